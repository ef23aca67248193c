"""More sequences than a grid has CTAs for: the layer's passes come in several launches."""
import pytest
import torch

from paper_2608_20172_gb300 import binding

pytestmark = pytest.mark.gpu


def test_more_sequences_than_a_grid_holds():
    """2^30 + 3 sequences of one position (rotation angle 0) with mixing angles of 0: both passes are
    the identity.  A sequence's two rows of 8 start 8 elements after the last one's, so that a buffer
    of 17 GB holds them all and every element is written by its rows' owners alike."""
    B, dev = (1 << 30) + 3, torch.device("cuda:0")
    n = 8 * (B + 1)
    x = torch.randint(-(1 << 15), 1 << 15, (n,), dtype=torch.int16, device=dev)
    x.bitwise_and_(0x3FFF)  # finite bf16 values
    y = torch.zeros(n, dtype=torch.int16, device=dev)
    rows = [t.view(torch.bfloat16).as_strided((B, 1, 2, 8), (8, 16, 8, 1)) for t in (x, y)]
    theta = torch.zeros(1, device=dev)
    q = rows[1]
    binding.layer_prep(rows[0], rows[0], rows[0], theta, out=(q, q, q))
    torch.cuda.synchronize()
    assert torch.equal(x, y)
    y.zero_()
    lib, shp = binding.load(), binding.shape_of(q)
    ws = torch.empty(binding.layer_grad_workspace_size(q), dtype=torch.uint8, device=dev)
    dth = torch.empty(1, device=dev)
    p, o = x.data_ptr(), y.data_ptr()
    rc = lib.relation_layer_grad(p, p, p, p, theta.data_ptr(), 0, 1.0e4, o, o, o, dth.data_ptr(), shp,
                                 binding.BF16, ws.data_ptr(), ws.numel(),
                                 torch.cuda.current_stream().cuda_stream)
    assert rc == binding.OK
    torch.cuda.synchronize()
    assert torch.equal(x, y)
    # dtheta's terms are a rounding error each (dv = info); every partial was written
    assert bool((ws.view(torch.float32).abs() < 1e-6).all())
