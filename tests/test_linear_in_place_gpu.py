"""The chunked Linear Relation backward with dalpha in alpha's place (C ABI): the same gradients, with
few small retentions in a block, many, or none."""
import pytest
import torch

from paper_2608_20172_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_small", [0, 1, 16, 17])
def test_dalpha_in_place(n_small):
    g = torch.Generator().manual_seed(n_small)
    dev = torch.device("cuda:0")
    B, T, H, d = 1, 300, 2, 64
    p1, p2, v, dy = (torch.randn((B, T, H, d), generator=g).to(torch.bfloat16).to(dev) for _ in range(4))
    alpha = 1.0 - 0.1 * torch.rand((B, T, H, d), generator=g)
    for h in range(H):
        for i in torch.randperm(128 * d, generator=g)[:n_small].tolist():
            alpha[0, 128 + i // d, h, i % d] = 2.0 ** -13
    alpha = alpha.to(dev)
    ref = binding.linear_bwd(p1, p2, v, alpha, dy, kernel="tcgen05")
    out, al = [torch.empty_like(p1) for _ in range(3)], alpha.clone()
    ws = torch.empty(binding.linear_bwd_workspace_size(p1, "tcgen05"), dtype=torch.uint8, device=dev)
    rc = binding.load().relation_linear_bwd_ex(
        *(t.data_ptr() for t in (p1, p2, v, al, dy, *out, al)), 2.0, binding.shape_of(p1), binding.BF16,
        binding.KERNELS["tcgen05"], ws.data_ptr(), ws.numel(), None,
        torch.cuda.current_stream().cuda_stream)
    assert rc == binding.OK
    torch.cuda.synchronize()
    for a, b in zip((*out, al), ref):
        assert torch.equal(a, b)
