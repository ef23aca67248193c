"""The CUDA-core backward with dQ in the place of Q or of dO (equal strides): the same gradients."""
import pytest
import torch

from paper_2608_20172_gb300 import binding

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("T,d,H", [(33, 64, 2), (700, 64, 4), (1500, 32, 6), (300, 128, 2)])
@pytest.mark.parametrize("place", ["q", "do"])
def test_dq_in_place(dtype, T, d, H, place):
    g = torch.Generator().manual_seed(T + d)
    q, k, v, do = (torch.randn((2, T, H, d), generator=g).to(dtype).to(DEV) for _ in range(4))
    y, lz = binding.fwd(q, k, v, 0.5, kernel="simt")
    ref = binding.bwd(q, k, v, y, do, lz, 0.5, kernel="simt")
    q2, do2 = q.clone(), do.clone()
    got = binding.bwd(q2, k, v, y, do2, lz, 0.5, kernel="simt", dq=q2 if place == "q" else do2)
    torch.cuda.synchronize()
    assert got[0].data_ptr() == (q2 if place == "q" else do2).data_ptr()
    tol = 2e-6 if dtype == torch.float32 else 2.0 ** -7
    for a, b in zip(got, ref):
        # (fp32 sums: one group of warps or two)
        assert float((a.float() - b.float()).abs().max()) <= tol * float(b.float().abs().max())
