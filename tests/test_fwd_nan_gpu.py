"""NaN in an input reaches the rows that read it, and no others, however a row's keys are shared out:
over clusters of CTAs, groups of warps or neither."""
import pytest
import torch

from paper_2608_20172_gb300 import binding

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
LAM = 0.5


def _inputs(T, H, d, dtype, seed):
    g = torch.Generator().manual_seed(seed)
    return [torch.randn((1, T, H, d), generator=g).to(dtype).to(DEV) for _ in range(3)]


def _rows(x):
    """[T] flags: rows of head 0 with a NaN."""
    return torch.isnan(x[0, :, 0].float()).any(-1)


# T 512 to 2048: clusters of 2, 4 and 8; T 100: one CTA per tile
@pytest.mark.parametrize("T,d", [(100, 64), (512, 64), (777, 64), (2048, 64), (1280, 128)])
def test_nan_query_split(T, d):
    q, k, v = _inputs(T, 1, d, torch.bfloat16, T)
    y0, lz0 = binding.fwd(q, k, v, LAM)
    m0, l0, z0 = binding.fwd_state(q, k, v, False)
    r = T - 3
    q[0, r] = float("nan")
    y, lz = binding.fwd(q, k, v, LAM)
    m, l, z = binding.fwd_state(q, k, v, False)
    torch.cuda.synchronize()
    others = torch.arange(T, device=DEV) != r
    assert bool(torch.isnan(y[0, r].float()).all()) and bool(torch.isnan(lz[0, 0, r]))
    assert torch.equal(y[0, others], y0[0, others]) and torch.equal(lz[0, 0, others], lz0[0, 0, others])
    assert bool(torch.isnan(l[0, 0, r])) and bool(torch.isnan(z[0, 0, r]).all())
    assert torch.equal(l[0, 0, others], l0[0, 0, others]) and torch.equal(z[0, 0, others], z0[0, 0, others])


# a key that is the only one of its CTA's share for the first rows behind it
@pytest.mark.parametrize("T,d,j", [(777, 64, 0), (777, 64, 640), (2048, 64, 1920), (1280, 128, 1152)])
def test_nan_key_split(T, d, j):
    q, k, v = _inputs(T, 1, d, torch.bfloat16, T + j)
    y0, _ = binding.fwd(q, k, v, LAM)
    k[0, j] = float("nan")
    y, lz = binding.fwd(q, k, v, LAM)
    torch.cuda.synchronize()
    bad = _rows(y)
    assert bool(bad[j + 1:].all()) and not bool(bad[:j].any())
    assert torch.equal(y[0, :j], y0[0, :j])


# T 65 and 70: the second group of warps has one to six keys of the last rows; T 300: several tiles;
# many heads: one group
@pytest.mark.parametrize("T,d,H,j", [(70, 64, 1, 64), (70, 32, 1, 0), (300, 64, 1, 64), (300, 128, 1, 192),
                                     (300, 64, 256, 64), (40, 64, 1, 0)])
def test_nan_key_simt(T, d, H, j):
    q, k, v = _inputs(T, H, d, torch.float32, T + j)
    y0, _ = binding.fwd(q, k, v, LAM)
    k[0, j] = float("nan")
    y, _ = binding.fwd(q, k, v, LAM)
    torch.cuda.synchronize()
    bad = _rows(y)
    assert bool(bad[j + 1:].all()) and not bool(bad[:j].any())
    assert torch.equal(y[0, :j], y0[0, :j])
