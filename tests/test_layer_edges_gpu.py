"""The layer's transforms where their rotation tables and item loops change form: positions on
both sides of the two-float angle's range, frequencies outside it, CTAs of one position and of
sixteen, item counts around the threads of a CTA."""
import numpy as np
import pytest
import torch

from oracle import layer as lay
from paper_2608_20172_gb300 import binding
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


def _np(t):
    return t.double().cpu().numpy()


@pytest.mark.parametrize("base", [1.0e4, 1.0, 0.25])
@pytest.mark.parametrize("T,H,d", [(1, 2, 8), (16, 2, 128), (17, 4, 24), (33, 8, 128), (15, 6, 256)])
def test_tables_and_item_loops(base, T, H, d):
    g = torch.Generator().manual_seed(T * H + d)
    x = [torch.randn((2, T, H, d), generator=g) for _ in range(4)]
    theta = (torch.rand(H // 2, generator=g) * 6.0 - 3.0).float()
    y = [t.to(DEV) for t in x]
    q, k, v = binding.layer_prep(*y[:3], theta.to(DEV), 1, base)
    g1, g2, gi, gt = binding.layer_grad(*y, theta.to(DEV), 1, base)
    torch.cuda.synchronize()
    th = theta.double().numpy()
    n = [_np(t) for t in x]
    _, _, rv = lay.prep(*n[:3], th, 1)
    _, _, ri, rt = lay.grad(*n, th, 1)
    for name, got, ref in [("q", q, lay.rope(n[0], base)), ("k", k, lay.rope(n[1], base)), ("v", v, rv),
                           ("dp1", g1, lay.rope(n[0], base, inverse=True)),
                           ("dp2", g2, lay.rope(n[1], base, inverse=True)), ("dinfo", gi, ri)]:
        pu.check(name, _np(got), ref, "fp32", "grad" if name[0] == "d" else "out")
    for j in range(len(rt)):
        pu.check_dlambda(float(gt[j].item()), float(rt[j]), "fp32")


def test_positions_around_the_two_float_range():
    """2^22 positions and a few more: the last two-float CTAs and the first fp64 ones.  An angle
    is good to a few 2^-24 pi, so the rotated rows (|x| < 6) to ~1e-5 at most."""
    T, n = (1 << 22) + 20, 64
    g = torch.Generator().manual_seed(9)
    tail = torch.randn((1, n, 2, 8), generator=g)
    x = torch.zeros((1, T, 2, 8), device=DEV)
    x[:, -n:] = tail.to(DEV)
    q, k, v = binding.layer_prep(x, x, x, torch.zeros(1, device=DEV), 0)
    torch.cuda.synchronize()
    a = lay.rope_angles(T, 8)[-n:][None, :, None, :]
    e, o = _np(tail)[..., 0::2], _np(tail)[..., 1::2]
    for got in (_np(q[:, -n:]), _np(k[:, -n:])):
        assert np.max(np.abs(got[..., 0::2] - (e * np.cos(a) - o * np.sin(a)))) <= 2e-5
        assert np.max(np.abs(got[..., 1::2] - (e * np.sin(a) + o * np.cos(a)))) <= 2e-5
    assert torch.equal(v, x)
