"""RoPE angles at long positions: what fp64 gives, rounded to fp32."""
import numpy as np
import pytest
import torch

from paper_2608_20172_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [(1 << 15) + 16, 1 << 18, (1 << 22) - 16])
def test_angles_are_fp64_rounded(T):
    """Rows (1, 0, 1, 0, ...) come back as the cosines and sines of the last positions' angles: of the
    angle modulo 2 pi in fp64, rounded to fp32, to 2 ulp (the bound of sincosf).  An angle one fp32
    unit off shows, where it is above 2, as up to 2.4e-7.  Where a rounding is close to a tie the last
    bit of a frequency's exponential may turn it: at T 2^22 2^22 2^-53 / 2^-23, 0.4 %, of them, of
    which a third is above 2."""
    d, n, dev = 64, 512, torch.device("cuda:0")
    x = torch.zeros((1, T, 2, d), device=dev)
    x[..., 0::2] = 1.0
    q, _, _ = binding.layer_prep(x, x, x, torch.zeros(1, device=dev), 0)
    got = q[0, -n:, 0].double().cpu().numpy()
    c = np.arange(d // 2)
    a = np.arange(T - n, T, dtype=np.float64)[:, None] * np.exp(-2.0 * c / d * np.log(1.0e4))
    turns = np.rint(a * 0.15915494309189533576888376337251)
    r = (a.astype(np.longdouble) - turns.astype(np.longdouble) * np.longdouble(6.283185307179586476925286766559))
    r = r.astype(np.float32).astype(np.float64)
    off = np.maximum(np.abs(got[:, 0::2] - np.cos(r)), np.abs(got[:, 1::2] - np.sin(r))) > 2.0 ** -23
    assert off.mean() <= 0.0015
