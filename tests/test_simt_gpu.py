"""The CUDA-core kernels at the edges of their 8-row warps, 32-row CTAs and 64-row tiles, and
their masks: rows outside a row's history hold anything and must not enter, not even times
zero."""
import numpy as np
import pytest
import torch

from paper_2608_20172_gb300 import binding, workloads
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

LAM = workloads.LAMBDA_INIT


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("T", [7, 8, 9, 31, 33, 63, 64, 97, 193])
def test_tile_edges(T, d):
    w = workloads.custom(1, 3, T, d, "fp32", qk_std=1.0)
    q, k, v, do = workloads.make_inputs(w, seed=10 * T + d)
    res = pu.gpu_run(q, k, v, do, LAM, kernel="simt")
    ref = pu.oracle_heads(q, k, v, do, LAM, [(0, h) for h in range(3)])
    pu.compare_heads(res, ref, "fp32")
    pu.check_dlambda(res["dlambda"], sum(r["dlambda"] for r in ref.values()), "fp32")


@pytest.mark.parametrize("cut", [5, 40, 64, 100])
def test_rows_outside_the_history_never_enter(cut):
    """NaN in V from row `cut` on leaves Y before it as it was; NaN in dO before row `cut`
    leaves dK and dV of the keys from `cut` on as they were."""
    w = workloads.custom(1, 2, 150, 64, "fp32")
    q, k, v, do = (t.cuda() for t in workloads.make_inputs(w, seed=3))
    y, logz = binding.fwd(q, k, v, LAM, kernel="simt")
    vn = v.clone()
    vn[:, cut:] = float("nan")
    yn, _ = binding.fwd(q, k, vn, LAM, kernel="simt")
    assert torch.equal(yn[:, :cut], y[:, :cut])
    _, dk, dv, _ = binding.bwd(q, k, v, y, do, logz, LAM, kernel="simt")
    dn = do.clone()
    dn[:, :cut] = float("nan")
    _, dkn, dvn, _ = binding.bwd(q, k, v, y, dn, logz, LAM, kernel="simt")
    assert torch.equal(dkn[:, cut:], dk[:, cut:]) and torch.equal(dvn[:, cut:], dv[:, cut:])
    assert np.isfinite(dk.cpu().numpy()).all()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("T,d", [(65, 64), (96, 32), (129, 64), (160, 128), (193, 32), (300, 64),
                                 (321, 128)])
def test_one_and_two_groups_of_warps(T, d, dtype):
    """A few heads take CTAs whose two groups of warps share a row's tiles, the same heads in a
    large batch CTAs of one group: the large batch against the oracle, and both against each other
    (fp32 sums in another order, a few 1e-7 of the largest value; bf16 outputs then rounded)."""
    H, n = 2, -(-1300 // (2 * (T // 32)))
    w = workloads.custom(1, H, T, d, dtype, qk_std=1.0)
    x = workloads.make_inputs(w, seed=T + d)
    many = [t.expand(n, T, H, d).contiguous() for t in x]
    out = []
    for q, k, v, do in (x, many):
        q, k, v, do = (t.cuda() for t in (q, k, v, do))
        y, lz = binding.fwd(q, k, v, LAM, kernel="simt")
        dq, dk, dv, dl = binding.bwd(q, k, v, y, do, lz, LAM, kernel="simt")
        out.append([t[:1].float() for t in (y, lz, dq, dk, dv)])
    for a, b in zip(*out):
        tol = 2e-6 if a.dtype == torch.float32 and dtype == "fp32" else 2.0 ** -7
        assert float((a - b).abs().max()) <= tol * float(b.abs().max())
    res = {k: t.cpu() for k, t in zip(("Y", "logZ", "dQ", "dK", "dV"), out[1])}
    ref = pu.oracle_heads(*x, LAM, [(0, h) for h in range(H)])
    pu.compare_heads(res, ref, dtype)
