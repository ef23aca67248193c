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
