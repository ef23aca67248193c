"""Few query tiles: a cluster of CTAs shares a tile's keys and merges (m, l, z).  The same heads in
a batch that fills the GPU take one CTA per tile; both against the oracle and each other."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_20172_gb300 import binding, workloads
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
LAM = workloads.LAMBDA_INIT


# clusters of 2, 4 and 8 at d_h <= 64 (T 512 is their first length), of 2 and 4 above (640, 1280), ragged
# last tiles, padded widths; the first query tiles of a head leave shares empty
@pytest.mark.parametrize("T,d,reps", [(512, 64, 320), (777, 40, 320), (1024, 64, 320),
                                      (2048, 64, 320), (2047, 8, 320), (640, 128, 64), (1280, 128, 64),
                                      (1409, 80, 64)])
def test_split_rows(T, d, reps):
    H = 2 if T < 2047 else 1
    g = torch.Generator().manual_seed(T)
    q, k, v = (torch.randn((1, T, H, d), generator=g).to(torch.bfloat16) for _ in range(3))
    dev = [t.to(DEV) for t in (q, k, v)]
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    y, lz, f = binding.fwd_flow(*dev, LAM, dev_status=status)
    n = -(-reps // H)
    ym, lm, fm = binding.fwd_flow(*(t.expand(n, T, H, d).contiguous() for t in dev), LAM)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    rows = sorted({0, 1, 127, 128, T // 2, T - 2, T - 1})
    for h in range(H):
        yr, lr = oracle.fwd_rows(q[0, :, h].double().numpy(), k[0, :, h].double().numpy(),
                                 v[0, :, h].double().numpy(), rows, LAM)
        pu.check(f"Y {h}", y[0, rows, h].double().cpu().numpy(), yr, "bf16", "out")
        pu.check_logz(f"logZ {h}", lz[0, h, rows].cpu().numpy(), lr, "bf16")
    pu.check("Y", y[0].double().cpu().numpy(), ym[0].double().cpu().numpy(), "bf16", "out")
    assert float((lz[0] - lm[0]).abs().max()) <= 2e-5  # fp32 sums in another order, |logZ| < 16
    assert float((f[0] - fm[0]).abs().max()) <= 2e-5


@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("Tq,Tk,d,reps", [(256, 1500, 64, 320), (129, 1290, 128, 160)])
def test_split_summaries(causal, Tq, Tk, d, reps):
    if causal:
        Tq = Tk
    g = torch.Generator().manual_seed(Tk)
    q = torch.randn((1, Tq, 1, d), generator=g).to(torch.bfloat16).to(DEV)
    k, v = (torch.randn((1, Tk, 1, d), generator=g).to(torch.bfloat16).to(DEV) for _ in range(2))
    one = binding.fwd_state(q, k, v, causal)
    many = binding.fwd_state(*(t.expand(reps, -1, -1, -1).contiguous() for t in (q, k, v)), causal)
    torch.cuda.synchronize()
    (m, l, z), (mm, lm, zm) = one, [t[:1] for t in many]
    live = lm > 0
    assert torch.equal(l > 0, live)
    # log of the row's sum, and the weighted mean of v (P rounds to bf16 at the row's own scale)
    a, b = (m + l.log())[live], (mm + lm.log())[live]
    assert float((a - b).abs().max()) <= 2e-5
    pu.check("mean", (z[live] / l[live][:, None]).double().cpu().numpy(),
             (zm[live] / lm[live][:, None]).double().cpu().numpy(), "bf16", "out")
    assert bool((z[~live] == 0).all())
