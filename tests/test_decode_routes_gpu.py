"""relation_decode's two routes (a cluster per head for few heads and short caches; partial and
combine pass otherwise) and its three row scans, on the same sequences: against the oracle's
row, and against each other."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_20172_gb300 import binding, workloads
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
LAM = workloads.LAMBDA_INIT


# head sizes: the specialised ones, 16-byte groups that fill a warp and that leave lanes idle,
# whole and broken groups, one channel; lengths: no history, fewer rows than CTAs, tile and
# chunk edges, and the longest cache of the cluster route and one more row
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("d", [1, 30, 48, 64, 72, 80, 120, 128])
@pytest.mark.parametrize("T,lengths", [(1, [1]), (70, [2, 9, 70]), (4097, [4097, 513, 514]),
                                       (4098, [4098, 1025])])
def test_routes_agree(dtype, d, T, lengths):
    H, reps = 3, 40  # reps * lengths * H heads: past the cluster route
    n = len(lengths)
    g = torch.Generator().manual_seed(T + d)
    dt = torch.float32 if dtype == "fp32" else torch.bfloat16
    std = 1.0 / np.sqrt(d) if dtype == "fp32" else 1.0
    q = (torch.randn((n, H, d), generator=g) * std).to(dt)
    k, v = ((torch.randn((n, T, H, d), generator=g) * s).to(dt) for s in (std, 1.0))
    lens = torch.tensor(lengths, dtype=torch.int32)
    y, lz = binding.decode(q.to(DEV), k.to(DEV), v.to(DEV), lens.to(DEV), LAM)
    ym, lm = binding.decode(*(t.to(DEV).repeat((reps,) + (1,) * (t.dim() - 1)) for t in (q, k, v, lens)),
                            LAM)
    # a head's rows at an odd stride: no 16-byte groups
    wide = [torch.zeros(t.shape[:-1] + (d + 1,), dtype=dt, device=DEV) for t in (k, v)]
    for w, t in zip(wide, (k, v)):
        w[..., :d] = t.to(DEV)
    yo, lo = binding.decode(q.to(DEV), wide[0][..., :d], wide[1][..., :d], lens.to(DEV), LAM)
    torch.cuda.synchronize()
    for i, L in enumerate(lengths):
        for h in range(H):
            qs = np.zeros((L, d))
            qs[L - 1] = q[i, h].double().numpy()
            yr, lr = oracle.fwd_rows(qs, k[i, :L, h].double().numpy(), v[i, :L, h].double().numpy(),
                                     [L - 1], LAM)
            for a, b in ((y, lz), (ym, lm), (yo, lo)):
                pu.check(f"Y {L}", a[i, h][None].double().cpu().numpy(), yr, dtype, "out")
                pu.check_logz(f"logZ {L}", b[i, h][None].cpu().numpy(), lr, dtype)
    # the routes: fp32 sums in another order (1e-5 of O(1) rows), then rounded (2^-8)
    tol = 1e-5 if dtype == "fp32" else 2.0 ** -6
    for other, lother in ((ym[:n], lm[:n]), (ym[-n:], lm[-n:]), (yo, lo)):
        assert float((y.float() - other.float()).abs().max()) <= tol
        assert float((lz - lother).abs().max()) <= 1e-5


def test_bad_length_on_both_routes():
    for B in (2, 400):
        k = torch.ones((B, 16, 1, 64), device=DEV, dtype=torch.bfloat16)
        q = torch.ones((B, 1, 64), device=DEV, dtype=torch.bfloat16)
        lens = torch.full((B,), 16, dtype=torch.int32, device=DEV)
        lens[B - 1] = 17
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        y, _ = binding.decode(q, k, k, lens, LAM, dev_status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == binding.ERR_INVALID_ARG
        assert bool((y[: B - 1] == 1).all())  # the others are done
