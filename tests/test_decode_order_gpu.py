"""Decode steps back to back: what the kernels launched before a step have written (lengths, the new
cache rows, the query) is what both of its passes read.  Chains against the same chain with a
synchronisation after every launch, on the route of two launches and on that of one."""
import pytest
import torch

from paper_2608_20172_gb300 import binding

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
STEPS = 12


def _chain(q0, k0, v0, lens0, sync):
    """STEPS tokens: every step advances the lengths, writes the new rows from the last output,
    which is also the next query, and decodes."""
    q, k, v, lens = (t.clone() for t in (q0, k0, v0, lens0))
    rows = torch.arange(q.shape[0], device=DEV)
    out = []
    for _ in range(STEPS):
        lens.add_(1)
        sync()
        at = (lens - 1).long()
        k[rows, at] = q
        sync()
        v[rows, at] = -q
        sync()
        y, lz = binding.decode(q, k, v, lens, 0.5)
        sync()
        q.copy_(y).mul_(1.5).add_(0.1)
        sync()
        out += [y, lz]
    return out


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,d", [(48, 64), (48, 128), (48, 80), (48, 30), (4, 64)])
def test_a_step_reads_what_came_before_it(dtype, B, d):
    H, T = 2, 1100
    g = torch.Generator().manual_seed(B + d)
    dt = torch.float32 if dtype == "fp32" else torch.bfloat16
    k, v = (torch.randn((B, T, H, d), generator=g).to(dt).to(DEV) for _ in range(2))
    q = torch.randn((B, H, d), generator=g).to(dt).to(DEV)
    lens = torch.randint(1, T - STEPS, (B,), generator=g, dtype=torch.int32).to(DEV)
    lens[0], lens[1] = 510, 1  # chunk edges on the way, and hardly any history
    ref = _chain(q, k, v, lens, torch.cuda.synchronize)
    for _ in range(3):
        got = _chain(q, k, v, lens, lambda: None)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, ref))
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            got = _chain(q, k, v, lens, lambda: None)
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, ref))
