"""Back-to-back launches: every kernel waits for the ones before it in the stream, whoever launched
them.  Chains of calls whose buffers each call overwrites for the next, against the same chain with
a synchronisation after every call; eager, captured in a graph, and on two streams at once."""
import pytest
import torch

from paper_2608_20172_gb300 import binding

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


class Chain:
    """Two rounds over the same buffers; the second round's inputs are the first's outputs."""

    def __init__(self, dtype, seed):
        g = torch.Generator().manual_seed(seed)
        dt = torch.bfloat16 if dtype == "bf16" else torch.float32
        self.x = [torch.randn((2, 600, 4, 64), generator=g).to(dt).to(DEV) for _ in range(4)]
        self.theta = torch.rand(2, generator=g).to(DEV)
        self.alpha = (1.0 - 0.1 * torch.rand((2, 600, 4, 64), generator=g)).to(DEV)
        self.lens = torch.tensor([600, 333], dtype=torch.int32, device=DEV)
        q = self.x[0]
        self.ws = torch.empty(binding.workspace_size(q), dtype=torch.uint8, device=DEV)
        self.dtype = dtype

    def run(self, sync=lambda: None):
        a, b, c, dy = (t.clone() for t in self.x)
        out = []
        for _ in range(2):
            q, k, v = binding.layer_prep(a, b, c, self.theta)
            sync()
            y, lz = binding.fwd(q, k, v, 0.5)
            sync()
            dq, dk, dv, dl = binding.bwd(q, k, v, y, dy, lz, 0.5, workspace=self.ws)
            sync()
            g1, g2, gi, gt = binding.layer_grad(dq, dk, dv, c, self.theta)
            sync()
            yd, lzd = binding.decode(y[:, -1].contiguous(), k, v, self.lens, 0.5)
            sync()
            lin = binding.linear_fwd_ws(q, k, v, self.alpha)
            sync()
            self.ws.fill_(255)  # (a stale workspace is no input)
            sync()
            out += [q, k, v, y, lz, yd, lzd, lin]  # deterministic
            tol = [dq, dk, dv, g1, g2, gi]         # dQ of bf16: sums in any order
            if self.dtype == "bf16":
                st = binding.fwd_state(q, k, v, True)
                sync()
                binding.state_merge(st, binding.fwd_state(q, k, v, False))
                sync()
                out += list(st) + list(binding.state_finish(q, k, v, st, 0.5))
                sync()
            a.copy_(y)
            b.copy_(lin)
            c.copy_(yd[:, None].expand_as(c))
            dy.mul_(0.5)
            sync()
        return out, tol


def _same(got, ref):
    for x, y in zip(got[0], ref[0]):
        assert torch.equal(x, y)
    for x, y in zip(got[1], ref[1]):
        n = float(y.double().norm())
        assert float((x.double() - y.double()).norm()) <= 1e-4 * n


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_back_to_back_calls(dtype):
    c = Chain(dtype, 1)
    ref = c.run(torch.cuda.synchronize)
    for _ in range(3):
        got = c.run()
        torch.cuda.synchronize()
        _same(got, ref)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        c.run()
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            got = c.run()
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        _same(got, ref)


def test_two_streams():
    chains = [Chain("bf16", 2), Chain("fp32", 3)]
    refs = [c.run(torch.cuda.synchronize) for c in chains]
    streams = [torch.cuda.Stream() for _ in chains]
    torch.cuda.synchronize()
    for _ in range(3):
        got = []
        for c, s in zip(chains, streams):
            with torch.cuda.stream(s):
                got.append(c.run())
        torch.cuda.synchronize()
        for g, r in zip(got, refs):
            _same(g, r)
