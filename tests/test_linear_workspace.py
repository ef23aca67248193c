"""The Linear Relation workspaces start at any 16-byte boundary: the library's arrays stand on a
boundary of their own inside the reported size."""
import pytest
import torch

from paper_2608_20172_gb300 import binding


def _up(n):
    return (n + 255) // 256 * 256


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,T", [(1, 1, 1), (1, 2, 128), (2, 3, 129), (1, 5, 700), (3, 1, 2048)])
def test_size_holds_the_arrays_and_the_alignment(B, H, T, d):
    """fp32 rows of 64 and their decays, for the backward a second set of rows: with 240 bytes in
    front of them (a base 16 bytes past a 256-byte boundary) they end inside the size."""
    rows = B * H * (d // 64) * -(-T // 128) * d
    one = _up(rows * 256) + _up(rows * 4)
    shp = binding.Shape(B, T, H, d, T * H * d, H * d, d)
    lib = binding.load()
    assert lib.relation_linear_fwd_workspace_size(shp, binding.BF16) >= 240 + one
    if d == 64:
        assert lib.relation_linear_bwd_workspace_size(shp, binding.BF16) >= 240 + one + rows * 256


@pytest.mark.gpu
@pytest.mark.parametrize("past", [0, 16, 48, 240])
def test_workspace_at_any_16_byte_boundary(past):
    """A workspace of exactly the reported size, `past` bytes past a 256-byte boundary in a larger
    buffer: the results of an aligned one, and nothing written outside it."""
    g = torch.Generator().manual_seed(past)
    dev = torch.device("cuda:0")
    B, T, H, d = 1, 700, 3, 64
    p1, p2, v, dy = (torch.randn((B, T, H, d), generator=g).to(torch.bfloat16).to(dev) for _ in range(4))
    alpha = (1.0 - 0.1 * torch.rand((B, T, H, d), generator=g)).to(dev)

    def ws(need):
        buf = torch.full((need + 1024,), 77, dtype=torch.uint8, device=dev)
        at = -buf.data_ptr() % 256 + past
        return buf, at, buf[at:at + need]

    def outside(buf, at, need):
        return bool((buf[:at] == 77).all()) and bool((buf[at + need:] == 77).all())

    need = binding.linear_fwd_workspace_size(p1)
    buf, at, part = ws(need)
    assert part.data_ptr() % 256 == past
    y = binding.linear_fwd_ws(p1, p2, v, alpha, workspace=part)
    ref = binding.linear_fwd_ws(p1, p2, v, alpha)
    torch.cuda.synchronize()
    assert torch.equal(y, ref) and outside(buf, at, need)
    assert bool((part != 77).any())  # the chunk-parallel form ran

    need = binding.linear_bwd_workspace_size(p1, "tcgen05")
    buf, at, part = ws(need)
    got = binding.linear_bwd(p1, p2, v, alpha, dy, kernel="tcgen05", workspace=part)
    ref = binding.linear_bwd(p1, p2, v, alpha, dy, kernel="tcgen05")
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, ref)) and outside(buf, at, need)


@pytest.mark.gpu
def test_stride_zero_along_one_entry():
    """A stride of 0 along a dimension of one entry: taken with few (head, column) pairs whatever the
    length, with the result of a plain stride, and refused with half as many pairs as SMs or more."""
    dev = torch.device("cuda:0")
    for T, H, ok in ((100, 3, True), (700, 3, True), (2048, 80, False), (100, 80, False)):
        g = torch.Generator().manual_seed(T + H)
        p1, p2, v = (torch.randn((1, T, H, 64), generator=g).to(torch.bfloat16).to(dev) for _ in range(3))
        alpha = (1.0 - 0.1 * torch.rand((1, T, H, 64), generator=g)).to(dev)
        x = [t.as_strided(t.shape, (0,) + t.stride()[1:]) for t in (p1, p2, v, alpha)]
        if not ok:
            with pytest.raises(binding.RelationError) as e:
                binding.linear_fwd_ws(*x)
            assert e.value.code == binding.ERR_INVALID_ARG
            continue
        y = binding.linear_fwd_ws(*x)
        ref = binding.linear_fwd_ws(p1, p2, v, alpha)
        torch.cuda.synchronize()
        assert float((y.float() - ref.float()).abs().max()) <= 2.0 ** -6 * float(ref.float().abs().max())
