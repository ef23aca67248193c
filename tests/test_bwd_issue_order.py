"""The issue order of the backward tile kernel's d_h = 64 form (relation_tc_bwd.cu): behind step s the
products of the steps up to s + NBUF, with no test that the Q / dO stages they load into have been
released.  The roles of test_bwd_protocol_model with this order for the MMA warp, at the kernel's
constants and on both sides of its two static assertions.  CPU only."""
import random

import pytest

from tests import test_bwd_protocol_model as model


def mma(units):
    NBUF, NQS, SPT, NKV = model.NBUF, model.NQS, model.SPT, model.NKV
    gs0 = gt0 = pre = issued = 0  # issued: tiles whose stage the issue loop has waited for

    def issue(base, s):
        nonlocal issued
        if s % SPT == 0:
            yield ("wait", f"QF{issued % NQS}", issued // NQS)
            issued += 1
        yield ("arrive", f"S{(base + s) % NBUF}")

    for ul, n_i in enumerate(units):
        total = n_i * SPT
        if pre == 0:
            yield ("wait", f"KV{ul % NKV}", ul // NKV)
        sn, pre = pre, 0
        while sn < total and sn < NBUF:
            yield from issue(gs0, sn)
            sn += 1
        for s in range(total):
            g = gs0 + s
            yield ("wait", f"P{g % NBUF}", g // NBUF)
            if s == total - 1:
                yield ("arrive", "ACC")
                if ul + 1 < len(units):
                    yield ("wait", f"KV{(ul + 1) % NKV}", (ul + 1) // NKV)
                    while pre < units[ul + 1] * SPT and pre < NBUF:
                        yield from issue(gs0 + total, pre)
                        pre += 1
            if s % SPT == SPT - 1:
                gt = gt0 + s // SPT
                if gt > 0:
                    yield ("wait", "DQE", gt - 1)
                yield ("arrive", "DQF")
                yield ("arrive", f"QE{gt % NQS}")
            while sn < total and sn <= s + NBUF:
                yield from issue(gs0, sn)
                sn += 1
        yield ("arrive", f"KVE{ul % NKV}")
        gs0 += total
        gt0 += n_i


def run(units, seed, monkeypatch):
    monkeypatch.setattr(model, "mma", mma)
    model.run(units, seed)


@pytest.mark.parametrize("n_t,BH,grid", [(1, 400, 152), (2, 400, 152), (8, 128, 152), (16, 96, 152)])
def test_issue_order_of_real_unit_sequences(n_t, BH, grid, monkeypatch):
    for c in sorted({0, 1, grid // 2, grid - 1}):
        units = model.cta_units(n_t, BH, grid, c)
        for seed in range(25):
            run(units, seed, monkeypatch)


# (NBUF, NQS, SPT): the kernel's; each assertion met with nothing to spare; each just broken
@pytest.mark.parametrize("nbuf,nqs,spt,ok", [(2, 2, 2, True), (3, 2, 4, True), (5, 2, 4, False),
                                             (4, 3, 2, True), (4, 2, 3, False), (3, 2, 2, False),
                                             (2, 3, 1, True), (3, 3, 1, False), (6, 2, 4, False)])
def test_assertions(nbuf, nqs, spt, ok, monkeypatch):
    assert ok == (nbuf <= (nqs - 1) * spt + 1 and (nbuf - 1) // spt <= nqs - 2)
    for name, value in (("NBUF", nbuf), ("NQS", nqs), ("SPT", spt)):
        monkeypatch.setattr(model, name, value)
    rng = random.Random(3)
    stuck = 0
    for trial in range(60):
        units = [rng.randint(1, 6) for _ in range(rng.randint(2, 5))]
        try:
            run(units, trial, monkeypatch)
        except AssertionError as e:
            assert "deadlock" in str(e)
            stuck += 1
    assert (stuck == 0) == ok
