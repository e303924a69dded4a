"""Requests of a wave that run as binary polynomials, one group of launches a length:
every kind at the edges of its operands, constant Dodis et al. inputs reported
alone, and never more scratch than admission reserved."""

import time

import numpy as np
import pytest
import torch

import oracle
from oracle import extractors as ex
from paper_2402_09481_gb300 import inputs, native
from conftest import from_dev, to_dev

pytestmark = pytest.mark.gpu
T, C, D = native.TOEPLITZ, native.CIRCULANT, native.DODIS


def ybits(kind, n, m):
    return n + m - 1 if kind == T else (n + 1 if kind == C else n)


def make(kind, n, m, s0, const_x=None):
    xw = inputs.bernoulli_half(s0, n)
    if const_x is not None:
        xw = ex.pack_bits(np.full(n, const_x, dtype=np.uint8))
    elif kind == D:
        xw[0] = (xw[0] | np.uint64(1)) & ~np.uint64(2)
    z = torch.full((native.words(m),), -1, dtype=torch.int64, device="cuda")
    return [kind, n, m, to_dev(xw), to_dev(inputs.bernoulli_half(s0 + 1, ybits(kind, n, m))), z]


def alone(ctx, r):
    kind, n, m, x, y, _ = r
    z = torch.full_like(r[5], -1)
    if kind == T:
        return ctx.toeplitz(x, n, y, m, z)
    if kind == C:
        return ctx.circulant(x, n, y, m, z)
    return ctx.dodis(x, y, n, m, z)


@pytest.fixture
def sctx():
    from paper_2402_09481_gb300 import build
    build.build()
    ctx = native.Context(0)
    yield ctx
    ctx.close()


@pytest.fixture(scope="module")
def q30():
    from paper_2402_09481_gb300 import build
    build.build()
    c = native.Context(0, field=native.FIELD_Q30)
    yield c
    c.close()


def busy(ctx, slots):
    end = time.time() + 20
    while ctx.server_stats()["busy_slots"] < slots:
        assert time.time() < end


def collect(ctx, tickets):
    out = []
    for t in tickets:
        s, r = ctx.poll(t, 60.0)
        assert s == native.CM_OK
        out.append(r)
    return out


def test_groups_within_the_admitted_scratch(sctx, cm_ctx):
    # two arrays of 2^24 bits (4 MB) do not fit what the planner's blocks take of a
    # 2 MB budget: in a wave with others such a request keeps its blocks.  The
    # first request holds the budget while the others queue behind it.
    n, m, budget = 16_000_000, 100_000, 2 << 20
    assert native.plan_query(T, n, m, hbm_budget_bytes=budget)["scratch_bytes"] + 4096 < budget < 1 << 22
    longs = [make(T, n, m, 100 + 2 * j) for j in range(2)]
    shorts = [make(T, 300 + j, 200, 110 + 2 * j) for j in range(4)]
    torch.cuda.synchronize()
    sctx.server_start(hbm_budget_bytes=budget, slots=1, express_slots=native.SERVER_NO_EXPRESS)
    sctx.profile_enable(True)
    sctx.profile_read(reset=True)
    tickets = [sctx.submit(*longs[0])]
    busy(sctx, 1)
    tickets.append(sctx.submit(*shorts[0]))  # takes the stream's second slot, behind the long one
    busy(sctx, 2)
    tickets += [sctx.submit(*r) for r in shorts[1:] + longs[1:]]
    res = collect(sctx, tickets)
    st = sctx.server_stats()
    sctx.server_stop()
    prof = sctx.profile_read(reset=True)
    sctx.profile_enable(False)
    assert all(r["status"] == native.CM_OK for r in res)
    assert len({r["wave"] for r in res[2:]}) == 1  # the second long one shared a wave
    assert not any(k in prof for k in ("k_gf_rows", "k_gf_units", "k_gf_mid")), prof
    assert st["max_inflight_bytes"] <= budget
    for r in longs + shorts:
        assert torch.equal(r[5], alone(cm_ctx, r))


def test_groups_every_kind(sctx, q30):
    # long requests hold the stream while the others queue: they make one wave
    specs = []
    for lg, copies in ((18, 4), (19, 2), (21, 1), (23, 1)):
        L = 1 << lg
        for j in range(copies):
            specs += [(T, L - L // 3 - j, L // 3 + 1, None), (T, 5, L - 4 - j, None),
                      (C, oracle.next_na(L // 2 + 7 + j) - 1, L // 4 + 3, None),
                      (D, oracle.next_na(L * 5 // 9), L // 3 + j, None),
                      (D, oracle.next_na(L * 5 // 9), L // 3 + j, j & 1)]
    reqs = [make(k, n, m, 200 + 2 * j, c) for j, (k, n, m, c) in enumerate(specs)]
    hold = [make(T, 2 ** 27, 2 ** 26, 900 + 2 * j) for j in range(2)]  # past the groups
    torch.cuda.synchronize()
    sctx.server_start(slots=1, express_slots=native.SERVER_NO_EXPRESS)
    sctx.profile_enable(True)
    sctx.profile_read(reset=True)
    tickets = [sctx.submit(*hold[0])]
    busy(sctx, 1)
    tickets.append(sctx.submit(*hold[1]))
    busy(sctx, 2)
    tickets += [sctx.submit(*r) for r in reqs]
    res = collect(sctx, tickets)[2:]
    sctx.server_stop()
    prof = sctx.profile_read(reset=True)
    sctx.profile_enable(False)
    assert {r["wave"] for r in res} == {res[0]["wave"]}
    assert prof["k_gf_mid"][0] == 4 and prof["k_gf_same"][0] == 1 and "k_batch" not in prof, prof
    for (kind, n, m, c), r, q in zip(specs, reqs, res):
        assert q["status"] == (native.CM_OK if c is None else native.CM_EPRECOND), (kind, n, m, c)
        if c is not None:
            assert not from_dev(r[5]).any()
        else:
            assert torch.equal(r[5], alone(q30, r)), (kind, n, m)
