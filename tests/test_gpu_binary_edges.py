"""The binary form's groups of short transforms, every kind and edge of the operands in
batches long enough that a length runs as a group, and the tensor-core form's
longest share of terms."""

import numpy as np
import pytest
import torch

import oracle
from oracle import extractors as ex
from paper_2402_09481_gb300 import inputs, native
from conftest import from_dev, to_dev

pytestmark = pytest.mark.gpu
T, C, D = native.TOEPLITZ, native.CIRCULANT, native.DODIS


@pytest.fixture(scope="module")
def q30():
    from paper_2402_09481_gb300 import build
    build.build()
    c = native.Context(0, field=native.FIELD_Q30)
    yield c
    c.close()


def ybits(kind, n, m):
    return n + m - 1 if kind == T else (n + 1 if kind == C else n)


def run(ctx, kind, n, m, x, y):
    z = torch.full((native.words(m),), -1, dtype=torch.int64, device="cuda")
    if kind == T:
        return ctx.toeplitz(x, n, y, m, z)
    if kind == C:
        return ctx.circulant(x, n, y, m, z)
    return ctx.dodis(x, y, n, m, z)


@pytest.mark.parametrize("lg,count", [(15, 64), (16, 32), (17, 32), (18, 16), (19, 16), (20, 8)])
def test_batch_group_every_kind(cm_ctx, q30, lg, count):
    L, s0 = 2 ** lg, 2000 + 20 * lg
    P = oracle.next_na(L * 5 // 9)
    specs = [(T, L - L // 3, L // 3 + 1, None), (T, L // 2, 2, None), (T, 5, L - 4, None),
             (C, oracle.next_na(L // 2 + 7) - 1, L // 4 + 3, None), (D, P, L // 3, None), (D, P, L // 3 - 1, 0),
             (D, P, L // 3 - 2, 1)]
    made = []
    for j, (kind, n, m, const) in enumerate(specs):
        xw = inputs.bernoulli_half(s0 + 2 * j, n) if const is None else ex.pack_bits(np.full(n, const, dtype=np.uint8))
        if kind == D and const is None:
            xw[0] = (xw[0] | np.uint64(1)) & ~np.uint64(2)
        x, y = to_dev(xw), to_dev(inputs.bernoulli_half(s0 + 2 * j + 1, ybits(kind, n, m)))
        made.append((kind, n, m, x, y, run(q30, kind, n, m, x, y) if const is None else None))
    items = []
    for i in range(count):  # copies of the seven share inputs
        kind, n, m, x, y, _ = made[i % len(made)]
        items.append((kind, n, m, x, y, torch.full((native.words(m),), -1, dtype=torch.int64, device="cuda")))
    cm_ctx.device_status()
    cm_ctx.profile_enable(True)
    cm_ctx.profile_read(reset=True)
    cm_ctx.batch_extract(items)
    prof = cm_ctx.profile_read(reset=True)
    cm_ctx.profile_enable(False)
    assert prof["k_gf_mid"][0] == 1 and "k_batch" not in prof, prof
    assert cm_ctx.device_status()[0] == native.CM_EPRECOND
    for i, it in enumerate(items):
        want = made[i % len(made)][5]
        assert torch.equal(it[5], want) if want is not None else not from_dev(it[5]).any(), (lg, i, it[:3])


@pytest.mark.parametrize("n", [1_500_000, 1_500_001])
def test_tensor_core_longest_share(cm_ctx, n):
    # 39 stages of 256 terms a CTA, all ones: counts of 9984, the most that the line
    # of 40 stages leaves to one accumulator but for 256
    m = 1000
    x = torch.full((native.words(n),), -1, dtype=torch.int64, device="cuda")
    y = torch.full((native.words(n + m - 1),), -1, dtype=torch.int64, device="cuda")
    cm_ctx.profile_enable(True)
    cm_ctx.profile_read(reset=True)
    z = from_dev(run(cm_ctx, T, n, m, x, y))
    prof = cm_ctx.profile_read(reset=True)
    cm_ctx.profile_enable(False)
    assert prof["k_gf_tc"][0] == 1
    assert int(sum(bin(int(w)).count("1") for w in z)) == (m if n & 1 else 0)
