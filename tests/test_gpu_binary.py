"""The binary-polynomial form of the products (additive transforms over packed
bits, products longer than 2^23 in a context with default options) against the
integer transforms of another context, every bit, and the oracle on sampled
rows: each transform length at its edges, ragged lengths, every kind, one
window of several blocks, several windows of one block, and both."""

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


def resolve(kind, n, m):
    if kind == C:
        n = oracle.next_na(n + 1) - 1
    elif kind == D:
        n = oracle.next_na(n)
    return n, m if kind == T else min(m, n)


CASES = [(T, 2 ** lg - m + 1 + d, m) for lg in (24, 25) for m, d in ((2 ** (lg - 2) + 17, 0), (77, 0), (2 ** (lg - 1) + 1, 1))
         if not (lg == 25 and d)]
CASES += [
    (T, 2 ** 23, 2), (T, 1, 2 ** 24), (T, 2 ** 24 + 1, 2 ** 24),
    (C, 12_000_000, 4_000_000), (C, 16777258, 8388629), (D, 9_000_000, 1), (D, 9_000_000, 8_999_999),
    # one window, several input blocks; one block, several windows; both
    (T, 40_000_000, 3), (T, 70_000_001, 5_000_011), (T, 5, 40_000_000), (T, 3_000_001, 70_000_003),
    (T, 40_000_003, 40_000_001), (C, 50_000_000, 20_000_003), (D, 60_000_000, 50_000_000),
]


@pytest.mark.parametrize("kind,n,m", CASES)
def test_binary_form_matches(cm_ctx, q30, kind, n, m):
    n, m = resolve(kind, n, m)
    xw = inputs.bernoulli_half(31 + n % 83, n)
    if kind == D:
        xw[0] = (xw[0] | np.uint64(1)) & ~np.uint64(2)
    yw = inputs.bernoulli_half(32 + m % 79, ybits(kind, n, m))
    x, y = to_dev(xw), to_dev(yw)
    cm_ctx.profile_enable(True)
    cm_ctx.profile_read(reset=True)
    z = run(cm_ctx, kind, n, m, x, y)
    prof = cm_ctx.profile_read(reset=True)
    cm_ctx.profile_enable(False)
    assert any(k.startswith("k_gf") for k in prof), prof
    assert torch.equal(z, run(q30, kind, n, m, x, y))
    zw = from_dev(z)
    rows = np.unique(np.concatenate([np.arange(min(m, 8)), np.arange(max(0, m - 8), m),
                                     np.random.default_rng(m).integers(0, m, 8)]))
    got = ((zw[rows >> 6] >> (rows & 63).astype(np.uint64)) & np.uint64(1)).astype(np.uint8)
    fn = {T: lambda: oracle.toeplitz_rows(xw, n, yw, m, rows), C: lambda: oracle.circulant_rows(xw, n, yw, m, rows),
          D: lambda: oracle.dodis_rows(xw, yw, n, m, rows)}[kind]
    assert (got == fn()).all()


@pytest.mark.parametrize("P,m", [(9_000_000, 70001), (40_000_000, 20_000_000)])
def test_binary_form_precondition(cm_ctx, P, m):
    # a constant Dodis et al. input: zero output, reported, flag cleared after
    P = oracle.next_na(P)
    y = to_dev(inputs.bernoulli_half(6, P))
    for fill in (0, 1):
        z = run(cm_ctx, D, P, m, to_dev(ex.pack_bits(np.full(P, fill, dtype=np.uint8))), y)
        assert cm_ctx.device_status()[0] == native.CM_EPRECOND
        assert not from_dev(z).any()
    assert cm_ctx.device_status() == (native.CM_OK, 0)


def test_binary_form_budget_falls_back(q30):
    # a scratch budget below the binary form's: the integer planner's blocks, same bits
    n, m = 9_000_000, 1_000_000
    ctx = native.Context(0, hbm_budget_bytes=4_000_000)
    try:
        x, y = to_dev(inputs.bernoulli_half(8, n)), to_dev(inputs.bernoulli_half(9, n + m - 1))
        assert torch.equal(run(ctx, T, n, m, x, y), run(q30, T, n, m, x, y))
    finally:
        ctx.close()


def test_batch_every_length_matches(cm_ctx, q30):
    # the batch's groups, 2^15 .. 2^25 and past them, every kind, K + m - 1 at
    # the edges of each length, and constant Dodis et al. inputs zeroed alone
    specs = []
    for lg in range(15, 26):
        L = 2 ** lg
        specs += [(T, L - L // 3, L // 3 + 1), (T, L // 2, 2), (T, 5, L - 4),
                  (C, oracle.next_na(L // 2 + 7) - 1, L // 4 + 3), (D, oracle.next_na(L * 5 // 9), L // 3)]
    specs += [(T, 2 ** 25, 2 ** 24), (T, 100, 50), (T, 9000, 7000)]
    items, bad = [], []
    for j, (kind, n, m) in enumerate(specs):
        xw, yw = inputs.bernoulli_half(500 + 2 * j, n), inputs.bernoulli_half(501 + 2 * j, ybits(kind, n, m))
        if kind == D:
            xw[0] = (xw[0] | np.uint64(1)) & ~np.uint64(2)
            if j % 3 == 1:
                xw = ex.pack_bits(np.full(n, j & 1, dtype=np.uint8))
                bad.append(j)
        items.append((kind, n, m, to_dev(xw), to_dev(yw),
                      torch.full((native.words(m),), -1, dtype=torch.int64, device="cuda")))
    want = [run(q30, k, n, m, x, y) for k, n, m, x, y, _ in items]
    assert q30.device_status()[0] == native.CM_EPRECOND and bad
    for graph in (True, False):
        b = cm_ctx.batch(items, graph=graph)
        b.launch()
        assert cm_ctx.device_status()[0] == native.CM_EPRECOND
        for j, it in enumerate(items):
            assert torch.equal(it[5], want[j]), (graph, specs[j])
            it[5].fill_(-1)
        b.launch()  # a replay writes the same bits
        torch.cuda.synchronize()
        for j, it in enumerate(items):
            assert torch.equal(it[5], want[j]), (graph, specs[j])
            it[5].fill_(-1)
        b.close()
    cm_ctx.device_status()


DENSE = [(T, 1, 1), (T, 33, 31), (T, 1, 8192), (T, 8192, 1), (T, 4096, 2048), (T, 4095, 4098), (T, 1025, 63),
         (C, 1000, 500), (C, 5000, 3100), (D, 30, 29), (D, 4093, 4093), (D, 8000, 65)]


@pytest.mark.parametrize("kind,n,m", DENSE)
def test_dense_form_matches(cm_ctx, q30, kind, n, m):
    # products of up to 2^13 terms: one launch, every output against the oracle
    n, m = resolve(kind, n, m)
    xw, yw = inputs.bernoulli_half(41 + n, n), inputs.bernoulli_half(42 + m, ybits(kind, n, m))
    if kind == D:
        xw[0] = (xw[0] | np.uint64(1)) & ~np.uint64(2)
    x, y = to_dev(xw), to_dev(yw)
    cm_ctx.profile_enable(True)
    cm_ctx.profile_read(reset=True)
    z = run(cm_ctx, kind, n, m, x, y)
    prof = cm_ctx.profile_read(reset=True)
    cm_ctx.profile_enable(False)
    assert prof["k_gf_dense"][0] == 1 and len(prof) == 1
    want = {T: lambda: oracle.toeplitz_packed(xw, n, yw, m), C: lambda: oracle.circulant_packed(xw, n, yw, m),
            D: lambda: oracle.dodis_packed(xw, yw, n, m)}[kind]()
    assert (from_dev(z) == want).all()
    zh = torch.zeros(native.words(m), dtype=torch.int64)
    assert cm_ctx.extract_host(kind, x.cpu(), n, y.cpu(), m, zh) == native.CM_OK
    assert (zh.numpy().view(np.uint64) == want).all()
    if kind == D:
        for fill in (0, 1):
            c = ex.pack_bits(np.full(n, fill, dtype=np.uint8))
            assert not from_dev(run(cm_ctx, D, n, m, to_dev(c), y)).any()
            assert cm_ctx.device_status()[0] == native.CM_EPRECOND
            assert cm_ctx.extract_host(D, torch.from_numpy(c.view(np.int64)), n, y.cpu(), m, zh) == native.CM_EPRECOND
            cm_ctx.device_status()


TENSOR = [(T, 2 ** 17, 2), (T, 3, 2 ** 17 - 1), (T, 300007, 150001), (T, 131000, 224 * 256), (T, 131000, 224 * 256 + 1),
          (T, 256 * 600 - 223, 223), (T, 256 * 600 - 222, 225), (C, 200000, 100001), (C, 140000, 77), (D, 150000, 149000),
          (D, 262000, 65)]


@pytest.mark.parametrize("kind,n,m", TENSOR)
def test_tensor_core_form_matches(cm_ctx, q30, kind, n, m):
    # dense products on the tensor cores: edges of its 256-window, 224-output and
    # 256-term tiles, against the integer transforms and the oracle
    n, m = resolve(kind, n, m)
    xw, yw = inputs.bernoulli_half(51 + n % 97, n), inputs.bernoulli_half(52 + m % 89, ybits(kind, n, m))
    if kind == D:
        xw[0] = (xw[0] | np.uint64(1)) & ~np.uint64(2)
    x, y = to_dev(xw), to_dev(yw)
    cm_ctx.profile_enable(True)
    cm_ctx.profile_read(reset=True)
    z = run(cm_ctx, kind, n, m, x, y)
    prof = cm_ctx.profile_read(reset=True)
    cm_ctx.profile_enable(False)
    assert prof["k_gf_tc"][0] == 1
    assert torch.equal(z, run(q30, kind, n, m, x, y))
    assert cm_ctx.device_status() == (native.CM_OK, 0)
    zw = from_dev(z)
    rows = np.unique(np.random.default_rng(m).integers(0, m, 8))
    got = ((zw[rows >> 6] >> (rows & 63).astype(np.uint64)) & np.uint64(1)).astype(np.uint8)
    fn = {T: lambda: oracle.toeplitz_rows(xw, n, yw, m, rows), C: lambda: oracle.circulant_rows(xw, n, yw, m, rows),
          D: lambda: oracle.dodis_rows(xw, yw, n, m, rows)}[kind]
    assert (got == fn()).all()
    if kind == D:
        for fill in (0, 1):
            c = to_dev(ex.pack_bits(np.full(n, fill, dtype=np.uint8)))
            assert not from_dev(run(cm_ctx, D, n, m, c, y)).any()
            assert cm_ctx.device_status()[0] == native.CM_EPRECOND


def test_tensor_core_form_largest_counts(cm_ctx):
    # all ones: every count is n, in shares of up to 2^14 terms
    for n, m in ((300_000, 1000), (300_001, 1000)):
        x = torch.full((native.words(n),), -1, dtype=torch.int64, device="cuda")
        y = torch.full((native.words(n + m - 1),), -1, dtype=torch.int64, device="cuda")
        z = from_dev(run(cm_ctx, T, n, m, x, y))
        assert int(sum(bin(int(w)).count("1") for w in z)) == (m if n & 1 else 0)


@pytest.mark.parametrize("kind,n,m", [(T, 2 ** 23 - 4_000_000, 4_000_001), (T, 4_900_007, 3_100_003),
                                      (C, 6_000_000, 2_000_003), (D, 4_194_389, 2_000_003), (T, 5_000_000, 64)])
def test_one_transform_of_2_23(cm_ctx, q30, kind, n, m):
    # above 2^22: either form, the same bits; the first is a single transform of 2^23
    n, m = resolve(kind, n, m)
    xw = inputs.bernoulli_half(41 + n % 83, n)
    if kind == D:
        xw[0] = (xw[0] | np.uint64(1)) & ~np.uint64(2)
    x, y = to_dev(xw), to_dev(inputs.bernoulli_half(42 + m % 79, ybits(kind, n, m)))
    cm_ctx.profile_enable(True)
    cm_ctx.profile_read(reset=True)
    z = run(cm_ctx, kind, n, m, x, y)
    prof = cm_ctx.profile_read(reset=True)
    cm_ctx.profile_enable(False)
    if m == 4_000_001:
        assert any(k.startswith("k_gf_mid") for k in prof), prof
    assert torch.equal(z, run(q30, kind, n, m, x, y))


@pytest.mark.parametrize("lg,count", [(22, 1), (22, 4), (22, 5), (23, 2), (23, 3), (24, 1), (24, 2)])
def test_batch_few_operands(cm_ctx, q30, lg, count):
    # both tile shapes of the last pass, on each side of the line between them
    items, want = [], []
    for j in range(count):
        m = 2 ** (lg - 2) + 3 * j + 1
        n = 2 ** lg - m + 1 - j
        x, y = to_dev(inputs.bernoulli_half(700 + j, n)), to_dev(inputs.bernoulli_half(800 + j, n + m - 1))
        items.append((T, n, m, x, y, torch.full((native.words(m),), -1, dtype=torch.int64, device="cuda")))
        want.append(run(q30, T, n, m, x, y))
    cm_ctx.batch_extract(items)
    for it, z in zip(items, want):
        assert torch.equal(it[5], z)


@pytest.mark.parametrize("lg,count", [(15, 63), (15, 64), (16, 32), (17, 31), (17, 32), (18, 16), (19, 15), (19, 16)])
def test_batch_group_line(cm_ctx, q30, lg, count):
    # the fewest instances of a length that run as a group, and one less
    items, want = [], []
    for j in range(count):
        m = 2 ** (lg - 1) + 3 * j - 40
        n = 2 ** lg - m + 1 - j
        x, y = to_dev(inputs.bernoulli_half(900 + j, n)), to_dev(inputs.bernoulli_half(980 + j, n + m - 1))
        items.append((T, n, m, x, y, torch.full((native.words(m),), -1, dtype=torch.int64, device="cuda")))
        want.append(run(q30, T, n, m, x, y))
    cm_ctx.profile_enable(True)
    cm_ctx.profile_read(reset=True)
    cm_ctx.batch_extract(items)
    prof = cm_ctx.profile_read(reset=True)
    cm_ctx.profile_enable(False)
    line = 21 if lg <= 16 else 22 if lg <= 18 else 23
    assert ("k_batch" in prof) == (count << lg < 1 << line), prof
    for it, z in zip(items, want):
        assert torch.equal(it[5], z)
