"""The shared-seed product on tcgen05 (e2m1 counts, parity epilogue) against the
CUDA-core engine and the oracle: edges of its 256-input, 224-output and
256-column tiles, and the largest counts (all ones at n = 2^14)."""

import numpy as np
import pytest
import torch

import oracle
from paper_2402_09481_gb300 import inputs, native
from conftest import from_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,count", [(1, 1, 1), (255, 223, 255), (256, 224, 256), (257, 225, 257), (300, 448, 3), (300, 480, 3), (1000, 333, 300),
                                       (64, 65, 1500), (4096, 2048, 700), (5000, 4000, 9), (16384, 300, 40000)])
def test_f4_engine_matches(cm_ctx, n, m, count):
    wx, wz = native.words(n), native.words(m)
    yw = inputs.bernoulli_half(61 + n, n + m - 1)
    g = torch.Generator(device="cuda")
    g.manual_seed(n + count)
    X = torch.randint(-2 ** 63, 2 ** 63 - 1, (wx * count,), dtype=torch.int64, device="cuda", generator=g)  # dirty tails
    y = to_dev(yw)
    Z = torch.full((wz * count,), -1, dtype=torch.int64, device="cuda")
    cm_ctx.toeplitz_shared_seed(y, n, m, X, count, Z, engine=native.ENGINE_F4)
    assert cm_ctx.device_status() == (native.CM_OK, 0)
    assert torch.equal(Z, cm_ctx.toeplitz_shared_seed(y, n, m, X, count, engine=native.ENGINE_GF2))
    for c in {0, count // 2, count - 1}:
        want = oracle.toeplitz_packed(from_dev(X[c * wx:(c + 1) * wx]), n, yw, m)
        assert (from_dev(Z[c * wz:(c + 1) * wz]) == want).all()


def test_f4_engine_largest_counts(cm_ctx):
    # all ones: every count is n; one input bit cleared: n - 1
    for n in (16384, 16383, 8191):
        m, wx = 256, native.words(n)
        y = torch.full((native.words(n + m - 1),), -1, dtype=torch.int64, device="cuda")
        X = torch.full((2, wx), -1, dtype=torch.int64, device="cuda")
        X[1, 0] = -2
        Z = cm_ctx.toeplitz_shared_seed(y, n, m, X.reshape(-1), 2, engine=native.ENGINE_F4).reshape(2, -1)
        assert (Z[0] == (-1 if n & 1 else 0)).all() and (Z[1] == (0 if n & 1 else -1)).all()


def test_f4_engine_limits(cm_ctx):
    d = to_dev(np.zeros(8, dtype=np.uint64))
    L, p, s = native.lib(), d.data_ptr(), torch.cuda.current_stream().cuda_stream
    assert L.cm_batch_toeplitz_shared_seed(cm_ctx.handle, p, 16385, 5, p, 1, p, native.ENGINE_F4, s) == native.CM_EINVAL
