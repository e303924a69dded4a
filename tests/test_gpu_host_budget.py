"""The host-buffer call's smallest budget: its copies of x, y, z and its scratch in
256-byte steps, nothing more, whichever form runs."""

import numpy as np
import pytest
import torch

import oracle
from paper_2402_09481_gb300 import inputs, native

pytestmark = pytest.mark.gpu
T, D = native.TOEPLITZ, native.DODIS


@pytest.mark.parametrize("kind,n,m", [(T, 600_000, 300_000), (T, 4096, 2048), (D, 4093, 2000)])
def test_exact_budget(kind, n, m):
    from paper_2402_09481_gb300 import build
    build.build()
    yb = n + m - 1 if kind == T else n
    io = 8 * (native.words(n) + native.words(yb) + native.words(m)) + 3 * 256
    need = (native.plan_query(kind, n, m)["scratch_bytes"] + 255) & ~255
    xw, yw = inputs.bernoulli_half(91, n), inputs.bernoulli_half(92, yb)
    xw[0] = (xw[0] | np.uint64(1)) & ~np.uint64(2)
    x, y = torch.from_numpy(xw.view(np.int64)), torch.from_numpy(yw.view(np.int64))
    z = torch.zeros(native.words(m), dtype=torch.int64)
    for budget, fits in ((io + need, True), (io + need - 1, False)):
        ctx = native.Context(0, hbm_budget_bytes=budget)
        try:
            if not fits:
                with pytest.raises(native.CMError) as e:
                    ctx.extract_host(kind, x, n, y, m, z)
                assert e.value.status == native.CM_ENOMEM
                continue
            assert ctx.extract_host(kind, x, n, y, m, z) == native.CM_OK
            rows = np.arange(0, m, max(1, m // 40))
            zw = z.numpy().view(np.uint64)
            got = ((zw[rows >> 6] >> (rows & 63).astype(np.uint64)) & np.uint64(1)).astype(np.uint8)
            want = oracle.toeplitz_rows(xw, n, yw, m, rows) if kind == T else oracle.dodis_rows(xw, yw, n, m, rows)
            assert (got == want).all()
        finally:
            ctx.close()
