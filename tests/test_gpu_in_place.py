"""Outputs written over an operand: the dense forms read the operands while other CTAs
write, so a call whose z lies in x's or y's words runs the transforms, which have
read them by then.  Lengths whose plan is one product (no tail that reads again)."""

import numpy as np
import pytest
import torch

import oracle
from paper_2402_09481_gb300 import inputs, native
from conftest import to_dev

pytestmark = pytest.mark.gpu
T, C, D = native.TOEPLITZ, native.CIRCULANT, native.DODIS


def ybits(kind, n, m):
    return n + m - 1 if kind == T else (n + 1 if kind == C else n)


def run(ctx, kind, n, m, x, y, z):
    if kind == T:
        return ctx.toeplitz(x, n, y, m, z)
    if kind == C:
        return ctx.circulant(x, n, y, m, z)
    return ctx.dodis(x, y, n, m, z)


# dense on the CUDA cores, then dense on the tensor cores
@pytest.mark.parametrize("kind,n,m", [(T, 4096, 2048), (T, 4500, 3600), (C, 5000, 3100), (D, 4093, 2000),
                                      (T, 300007, 150001), (T, 140000, 110000), (C, 200000, 40001), (D, 150000, 90000)])
def test_output_over_an_operand(cm_ctx, kind, n, m):
    if kind == C:
        n = oracle.next_na(n + 1) - 1
    elif kind == D:
        n = oracle.next_na(n)
    q = native.plan_query(kind, n, m)
    assert q["products"] == 1 and q["tail_terms"] == 0
    xw, yw = inputs.bernoulli_half(81 + n % 97, n), inputs.bernoulli_half(82 + m % 89, ybits(kind, n, m))
    if kind == D:
        xw[0] = (xw[0] | np.uint64(1)) & ~np.uint64(2)
    want = run(cm_ctx, kind, n, m, to_dev(xw), to_dev(yw), None)
    for over in ("x", "y", "y's end"):
        x, y = to_dev(xw), to_dev(yw)
        z = {"x": x[:native.words(m)], "y": y[:native.words(m)], "y's end": y[y.numel() - native.words(m):]}[over]
        assert torch.equal(run(cm_ctx, kind, n, m, x, y, z), want), over
    # the same as a lone served request
    x, y = to_dev(xw), to_dev(yw)
    z = x[:native.words(m)]
    torch.cuda.synchronize()
    cm_ctx.server_start()
    try:
        s, r = cm_ctx.poll(cm_ctx.submit(kind, n, m, x, y, z), 60.0)
    finally:
        cm_ctx.server_stop()
    assert s == native.CM_OK and r["status"] == native.CM_OK and torch.equal(z, want)
