"""Trevisan's one-bit step in its grouped form (many outputs: the chunks' matrix on
the tensor cores) against the plain form, which a context with a small scratch
budget keeps, every output bit, and the oracle on a few: element sizes of one
to four words, l a multiple of 64, s at and around whole groups, ragged m."""

import numpy as np
import pytest

from oracle import extractors as ex
from oracle import trevisan as tv
from paper_2402_09481_gb300 import inputs, native
from conftest import from_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,l,m", [(1_000_003, 40, 20001), (64 * 15625, 64, 16384), (600_000, 63, 33000),
                                   (300_001, 121, 40007), (121 * 64 * 64, 121, 4160), (250_000, 128, 20000),
                                   (200_000, 129, 9999), (150_000, 200, 12000), (130_000, 256, 8192)])
def test_grouped_form_matches_plain(cm_ctx, n, l, m):
    xw, sw = inputs.bernoulli_half(1500 + l, n), inputs.bernoulli_half(1501 + m, 2 * l * m)
    x, s = to_dev(xw), to_dev(sw)
    cm_ctx.profile_enable(True)
    cm_ctx.profile_read(reset=True)
    z = from_dev(cm_ctx.trevisan_rsh(x, n, l, s, m))
    prof = cm_ctx.profile_read(reset=True)
    cm_ctx.profile_enable(False)
    assert "k_rsh_join" in prof and cm_ctx.device_status() == (native.CM_OK, 0)
    small = native.Context(0, hbm_budget_bytes=4 << 20)
    try:
        assert (z == from_dev(small.trevisan_rsh(x, n, l, s, m))).all()
    finally:
        small.close()
    xb, sb, f = ex.unpack_bits(xw, n), ex.unpack_bits(sw, 2 * l * m), tv.rsh_modulus(l)
    for i in (0, m - 1):
        assert int(z[i >> 6] >> np.uint64(i & 63)) & 1 == int(tv.rsh_onebit(xb, n, sb[2 * l * i:2 * l * (i + 1)], l, f))
    if m & 63:
        assert int(z[-1]) >> (m & 63) == 0
