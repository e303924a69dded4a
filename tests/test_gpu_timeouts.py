"""A bounded wait of the tensor-core form that runs out is reported to whoever made
the call: by the device status, by the host-buffer call's return and by a served
request's result, and the context works on."""

import numpy as np
import pytest
import torch

from paper_2402_09481_gb300 import inputs, native
from conftest import from_dev, to_dev

pytestmark = pytest.mark.gpu
T = native.TOEPLITZ


@pytest.fixture
def ctx():
    from paper_2402_09481_gb300 import build
    build.build()
    c = native.Context(0)
    yield c
    c.close()


def case():
    n, m = 100_000, 50_000
    x, y = to_dev(inputs.bernoulli_half(61, n)), to_dev(inputs.bernoulli_half(62, n + m - 1))
    return n, m, x, y, torch.zeros(native.words(m), dtype=torch.int64, device="cuda")


def test_single_call_and_host_call(ctx):
    n, m, x, y, z = case()
    want = from_dev(ctx.toeplitz(x, n, y, m))
    zh = torch.zeros(native.words(m), dtype=torch.int64)
    ctx.test_stall(True)
    ctx.toeplitz(x, n, y, m, z)
    assert ctx.device_status() == (native.CM_ETIMEDOUT, native.FLAG_TIMEOUT)
    with pytest.raises(native.CMError) as e:
        ctx.extract_host(T, x.cpu(), n, y.cpu(), m, zh)
    assert e.value.status == native.CM_ETIMEDOUT
    assert ctx.device_status() == (native.CM_OK, 0)  # reported once, to its own caller
    ctx.test_stall(False)
    assert ctx.extract_host(T, x.cpu(), n, y.cpu(), m, zh) == native.CM_OK
    assert (zh.numpy().view(np.uint64) == want).all()


def test_lone_served_request(ctx):
    n, m, x, y, z = case()
    want = from_dev(ctx.toeplitz(x, n, y, m))
    torch.cuda.synchronize()
    ctx.server_start()
    for stall, status in ((True, native.CM_ETIMEDOUT), (False, native.CM_OK)):
        ctx.test_stall(stall)
        s, r = ctx.poll(ctx.submit(T, n, m, x, y, z), 60.0)
        assert s == native.CM_OK and r["status"] == status
    ctx.server_stop()
    assert (from_dev(z) == want).all()
    assert ctx.device_status() == (native.CM_OK, 0)
