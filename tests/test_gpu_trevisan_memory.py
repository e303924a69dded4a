"""Trevisan's one-bit step where the grouped form's scratch fits the context's budget
but not the memory that is free when the call is made: the plain form runs.  In a
process of its own: CUDA would serve the call from what other contexts'
pools hold unused in this one."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def check():
    import torch

    from paper_2402_09481_gb300 import inputs, native
    from conftest import from_dev, to_dev
    n, l, m, t = 1 << 18, 121, 1 << 20, 242  # grouped scratch 1.5 GB, plain 35 KB
    x, s = to_dev(inputs.bernoulli_half(71, n)), to_dev(inputs.bernoulli_half(72, 2 * l * m))
    sets = torch.arange(m * t, dtype=torch.int32, device="cuda")  # the seeds in order
    ctx = native.Context(0)
    want = from_dev(ctx.trevisan_rsh(x, n, l, s, m))
    torch.cuda.synchronize()
    ctx.close()
    ctx = native.Context(0)  # its budget is 80% of what is free now
    torch.cuda.empty_cache()
    taken = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device="cuda")
    ctx.profile_enable(True)
    ctx.profile_read(reset=True)
    z = from_dev(ctx.trevisan_rsh(x, n, l, s, m))
    prof = ctx.profile_read(reset=True)
    assert "k_rsh" in prof and "k_rsh_join" not in prof, prof
    assert (z == want).all()
    assert (from_dev(ctx.trevisan(x, n, s, 2 * l * m, sets, t, m, l)) == want).all()
    del taken
    ctx.close()


def test_plain_form_where_memory_is_taken():
    from paper_2402_09481_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env={**os.environ, "PYTHONPATH": ROOT})
    assert r.returncode == 0 and "checked" in r.stdout, r.stderr[-2000:]


if __name__ == "__main__":
    check()
    print("checked")
