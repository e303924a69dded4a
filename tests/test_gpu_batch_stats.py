"""cm_batch_stats.kernel_launches against the launches that a run traces, for every
form an instance can take."""

import pytest
import torch

import oracle
from paper_2402_09481_gb300 import inputs, native
from conftest import to_dev

pytestmark = pytest.mark.gpu
T, D = native.TOEPLITZ, native.DODIS


def specs(case):
    return {"tensor cores": [(T, 30_000, 2_100_000), (T, 100, 50), (T, 9000, 7000)],
            "integer": [(T, 2 ** 21, 2 ** 20)],
            "integer, checked": [(D, oracle.next_na(2_000_000), 1_500_000)],
            "sums": [(T, 2 ** 25, 2 ** 24), (D, oracle.next_na(3 << 24), 2 ** 24)],
            "groups": [(T, 2 ** 21, 2 ** 20), (T, 2 ** 21, 2 ** 20 + 1), (D, oracle.next_na(3 << 21), 2 ** 20)]}[case]


@pytest.mark.parametrize("case", ["tensor cores", "integer", "integer, checked", "sums", "groups"])
def test_launches_as_traced(cm_ctx, case):
    items = []
    for j, (kind, n, m) in enumerate(specs(case)):
        yb = n + m - 1 if kind == T else n
        items.append((kind, n, m, to_dev(inputs.bernoulli_half(600 + 2 * j, n)),
                      to_dev(inputs.bernoulli_half(601 + 2 * j, yb)),
                      torch.zeros(native.words(m), dtype=torch.int64, device="cuda")))
    b = cm_ctx.batch(items, graph=False)
    cm_ctx.profile_enable(True)
    cm_ctx.profile_read(reset=True)
    b.launch()
    prof = cm_ctx.profile_read(reset=True)
    cm_ctx.profile_enable(False)
    assert ("k_gf_tc" in prof) == (case == "tensor cores"), prof
    assert b.info()["kernel_launches"] == sum(c for c, _ in prof.values()), prof
    b.close()
