"""Proposals do not depend on how many requests share a cluster: one request, a tile and its
neighbours, two to four tiles per cluster, and more requests than there are rows, against the
same requests planned in small groups.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2008_03518_gb300 import scenarios as S  # noqa: E402
from paper_2008_03518_gb300.fmdp import Scheduler  # noqa: E402


@pytest.fixture(scope="module")
def proposals():
    sc = S.c1_plain_small()
    sc.requests = np.tile(sc.requests, 3000 // len(sc.requests) + 1)[:3000].copy()
    rng = np.random.default_rng(1)
    sc.requests["horizon"] = rng.integers(1, 60, size=3000)  # rows are refilled at different steps
    sc.requests["horizon"][7] = 0
    with Scheduler.from_scenario(sc) as s:
        s.learned_init(seed=9)

        def steps(n):
            return np.asarray(s.learned_evaluate(sc.requests[:n])[2])

        want = np.concatenate([np.asarray(s.learned_evaluate(sc.requests[i:i + 40])[2]) for i in range(0, 3000, 40)])
        yield steps, want


@pytest.mark.parametrize("n", [1, 15, 16, 17, 609, 1217, 1825, 2433, 3000])
def test_groups_of_any_size(proposals, n):
    steps, want = proposals
    np.testing.assert_array_equal(steps(n), want[:n])
