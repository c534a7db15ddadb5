"""Checks on both sides of the line between reading every slot and reading cells (1024 samples,
3 x 2^18 sample-slot pairs): the allocation-free check and the check of a scheduled request,
which take the rule, against the one-launch check, which always reads cells.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2008_03518_gb300 import scenarios as S  # noqa: E402
from paper_2008_03518_gb300.fmdp import Scheduler  # noqa: E402


@pytest.mark.parametrize("plans,samples", [(0, 1), (1, 1), (32, 1024), (32, 1025), (768, 1024), (800, 1024), (3071, 256),
                                           (3073, 256), (3000, 1)])
def test_reports_are_equal(plans, samples):
    sc = S.crowded_batch(seed=401, n_plans=plans, n_requests=4)
    rng = np.random.default_rng(plans + samples)
    with Scheduler.from_scenario(sc, max_slots=4096) as s:
        for k in range(4):
            a, b = rng.uniform(2000.0, 8000.0, (2, 2))
            xy = a + (b - a) * np.linspace(0.0, 1.0, samples)[:, None]
            path = np.concatenate([xy, np.full((samples, 1), 150.0 + 60.0 * k)], axis=1)
            assert s.sep_check_noalloc(10 * k, path) == s.sep_check(10 * k, path)
        s.snapshot()
        for r in sc.requests:  # (checked before it is stored)
            s.restore()
            got = s.schedule(r)
            s.restore()
            want = s.sep_check(int(r["depart"]), got["xyz"])
            for k in ("first_conflict_step", "first_terrain_step", "min_sep_h", "min_sep_v"):
                assert got[k] == want[k], k
