"""Lookahead rollouts and co-simulations that read the spatial index, against the same kernel
reading every slot of every slice (full_scan): bit for bit, for the smallest, an odd and the
largest window, tables on both sides of the line between the two ways, more samples in reach
than a step's list holds, fast plans in the extra list, and co-simulated aircraft that depart
together, one by one, or after the others have landed.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2008_03518_gb300 import scenarios as S  # noqa: E402
from paper_2008_03518_gb300.fmdp import Scheduler  # noqa: E402
from test_gpu_batch import same_results, same_tables, table_of  # noqa: E402

KEYS = ("xyz", "actions", "q", "headings", "ties")


def scene(n_plans, n_requests, spread=1500.0):
    sc = S.crowded_batch(seed=211, n_plans=n_plans, n_requests=n_requests, spread_m=spread)
    t = np.arange(200)[:, None]
    fast = np.array([5000.0, 5000.0, 210.0]) + (t - 60.0) * np.array([[60.0, 90.0, 0.0]])
    sc.plans = list(sc.plans) + [S.Plan(3, np.clip(fast, 0.0, 10000.0).astype(np.float32))]
    sc.requests["horizon"] = np.minimum(sc.requests["horizon"], 150)
    return sc


@pytest.mark.parametrize("combine", [0, 1])
@pytest.mark.parametrize("window", [2, 7, 16])
@pytest.mark.parametrize("n_plans", [255, 256, 900])
def test_index_equals_every_slot(n_plans, window, combine):
    sc = scene(n_plans, 3)
    with Scheduler.from_scenario(sc, full_scan=True, lookahead_W=window, combine=combine) as full, \
            Scheduler.from_scenario(sc, lookahead_W=window, combine=combine) as idx:
        for r in sc.requests:
            a, b = full.rollout_trace(r), idx.rollout_trace(r)
            for k in KEYS:
                np.testing.assert_array_equal(a[k], b[k], err_msg=k)


def test_more_samples_than_the_list_holds():
    """Plans that hover around one point: every one of them is in reach at every sub-step."""
    sc = scene(10, 2)
    rng = np.random.default_rng(3)
    xyz = np.array([5000.0, 5000.0, 200.0]) + rng.uniform(-150.0, 150.0, size=(400, 1, 3)) * [1.0, 1.0, 0.3]
    sc.plans = list(sc.plans) + [S.Plan(0, np.repeat(p, 300, axis=0).astype(np.float32)) for p in xyz]
    for c, v in (("ox", 4990.0), ("oy", 5010.0), ("oz", 200.0), ("depart", 20), ("horizon", 30)):
        sc.requests[c] = v
    with Scheduler.from_scenario(sc, full_scan=True, lookahead_W=5, max_slots=1024) as full, \
            Scheduler.from_scenario(sc, lookahead_W=5, max_slots=1024) as idx:
        for r in sc.requests:
            a, b = full.rollout_trace(r), idx.rollout_trace(r)
            for k in KEYS:
                np.testing.assert_array_equal(a[k], b[k], err_msg=k)


@pytest.mark.parametrize("departures", ["together", "one by one", "after the others"])
@pytest.mark.parametrize("window", [1, 3])
def test_cosim_equals_every_slot(window, departures):
    sc = scene(1100, 24, spread=800.0)
    n = len(sc.requests)
    sc.requests["depart"] = {"together": np.full(n, 10), "one by one": 10 + 3 * np.arange(n)[::-1],
                             "after the others": 10 + 400 * (np.arange(n) % 2)}[departures]
    sc.requests["horizon"][3] = 1
    with Scheduler.from_scenario(sc, full_scan=True, lookahead_W=window) as full, \
            Scheduler.from_scenario(sc, lookahead_W=window) as idx:
        same_results(full.schedule_cosim(sc.requests), idx.schedule_cosim(sc.requests))
        same_tables(table_of(full), table_of(idx))
