"""Indexed rollouts at every division of a CTA's warps into roles, against the full scan.

The number of warps decides which roles have a warp of their own (recorder, terrain, second
well-folding warp) and how many warps prepare lists; options.index_stage_items decides when a
step's samples no longer fit its list. Trajectories, actions, action values and near-tie flags
of the full scan must come out bit for bit, also along the clearance limit (where fp32 leaves
the decision to double-float or FP64), with static wells, with fast plans in the extra list,
and when the plan ends at once (goal at the origin, a horizon of one step).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2008_03518_gb300 import scenarios as S  # noqa: E402
from paper_2008_03518_gb300.fmdp import Scheduler  # noqa: E402


def scene(terrain):
    rng = np.random.default_rng(31)
    if terrain:
        hm = S.fractal_heightmap(5, n=129, top=300.0)
        box = (0.0, 0.0, 0.0, 12000.0, 12000.0, 1000.0)
        plans = S.multileg_plans(rng, box, 300, hm, legs=(2, 4), leg_len=(1500.0, 5000.0), tlo=0, thi=300)
        reqs = S.make_requests(rng, box, 5, hm=hm, zspan=(0.0, 90.0), tlo=0, thi=300, horizon=600)
        sw = np.array([[6000.0, 6000.0, 300.0, 800.0, 1000.0, 0.99], [3000.0, 9000.0, 200.0, 400.0, 500.0, 0.98]])
        sc = S.Scenario("roles_terrain", box, 1.0, 0.99, S.action_grid((-2.0, 0.0, 2.0)), (150.0, 30.0), plans, reqs,
                        heightmap=hm, clearance=60.0, static_wells=sw, n_slices_window=2048, max_slots=400)
    else:
        sc = S.crowded_batch(seed=109, n_plans=500, n_requests=5)
        t = np.arange(300)[:, None]
        fast = np.clip(np.array([5000.0, 5000.0, 210.0]) + (t - 150.0) * np.array([[60.0, 90.0, 0.0]]), 0.0, 10000.0)
        sc.plans = list(sc.plans) + [S.Plan(5, fast.astype(np.float32))]  # over the index's speed bound: extra list
        reqs = sc.requests
    reqs["horizon"][3] = 1
    for g, o in (("gx", "ox"), ("gy", "oy"), ("gz", "oz")):
        reqs[g][4] = reqs[o][4]
    return sc


@pytest.mark.parametrize("terrain", [False, True])
@pytest.mark.parametrize("combine", [0, 1])
def test_every_warp_count_equals_the_full_scan(terrain, combine):
    sc = scene(terrain)
    with Scheduler.from_scenario(sc, full_scan=True, combine=combine) as full:
        want = [full.rollout_trace(r) for r in sc.requests]
    assert max(w["n_points"] for w in want) > 50
    for threads in range(128, 385, 32):
        for items in (16, 512):
            with Scheduler.from_scenario(sc, combine=combine, threads_per_cta=threads, index_stage_items=items) as s:
                for r, w in zip(sc.requests, want):
                    g = s.rollout_trace(r)
                    assert (g["verdict"], g["n_points"]) == (w["verdict"], w["n_points"]), (threads, items)
                    for k in ("xyz", "actions", "q", "headings", "ties"):
                        np.testing.assert_array_equal(g[k], w[k], err_msg=f"{k} {threads} {items}")
