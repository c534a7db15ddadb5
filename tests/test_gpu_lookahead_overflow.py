"""Lookahead steps with more samples in reach than their list holds, against the oracle: the
samples that no longer fit are scored while the others are still collected, with well edges
in the FP64 band among them. Other aircraft of a co-simulation, whose records change from
step to step, and plans up to the table window's last row, whose next sample is not there.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import Oracle  # noqa: E402
from paper_2008_03518_gb300 import scenarios as S  # noqa: E402
from paper_2008_03518_gb300.fmdp import Scheduler  # noqa: E402
from test_gpu_cosim import cosim_parity  # noqa: E402
from tests.parity_util import check_q  # noqa: E402


def near(rng, n, spread=150.0):
    return np.array([5000.0, 5000.0, 200.0]) + rng.uniform(-spread, spread, size=(n, 3)) * [1.0, 1.0, 0.5]


@pytest.mark.parametrize("combine", [0, 1])
def test_cosimulated_aircraft(combine):
    """100 aircraft within 200 m of one another at W = 16: 1600 samples in reach of each."""
    rng = np.random.default_rng(17)
    o, g = near(rng, 100), near(rng, 100) + rng.uniform(-1.0, 1.0, size=(100, 3)) * [3000.0, 3000.0, 0.0]
    reqs = [dict(id=i + 1, ox=o[i, 0], oy=o[i, 1], oz=o[i, 2], gx=g[i, 0], gy=g[i, 1], gz=g[i, 2], speed=3.0 + 0.02 * i,
                 depart=5 + i % 3, horizon=14) for i in range(100)]
    args = dict(box=(0.0, 0.0, 0.0, 10000.0, 10000.0, 500.0), dt=1.0, gamma=0.99, actions=S.action_grid((-2.0, 0.0, 2.0)),
                sep=(150.0, 30.0), lookahead_W=16, combine=combine)
    with Scheduler(n_slices_window=256, max_slots=256, **args) as s:
        got, _ = cosim_parity(s, Oracle(**args), reqs)
    assert max(r["n_points"] for r in got) == 15


@pytest.mark.parametrize("full_scan", [False, True])
def test_plans_at_the_end_of_the_window(full_scan):
    rng = np.random.default_rng(23)
    v = rng.uniform(-2.0, 2.0, size=(300, 3)) * [1.0, 1.0, 0.2]
    plans = [(0, (p + np.arange(-52, 12)[:, None] * q).astype(np.float32)) for p, q in zip(near(rng, 300), v)]
    args = dict(box=(0.0, 0.0, 0.0, 10000.0, 10000.0, 500.0), dt=1.0, gamma=0.99, actions=S.action_grid((-2.0, 0.0, 2.0)),
                sep=(150.0, 30.0), lookahead_W=5)
    o = Oracle(**args)
    for t0, xyz in plans:
        o.add_plan(t0, xyz)
    with Scheduler(n_slices_window=64, max_slots=512, full_scan=full_scan, **args) as s:
        s.add_plans(plans)
        for i, p in enumerate(near(rng, 8)):
            req = dict(id=i + 1, ox=p[0], oy=p[1], oz=p[2], gx=8000.0, gy=4000.0 + 300.0 * i, gz=200.0, speed=15.0, depart=50,
                       horizon=13)
            t = s.rollout_trace(req)
            d = o.rollout(req, follow=np.asarray(t["actions"], dtype=np.int32), trace=True)
            assert d["mismatch_step"] == -1 and t["n_points"] == 14
            np.testing.assert_array_equal(d["xyz"], t["xyz"])
            check_q(t["q"], d["q"], d["scale"], where=f"request {i}")
