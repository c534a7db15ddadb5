"""A flight a tenth of a millimetre beside a node line of the heightmap, level at the clearance
limit: its fp32 position lies on the line, in the cell FP64 does not take. Along a ridge the
neighbouring cell's surface, continued to the flight, is higher than the limit allows, so a
penalty taken from it turns the flight away; FP64 sees it clear. The rollouts have to follow
the oracle (and, without lookahead, the full scan bit for bit).
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
from tests.parity_util import check_q  # noqa: E402

BOX = (0.0, 0.0, 0.0, 12000.0, 12000.0, 1000.0)
CELL = 12000.0 / 64


@pytest.mark.parametrize("window", [1, 3])
@pytest.mark.parametrize("along", ["x", "y"])
@pytest.mark.parametrize("side", [-1.0, 1.0])
def test_flight_beside_a_node_line(window, along, side):
    hm = np.zeros((65, 65), dtype=np.float32)
    hm[20, :] = 100.0  # a ridge along x ...
    line = 20 * CELL + side * 1e-4
    req = dict(id=1, ox=1000.0, oy=line, oz=160.0, gx=9000.0, gy=line, gz=160.0, speed=30.0, depart=0, horizon=100)
    if along == "y":  # ... or along y
        hm = np.ascontiguousarray(hm.T)
        req.update(ox=line, oy=1000.0, gx=line, gy=9000.0)
    args = dict(box=BOX, dt=1.0, gamma=0.99, actions=S.action_grid((0.0,)), sep=(150.0, 30.0), heightmap=hm, clearance=60.0,
                lookahead_W=window)
    o = Oracle(**args)
    with Scheduler(n_slices_window=1024, max_slots=64, **args) as s:
        t = s.rollout_trace(req)
    d = o.rollout(req, follow=np.asarray(t["actions"], dtype=np.int32), trace=True)
    assert d["mismatch_step"] == -1
    np.testing.assert_array_equal(d["xyz"], t["xyz"])
    check_q(t["q"], d["q"], d["scale"])
    np.testing.assert_array_equal(t["xyz"][:, 1 if along == "x" else 0], np.float32(line))  # (straight along the ridge)
    if window == 1:
        with Scheduler(n_slices_window=1024, max_slots=64, full_scan=True, **args) as full:
            f = full.rollout_trace(req)
        for k in ("xyz", "actions", "q", "headings", "ties"):
            np.testing.assert_array_equal(t[k], f[k], err_msg=k)
