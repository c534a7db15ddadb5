"""The separation check that reads only the cells around each sample, against the full scan.

With the spatial index a check reads, of each row, a square around the sample and widens it
until no unread plan can conflict or lower the least separation; without the index
(full_scan) it reads every slot. The reports must be equal in every field, whatever the
density, wherever the plans and samples lie (outside the box, in edge cells, on cell edges),
for plans kept in the extra list (fast ones, appended ones), and for minima from below a
metre to wider than the airspace.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2008_03518_gb300 import scenarios as S  # noqa: E402
from paper_2008_03518_gb300.fmdp import Scheduler  # noqa: E402

BOX = (0.0, 0.0, 0.0, 20000.0, 20000.0, 1000.0)


def table(rng, n, spread, z, speed):
    """n plans of 20 to 60 samples from step 0 on, from a square `spread` box widths wide."""
    plans = []
    for _ in range(n):
        m = int(rng.integers(20, 61))
        p = 10000.0 + (rng.uniform(-1.0, 1.0, 2) * 10000.0 * spread)
        a = rng.uniform(0.0, 2.0 * np.pi)
        t = np.arange(m)[:, None] * speed
        xy = p + t * np.array([np.cos(a), np.sin(a)])
        plans.append((0, np.concatenate([xy, np.full((m, 1), rng.uniform(*z))], axis=1).astype(np.float32)))
    return plans


CASES = {
    "flat rows": dict(n=60, spread=1.0, z=(100.0, 400.0)),
    "dense": dict(n=3000, spread=1.0, z=(100.0, 400.0)),
    "one corner": dict(n=2000, spread=0.05, z=(100.0, 400.0)),
    "outside the box": dict(n=800, spread=2.5, z=(100.0, 400.0)),
    "no plan at the height": dict(n=1500, spread=1.0, z=(800.0, 900.0)),
    "fast plans": dict(n=900, spread=0.8, z=(100.0, 400.0), speed=90.0),
    "sub-metre minima": dict(n=1500, spread=1.0, z=(200.0, 201.0), sep=(0.5, 0.25)),
    "minima wider than the box": dict(n=700, spread=1.0, z=(100.0, 900.0), sep=(60000.0, 5000.0)),
    "wide horizontal minimum": dict(n=2500, spread=1.0, z=(100.0, 400.0), sep=(2500.0, 30.0)),
}


@pytest.mark.parametrize("name", CASES)
def test_reports_equal_the_full_scan(name):
    c = dict(dict(speed=30.0, sep=(150.0, 30.0)), **CASES[name])
    rng = np.random.default_rng(sorted(CASES).index(name))
    plans = table(rng, c["n"], c["spread"], c["z"], c["speed"])
    late = table(rng, 6, 0.5, c["z"], 30.0)  # appended to the rows' extra lists
    hm = S.fractal_heightmap(3, n=64)
    args = dict(box=BOX, dt=1.0, gamma=0.99, actions=S.action_grid((-2.0, 0.0, 2.0)), sep=c["sep"], n_slices_window=64,
                max_slots=c["n"] + 64, heightmap=hm, clearance=60.0)
    with Scheduler(full_scan=True, **args) as full, Scheduler(**args) as idx:
        for s in (full, idx):
            s.add_plans(plans)
            for p in late:
                s.add_plan(*p)
        reports = []
        for t0, n in ((0, 60), (-3, 7), (20, 1), (59, 40)):
            paths = [np.concatenate([rng.uniform(-4000.0, 24000.0, (n, 2)), rng.uniform(50.0, 450.0, (n, 1))], axis=1),
                     plans[0][1][:1] + np.cumsum(rng.normal(0.0, 40.0, (n, 3)), axis=0) * [1.0, 1.0, 0.1],
                     np.tile([[0.0, 20000.0, 210.0]], (n, 1)) + np.arange(n)[:, None] * [570.0, -570.0, 0.0]]
            for path in paths:
                a, b = full.sep_check(t0, path), idx.sep_check(t0, path)
                assert a == b, (name, t0, n, a, b)
                assert idx.sep_check_noalloc(t0, path) == b
                reports.append(b)
    if name in ("dense", "one corner", "wide horizontal minimum", "minima wider than the box"):
        assert any(r["conflicts"] > 0 for r in reports)
    # (a path 600 m below every plan has no pair inside the vertical minimum: the whole row is read)
    assert any(np.isinf(r["min_sep_h"]) for r in reports) or name != "no plan at the height"
