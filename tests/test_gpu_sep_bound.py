"""Reports of many trajectories whose samples lower one another's least distance while they are
read, with squares of more than 32 cell rows (fine cells, sparse rows): batches in waves and
pipelined, and checks of one trajectory, against the scan of every slot.
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


@pytest.mark.parametrize("sep", [(150.0, 30.0), (2600.0, 4.0)])
@pytest.mark.parametrize("n_plans", [400, 1500])
def test_wide_squares_and_shared_bounds(n_plans, sep):
    sc = S.crowded_batch(seed=307, n_plans=n_plans, n_requests=64)
    sc.sep = sep
    with Scheduler.from_scenario(sc, full_scan=True) as full:
        want = full.schedule_batch(sc.requests)
        table = table_of(full)
        paths = [w["xyz"] for w in want if w["n_points"] > 40][:12]
        starts = [int(r["depart"]) for r, w in zip(sc.requests, want) if w["n_points"] > 40][:12]
        checks = [full.sep_check(t, p) for t, p in zip(starts, paths)]
    assert any(c["conflicts"] for c in checks)
    for mode in (0, 1):
        with Scheduler.from_scenario(sc, index_cell_m=100.0, batch_mode=mode) as s:
            same_results(s.schedule_batch(sc.requests), want)
            same_tables(table_of(s), table)
            assert [s.sep_check(t, p) for t, p in zip(starts, paths)] == checks
