"""The conflict check at the end of a pipelined plan, against sequential scheduling: separation
minima from a metre to several index cells (more cell rows than it loads at once), rows whose
appended lists are shorter and longer than the items it loads at once, and no plans at all.
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


@pytest.mark.parametrize("n_plans", [0, 5, 300])
@pytest.mark.parametrize("sep", [(1.0, 1.0), (150.0, 30.0), (4000.0, 3.0)])
def test_verdicts_equal_sequential(sep, n_plans):
    sc = S.crowded_batch(seed=311, n_plans=max(n_plans, 1), n_requests=40)
    sc.plans = sc.plans[:n_plans]
    sc.sep = sep
    with Scheduler.from_scenario(sc) as one, Scheduler.from_scenario(sc) as many:
        a, b = one.schedule_many(sc.requests), many.schedule_batch(sc.requests)
        same_results(a, b)
        same_tables(table_of(one), table_of(many))
    if n_plans == 300 and sep[0] == 150.0:  # (with 4 km every request is rejected)
        assert len({r["verdict"] for r in a}) > 1
