"""GPU: an explicit kernel form is the one that runs. A product that the planner would give the
64-column form keeps the form with C store warps (store_warps = 2) or without (1) when the
options ask for it, with the same bits."""
import numpy as np
import pytest

import paper_1504_05046_gb300 as P
from test_gpu_split import _scaled_problem, check
from test_gpu_wide import CLASSES, _is_wide, _sizes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,cluster", [(6, 4), (4, 2), (3, 2)])
def test_store_warps_are_kept(s, cluster):
    r, q, c = _sizes(31, 30, [40, 3, 90, 17])
    prob = _scaled_problem(31, r, q, c, *CLASSES["changes"])
    runs = {}
    for sw in (0, 1, 2):
        got, plan, _ = check(prob, s, cluster=cluster, ksplit=1, bar=np.inf, store_warps=sw)
        runs[sw] = got
        assert _is_wide(plan) == (sw == 0)
        assert P.bsmm_plan_form(plan)["store_warps"] == (1 if sw == 2 else 0)
    assert np.array_equal(runs[0], runs[1]) and np.array_equal(runs[0], runs[2])
