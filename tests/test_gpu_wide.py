"""GPU parity of the contraction's 64-column form (products of deep inner sums whose column
blocks come in pairs): every slice count it is built for, groups of 2 and 4, a last column
block without a partner, a last row block of a few rows, tiles that begin and end inside the
pair, classes of scale that stay, change half way, or differ by row or column tile, cut k
lists, each element type, either storage order. Bit for bit against the split oracle."""
import numpy as np
import pytest

import bsmm_gen as G
import paper_1504_05046_gb300 as P
from test_gpu_split import _scaled_problem, check
from test_gpu_split_complex import run_c
from test_gpu_split_f32 import run_f32

pytestmark = pytest.mark.gpu


def _sizes(seed, n_inner, c):
    rng = np.random.default_rng(seed)
    q = rng.integers(20, 200, n_inner)
    q[-1] += max(0, 3100 - int(q.sum()))
    while q[-1] > 500:  # within the exact depth of every slice count
        q = np.append(q, 200)
        q[-2] -= 200
    return np.asarray([70, 1, 64, 6], np.int32), q.astype(np.int32), np.asarray(c, np.int32)


def _is_wide(plan):
    f = P.bsmm_plan_form(plan)
    return f["cluster"] >= 2 and f["store_warps"] == 0 and f["epi_walk"] == 1


CLASSES = {
    "one": (lambda i, k: 0, lambda k, j: 0),
    "changes": (lambda i, k: 0 if k < 12 else -3, lambda k, j: 0 if k < 20 else 2),
    "rows": (lambda i, k: i % 2, lambda k, j: 0),
    "columns": (lambda i, k: 0, lambda k, j: -(j % 2)),
    "late": (lambda i, k: (i * (k % 7 == 6 and k > 15)), lambda k, j: 0),
}


@pytest.mark.parametrize("classes", list(CLASSES))
@pytest.mark.parametrize("s,cluster", [(6, 4), (6, 2), (5, 2), (4, 4), (3, 2)])
def test_forms_and_scale_classes(s, cluster, classes):
    # 32-column blocks: 0-31 and 32-63 share every tile boundary's inner blocks; 165 columns
    # leave a sixth block of 5 (a pair with the fifth) or, with 150, a fifth alone
    r, q, c = _sizes(s, 30, [40, 3, 90, 17] if cluster == 2 else [40, 3, 90, 32])
    prob = _scaled_problem(7 * s + cluster, r, q, c, *CLASSES[classes])
    prob.alpha, prob.beta = (1.0, 0.0) if classes == "one" else (0.75, -0.5)
    _, plan, _ = check(prob, s, P.BSMM_SPLIT_FP16 if s == 5 else P.BSMM_SPLIT_BF16, cluster=cluster, ksplit=1,
                       bar=np.inf)
    assert _is_wide(plan)


@pytest.mark.parametrize("ksplit", [2, 5, 0])
@pytest.mark.parametrize("classes", ["one", "changes"])
def test_cut_k_lists(classes, ksplit):
    r, q, c = _sizes(11, 30, [40, 3, 90, 17])
    prob = _scaled_problem(12, r, q, c, *CLASSES[classes])
    _, plan, _ = check(prob, 6, cluster=2, ksplit=ksplit)
    assert _is_wide(plan) and (P.bsmm_plan_ksplit(plan)["n_regions"] > 0)


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-0.5, 0.25)])
@pytest.mark.parametrize("trans", [(0, 0), (1, 1)])
def test_element_types(alpha, beta, trans):
    r, q, c = _sizes(13, 30, [40, 3, 90, 17])
    rng = np.random.default_rng(3)
    am, bm = np.ones((len(r), len(q)), np.uint8), np.ones((len(q), len(c)), np.uint8)
    am[0, 3] = am[2, 5] = 0
    bm[7] = 0
    prob = G._assemble("wide", r, c, q, am, bm, rng, "uniform", "wide", alpha, beta)
    t = G.transposed_storage(prob, True, True) if trans[0] else prob
    plan, _ = run_f32(G.as_float32(t), 4, cluster=2, ksplit=1)
    assert _is_wide(plan)
    plan, _ = run_c(G.as_complex(prob, 3), 6, trans=trans, cluster=4, ksplit=1)
    assert _is_wide(plan)


def test_pairs_that_differ_take_the_other_form():
    r, q, c = _sizes(14, 30, [40, 3, 90, 17])
    rng = np.random.default_rng(4)
    am, bm = np.ones((len(r), len(q)), np.uint8), np.ones((len(q), len(c)), np.uint8)
    bm[4, :2] = 0  # columns 0-42: block 0 lacks an inner block that block 1 has through tile 2
    prob = G._assemble("pairs", r, c, q, am, bm, rng, "uniform", "pairs")
    _, plan, _ = check(prob, 6, cluster=2, ksplit=1)
    assert P.bsmm_plan_form(plan)["store_warps"] == 1


@pytest.mark.parametrize("s", [3, 4, 6])
def test_plans_of_the_form_in_a_batch(s):
    """A batch runs every plan with the 32-column kernel: the same bits as each plan's own
    execute, also with the column blocks packed in pairs (3 and 4 slices)."""
    import torch
    r, q, c = _sizes(15, 30, [40, 3, 90, 17])
    probs = [_scaled_problem(20 + i, r, q, c, *CLASSES[k]) for i, k in enumerate(("one", "changes"))]
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    plans, args, alone = [], [], []
    for p in probs:
        plan = P.bsmm_plan(r, c, q, p.a_mask, p.b_mask, nslices=s, mode=P.BSMM_SPLIT_BF16, cluster=2, ksplit=1)
        assert _is_wide(plan)
        off, tot = G.layout_arena(P.bsmm_plan_query(plan)["c_mask"], r, c)
        a = [d(p.A), d(p.a_off), d(p.B), d(p.b_off), torch.zeros(tot, dtype=torch.float64, device="cuda"), d(off)]
        P.bsmm_execute(plan, 1.0, a[0], a[1], a[2], a[3], 0.0, a[4], a[5])
        P.bsmm_status_device(plan)
        alone.append(a[4].cpu().numpy())
        a[4].zero_()
        plans.append(plan)
        args.append(a)
    batch = P.bsmm_batch_create(plans)
    P.bsmm_batch_set_args(batch, [1.0, 1.0], *[[a[i] for a in args] for i in range(4)], [0.0, 0.0],
                          [a[4] for a in args], [a[5] for a in args])
    P.bsmm_batch_execute(batch)
    P.bsmm_batch_status_device(batch)
    for a, want in zip(args, alone):
        assert np.array_equal(a[4].cpu().numpy(), want)
