"""GPU: with 5 and 6 slices the scale classes of the data decide, at each execute, which of the
two contraction forms runs. Same bits either way (against the split oracle), for data that
falls on either side and changes from one execute to the next, with cut k lists, row and
column scaling and under graph replay; and products whose classes change at every inner block
take no longer than with the 32-column form."""
import dataclasses

import numpy as np
import pytest

import bsmm_gen as G
import oracle
from oracle import split as OS
import paper_1504_05046_gb300 as P
from gpu_helpers import to_dev
from helpers import c_arena, struct_elements
from test_gpu_split import _scaled_problem
from test_gpu_wide import _is_wide, _sizes

pytestmark = pytest.mark.gpu

# A's scale per (row tile, inner block): the share of changes below, near and above the limits
SCALES = {
    "one": lambda i, k: 0,
    "few": lambda i, k: -(k // 10),
    "some": lambda i, k: -(k % 8 == 7),
    "rows": lambda i, k: -(i % 2) * (k % 3 == 1),
    "all": lambda i, k: -(k % 2),
}


def _problems(s, c, scaling="tile"):
    r, q, c = _sizes(40 + s, 34, c)
    out = []
    for n, f in enumerate(SCALES.values()):
        prob = _scaled_problem(50 + n, r, q, c, f, lambda k, j: 0)
        out.append(dataclasses.replace(prob, alpha=0.75, beta=-0.5))
    return out


@pytest.mark.parametrize("scaling", ["tile", "rows"])
@pytest.mark.parametrize("s,ksplit", [(6, 1), (5, 1), (6, 3)])
def test_bits_on_both_sides(s, ksplit, scaling):
    import torch
    probs = _problems(s, [40, 3, 90, 17])
    p0 = probs[0]
    plan = P.bsmm_plan(p0.row_sizes, p0.col_sizes, p0.inner_sizes, p0.a_mask, p0.b_mask, mode=P.BSMM_SPLIT_BF16, nslices=s,
                       cluster=2, ksplit=ksplit, split_scale=int(scaling == "rows"))
    assert _is_wide(plan)
    cs, _, _ = oracle.structure(p0)
    off, C0 = c_arena(p0, cs, rng=np.random.default_rng(0))
    A, B, ao, bo, co = (to_dev(x) for x in (p0.A, p0.B, p0.a_off, p0.b_off, off))
    C = to_dev(C0)
    run = lambda: P.bsmm_execute(plan, p0.alpha, A, ao, B, bo, p0.beta, C, co)
    run()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    for prob in probs + probs[::-1]:
        want = C0.copy()
        OS.bsmm_split(prob, cs, want, off, s, scaling=scaling)
        A.copy_(to_dev(prob.A))
        B.copy_(to_dev(prob.B))
        for step in (run, graph.replay):
            C.copy_(to_dev(C0))
            step()
            torch.cuda.synchronize()
            P.bsmm_status_device(plan)
            g, w = (struct_elements(prob, cs, off, x) for x in (C.cpu().numpy(), want))
            assert np.array_equal(g, w)


@pytest.mark.parametrize("s", [5, 6])
def test_changing_classes_cost_no_more_than_the_other_form(s):
    """2048 x 2048 x 4096, inner blocks of 96, a class of its own for each: before the choice the
    64-column form took 1.4 times as long as the 32-column one (store_warps = 2)."""
    import torch
    tiles = lambda n, b: np.asarray([b] * (n // b) + ([n % b] if n % b else []), np.int32)
    t, q = tiles(2048, 128), tiles(4096, 96)
    am, bm = np.ones((len(t), len(q)), np.uint8), np.ones((len(q), len(t)), np.uint8)
    offs = [G.layout_arena(m, a, b) for m, a, b in ((am, t, q), (bm, q, t), (np.ones((len(t),) * 2, np.uint8), t, t))]
    gen = torch.Generator(device="cuda").manual_seed(1)
    A, B = (torch.rand(tot, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1 for _, tot in offs[:2])
    for i in range(len(t)):
        for k in range(1, len(q), 2):
            o = int(offs[0][0][i, k])
            A[o:o + int(t[i]) * int(q[k])] *= 0.5
    C = torch.zeros(offs[2][1], dtype=torch.float64, device="cuda")
    ao, bo, co = (torch.from_numpy(o).cuda() for o, _ in offs)
    plans = [P.bsmm_plan(t, t, q, am, bm, mode=P.BSMM_SPLIT_BF16, nslices=s, cluster=4, store_warps=sw) for sw in (0, 2)]
    assert _is_wide(plans[0]) and not _is_wide(plans[1])

    def us(plan, passes=10):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(passes):
            P.bsmm_execute(plan, 1.0, A, ao, B, bo, 0.0, C, co)
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b) / passes

    for p in plans:
        us(p)
    ratio = [us(plans[0]) / us(plans[1]) for _ in range(9)]
    for p in plans:
        P.bsmm_status_device(p)
    assert np.median(ratio) <= 1.12, ratio
