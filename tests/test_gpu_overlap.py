"""The kernels of one product placed while their predecessors end: calls issued back to back,
eagerly and from a captured graph, have the bits of a plan that records an event between any
two of its kernels (which orders them fully)."""
import numpy as np
import pytest

import bsmm_gen as G
import paper_1504_05046_gb300 as P
from test_gpu_split import _scaled_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_inner,options", [
    (2, {}),                                   # exponents, slices, contraction
    (2, {"split_scale": 1}),                   # one scale per line: a kernel more
    (24, {"ksplit": 4}),                       # and the reduction of cut k lists
    (30, {"cluster": 2}), (30, {"cluster": 2, "ksplit": 3}),
])
def test_back_to_back_calls(n_inner, options):
    import torch
    rng = np.random.default_rng(n_inner)
    q = rng.integers(100, 200, n_inner).astype(np.int32)
    r, c = np.asarray([70, 1, 130], np.int32), np.asarray([40, 3, 90], np.int32)
    probs = [_scaled_problem(3 + i, r, q, c, lambda i, k: i - k % 3, lambda k, j: j) for i in range(6)]
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    ins = [(d(p.A), d(p.B)) for p in probs]
    p = probs[0]
    a_off, b_off = d(p.a_off), d(p.b_off)

    def plan(**k):
        return P.bsmm_plan(r, c, q, p.a_mask, p.b_mask, mode=P.BSMM_SPLIT_BF16, **options, **k)

    def call(pl, A, B, C):
        P.bsmm_execute(pl, 0.75, A, a_off, B, b_off, 0.0, C, c_off)

    ordered = plan(profile=1)
    off, total = G.layout_arena(P.bsmm_plan_query(ordered)["c_mask"], r, c)
    c_off = d(off)
    want = [torch.zeros(total, dtype=torch.float64, device="cuda") for _ in ins]
    for (A, B), C in zip(ins, want):
        call(ordered, A, B, C)
        torch.cuda.synchronize()
    overlapped = plan()
    got = [torch.zeros_like(C) for C in want]
    for _ in range(3):
        for (A, B), C in zip(ins, got):
            call(overlapped, A, B, C)
    P.bsmm_status_device(overlapped)
    assert all(torch.equal(x, y) for x, y in zip(got, want))

    for C in got:
        C.zero_()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        for (A, B), C in zip(ins, got):
            call(overlapped, A, B, C)
    g.replay()
    g.replay()
    P.bsmm_status_device(overlapped)
    assert all(torch.equal(x, y) for x, y in zip(got, want))
