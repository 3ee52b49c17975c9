"""GPU parity of the 64-column form's store and scales on rare values: results below the
normal range and beyond the largest number next to ordinary ones, row and column scaling
with all-zero lines, factors that are no powers of two. Bit for bit against the split
oracle."""
import dataclasses

import numpy as np
import pytest

import bsmm_gen as G
import oracle
from oracle import split as OS
import paper_1504_05046_gb300 as P
from gpu_helpers import run_lib
from helpers import c_arena, struct_elements
from test_gpu_split import _scaled_problem
from test_gpu_split_complex import run_c
from test_gpu_split_f32 import run_f32
from test_gpu_wide import _is_wide, _sizes

pytestmark = pytest.mark.gpu


def _check(prob, s, scaling="tile", **opt):
    cs, _, _ = oracle.structure(prob)
    off, C0 = c_arena(prob, cs, rng=np.random.default_rng(0))
    want = C0.copy()
    OS.bsmm_split(prob, cs, want, off, s, scaling=scaling)
    got, plan = run_lib(prob, cs, C0, off, mode=P.BSMM_SPLIT_BF16, nslices=s, ksplit=1,
                        split_scale=int(scaling == "rows"), **opt)
    assert _is_wide(plan)
    g, w = (struct_elements(prob, cs, off, x) for x in (got, want))
    assert np.array_equal(g, w)
    return w


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (0.5, 0.25), (-0.3, 1.7)])
@pytest.mark.parametrize("s", [3, 4, 6])
def test_results_at_both_ends_of_the_range(s, alpha, beta):
    r, q, c = _sizes(61, 30, [40, 3, 90, 17])
    ends = [-1075, 1020, -1055, 1020]  # by row tile: 2^end times sums of 3000 products in (-1, 1)
    prob = _scaled_problem(62, r, q, c, lambda i, k: ends[i] // 2, lambda k, j: 0)
    a = prob.A.copy()
    for i, e in enumerate(ends):
        for k in range(len(q)):
            o = prob.a_off[i, k]
            a[o:o + r[i] * q[k]] *= 2.0 ** (e - e // 2)
    prob = dataclasses.replace(prob, A=a, alpha=alpha, beta=beta)
    w = _check(prob, s, cluster=2)
    assert np.isinf(w).sum() > 10
    assert beta != 0.0 or ((w != 0) & (np.abs(w) < 2.0 ** -1022)).sum() > 1000


@pytest.mark.parametrize("s", [3, 4])
def test_float32_results_at_both_ends_of_the_range(s):
    r, q, c = _sizes(63, 30, [40, 3, 90, 17])
    ends = [-147, 124, -130, 124]
    prob = _scaled_problem(64, r, q, c, lambda i, k: -100 if ends[i] < 0 else ends[i] // 2,
                           lambda k, j: 0)
    b = lambda i: ends[i] + 100 if ends[i] < 0 else ends[i] - ends[i] // 2
    a = prob.A.copy()
    for i in range(len(r)):
        for k in range(len(q)):
            o = prob.a_off[i, k]
            a[o:o + r[i] * q[k]] *= 2.0 ** b(i)
    plan, _ = run_f32(G.as_float32(dataclasses.replace(prob, A=a)), s, cluster=2, ksplit=1)
    assert _is_wide(plan)


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-0.3, 1.7)])
@pytest.mark.parametrize("s,cluster", [(3, 2), (4, 4), (6, 2), (6, 4)])
def test_row_and_column_scaling_with_zero_lines(s, cluster, alpha, beta):
    r, q, c = _sizes(65, 30, [40, 3, 90, 32])
    prob = _scaled_problem(66, r, q, c, lambda i, k: -(k // 15), lambda k, j: 0)
    A, B = prob.A.copy(), prob.B.copy()
    rng = np.random.default_rng(67)
    for i in range(len(r)):
        for k in range(len(q)):
            t = G.tile_view(A, prob.a_off, r, q, i, k)
            t *= 2.0 ** -(np.arange(r[i]) % 7)[:, None]
            t[rng.random(r[i]) < 0.1] = 0.0
            if i == 0:
                t[5] = 0.0  # a row that is zero everywhere
    for k in range(len(q)):
        for j in range(len(c)):
            t = G.tile_view(B, prob.b_off, q, c, k, j)
            t *= 2.0 ** -(np.arange(c[j]) % 5)
            t[:, rng.random(c[j]) < 0.1] = 0.0
            if j == 2:
                t[:, 31] = 0.0
    _check(dataclasses.replace(prob, A=A, B=B, alpha=alpha, beta=beta), s, "rows", cluster=cluster)


def test_complex_row_scaling_with_zero_lines():
    r, q, c = _sizes(68, 30, [40, 3, 90, 17])
    prob = _scaled_problem(69, r, q, c, lambda i, k: 0, lambda k, j: 0)
    prob = G.as_complex(dataclasses.replace(prob, alpha=-0.3, beta=1.7), 3)
    A = prob.A.copy()
    for i in range(len(r)):
        for k in range(0, len(q), 7):
            G.tile_view(A, prob.a_off, r, q, i, k)[:: 3] = 0.0
    plan, _ = run_c(dataclasses.replace(prob, A=A), 6, cluster=4, ksplit=1, split_scale=1)
    assert _is_wide(plan)
