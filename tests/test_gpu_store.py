"""GPU parity of the C store and its rounding on the row tilings where they can go wrong:
tiles of 0, 1 and 2 rows, tiles that end one row before, at and after a warp's 32 rows, a
last row block of a few rows, columns of several tiles in one 32-column block. Each
element type, with and without alpha and beta, in both kernel forms and through the
split-k reduction; bit for bit against the split oracle."""

import dataclasses

import numpy as np
import pytest

import bsmm_gen as G
import paper_1504_05046_gb300 as P
from test_gpu_split_complex import run_c
from test_gpu_split_f32 import run_f32
from test_gpu_split import check

pytestmark = pytest.mark.gpu

ROWS = [0, 1, 2, 0, 28, 1, 33, 31, 32, 0, 64, 7, 3]  # 202 rows: boundaries at 31, 32, 65, 96, 128, 192
COLS = [5, 0, 1, 26, 33, 2]


def _problem(alpha, beta):
    rng = np.random.default_rng(5)
    r, c, q = (np.asarray(x, np.int32) for x in (ROWS, COLS, [17, 40, 3]))
    am = (rng.random((len(r), len(q))) < 0.7).astype(np.uint8)
    bm = (rng.random((len(q), len(c))) < 0.7).astype(np.uint8)
    return G._assemble("store", r, c, q, am, bm, rng, "uniform", "store", alpha, beta)


@pytest.mark.parametrize("form", [dict(store_warps=2), dict(store_warps=1), dict(ksplit=2)])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-0.5, 0.0), (1.0, 0.75), (0.375, -2.0)])
@pytest.mark.parametrize("elem", ["f64", "f32", "c128"])
def test_row_segments(elem, alpha, beta, form):
    prob = _problem(alpha, beta)
    if elem == "f64":
        check(prob, 6, **form)
    elif elem == "f32":
        run_f32(G.as_float32(prob), **form)
    else:
        run_c(G.as_complex(prob, 3), **form)


@pytest.mark.parametrize("form", [dict(store_warps=2), dict(store_warps=1), dict(ksplit=2)])
@pytest.mark.parametrize("alpha,beta", [(-1.0, 1.0), (1.0, -1.0), (0.5, -0.25), (2.0 ** -1021, 1.0), (1.0, 2.0 ** -1000),
                                        (2.0 ** 900, 2.0 ** 200), (2.0 ** -1030, 0.5), (0.0, 2.0), (3.0, 2.0 ** -3)])
def test_factors_that_are_powers_of_two(alpha, beta, form):
    """alpha and beta formed on the bits: signs, zeros, subnormal and overflowing results, and
    zeros, subnormals, infinities and the extremes in C; the two-multiplication epilogue's bits."""
    import oracle
    from gpu_helpers import run_lib
    from helpers import c_arena, struct_elements
    from oracle import split as OS
    prob = _problem(alpha, beta)
    cs, _, _ = oracle.structure(prob)
    off, C0 = c_arena(prob, cs, rng=np.random.default_rng(2))
    special = np.array([0.0, -0.0, 5e-324, -2.0 ** -1022, 1.7e308, -1.7e308, np.inf, -np.inf, 2.0 ** -1000, 1.5e-320])
    C0[::3] = np.resize(special, C0[::3].size)
    # the product's own sums from the oracle with alpha = 1, beta = 0, then the epilogue as stated
    plain = dataclasses.replace(prob, alpha=1.0, beta=0.0)
    acc = C0.copy()
    OS.bsmm_split(plain, cs, acc, off, 6)
    with np.errstate(all="ignore"):
        want = alpha * acc + beta * C0 if beta else alpha * acc
    got, _ = run_lib(prob, cs, C0, off, mode=P.BSMM_SPLIT_BF16, nslices=6, **form)
    g, w = struct_elements(prob, cs, off, got), struct_elements(prob, cs, off, want)
    same = (g.view(np.int64) == w.view(np.int64)) | (np.isnan(g) & np.isnan(w))
    assert same.all(), (g[~same][:4], w[~same][:4])
