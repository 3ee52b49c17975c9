"""GPU parity of the slicing of tiles near the bottom of the float32 range (and of the float64
range): zeros, subnormal elements and the padding of ragged inner blocks next to elements
whose window reaches below the smallest normal number, for every slice count, either slice
format, either storage order, one scale per tile or per line. Bit for bit against the split
oracle."""
import dataclasses

import numpy as np
import pytest

import bsmm_gen as G
import paper_1504_05046_gb300 as P
from test_gpu_slices import _problem
from test_gpu_split import check
from test_gpu_split_f32 import run_f32

pytestmark = pytest.mark.gpu

# A zero's window is empty by itself down to a largest element of 2^(7s - 124) (2^-117 for
# one slice, 2^-82 for six); below that it has to be decoded as a zero.
SHIFTS = [-75, -82, -83, -84, -90, -97, -104, -111, -118]


def _small(shift_a, shift_b, trans, odd):
    prob = _problem(0, 0, False, odd, seed=5)
    A, B = np.ldexp(prob.A, shift_a), np.ldexp(prob.B, shift_b)
    prob = dataclasses.replace(prob, A=A, B=B)
    return G.as_float32(G.transposed_storage(prob, True, True) if trans else prob)


@pytest.mark.parametrize("s", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("shift", SHIFTS)
def test_small_tiles(shift, s):
    mode = P.BSMM_SPLIT_FP16 if s % 2 else P.BSMM_SPLIT_BF16
    run_f32(_small(shift, 100, s % 2 == 1, True), s, mode)
    if s == 4:
        run_f32(_small(100, shift, False, False), s, mode)


@pytest.mark.parametrize("s", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("shift", [-125, -126, -127, -133, -140, -147, -148])
def test_tiles_of_subnormals(shift, s):
    """Tiles (lines) whose largest element is subnormal: its exponent is that of its leading one."""
    run_f32(_small(shift, 100, s % 2 == 1, True), s)
    run_f32(_small(100, shift, False, False), s, scaling="rows")


@pytest.mark.parametrize("s", [3, 6])
@pytest.mark.parametrize("shift", [-950, -978, -979, -980, -999, -1000, -1001, -1040])
def test_small_float64_tiles(shift, s):
    prob = _problem(0, 0, False, True, seed=7)
    prob = dataclasses.replace(prob, A=np.ldexp(prob.A, shift), B=np.ldexp(prob.B, 900))
    check(prob, s, bar=np.inf)


@pytest.mark.parametrize("trans", [False, True])
@pytest.mark.parametrize("s", [3, 4, 6])
def test_small_lines_of_ordinary_tiles(s, trans):
    """One scale per row and column: rows and columns of every size in the same tiles."""
    prob = _problem(0, 0, False, True, seed=6)
    rng = np.random.default_rng(6)
    A, B = (rng.uniform(0.25, 1.0, x.size) * rng.choice([-1.0, 0.0, 1.0], x.size) for x in (prob.A, prob.B))
    for (rows, cols, off, x, axis) in ((prob.row_sizes, prob.inner_sizes, prob.a_off, A, 0),
                                       (prob.inner_sizes, prob.col_sizes, prob.b_off, B, 1)):
        for u, v in zip(*np.nonzero(off >= 0)):
            t = G.tile_view(x, off, rows, cols, u, v)
            t = t if axis == 0 else t.T
            for line in range(len(t)):  # (the same scale at every inner block)
                t[line] *= 2.0 ** (0 if line % 3 == 0 else SHIFTS[(line + (u, v)[axis]) % len(SHIFTS)])
    prob = dataclasses.replace(prob, A=A, B=B)
    prob = G.as_float32(G.transposed_storage(prob, True, True) if trans else prob)
    run_f32(prob, s, scaling="rows")
