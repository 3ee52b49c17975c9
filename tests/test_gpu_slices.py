"""GPU parity of the slicing where its rounding can go wrong: elements at and next to an
exact tie of every level, elements far below their tile's largest, zeros, tiles near both
ends of the exponent range; for every slice count, both slice formats, float64 and float32
elements, either storage order, and inner blocks that leave part of a 16-byte load, of a
32-deep chunk, of a pair of chunks or of a group of four column blocks. Bit for bit against
the split oracle."""
import dataclasses

import numpy as np
import pytest

import bsmm_gen as G
import paper_1504_05046_gb300 as P
from test_gpu_split import check
from test_gpu_split_f32 import run_f32

pytestmark = pytest.mark.gpu


def _tie_values(n, rng, dtype):
    """Values in (-1, 1) whose lowest set bit is at or near a rounding position of a level."""
    t = rng.integers(0, 7, n)  # (N + 1/2) 2^(-7t): a tie of level t
    x = (np.floor(rng.random(n) * 2.0 ** (7 * t)) + 0.5) * 2.0 ** (-7.0 * t)
    bits = 53 if dtype == np.float64 else 24
    x = x + rng.integers(-1, 2, n) * 2.0 ** -rng.integers(7 * t + 2, 55).astype(float)  # and just off it
    x = x * 2.0 ** (-rng.integers(0, 70, n) * (rng.random(n) < 0.2))  # some far below the rest
    x = np.where(rng.random(n) < 0.05, 0.0, x)
    x = np.clip(x, -(1 - 2.0 ** -bits), 1 - 2.0 ** -bits) * rng.choice([-1.0, 1.0], n)
    return x.astype(dtype)


def _problem(shift_a, shift_b, trans, odd, dtype=np.float64, seed=0):
    rng = np.random.default_rng(seed)
    r, c = np.asarray([40, 3, 100], np.int32), np.asarray([33, 130, 8], np.int32)
    q = np.asarray([33, 95, 1, 161] if odd else [32, 96, 4, 164], np.int32)
    am, bm = np.ones((3, 4), np.uint8), np.ones((4, 3), np.uint8)
    am[1, 2] = bm[3, 0] = 0
    prob = G._assemble("slices", r, c, q, am, bm, rng, "uniform", "slices")
    prob = dataclasses.replace(prob, A=np.ldexp(_tie_values(prob.A.size, rng, np.float64), shift_a),
                               B=np.ldexp(_tie_values(prob.B.size, rng, np.float64), shift_b))
    if trans:
        prob = G.transposed_storage(prob, True, True)
    return prob


@pytest.mark.parametrize("trans,odd", [(False, False), (False, True), (True, False), (True, True)])
@pytest.mark.parametrize("s", [1, 2, 3, 4, 5, 6])
def test_ties_float64(s, trans, odd):
    mode = P.BSMM_SPLIT_FP16 if s % 2 else P.BSMM_SPLIT_BF16
    check(_problem(0, 0, trans, odd), s, mode, bar=np.inf)


@pytest.mark.parametrize("trans,odd", [(False, False), (True, True)])
@pytest.mark.parametrize("s", [3, 4, 6])
def test_ties_float32(s, trans, odd):
    prob = _problem(0, 0, False, odd)
    prob = G.as_float32(G.transposed_storage(prob, True, True) if trans else prob)
    run_f32(prob, s, P.BSMM_SPLIT_FP16 if s == 4 else P.BSMM_SPLIT_BF16)


@pytest.mark.parametrize("shift", [-899, -900, -901, -1022, -1060, 900])
def test_ties_at_the_ends_of_the_exponent_range(shift):
    for s in (3, 6):
        check(_problem(shift, -shift if abs(shift) < 1000 else 900, False, False, seed=1), s, bar=np.inf)
