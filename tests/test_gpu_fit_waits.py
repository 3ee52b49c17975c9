"""The training kernel's grid barrier, exercised on the GPU without a fault, trap or hang: a
barrier that waits for one arrival too many runs out of its short limit, every CTA leaves, the
call reports BSMM_ERR_TIMEOUT, and the context then trains a model correctly."""
import time

import numpy as np
import pytest

import paper_1504_05046_gb300 as P
from test_gpu_mlp import _data

pytestmark = pytest.mark.gpu


def _fits(n=300):
    import torch
    X, t = (torch.from_numpy(x).cuda() for x in _data(n, 1))
    losses = []
    for _ in range(2):
        mlp = P.bsmm_mlp_create(3)
        losses.append(P.bsmm_mlp_fit(mlp, X, t, 5, 1e-3))
    return losses


@pytest.mark.parametrize("with_loss", [True, False])
def test_barrier_that_runs_out_is_reported(with_loss):
    import torch
    before = _fits()
    limit = 50_000_000  # 50 ms
    for _ in range(3):
        t0 = time.perf_counter()
        with pytest.raises(P.BsmmError) as ei:
            P.bsmm_selftest_fit(limit, with_loss=with_loss)
        assert ei.value.status == 4
        assert time.perf_counter() - t0 < 1.0  # one limit, not one per barrier
    torch.cuda.synchronize()
    after = _fits()
    assert np.isfinite(after).all() and before == after
