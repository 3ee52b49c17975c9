"""The training kernel at the sample counts where its tiling changes: one short tile, one
sample more than a tile, one tile per CTA, two tiles per CTA with their inputs kept, more;
loss, gradient and several Adam steps against the FP64 oracle."""
import numpy as np
import pytest

from oracle import mlp as OM
import paper_1504_05046_gb300 as P
from test_gpu_mlp import F, H, _data, _identity_norm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [127, 128, 129, 152 * 128, 152 * 128 + 1, 2 * 152 * 128 + 77])
def test_gradient_and_steps(n):
    import torch
    X, t = _data(n, n)
    Xd, td = torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda()
    mlp = P.bsmm_mlp_create(5)
    _identity_norm(mlp)
    theta = P.bsmm_mlp_get_params(mlp).astype(np.float64)
    loss, g = P.bsmm_mlp_loss_grad(mlp, Xd, td)
    L, gref = OM.loss_and_grad(theta, X.astype(np.float64), t.astype(np.float64), F, H)
    assert abs(loss - L) <= 1e-5 * max(1.0, L)
    assert np.linalg.norm(g - gref) <= 1e-4 * np.linalg.norm(gref)
    # Adam: 4 steps at a rate small enough that float32 and float64 trajectories stay together
    # (each step moves a coordinate by at most about lr; a sign that differs costs 2 lr)
    steps, lr = 4, 1e-3
    final = P.bsmm_mlp_fit(mlp, Xd, td, steps, lr)
    mu, sd = OM.standardise(X)
    tm, ts = float(t.astype(np.float64).mean()), float(t.astype(np.float64).std())
    m, v = np.zeros_like(theta), np.zeros_like(theta)
    w, settled = theta, np.ones(theta.size, bool)
    for k in range(1, steps + 1):
        _, gk = OM.loss_and_grad(w, (X - mu) / sd, (t - tm) / ts, F, H)
        settled &= np.abs(gk) > 1e-4
        w, m, v = OM.adam_step(w, m, v, gk, k, lr)
    got = P.bsmm_mlp_get_params(mlp).astype(np.float64)
    assert np.max(np.abs(got - w)[settled]) <= 0.02 * lr * steps
    Lw, _ = OM.loss_and_grad(w, (X - mu) / sd, (t - tm) / ts, F, H)
    assert abs(final - Lw) <= 1e-3 * max(1.0, Lw)
