"""GPU parity on both sides of dispatch rules that depend on the size of a system: the CG
direction's own kernel above 4096 rows, the implicit step's reductions by a warp above 64
row tiles, and the many-dimension forward with several items per CTA and several folds per
item.  Tolerances are those of test_gpu_hmc.py, test_gpu_implicit.py and test_gpu_kmv.py."""
import numpy as np
import pytest
import torch

import workloads as wl
from oracle import se_kernel as sk
from helpers import abs_row_products, componentwise_err, f32, to_dev
from test_gpu_kmv import TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", [False, True])
@pytest.mark.parametrize("n", [4096, 4097])
def test_cg_direction_by_a_kernel_or_the_last_block(kmv_handle, n, precond):
    w = wl.ragged([n, 50], d=2, chains=1, m=1, seed=9000, sigma2=0.1)
    pts, theta, _, _ = to_dev(w)
    y = torch.tensor(w.y, dtype=torch.float32, device="cuda")
    if precond:
        om = torch.tensor(np.random.default_rng(9001).standard_normal((1, w.n_total, 32)), dtype=torch.float32,
                          device="cuda")
        U, lam, _ = kmv_handle.nystrom_build(pts, theta, om)
        kmv_handle.set_preconditioner(pts, U, lam)
    try:
        x, st, _ = kmv_handle.kmv_cg_solve(pts, theta, y, tol=1e-6, maxiter=5000)
    finally:
        kmv_handle.set_preconditioner(pts)
    assert torch.all(st == 0)
    X, yh, xh = f32(w.X), f32(w.y), f32(x[0].cpu().numpy())
    for b in range(2):
        r = slice(w.offsets[b], w.offsets[b + 1])
        res = yh[r] - sk.kmv(X[r], w.theta[b], xh[r], True)
        A_norm = np.abs(sk.A_matrix(X[r], w.theta[b], True)).sum(1).max()
        floor = 20 * 2.0 ** -24 * A_norm * np.linalg.norm(xh[r])
        assert np.linalg.norm(res) <= 1e-6 * np.linalg.norm(yh[r]) + floor


def test_implicit_step_of_many_tiles(kmv_handle):
    # 8,200 rows = 65 tiles of 128; a smooth kernel, whose leading 64 eigenvectors leave the
    # preconditioned system near the identity
    w = wl.ragged([8200], d=2, chains=1, m=1, seed=9100, ell_range=(1.0, 2.0), sigma2=0.5)
    rng = np.random.default_rng(9101)
    phi, pi0 = rng.standard_normal((1, 8200)).astype(np.float32), 0.5 * rng.standard_normal(w.theta.shape)
    dt, tol = 1e-3, 1e-4
    pts, theta, _, _ = to_dev(w)
    th, pi = theta.clone(), torch.tensor(pi0, dtype=torch.float64, device="cuda")
    U, lam, _ = kmv_handle.nystrom_build(pts, theta, torch.tensor(rng.standard_normal((1, 8200, 64)),
                                                                  dtype=torch.float32, device="cuda"))
    kmv_handle.set_preconditioner(pts, U, lam)
    try:
        st, _, x = kmv_handle.implicit_step(pts, torch.tensor(w.y, dtype=torch.float32, device="cuda"),
                                            torch.tensor(phi, device="cuda"), th, pi, dt, tol=tol, maxiter=1500)
    finally:
        kmv_handle.set_preconditioner(pts)
    assert int(st[0]) == 0
    th, pi, xs = th.cpu().numpy()[0], pi.cpu().numpy()[0], x.cpu().numpy()[0].astype(np.float64)
    X, yh = f32(w.X), f32(w.y)
    tb = 0.5 * (w.theta[0] + th)
    assert np.linalg.norm(sk.kmv(X, tb, xs, True) - yh) <= 5 * tol * np.linalg.norm(yh)
    # theta and pi moved by at most tol (1 + |.|) in the last iteration
    slack = 2 * tol * (1.0 + max(np.abs(th).max(), np.abs(pi).max()))
    np.testing.assert_allclose(th, w.theta[0] + 0.5 * dt * (pi0[0] + pi), rtol=0, atol=dt * slack)
    # the force with x held fixed: -x'Kx/2 + phi'K phi/2 differentiated
    ph = f32(phi[0])
    F, _ = sk.kmv_adjoint(X, tb, np.stack([xs, ph], 1), np.stack([-0.5 * xs, 0.5 * ph], 1), True)
    np.testing.assert_allclose(pi, pi0[0] - dt * F, rtol=0, atol=dt * 1e-3 * max(np.abs(F).max(), 1.0) + slack)


# 20,000 rows: 157 J tiles (a fold every 32), 4 chains: more items than SMs
@pytest.mark.parametrize("d,m", [(24, 16), (25, 16), (31, 3)])
def test_many_dimension_forward_of_several_items(kmv_handle, d, m):
    n = 20000
    w = wl.ragged([n], d=d, chains=4, m=m, seed=9200 + d, ell_range=(1.0, 3.0))
    pts, theta, V, _ = to_dev(w)
    Y = kmv_handle.kmv_forward(pts, theta, V, prec="bf16_hilo").cpu().numpy()
    X, Vh = f32(w.X), f32(w.V)
    rows = np.r_[0:3, 8190:8194, n - 3:n]
    for c in range(4):
        ref = sk.kmv(X, w.theta[c], Vh[c], True, rows=rows)
        scale = abs_row_products(X, w.theta[c], Vh[c], True, rows)
        assert componentwise_err(Y[c, rows], ref, scale) <= TOL["bf16_hilo"][0]
