"""GPU parity at the sizes where a launch plan changes: tile edges of the
tensor-core forward, the FP32 kernels with several rows per thread, the
eigensolver's cluster sizes, and the column counts of the shifted solves,
against the FP64 oracle.  Tolerances are the method's stated targets of
test_gpu_kmv.py and the bounds that test_gpu_nystrom.py and test_gpu_phi.py
derive."""
import math

import numpy as np
import pytest
import torch

import workloads as wl
from oracle import poles, se_kernel as sk
from helpers import to_dev, f32, abs_row_products, componentwise_err, grad_err
from test_gpu_kmv import TOL, _check_backward, _check_forward
from test_gpu_nystrom import _check_factor, _omega

pytestmark = pytest.mark.gpu


# I tiles come in pairs of 128 rows and J tiles in halves of 64 columns; up to 16 columns
# keep their fold sums in shared memory, in halves of 8
@pytest.mark.parametrize("m", [3, 9, 16, 17, 40, 64])
@pytest.mark.parametrize("sizes,d", [([1, 127], 3), ([128, 129, 0, 255], 8), ([257, 513], 20)])
def test_tensor_forward_tile_edges(kmv_handle, sizes, d, m):
    _check_forward(kmv_handle, wl.ragged(sizes, d=d, chains=1, m=m, seed=1000 + d + m), "bf16_hilo")


# 4 chains of 4,609 rows = 9 x 512 + 1 give each SM two CTAs of the several-row FP32
# kernels (2 or 4 rows a thread by d and m) with a last tile of one row; 1,537 rows do not
@pytest.mark.parametrize("n", [1537, 4609])
@pytest.mark.parametrize("d,m", [(1, 1), (3, 2), (4, 5), (8, 16), (13, 3), (32, 2)])
def test_fp32_rows_per_thread(kmv_handle, n, d, m):
    w = wl.ragged([n, 3], d=d, chains=4, m=m, seed=2000 + d + m)
    pts, theta, V, G = to_dev(w)
    Y = kmv_handle.kmv_forward(pts, theta, V, prec="fp32").cpu().numpy()
    gth, gV = kmv_handle.kmv_backward(pts, theta, V, G, prec="fp32")
    gth, gV = gth.cpu().numpy(), gV.cpu().numpy()
    X, Vh, Gh = f32(w.X), f32(w.V), f32(w.G)
    rows = np.r_[0:3, 509:515, n - 3:n]
    for c in (0, 3):
        ref = sk.kmv(X[:n], w.theta[c], Vh[c, :n], w.ard, rows=rows)
        scale = abs_row_products(X[:n], w.theta[c], Vh[c, :n], w.ard, rows)
        assert componentwise_err(Y[c, rows], ref, scale) <= TOL["fp32"][0]
        # grad_V = A G row by row (A is symmetric)
        ref = sk.kmv(X[:n], w.theta[c], Gh[c, :n], w.ard, rows=rows)
        scale = abs_row_products(X[:n], w.theta[c], Gh[c, :n], w.ard, rows)
        assert componentwise_err(gV[c, rows], ref, scale) <= TOL["fp32"][0]
    g_ref, _ = sk.kmv_adjoint(X[:n], w.theta[1], Vh[1, :n], Gh[1, :n], w.ard)
    assert grad_err(gth[1], g_ref) <= TOL["fp32"][1]


# XA in shared memory (3 d > 32 columns of tensor memory) or in tensor memory, tile edges
@pytest.mark.parametrize("d", [5, 10, 11, 18])
@pytest.mark.parametrize("sizes", [[64, 65], [127, 129, 1], [384]])
def test_tensor_adjoint_tile_edges(kmv_handle, sizes, d):
    _check_backward(kmv_handle, wl.ragged(sizes, d=d, chains=1, m=4, seed=3000 + d), "bf16_hilo")


# one system takes the largest cluster of the eigensolver, many take one block each; odd
# ranks leave one column out of every sweep's pairs
@pytest.mark.parametrize("n_inst,rank", [(1, 1), (1, 2), (1, 33), (1, 64), (3, 31), (40, 7)])
def test_eigensolver_clusters(kmv_handle, n_inst, rank):
    w = wl.ragged([140] * n_inst, d=2, chains=1, m=1, seed=4000 + rank)
    pts, theta, _, _ = to_dev(w)
    Om = _omega(w, rank, rank)
    U, lam, st = kmv_handle.nystrom_build(pts, theta, torch.tensor(Om, device="cuda"))
    _check_factor(w, U.cpu().numpy(), lam.cpu().numpy(), st.cpu().numpy(), Om, rank,
                  lambda X, s: sk.kernel_matrix(X, X, w.theta[s], True))


# 16 columns are the most that the block reduction of the several-column solve takes at once
@pytest.mark.parametrize("n_poles", [3, 16, 17, 32])
@pytest.mark.parametrize("precond", [False, True])
def test_shifted_solves_column_counts(kmv_handle, n_poles, precond):
    w = wl.ragged([300, 129], d=2, chains=2, m=1, seed=5000 + n_poles)
    pts, theta, _, _ = to_dev(w)
    xi = np.random.default_rng(n_poles).standard_normal((w.chains, w.n_total)).astype(np.float32)
    if precond:
        U, lam, _ = kmv_handle.nystrom_build(pts, theta, torch.tensor(_omega(w, 24, 5), device="cuda"))
        kmv_handle.set_preconditioner(pts, U, lam)
    try:
        phi, st, _, pl = kmv_handle.phi_refresh(pts, theta, torch.tensor(xi, device="cuda"), n_poles=n_poles,
                                                cg_tol=1e-6, cg_maxiter=3000, want_poles=True)
    finally:
        kmv_handle.set_preconditioner(pts)
    assert torch.all(st == 0)
    phi, pl = phi.cpu().numpy(), pl.cpu().numpy()
    X = f32(w.X)
    for s in range(4):
        b, c = divmod(s, 2)
        r0, r1 = w.offsets[b], w.offsets[b + 1]
        A = sk.A_matrix(X[r0:r1], w.theta[s], True)
        ref = poles.inv_sqrt_apply(A, xi[c, r0:r1].astype(np.float64), pl[s, 0], pl[s, 1], n_poles)
        bound = 20 * 1e-6 * np.linalg.norm(xi[c, r0:r1]) / math.sqrt(pl[s, 0]) + 1e-5 * np.linalg.norm(ref)
        assert np.linalg.norm(phi[c, r0:r1] - ref) <= bound
