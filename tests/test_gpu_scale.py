"""The solves do not depend on the scale of their right-hand side: with y and xi scaled by
a power of two every FP32 value and FP64 sum of the iteration scales exactly, so the
iteration counts are the same and the solutions the scaled ones, bit for bit.  At 2^-56
the residuals at convergence are about 1e-23, whose squares FP32 cannot hold; at 2^66
the squares of y are above FP32's largest value."""
import numpy as np
import pytest
import torch

import workloads as wl
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "bf16_hilo"])
@pytest.mark.parametrize("precond", [False, True])
@pytest.mark.parametrize("k", [-56, 66])
def test_solves_scale_exactly(kmv_handle, k, precond, prec):
    w = wl.ragged([300, 129], d=2, chains=2, m=1, seed=6000, sigma2=0.1)
    pts, theta, _, _ = to_dev(w)
    rng = np.random.default_rng(6001)
    y = torch.tensor(w.y, dtype=torch.float32, device="cuda")
    xi = torch.tensor(rng.standard_normal((w.chains, w.n_total)), dtype=torch.float32, device="cuda")
    if precond:
        om = torch.tensor(rng.standard_normal((w.chains, w.n_total, 16)), dtype=torch.float32, device="cuda")
        U, lam, _ = kmv_handle.nystrom_build(pts, theta, om)
        kmv_handle.set_preconditioner(pts, U, lam)

    def solves(scale):
        x, st, it = kmv_handle.kmv_cg_solve(pts, theta, scale * y, tol=1e-6, maxiter=1000, prec=prec)
        phi, st2, it2 = kmv_handle.phi_refresh(pts, theta, scale * xi, n_poles=15, cg_tol=1e-6, cg_maxiter=2000,
                                               prec=prec)[:3]
        return x, phi, it, it2, st, st2

    try:
        ref, got = solves(1.0), solves(2.0 ** k)
    finally:
        kmv_handle.set_preconditioner(pts)
    for a in ref[4:] + got[4:]:
        assert torch.all(a == 0)
    assert torch.equal(got[2], ref[2]) and torch.equal(got[3], ref[3])
    assert torch.equal(got[0], ref[0] * 2.0 ** k) and torch.equal(got[1], ref[1] * 2.0 ** k)
