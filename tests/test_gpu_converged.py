"""A solve that starts converged queues at most one masked iteration before the host sees
that no system is active."""
import pytest
import torch

import workloads as wl
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "bf16_hilo"])
@pytest.mark.parametrize("precond", [False, True])
def test_converged_start_queues_one_iteration(kmv_handle, precond, prec):
    w = wl.ragged([300, 129], d=2, chains=2, m=1, seed=9500, sigma2=0.1)
    pts, theta, _, _ = to_dev(w)
    y = torch.zeros(w.n_total, device="cuda")
    if precond:
        om = torch.randn(w.chains, w.n_total, 16, device="cuda")
        U, lam, _ = kmv_handle.nystrom_build(pts, theta, om)
        kmv_handle.set_preconditioner(pts, U, lam)
    kmv_handle.profile_enable()
    try:
        kmv_handle.profile_read(0)
        x, st, it = kmv_handle.kmv_cg_solve(pts, theta, y, tol=1e-6, maxiter=100, prec=prec)
        torch.cuda.synchronize()
        launches = kmv_handle.profile_read(0)[1]
    finally:
        kmv_handle.profile_enable(False)
        kmv_handle.set_preconditioner(pts)
    assert torch.all(st == 0) and torch.all(it == 0) and torch.all(x == 0)
    assert launches <= 1
