"""The FP32 product and adjoint of points with more than 32 dimensions: parity at the edges of its
dimension classes (48, 64) and column widths (16, 32), and the time of wide V."""
import numpy as np
import pytest
import torch

import workloads as wl
from helpers import abs_row_products, componentwise_err, f32, to_dev
from oracle import se_kernel as sk
from test_gpu_kmv import TOL, _check_backward, _check_forward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 16, 17, 33, 65])
@pytest.mark.parametrize("sizes,d", [([1, 127, 129], 33), ([513], 48), ([64, 300], 49), ([257], 64)])
def test_forward_of_small_sets(kmv_handle, sizes, d, m):
    _check_forward(kmv_handle, wl.ragged(sizes, d=d, chains=2, m=m, seed=9700 + d + m, ell_range=(1.0, 4.0)), "fp32")


# 4 chains of 4,609 rows fill the chip: the wide chunks, and several folds per unit
@pytest.mark.parametrize("d,m", [(33, 17), (48, 64), (49, 32), (64, 65)])
def test_forward_of_large_sets(kmv_handle, d, m):
    n = 4609
    w = wl.ragged([n], d=d, chains=4, m=m, seed=9800 + d, ell_range=(1.0, 4.0))
    pts, theta, V, _ = to_dev(w)
    Y = kmv_handle.kmv_forward(pts, theta, V, prec="fp32").cpu().numpy()
    X, Vh, rows = f32(w.X), f32(w.V), np.r_[0:3, 509:515, n - 3:n]
    for c in (0, 3):
        ref = sk.kmv(X, w.theta[c], Vh[c], True, rows=rows)
        scale = abs_row_products(X, w.theta[c], Vh[c], True, rows)
        assert componentwise_err(Y[c, rows], ref, scale) <= TOL["fp32"][0]


# 1,100 rows: sums over several folds, kept in local memory
@pytest.mark.parametrize("prec", ["fp32", "bf16_hilo"])
@pytest.mark.parametrize("d,m", [(33, 2), (33, 40), (48, 17), (64, 5)])
def test_adjoint(kmv_handle, d, m, prec):
    _check_backward(kmv_handle, wl.ragged([1100, 65], d=d, chains=1, m=m, seed=9850 + d + m, ell_range=(1.0, 4.0)), prec)


def test_many_dimensions_keep_the_wide_chunks(kmv_handle):
    # Per pair 2 d operations for the distance and one per column: 40 dimensions (computed
    # as 48) and 64 columns take (2 * 48 + 64) / (2 * 32 + 64) = 1.25 times as long as 32;
    # with the distance formed for every 16 columns, padded to 64, 3.8 times
    def ms(d):
        w = wl.ragged([9001], d=d, chains=1, m=64, seed=9900, ell_range=(1.0, 4.0))
        pts, theta, V, _ = to_dev(w)
        best = 1e9
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                kmv_handle.kmv_forward(pts, theta, V, prec="fp32")
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    assert ms(40) <= 2.0 * ms(32)
