"""FP32 products at the ends of FP32's range: the sums over more than 512 columns are kept
in FP64, so an infinite entry of V (or G) gives infinite sums where every kernel entry is
positive, not NaN, and sums above FP32's largest value are exact until they are scaled by
alpha and rounded."""
import numpy as np
import pytest
import torch

from oracle import se_kernel as sk
from helpers import f32
from test_gpu_kmv import TOL

pytestmark = pytest.mark.gpu

# 1,100 rows: one row a thread, sums of several units by the last CTA (m <= 2) or by a
# kernel of their own; 4 chains of 4,609: several rows a thread, several folds per unit
SHAPES = [(1100, 1, 1, 1), (1100, 1, 3, 2), (1100, 1, 2, 5), (4609, 4, 1, 1), (4609, 4, 3, 2), (4609, 4, 8, 16),
          (4609, 4, 40, 3)]


def _inputs(n, chains, d, log_alpha, seed):
    from paper_2412_20884_gb300 import Points
    rng = np.random.default_rng(seed)
    X = 0.5 * rng.random((n, d)) / np.sqrt(d)          # |x_i - x_j| <= 0.5, l = 1: K0 >= 0.88
    th = np.tile(np.concatenate([[log_alpha], np.zeros(d), [np.log(1e-3)]]), (chains, 1))
    pts = Points(torch.tensor(X, dtype=torch.float32, device="cuda"), [0, n], ard=True)
    return rng, f32(X), th, pts, torch.tensor(th, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n,chains,d,m", SHAPES)
def test_infinite_entries_give_infinite_sums(kmv_handle, n, chains, d, m):
    rng, _, _, pts, theta = _inputs(n, chains, d, 0.0, 7000 + m)
    V = torch.tensor(0.1 + rng.random((chains, n, m)), dtype=torch.float32, device="cuda")
    V[0, n // 3, 0] = float("inf")
    Y = kmv_handle.kmv_forward(pts, theta, V, prec="fp32")
    assert torch.all(Y[0, :, 0] == float("inf"))
    Y[0, :, 0] = 0.0
    assert torch.all(torch.isfinite(Y))
    G, V = V, torch.tensor(0.1 + rng.random((chains, n, m)), dtype=torch.float32, device="cuda")
    gth, gV = kmv_handle.kmv_backward(pts, theta, V, G, prec="fp32")
    # (dL/dtheta of that system is NaN: its W = G V^T holds infinity times the padding's zeros)
    assert torch.all(gV[0, :, 0] == float("inf"))
    gV[0, :, 0] = 0.0
    assert torch.all(torch.isfinite(gV)) and torch.all(torch.isfinite(gth[1:]))


@pytest.mark.parametrize("n,chains,d,m", SHAPES)
def test_sums_above_fp32_range(kmv_handle, n, chains, d, m):
    # 512 columns of 5e35 stay below FP32's 3.4e38, all of them do not; alpha = e^-7 brings
    # the result back
    rng, X, th, pts, theta = _inputs(n, chains, d, -7.0, 7100 + m)
    Vh = f32(5e35 * (0.9 + 0.1 * rng.random((chains, n, m))))
    V = torch.tensor(Vh, dtype=torch.float32, device="cuda")
    assert Vh[0, :, 0].sum() > 3.5e38
    rows = np.r_[0:4, n - 4:n]
    ref = sk.kmv(X, th[0], Vh[0], True, rows=rows)
    Y = kmv_handle.kmv_forward(pts, theta, V, prec="fp32")[0, rows].cpu().numpy()
    assert np.max(np.abs(Y - ref) / ref) <= TOL["fp32"][0]
    one = torch.full_like(V, 1e-35)
    gV = kmv_handle.kmv_backward(pts, theta, one, V, prec="fp32")[1][0, rows].cpu().numpy()
    assert np.max(np.abs(gV - ref) / ref) <= TOL["fp32"][0]


def test_infinite_entries_in_the_wide_tensor_core_form(kmv_handle):
    # 20 columns, 8 chains of 20,000 rows: items of more than 32 J tiles, whose sums over
    # 4096 columns are folded several times; K0 >= 0.88 keeps every probability positive
    n, chains, m = 20000, 8, 20
    rng, _, _, pts, theta = _inputs(n, chains, 3, 0.0, 7200)
    V = torch.tensor(0.1 + rng.random((chains, n, m)), dtype=torch.float32, device="cuda")
    V[0, n // 3, 0] = float("inf")
    Y = kmv_handle.kmv_forward(pts, theta, V, prec="bf16_hilo")
    assert torch.all(Y[0, :, 0] == float("inf"))
    Y[0, :, 0] = 0.0
    assert torch.all(torch.isfinite(Y))
