"""Device memory of the FP32 products: what a handle holds is what workspace_bytes reports,
a call with one work unit per row needs no scratch whatever its size, and a captured call
that has none takes the plan without."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _inputs(rows, n_inst, chains, d, m, seed=8000):
    from paper_2412_20884_gb300 import Points
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = rows * n_inst
    pts = Points(torch.rand(n, d, device="cuda", generator=g), np.arange(n_inst + 1) * rows, ard=True)
    theta = torch.zeros(n_inst * chains, d + 2, dtype=torch.float64, device="cuda")
    V = torch.randn(chains, n, m, device="cuda", generator=g)
    G = torch.randn(chains, n, m, device="cuda", generator=g)
    return pts, theta, V, G


# 20,000 rows are split into units of several hundred columns (sums in scratch); 1,500
# instances of 800 rows have a unit per row, whose sums would be 614 MB at m = 64.  16 MB:
# the granularity of the handle's allocations.
@pytest.mark.parametrize("rows,n_inst,d,m,most", [(20000, 1, 8, 16, None), (800, 1500, 3, 64, 64 << 20)])
def test_memory_held_is_reported_and_bounded(rows, n_inst, d, m, most):
    from paper_2412_20884_gb300 import Kmv
    pts, theta, V, G = _inputs(rows, n_inst, 1, d, m)
    Y, gV, gth = torch.empty_like(V), torch.empty_like(V), torch.empty_like(theta)

    def calls(h):
        h.kmv_forward(pts, theta, V, Y=Y, prec="fp32")
        h.kmv_backward(pts, theta, V, G, grad_theta=gth, grad_V=gV, prec="fp32")
        torch.cuda.synchronize()

    h = Kmv(0)   # loads the kernels
    calls(h)
    h.close()
    h = Kmv(0)
    before = torch.cuda.mem_get_info()[0]
    calls(h)
    held, reported = before - torch.cuda.mem_get_info()[0], h.workspace_bytes()
    h.close()
    assert held <= reported + (16 << 20)
    assert reported <= (most or 1 << 30)


@pytest.mark.parametrize("adjoint", [False, True])
def test_capture_without_prepared_scratch(adjoint):
    from paper_2412_20884_gb300 import Kmv
    # 400 items of 128 rows: one chunk of columns, split into units only with scratch
    pts, theta, V, G = _inputs(1200, 10, 4, 3, 5)
    h = Kmv(0)

    def call(prec):
        if adjoint:
            return h.kmv_backward(pts, theta, V, G, prec=prec)
        return (h.kmv_forward(pts, theta, V, prec=prec),)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):   # layout and workspace, not the FP32 scratch
        call("bf16_hilo")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = call("fp32")
    graph.replay()
    torch.cuda.synchronize()
    got = [t.clone() for t in got]
    want = call("fp32")
    torch.cuda.synchronize()
    h.close()
    # the same FP32 sums of 512 columns, added in FP64 in another order
    for a, b in zip(got, want):
        assert float((a - b).abs().max()) <= 2.0 ** -23 * float(b.abs().max())
