"""hss_apply of several vectors costs no more than the vectors one at a time: over
small and large fronts, both precisions (FP64 is bound by a pipe of two products
per clock and SM, so a level has to be spread over all of them)."""
import pytest

from paper_1508_07798_gb300 import dg_inputs as dg

pytestmark = pytest.mark.gpu


def _time(fn):
    import torch
    for _ in range(3):
        fn()
    best = float("inf")
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / 5)
    return best


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("op,n,p", [("poisson", 16, 1), ("poisson", 16, 3), ("poisson", 32, 2), ("poisson", 64, 2),
                                    ("diffusion", 12, 1), ("diffusion", 16, 1)])
def test_several_vectors_cost_no_more_than_one_at_a_time(op, n, p, precision):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    mesh, A = dg.poisson_2d(n, p) if op == "poisson" else dg.diffusion_3d(n, p, 0)
    dA = hs.DeviceBSR.from_host(A)
    F = hs.hss_factor(dA, hs.nd_order((mesh.dim, mesh.n[:mesh.dim], p), dA), tol=1e-6, precision=precision)
    X = torch.as_tensor(dg.random_rhs(A.n, 20, 5, kind="normal"), device="cuda")
    x = X[:, 0].contiguous()
    one = _time(lambda: hs.hss_apply(F, x))
    for k in (2, 3, 8, 20):
        Xk = X[:, :k]
        # (a tenth for the spread of the timings)
        assert _time(lambda: hs.hss_apply(F, Xk)) <= 1.1 * k * one, k
