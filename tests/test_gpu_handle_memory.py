"""The device memory of factors and trees: giving handles up in one thread leaves a
stream capture of another thread alone, and their memory is not handed to a later
handle while kernels still use it."""
import threading

import pytest

from paper_1508_07798_gb300 import dg_inputs as dg

pytestmark = pytest.mark.gpu


def _handles(n=8, applied=False, solved=False):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    mesh, A = dg.poisson_2d(n, 1)
    dA = hs.DeviceBSR.from_host(A)
    tree = hs.nd_order((2, mesh.n[:2], 1), dA)
    F = hs.hss_factor(dA, tree)
    b = torch.ones(A.n, dtype=torch.float64, device="cuda")
    if applied:
        hs.hss_apply(F, b)
    if solved:
        hs.fgmres_solve(dA, F, b)
        hs.fgmres_solve(dA, F, torch.stack([b, 2 * b], dim=1))
    return [F, tree]


@pytest.mark.parametrize("kw", [{}, {"applied": True}, {"solved": True}])
def test_destroying_handles_leaves_other_threads_captures_alone(kw):
    import torch
    box = _handles(**kw)
    x = torch.ones(1024, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=torch.cuda.Stream(), capture_error_mode="thread_local"):
        y = x * 2
        t = threading.Thread(target=box.clear)
        t.start()
        t.join()
        z = y + 1
    g.replay()
    torch.cuda.synchronize()
    assert torch.all(z == 3)


def test_memory_of_a_destroyed_factor_is_not_reused_under_its_apply():
    """An apply is still queued behind other work when its factor and tree are given
    up and other factorizations take memory on another stream."""
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    mesh, A = dg.poisson_2d(32, 2)
    dA = hs.DeviceBSR.from_host(A)
    desc = (2, mesh.n[:2], 2)
    b = torch.ones(A.n, dtype=torch.float64, device="cuda")

    def factor():
        tree = hs.nd_order(desc, dA)
        return hs.hss_factor(dA, tree)

    ref = hs.hss_apply(factor(), b)
    mesh2, A2 = dg.helmholtz_2d(32, 2, 1)
    dA2 = hs.DeviceBSR.from_host(A2)
    big = torch.randn(6000, 6000, device="cuda")
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    F = factor()
    with torch.cuda.stream(s1):
        for _ in range(20):
            big = torch.tanh(big @ big)
        y = hs.hss_apply(F, b)
    del F
    with torch.cuda.stream(s2):
        for _ in range(3):
            hs.hss_factor(dA2, hs.nd_order((2, mesh2.n[:2], 2), dA2))
    torch.cuda.synchronize()
    assert torch.equal(y, ref)


def test_cached_memory_can_be_given_back_and_small_handles_leave_large_chunks():
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    mesh, A = dg.diffusion_3d(12, 1, 0)
    dA = hs.DeviceBSR.from_host(A)
    tree = hs.nd_order((mesh.dim, mesh.n[:mesh.dim], 1), dA)
    hs.cache_trim()
    free0 = torch.cuda.mem_get_info()[0]
    F = hs.hss_factor(dA, tree, precision="fp64")
    large = F.info()["factor_bytes"]
    del F
    # half its size: the FP32 factor must not sit on the FP64 one's memory
    F = hs.hss_factor(dA, tree, precision="fp32")
    assert hs.cache_trim() >= large
    del F
    assert hs.cache_trim() > 0 and hs.cache_trim() == 0
    assert torch.cuda.mem_get_info()[0] >= free0 - (64 << 20)   # (modules loaded meanwhile)
