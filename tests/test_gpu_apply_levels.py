"""hss_apply of one vector: row tiles worked on by one warp up to a cluster of
eight CTAs (fronts of a few dofs up to more than 4,096 columns, where a warp takes
several chunks).  Without compression the factor is a direct solver, so the
residual shows every level's products; FP32 factors are compared with the
several-vector kernels, which sum on their own."""
import numpy as np
import pytest

from paper_1508_07798_gb300 import dg_inputs as dg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("autotune", [0, 1])
@pytest.mark.parametrize("op,n,p", [("poisson", 5, 1), ("poisson", 31, 2), ("diffusion", 9, 1), ("diffusion", 16, 1)])
def test_one_vector_over_every_level_shape(op, n, p, autotune):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    mesh, A = dg.poisson_2d(n, p) if op == "poisson" else dg.diffusion_3d(n, p, 0)
    dA = hs.DeviceBSR.from_host(A)
    tree = hs.nd_order((mesh.dim, mesh.n[:mesh.dim], p), dA)
    b = dg.random_rhs(A.n, 2, 3, kind="normal")
    B = torch.as_tensor(np.asfortranarray(b), device="cuda")
    F = hs.hss_factor(dA, tree, precision="fp64", compress=0, autotune=autotune)
    x = hs.hss_apply(F, B[:, 0].contiguous()).cpu().numpy()
    M = dg.bsr_to_csr(A)
    # backward error of the elimination: n u with room for its growth
    assert np.linalg.norm(M @ x - b[:, 0]) <= 1e-9 * (abs(M).sum(axis=1).max() * np.linalg.norm(x) + np.linalg.norm(b[:, 0]))
    F = hs.hss_factor(dA, tree, precision="fp32", compress=0, autotune=autotune)
    one = hs.hss_apply(F, B[:, 0].contiguous())
    two = hs.hss_apply(F, B)[:, 0]
    assert ((one - two).norm() / two.norm()).item() <= 2e-4   # as for several vectors
