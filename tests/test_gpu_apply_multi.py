"""hss_apply of several vectors (tiles of 128 rows, blocks of 8, 16 or 32 vectors,
512-column items) against one vector at a time, which has its own kernel: sizes
with and without 16-byte columns, fronts below one tile and above one item,
subtree levels, every block width and its remainders, strided output."""
import numpy as np
import pytest

from paper_1508_07798_gb300 import dg_inputs as dg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("op,n,p,compress", [("poisson", 7, 2, 1), ("poisson", 20, 1, 1), ("poisson", 33, 2, 1),
                                             ("poisson", 40, 3, 1), ("diffusion", 9, 1, 1), ("poisson", 24, 2, 0),
                                             ("diffusion", 12, 1, 0)])
def test_several_vectors_equal_one_at_a_time(op, n, p, compress, precision):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    mesh, A = dg.poisson_2d(n, p) if op == "poisson" else dg.diffusion_3d(n, p, 0)
    dA = hs.DeviceBSR.from_host(A)
    F = hs.hss_factor(dA, hs.nd_order((mesh.dim, mesh.n[:mesh.dim], p), dA), tol=1e-6, precision=precision,
                      compress=compress)
    X = torch.as_tensor(dg.random_rhs(A.n, 41, 5, kind="normal"), device="cuda")
    one = torch.stack([hs.hss_apply(F, X[:, k].contiguous()) for k in range(41)], dim=1)
    # sums of up to 3,000 products in another order, through up to 10 levels
    tol = 1e-12 if precision == "fp64" else 2e-4
    for k in (2, 3, 7, 8, 9, 16, 17, 20, 31, 32, 33, 41):
        Y = hs.hss_apply(F, X[:, :k])
        err = ((Y - one[:, :k]).norm(dim=0) / one[:, :k].norm(dim=0)).max().item()
        assert err <= tol, (k, err)
    # in place, with a leading dimension beyond the vectors
    ld = A.n + 37
    buf = torch.full((11, ld), 7.0, dtype=torch.float64, device="cuda")
    buf[:, :A.n] = X[:, :11].t()
    hs.hss_apply_raw(F, 11, buf, buf, ld)
    assert ((buf[:, :A.n].t() - one[:, :11]).norm() / one[:, :11].norm()).item() <= tol
    assert torch.all(buf[:, A.n:] == 7.0)
