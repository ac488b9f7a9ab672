"""A failed device allocation in hss_apply leaves a factor that the next call
can use: every allocation of the first apply to several vectors fails once."""
import numpy as np
import pytest

from paper_1508_07798_gb300 import dg_inputs as dg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_apply_after_a_failed_allocation(precision):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    mesh, A = dg.diffusion_3d(12, 1, 0)   # fronts whose row tiles are split over several items
    dA = hs.DeviceBSR.from_host(A)
    tree = hs.nd_order((mesh.dim, mesh.n[:mesh.dim], 1), dA)
    X = torch.as_tensor(np.asfortranarray(dg.random_rhs(A.n, 20, 1, kind="normal")), device="cuda")
    ref = hs.hss_apply(hs.hss_factor(dA, tree, precision=precision), X)
    failures = 0
    for nth in range(1, 12):
        F = hs.hss_factor(dA, tree, precision=precision)
        hs.alloc_fail_next(nth)
        try:
            hs.hss_apply(F, X)
        except hs.HssError as e:
            assert e.code == hs.HSS_ENOMEM
            failures += 1
        finally:
            hs.alloc_fail_next(0)
        assert torch.equal(hs.hss_apply(F, X), ref), nth
    assert failures >= 2   # the sweep's vectors and parameters at least
