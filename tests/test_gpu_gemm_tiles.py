"""The SIMT GEMM's tiles (32 x 32 and 64 x 64, K in chunks of 16) at their edges,
through hss_gemm_f32 (engine 0) and through one elimination step in both
precisions, whose updates mask rows and columns."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (31, 33, 15), (32, 32, 16), (33, 31, 17), (64, 64, 32), (65, 63, 33),
                                   (129, 1, 100), (1, 200, 48), (700, 900, 31), (3000, 2900, 33)])
def test_gemm_f32_simt_tiles(m, n, k):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    A = torch.randn(m, k, device="cuda", generator=g)
    B = torch.randn(k, n, device="cuda", generator=g)
    C = torch.randn(m, n, device="cuda", generator=g)
    ref = 0.5 * (A.double() @ B.double()) - 2.0 * C.double()
    out = hs.gemm_f32(A, B, C.clone(), alpha=0.5, beta=-2.0, engine=0)
    # k products and a sum, each rounded once: (k + 3) u relative to the terms
    bound = (k + 3) * 6e-8 * (0.5 * A.abs().double() @ B.abs().double() + 2.0 * C.abs().double())
    assert torch.all((out.double() - ref).abs() <= bound + 1e-30)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("fp32", 5e-4)])
@pytest.mark.parametrize("n,ni", [(5, 3), (33, 32), (97, 31), (130, 65), (321, 100), (1000, 40)])
def test_masked_updates_of_an_elimination(n, ni, precision, tol):
    from paper_1508_07798_gb300 import hssnd as hs
    rng = np.random.default_rng(n)
    F = rng.standard_normal((n, n)) / np.sqrt(n)
    F[np.arange(n), np.arange(n)] += 3.0
    out, perm, rc = hs.front_eliminate(F, ni, precision)
    assert rc == 0
    W = np.linalg.solve(F[:ni, :ni], F[:ni, ni:])
    S = F[ni:, ni:] - F[ni:, :ni] @ W
    assert np.abs(out[:ni, ni:] - W).max() <= tol and np.abs(out[ni:, ni:] - S).max() <= tol
