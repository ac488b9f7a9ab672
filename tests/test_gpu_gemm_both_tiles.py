"""Both tiles of the FP32 SIMT GEMM (hss_gemm_f32 and hss_gemm_f32_static: 32 x 32
below 1,000 tiles of 64, else 64 x 64) at the edges of the tiles and of the
three-stage ring of K chunks of 16.  Both add the products in order of K, so they
agree bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


def _data(m, n, k):
    import torch
    g = torch.Generator(device="cuda").manual_seed(m * n + k)
    A = torch.randn(m, k, device="cuda", generator=g)
    B = torch.randn(k, n, device="cuda", generator=g)
    C = torch.randn(m, n, device="cuda", generator=g)
    ref = 0.5 * (A.double() @ B.double()) - 2.0 * C.double()
    # k products and a sum, each rounded once: (k + 3) u relative to the terms
    bound = (k + 3) * 6e-8 * (0.5 * A.abs().double() @ B.abs().double() + 2.0 * C.abs().double()) + 1e-30
    return A, B, C, ref, bound


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (31, 33, 15), (32, 32, 16), (33, 31, 17), (63, 65, 31), (64, 64, 32),
                                   (65, 63, 33), (95, 97, 47), (96, 96, 48), (97, 95, 49), (200, 7, 64), (7, 200, 65)])
def test_small_tile_at_its_edges(m, n, k):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    A, B, C, ref, bound = _data(m, n, k)
    out = hs.gemm_f32(A, B, C.clone(), alpha=0.5, beta=-2.0, engine=0)
    fixed = C.clone()
    hs.gemm_f32_static(A, B, fixed, alpha=0.5, beta=-2.0, engine=0)
    assert torch.all((out.double() - ref).abs() <= bound)
    assert torch.equal(out, fixed)


@pytest.mark.parametrize("k", [1, 15, 16, 17, 31, 32, 33, 47, 48, 49])
def test_large_tile_at_its_edges_with_the_sums_of_the_small_one(k):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    A, B, C, ref, bound = _data(2881, 2945, k)   # 46 x 47 tiles of 64, one row and one column over
    out = hs.gemm_f32(A, B, C.clone(), alpha=0.5, beta=-2.0, engine=0)
    fixed = C.clone()
    hs.gemm_f32_static(A, B, fixed, alpha=0.5, beta=-2.0, engine=0)
    assert torch.all((out.double() - ref).abs() <= bound)
    assert torch.equal(out, fixed)
    part = hs.gemm_f32(A[2000:].contiguous(), B, C[2000:].clone(), alpha=0.5, beta=-2.0, engine=0)   # 14 x 47: the small one
    assert torch.equal(out[2000:], part)
