"""Both tiles of the FP32 SIMT GEMM (32 x 32: hss_gemm_f32 below 2,000 tiles of 64,
as the launches of a factorization; 64 x 64: hss_gemm_f32_static, and hss_gemm_f32
above) at the edges of the tiles and of the three-stage ring of K chunks of 16.
Both add the products in order of K, so they agree bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (31, 33, 15), (32, 32, 16), (33, 31, 17), (63, 65, 31), (64, 64, 32),
                                   (65, 63, 33), (95, 97, 47), (96, 96, 48), (97, 95, 49), (200, 7, 64), (7, 200, 65)])
def test_both_tiles_at_their_edges(m, n, k):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    g = torch.Generator(device="cuda").manual_seed(m * n + k)
    A = torch.randn(m, k, device="cuda", generator=g)
    B = torch.randn(k, n, device="cuda", generator=g)
    C = torch.randn(m, n, device="cuda", generator=g)
    ref = 0.5 * (A.double() @ B.double()) - 2.0 * C.double()
    # k products and a sum, each rounded once: (k + 3) u relative to the terms
    bound = (k + 3) * 6e-8 * (0.5 * A.abs().double() @ B.abs().double() + 2.0 * C.abs().double()) + 1e-30
    small = hs.gemm_f32(A, B, C.clone(), alpha=0.5, beta=-2.0, engine=0)
    large = C.clone()
    hs.gemm_f32_static(A, B, large, alpha=0.5, beta=-2.0, engine=0)
    assert torch.all((small.double() - ref).abs() <= bound)
    assert torch.equal(small.cpu(), large.cpu())


@pytest.mark.parametrize("k", [15, 49])
def test_large_launch_takes_the_large_tile_with_the_same_sums(k):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    m, n = 2881, 2945   # 46 x 47 tiles of 64, ragged on both sides
    g = torch.Generator(device="cuda").manual_seed(k)
    A = torch.randn(m, k, device="cuda", generator=g)
    B = torch.randn(k, n, device="cuda", generator=g)
    C = torch.randn(m, n, device="cuda", generator=g)
    whole = hs.gemm_f32(A, B, C.clone(), engine=0)
    part = hs.gemm_f32(A[:1000].contiguous(), B, C[:1000].clone(), engine=0)
    assert torch.equal(whole[:1000].cpu(), part.cpu())
