"""Block updates as three-term BF16 products (tensor_cores = 3) of fronts whose
rows differ in scale by up to 2^40 inside one block of pivots: one block of 256 or
128 pivots (row pivoting sorts rows by magnitude over several blocks, which
narrows a block's range), sizes with and without 16-byte columns.  A value's
accuracy must not depend on the scale of its row or of its contraction index."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spread", [12, 20])
@pytest.mark.parametrize("n,ni", [(2304, 256), (2305, 256), (2600, 128), (4096, 256)])
def test_rows_of_different_scale_inside_one_block(n, ni, spread):
    from paper_1508_07798_gb300 import hssnd as hs
    rng = np.random.default_rng(n + ni + spread)
    F = rng.standard_normal((n, n)) / np.sqrt(n)
    F[np.arange(n), np.arange(n)] += 4.0
    F *= np.exp2(rng.integers(-spread, spread + 1, n).astype(float))[:, None]
    F = F.astype(np.float32).astype(np.float64)
    W = np.linalg.solve(F[:ni, :ni], F[:ni, ni:])
    ref = F[ni:, ni:] - F[ni:, :ni] @ W
    w = np.abs(F[ni:, ni:]) + np.abs(F[ni:, :ni]) @ np.abs(W)
    err = {}
    for tc in (0, 1, 3):
        hs.profile_enable(True)
        hs.profile_reset()
        out, perm, rc = hs.front_eliminate(F, ni, "fp32", tensor_cores=tc)
        tags = set(hs.profile_read())
        hs.profile_enable(False)
        assert rc == 0 and ("gemm_h2_split" in tags) == (tc == 3)
        err[tc] = (np.abs(out[ni:, ni:] - ref) / w).max()
    print(f"\nn {n} ni {ni} spread {spread}: FP32 {err[0]:.2e}, TF32 split {err[1]:.2e}, BF16 terms {err[3]:.2e}")
    assert err[3] <= 1.5 * max(err[0], err[1])   # the bound of the other block updates
