"""Width of the pivot blocks of a blocked sweep (fronts of 2,048 rows and more) in
FP32.  A block update multiplies by the explicit inverse of the block's pivot rows,
and its rounding grows with the block's width: fronts of 1,537 to 6,144 interior
dofs take 128 (to 3,072) or 64 pivots per block although their panels have 32
columns, with the tensor-core updates (tensor_cores = 3) 128; smaller and larger
ones 256.  Checked by the number of block ends, and W and S against FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ni,tc,width", [(2100, 1536, 0, 256), (2100, 1537, 0, 128), (2300, 1600, 3, 128),
                                           (3300, 3072, 0, 128), (3400, 3073, 0, 64), (3400, 3200, 3, 128)])
def test_pivots_per_block(n, ni, tc, width):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    rng = np.random.default_rng(n + ni)
    F = rng.standard_normal((n, n)) / np.sqrt(n)
    F[np.arange(n), np.arange(n)] += 4.0
    F = F.astype(np.float32).astype(np.float64)
    hs.profile_enable(True)
    hs.profile_reset()
    out, perm, rc = hs.front_eliminate(F, ni, "fp32", tensor_cores=tc)
    launches = {k: v[1] for k, v in hs.profile_read().items()}
    hs.profile_enable(False)
    assert rc == 0
    # one launch after every panel of 32 columns and one at the end of every block
    assert launches["gj_post_f32"] == -(-ni // 32) + -(-ni // width)
    Fd, o = torch.as_tensor(F, device="cuda"), torch.as_tensor(out, device="cuda")
    W = torch.linalg.solve(Fd[:ni, :ni], Fd[:ni, ni:])
    S = Fd[ni:, ni:] - Fd[ni:, :ni] @ W
    # FP32's unit (6e-8) times the condition (about 2) and a sum of ni products' growth
    assert (o[:ni, ni:] - W).norm() <= 1e-5 * W.norm() and (o[ni:, ni:] - S).norm() <= 1e-5 * S.norm()
