"""Block-end updates as FP16 two-term products (tensor_cores = 3, fronts of at
least 2,048 rows): the eliminated front against FP64, at sizes around the tiles
(128 rows, 256 columns, 32 of K), with odd leading dimensions, with rows and
columns of very different magnitude, and no further from FP64 than the TF32
split (tensor_cores = 1) and FP32 arithmetic (tensor_cores = 0)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _front(n, ni, seed, spread):
    rng = np.random.default_rng(seed)
    F = rng.standard_normal((n, n)) / np.sqrt(n)
    F[np.arange(n), np.arange(n)] += 4.0
    if spread:   # rows and columns over 2^+-spread
        F *= np.exp2(rng.integers(-spread, spread + 1, n).astype(float))[:, None]
        F *= np.exp2(rng.integers(-spread, spread + 1, n).astype(float))[None, :]
    return F.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("n,ni,spread", [(2048, 256, 0), (2049, 257, 0), (2303, 511, 0), (2305, 640, 8), (2560, 1100, 0),
                                         (3001, 700, 20), (2048, 2048, 0), (2200, 128, 0)])
def test_block_updates_no_further_from_fp64_than_fp32(n, ni, spread):
    from paper_1508_07798_gb300 import hssnd as hs
    F = _front(n, ni, n + ni, spread)
    S64 = np.linalg.solve(F[:ni, :ni], F[:ni, ni:]) if ni < n else np.linalg.inv(F)
    ref = F[ni:, ni:] - F[ni:, :ni] @ S64 if ni < n else S64
    err, bytag = {}, {}
    for tc in (0, 1, 3):
        hs.profile_enable(True)
        hs.profile_reset()
        out, perm, rc = hs.front_eliminate(F, ni, "fp32", tensor_cores=tc)
        bytag[tc] = set(hs.profile_read())
        hs.profile_enable(False)
        assert rc == 0
        if ni < n:   # every entry on the scale of what is added up in it
            w = np.abs(F[ni:, ni:]) + np.abs(F[ni:, :ni]) @ np.abs(S64)
            err[tc] = (np.abs(out[ni:, ni:] - ref) / w).max()
        else:
            X = np.zeros_like(out)
            X[:, perm] = out      # out = F^-1 P^t: column j belongs to row perm[j]
            err[tc] = np.abs(X - ref).max() / np.abs(ref).max()
    print(f"\nn {n} ni {ni} spread {spread}: largest error, FP32 {err[0]:.2e}, TF32 split {err[1]:.2e}, FP16 terms {err[3]:.2e}")
    assert ("gemm_h2_split" in bytag[3]) == (ni >= 128) and "gemm_h2_split" not in bytag[1] | bytag[0]
    assert err[3] <= 1.5 * max(err[0], err[1])
