"""hss_spmv: one kernel per block size of p = 1, 2, 3 (2D, 3D), vector loads where
the arrays allow them, a general kernel for the others.  All of them add a
row's products in the order of the several-vector kernel, so one vector has to
give the same bits as the same vector beside another one.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("bs", [1, 4, 5, 8, 9, 16, 25, 27, 64])
def test_spmv_one_vector_equals_one_of_several_bit_for_bit(bs, shift):
    """shift: doubles by which x and the values start past a 16-byte boundary."""
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    rng = np.random.default_rng(bs)
    nb = 37
    pattern = [np.sort(rng.choice(nb, size=rng.integers(0, 7), replace=False)) for _ in range(nb)]
    row_ptr = np.concatenate([[0], np.cumsum([len(c) for c in pattern])]).astype(np.int32)
    col = np.concatenate(pattern).astype(np.int32)
    val = rng.standard_normal(len(col) * bs * bs)
    A = hs.DeviceBSR(nb, bs, row_ptr, col, val)
    buf = torch.zeros(val.size + shift, dtype=torch.float64, device="cuda")
    buf[shift:] = torch.as_tensor(val, device="cuda")
    A.val = buf[shift:]
    A.c.val = A.val.data_ptr()
    N = nb * bs
    X = rng.standard_normal((N, 2))
    xb = torch.zeros(N + shift, dtype=torch.float64, device="cuda")
    xb[shift:] = torch.as_tensor(X[:, 0], device="cuda")
    y1 = hs.hss_spmv(A, xb[shift:]).cpu().numpy()
    y2 = hs.hss_spmv(A, torch.as_tensor(X, device="cuda")).cpu().numpy()
    assert np.array_equal(y1, y2[:, 0])
    dense = np.zeros((N, N))
    for e in range(nb):
        for t in range(row_ptr[e], row_ptr[e + 1]):
            dense[e * bs:(e + 1) * bs, col[t] * bs:(col[t] + 1) * bs] = val[t * bs * bs:(t + 1) * bs * bs].reshape(bs, bs)
    # sums of at most 6 bs products: bs * 6 * u relative to |A| |x|
    bound = 6 * bs * np.finfo(float).eps * (np.abs(dense) @ np.abs(X[:, 0])) + 1e-300
    assert np.all(np.abs(y1 - dense @ X[:, 0]) <= bound)
