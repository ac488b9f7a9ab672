"""The Gram-Schmidt kernels of one right-hand side against the oracle's GMRES:
sizes around a block of 256 rows, one block per CTA (152 x 256 rows), two
(304 x 256) and more; 31 Arnoldi steps pass through every width of the kernels
(4, 8, 16, 32 basis vectors), short restarts through the restart path.
"""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle

pytestmark = pytest.mark.gpu


def _system(n, bs=5):
    nb = n // bs
    rng = np.random.default_rng(n)
    off = [o for o in (0, 1, 7) if o < nb]
    col = np.sort(np.stack([(np.arange(nb) + o) % nb for o in off], 1), axis=1)
    val = rng.uniform(-0.5, 0.5, (nb, len(off), bs, bs)) / bs
    for e in range(nb):
        val[e, list(col[e]).index(e)] += np.eye(bs)
    row_ptr = (len(off) * np.arange(nb + 1)).astype(np.int32)
    M = sp.bsr_matrix((val.reshape(-1, bs, bs), col.ravel(), row_ptr), shape=(n, n)).tocsr()
    return row_ptr, col.ravel().astype(np.int32), np.ascontiguousarray(val.reshape(-1)), M, rng.standard_normal(n)


@pytest.mark.parametrize("n,restart,maxit", [(5, 3, 3), (255, 31, 31), (260, 4, 10), (38910, 31, 31), (38915, 5, 12),
                                             (77820, 17, 20), (77825, 31, 31), (120005, 9, 20)])
def test_history_and_solution_match_the_oracle(n, restart, maxit):
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    row_ptr, col, val, M, b = _system(n)
    A = hs.DeviceBSR(n // 5, 5, row_ptr, col, val)
    xo, info = oracle.fgmres(lambda v: M @ v, None, b, restart=restart, rtol=1e-30, maxit=maxit)
    x, st = hs.fgmres_solve(A, None, torch.as_tensor(b, device="cuda"), restart=restart, rtol=1e-30, maxit=maxit)
    h = hs.fgmres_history(0)
    assert len(h) == len(info["hist"]) == st.iters == maxit
    # estimates relative to ||b||: 31 steps, each with rounding of a few hundred u at
    # the condition number (< 10) of these matrices
    assert np.abs(h - np.array(info["hist"])).max() <= 1e-12
    assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-11 * np.linalg.norm(xo)


def test_zero_right_hand_side_and_converged_start():
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    row_ptr, col, val, M, b = _system(500)
    A = hs.DeviceBSR(100, 5, row_ptr, col, val)
    x0 = torch.as_tensor(b, device="cuda")
    x, st = hs.fgmres_solve(A, None, torch.zeros_like(x0), x0=x0.clone(), rtol=1e-10)   # (the solve writes into x0)
    assert st.converged and st.iters == 0 and st.relres == 0.0 and not x.any()
    rhs = torch.as_tensor(M @ b, device="cuda")
    x, st = hs.fgmres_solve(A, None, rhs, x0=x0.clone(), rtol=1e-10)
    assert st.converged and st.iters == 0 and torch.equal(x, x0)
