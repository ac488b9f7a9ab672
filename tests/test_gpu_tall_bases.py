"""Tall bases of the HSS construction (64-row tiles of a child's part, register
blocks of 16, 32, 64 or 128 columns): H of a Schur complement whose ranks reach
into each block, built by hss_front_compress, against the oracle's construction
of the same S.
"""
import numpy as np
import pytest

import oracle
from paper_1508_07798_gb300 import dg_inputs as dg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,rank", [(16, 1, 1), (17, 1, 14), (16, 2, 17), (19, 2, 31), (24, 2, 33), (23, 3, 62),
                                      (24, 3, 65), (24, 3, 80)])
def test_compressed_front_of_given_rank_matches_oracle(n, p, rank):
    """S = diagonal + a rank-`rank` part whose pivots fall off slowly, so every
    HSS node of at least that size has that rank and no rank decision is near
    the cut: H of the GPU equals the oracle's to 1e-10 (the bar of the step
    tests), in FP32 to 1e-3 (u_32 1e-7 times |T| growth over the tree)."""
    from paper_1508_07798_gb300 import hssnd as hs
    mesh, A = dg.poisson_2d(n, p)
    dA = hs.DeviceBSR.from_host(A)
    tree = hs.nd_order((2, (n, n), p), dA)
    nd = oracle.nd_order(2, mesh.n, p, A.row_ptr, A.col_idx)
    ex = tree.export()
    box = int(np.argmax(ex["nb"]))
    nb = int(ex["nb"][box])
    rng = np.random.default_rng(n * 100 + rank)
    U, V = (np.linalg.qr(rng.standard_normal((nb, rank)))[0] for _ in range(2))
    S = U @ np.diag(np.linspace(2.0, 1.0, rank)) @ V.T
    nodes = oracle.hss_tree_for_front(nd, box)
    for N in nodes:
        if not N["children"]:
            lo, hi = N["lo"], N["hi"]
            S[lo:hi, lo:hi] += np.diag(np.linspace(3.0, 4.0, hi - lo))
    Ho, rep = oracle.hss_compress(S, nodes, 1e-9, 0, box, rmax=96)
    H, k, r, rounds = hs.front_compress(tree, box, S, tol=1e-9)
    assert (k, r) == (max(*rep["krow"].values(), *rep["kcol"].values()), rep["r"])
    assert np.linalg.norm(H - Ho) <= 1e-10 * np.linalg.norm(Ho)
    H32 = hs.front_compress(tree, box, S, tol=1e-5, precision="fp32")[0]
    assert np.linalg.norm(H32 - S) <= 1e-3 * np.linalg.norm(S)
