"""The forms of the ID kernel at the edges of their ranges: sample widths around
32, 64 and 96 (registers per lane), leaf and parent nodes around 64, 128 and
192 columns (threads per node), the general form beyond, and sampling rounds
that are abandoned because a node ran short of samples.  S has a low-rank part
with slowly falling pivots, so no rank decision is near the cut: the FP32 ranks,
widths and rounds equal the FP64 oracle's."""
import numpy as np
import pytest

import oracle
from paper_1508_07798_gb300 import dg_inputs as dg

pytestmark = pytest.mark.gpu


def _front(n, p, leaf_max, rank):
    from paper_1508_07798_gb300 import hssnd as hs
    mesh, A = dg.poisson_2d(n, p)
    tree = hs.nd_order((2, (n, n), p), hs.DeviceBSR.from_host(A), leaf_max=leaf_max)
    nd = oracle.nd_order(2, mesh.n, p, A.row_ptr, A.col_idx, leaf_max=leaf_max)
    box = int(np.argmax(tree.export()["nb"]))
    nb = int(tree.export()["nb"][box])
    rng = np.random.default_rng(n * 100 + rank)
    U, V = (np.linalg.qr(rng.standard_normal((nb, rank)))[0] for _ in range(2))
    S = U @ np.diag(np.linspace(2.0, 1.0, rank)) @ V.T
    nodes = oracle.hss_tree_for_front(nd, box)
    for N in nodes:
        if not N["children"]:
            S[N["lo"]:N["hi"], N["lo"]:N["hi"]] += np.diag(np.linspace(3.0, 4.0, N["hi"] - N["lo"]))
    return hs, tree, box, nodes, S


@pytest.mark.parametrize("n,p,leaf_max,rank,r0,dr", [
    (16, 2, 64, 9, 24, 32), (16, 2, 64, 21, 32, 32), (16, 2, 64, 22, 33, 32), (24, 3, 64, 30, 40, 8),
    (24, 3, 64, 53, 64, 32), (24, 3, 64, 53, 65, 32), (24, 3, 64, 85, 96, 32), (24, 3, 64, 85, 97, 31),
    (24, 3, 64, 100, 128, 32), (24, 3, 128, 40, 64, 32), (24, 3, 256, 60, 96, 32), (24, 3, 600, 60, 96, 32),
    (24, 3, 64, 70, 8, 8), (24, 2, 64, 40, 32, 32),
])
def test_id_form_matches_oracle(n, p, leaf_max, rank, r0, dr):
    hs, tree, box, nodes, S = _front(n, p, leaf_max, rank)
    rmax = max(96, r0)
    Ho, rep = oracle.hss_compress(S, nodes, 1e-4, 0, box, r0=r0, dr=dr, rmax=rmax)
    H, k, r, rounds = hs.front_compress(tree, box, S, tol=1e-4, precision="fp32", r0=r0, dr=dr, rmax=rmax)
    assert (k, r, rounds) == (max(*rep["krow"].values(), *rep["kcol"].values()), rep["r"], rep["rounds"])
    # u_32 (6e-8) times the growth of the nested |T| <= 2 bases (ranks to 100, depth to 6) stays below 1e-3
    assert np.linalg.norm(H - Ho) <= 1e-3 * np.linalg.norm(Ho)
