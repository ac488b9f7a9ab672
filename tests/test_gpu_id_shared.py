"""Shared memory of an ID launch: fronts of one level whose widths differ (r_init).
One has few samples of many columns, one many samples of few; either fits the
kernel's 220 KB, the largest width times the largest column count does not."""
import numpy as np
import pytest

import oracle
from paper_1508_07798_gb300 import dg_inputs as dg

pytestmark = pytest.mark.gpu

WIDE, LEAF = 128, 256


def _smem(r, m):   # bytes of an FP64 node's samples: odd multiples of 16 bytes per column
    lda = 2 * ((r + 1) // 2 | 1)
    return 8 * (lda * m + r + m) + 4 * m + 16


def _columns(nodes, r):
    """Depth and columns of every node but the root."""
    depth, m, k = [0] * len(nodes), [0] * len(nodes), [0] * len(nodes)
    for i in reversed(range(len(nodes))):
        for c in nodes[i]["children"]:
            depth[c] = depth[i] + 1
    for i, N in enumerate(nodes):
        ch = N["children"]
        m[i] = k[ch[0]] + k[ch[1]] if ch else N["hi"] - N["lo"]
        k[i] = min(m[i], r)
    return [(d, c) for d, c in zip(depth, m) if d > 0]


def test_fronts_of_one_level_with_different_widths():
    import torch
    from paper_1508_07798_gb300 import hssnd as hs
    mesh, A = dg.diffusion_3d(9, 1, 0)
    nd = oracle.nd_order(3, mesh.n, 1, A.row_ptr, A.col_idx, leaf_max=LEAF)
    level = np.asarray(nd["level"])
    cols = {(b, r): _columns(oracle.hss_tree_for_front(nd, b), r) for b in range(len(level)) for r in (32, WIDE)}
    # a front that fits at the wide setting, beside one of its level with more columns at the narrow one
    wide = next(b for b in range(len(level)) if cols[b, WIDE] and all(_smem(WIDE, m) <= 220 * 1024 for _, m in cols[b, WIDE])
                and any(_smem(WIDE, m) > 220 * 1024 and any(d == e for e, _ in cols[b, WIDE])
                        for c in np.nonzero(level == level[b])[0] if c != b for d, m in cols[c, 32]))
    assert all(_smem(32, m) <= 220 * 1024 for (b, r), v in cols.items() if r == 32 for _, m in v)
    r = np.full(len(level), 32, dtype=np.int32)
    r[wide] = WIDE
    dA = hs.DeviceBSR.from_host(A)
    tree = hs.nd_order((3, mesh.n[:3], 1), dA, leaf_max=LEAF)
    # (dr: no front samples again)
    F = hs.hss_factor(dA, tree, tol=1e-3, precision="fp64", r_init=r, rmax=WIDE, dr=WIDE, cap_policy="accept")
    log = F.export_log()
    assert dict(zip(log["box"].tolist(), log["r"].tolist()))[wide] == WIDE
    assert torch.all(torch.isfinite(hs.hss_apply(F, torch.ones(A.n, dtype=torch.float64, device="cuda"))))
