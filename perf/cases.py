"""The work a program asks of this library, as cases that can be timed.

A program orders and factors a DG system matrix, solves with it by FGMRES, and
either discards the factor (a new operator in every step) or keeps it for
further right-hand sides.  The listed cases cover that over the operators,
sizes, precisions and options of the repository's configurations, benchmark
and tests, from the 1,024-dof Poisson problem to the 262,144-dof diffusion
problem with 20 right-hand sides; draw() gives other cases of the same ranges.

Every solve goes to a true relative residual of 1e-11, so that the solution is
determined by the system and not by the preconditioner's rounding.
"""
import math

import numpy as np
import torch

from paper_1508_07798_gb300 import dg_inputs as dg
from paper_1508_07798_gb300 import hssnd

RTOL = 1e-11
MAXIT = 400
LEAF = 64


def listed():
    return [
        # the smallest configuration, library defaults: FP64, one call after another on
        # 1,024 dofs; launches, read-backs and host scheduling count, not arithmetic
        _solve("poisson16_fp64", "poisson", 16, 1, "fp64", 1e-6),
        # the benchmark's operator in the plain FP64 form
        _solve("helmholtz64_fp64", "helmholtz", 64, 2, "fp64", 1e-4),
        # the benchmark's operator in the mixed form: FP32 factor, FP64 Krylov, with the
        # tuned apply split and GEMM engine as the benchmark runs it
        _solve("helmholtz64_mixed", "helmholtz", 64, 2, "fp32", 1e-6, tuned=True),
        # the known-width form (sample widths predicted from earlier factorizations,
        # checked by the residual probe), at the degree-3 size of the width model's runs
        _solve("helmholtz64p3_widths", "helmholtz", 64, 3, "fp32", 1e-6, tuned=True, widths=True),
        # a larger 2D problem, between the benchmark's and the million-dof configuration
        _solve("helmholtz128_mixed", "helmholtz", 128, 2, "fp32", 1e-6, tuned=True),
        # an odd mesh: uneven boxes, fronts whose sizes are no multiple of any tile
        _solve("poisson51p3_mixed", "poisson", 51, 3, "fp32", 1e-5),
        # the 3D configuration: tall fronts, ranks at the width cap, BF16 sampling, 20 right-hand sides
        _solve("diffusion32_20rhs", "diffusion", 32, 1, "fp32", 1e-5, nrhs=20, tuned=True, bf16=True),
        # the 3D operator at the size of the width model's runs, one right-hand side
        _solve("diffusion16", "diffusion", 16, 1, "fp32", 1e-5, tuned=True),
        # many uneven instances factored and solved together, 32 right-hand sides each
        {"name": "batch24_32rhs", "kind": "batch", "count": 24, "first": 7, "lo": 16, "hi": 64, "p": 2, "tol": 1e-6,
         "precision": "fp32", "nrhs": 32},
        # a kept FP32 factor and a new right-hand side: the Krylov loop alone
        {"name": "resolve64_mixed", "kind": "resolve", "op": "helmholtz", "n": 64, "p": 2, "field": 0, "tol": 1e-6,
         "precision": "fp32", "nrhs": 1, "tuned": True},
        # the preconditioner inside somebody else's Krylov method: one vector at a time
        {"name": "apply64_fp64", "kind": "apply", "op": "poisson", "n": 64, "p": 2, "field": 0, "tol": 1e-6,
         "precision": "fp64", "nrhs": 1, "tuned": True},
        # the residual check of such a method: A x alone
        {"name": "spmv128p3", "kind": "spmv", "op": "helmholtz", "n": 128, "p": 3, "field": 0, "nrhs": 1},
    ]


def _solve(name, op, n, p, precision, tol, nrhs=1, tuned=False, bf16=False, widths=False, field=0):
    return {"name": name, "kind": "solve", "op": op, "n": n, "p": p, "field": field, "tol": tol,
            "precision": precision, "nrhs": nrhs, "tuned": tuned, "bf16": bf16, "widths": widths}


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve"] * 6 + ["batch", "resolve", "apply", "spmv"])
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(2, 16), "first": rng.randint(0, 10 ** 6), "lo": rng.randint(4, 16),
                "hi": rng.randint(20, 48), "p": rng.choice([1, 2, 3]), "tol": 1e-6, "precision": "fp32",
                "nrhs": rng.choice([1, 2, 7, 16, 32])}
    op = rng.choice(["poisson", "poisson", "helmholtz", "helmholtz", "diffusion"])
    p = 1 if op == "diffusion" else rng.choice([1, 2, 3])
    field = rng.randint(0, 9)
    nrhs = rng.choice([1, 1, 1, 3, 8, 20])
    fp64 = rng.random() < 0.3
    if kind == "spmv":
        n = size(4, 32) if op == "diffusion" else size(8, 192)
        return {"kind": kind, "op": op, "n": n, "p": p, "field": field, "nrhs": nrhs}
    if op == "diffusion":
        n = size(4, 12 if fp64 else 20)
    else:
        n = size(8, 64 if fp64 else 112)
    tol = 1e-6 if op == "helmholtz" else 1e-5 if op == "diffusion" else rng.choice([1e-4, 1e-5, 1e-6])
    precision = "fp64" if fp64 else "fp32"
    tuned = rng.random() < 0.5
    if kind == "apply":
        n, op, precision, tol = min(n, 48), "poisson", "fp64", 1e-6
    if kind in ("apply", "resolve"):
        return {"kind": kind, "op": op, "n": n, "p": p, "field": field, "tol": tol, "precision": precision,
                "nrhs": nrhs, "tuned": tuned}
    case = _solve("", op, n, p, precision, tol, nrhs, tuned, op == "diffusion" and not fp64 and rng.random() < 0.5,
                  rng.random() < 0.25, field)
    del case["name"]
    return case


# ------------------------------------------------------------------ inputs
def _operator(op, n, p, field):
    """(mesh descriptor, mesh, matrix) on the host."""
    if op == "poisson":
        mesh, A = dg.poisson_2d(n, p)
    elif op == "helmholtz":
        mesh, A = dg.helmholtz_2d(n, p, field)
    else:
        mesh, A = dg.diffusion_3d(n, p, field)
    return (mesh.dim, tuple(mesh.n[:mesh.dim]), p), mesh, A


def _rhs(op, mesh, N, nrhs, seed):
    """Right-hand sides as the configurations have them: Gaussian point sources for
    Helmholtz, U(-1, 1) per dof for Poisson, N(0, 1) for diffusion."""
    if op == "helmholtz":
        b = np.concatenate([dg.point_source_rhs(mesh, 1000 * seed + k) for k in range(nrhs)], axis=1)
    else:
        b = dg.random_rhs(N, nrhs, seed, kind="uniform" if op == "poisson" else "normal")
    return b[:, 0] if nrhs == 1 else np.asfortranarray(b)


def _factor_options(case):
    o = {"tol": case["tol"], "precision": case["precision"]}
    if case.get("tuned"):
        o.update(autotune=1, tensor_cores=3)
    if case.get("bf16"):
        o["sample_bf16"] = 1
    return o


def _instances(case):
    """Meshes, matrices and operators of a batch, drawn from case["first"]."""
    rng = np.random.default_rng(case["first"])
    out = []
    for _ in range(case["count"]):
        n, op, field = int(rng.integers(case["lo"], case["hi"] + 1)), ("poisson", "helmholtz")[rng.integers(2)], int(rng.integers(10))
        out.append((op,) + _operator(op, n, case["p"], field))
    return out


def prepare(case, seed):
    seed = int(seed) % 100003
    if case["kind"] == "batch":
        inst = _instances(case)
        dAs = [hssnd.DeviceBSR.from_host(A) for _, _, _, A in inst]
        B = np.concatenate([dg.random_rhs(A.n, case["nrhs"], seed + 31 * i, kind="normal") for i, (_, _, _, A) in
                            enumerate(inst)], axis=0)
        return {"case": case, "meshes": [m for _, m, _, _ in inst], "A": dAs,
                "b": torch.as_tensor(np.asfortranarray(B), device="cuda"), "options": _factor_options(dict(case, tuned=True))}
    desc, mesh, A = _operator(case["op"], case["n"], case["p"], case["field"])
    dA = hssnd.DeviceBSR.from_host(A)
    s = {"case": case, "mesh": desc, "A": dA}
    if case["kind"] in ("spmv", "apply"):
        x = dg.random_rhs(A.n, case["nrhs"], seed, kind="normal")
        s["b"] = torch.as_tensor(x[:, 0] if case["nrhs"] == 1 else x, device="cuda")
    else:
        s["b"] = torch.as_tensor(_rhs(case["op"], mesh, A.n, case["nrhs"], seed), device="cuda")
    if case["kind"] == "spmv":
        return s
    s["options"] = _factor_options(case)
    if case.get("widths"):
        # widths a program has from a factorization of the same operator with another
        # coefficient field: each front's largest rank plus the oversampling, in eights
        dB = hssnd.DeviceBSR.from_host(_operator(case["op"], case["n"], case["p"], case["field"] + 1)[2])
        tree = hssnd.nd_order(desc, dB, leaf_max=LEAF)
        log = hssnd.hss_factor(dB, tree, **s["options"]).export_log()
        r = np.full(tree.desc.nbox, 32, dtype=np.int32)
        r[log["box"]] = np.clip(-(-(log["kmax"] + 10) // 8) * 8, 16, 96)
        s["options"].update(r_init=r, probe=4)
    if case["kind"] in ("apply", "resolve"):
        s["tree"] = hssnd.nd_order(desc, dA, leaf_max=LEAF)
        s["factor"] = hssnd.hss_factor(dA, s["tree"], **s["options"])
    return s


def run(state):
    kind = state["case"]["kind"]
    if kind == "spmv":
        return hssnd.hss_spmv(state["A"], state["b"])
    if kind == "apply":
        return hssnd.hss_apply(state["factor"], state["b"])
    if kind == "resolve":
        return hssnd.fgmres_solve(state["A"], state["factor"], state["b"], rtol=RTOL, maxit=MAXIT)[0]
    if kind == "batch":
        forest = hssnd.nd_order_batched(state["meshes"], state["A"], leaf_max=LEAF)
        F = hssnd.hss_factor_batched(state["A"], forest, **state["options"])
        return hssnd.fgmres_solve_batched(F, state["b"], rtol=RTOL, maxit=MAXIT)[0]
    tree = hssnd.nd_order(state["mesh"], state["A"], leaf_max=LEAF)
    F = hssnd.hss_factor(state["A"], tree, **state["options"])
    return hssnd.fgmres_solve(state["A"], F, state["b"], rtol=RTOL, maxit=MAXIT)[0]


# ------------------------------------------------------------------ work
def _boxes(n, p, dim):
    """(interior, boundary) dofs of every front of the nested-dissection box tree and the
    size of the top block: a box's boundary elements are those with a neighbour outside it."""
    bs, out = (p + 1) ** dim, []

    def boundary(lo, hi):
        v = c = 1
        for a in range(dim):
            v *= hi[a] - lo[a]
            c *= max(0, hi[a] - lo[a] - (lo[a] > 0) - (hi[a] < n))
        return (v - c) * bs, v * bs

    def cut(lo, hi):
        ext = [hi[a] - lo[a] for a in range(dim)]
        a = max(range(dim), key=lambda k: (ext[k], k))
        mid = lo[a] + ext[a] // 2
        return (lo, [mid if k == a else hi[k] for k in range(dim)]), ([mid if k == a else lo[k] for k in range(dim)], hi)

    def visit(lo, hi):
        nb, vol = boundary(lo, hi)
        if vol <= LEAF or vol == bs:
            out.append((vol - nb, nb))
            return nb
        below = sum(visit(*half) for half in cut(lo, hi))
        out.append((below - nb, nb))
        return nb

    lo, hi = [0] * dim, [n] * dim
    top = sum(visit(*half) for half in cut(lo, hi))
    return out, top


def _work_of(op, n, p, nrhs, kind, esize):
    """Bytes of the matrix, the vectors and (kept factors) the factor entries of one apply;
    flops of the dense elimination of every front, by LU, or two per entry and vector."""
    dim = 3 if op == "diffusion" else 2
    ne, bs = n ** dim, (p + 1) ** dim
    nnz = (ne + 2 * dim * n ** (dim - 1) * (n - 1)) * bs * bs
    N = ne * bs
    matrix = 8.0 * nnz + 4.0 * (nnz // (bs * bs) + ne + 1)
    vectors = 16.0 * N * nrhs
    if kind == "spmv":
        return matrix + vectors, 2.0 * nnz * nrhs
    fronts, top = _boxes(n, p, dim)
    if kind in ("apply", "resolve"):
        entries = float(top) ** 2 + sum(float(i) * (i + 2 * b) for i, b in fronts)
        extra, fl = (matrix, 2.0 * nnz * nrhs) if kind == "resolve" else (0.0, 0.0)
        return esize * entries + vectors + extra, 2.0 * entries * nrhs + fl
    lu = 2.0 / 3.0 * float(top) ** 3 + sum(2.0 / 3.0 * i ** 3 + 2.0 * i * i * b + 2.0 * i * b * b for i, b in fronts)
    return matrix + vectors, lu


def work(case):
    if case["kind"] == "batch":
        rng, parts = np.random.default_rng(case["first"]), []
        for _ in range(case["count"]):
            n, _, _ = int(rng.integers(case["lo"], case["hi"] + 1)), rng.integers(2), rng.integers(10)
            parts.append(_work_of("poisson", n, case["p"], case["nrhs"], "solve", 4))
    else:
        parts = [_work_of(case["op"], case["n"], case["p"], case["nrhs"], case["kind"],
                          4 if case.get("precision") == "fp32" else 8)]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


# ------------------------------------------------------------------ exact values
def _dense_lines(A, lines):
    """The matrix as block tridiagonal over `lines` equal groups of elements (mesh lines in 2D,
    planes in 3D): a function that makes its dense block (i, j) on the device."""
    ne_l, bs = A.nb // lines, A.bs
    rows = torch.as_tensor(np.repeat(np.arange(A.nb), np.diff(A.row_ptr)), device="cuda")
    cols = torch.as_tensor(A.col_idx.astype(np.int64), device="cuda")
    val = torch.as_tensor(A.val, device="cuda")

    def block(i, j):
        M = torch.zeros(ne_l, bs, ne_l, bs, dtype=torch.float64, device="cuda")
        at = torch.nonzero((rows // ne_l == i) & (cols // ne_l == j))[:, 0]
        M[rows[at] - i * ne_l, :, cols[at] - j * ne_l, :] = val[at]
        return M.reshape(ne_l * bs, ne_l * bs)

    return block


def _times(A, x):
    """A x in 64 bits, block by block."""
    rows = torch.as_tensor(np.repeat(np.arange(A.nb), np.diff(A.row_ptr)), device="cuda")
    cols = torch.as_tensor(A.col_idx.astype(np.int64), device="cuda")
    X = x.reshape(A.nb, A.bs, -1)
    y = torch.zeros_like(X)
    val = torch.as_tensor(A.val, device="cuda")
    for k in range(0, len(cols), 1 << 16):
        y.index_add_(0, rows[k:k + (1 << 16)], torch.bmm(val[k:k + (1 << 16)], X[cols[k:k + (1 << 16)]]))
    return y.reshape(A.n, -1)


def _solve_exact(A, lines, B):
    """A^-1 B by block elimination over the mesh lines, refined once."""
    block, N = _dense_lines(A, lines), A.n
    lus, ups = [], []
    for i in range(lines):
        D = block(i, i)
        if i > 0:
            D -= block(i, i - 1) @ ups[-1]
        lus.append(torch.linalg.lu_factor(D))
        ups.append(torch.linalg.lu_solve(*lus[-1], block(i, i + 1)) if i + 1 < lines else None)

    def solve(R):
        R, y = R.reshape(lines, N // lines, -1), []
        for i in range(lines):
            y.append(torch.linalg.lu_solve(*lus[i], R[i] - block(i, i - 1) @ y[-1] if i > 0 else R[i].clone()))
        for i in range(lines - 2, -1, -1):
            y[i] = y[i] - ups[i] @ y[i + 1]
        return torch.cat(y).reshape(N, -1)

    x = solve(B)
    return x + solve(B - _times(A, x))


def exact(case, seed):
    seed = int(seed) % 100003
    if case["kind"] == "apply":
        return None   # the approximate inverse of a compressed factor has no other definition than the method
    if case["kind"] == "batch":
        parts = []
        for i, (_, _, mesh, A) in enumerate(_instances(case)):
            B = torch.as_tensor(dg.random_rhs(A.n, case["nrhs"], seed + 31 * i, kind="normal"), device="cuda")
            parts.append(_solve_exact(A, mesh.n[1], B))
        return torch.cat(parts)
    _, mesh, A = _operator(case["op"], case["n"], case["p"], case["field"])
    nrhs = case["nrhs"]
    if case["kind"] == "spmv":
        b = dg.random_rhs(A.n, nrhs, seed, kind="normal")
        y = _times(A, torch.as_tensor(b, device="cuda"))
        return y[:, 0] if nrhs == 1 else y
    if case["op"] == "diffusion" and case["n"] > 20:
        return None   # planes of more than 3,200 dofs: too long in 64 bits
    b = torch.as_tensor(_rhs(case["op"], mesh, A.n, nrhs, seed), device="cuda").reshape(A.n, -1)
    x = _solve_exact(A, mesh.n[mesh.dim - 1], b)
    return x[:, 0] if nrhs == 1 else x
