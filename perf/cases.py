"""The work that a user of this framework has it do, as measurable cases.

A case is a dict of plain values; ``listed()`` gives the fixed ones, ``draw(rng)`` one
more of the same ranges.  ``prepare`` makes what a program has in hand before the call
(seeded inputs on the GPU, the plan, the workspace, the analysis or factors it keeps),
``run`` makes one pass through the public entry points of ``ctp`` and returns its
outputs whole, ``work`` says what the pass cannot do without, and ``exact`` computes the
outputs in 64 bits with torch alone.

Kinds:
  compress   one compression of A21 (strict, Section 4.1; relaxed, Section 4.2)
  supernode  one supernode: compression, pivot search, Solve and (smode) Form
  batch      many uneven fronts through one plan (Batch)
  dense      a complete dense symmetric system, forward and backward (sym_solve)
  sparse     a sparse system, factored multifrontally, forward and backward
             (SparseSymSolver)
  mf_solve   solves with kept multifrontal factors (Multifrontal.solve)
"""
import math

import numpy as np
import torch

from paper_1305_2353_gb300 import ctp, inputs

_MODES = {"none": 0, "fp64": 1, "fp32": 2, "fp64_packed": 3, "fp32_packed": 4, "fp32_tiled": 5}


def listed():
    return [
        # the compression that every supernode begins with, at the size of the
        # paper's large random supernodes (bench.py's headline shape)
        {"name": "compress_strict_large", "kind": "compress", "pivot": "strict", "m": 199744, "p": 256},
        # the smallest whole call: one small supernode with a few tiny columns
        # (inputs.single_small), where latency and launches count
        {"name": "supernode_small", "kind": "supernode", "n": 2000, "p": 64, "pivot": "strict", "prec": "fp64",
         "smode": "fp64", "solve": "fp64", "dist": "normal", "tiny": 8},
        # full-column threshold pivoting, which a user takes as the reference of
        # the compressed methods and as the pivoting of a root; odd, ragged sizes
        {"name": "supernode_tpp_ragged", "kind": "supernode", "n": 20011, "p": 127, "pivot": "tpp", "prec": "fp64",
         "smode": "none", "solve": "fp64", "dist": "uniform", "tiny": 0},
        # factor and solve of a large supernode without a Form (the part of the
        # work that the paper's timings are about)
        {"name": "supernode_factor_solve", "kind": "supernode", "n": 200000, "p": 256, "pivot": "relaxed",
         "prec": "fp64", "smode": "none", "solve": "fp64", "dist": "uniform", "tiny": 0},
        # the whole supernode in FP64 with its Schur complement
        {"name": "supernode_fp64", "kind": "supernode", "n": 20000, "p": 256, "pivot": "relaxed", "prec": "fp64",
         "smode": "fp64_packed", "solve": "fp64", "dist": "uniform", "tiny": 0},
        # the same in mixed precision: Solve and Form on the tensor cores
        {"name": "supernode_mixed", "kind": "supernode", "n": 40000, "p": 256, "pivot": "relaxed", "prec": "bf16x3",
         "smode": "fp32_tiled", "solve": "tc", "dist": "uniform", "tiny": 0},
        # a tree level's worth of uneven fronts, FP64 and mixed precision
        {"name": "batch_fp64", "kind": "batch", "count": 1024, "prec": "fp64", "smode": "fp64_packed"},
        {"name": "batch_mixed", "kind": "batch", "count": 1024, "prec": "bf16x3", "smode": "fp32_tiled"},
        # a complete dense system inside a differentiable program
        {"name": "dense_forward_backward", "kind": "dense", "N": 1999, "p_first": 64, "nrhs": 4},
        # a sparse system inside a differentiable program, FP64
        {"name": "sparse_forward_backward", "kind": "sparse", "k": 36, "nrhs": 8, "prec": "fp64"},
        # the largest sparse system, mixed precision with FP64 refinement
        {"name": "sparse_large_mixed", "kind": "sparse", "k": 64, "nrhs": 16, "prec": "bf16x6"},
        # one more right-hand side on kept factors (a time step, a Newton step)
        {"name": "sparse_solve_kept_factors", "kind": "mf_solve", "k": 48, "nrhs": 1},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["compress", "supernode", "supernode", "supernode", "batch", "dense", "sparse", "mf_solve"])
    if kind == "compress":
        return {"kind": kind, "pivot": rng.choice(["strict", "relaxed"]), "m": _log_int(rng, 300, 200000),
                "p": _log_int(rng, 8, 256)}
    if kind == "supernode":
        p = _log_int(rng, 8, 256)
        pivot = rng.choice(["strict", "relaxed", "relaxed", "tpp", "restricted", "single_row"])
        prec = "fp64" if pivot == "tpp" else rng.choice(["fp64", "fp64", "bf16x3", "bf16x6", "bf16"])
        smode = rng.choice(["none", "fp64", "fp64_packed", "fp32"] if prec == "fp64" else
                           ["fp32", "fp32_packed", "fp32_tiled"])
        n = p + _log_int(rng, 1, 60000 if smode == "none" else 20000)
        # the tensor-core Solve is the mixed-precision path's faster choice
        solve = rng.choice(["fp64", "tc"]) if prec != "fp64" else "fp64"
        return {"kind": kind, "n": n, "p": p, "pivot": pivot, "prec": prec, "smode": smode, "solve": solve,
                "dist": rng.choice(["normal", "uniform"]), "tiny": rng.choice([0, 0, min(8, p // 4)])}
    if kind == "batch":
        prec, smode = rng.choice([("fp64", "fp64_packed"), ("fp64", "none"), ("fp64", "fp32_packed"),
                                  ("bf16x3", "fp32_tiled"), ("bf16x6", "fp32_tiled")])
        return {"kind": kind, "count": _log_int(rng, 16, 1024), "prec": prec, "smode": smode}
    if kind == "dense":
        N = _log_int(rng, 100, 3000)
        return {"kind": kind, "N": N, "p_first": rng.choice([32, 64, 100, 256]), "nrhs": _log_int(rng, 1, 16)}
    if kind == "sparse":
        return {"kind": kind, "k": rng.randint(10, 44), "nrhs": _log_int(rng, 1, 32),
                "prec": rng.choice(["fp64", "fp64", "bf16x6"])}
    return {"kind": kind, "k": rng.randint(12, 56), "nrhs": _log_int(rng, 1, 32)}


# ---------------------------------------------------------------------------
# inputs (from the seed alone)

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _panel(n, p, dist, seed, tiny=0):
    """An n x p supernode as a (p, n) tensor (row j is column j); A11 is symmetric,
    `tiny` of its rows and columns are scaled by 1e-8."""
    g = _gen(seed)
    if dist == "normal":
        A = torch.randn((p, n), dtype=torch.float64, device="cuda", generator=g)
    else:
        A = torch.rand((p, n), dtype=torch.float64, device="cuda", generator=g).mul_(2.0).sub_(1.0)
    A11 = A[:, :p].triu()  # row j from the diagonal on: the lower triangle of A11
    A[:, :p] = A11 + A11.triu(1).t()
    if tiny:
        idx = torch.randperm(p, device="cuda", generator=g)[:tiny]
        A[idx, :p] *= 1e-8
        A[:, idx] *= 1e-8
    return A


def _batch_fronts(count, seed):
    """The uneven fronts of inputs.batch (p log-uniform in [8, 256], A21 rows log-uniform
    in [0, 16 p], N(0,1), 2% zero diagonals), drawn as one block.  The shapes are one
    fixed draw: a plan belongs to shapes, new values to a pass."""
    shapes = inputs.batch_shapes(count, seed=count)
    rng = np.random.default_rng(seed)
    flat = rng.standard_normal(int((shapes[:, 0] * shapes[:, 1]).sum()))
    out, at = [], 0
    for n, p in shapes:
        n, p = int(n), int(p)
        A = flat[at:at + n * p].reshape(p, n).T
        at += n * p
        low = np.tril(A[:p])
        A[:p] = low + np.tril(low, -1).T
        nz = int(round(0.02 * p))
        if nz:
            idx = rng.choice(p, size=nz, replace=False)
            A[idx, idx] = 0.0
        out.append(A)
    return out, [int(p) for p in shapes[:, 1]]


def _grid(k, seed):
    """The 7-point Laplacian of a k x k x k grid with one weight per direction, shifted to
    be indefinite: (colptr, rowind, val, weights, sigma).  The shift sits in the widest
    gap of the spectrum near half the mean eigenvalue."""
    rng = np.random.default_rng(int(seed) + 1000 * k)
    w = rng.uniform(0.7, 1.3, 3)
    lam = _spectrum(k, w).ravel()
    near = np.sort(lam[(lam > 0.9 * w.sum()) & (lam < 1.1 * w.sum())])
    i = int(np.argmax(np.diff(near)))
    sigma = 0.5 * (near[i] + near[i + 1])
    colptr, rowind, _ = inputs.laplacian_3d(k)
    step = rowind - np.repeat(np.arange(k ** 3), np.diff(colptr))
    val = np.where(step == 0, 2.0 * w.sum() - sigma,
                   np.where(step == 1, -w[0], np.where(step == k, -w[1], -w[2])))
    return colptr, rowind, val, w, sigma


def _spectrum(k, w):
    """Eigenvalues of the unshifted operator, indexed [z, y, x]."""
    mu = 2.0 - 2.0 * np.cos(np.arange(1, k + 1) * np.pi / (k + 1))
    return w[2] * mu[:, None, None] + w[1] * mu[None, :, None] + w[0] * mu[None, None, :]


def _randn(shape, seed, salt):
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=_gen(int(seed) + 104729 * salt))


def _s_buffer(m, smode):
    if smode == "none":
        return None
    dt = torch.float64 if smode in ("fp64", "fp64_packed") else torch.float32
    if smode in ("fp64_packed", "fp32_packed"):
        return torch.zeros(max(m * (m + 1) // 2, 1), dtype=dt, device="cuda")
    if smode == "fp32_tiled":
        nb = (m + 127) // 128
        return torch.zeros(max(nb * (nb + 1) // 2 * 16384, 1), dtype=dt, device="cuda")
    return torch.zeros((m, m), dtype=dt, device="cuda")


# ---------------------------------------------------------------------------
# prepare and run

def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("compress", "supernode", "batch", "mf_solve"):
        st["ctx"] = ctx = ctp.Context(torch.cuda.current_device())
    if kind == "compress":
        m, p = case["m"], case["p"]
        st["A21"] = _panel(m + p, p, "uniform", seed)[:, p:].contiguous()
        st["C"] = torch.empty((p, p), dtype=torch.float64, device="cuda")
        st["rows"] = torch.empty(m if case["pivot"] == "strict" else p, dtype=torch.int32, device="cuda")
        st["ws"] = ctx.workspace(m + p, p, ctp.options(pivot=case["pivot"]))
    elif kind == "supernode":
        n, p = case["n"], case["p"]
        st["opt"] = opt = ctp.options(pivot=case["pivot"], prec=case["prec"], smode=case["smode"],
                                      solve=case["solve"])
        st["A0"] = _panel(n, p, case["dist"], seed, case["tiny"])
        st["A"] = torch.empty_like(st["A0"])
        st["perm"] = torch.empty(p, dtype=torch.int32, device="cuda")
        st["piv"] = torch.empty(p, dtype=torch.int32, device="cuda")
        st["D"] = torch.empty(2 * p, dtype=torch.float64, device="cuda")
        st["nelim"] = torch.empty(1, dtype=torch.int32, device="cuda")
        st["S"] = _s_buffer(n - p, case["smode"])
        st["ws"] = ctx.workspace(n, p, opt)
    elif kind == "batch":
        fronts, ps = _batch_fronts(case["count"], seed)
        st["batch"] = ctp.Batch(ctx, fronts, ps, ctp.options(prec=case["prec"], smode=case["smode"]))
    elif kind == "dense":
        N = case["N"]
        X = _randn((N, N), seed, 1)
        st["A"] = (X.tril() + X.tril(-1).t()).requires_grad_(True)
        st["B"] = _randn((N, case["nrhs"]), seed, 2).requires_grad_(True)
        st["G"] = _randn((N, case["nrhs"]), seed, 3)
        st["ctx"] = ctp.Context(torch.cuda.current_device())
    else:
        k, nrhs = case["k"], case["nrhs"]
        colptr, rowind, val, _, _ = _grid(k, seed)
        perm, blocks = inputs.nested_dissection_3d(k)
        N = k ** 3
        if kind == "sparse":
            st["ctx"] = ctx = ctp.Context(torch.cuda.current_device())
            st["solver"] = ctp.SparseSymSolver(ctx, colptr, rowind, perm, blocks, prec=case["prec"])
            st["val"] = torch.from_numpy(val).cuda().requires_grad_(True)
            st["B"] = _randn((N, nrhs), seed, 2).requires_grad_(True)
            st["G"] = _randn((N, nrhs), seed, 3)
        else:
            st["mf"] = mf = ctp.Multifrontal(ctx, colptr, rowind, val, perm, blocks)
            mf.factor(ctp.options())
            st["B"] = _randn((nrhs, N), seed, 2)
            st["X"] = torch.empty_like(st["B"])
            st["ws"] = mf.refine_workspace(nrhs)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "compress":
        f = st["ctx"].compress_strict if case["pivot"] == "strict" else st["ctx"].compress_relaxed
        f(st["A21"], case["m"], case["p"], case["m"], st["C"], st["rows"], st["ws"])
        return {"C": st["C"], "rows": st["rows"]}
    if kind == "supernode":
        n, p = case["n"], case["p"]
        st["A"].copy_(st["A0"])  # factored in place
        st["ctx"].factor_supernode(st["A"], n, p, n, st["opt"], st["perm"], st["piv"], st["D"], st["nelim"],
                                   st["S"], max(n - p, 1), st["ws"])
        out = {key: st[key] for key in ("A", "perm", "piv", "D", "nelim")}
        if st["S"] is not None:
            out["S"] = st["S"]
        return out
    if kind == "batch":
        b = st["batch"]
        b.reset()  # factored in place
        b.run()
        out = {"A": b.A, "perm": b.perm, "piv": b.piv, "D": b.D, "nelim": b.nelim}
        if b.S is not None:
            out["S"] = b.S
        return out
    if kind == "dense":
        X = ctp.sym_solve(st["A"], st["B"], ctx=st["ctx"], p_first=case["p_first"])
        gA, gB = torch.autograd.grad(X, [st["A"], st["B"]], st["G"])
        return {"X": X.detach(), "gA": gA, "gB": gB}
    if kind == "sparse":
        X = st["solver"](st["val"], st["B"])
        gv, gB = torch.autograd.grad(X, [st["val"], st["B"]], st["G"])
        return {"X": X.detach(), "gval": gv, "gB": gB}
    st["X"].copy_(st["B"])  # solved in place
    st["mf"].solve(st["X"], st["ws"])
    return st["X"]


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _supernode_work(n, p, pivot, smode):
    m = n - p
    # strict and single-row pivoting accept about a dozen columns of random data, the others all
    e = min(p, 12) if pivot in ("strict", "single_row") else p
    width = {"none": 0, "fp64": 8, "fp64_packed": 8}.get(smode, 4)
    k = np.arange(1, e + 1, dtype=np.float64)
    flops = float(((n - k) + 2 * ((n - p) * (p - k) + (p - k) * (p - k + 1) / 2)).sum())
    if smode != "none":
        flops += float(m) * (m + 1) * e
    return 16.0 * n * p + width * m * (m + 1) / 2, flops


def work(case):
    kind = case["kind"]
    if kind == "compress":
        m, p = case["m"], case["p"]
        return {"bytes": 8.0 * m * p + 8.0 * p * p + 4.0 * (m if case["pivot"] == "strict" else p), "flops": 0.0}
    if kind == "supernode":
        b, f = _supernode_work(case["n"], case["p"], case["pivot"], case["smode"])
        return {"bytes": b, "flops": f}
    if kind == "batch":
        bf = [_supernode_work(int(n), int(p), "strict", case["smode"])
              for n, p in inputs.batch_shapes(case["count"], seed=case["count"])]
        return {"bytes": sum(x for x, _ in bf), "flops": sum(x for _, x in bf)}
    if kind == "dense":
        N, r = float(case["N"]), case["nrhs"]
        # one factorization, two solves, the gradient of the lower triangle
        return {"bytes": 16.0 * N * N + 40.0 * N * r, "flops": N ** 3 / 3 + 4 * N * N * r + 2 * N * N * r}
    k, r = float(case["k"]), case["nrhs"]
    # nested dissection of a cube: factor flops and fill counted once on 64^3 (strict pivoting)
    fill, flops = 10.25 * k ** 4, 6.17 * k ** 6
    if kind == "sparse":
        return {"bytes": 8 * 8 * k ** 3 + 40 * k ** 3 * r, "flops": flops + 8 * fill * r}
    return {"bytes": 8 * fill + 16 * k ** 3 * r, "flops": 4 * fill * r}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from torch alone

def _strict_c(A21):
    """Eq. (4.1): rows of A21 by the column of their largest entry; (p, p) C and J."""
    p, m = A21.shape
    C = torch.zeros((p, p), dtype=torch.float64, device=A21.device)
    if m == 0:
        return C, torch.empty(0, dtype=torch.int64, device=A21.device)
    absA = A21.abs()
    J = absA.argmax(0)
    for k in range(p):
        C[:, k].scatter_reduce_(0, J, absA[k], "amax")
    return C, J


def _relaxed_c(A21):
    """Section 4.2: column by column, the largest entry's row among the rows not taken."""
    p, m = A21.shape
    rows = torch.full((p,), -1, dtype=torch.int64, device=A21.device)
    taken = torch.zeros(m, dtype=torch.bool, device=A21.device)
    C = torch.zeros((p, p), dtype=torch.float64, device=A21.device)
    for j in range(min(p, m)):
        i = A21[j].abs().masked_fill(taken, -1.0).argmax()
        rows[j] = i
        taken[i] = True
        C[j] = A21[:, i]
    return C, rows


def _pivots(W, p, abs_outer, u=0.01, small=1e-20):
    """Threshold pivoting (Listing 1) on W, the LD x p matrix whose first p rows are A11 in
    full; the tests see all its rows.  Returns (order, kinds)."""
    W = W.clone()
    dev = W.device
    live = torch.ones(p, dtype=torch.bool, device=dev)
    order, kinds, m, accepted = [], [], (1 if p >= 2 else 0), False
    while len(order) < p:
        cand = torch.nonzero(live[m:]).flatten() + m
        if cand.numel() == 0:
            if not accepted:
                break
            accepted, m = False, 0
            continue
        M = W.abs()
        M[:p].masked_fill_(~live[:, None], 0.0)
        # a few candidates at a time: most searches end soon (all of them when they do not)
        hit = None
        for c in (cand[:2], cand[2:]):
            if c.numel() == 0:
                continue
            nc = torch.arange(c.numel(), device=dev)
            rows = torch.arange(p, device=dev)[:, None]
            part = torch.where(live[:, None] & (rows < c[None]), M[:p, c], -1.0)
            best, t = part.max(0)[0], part.argmax(0)
            has = best >= 0
            t = torch.where(has, t, c)
            Mc, Mt = M[:, c], M[:, t]
            allmax = Mc.max(0)[0]
            for X in (Mc, Mt):
                X[c, nc] = 0.0
                X[t, nc] = 0.0
            vm, vt = Mc.max(0)[0], Mt.max(0)[0]
            att, atm, amm = W[t, t], W[t, c], W[c, c]
            amax = torch.maximum(att.abs(), torch.maximum(atm.abs(), amm.abs()))
            sc = 1.0 / amax.clamp_min(1e-300)
            d0, d1 = amm * sc * att, atm * sc * atm
            det = d0 - d1
            guard = torch.maximum(0.5 * d0.abs(), 0.5 * d1.abs()).clamp_min(small)
            grow = torch.maximum(amm.abs() * vt + atm.abs() * vm, atm.abs() * vt + att.abs() * vm) * sc
            ok2 = has & (amax >= small) & (det.abs() > guard) & (
                (torch.maximum(vm, vt) < small) | (grow <= det.abs() / u))
            ok1 = amm.abs() >= u * torch.where(has, torch.maximum(vm, atm.abs()), vm)
            kind = torch.where(allmax < small, -1, torch.where(ok2, 2, torch.where(ok1, 1, 0)))
            pos = torch.nonzero(kind).flatten()
            if pos.numel():
                i = int(pos[0])
                hit = (int(kind[i]), int(t[i]), int(c[i]))
                break
        if hit is None:
            m = p
            continue
        kd, t, c = hit
        accepted, m = True, c + 1
        q = [t, c] if kd == 2 else [c]
        live[q] = False
        order += q
        kinds += [2, 0] if kd == 2 else [kd]
        if kd != -1:
            B = W[:, q]
            Dinv = torch.linalg.inv(W[q][:, q])
            lv = torch.nonzero(live).flatten()
            upd = (B @ Dinv) @ W[q][:, lv]
            if abs_outer and W.shape[0] > p:
                upd[p:] = -((B[p:].abs() @ Dinv.abs()) @ W[q][:, lv].abs())
            W[:, lv] -= upd
    rest = torch.nonzero(live).flatten().tolist()
    return order + rest, kinds + [3] * len(rest)


def _factor(A0, p, pivot):
    """The supernode's factor for its pivot order: (A, perm, piv, D, e, W21) with A laid out
    as the framework leaves it."""
    A21 = A0[:, p:]
    A11 = A0[:, :p]
    outer = {"strict": lambda: _strict_c(A21)[0], "relaxed": lambda: _relaxed_c(A21)[0],
             "tpp": lambda: A21.t(), "restricted": lambda: A21[:, :0].t(),
             "single_row": lambda: A21.abs().amax(1)[None] if A21.shape[1] else A21[:, :0].t()}[pivot]()
    # the search runs where its many small steps are quick
    where = "cuda" if outer.shape[0] > 2048 else "cpu"
    W = torch.cat([A11, outer]).to(where)
    order, kinds = _pivots(W, p, pivot in ("strict", "single_row"))
    e = sum(1 for k in kinds if k != 3)
    o = torch.tensor(order, device="cuda")
    T = torch.cat([A11[o][:, o], A0[o, p:]], 1)  # columns in pivot order, full A11
    D = torch.zeros(2 * p, dtype=torch.float64, device="cuda")
    L, Y = torch.zeros_like(T), torch.zeros_like(T)
    k = 0
    while k < e:
        w = 2 if kinds[k] == 2 else 1
        if kinds[k] == -1:
            k += 1
            continue
        q = slice(k, k + w)
        blk = T[q, q].clone()
        D[2 * k] = blk[0, 0]
        if w == 2:
            D[2 * k + 1], D[2 * k + 2] = blk[0, 1], blk[1, 1]
        Y[q] = T[q]
        L[q] = torch.linalg.inv(blk) @ T[q]
        T[k + w:] -= T[q, k + w:p].t() @ L[q]
        k += w
    out = A0.clone()
    out[:, p:] = torch.cat([L[:e, p:], T[e:, p:]])
    low = torch.cat([L[:e, :p], T[e:, :p]])
    for k in range(e):
        if kinds[k] != -1:
            low[k, k] = D[2 * k]
        if kinds[k] == 2:
            low[k, k + 1] = D[2 * k + 1]
    up = torch.ones((p, p), dtype=torch.bool, device="cuda").triu()
    out[:, :p] = torch.where(up, low, A0[:, :p])
    return (out, torch.tensor(order, dtype=torch.int32, device="cuda"),
            torch.tensor(kinds, dtype=torch.int32, device="cuda"), D, e, Y[:e, p:])


def _schur(L21, W21, smode):
    """S = W21 L21^T in the layout `smode` (rows of the arguments are columns)."""
    m = L21.shape[1]
    if smode in ("fp64", "fp32"):
        return (L21.t() @ W21).triu()  # [j, i] = S(i, j), the lower triangle of S
    if smode in ("fp64_packed", "fp32_packed"):
        out, at, step = torch.empty(max(m * (m + 1) // 2, 1), dtype=torch.float64, device="cuda").zero_(), 0, 4096
        for j0 in range(0, m, step):
            blk = L21[:, j0:j0 + step].t() @ W21[:, j0:]
            sel = blk[torch.ones_like(blk, dtype=torch.bool).triu()]
            out[at:at + sel.numel()] = sel
            at += sel.numel()
        return out
    nb = (m + 127) // 128
    pad = nb * 128 - m
    Lp, Wp = (torch.nn.functional.pad(x, (0, pad)) for x in (L21, W21))
    out, at = torch.zeros(max(nb * (nb + 1) // 2 * 16384, 1), dtype=torch.float64, device="cuda"), 0
    for b in range(nb):  # block column b, blocks from the diagonal down, columns first inside
        blk = Lp[:, b * 128:(b + 1) * 128].t() @ Wp[:, b * 128:]
        blk = blk.reshape(128, nb - b, 128).transpose(0, 1)
        out[at:at + blk.numel()] = blk.reshape(-1)
        at += blk.numel()
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "compress":
        A21 = _panel(case["m"] + case["p"], case["p"], "uniform", seed)[:, case["p"]:]
        C, rows = (_strict_c if case["pivot"] == "strict" else _relaxed_c)(A21)
        return {"C": C, "rows": rows.to(torch.int32)}
    if kind == "supernode":
        n, p, smode = case["n"], case["p"], case["smode"]
        A0 = _panel(n, p, case["dist"], seed, case["tiny"])
        A, perm, piv, D, e, W21 = _factor(A0, p, case["pivot"])
        out = {"A": A, "perm": perm, "piv": piv, "D": D, "nelim": torch.tensor([e], dtype=torch.int32)}
        if smode != "none":
            out["S"] = _schur(A[:e, p:], W21, smode)
        return out
    if kind == "batch":
        fronts, ps = _batch_fronts(case["count"], seed)
        parts = {"A": [], "perm": [], "piv": [], "D": [], "nelim": [], "S": []}
        for F, p in zip(fronts, ps):
            A, perm, piv, D, e, W21 = _factor(torch.from_numpy(np.ascontiguousarray(F.T)).cuda(), p, "strict")
            for key, x in (("A", A), ("perm", perm), ("piv", piv), ("D", D)):
                parts[key].append(x.flatten())
            parts["nelim"].append(torch.tensor([e], dtype=torch.int32))
            if case["smode"] != "none":
                if F.shape[0] > p:
                    parts["S"].append(_schur(A[:e, p:], W21, case["smode"]))
        return {key: torch.cat(x) for key, x in parts.items() if x}
    if kind == "dense":
        N = case["N"]
        R = _randn((N, N), seed, 1)
        A = R.tril() + R.tril(-1).t()
        B, G = _randn((N, case["nrhs"]), seed, 2), _randn((N, case["nrhs"]), seed, 3)
        lu, piv = torch.linalg.lu_factor(A)

        def solve(b):
            x = torch.linalg.lu_solve(lu, piv, b)
            for _ in range(3):
                x = x + torch.linalg.lu_solve(lu, piv, b - A @ x)
            return x
        X, g = solve(B), solve(G)
        gA = -(g @ X.t() + X @ g.t()).tril(-1) - torch.diag((g * X).sum(1))
        return {"X": X, "gA": gA, "gB": g}
    k = case["k"]
    colptr, rowind, _, w, sigma = _grid(k, seed)
    i = np.arange(1, k + 1)
    Q = torch.from_numpy(np.sqrt(2.0 / (k + 1)) * np.sin(np.outer(i, i) * np.pi / (k + 1))).cuda()
    lam = torch.from_numpy(_spectrum(k, w) - sigma).cuda()

    def solve(b):  # (N, nrhs): the operator is diagonal in the sine basis of each direction
        t = b.t().reshape(-1, k, k, k)

        def transform(t):
            for _ in range(3):
                t = (t @ Q).permute(0, 3, 1, 2)
            return t
        return transform(transform(t) / lam).reshape(b.shape[1], -1).t()
    B = _randn((k ** 3, case["nrhs"]), seed, 2) if kind == "sparse" else _randn((case["nrhs"], k ** 3), seed, 2).t()
    X = solve(B)
    if kind == "mf_solve":
        return X.t()
    g = solve(_randn((k ** 3, case["nrhs"]), seed, 3))
    row = torch.from_numpy(rowind.astype(np.int64)).cuda()
    col = torch.from_numpy(np.repeat(np.arange(k ** 3), np.diff(colptr))).cuda()
    gv = -(g[row] * X[col] + g[col] * X[row]).sum(1)
    return {"X": X, "gval": torch.where(row == col, 0.5 * gv, gv), "gB": g}
