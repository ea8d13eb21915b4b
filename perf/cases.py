"""The workloads that the library's speed is judged by, through its public entry points.

``listed()`` names the cases, ``draw`` gives further ones of the same ranges,
``prepare`` makes what a program has in hand before the call (the matrix on the
device, the right-hand side, the split and preconditioner where a program keeps
them), ``run`` is one pass through the call, ``work`` what a pass cannot do
without, ``exact`` the outputs in 64 bits where they are known.

The matrices are those of ``workloads`` (convection-diffusion stencils with a few
dense columns, the rotated anisotropic 9-point operator, heavy-tailed column
counts, random geometric graphs), generated here in numpy with the sort on the
device. Every solution is a smooth vector chosen from the seed and the right-hand
side is A times it, so the exact solution is known. The solves run to an eps at
which x itself is good to ten digits (a program that differentiates through the
solve, or compares two solves, asks for that); the work per iteration is that of
the paper's 1e-8, with more iterations.
"""
import math

import numpy as np
import torch

import paper_1211_6866_gb300 as sai

# ||b - A x|| / ||b|| asked for, by the conditioning of the matrices
_EPS = {"solve2d": 1e-13, "grad_zipf": 1e-14, "many_zipf": 1e-14}

# entries of M per column: SPAI's bound 1 + mn max_aug; PSAI's patterns on the 7-point grid stay below this
_ROOM = {"spai": 51, "psai": 28}

# size limits of the drawn cases, per kind: (name of the size, least, most)
_RANGES = {
    "solve2d": ("m", 16, 180),      # m^2 unknowns
    "solve3d": ("m", 10, 64),       # m^3 unknowns
    "repair3d": ("m", 12, 40),
    "reuse3d": ("m", 10, 48),
    "adjoint3d": ("m", 10, 48),
    "block3d": ("m", 10, 34),
    "build3d": ("m", 12, 64),
    "build_aniso": ("m", 24, 300),  # m^2 unknowns
    "grad_zipf": ("n", 500, 4000),
    "many_zipf": ("n", 8000, 20000),
    "batch": ("nmax", 1500, 16000),
}


def listed():
    return [
        # The smallest call: all of the method on the paper-sized 2D system (n = 2025, 3 dense columns) with the
        # defaults of solve() (SPAI(0.4, 5, 10), BiCGStab, FP64 throughout).
        dict(name="solve_2d_45", kind="solve2d", m=45, s=3, sai="spai", precision=0, krylov="bicgstab"),
        # The benchmark's system, n = 262144 with ten 5% columns: SPAI(0.3, 5, 10) and GMRES(50) in the refined
        # forms.
        dict(name="solve_3d_64_refined", kind="solve3d", m=64, s=10, sai="spai", precision=1, krylov="gmres"),
        # The same call in plain FP64 with PSAI(0.3, tol 1e-3) on an odd grid.
        dict(name="solve_3d_37_psai_gmres", kind="solve3d", m=37, s=7, sai="psai", precision=0, krylov="gmres"),
        # BiCGStab, the paper's solver, in FP64 at an ordinary size.
        dict(name="solve_3d_49_bicgstab", kind="solve3d", m=49, s=10, sai="spai", precision=0, krylov="bicgstab"),
        # A system with zeros on its diagonal: the row permutation comes first.
        dict(name="solve_3d_33_repair", kind="repair3d", m=33, s=5, sai="spai", precision=1, krylov="gmres"),
        # A further right-hand side on a kept split and M of the heavy-tailed matrix: a thousand dense columns, so a
        # thousand systems at once and a large recovery system.
        dict(name="reuse_zipf_20000", kind="many_zipf", n=20000, sai="spai"),
        # The backward pass of such a solve: transposed solves, the adjoint recovery, dL/dA.
        dict(name="adjoint_3d_40", kind="adjoint3d", m=40, s=10, sai="spai", precision=0, krylov="bicgstab"),
        # Block GMRES(50) over the s+1 systems, refined form.
        dict(name="block_3d_30_refined", kind="block3d", m=30, s=10, sai="spai", precision=1, krylov="bgmres"),
        # Split and SPAI build alone in FP64 with patterns of dozens of entries per column (9-point operator): M is
        # built once and kept.
        dict(name="build_aniso_255", kind="build_aniso", m=255, s=12, sai="spai", precision=0),
        # Split and refined PSAI build alone on the benchmark's grid.
        dict(name="build_3d_64_psai", kind="build3d", m=64, s=10, sai="psai", precision=1),
        # A training step through the solve (autograd) on the heavy-tailed matrix: forward and both gradients with
        # about a hundred dense columns.
        dict(name="grad_zipf_2000", kind="grad_zipf", n=2000, sai="spai"),
        # Many independent matrices of different orders in one call, refined build.
        dict(name="batch_24", kind="batch", count=24, nmin=1000, nmax=12000, sai="spai", precision=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(sorted(_RANGES))
    size, lo, hi = _RANGES[kind]
    c = {"kind": kind, size: _log_int(rng, lo, hi)}
    c["sai"] = rng.choice(("spai", "psai"))
    if kind in ("solve2d", "solve3d", "repair3d", "reuse3d", "adjoint3d", "block3d", "build3d", "build_aniso"):
        c["s"] = rng.randint(1, 10)
        c["precision"] = rng.randint(0, 1)
    if kind in ("solve2d", "solve3d", "repair3d", "reuse3d", "adjoint3d"):
        c["krylov"] = "gmres" if c["precision"] else rng.choice(("bicgstab", "gmres", "bicgstab"))
        if c["krylov"] == "gmres" and not c["precision"] and kind != "solve2d" and c["m"] > 42:
            c["m"] = rng.randint(20, 42)  # FP64 GMRES on the larger grids costs more than the largest listed case
        if c["krylov"] == "gmres" and kind == "solve2d" and c["m"] > 90:
            c["m"] = rng.randint(45, 90)  # restarted GMRES takes thousands of steps on larger 2D grids
    if kind == "block3d":
        c["krylov"] = "bgmres"
        if not c["precision"] and c["m"] > 22:
            c["m"] = rng.randint(11, 22)
    if kind in ("build_aniso", "many_zipf", "grad_zipf"):
        c["sai"] = "spai"
    if kind == "batch":
        c.update(sai="spai", count=rng.randint(3, 24), nmin=rng.randint(300, 1000), precision=rng.randint(0, 1))
    return c


# ------------------------------------------------------------------ matrices
def _csc(n, rows, cols, vals):
    """Canonical CSC on the device; of entries at one place the first stays."""
    key = torch.from_numpy(cols.astype(np.int64) * n + rows.astype(np.int64)).cuda()
    key, at = torch.sort(key, stable=True)
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    key = key[first]
    v = torch.from_numpy(np.ascontiguousarray(vals, dtype=np.float64)).cuda()[at][first]
    col, row = key // n, key % n
    cp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    cp[1:] = torch.cumsum(torch.bincount(col, minlength=n), 0)
    return sai.CscMatrix(n, cp, row.to(torch.int32).contiguous(), v.contiguous())


def _host(A):
    """(rows, cols, vals) of a device matrix as numpy arrays, column by column."""
    cp = A.col_ptr.cpu().numpy()
    return A.row_idx.cpu().numpy().astype(np.int64), np.repeat(np.arange(A.n), np.diff(cp)), A.val.cpu().numpy()


def _times(A, x):
    """A x in a fixed order of summation."""
    r, c, v = _host(A)
    return np.bincount(r, weights=v * x[c], minlength=A.n)


def _times_t(A, x):
    r, c, v = _host(A)
    return np.bincount(c, weights=v * x[r], minlength=A.n)


def _stencil(m, dim, pe=10.0):
    """Upwind convection-diffusion on an m^dim grid, scaled by h^2."""
    h, n = 1.0 / (m + 1), m ** dim
    idx = np.arange(n, dtype=np.int64)
    rows, cols, vals = [idx], [idx], [np.full(n, 2.0 * dim + h * dim * pe)]
    for d in range(dim):
        st = m ** d
        c = (idx // st) % m
        lo, hi = idx[c > 0], idx[c < m - 1]
        rows += [lo, hi]
        cols += [lo - st, hi + st]
        vals += [np.full(lo.size, -1.0 - h * pe), np.full(hi.size, -1.0)]
    return n, rows, cols, vals


def _aniso(m, eps=1e-3, degrees=30.0):
    """Rotated anisotropic diffusion, 9-point, on m x m, scaled by h^2."""
    c, s = math.cos(math.radians(degrees)), math.sin(math.radians(degrees))
    k11, k22, k12 = c * c + eps * s * s, s * s + eps * c * c, (1.0 - eps) * c * s
    n = m * m
    idx = np.arange(n, dtype=np.int64)
    x, y = idx % m, idx // m
    rows, cols, vals = [idx], [idx], [np.full(n, 2.0 * (k11 + k22))]
    for dx, dy, v in ((-1, 0, -k11), (1, 0, -k11), (0, -1, -k22), (0, 1, -k22),
                      (1, 1, -0.5 * k12), (-1, -1, -0.5 * k12), (1, -1, 0.5 * k12), (-1, 1, 0.5 * k12)):
        ok = idx[(x + dx >= 0) & (x + dx < m) & (y + dy >= 0) & (y + dy < m)]
        rows.append(ok)
        cols.append(ok + dx + dy * m)
        vals.append(np.full(ok.size, v))
    return n, rows, cols, vals


def _with_dense(body, s, density, rng, scale=None):
    """The body's entries plus s columns with round(density n) further entries, N(0,1) at random rows outside the
    column's pattern; scale: sum |added| = scale |a_jj|."""
    n, rows, cols, vals = body
    diag = float(vals[0][0])
    dense = np.sort(rng.choice(n, size=s, replace=False))
    at = np.concatenate(cols)
    pattern = np.concatenate(rows)
    rows, cols, vals = list(rows), list(cols), list(vals)
    for j in dense:
        free = np.setdiff1d(np.arange(n), pattern[at == j], assume_unique=True)
        r = rng.choice(free, size=max(1, round(density * n)), replace=False)
        v = rng.standard_normal(r.size)
        if scale is not None:
            v *= scale * diag / np.abs(v).sum()
        rows.append(r)
        cols.append(np.full(r.size, j))
        vals.append(v)
    return _csc(n, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals))


def _zipf(n, rng):
    """Column j: min(Zipf(1.5), cap) random rows (one in each of as many strata of rows), N(0,1) values,
    a_jj = 1.2 sum |a_ij|. The column counts are the same for every seed."""
    count = np.minimum(np.random.default_rng(n).zipf(1.5, size=n), min(5000, n // 2))
    cols = np.repeat(np.arange(n), count)
    t = np.arange(cols.size) - np.repeat(np.cumsum(count) - count, count)
    k = count[cols]
    lo, hi = -(-(t * (n - 1)) // k), -(-((t + 1) * (n - 1)) // k)
    rows = lo + np.floor(rng.random(cols.size) * (hi - lo)).astype(np.int64)
    rows += rows >= cols
    vals = rng.standard_normal(cols.size)
    diag = 1.2 * np.bincount(cols, weights=np.abs(vals), minlength=n) + 1e-3
    idx = np.arange(n)
    return _csc(n, np.concatenate([idx, rows]), np.concatenate([idx, cols]), np.concatenate([diag, vals]))


def _rgg(n, rng, smax=20):
    """Perturbed Laplacian of a random geometric graph of average degree 8, raised to column dominance, plus up to
    smax dense columns."""
    pts = torch.from_numpy(rng.random((n, 2))).cuda()
    at = []
    for b in range(0, n, 2048):
        q = pts[b:b + 2048]
        d2 = (q[:, None, 0] - pts[None, :, 0]) ** 2 + (q[:, None, 1] - pts[None, :, 1]) ** 2
        i, j = torch.nonzero(d2 < 8.0 / (math.pi * n), as_tuple=True)
        at.append(torch.stack([i + b, j]))
    at = torch.cat(at, 1).cpu().numpy()
    r, c = at[:, at[0] != at[1]]
    deg = np.bincount(r, minlength=n).astype(np.float64)
    v = -1.0 + rng.uniform(-0.1, 0.1, size=r.size) * deg[r]
    density = float(rng.uniform(0.01, 0.10))
    for j in rng.choice(n, size=int(rng.integers(1, smax + 1)), replace=False):
        k = np.nonzero(rng.random(n) < density)[0]
        k = k[k != j]
        r, c, v = np.concatenate([r, k]), np.concatenate([c, np.full(k.size, j)]), \
            np.concatenate([v, rng.standard_normal(k.size)])
    off = np.bincount(c, weights=np.abs(v), minlength=n)
    idx = np.arange(n)
    return _csc(n, np.concatenate([idx, r]), np.concatenate([idx, c]), np.concatenate([np.maximum(1.05 * off, 1.0), v]))


def _smooth(n, rng):
    """A smooth solution around 1, as a field on an ordered grid has it."""
    t = np.arange(n) / n
    x = np.ones(n)
    for f in (1, 2, 3):
        x += 0.2 / f * np.sin(2.0 * np.pi * f * t + rng.uniform(0, 2.0 * np.pi))
    return x


def _matrix(case, rng):
    kind = case["kind"]
    if kind == "solve2d":
        return _with_dense(_stencil(case["m"], 2), case["s"], 0.3, rng)
    if kind == "build_aniso":
        return _with_dense(_aniso(case["m"]), case["s"], 0.02, rng)
    if kind in ("grad_zipf", "many_zipf"):
        return _zipf(case["n"], rng)
    A = _with_dense(_stencil(case["m"], 3), case["s"], 0.05 if case["m"] >= 20 else 0.2, rng, scale=0.5)
    if kind == "repair3d":  # a cycle over 5% of the rows puts zeros on the diagonal
        r, c, v = _host(A)
        moved = rng.choice(A.n, size=max(2, A.n // 20), replace=False)
        to = np.arange(A.n)
        to[np.roll(moved, -1)] = moved
        A = _csc(A.n, to[r], c, v)
    return A


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _build_options(case):
    grid3 = case["kind"] in ("solve3d", "repair3d", "reuse3d", "adjoint3d", "block3d", "build3d")
    if case["sai"] == "spai":
        return dict(delta=0.3 if grid3 else 0.4, mn=5, max_aug=10)
    return dict(delta=0.3 if grid3 else 0.4, tol=1e-3, tol_mode=1, lmax=10)


def _solve_options(case):
    # the refined Krylov form (FP32 inner solves) is GMRES's
    refined = int(case.get("krylov") in ("gmres", "bgmres") and case["precision"] == 1)
    return dict(krylov=case.get("krylov", "bicgstab"), eps=_EPS.get(case["kind"], 1e-12), maxit=4000, restart=50,
                krylov_precision=refined)


def _build(case, sp):
    make = sai.build_spai if case["sai"] == "spai" else sai.build_psai
    return make(sp, precision=case.get("precision", 0), **_build_options(case))


def _batch_orders(case):
    """Orders spread over [nmin, nmax], the same for every seed."""
    return [int(v) for v in np.random.default_rng(case["nmax"]).integers(case["nmin"], case["nmax"] + 1,
                                                                        size=case["count"])]


def _whole(case, M):
    """M's entries at the head of arrays with room for the largest M of the options, so that their lengths do not
    depend on the values."""
    room = _ROOM[case["sai"]] * M.n
    rows = torch.full((room,), -1, dtype=torch.int32, device="cuda")
    vals = torch.zeros(room, dtype=torch.float64, device="cuda")
    rows[:M.nnz] = M.row_idx
    vals[:M.nnz] = M.val
    return {"col_ptr": M.col_ptr, "row_idx": rows, "val": vals}


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "batch":
        As = [_rgg(n, rng) for n in _batch_orders(case)]
        bs = [_dev(_times(A, _smooth(A.n, rng))) for A in As]
        return dict(case=case, As=As, bs=bs)
    A = _matrix(case, rng)
    st = dict(case=case, A=A)
    if kind in ("build3d", "build_aniso"):
        return st
    x = _smooth(A.n, rng)
    st["b"] = _dev(_times(A, x))
    if kind in ("reuse3d", "many_zipf", "adjoint3d"):
        st["sp"] = sai.split(A, abs_tau=200.0 if kind == "many_zipf" else -1.0)
        st["P"] = _build(case, st["sp"])
    if kind in ("adjoint3d", "grad_zipf"):
        st["x"] = _dev(x)
        st["g"] = _dev(_times_t(A, _smooth(A.n, rng)))  # dL/dx
    if kind == "grad_zipf":
        st["val"] = A.val.detach().clone().requires_grad_(True)
        st["b"].requires_grad_(True)
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind in ("solve2d", "solve3d", "repair3d", "block3d"):
        x, _, _ = sai.solve(st["A"], st["b"], sai=case["sai"], sai_precision=case["precision"],
                            zero_diag=kind == "repair3d", **_build_options(case), **_solve_options(case))
        return {"x": x}
    if kind == "reuse3d":
        x, _, _ = sai.solve_with(st["A"], st["sp"], st["P"], st["b"], **_solve_options(case))
        return {"x": x}
    if kind == "many_zipf":
        x, _, _ = sai.solve_with(st["A"], st["sp"], st["P"], st["b"], **_solve_options(case))
        return {"x": x}
    if kind == "adjoint3d":
        lam, gv, _, _ = sai.backward(st["A"], st["sp"], st["P"], st["x"], st["g"], **_solve_options(case))
        return {"lambda": lam, "grad_vals": gv}
    if kind in ("build3d", "build_aniso"):
        sp = sai.split(st["A"])
        M, loops, res, post = _build(case, sp).arrays()
        return dict(_whole(case, M), loops=loops, res=res, res_post=post)
    if kind == "grad_zipf":
        st["val"].grad = st["b"].grad = None
        opts = dict(_build_options(case), sai=case["sai"], abs_tau=200.0, krylov="bicgstab", eps=_EPS[kind], maxit=4000)
        x = sai.SparseSolve.apply(st["A"].col_ptr, st["A"].row_idx, st["val"], st["b"], opts)
        x.backward(st["g"])
        return {"x": x.detach(), "grad_vals": st["val"].grad, "grad_b": st["b"].grad}
    xs, _, _ = sai.solve_batched(st["As"], st["bs"], sai=case["sai"], sai_precision=case["precision"], eps=1e-12,
                                 maxit=4000, **_build_options(case))
    return {"x": xs}


def exact(case, seed):
    """The chosen solution (the right-hand side is A times it), and for the gradients lambda = A^-T g and
    dL/dA_ij = -lambda_i x_j; M has no closed form."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind in ("build3d", "build_aniso"):
        return None
    if kind == "batch":
        As = [_rgg(n, rng) for n in _batch_orders(case)]
        return {"x": [_dev(_smooth(A.n, rng)) for A in As]}
    A = _matrix(case, rng)
    x = _smooth(A.n, rng)
    if kind not in ("adjoint3d", "grad_zipf"):
        return {"x": _dev(x)}
    lam = _smooth(A.n, rng)
    r, c, _ = _host(A)
    gv = _dev(-lam[r] * x[c])
    if kind == "adjoint3d":
        return {"lambda": _dev(lam), "grad_vals": gv}
    return {"x": _dev(x), "grad_vals": gv, "grad_b": _dev(lam)}


def work(case):
    """Inputs and outputs once; flops: a nominal count of the Krylov iterations (by the grid's width) times the two
    products with A~ and M for every system, or the least squares of the build."""
    kind = case["kind"]
    if kind == "batch":
        n = 0.5 * (case["nmin"] + case["nmax"]) * case["count"]
        nnz, k, iters, passes = 9.5 * n, 10.0, 45.0, 2.0
    elif kind in ("grad_zipf", "many_zipf"):
        n = float(case["n"])
        nnz, k, iters = 2.6 * math.sqrt(min(5000.0, n / 2)) * n * 0.75, 0.053 * n + 1.0, 25.0
        passes = 2.0 if kind == "many_zipf" else 4.0
    else:
        dim = 2 if kind in ("solve2d", "build_aniso") else 3
        n = float(case["m"]) ** dim
        density = {"solve2d": 0.3, "build_aniso": 0.02}.get(kind, 0.05 if case["m"] >= 20 else 0.2)
        nnz = {"solve2d": 5.0, "build_aniso": 9.0}.get(kind, 7.0) * n + case["s"] * density * n
        if kind in ("build3d", "build_aniso"):
            per = 8.0 if kind == "build3d" else 30.0  # entries of a column of M
            # Householder on |L| x |S| with |L| about three times |S|, per column
            return {"bytes": 12.0 * nnz + 12.0 * per * n + 24.0 * n, "flops": n * (6.0 * per ** 3)}
        k, iters = case["s"] + 1.0, 3.0 * case["m"]
        passes = 2.0 if case["krylov"] == "bicgstab" else 1.0
    body = 7.0 * n if kind not in ("grad_zipf", "many_zipf") else 15.0 * n
    return {"bytes": 12.0 * nnz + 8.0 * n + 8.0 * n * (1.0 if passes < 4.0 else 3.0),
            "flops": k * iters * passes * 2.0 * (2.0 * body + 5.0 * n)}
