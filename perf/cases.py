"""Performance cases of the sparse path, run through the public entry points
of ``paper_2006_14290_gb300.gko``: SpMV per format and value type, the Krylov
solvers, the batched solver and the request server.

A case is a dict of plain values; ``prepare`` makes its inputs from the seed
on the GPU (the matrix families of ``inputs.py``, generated with torch),
``run`` is one call of a user's program, ``exact`` the same result in 64-bit
torch arithmetic without the library, ``work`` the bytes and floating-point
operations the call cannot do without.

Solves come in two forms.  ``iters`` > 0: a fixed number of iterations (the
paper times 1,000 CG iterations; the tolerance 0 never stops early).
``iters`` = 0: to ``tol``, with b = A v for a known v, so the exact result is v.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2006_14290_gb300 import gko as G

# row lengths clip(ceil(lam Z), 1, 1e4), Z ~ Zipf(2): mean 6.5 (lam = 1) and 16 (lam = 2.65)
ZIPF_MEAN = {1.0: 6.5, 2.65: 16.0}
BAND_HALF, BAND_FILL = 64, 0.3
L2_BYTES = 126e6


def listed():
    return [
        # the smallest call: one SpMV of the 64 x 64 grid Laplacian
        dict(name="spmv_csr_f64_lap64", kind="spmv", matrix="lap2d", side=64, fmt="csr", dtype="f64", general=False),
        # the sweep's large regular matrix in the default format
        dict(name="spmv_csr_f64_27pt_128", kind="spmv", matrix="s27", side=128, fmt="csr", dtype="f64", general=False),
        # COO (the paper's format), ragged rows of about 39
        dict(name="spmv_coo_f64_banded_1m", kind="spmv", matrix="banded", side=1_000_000, fmt="coo", dtype="f64",
             general=False),
        # skewed rows, FP32: graph-like matrices
        dict(name="spmv_csr_f32_power16_1m", kind="spmv", matrix="power16", side=1_000_000, fmt="csr", dtype="f32",
             general=False),
        # hybrid ELL + COO on skewed rows, y = alpha A x + beta y
        dict(name="spmv_hybrid_f64_power_1m", kind="spmv", matrix="power", side=1_000_000, fmt="hybrid", dtype="f64",
             general=True),
        # the smallest solve
        dict(name="cg_f64_lap64", kind="solve", solver="cg", matrix="lap2d", side=64, fmt="csr", precision="f64",
             precond="none", iters=0, peclet=0.0),
        # the paper's measurement: a fixed number of CG iterations on a large 7-point Poisson matrix
        dict(name="cg_f64_poisson256_100it", kind="solve", solver="cg", matrix="s7", side=256, fmt="csr",
             precision="f64", precond="none", iters=100, peclet=0.0),
        # a nonsymmetric system of the size most serving requests have, odd side
        dict(name="bicgstab_f64_convdiff31", kind="solve", solver="bicgstab", matrix="convdiff", side=31, fmt="csr",
             precision="f64", precond="none", iters=0, peclet=1.0),
        # restarted GMRES, three cycles, on a large convection-diffusion matrix
        dict(name="gmres_f64_convdiff128_90it", kind="solve", solver="gmres", matrix="convdiff", side=128, fmt="csr",
             precision="f64", precond="none", iters=90, peclet=10.0),
        # the solver users of mixed precision run: Jacobi CG, FP32 recurrences, FP64 solution
        dict(name="cg_mixed_jacobi_varcoef128", kind="solve", solver="cg", matrix="varcoef", side=128, fmt="csr",
             precision="f32", precond="jacobi", iters=0, peclet=0.0),
        # thousands of small independent systems in one call
        dict(name="batch_mixed_4096", kind="batch", count=4096, lo=8, hi=64, precision="f32"),
        # a burst of requests of mixed sizes, solvers and precisions against resident matrices
        dict(name="serve_burst_24", kind="serve", requests=24, pool=8, lo=10, hi=60, slots=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmv"] * 6 + ["solve"] * 5 + ["batch", "serve"])
    if kind == "spmv":
        matrix = rng.choice(["lap2d", "s7", "s27", "banded", "power", "power16"])
        side = {"lap2d": (20, 1000), "s7": (10, 160), "s27": (8, 120), "banded": (1000, 900_000),
                "power": (2000, 1_000_000), "power16": (2000, 1_000_000)}[matrix]
        formats = ["csr", "csr", "coo", "hybrid"] + ([] if matrix.startswith("power") else ["ell", "sellp"])
        return dict(kind="spmv", matrix=matrix, side=_log_int(rng, *side), fmt=rng.choice(formats),
                    dtype=rng.choice(["f64", "f64", "f32", "f32", "bf16"]), general=rng.random() < 0.25)
    if kind == "solve":
        solver = rng.choice(["cg", "cg", "bicgstab", "bicgstab", "gmres"])
        fixed = rng.random() < 0.4
        if solver == "cg":
            matrix = rng.choice(["lap2d", "s7", "varcoef"])
        else:
            matrix = "convdiff"
        side = _log_int(rng, *((20, 300) if matrix == "lap2d" else (10, 100)))
        precision = "f64" if fixed else rng.choice(["f64", "f64", "f32"])
        precond = "none" if solver == "gmres" else rng.choice(["none", "none", "jacobi", "bjacobi"])
        fmt = "csr" if precond == "bjacobi" else rng.choice(["csr", "csr", "csr", "ell", "sellp"])
        # BiCGSTAB's iterates keep few digits of their rounding after many steps, GMRES fills whole cycles
        iters = 0 if not fixed else {"cg": rng.randint(40, 160), "bicgstab": rng.randint(8, 24),
                                     "gmres": 30 * rng.randint(1, 3)}[solver]
        return dict(kind="solve", solver=solver, matrix=matrix, side=side, fmt=fmt, precision=precision,
                    precond=precond, iters=iters, peclet=round(rng.uniform(0.5, 2.0), 2) if matrix == "convdiff" else 0.0)
    if kind == "batch":
        return dict(kind="batch", count=_log_int(rng, 64, 4096), lo=rng.randint(5, 12), hi=rng.randint(30, 64),
                    precision=rng.choice(["f64", "f32"]))
    return dict(kind="serve", requests=rng.randint(8, 24), pool=rng.randint(4, 8), lo=rng.randint(8, 14),
                hi=rng.randint(30, 60), slots=rng.choice([4, 8]))


# ------------------------------------------------------------------ matrices --

DIAG = {"lap2d": 4.0, "s7": 6.0, "s27": 26.0}
TORCH = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.float32}


def _gen(seed, what):
    """A torch generator on the GPU for one of the inputs of a seed."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * (seed % (1 << 40)) + what)
    return g


def _uniform(n, lo, hi, gen):
    return torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) * (hi - lo) + lo


def _offsets(matrix):
    """Stencil offsets (x fastest) in ascending column order."""
    dims = 2 if matrix == "lap2d" else 3
    near = [-1, 0, 1]
    offs = [(i, j, k) for k in (near if dims == 3 else [0]) for j in near for i in near]
    if matrix != "s27":
        offs = [o for o in offs if abs(o[0]) + abs(o[1]) + abs(o[2]) <= 1]
    return offs


def _stencil(matrix, side, peclet, gen):
    """(n, S) slots of a stencil matrix: columns, values, which are present."""
    offs = _offsets(matrix)
    nx, ny, nz = side, side, 1 if matrix == "lap2d" else side
    n = nx * ny * nz
    i = torch.arange(n, dtype=torch.int32, device="cuda")
    xyz = (i % nx, (i // nx) % ny, i // (nx * ny))
    cols = torch.empty((n, len(offs)), dtype=torch.int32, device="cuda")
    vals = torch.empty((n, len(offs)), dtype=torch.float64, device="cuda")
    valid = torch.empty((n, len(offs)), dtype=torch.bool, device="cuda")
    # variable coefficients exp(N(0,1)) per cell, harmonic means on the faces
    coef = torch.randn(n, dtype=torch.float64, device="cuda", generator=gen).exp() if matrix == "varcoef" else None
    diag = torch.zeros(n, dtype=torch.float64, device="cuda") if coef is not None else None
    for s, o in enumerate(offs):
        ok = torch.ones(n, dtype=torch.bool, device="cuda")
        for c, d, m in zip(xyz, o, (nx, ny, nz)):
            if d:
                ok &= (c + d >= 0) & (c + d < m)
        nb = torch.where(ok, i + (o[0] + nx * (o[1] + ny * o[2])), i)
        cols[:, s] = nb
        valid[:, s] = ok
        if o == (0, 0, 0):
            centre = s
            vals[:, s] = DIAG.get(matrix, 6.0 + 3.0 * peclet)
        elif coef is not None:
            other = coef[nb.long()]
            face = torch.where(ok, 2.0 * coef * other / (coef + other), coef)
            diag += face
            vals[:, s] = -face
        else:
            vals[:, s] = -1.0 - (peclet if min(o) < 0 else 0.0)
    if coef is not None:
        vals[:, centre] = diag
    return cols, vals, valid


def _arrays(case, seed):
    """CSR arrays (row_ptr, col, val) on the GPU, FP64 values."""
    m, n = case["matrix"], case["side"]
    if m in ("power", "power16"):
        lam = 2.65 if m == "power16" else 1.0
        z = np.random.default_rng(seed).zipf(2.0, n).astype(np.float64)
        lens = torch.from_numpy(np.clip(np.ceil(lam * z), 1, min(10000, n)).astype(np.int64)).cuda()
        nnz = int(lens.sum())
        g = _gen(seed, 1)
        col = torch.randint(0, n, (nnz,), dtype=torch.int32, device="cuda", generator=g)
        val = torch.randn(nnz, dtype=torch.float64, device="cuda", generator=g)
    elif m == "banded":
        g = _gen(seed, 1)
        offs = torch.arange(-BAND_HALF, BAND_HALF + 1, dtype=torch.int32, device="cuda")
        cols = torch.arange(n, dtype=torch.int32, device="cuda")[:, None] + offs[None, :]
        valid = torch.rand((n, offs.numel()), dtype=torch.float32, device="cuda", generator=g) < BAND_FILL
        valid[:, BAND_HALF] = True
        valid &= (cols >= 0) & (cols < n)
        lens, col = valid.sum(1), cols[valid]
        val = _uniform(col.numel(), -1.0, 1.0, g)
    else:
        cols, vals, valid = _stencil(m, n, case.get("peclet", 0.0), _gen(seed, 1))
        lens, col, val = valid.sum(1), cols[valid], vals[valid]
    rp = torch.zeros(lens.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=rp[1:])
    return rp.to(torch.int32), col.contiguous(), val.contiguous()


def _product(rp, col, val, x):
    """A x in 64 bits with torch."""
    return torch.segment_reduce(val * x[col.long()], "sum", lengths=(rp[1:] - rp[:-1]).long(), initial=0.0)


def _handle(rp, col, val, fmt, dtype):
    n = rp.numel() - 1
    if dtype == "f32":
        M = G.gko_matrix_create_csr(n, n, rp, col, val.float(), G.F32)
    else:
        M = G.gko_matrix_create_csr(n, n, rp, col, val, G.F64)
        if dtype == "bf16":
            M = G.gko_matrix_convert_values(M, G.BF16)
    convert = {"ell": G.gko_matrix_convert_to_ell, "coo": G.gko_matrix_convert_to_coo,
               "hybrid": G.gko_matrix_convert_to_hybrid, "sellp": G.gko_matrix_convert_to_sellp}
    return convert[fmt](M) if fmt in convert else M


# ---------------------------------------------------------------------- SpMV --

def _scalars(case):
    return (-0.75, 1.5) if case["general"] else (1.0, 0.0)


def _spmv_vectors(case, seed, n):
    g = _gen(seed, 2)
    x, y = _uniform(n, -1.0, 1.0, g), _uniform(n, -1.0, 1.0, g)
    return x.to(TORCH[case["dtype"]]), y.to(TORCH[case["dtype"]])


def _prepare_spmv(case, seed):
    rp, col, val = _arrays(case, seed)
    x, y0 = _spmv_vectors(case, seed, rp.numel() - 1)
    M = _handle(rp, col, val, case["fmt"], case["dtype"])
    return dict(M=M, x=x, y0=y0, y=torch.zeros_like(y0))


def _run_spmv(case, st):
    alpha, beta = _scalars(case)
    if case["general"]:  # a fresh y each pass: beta y is read
        st["y"].copy_(st["y0"])
    return G.gko_spmv(alpha, st["M"], st["x"], beta, st["y"])


def _exact_spmv(case, seed):
    rp, col, val = _arrays(case, seed)
    x, y0 = _spmv_vectors(case, seed, rp.numel() - 1)
    if case["dtype"] != "f64":
        val = (val.to(torch.bfloat16) if case["dtype"] == "bf16" else val.float()).double()
    alpha, beta = _scalars(case)
    y = alpha * _product(rp, col, val, x.double())
    return y + beta * y0.double() if beta else y


def _rows_nnz(case):
    m, s = case["matrix"], case["side"]
    if m in ("power", "power16"):
        return s, ZIPF_MEAN[2.65 if m == "power16" else 1.0] * s
    if m == "banded":
        return s, (1.0 + 2 * BAND_HALF * BAND_FILL) * s
    if m == "lap2d":
        return s * s, 5.0 * s * s - 4 * s
    if m == "s27":
        return s ** 3, float((3 * s - 2) ** 3)
    return s ** 3, 7.0 * s ** 3 - 6 * s * s


def _work_spmv(case):
    n, nnz = _rows_nnz(case)
    sv = {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
    sx = 8 if case["dtype"] == "f64" else 4
    per = sv + (8 if case["fmt"] == "coo" else 4)
    fixed = 4 * n if case["fmt"] == "csr" else 0
    return dict(bytes=nnz * per + fixed + sx * n * (3 if case["general"] else 2), flops=2 * nnz)


# ------------------------------------------------------------------- solvers --

SOLVE = {"cg": G.gko_solve_cg, "bicgstab": G.gko_solve_bicgstab, "gmres": G.gko_solve_gmres}
TOL = 1e-12


def _opts(precision, precond):
    return G.opts(precision=G.PRECISION_MIXED_F32 if precision == "f32" else G.PRECISION_F64,
                  preconditioner={"none": G.PRECOND_NONE, "jacobi": G.PRECOND_JACOBI,
                                  "bjacobi": G.PRECOND_BLOCK_JACOBI}[precond])


def _solution(n, seed):
    return _uniform(n, 0.5, 1.5, _gen(seed, 3))


def _prepare_solve(case, seed):
    rp, col, val = _arrays(case, seed)
    n = rp.numel() - 1
    b = _product(rp, col, val, _solution(n, seed))
    return dict(M=_handle(rp, col, val, case["fmt"], "f64"), b=b, x=torch.zeros_like(b),
                opts=_opts(case["precision"], case["precond"]))


def _run_solve(case, st):
    st["x"].zero_()
    tol, cap = (0.0, case["iters"]) if case["iters"] else (TOL, 20000)
    res = SOLVE[case["solver"]](st["M"], st["b"], st["x"], tol, cap, st["opts"])
    return dict(x=st["x"], status=res.status)


def _preconditioner(case, rp, col, val):
    """v -> M^-1 v in 64 bits (diagonal, or diagonal blocks of 8 rows)."""
    n = rp.numel() - 1
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
    cl = col.long()
    if case["precond"] == "jacobi":
        d = torch.zeros(n, dtype=torch.float64, device="cuda")
        at = rows == cl
        d[rows[at]] = val[at]
        return lambda v: v / d
    if case["precond"] == "bjacobi":
        nb = -(-n // 8)
        D = torch.eye(8, dtype=torch.float64, device="cuda").repeat(nb, 1, 1)
        at = (rows // 8) == (cl // 8)
        D[rows[at] // 8, rows[at] % 8, cl[at] % 8] = val[at]
        inv = torch.linalg.inv(D)
        pad = nb * 8 - n
        return lambda v: (inv @ torch.nn.functional.pad(v, (0, pad)).view(nb, 8, 1)).reshape(-1)[:n]
    return lambda v: v


def _plain_cg(mul, prec, b, iters):
    x, r = torch.zeros_like(b), b.clone()
    z = prec(r)
    p, rho = z.clone(), torch.dot(r, z)
    for _ in range(iters):
        q = mul(p)
        a = rho / torch.dot(p, q)
        x += a * p
        r -= a * q
        z = prec(r)
        new = torch.dot(r, z)
        p = z + (new / rho) * p
        rho = new
    return x


def _plain_bicgstab(mul, prec, b, iters):
    x, r, rh = torch.zeros_like(b), b.clone(), b.clone()
    p, rho = r.clone(), torch.dot(rh, r)
    for _ in range(iters):
        ph = prec(p)
        v = mul(ph)
        a = rho / torch.dot(rh, v)
        s = r - a * v
        sh = prec(s)
        t = mul(sh)
        w = torch.dot(t, s) / torch.dot(t, t)
        x += a * ph + w * sh
        r = s - w * t
        new = torch.dot(rh, r)
        p = r + (new / rho) * (a / w) * (p - w * v)
        rho = new
    return x


def _plain_gmres(mul, b, iters, m=30):
    x = torch.zeros_like(b)
    for start in range(0, iters, m):
        r = b - mul(x)
        beta = torch.linalg.norm(r)
        k = min(m, iters - start)
        V = torch.empty((k + 1, b.numel()), dtype=torch.float64, device="cuda")
        H = torch.zeros((k + 1, k), dtype=torch.float64, device="cuda")
        V[0] = r / beta
        for j in range(k):
            w = mul(V[j])
            for _ in range(2):
                h = V[:j + 1] @ w
                w -= h @ V[:j + 1]
                H[:j + 1, j] += h
            H[j + 1, j] = torch.linalg.norm(w)
            V[j + 1] = w / H[j + 1, j]
        e = torch.zeros((k + 1, 1), dtype=torch.float64, device="cuda")
        e[0] = beta
        Q, R = torch.linalg.qr(H)
        x += torch.linalg.solve_triangular(R, Q.T @ e, upper=True).flatten() @ V[:k]
    return x


def _exact_solve(case, seed):
    rp, col, val = _arrays(case, seed)
    v = _solution(rp.numel() - 1, seed)
    if not case["iters"]:
        return dict(x=v, status=None)

    def mul(u):
        return _product(rp, col, val, u)

    b = mul(v)
    if case["solver"] == "gmres":
        return dict(x=_plain_gmres(mul, b, case["iters"]), status=None)
    plain = _plain_cg if case["solver"] == "cg" else _plain_bicgstab
    return dict(x=plain(mul, _preconditioner(case, rp, col, val), b, case["iters"]), status=None)


def _iterations(solver, matrix, side, precond):
    """About how many iterations a solve to TOL takes."""
    if solver == "cg":
        return {"lap2d": 4.1, "s7": 3.6, "varcoef": 12.0 if precond == "none" else 5.0}[matrix] * side + 20
    return (3.6 if solver == "bicgstab" else 6.0) * side + 20


def _work_solve(case):
    n, nnz = _rows_nnz(case)
    it = case["iters"] or _iterations(case["solver"], case["matrix"], case["side"], case["precond"])
    low = case["precision"] == "f32"
    sv = 4 if low else 8
    # per iteration: products, and vector passes (CG: q written, x, r, p read and written, q read;
    # BiCGSTAB twice that; GMRES: the basis read twice, 16 vectors on average)
    products = 2 if case["solver"] == "bicgstab" else 1
    passes = {"cg": 8, "bicgstab": 14, "gmres": 34}[case["solver"]]
    matrix, vector = nnz * (sv + 4) + 4 * n, sv * n
    per = products * matrix + passes * vector
    resident = matrix + 4 * vector < L2_BYTES  # stays on the chip: read once
    once = nnz * 12 + 4 * n + 16 * n
    return dict(bytes=once + (0 if resident else it * per),
                flops=it * (2 * nnz * products + n * {"cg": 10, "bicgstab": 20, "gmres": 66}[case["solver"]]))


# --------------------------------------------------------------------- batch --

class _System:
    """What gko.Batch takes: host CSR of one system."""

    def __init__(self, rp, col, val):
        self.n_rows, self.row_ptr, self.col, self.val = rp.size - 1, rp, col, val


def _batch_sides(case):
    # the sizes belong to the workload, the coefficients and right-hand sides to the seed
    r = np.random.default_rng(case["count"])
    return np.rint(np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), case["count"]))).astype(np.int64)


def _batch_systems(case, seed):
    """2D 5-point variable-coefficient systems, one coefficient per cell."""
    sides, rng = _batch_sides(case), np.random.default_rng(seed)
    systems = [None] * case["count"]
    for s in np.unique(sides):
        at, n = np.flatnonzero(sides == s), int(s * s)
        c = np.exp(rng.standard_normal((at.size, s, s)))
        i = np.arange(n, dtype=np.int32).reshape(s, s)
        cols, vals, valid = [], [], []
        diag = np.zeros_like(c)
        for dy, dx in ((-1, 0), (0, -1), (0, 0), (0, 1), (1, 0)):
            ok = np.zeros((s, s), bool)
            here = (slice(max(0, -dy), s - max(0, dy)), slice(max(0, -dx), s - max(0, dx)))
            there = (slice(max(0, dy), s + min(0, dy)), slice(max(0, dx), s + min(0, dx)))
            ok[here] = True
            cols.append(i + dy * s + dx)
            valid.append(ok)
            if (dy, dx) == (0, 0):
                vals.append(diag)
                continue
            face = c.copy()
            a, b = c[(slice(None),) + here], c[(slice(None),) + there]
            face[(slice(None),) + here] = 2.0 * a * b / (a + b)
            diag += face
            vals.append(-face)
        keep = np.stack(valid, -1).reshape(-1)
        col = np.ascontiguousarray(np.stack(cols, -1).reshape(-1)[keep])
        rp = np.concatenate([[0], np.cumsum(keep.reshape(n, 5).sum(1))]).astype(np.int32)
        val = np.ascontiguousarray(np.stack(vals, -1).reshape(at.size, -1)[:, keep])
        for j, k in enumerate(at):
            systems[k] = _System(rp, col, val[j])
    return systems


def _batch_arrays(systems):
    """The systems as one block-diagonal CSR on the GPU."""
    lens = np.concatenate([np.diff(s.row_ptr) for s in systems])
    rp = torch.from_numpy(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)).cuda()
    off = np.cumsum([0] + [s.n_rows for s in systems])
    col = torch.from_numpy(np.concatenate([s.col + o for s, o in zip(systems, off)]).astype(np.int32)).cuda()
    return rp, col, torch.from_numpy(np.concatenate([s.val for s in systems])).cuda()


def _prepare_batch(case, seed):
    systems = _batch_systems(case, seed)
    rp, col, val = _batch_arrays(systems)
    b = _product(rp, col, val, _solution(rp.numel() - 1, seed))
    B = G.Batch(systems)
    if case["precision"] == "f32":
        B.set_precision(G.PRECISION_MIXED_F32)
    return dict(B=B, b=b, x=torch.zeros_like(b))


def _run_batch(case, st):
    st["x"].zero_()
    code, _, _, status = st["B"].cg(st["b"], st["x"], TOL, 20000)
    return dict(x=st["x"], code=code, status=status)


def _exact_batch(case, seed):
    n = int((_batch_sides(case) ** 2).sum())
    return dict(x=_solution(n, seed), code=None, status=None)


def _work_batch(case):
    s = _batch_sides(case).astype(np.float64)
    n, nnz = s * s, 5 * s * s - 4 * s
    it = 8.5 * s + 20
    return dict(bytes=float((nnz * 12 + n * 20).sum()), flops=float((it * (2 * nnz + 10 * n)).sum()))


# ------------------------------------------------------------------- serving --

def _serve_plan(case):
    """Per resident matrix its solver and side, per request its matrix and precision (parts of the workload)."""
    r = np.random.default_rng([case["requests"], case["pool"], case["hi"]])
    side = np.rint(np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), case["pool"]))).astype(int)
    mats = [dict(solver="cg" if k % 10 < 7 and k % 3 != 2 else "bicgstab", side=int(s)) for k, s in enumerate(side)]
    for m in mats:
        m["matrix"], m["peclet"] = ("varcoef", 0.0) if m["solver"] == "cg" else ("convdiff", 1.0)
    reqs = [(int(r.integers(case["pool"])), "f32" if q % 2 else "f64") for q in range(case["requests"])]
    return mats, reqs


def _serve_solutions(case, seed):
    mats, reqs = _serve_plan(case)
    return [_uniform(mats[k]["side"] ** 3, 0.5, 1.5, _gen(seed, 100 + q)) for q, (k, _) in enumerate(reqs)]


def _prepare_serve(case, seed):
    mats, reqs = _serve_plan(case)
    arrays = [_arrays(m, seed + 7919 * k) for k, m in enumerate(mats)]
    server = G.Server(slots=case["slots"])
    ids = [server.add_matrix(_handle(*a, "csr", "f64")) for a in arrays]
    calls = []
    for (k, precision), v in zip(reqs, _serve_solutions(case, seed)):
        cg = mats[k]["solver"] == "cg"
        calls.append((ids[k], 0 if cg else 1, _product(*arrays[k], v).cpu().numpy(),
                      _opts(precision, "jacobi" if cg else "none")))
    return dict(server=server, calls=calls)


def _run_serve(case, st):
    server = st["server"]
    ids = [server.submit(m, solver, b, TOL, 20000, o) for m, solver, b, o in st["calls"]]
    done = [server.result(i) for i in ids]
    return dict(x=[d[2] for d in done], status=np.array([d[0] for d in done], np.int32))


def _exact_serve(case, seed):
    return dict(x=_serve_solutions(case, seed), status=None)


def _work_serve(case):
    mats, reqs = _serve_plan(case)
    total = dict(bytes=0.0, flops=0.0)
    for k, precision in reqs:
        pc = "jacobi" if mats[k]["solver"] == "cg" else "none"
        w = _work_solve(dict(mats[k], precision=precision, precond=pc, iters=0))
        for f in total:
            total[f] += w[f]
    return total


# ----------------------------------------------------------------- interface --

def prepare(case, seed):
    make = {"spmv": _prepare_spmv, "solve": _prepare_solve, "batch": _prepare_batch, "serve": _prepare_serve}
    return dict(make[case["kind"]](case, seed), case=case)


def run(state):
    do = {"spmv": _run_spmv, "solve": _run_solve, "batch": _run_batch, "serve": _run_serve}
    return do[state["case"]["kind"]](state["case"], state)


def exact(case, seed):
    return {"spmv": _exact_spmv, "solve": _exact_solve, "batch": _exact_batch, "serve": _exact_serve}[case["kind"]](case, seed)


def work(case):
    return {"spmv": _work_spmv, "solve": _work_solve, "batch": _work_batch, "serve": _work_serve}[case["kind"]](case)
