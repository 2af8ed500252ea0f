"""The single-launch CG and BiCGSTAB at the edges of their launch shapes
(blocks of 32-512 rows in one cluster, then one block per SM) against the
oracle: both sides to 1e-12, solutions within 1e-8 (kappa * 1e-12 << 1e-8),
the reported residual the true one, as tests/test_gpu_solvers.py."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle as O
from gpu_util import dev, host
from paper_2006_14290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def banded_system(n, half, spd, seed):
    """Diagonally dominant band matrix: rows of 1 to 2*half+1 entries, ragged ends."""
    rng = np.random.default_rng(seed)
    offs = [k for k in range(-half, half + 1) if k == 0 or abs(k) in (1, half)]
    cols = np.arange(n)[:, None] + np.array(offs)[None, :]
    vals = rng.uniform(-1.0, -0.2, cols.shape)
    if spd:
        vals[:] = -1.0
    vals[:, offs.index(0)] = len(offs) - 1 + 0.5
    ok = (cols >= 0) & (cols < n)
    rp = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32)
    return I.Csr(n, n, rp, cols[ok].astype(np.int32), vals[ok], f"band_{n}")


def solve(G, name, M, b, tol=1e-12, maxit=3000, **opt):
    xd = dev(np.zeros(b.size))
    fn = G.gko_solve_cg if name == "cg" else G.gko_solve_bicgstab
    res = fn(M, dev(b), xd, tol, maxit, G.opts(**opt) if opt else None)
    return host(xd), res


def check(G, name, A, M, seed=1, **opt):
    b = np.random.default_rng(seed).uniform(-1, 1, A.n_rows)
    x, res = solve(G, name, M, b, **opt)
    xo, ro = O.solve(O.CG if name == "cg" else O.BICGSTAB, A, b, tol=1e-12, maxit=3000)
    assert res.status == G.OK and ro.status == 0, res
    assert np.linalg.norm(x - xo) <= 1e-8 * np.linalg.norm(xo)
    true = np.linalg.norm(b - O.spmv_csr(A, x)) / np.linalg.norm(b)
    assert true <= 1.01e-12 and abs(true - res.rel_residual) <= 1e-13
    return b, x


# block and cluster edges: 1 row, one warp, 16 blocks of 32/64/128/256/512 rows and one row more
SIZES = [1, 2, 31, 32, 33, 512, 513, 1024, 1025, 2048, 2049, 4096, 4097, 8192, 8193, 9729, 19457, 38913, 77825]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("name", ["cg", "bicgstab"])
def test_shape_edges(gko, name, n):
    G = gko
    A = banded_system(n, 7, name == "cg", n)
    b, x = check(G, name, A, G.from_csr(A))
    x2, _ = solve(G, name, G.from_csr(A), b)
    assert x.tobytes() == x2.tobytes()
    check(G, name, A, G.from_csr(A), precision=G.PRECISION_MIXED_F32, preconditioner=G.PRECOND_JACOBI)


@pytest.mark.parametrize("fmt", ["ell", "sellp32", "sellp128"])
@pytest.mark.parametrize("n", [700, 9001, 100003])
@pytest.mark.parametrize("name", ["cg", "bicgstab"])
def test_padded_formats(gko, name, n, fmt):
    """ELL and SELL-P (slices that end inside a block) against the same solve from CSR."""
    G = gko
    A = banded_system(n, 11, name == "cg", n)
    M = G.from_csr(A)
    M = G.gko_matrix_convert_to_ell(M) if fmt == "ell" else G.gko_matrix_convert_to_sellp(M, int(fmt[5:]))
    check(G, name, A, M)
    check(G, name, A, M, precision=G.PRECISION_MIXED_F32, refinement=G.REFINE_AUTO)


@pytest.mark.parametrize("name", ["cg", "bicgstab"])
def test_entries_that_do_not_fit_in_shared_memory(gko, name):
    """Rows of about 400 entries: read from the matrix every iteration."""
    G = gko
    n, half = 20000, 200
    rng = np.random.default_rng(4)
    cols = np.arange(n)[:, None] + np.arange(-half, half + 1)[None, :]
    vals = np.full(cols.shape, -1.0) if name == "cg" else rng.uniform(-1, 0, cols.shape)
    vals[:, half] = 2 * half + 1.0
    ok = (cols >= 0) & (cols < n)
    rp = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32)
    A = I.Csr(n, n, rp, cols[ok].astype(np.int32), vals[ok], "wide")
    check(G, name, A, G.from_csr(A))


@pytest.mark.parametrize("n", [300, 20000])
@pytest.mark.parametrize("name", ["cg", "bicgstab"])
def test_scaled_and_special_right_hand_sides(gko, name, n):
    """The sums keep their accuracy at any scale of b, zero stays zero, and
    infinities and NaN end the solve as the reductions in FP64 do."""
    G = gko
    A = banded_system(n, 7, name == "cg", 3)
    M = G.from_csr(A)
    b = np.random.default_rng(2).uniform(-1, 1, n)
    x1, r1 = solve(G, name, M, b)
    for k in (-400, -100, 100, 400):  # powers of two: the same digits
        xs, rs = solve(G, name, M, np.ldexp(b, k))
        assert rs.status == G.OK and rs.iterations == r1.iterations and np.array_equal(xs, np.ldexp(x1, k))
    xz, rz = solve(G, name, M, np.zeros(n))
    assert rz.status == G.OK and rz.iterations == 0 and np.all(xz == 0) and rz.rel_residual == 0
    bn = b.copy()
    bn[n // 2] = np.nan
    _, rn = solve(G, name, M, bn, maxit=5)
    assert rn.status in (G.BREAKDOWN, G.NOT_CONVERGED) and np.isnan(rn.rel_residual)
    bn[n // 2] = np.inf  # ||b|| is infinite: every finite residual meets rel_tol ||b||
    _, ri = solve(G, name, M, bn, maxit=5)
    assert np.isnan(ri.rel_residual)


def test_batch_mixed_widths_and_long_rows(gko):
    """The batched mixed solve at the edges of its block widths, and next to
    systems whose rows are too long for it (the queued kernels take those):
    per system the oracle's solution within 1e-8, the true residual reported."""
    G = gko
    rng = np.random.default_rng(6)
    sizes = [1, 3, 63, 64, 65, 128, 129, 255, 256, 257, 1023, 1024, 1025, 1281, 2049, 4095, 4096, 4097, 5000]
    systems = [banded_system(n, 7, True, n) for n in sizes]
    for n in (40, 300, 1500):  # 61 entries a row
        half = 30
        cols = np.arange(n)[:, None] + np.arange(-half, half + 1)[None, :]
        vals = np.full(cols.shape, -1.0)
        vals[:, half] = 2 * half + 0.5
        ok = (cols >= 0) & (cols < n)
        rp = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32)
        systems.append(I.Csr(n, n, rp, cols[ok].astype(np.int32), vals[ok], "long"))
    bs = [rng.uniform(-1, 1, A.n_rows) for A in systems]
    bs[4][:] = 0.0
    bs[7] = np.ldexp(bs[7], -60)
    B = G.Batch(systems)
    B.set_precision(G.PRECISION_MIXED_F32)
    xd = dev(np.zeros(B.total_rows))
    code, it, rr, st = B.cg(dev(np.concatenate(bs)), xd, 1e-12, 5000)
    assert code == G.OK and np.all(st == G.OK)
    x = host(xd)
    for i, A in enumerate(systems):
        xi = x[B.row_off[i]:B.row_off[i + 1]]
        if i == 4:
            assert it[i] == 0 and np.all(xi == 0) and rr[i] == 0
            continue
        xo, ro = O.cg(A, bs[i], tol=1e-12, maxit=5000)
        assert ro.status == 0 and np.linalg.norm(xi - xo) <= 1e-8 * np.linalg.norm(xo), i
        true = np.linalg.norm(bs[i] - O.spmv_csr(A, xi)) / np.linalg.norm(bs[i])
        assert true <= 1.01e-12 and abs(true - rr[i]) <= 1e-14


@pytest.mark.parametrize("bs", [1, 2, 8, 32, 5])
@pytest.mark.parametrize("n", [37, 700, 4101, 9001, 30011, 80000])
@pytest.mark.parametrize("name", ["cg", "bicgstab"])
def test_block_jacobi_shapes(gko, name, n, bs):
    """Block-Jacobi in the single-launch solvers (sizes that leave a short last
    block; block size 5 takes the multi-kernel solve), FP64 and mixed."""
    G = gko
    A = banded_system(n, 7, name == "cg", n)
    M = G.from_csr(A)
    bj = dict(preconditioner=G.PRECOND_BLOCK_JACOBI, block_size=bs)
    check(G, name, A, M, **bj)
    check(G, name, A, M, precision=G.PRECISION_MIXED_F32, **bj)


@pytest.mark.parametrize("restart", [1, 7, 30, 31, 32, 128])
@pytest.mark.parametrize("n", [1, 33, 700, 9001, 40000, 77825, 200000])
def test_gmres_shapes_and_restarts(gko, n, restart):
    """The single-launch GMRES over its launch shapes and restart lengths (32 and 128
    take the multi-kernel solve): the oracle's solution at 1e-12, the true
    residual reported, repeatable, and capped in the middle of a cycle."""
    G = gko
    A = banded_system(n, 7, False, n)
    M = G.from_csr(A)
    b = np.random.default_rng(1).uniform(-1, 1, n)
    for opt in ({}, {"precision": G.PRECISION_MIXED_F32}):
        xd = dev(np.zeros(n))
        res = G.gko_solve_gmres(M, dev(b), xd, 1e-12, 3000, G.opts(restart=restart, **opt))
        x = host(xd)
        xo, ro = O.gmres(A, b, tol=1e-12, maxit=3000, restart=restart)
        assert res.status == G.OK and ro.status == 0, res
        assert np.linalg.norm(x - xo) <= 1e-8 * np.linalg.norm(xo)
        true = np.linalg.norm(b - O.spmv_csr(A, x)) / np.linalg.norm(b)
        assert true <= 1.01e-12 and abs(true - res.rel_residual) <= 1e-13
        xd2 = dev(np.zeros(n))
        G.gko_solve_gmres(M, dev(b), xd2, 1e-12, 3000, G.opts(restart=restart, **opt))
        assert host(xd2).tobytes() == x.tobytes()
    xd = dev(np.zeros(n))
    res = G.gko_solve_gmres(M, dev(b), xd, 1e-15, 2, G.opts(restart=restart))
    assert res.iterations <= 2
    true = np.linalg.norm(b - O.spmv_csr(A, host(xd))) / np.linalg.norm(b)
    assert abs(true - res.rel_residual) <= 1e-13


FRESH = """
import sys, numpy as np, torch
sys.path.insert(0, {root!r}); sys.path.insert(0, {root!r} + '/tests')
from gpu_util import dev, host
from paper_2006_14290_gb300 import gko as G, inputs as I
def rows_of(K, n):
    cols = np.arange(n)[:, None] + np.arange(-(K // 2), K - K // 2)[None, :]
    vals = np.full(cols.shape, -1.0); vals[:, K // 2] = K + 1.0
    ok = (cols >= 0) & (cols < n)
    rp = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32)
    return G.from_csr(I.Csr(n, n, rp, cols[ok].astype(np.int32), vals[ok], 'rows'))
def solve(K, n, opt):
    xd = dev(np.zeros(n))
    res = G.gko_solve_bicgstab(rows_of(K, n), dev(np.linspace(1, 2, n)), xd, 1e-12, 500, G.opts(**opt))
    assert res.status == G.OK, res
    return host(xd).tobytes()
opt = {opt}
first = solve({K}, {n}, opt)
solve({K} + 2, {n}, opt)  # more shared memory: raises the kernel's limit
assert solve({K}, {n}, opt) == first
"""


# entries (and published vectors) of 46 to 48 KB a block: 12 bytes an entry in FP64, 8 in FP32
@pytest.mark.parametrize("K,n,opt", [(8, 40000, {}), (4, 80000, {}), (6, 8000, {}),
                                     (12, 40000, {"precision": 1}), (6, 80000, {"precision": 1}),
                                     (5, 8000, {"preconditioner": 2, "block_size": 8})])
def test_shared_memory_just_below_the_default_limit(gko, K, n, opt):
    """The same solve, bit for bit, before and after a larger one has raised
    the kernel's shared-memory limit (in a process of its own: the limit stays
    raised once any solve has done it)."""
    G = gko
    assert G.PRECISION_MIXED_F32 == 1 and G.PRECOND_BLOCK_JACOBI == 2
    code = FRESH.format(root=ROOT, K=K, n=n, opt=opt)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("precond", [0, 1, 2])
@pytest.mark.parametrize("n,fmt", [(33, "csr"), (300, "csr"), (300, "ell"), (20000, "csr"), (300, "coo")])
@pytest.mark.parametrize("name", ["cg", "bicgstab"])
def test_iteration_cap_near_attainable_accuracy(gko, name, n, fmt, precond):
    """A tolerance below what FP64 can reach: the recurrence residual meets it
    again and again, the true residual never, and max_iters still ends the
    solve wherever it falls (COO: the multi-kernel solve)."""
    G = gko
    if precond == 2 and fmt != "csr":
        pytest.skip("block-Jacobi reads a CSR matrix")
    A = banded_system(n, 7, name == "cg", 5)
    M = G.from_csr(A)
    M = {"csr": lambda m: m, "ell": G.gko_matrix_convert_to_ell, "coo": G.gko_matrix_convert_to_coo}[fmt](M)
    b = np.random.default_rng(5).uniform(-1, 1, n)
    for cap in range(1, 140 if n <= 300 and fmt != "coo" else 90):
        x, res = solve(G, name, M, b, tol=1e-17, maxit=cap, preconditioner=precond)
        assert res.iterations <= cap and res.status in (G.NOT_CONVERGED, G.BREAKDOWN), (cap, res)
        true = np.linalg.norm(b - O.spmv_csr(A, x)) / np.linalg.norm(b)
        assert abs(true - res.rel_residual) <= 1e-13


@pytest.mark.parametrize("ka,kb", [(0, 0), (-45, -75), (45, 60), (-45, 60)])
@pytest.mark.parametrize("n", [700, 9001])
def test_gmres_mixed_at_any_scale_of_matrix_and_right_hand_side(gko, n, ka, kb):
    """Mixed GMRES on 2^ka A x = 2^kb b: residuals and entries are FP32
    numbers, their products need not be; the same iterations and digits as
    without the powers of two."""
    G = gko
    A = banded_system(n, 7, False, n)
    b = np.random.default_rng(1).uniform(-1, 1, n)
    As = I.Csr(A.n_rows, A.n_cols, A.row_ptr, A.col, np.ldexp(A.val, ka), A.name)
    runs = []
    for M, rhs in ((G.from_csr(A), b), (G.from_csr(As), np.ldexp(b, kb))):
        xd = dev(np.zeros(n))
        res = G.gko_solve_gmres(M, dev(rhs), xd, 1e-12, 3000, G.opts(precision=G.PRECISION_MIXED_F32))
        assert res.status == G.OK, res
        runs.append((res.iterations, host(xd)))
    assert runs[1][0] == runs[0][0] and np.array_equal(runs[1][1], np.ldexp(runs[0][1], kb - ka))


# longest row K on both sides of the lines between cluster, recomputed and published vectors, entries in
# shared memory and in the matrix, and the multi-kernel solve
LONG_ROWS = [(2000, 17), (2000, 33), (2000, 57), (2000, 59), (4096, 15), (4096, 27), (4096, 29), (600, 265), (600, 267),
             (12000, 131), (12000, 135), (14000, 161), (20000, 101), (20000, 321), (20000, 323), (45000, 33),
             (45000, 35), (78000, 17), (78000, 95), (78000, 97), (100000, 65), (160000, 7), (160000, 9), (160000, 33),
             (160000, 41)]


@pytest.mark.parametrize("n,K", LONG_ROWS)
@pytest.mark.parametrize("name", ["cg", "bicgstab", "gmres"])
def test_long_rows(gko, name, n, K):
    G = gko
    half = K // 2
    rng = np.random.default_rng(K)
    cols = np.arange(n)[:, None] + np.arange(-half, half + 1)[None, :]
    vals = np.full(cols.shape, -1.0) if name == "cg" else rng.uniform(-1, 0, cols.shape)
    vals[:, half] = 1.5 * K
    ok = (cols >= 0) & (cols < n)
    rp = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32)
    A = I.Csr(n, n, rp, cols[ok].astype(np.int32), vals[ok], "long")
    M = G.from_csr(A)
    b = np.random.default_rng(1).uniform(-1, 1, n)
    x0, r0 = O.solve({"cg": O.CG, "bicgstab": O.BICGSTAB, "gmres": O.GMRES}[name], A, b, tol=1e-12, maxit=500)
    assert r0.status == 0
    fn = {"cg": G.gko_solve_cg, "bicgstab": G.gko_solve_bicgstab, "gmres": G.gko_solve_gmres}[name]
    for M in (M, G.gko_matrix_convert_to_ell(M)):
        for precision in (G.PRECISION_F64, G.PRECISION_MIXED_F32):
            xd = dev(np.zeros(n))
            res = fn(M, dev(b), xd, 1e-12, 500, G.opts(precision=precision))
            x = host(xd)
            assert res.status == G.OK and np.linalg.norm(x - x0) <= 1e-8 * np.linalg.norm(x0), res
            true = np.linalg.norm(b - O.spmv_csr(A, x)) / np.linalg.norm(b)
            assert true <= 1.01e-12 and abs(true - res.rel_residual) <= 1e-13


def test_mixed_cluster_solves_repeat_on_concurrent_streams(gko):
    """Mixed Jacobi-CG on 4,000-8,000 rows, whose FP32 inner solves run in one
    cluster each with two rows a thread, 480 times on four threads and streams:
    every solve converges in the steps and to the bits of the first."""
    import concurrent.futures as cf

    import torch

    G = gko
    systems = []
    for n in (4097, 4913, 5000, 6000, 6859, 7001, 8000, 8192):
        A = banded_system(n, 17, True, n)
        A.val = A.val * np.exp(np.random.default_rng(n).uniform(-2, 2)).astype(np.float64)
        systems.append((G.from_csr(A), dev(np.random.default_rng(n + 1).uniform(-1, 1, n))))
    opt = G.opts(precision=G.PRECISION_MIXED_F32, preconditioner=G.PRECOND_JACOBI)

    def run(M, b, stream):
        with torch.cuda.stream(stream):
            x = torch.zeros_like(b)
            res = G.gko_solve_cg(M, b, x, 1e-11, 2000, opt)
            stream.synchronize()
        assert res.status == G.OK and res.rel_residual <= 1e-11, res
        return res.iterations, host(x).tobytes()

    torch.cuda.synchronize()
    first = [run(M, b, torch.cuda.current_stream()) for M, b in systems]

    def worker(k):
        stream = torch.cuda.Stream()
        for rep in range(15):
            for i in np.random.default_rng(100 * k + rep).permutation(len(systems)):
                assert run(*systems[i], stream) == first[i], (k, rep, i)

    with cf.ThreadPoolExecutor(4) as ex:
        for f in [ex.submit(worker, k) for k in range(4)]:
            f.result()
