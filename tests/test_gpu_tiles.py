"""COO, hybrid and nonzero-split SpMV in row-aligned tiles at the edges of the
tiles and of the rule that selects them, against the oracle."""
import numpy as np
import pytest

from gpu_util import bf16_round, check_spmv_f32, check_spmv_f64, dev, host
from paper_2006_14290_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def cases():
    rng = np.random.default_rng(77)
    yield "one_entry", [0, 0, 1, 0]
    yield "row_fills_window", [1024, 1, 1023, 3]
    # rows that end on, one before and one after every tile (W = 960 with rows of 64 and more) and window
    yield "tile_ends", [960, 960, 959, 1, 961, 0, 0, 958, 2, 64, 896, 0] * 7
    yield "beyond_window", [5, 0, 1500, 0, 0, 3] * 40 + [2048, 0, 2048, 1, 2047]  # whole tiles inside a row
    yield "longest_tiled", [2048] * 20
    yield "too_long", [7] * 500 + [2049] + [7] * 500  # carries
    yield "empty_runs", [0] * 5000 + [3] * 200 + [0] * 4000 + [9, 0] * 300 + [0] * 3000
    yield "short", list(rng.integers(0, 5, 9000))
    yield "skewed", list(np.minimum(rng.zipf(2.0, 4000), 2000))
    yield "tail_of_one", [8] * 119 + [7] + [1]


CASES = [(n, I.rows_csr(L, 3000, np.random.default_rng(len(L)))) for n, L in cases()]


@pytest.mark.parametrize("name,A", CASES, ids=[c[0] for c in CASES])
@pytest.mark.parametrize("fmt", ["coo", "split", "hybrid0", "hybrid2"])
@pytest.mark.parametrize("dt", ["f64", "f32", "bf16"])
def test_tiles_match_oracle(gko, name, A, fmt, dt):
    G = gko
    M = G.from_csr(A)
    if dt != "f64":
        M = G.gko_matrix_convert_values(M, G.F32 if dt == "f32" else G.BF16)
    if fmt == "coo":
        M = G.gko_matrix_convert_to_coo(M)
    elif fmt == "split":
        M.set_plan(3, 1, 1, 1024)
    else:
        M = G.gko_matrix_convert_to_hybrid(M, int(fmt[-1]))
    rng = np.random.default_rng(5)
    x, y0 = rng.uniform(-1, 1, A.n_cols), rng.uniform(-1, 1, A.n_rows)
    for alpha, beta in [(1.0, 0.0), (-0.75, 1.5)]:
        if dt == "f64":
            yd = dev(y0 if beta else np.full(A.n_rows, np.nan))
            G.gko_spmv(alpha, M, dev(x), beta, yd)
            check_spmv_f64(host(yd), A, x, alpha, beta, y0)
        else:
            x32, v = x.astype(np.float32), A.val.astype(np.float32).astype(np.float64)
            yd = dev(y0, np.float32)
            G.gko_spmv(alpha, M, dev(x32), beta, yd)
            check_spmv_f32(host(yd), A, x32.astype(np.float64), alpha, beta, y0.astype(np.float32).astype(np.float64),
                           v if dt == "f32" else bf16_round(A.val))


@pytest.mark.parametrize("S", [2, 4])
@pytest.mark.parametrize("extra", [0, 1, 64])
@pytest.mark.parametrize("waves", [0, 1, 2, 3, 5])
def test_deferred_row_sums(gko, S, extra, waves):
    """FP64 row-block CSR with S lanes a row keeps the sums of up to S row
    blocks before it reduces them: 0 to 5 row blocks per thread block and a
    ragged last one, plain, with alpha and beta, and with the fused dot."""
    G = gko
    n = max(1, waves * 152 * 9 * (128 // S) + extra)
    rng = np.random.default_rng(n)
    lens = rng.integers(0, 12, n)
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    row = np.repeat(np.arange(n), lens)
    col = (row + rng.integers(0, 40, row.size)) % n
    A = I.Csr(n, n, rp, col.astype(np.int32), rng.uniform(-1, 1, row.size), "rows of 0..11")
    M = G.from_csr(A)
    M.set_plan(1, S, 1, 1024)
    x, y = rng.uniform(-1, 1, n), rng.uniform(-1, 1, n)
    yo = np.bincount(row, A.val * x[col], n)
    bound = 2.0**-53 * (14 * np.bincount(row, np.abs(A.val * x[col]), n) + 1e-300)
    yd = dev(y)
    G.gko_spmv(1.0, M, dev(x), 0.0, yd)
    assert np.all(np.abs(host(yd) - yo) <= bound)
    yd = dev(y)
    G.gko_spmv(-1.5, M, dev(x), 0.5, yd)
    assert np.all(np.abs(host(yd) - (-1.5 * yo + 0.5 * y)) <= 2 * bound + 2.0**-52 * np.abs(y))
    yd = dev(np.zeros(n))
    d = G.gko_spmv_dot(M, dev(x), yd)  # x . (A x)
    assert abs(d - x @ yo) <= 1e-13 * (np.abs(x) @ np.abs(yo)) + np.abs(x) @ bound


# both sides of the rule's lines: FP64 3 * 2^19 and 9 * 2^26 / L, FP32 2^21 and 3 * 2^30 / L, 2^23 for stencils
@pytest.mark.parametrize("L,rows", [(2000, 786), (2000, 787), (200, 15099), (200, 15100), (48, 174762), (48, 174763),
                                    (2000, 1048), (2000, 1049), (600, 8947), (600, 8948)])
@pytest.mark.parametrize("fmt", ["coo", "split", "hybrid0"])
def test_both_sides_of_the_tile_rule(gko, L, rows, fmt):
    """FP64, and the FP32 handle made from it (which may tile where FP64
    does not), before and after the plan is set again."""
    G = gko
    A = I.rows_csr([L] * rows, 3000, np.random.default_rng(L))
    M = G.from_csr(A)
    if fmt == "split":
        M.set_plan(3, 1, 1, 1024)
    else:
        M = G.gko_matrix_convert_to_coo(M) if fmt == "coo" else G.gko_matrix_convert_to_hybrid(M, 0)
    rng = np.random.default_rng(5)
    x, y0 = rng.uniform(-1, 1, A.n_cols), rng.uniform(-1, 1, A.n_rows)
    yd = dev(y0)
    G.gko_spmv(-0.75, M, dev(x), 1.5, yd)
    check_spmv_f64(host(yd), A, x, -0.75, 1.5, y0)
    x32, v32 = x.astype(np.float32), A.val.astype(np.float32).astype(np.float64)
    M32 = G.gko_matrix_convert_values(M, G.F32)
    for again in range(2):
        yd = dev(y0, np.float32)
        G.gko_spmv(-0.75, M32, dev(x32), 1.5, yd)
        check_spmv_f32(host(yd), A, x32.astype(np.float64), -0.75, 1.5, y0.astype(np.float32).astype(np.float64), v32)
        if fmt != "split":
            break
        M32.set_plan(3, 1, 1, 1024)
