"""The bench's algorithmic bytes per SpMV against the arrays they count: each
stored value and index read once (padding excluded), x read once, y written
once.  CPU only."""
import numpy as np

import bench
from paper_2006_14290_gb300 import inputs as I


def arrays_bytes(A, fmt, sv, sx=None, sy=None, ell_width=None):
    sx = sv if sx is None else sx
    sy = sv if sy is None else sy
    L = A.row_lengths()
    xy = sx * A.n_cols + sy * A.n_rows
    if fmt == "csr":  # values, column indices, row pointers
        return A.nnz * sv + A.col.nbytes + A.row_ptr.nbytes + xy
    if fmt == "coo":  # values, column and row index per entry
        rows = np.repeat(np.arange(A.n_rows, dtype=np.int32), L)
        return A.nnz * sv + A.col.nbytes + rows.nbytes + xy
    if fmt == "ell":  # stored (non-padding) entries: value + column index
        return int(L.sum()) * (sv + 4) + xy
    # hybrid: the first min(len, K) entries of a row in ELL, the rest in COO
    ell = np.minimum(L, ell_width)
    tail = L - ell
    return int(ell.sum()) * (sv + 4) + int(tail.sum()) * (sv + 8) + xy


def test_spmv_bytes_match_the_arrays():
    rng = np.random.default_rng(4)
    for A in (I.stencil3d_27pt(6), I.rows_csr([0, 3, 9, 1, 0, 17, 2], 40, rng), I.powerlaw(500, seed=2)):
        L = A.row_lengths()
        for sv in (8, 4, 2):
            for fmt in ("csr", "coo", "ell"):
                got = bench.spmv_bytes(fmt, A.n_rows, A.n_cols, A.nnz, 0, 0, sv, sv, sv)
                assert got == arrays_bytes(A, fmt, sv), (fmt, sv)
            K = 3
            ell_nnz = int(np.minimum(L, K).sum())
            got = bench.spmv_bytes("hybrid", A.n_rows, A.n_cols, A.nnz, ell_nnz, A.nnz - ell_nnz, sv, sv, sv)
            assert got == arrays_bytes(A, "hybrid", sv, ell_width=K)


def test_roofline_case_bytes_closed_form():
    """27-point stencil 128^3 in FP64 COO, the bench's roofline case: n = 128^3,
    nnz = (3*128 - 2)^3, 16 bytes per entry plus x and y."""
    n, nnz = 128 ** 3, (3 * 128 - 2) ** 3
    assert nnz == 55_742_968
    assert bench.spmv_bytes("coo", n, n, nnz, 0, 0, 8, 8, 8) == 925_441_920
    assert I.stencil3d_27pt(10).nnz == (3 * 10 - 2) ** 3


def test_output_line_is_short_and_complete():
    """The line on standard output parses, holds the headline and the legs'
    short forms, and stays within what a tail of the output keeps."""
    import json

    leg = {"status": 0, "time_ms": 123.456, "oracle_sample": "x" * 300}
    full = {"metric": bench.METRIC, "value": 3765.35, "unit": "GB/s", "n_gpus": 1, "steps": 200, "warmup": 3,
            "ms_per_step": 2.7969, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64/f32", "data": "synthetic",
            "config": {"workload": bench.WORKLOAD, "l2": "flushed", "matrices": {f"m{i}": {"n": 10**6} for i in range(4)},
                       "tuned_plans": {str(i): {"kernel": 1} for i in range(200)}, "parallelism": "replicas x1"},
            "roofline": {"frac": 0.7}, "per_case": {str(i): {"ms": 0.1} for i in range(28)},
            "e2e": {"value": 3161.1, "unit": "GB/s", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}, "gpu_launches": 104000,
            "solvers": dict({f"cg_case_{i}": leg for i in range(18)}, speedup=1.8,
                            batched_cg={"f64": leg, "systems": 4096}),
            "serving": {f"rate{r}_f64": {"converged": 500, "p99_ms": 1.0, "solves_per_s": 2.0} for r in range(10)},
            "cpu_baseline": {"value": 141.6, "unit": "GB/s", "sample": "y" * 150}}
    text = bench.summary_line(full)
    line = json.loads(text)
    assert len(text) <= bench.LINE_MAX and "\n" not in text
    for k in ("metric", "value", "unit", "config", "e2e", "clocks", "gpu_launches", "roofline", "cpu_baseline"):
        assert k in line
    assert line["value"] == 3765.35 and line["solvers_ms"]["batch4096_f64"] == 123.456
    full["solvers"].update({f"more_{i}": leg for i in range(300)})  # never longer, whatever the legs hold
    assert len(bench.summary_line(full)) <= bench.LINE_MAX
