"""The benchmark's count of the solver's FP64 operations against a count over the
rows: products with every entry of the red rows and with the off-diagonal ones
of the black rows, vector work on the red rows alone."""
import numpy as np
import pytest

import bench
from oracle import galerkin as ogal
from oracle import stamp as ostamp


@pytest.mark.parametrize("N", [1, 2, 3])
@pytest.mark.parametrize("half,real", [(True, True), (False, False)])
def test_solver_flops(N, half, real):
    p = np.array([[5, 0, 1, 0], [0, 7, 0, 2], [1, 1, 11, 0]])
    q = np.array([[1, 2, 3, 40], [50, 1, 0, 3]])
    af, F = np.vstack([np.zeros((1, 4), int), p, -p]), np.vstack([q, -q])
    S, level = ostamp.stamp_bfs(af, F, N)
    L = ogal.galerkin_matrix(S, af, np.array([1.0] + [0.1] * 6, complex))[0].tocsr()
    red = (N - np.asarray(level)) % 2 == 1
    per_row = np.diff(L.indptr)
    applies, iters = 5, 3
    rows = 0.5 if half else 1.0
    want = rows * ((4.0 if real else 8.0) * (per_row.sum() - (~red).sum()) * applies + 30.0 * red.sum() * iters)
    ctx = {"nnz": L.nnz, "size": len(S), "red_rows": int(red.sum()),
           "solve_stats": {"half_system": half, "real_coefficients": real, "applies": applies, "inner_iters": iters}}
    got = bench.roofline_of("k_solve<0>", 1.0, ctx, {"fp64_tflops": 1.0})
    assert got["algorithmic_flops"] == want
