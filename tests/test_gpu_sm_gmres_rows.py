"""GMRES with the matrix in shared memory on rows of very different lengths and scales, up to the longest that
the loop takes (4,096 entries): R and xi of the first cycle at the bars of the launched form."""
import pytest

from paper_1410_4054_gb300 import pk
from paper_1410_4054_gb300 import workloads as W

import test_gpu_gmres as G

pytestmark = pytest.mark.gpu

MATRICES = {
    "rows_4000": lambda: W.spd_dense_rows(k=120, dense=(0, 17, 5000), per_row=4000),
    "rows_4000_scaled": lambda: W.diag_scaled(W.spd_dense_rows(k=120, per_row=4000), seed=1, spread=100.0),
    "rows_1500": lambda: W.spd_dense_rows(k=150, dense=(0, 17, 5000, 9000, 20000), per_row=1500),
}


@pytest.mark.parametrize("name", list(MATRICES))
def test_first_cycle_on_uneven_rows(name):
    a, m = MATRICES[name](), 30
    _, b, _ = W.manufactured(a, seed=3)
    ref, _, sR, sX, _, _ = G.oracle_sensitivity(a, b, "pipelined", m, 1e-8, m)
    A = pk.CSRMatrix.from_workload(a)
    info, _, tr = G.solve(a, b, A=A, tol=1e-8, maxit=m, restart=m)
    assert info["launches"] == 5  # state, setup, r_0, the loop, b = 0
    G.first_cycle_check(tr, ref, sR, sX, ref["iters"], name)
    k = min(*G.first_cycle_lengths(tr, ref, ref["iters"]), len(sR))
    G.full_R_check(A, a, b, ref, sR, sX, k, name, m=m)
