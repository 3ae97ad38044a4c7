"""The automatic choice for CG on small systems with rows of very different lengths: one thread of the cluster loop
walks a row, so they run with the matrix in shared memory (several lanes per row), or, with rows longer than a
tile, on the graph loop; counts and x against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1410_4054_gb300 import pk
from paper_1410_4054_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "dense_300": (lambda: W.spd_dense_rows(k=30, dense=(0, 17, 100), per_row=300), True),
    "dense_1000": (lambda: W.spd_dense_rows(k=85, dense=(0, 17, 100), per_row=1000), True),
    "dense_5000": (lambda: W.spd_dense_rows(k=85, dense=(0, 17, 100), per_row=5000), False),  # rows beyond a tile
    "powerlaw_500": (lambda: W.spd_power_law(500, seed=3, mean=8.0), True),
    "powerlaw_4000": (lambda: W.spd_power_law(4000, seed=3, mean=8.0), True),
}


@pytest.mark.parametrize("name", list(CASES))
def test_uneven_rows(name):
    make, shared = CASES[name]
    a = make()
    assert a.nnz + 6 * a.n <= 120_000
    _, b, _ = W.manufactured(a, seed=4)
    A = pk.CSRMatrix.from_workload(a)
    bd = torch.from_numpy(b).cuda()
    ref = O.cg(a, b, tol=1e-8, maxit=2000, variant="pipelined")

    def solve(**kw):
        x = torch.zeros_like(bd)
        info = pk.cg_solve(A, bd, x, **{"tol": 1e-8, "maxit": 2000, **kw})
        return info, x.cpu().numpy()

    info, _ = solve()
    assert info["status"] == pk.PK_OK and abs(info["iters"] - ref["iters"]) <= 2
    assert (info["launches"] == 3) == shared  # (setup, x = 0 guard, the loop) or a launch per kernel
    k = ref["iters"]
    fixed = O.cg(a, b, tol=0.0, maxit=k, variant="pipelined")
    _, x = solve(tol=0.0, maxit=k)
    assert np.linalg.norm(x - fixed["x"]) <= 1e-9 * np.linalg.norm(fixed["x"])
    # not the cluster's bits: its sums are in another order
    assert shared is False or not np.array_equal(x, solve(tol=0.0, maxit=k, loop="persistent")[1])
