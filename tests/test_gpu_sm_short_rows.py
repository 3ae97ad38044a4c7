"""Shared-memory loops of small systems with rows of at most eight entries, whose blocks and tiles the device forms:
even and very uneven shares (blocks of more rows than a tile, short last blocks), a handle used by one solver and
then by another, against the launched loop and the exact solution."""
import numpy as np
import pytest
import torch

from paper_1410_4054_gb300 import pk
from paper_1410_4054_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def band_after(n, split, half):
    """Rows before `split` hold their diagonal alone, the others a symmetric band of `half` entries each way."""
    i = np.arange(n)
    rows, cols, vals = [i], [i], [np.where(i < split, 1.5, 2.0 * half + 0.5)]
    for k in range(1, half + 1):
        j = i[split:n - k]
        for r, c in ((j, j + k), (j + k, j)):
            rows.append(r)
            cols.append(c)
            vals.append(np.full(len(j), -1.0 / k))
    return W._from_coo(n, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals), f"band_{n}_{split}_{half}")


MATRICES = {
    "even_20000": lambda: band_after(20_000, 0, 3),
    "half_40001": lambda: band_after(40_001, 20_000, 3),   # the first blocks have three times the rows
    "most_65536": lambda: band_after(65_536, 60_000, 3),
    "all_65535": lambda: band_after(65_535, 65_535, 1),    # a diagonal matrix
    "lap2d_1x50001": lambda: W.laplace_2d(50_001, 1),
    "lap3d_40": lambda: W.laplace_3d(40),
    "convdiff_33": lambda: W.convdiff_3d(33),
}


@pytest.mark.parametrize("name", list(MATRICES))
def test_small_systems_match_the_launched_loop(name):
    a = MATRICES[name]()
    assert np.diff(a.row_ptr).max() <= 8 and a.nnz + 6 * a.n > 120_000 and a.n <= 65_536
    xs, b, _ = W.manufactured(a, seed=5)
    A = pk.CSRMatrix.from_workload(a)
    bd = torch.from_numpy(b).cuda()
    for solver, kw, launches in ((pk.cg_solve, {}, 3), (pk.gmres_solve, dict(restart=20), 5), (pk.bicgstab_solve, {}, 4),
                                 (pk.cg_solve, dict(precond="jacobi"), 4), (pk.cg_solve, {}, 3)):
        if solver is pk.cg_solve and name.startswith("convdiff"):
            continue
        for maxit in (1, 12):
            x, y = torch.zeros_like(bd), torch.zeros_like(bd)
            i1 = solver(A, bd, x, tol=1e-14, maxit=maxit, **kw)
            i2 = solver(A, bd, y, tol=1e-14, maxit=maxit, loop="graph", **kw)
            assert i1["launches"] == launches
            assert (i1["iters"], i1["status"]) == (i2["iters"], i2["status"]), (solver.__name__, kw, maxit)
            assert float((x - y).norm()) <= 1e-9 * float(y.norm()), (solver.__name__, kw, maxit)
    if not name.startswith("lap2d"):  # (that one is far too badly conditioned for an error bound)
        x = torch.zeros_like(bd)
        pk.bicgstab_solve(A, bd, x, tol=1e-10, maxit=5000)
        assert np.linalg.norm(x.cpu().numpy() - xs) <= 1e-6 * np.linalg.norm(xs)
    A.close()
