"""A caller's x that is not 16-byte aligned, in every form of CG, BiCGStab and GMRES: the same bits as an aligned
one (the update kernels read x in 16-byte units; such an x is iterated in a library copy)."""
import numpy as np
import pytest
import torch

from paper_1410_4054_gb300 import pk
from paper_1410_4054_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FORMS = [("cg", pk.cg_solve, kw) for kw in (
    dict(flags=pk.FLAG_NO_TMA, loop="graph"), dict(flags=pk.FLAG_NO_TMA), dict(flags=pk.FLAG_NO_TMA, loop="host"),
    dict(flags=pk.FLAG_NO_TMA | pk.FLAG_TIMING), dict(flags=pk.FLAG_NO_TMA, variant="split", loop="graph"),
    dict(flags=pk.FLAG_NO_TMA, variant="classical"), dict(loop="graph"), dict(variant="split"), dict(precond="jacobi", loop="graph"),
    dict(precision="mixed"), dict(flags=pk.FLAG_SELL, loop="graph"), {})]
FORMS += [("bicgstab", pk.bicgstab_solve, kw) for kw in (dict(flags=pk.FLAG_NO_TMA, variant="classical"), dict(loop="graph"), {})]
FORMS += [("gmres", pk.gmres_solve, kw) for kw in (dict(loop="graph"), {})]


@pytest.mark.parametrize("dims", [(2, 1), (40, 41), (61, 51), (260, 270)], ids=str)
@pytest.mark.parametrize("name, solver, kw", FORMS, ids=lambda v: str(v) if isinstance(v, (str, dict)) else None)
def test_unaligned_x_gives_the_same_bits(name, solver, kw, dims):
    a = W.laplace_2d(*dims)
    _, b, _ = W.manufactured(a, seed=2)
    A = pk.CSRMatrix.from_workload(a)
    bd = torch.from_numpy(b).cuda()
    buf = torch.zeros(a.n + 1, dtype=torch.float64, device="cuda")
    x = torch.zeros(a.n, dtype=torch.float64, device="cuda")
    i1 = solver(A, bd, x, tol=1e-12, maxit=9, **kw)
    i2 = solver(A, bd, buf[1:], tol=1e-12, maxit=9, **kw)
    assert x.data_ptr() % 16 == 0 and buf[1:].data_ptr() % 16 == 8
    assert (i1["iters"], i1["status"]) == (i2["iters"], i2["status"])
    assert np.array_equal(x.cpu().numpy(), buf[1:].cpu().numpy())
    A.close()
