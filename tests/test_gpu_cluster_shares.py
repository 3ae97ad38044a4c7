"""Row shares of the cluster loops at the edges of their sizes: batches that leave the device partly
empty and batches that fill it, and single systems whose CTAs do not all own rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1410_4054_gb300 import pk  # noqa: E402

DEV = "cuda:0"
# Tridiagonal matrices with diagonal 2.5 and neighbours -1: eigenvalues in (0.5, 4.5).  A solve to a
# relative residual of 1e-12 is within 9e-12 of x* (condition number 9) up to rounding.
BAR = 2e-11


def tridiagonal(n):
    i = np.arange(n)
    col = np.stack([i - 1, i, i + 1], 1)
    val = np.tile([-1.0, 2.5, -1.0], (n, 1))
    keep = (col >= 0) & (col < n)
    rp = np.concatenate([[0], np.cumsum(keep.sum(1))])
    return rp.astype(np.int32), col[keep].astype(np.int32), val[keep]


def system(n, seed):
    rp, ci, va = tridiagonal(n)
    x = np.random.default_rng([n, seed]).uniform(-1, 1, n)
    b = 2.5 * x
    b[1:] -= x[:-1]
    b[:-1] -= x[1:]
    return pk.CSRMatrix(rp, ci, va), torch.from_numpy(b).to(DEV), x


SIZES = [1, 31, 33, 511, 513, 2049, 8191, 8193, 16385, 32769, 65536]


@pytest.mark.parametrize("copies", [1, 24])  # 55 CTAs of 4,096 rows, and 1,320 (the device holds 304)
def test_batches_of_uneven_systems(copies):
    sys = [system(n, k) for n in SIZES for k in range(copies)]
    xs = [torch.zeros_like(b) for _, b, _ in sys]
    infos = pk.batched_solve([A for A, _, _ in sys], [b for _, b, _ in sys], xs, tol=1e-12, maxit=200)
    assert pk.batched_last_lanes() == -2
    ys = [torch.zeros_like(b) for _, b, _ in sys]
    rows = pk.batched_solve([A for A, _, _ in sys], [b for _, b, _ in sys], ys, tol=1e-12, maxit=200, lanes=1)
    for (_, _, want), x, info, row in zip(sys, xs, infos, rows):
        assert info["status"] == 0 and abs(info["iters"] - row["iters"]) <= 1
        assert np.linalg.norm(x.cpu().numpy() - want) <= BAR * np.linalg.norm(want)


@pytest.mark.parametrize("n", [1, 33, 513, 4900, 65536])
@pytest.mark.parametrize("solver", ["cg_solve", "bicgstab_solve", "gmres_solve"])
def test_single_systems_on_one_cluster(solver, n):
    A, b, want = system(n, 7)
    x = torch.zeros_like(b)
    if solver == "gmres_solve" and n > 32768:
        pytest.skip("past the GMRES cluster's sizes")
    info = getattr(pk, solver)(A, b, x, tol=1e-12, maxit=300, loop="persistent")
    assert info["status"] == 0
    assert np.linalg.norm(x.cpu().numpy() - want) <= BAR * np.linalg.norm(want)
    # maxit ends the loop with that many iterations
    if n > 100:
        x.zero_()
        info = getattr(pk, solver)(A, b, x, tol=1e-12, maxit=3, loop="persistent")
        assert info["iters"] == 3 and info["status"] == pk.PK_NOT_CONVERGED
