"""The launched CG update kernel on a matrix whose row lengths change along its numbering: its time goes with the
rows, not with the nonzeros of the blocks that the products take.  Systems that the shared-memory loop holds share
their blocks with it (bit equality, test_gpu_sm.py); this one is far too large for it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1410_4054_gb300 import pk  # noqa: E402
from paper_1410_4054_gb300 import workloads as W  # noqa: E402


def two_bands(n, half_first, half_second):
    """Symmetric, diagonally dominant: a band of half_first in the first half of the rows, half_second after."""
    i = np.arange(n)
    rows, cols, vals = [i], [i], [np.where(i < n // 2, 2.0 * half_first, 2.0 * half_second) + 1.0]
    for k in range(1, half_second + 1):
        j = i[:n - k] if k <= half_first else i[n // 2:n - k]
        for r, c in ((j, j + k), (j + k, j)):
            rows.append(r)
            cols.append(c)
            vals.append(np.full(len(j), -1.0))
    return W._from_coo(n, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals), f"two_bands_{n}")


def update_us(a):
    A = pk.CSRMatrix.from_workload(a)
    b = torch.from_numpy(W.manufactured(a, seed=1)[1]).cuda()
    best = min(pk.cg_solve(A, b, torch.zeros_like(b), tol=0.0, maxit=20, flags=pk.FLAG_TIMING)["kernel_ms"]["update"]
               for _ in range(4))
    A.close()
    return 1e3 * best


def test_update_time_does_not_follow_the_row_lengths():
    n = 600_000
    even, uneven = update_us(two_bands(n, 1, 1)), update_us(two_bands(n, 1, 30))
    print(f"update kernel: {even:.2f} us on even rows, {uneven:.2f} us on uneven ones")
    assert uneven <= 1.5 * even


def test_sell_loop_keeps_its_own_rows():
    """SELL sums in an order of its own, so its update kernel has no reason to take the tile blocks' rows: on 39,744
    unknowns of 45 entries these are 304 blocks of 130 rows, where equal chunks are 78 (5 us per iteration more)."""
    a = W.fe_elasticity_3d(23)
    A = pk.CSRMatrix.from_workload(a)
    b = torch.from_numpy(W.manufactured(a, seed=1)[1]).cuda()

    def us(flags):
        return min(pk.cg_solve(A, b, torch.zeros_like(b), tol=0.0, maxit=60, loop="graph", flags=flags)["solve_ms"]
                   for _ in range(10)) * 1e3 / 60

    tiles, sell = us(0), us(pk.FLAG_SELL)
    print(f"CG on the CSR tiles {tiles:.1f} us per iteration, on SELL {sell:.1f}")
    assert sell <= 1.05 * tiles
