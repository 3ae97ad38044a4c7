"""Tiles of rows of very different lengths: every number of lanes per row and its limits, in the
launched kernels and in the loop with the matrix in shared memory."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1410_4054_gb300 import pk  # noqa: E402

DEV = "cuda:0"
# row lengths around the limits of 8 entries per lane, repeated so that tiles start anywhere
LENGTHS = {
    "limits": [1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 300],
    "one_long": [600] + [2] * 300,
    "short_and_long": [1] * 400 + [40],
}


@pytest.mark.parametrize("name", sorted(LENGTHS))
@pytest.mark.parametrize("n", [700, 6000])
def test_rows_of_very_different_lengths(name, n):
    r = np.random.default_rng([n, len(LENGTHS[name])])
    lens = np.resize(np.array(LENGTHS[name]), n)
    cols = [np.sort(np.append(r.choice(n - 1, size=k - 1, replace=False), -1)) for k in lens]
    cols = [np.sort(np.where(c < 0, i, c + (c >= i))) for i, c in enumerate(cols)]  # the diagonal, k - 1 others
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    ci = np.concatenate(cols).astype(np.int32)
    row = np.repeat(np.arange(n), lens)
    va = np.where(ci == row, 2.0, r.uniform(-1, 1, len(ci)) / np.repeat(lens, lens))  # dominant by rows
    x0 = r.uniform(-1, 1, n)
    delta = r.uniform(-1, 1, n)
    b = delta.copy()
    np.add.at(b, row, va * x0[ci])
    A = pk.CSRMatrix(rp, ci, va)
    bd = torch.from_numpy(b).to(DEV)
    # the setup product: r0 = b - A x0 = delta, within the rounding of sums of at most 600 terms of
    # magnitude 1 or less (3 in all per row): 600 * 2^-53 * 3 per entry, delta's rms is 0.58
    x = torch.from_numpy(x0).to(DEV)
    info = pk.bicgstab_solve(A, bd, x, tol=1e-12, maxit=0, loop="graph")
    want = np.linalg.norm(delta) / np.linalg.norm(b)
    assert abs(info["rel_res_est"] - want) <= 1e-12 * want + 600 * 3 * 2.0 ** -53 * want / 0.5
    # one iteration, launched and with the matrix in shared memory: the same up to the rounding of its
    # products and of five inner products of n terms without cancellation to speak of (A is dominated by
    # its diagonal 2): n * 2^-53 < 1e-12, with two orders of room
    out = []
    for loop in ("graph", "auto"):
        y = torch.from_numpy(x0).to(DEV)
        info = pk.bicgstab_solve(A, bd, y, tol=1e-12, maxit=1, loop=loop)
        assert info["iters"] == 1 and info["status"] == pk.PK_NOT_CONVERGED
        out.append(y.cpu().numpy())
    assert np.linalg.norm(out[0] - out[1]) <= 1e-10 * np.linalg.norm(out[0])
