"""BiCGStab with the matrix in shared memory (PK_LOOP_AUTO past the cluster's sizes) against the oracle at the
bars of the launched form, at sizes for each of its layouts: all seven vectors in shared memory, then without
x, without r0* too, and with the four that the loop cannot do without."""
import numpy as np
import pytest
import torch

from paper_1410_4054_gb300 import pk
from paper_1410_4054_gb300 import workloads as W

import test_gpu_bicgstab as B

pytestmark = pytest.mark.gpu

# vectors in shared memory (two blocks of up to 113 KB per SM past 152 blocks; up to 225 KB below)
MATRICES = {
    "convdiff_24": lambda: W.convdiff_3d(24),       # 7; blocks finer than the launched kernels'
    "convdiff_41": lambda: W.convdiff_3d(41),       # 7; odd n
    "convdiff_61": lambda: W.convdiff_3d(61),       # 6; odd n
    "convdiff_63": lambda: W.convdiff_3d(63),       # 5; odd n
    "convdiff_64": lambda: W.convdiff_3d(64),       # 4
    "jacobi:powerlaw_50000": lambda: W.power_law(50_000),    # 7; rows in sorted rounds
    "jacobi:powerlaw_120000": lambda: W.power_law(120_000),  # 4
}


@pytest.mark.parametrize("name", list(MATRICES))
def test_parity_with_the_oracle(name):
    """alpha, beta, omega within max(1e-12, 100 x the oracle's one-ulp spread), the median count over b and its
    perturbations within the gate of the launched form, x at the oracle's count within max(1e-9, 10 x its spread)."""
    a = MATRICES[name]()
    _, b, _ = W.manufactured(a, seed=0)
    pre = "jacobi" if name.startswith("jacobi:") else "none"
    ref, fixed, spread, counts, x_spread = B.oracle_sensitivity(a, b, "pipelined", nsamp=4, nsamp_x=2, precond=pre)
    A = pk.CSRMatrix.from_workload(a)
    info, _, tr = B.solve(a, b, A=A, tol=1e-8, maxit=5000, precond=pre)
    assert info["status"] == pk.PK_OK
    assert info["launches"] == 4 + 2 * (pre == "jacobi")  # setup, x = 0 guard, p_0, the loop
    gpu = [info["iters"]] + [B.solve(a, B.perturbed_b(W, b, k), A=A, tol=1e-8, maxit=5000, precond=pre)[0]["iters"]
                             for k in range(len(counts) - 1)]
    assert abs(B.median(gpu) - B.median(counts)) <= B.count_gate(counts), (gpu, counts)
    k = min(20, ref["iters"] - 1)
    for col, key in ((0, "alpha"), (2, "omega"), (1, "beta")):
        off = np.abs(tr[:k, col] - ref[key][:k]) / np.abs(ref[key][:k])
        assert np.all(off <= np.maximum(1e-12, 100 * spread[:k])), (key, off)
    info, x, _ = B.solve(a, b, A=A, tol=0.0, maxit=ref["iters"], precond=pre)
    assert info["iters"] == ref["iters"]
    assert B.rel(x, fixed["x"]) <= max(1e-9, 10 * x_spread)
    # an x that is not 16-byte aligned: the same bits
    buf = torch.zeros(a.n + 1, dtype=torch.float64, device="cuda")
    pk.bicgstab_solve(A, B.dev(b), buf[1:], tol=0.0, maxit=ref["iters"], precond=pre)
    assert np.array_equal(buf[1:].cpu().numpy(), x)


@pytest.mark.parametrize("k", [41, 64])
def test_ends_match_the_graph_loop(k):
    a = W.convdiff_3d(k)
    n = a.n
    xs, b, _ = W.manufactured(a, seed=1)
    bad = b.copy()
    bad[n // 2] = np.nan
    one, cols = np.ones(n), np.arange(n, dtype=np.int32)
    rp = np.arange(n + 1, dtype=np.int32)
    e0 = np.zeros(n)
    e0[0] = 1.0
    A = pk.CSRMatrix.from_workload(a)
    D = pk.CSRMatrix.from_workload(W.CSR(n, rp, cols, np.full(n, 2.5)))              # s_0 = 0: the early exit
    Z = pk.CSRMatrix.from_workload(W.CSR(n, rp, ((cols + 1) % n).astype(np.int32), one))  # <A p, r0*> = 0: breakdown
    for M, rhs, kw in ((A, np.zeros(n), dict(x0=one)), (A, b, dict(maxit=0)), (A, b, dict(tol=0.0, maxit=1)), (A, bad, {}),
                       (A, b, dict(x0=xs, tol=1e-6)), (A, 1e-140 * b, {}), (D, one, {}), (Z, e0, {}),
                       (A, b, dict(tol=0.5)), (A, b, dict(tol=1e-3)), (A, b, {})):
        i1, x1, _ = B.solve(a, rhs, A=M, **kw)
        i2, x2, _ = B.solve(a, rhs, A=M, loop="graph", **kw)
        assert i1["launches"] == 4
        assert (i1["iters"], i1["status"]) == (i2["iters"], i2["status"]), kw
        scale = max(1e-300, np.abs(x2[np.isfinite(x2)]).max(initial=0.0))
        assert np.allclose(x1, x2, rtol=0, atol=1e-9 * scale, equal_nan=True), kw
    assert B.solve(a, one, A=D)[0]["iters"] == 1
    assert B.solve(a, e0, A=Z)[0]["status"] == pk.PK_BREAKDOWN
