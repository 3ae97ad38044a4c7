"""The loops that keep the matrix in shared memory (chosen by PK_LOOP_AUTO between the cluster's
sizes and what the SMs hold): the same rows, threads and summation orders as the launched kernels,
so every iterate must equal the graph loop's bit for bit."""
import threading

import numpy as np
import pytest
import torch

from paper_1410_4054_gb300 import pk
from paper_1410_4054_gb300 import workloads as W

import test_gpu_gmres as G

pytestmark = pytest.mark.gpu


def dev(v):
    return torch.from_numpy(np.ascontiguousarray(v)).cuda()


def shifted_dense_band(n, half):
    """Rows of 2 half + 1 entries: the block's columns reach only its neighbours."""
    r = np.repeat(np.arange(n), 2 * half + 1)
    c = (np.arange(n)[:, None] + np.arange(-half, half + 1)).ravel()
    keep = (c >= 0) & (c < n)
    v = np.where(r == c, 2.0 * half + 1.0, -1.0 / (1.0 + np.abs(r - c)))
    return W._from_coo(n, r[keep], c[keep], v[keep], f"band_{n}_{half}")


CG_MATRICES = {
    "lap3d_41": lambda: W.laplace_3d(41),                  # odd n, half the SMs
    "lap3d_64": lambda: W.laplace_3d(64),                  # two blocks on every SM
    "lap2d_513x400": lambda: W.laplace_2d(513, 400),
    "lap2d_1x70001": lambda: W.laplace_2d(70001, 1),       # halos of one or two columns
    "lap3d_66": lambda: W.laplace_3d(66),                  # x has no room in shared memory
    "band_70000": lambda: shifted_dense_band(70_000, 6),   # rows of 13: lane groups
    "fe_elasticity_23": lambda: W.fe_elasticity_3d(23),    # rows of up to 45
    "spd_powerlaw_70000": lambda: W.spd_power_law(70_000, seed=3, mean=8.0),  # whole-warp rows
}


def solve(A, n, b, trace=0, x0=None, **kw):
    x = dev(np.zeros(n) if x0 is None else x0)
    tr = torch.full((trace, 4), float("nan"), dtype=torch.float64, device="cuda") if trace else None
    info = pk.cg_solve(A, dev(b), x, trace=tr, **kw)
    return info, x.cpu().numpy(), tr.cpu().numpy() if trace else None


@pytest.mark.parametrize("name", sorted(CG_MATRICES))
def test_cg_equals_the_graph_loop_bitwise(name):
    a = CG_MATRICES[name]()
    _, b, _ = W.manufactured(a, seed=2)
    A = pk.CSRMatrix.from_workload(a)
    for kw in (dict(tol=1e-8, maxit=5000), dict(tol=0.0, maxit=1), dict(tol=0.0, maxit=7)):
        i1, x1, t1 = solve(A, a.n, b, trace=30, **kw)
        i2, x2, t2 = solve(A, a.n, b, trace=30, loop="graph", **kw)
        assert i1["launches"] == 3 and i2["launches"] > 3  # (setup, x = 0 guard, the loop)
        assert (i1["iters"], i1["status"], i1["rel_res_est"]) == (i2["iters"], i2["status"], i2["rel_res_est"])
        assert np.array_equal(x1, x2) and np.array_equal(t1, t2, equal_nan=True)


def test_cg_edges_match_the_graph_loop():
    a = W.laplace_3d(41)
    _, b, _ = W.manufactured(a, seed=1)
    A = pk.CSRMatrix.from_workload(a)
    bad = b.copy()
    bad[12345] = np.nan
    neg = W.CSR(a.n, a.row_ptr, a.col, -a.val)
    N = pk.CSRMatrix.from_workload(neg)
    rng = np.random.default_rng(0)
    for M, rhs, kw in ((A, np.zeros(a.n), dict(x0=np.ones(a.n))), (A, b, dict(maxit=0)), (A, bad, {}), (N, b, {}),
                       (A, b, dict(x0=rng.standard_normal(a.n), tol=1e-6)), (A, 1e-200 * b, {}), (A, 1e140 * b, {})):
        i1, x1, _ = solve(M, a.n, rhs, **kw)
        i2, x2, _ = solve(M, a.n, rhs, loop="graph", **kw)
        assert (i1["iters"], i1["status"]) == (i2["iters"], i2["status"])
        assert np.array_equal(x1, x2, equal_nan=True)


def test_cg_unaligned_x_and_host_vectors():
    a = W.laplace_3d(41)
    _, b, _ = W.manufactured(a, seed=1)
    A = pk.CSRMatrix.from_workload(a)
    _, want, _ = solve(A, a.n, b)
    buf = torch.zeros(a.n + 1, dtype=torch.float64, device="cuda")
    pk.cg_solve(A, dev(b), buf[1:])
    assert np.array_equal(buf[1:].cpu().numpy(), want)
    x = np.zeros(a.n)
    pk.cg_solve(A, b, x)
    assert np.array_equal(x, want)


def test_solves_of_several_threads_and_streams():
    """Only one such loop runs at a time; a solve that finds the GPU taken runs the launched loop
    with the same result."""
    mats = [W.laplace_3d(41), W.laplace_3d(48), W.laplace_2d(300, 290)]
    rhs = [W.manufactured(a, seed=k)[1] for k, a in enumerate(mats)]
    As = [pk.CSRMatrix.from_workload(a) for a in mats]
    want = [solve(A, a.n, b)[1] for A, a, b in zip(As, mats, rhs)]
    got = [[] for _ in mats]

    def work(k):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            b = dev(rhs[k])
            for _ in range(6):
                x = torch.zeros(mats[k].n, dtype=torch.float64, device="cuda")
                pk.cg_solve(As[k], b, x)
                got[k].append(x.cpu().numpy())

    ts = [threading.Thread(target=work, args=(k,)) for k in range(len(mats))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for k in range(len(mats)):
        assert len(got[k]) == 6 and all(np.array_equal(x, want[k]) for x in got[k])


# ------------------------------------------------------------------ GMRES, Jacobi CG
# (sums in another order than the launched kernels: the method's parity bars, 1e-12 for the scalars
# of the first steps and 1e-9 for x at the same count)

GMRES_MATRICES = {
    "convdiff_41": lambda: W.convdiff_3d(41),
    "convdiff_64": lambda: W.convdiff_3d(64),
    "band_70000": lambda: shifted_dense_band(70_000, 6),
    "fe_elasticity_11": lambda: W.fe_elasticity_3d(11),      # 4,752 rows of up to 45
    "powerlaw_20000": lambda: W.power_law(20_000),           # whole-warp rows
}


def gmres(A, n, b, x0=None, trace=40, **kw):
    x = dev(np.zeros(n) if x0 is None else x0)
    tr = torch.full((trace, 4), float("nan"), dtype=torch.float64, device="cuda")
    info = pk.gmres_solve(A, dev(b), x, trace=tr, **kw)
    return info, x.cpu().numpy(), tr.cpu().numpy()


@pytest.mark.parametrize("m", [1, 2, 3, 5, 9])
@pytest.mark.parametrize("name", sorted(GMRES_MATRICES))
def test_gmres_counts_and_x_match_the_graph_loop(name, m):
    """Few steps per cycle: every schedule of the column products (parts of a column per warp, then
    columns), restarts, and ends of the solve inside and at the end of a cycle."""
    a = GMRES_MATRICES[name]()
    _, b, _ = W.manufactured(a, seed=3)
    A = pk.CSRMatrix.from_workload(a)
    pre = "jacobi" if name == "powerlaw_20000" else "none"
    for maxit in (1, m, m + 2, 2 * m + 1):
        i1, x1, t1 = gmres(A, a.n, b, tol=1e-13, maxit=maxit, restart=m, precond=pre)
        i2, x2, t2 = gmres(A, a.n, b, tol=1e-13, maxit=maxit, restart=m, precond=pre, loop="graph")
        assert i1["launches"] == 5 + 2 * (pre == "jacobi")  # state, setup, r_0, the loop, b = 0
        assert (i1["iters"], i1["status"], i1["cycles"]) == (i2["iters"], i2["status"], i2["cycles"])
        assert np.linalg.norm(x1 - x2) <= 1e-9 * np.linalg.norm(x2)


@pytest.mark.parametrize("m", [30, 64])
@pytest.mark.parametrize("name", ["convdiff_41", "fe_elasticity_11", "powerlaw_20000"])
def test_gmres_parity_with_the_oracle(name, m):
    """R, xi, counts and x against the oracle, within max(1e-12, 100 x the oracle's own one-ulp
    spread) and max(1e-9, 10 x that of x): the bars of the launched form."""
    a = GMRES_MATRICES[name]()
    _, b, _ = W.manufactured(a, seed=3)
    pre = "jacobi" if name == "powerlaw_20000" else "none"
    k = 2 * m
    ref, fixed, sR, sX, it_spread, x_spread = G.oracle_sensitivity(a, b, "pipelined", m, 1e-8, k, precond=pre)
    A = pk.CSRMatrix.from_workload(a)
    info, x, tr = G.solve(a, b, A=A, tol=1e-8, maxit=k, restart=m, precond=pre)
    assert info["launches"] == 5 + 2 * (pre == "jacobi") and info["status"] == ref["status"]
    G.first_cycle_check(tr, ref, sR, sX, ref["iters"], name)
    k_orc, k_gpu = G.first_cycle_lengths(tr, ref, ref["iters"])
    G.full_R_check(A, a, b, ref, sR, sX, min(k_orc, k_gpu, len(sR)), name, m=m, precond=pre)
    if k_orc == k_gpu or ref["iters"] <= min(k_orc, k_gpu):
        assert abs(info["iters"] - ref["iters"]) <= max(2, 2 * it_spread)
        _, x2, _ = G.solve(a, b, A=A, tol=0.0, maxit=ref["iters"], restart=m, precond=pre)
        assert G.rel(x2, fixed["x"]) <= max(1e-9, 10 * x_spread)


def test_gmres_edges_match_the_graph_loop():
    a = W.convdiff_3d(41)
    xs, b, _ = W.manufactured(a, seed=1)
    A = pk.CSRMatrix.from_workload(a)
    bad = b.copy()
    bad[5] = np.nan
    d = W.CSR(70_000, np.arange(70_001, dtype=np.int32), np.arange(70_000, dtype=np.int32), np.full(70_000, 2.5))
    D = pk.CSRMatrix.from_workload(d)
    one = np.ones(d.n)
    z = W.CSR(d.n, d.row_ptr, ((d.col + 1) % d.n).astype(np.int32), np.ones(d.n))  # a cyclic shift
    Z = pk.CSRMatrix.from_workload(z)
    e0 = np.zeros(d.n)
    e0[0] = 1.0
    for M, n, rhs, kw in ((A, a.n, np.zeros(a.n), dict(x0=np.ones(a.n))), (A, a.n, b, dict(maxit=0)), (A, a.n, bad, {}),
                          (A, a.n, b, dict(x0=xs, tol=1e-6)), (D, d.n, one, {}), (Z, d.n, e0, dict(maxit=12, restart=5)), (A, a.n, b, dict(tol=1e-8, restart=30))):
        i1, x1, _ = gmres(M, n, rhs, **kw)
        i2, x2, _ = gmres(M, n, rhs, loop="graph", **kw)
        assert (i1["iters"], i1["status"], i1["cycles"]) == (i2["iters"], i2["status"], i2["cycles"]), kw
        assert np.allclose(x1, x2, rtol=0, atol=1e-9 * max(1e-300, np.abs(x2[np.isfinite(x2)]).max(initial=0.0)), equal_nan=True)


@pytest.mark.parametrize("name", ["lap3d_41", "lap3d_64", "fe_elasticity_23", "spd_powerlaw_70000", "lap2d_1x70001"])
def test_jacobi_cg_matches_the_graph_loop(name):
    a = W.diag_scaled(CG_MATRICES[name](), seed=1)
    _, b, _ = W.manufactured(a, seed=2)
    A = pk.CSRMatrix.from_workload(a)
    for kw in (dict(tol=0.0, maxit=1), dict(tol=0.0, maxit=25), dict(tol=1e-8, maxit=5000)):
        i1, x1, t1 = solve(A, a.n, b, trace=20, precond="jacobi", **kw)
        i2, x2, t2 = solve(A, a.n, b, trace=20, precond="jacobi", loop="graph", **kw)
        assert i1["launches"] == 4 and i2["launches"] > 4
        assert abs(i1["iters"] - i2["iters"]) <= (2 if kw["tol"] else 0) and i1["status"] == i2["status"]
        np.testing.assert_allclose(t1[:20, :2], t2[:20, :2], rtol=1e-12)
        if not kw["tol"]:
            assert np.linalg.norm(x1 - x2) <= 1e-9 * np.linalg.norm(x2)
    neg = W.CSR(a.n, a.row_ptr, a.col, -a.val)
    N = pk.CSRMatrix.from_workload(neg)
    assert solve(N, a.n, b, precond="jacobi")[0]["status"] == pk.PK_NOT_SPD
