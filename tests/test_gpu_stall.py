"""The loops' bounded waits run out, not only the setup's: with PK_FLAG_TEST_STALL the setup product completes
(the residual estimate is that of x0), the loop gives up after its short bound with x as it was, and the next
solve on the handle, whose exchange buffers an unfinished solve has used, is right."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1410_4054_gb300 import pk  # noqa: E402
from paper_1410_4054_gb300 import workloads as W  # noqa: E402

CASES = [
    ("pk_cg_solve", "auto", {}, 3), ("pk_cg_solve", "graph", {}, None), ("pk_cg_solve", "resident", {}, 3),
    ("pk_cg_solve", "auto", {"precond": "jacobi"}, 4), ("pk_cg_solve", "graph", {"precond": "jacobi"}, None),
    ("pk_bicgstab_solve", "auto", {}, 4), ("pk_bicgstab_solve", "graph", {}, None),
    ("pk_bicgstab_solve", "auto", {"precond": "jacobi"}, None),
    ("pk_gmres_solve", "auto", {}, 5), ("pk_gmres_solve", "graph", {}, None),
]


@pytest.mark.parametrize("entry, loop, kw, launches", CASES, ids=lambda v: str(v) if isinstance(v, str) else None)
def test_the_loops_own_waits_run_out(entry, loop, kw, launches):
    a = W.laplace_3d(64)  # 304 blocks: setup on the tiles where the flag is not given
    xs, b, _ = W.manufactured(a, seed=3)
    A = pk.CSRMatrix.from_workload(a)
    bd = torch.from_numpy(b).cuda()
    x = torch.zeros_like(bd)

    def solve(**opts):
        o, info = pk.make_opts(loop=loop, tol=1e-8, maxit=5000, **opts, **kw), pk.Info()
        st = getattr(pk.lib(), entry)(A.handle, C.c_void_p(bd.data_ptr()), C.c_void_p(x.data_ptr()), C.byref(o),
                                      C.byref(info), None)
        return st, info

    st, info = solve(flags=pk.FLAG_TEST_STALL, wait_ns=1_000_000)
    assert st == info.status == pk.PK_TIMEOUT and info.iters <= 1  # (GMRES: its first step needs no column)
    if not (entry == "pk_gmres_solve" and loop == "graph"):  # (there the first residual is part of the loop)
        assert info.rel_res_est == 1.0  # x0 = 0, and the setup's sums are complete
    if launches:
        assert info.launches == launches
    assert not x.any()
    st, info = solve(flags=pk.FLAG_TRUE_RES)
    assert st == pk.PK_OK and info.rel_res_true <= 1.5e-8
    assert np.linalg.norm(x.cpu().numpy() - xs) <= 1e-5 * np.linalg.norm(xs)
    A.close()
