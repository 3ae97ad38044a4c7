"""An automatic solve takes its loop by the system alone: solves of several host threads at once, each on a
cooperative loop that wants every SM, give the bits and the launch counts that they give alone, and none of
their (short) waits runs out while they queue for the SMs that the others hold."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1410_4054_gb300 import pk  # noqa: E402
from paper_1410_4054_gb300 import workloads as W  # noqa: E402

CASES = {
    "cg_small": (lambda: W.laplace_3d(24), pk.cg_solve, {}),
    "cg": (lambda: W.laplace_3d(64), pk.cg_solve, {}),
    "cg_jacobi": (lambda: W.fe_elasticity_3d(15), pk.cg_solve, dict(precond="jacobi", tol=0.0, maxit=200)),
    "cg_resident": (lambda: W.laplace_3d(72), pk.cg_solve, dict(loop="resident")),
    "bicgstab": (lambda: W.convdiff_3d(64), pk.bicgstab_solve, {}),
    "bicgstab_jacobi": (lambda: W.power_law(50_000), pk.bicgstab_solve, dict(precond="jacobi")),
    "gmres": (lambda: W.convdiff_3d(41), pk.gmres_solve, {}),
}


def test_threads_do_not_change_each_others_loops():
    run, want, got, errors = {}, {}, {k: [] for k in CASES}, []
    for name, (make, solver, kw) in CASES.items():
        a = make()
        A, b = pk.CSRMatrix.from_workload(a), torch.from_numpy(W.manufactured(a, seed=3)[1]).cuda()

        def once(A=A, b=b, solver=solver, kw=kw):
            x = torch.zeros_like(b)
            info = solver(A, b, x, stream=torch.cuda.current_stream(), wait_ns=100_000_000, **{"maxit": 5000, **kw})
            return x.cpu().numpy(), info["status"], info["iters"], info["launches"]

        run[name], want[name] = once, once()
    torch.cuda.synchronize()

    def work(name):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(12):
                    got[name].append(run[name]())
        except Exception as e:  # noqa: BLE001
            errors.append((name, str(e)))

    ts = [threading.Thread(target=work, args=(k,)) for k in CASES]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors
    for name in CASES:
        assert len(got[name]) == 12
        for x, *rest in got[name]:
            assert rest == list(want[name][1:]), name
            assert np.array_equal(x, want[name][0]), name
