"""fp64 solves of 27-point matrices on both sides of the line between the shared-memory form and
the graph form, against the oracle.

Tolerances as in test_gpu_resident.py: iteration counts within max(3, 2 %), the fp64 true
residual recomputed by the oracle <= tol, the solution to 1e-4 relative of the oracle's."""
import math

import numpy as np
import pytest

import cgproblems as gen
import oracle
from helpers import to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2608_09647_gb300 as cg  # noqa: E402


@pytest.mark.parametrize("side,form", [(72, 1), (73, 2)])  # 77.6 and 80.9 MB of loop matrix; the line lies at 80
def test_form_and_result(side, form):
    A = gen.diff3d27(side, 0.5, 3)
    on = A.colind == np.repeat(np.arange(A.n), np.diff(A.rowptr))
    A = gen.CSR(A.n, A.rowptr, A.colind, np.where(on, A.vals * 1.05, A.vals), A.name + "_shifted")
    b = oracle.spmv(A, gen.xstar(A.n, 3))
    h = cg.cg_create(A.n, *to_device(A))
    x = torch.zeros(A.n, dtype=torch.float64, device="cuda")
    st, it, rel = cg.cg_solve(h, torch.from_numpy(b).cuda(), x, 1e-9, 2000, cg.CG_PRECOND_JACOBI)
    got = cg.cg_get_solve_info(h)["loop_form"]
    cg.cg_destroy(h)
    assert got == form
    ref = oracle.pcg(A, b, tol=1e-9, maxit=2000, precond=1)
    x = x.cpu().numpy()
    assert st == ref.status == cg.CG_OK
    assert abs(it - ref.iters) <= max(3, math.ceil(0.02 * ref.iters)), (it, ref.iters)
    assert rel <= 1e-9 and oracle.true_relres(A, b, x) <= 1e-9 * (1 + 1e-6)
    assert np.linalg.norm(x - ref.x) <= 1e-4 * np.linalg.norm(ref.x)
