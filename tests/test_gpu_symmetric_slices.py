"""Refinement on matrices whose slices equal their transpose bit for bit (half of the slices is
read from 1 MB of half matrix and vectors up) and on one that differs from it in a single entry,
against the oracle.

Tolerances as in test_gpu_fsai.py: the fp64 true residual recomputed by the oracle <= tol, the
iteration count within 10 % (reliable updates decide on fp32 residuals), the solution to 1e-6.
"""
import math

import numpy as np
import pytest

import cgproblems as gen
import oracle
from helpers import to_device
from oracle import fsai

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2608_09647_gb300 as cg  # noqa: E402


def one_sided(A):
    """A with the last entry of row n/2 (right of the diagonal) scaled by 1 + 2^-20."""
    vals = A.vals.copy()
    vals[A.rowptr[A.n // 2 + 1] - 1] *= 1.0 + 2.0 ** -20
    return gen.CSR(A.n, A.rowptr, A.colind, vals, A.name + "_one_sided")


CASES = [
    ("5pt", lambda: gen.lap2d(211, 5, 0.5)),          # 4 slots, 44,521 rows: a ragged last slice
    ("7pt", lambda: gen.lap3d7(37)),                  # 6 slots
    ("q1", lambda: gen.q1aniso(181, 1.5, 1.9, 0.05, 8)),  # 8 slots
    ("q1_one_sided", lambda: one_sided(gen.q1aniso(181, 1.5, 1.9, 0.05, 8))),
    ("5pt_below", lambda: gen.lap2d(201, 5, 0.5)),    # just below 1 MB
]


@pytest.mark.parametrize("precond", ["jacobi", "none", "fsai"])
@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_refinement_matches_oracle(name, make, precond):
    A = make()
    b = oracle.spmv(A, gen.xstar(A.n, 5))
    tol = 1e-10
    h = cg.cg_create(A.n, *to_device(A))
    try:
        bd = torch.from_numpy(b).cuda()
        x = torch.zeros_like(bd)
        if precond == "fsai":
            g = fsai.classic(A)
            assert cg.cg_fsai_set_factor(h, torch.from_numpy(g).cuda()) == cg.CG_OK
            ref = fsai.pcg_ir(A, g, b, tol=tol, tol_in=0.1, carry=True)
            code = cg.CG_PRECOND_FSAI
        else:
            ref = oracle.pcg_ru(A, b, tol=tol, tol_in=0.1, precond=int(precond == "jacobi"))
            code = cg.CG_PRECOND_JACOBI if precond == "jacobi" else cg.CG_PRECOND_NONE
        st, it, rel = cg.cg_solve(h, bd, x, tol, 100000, code, cg.CG_PREC_FP32_RU)
        assert st == ref.status == cg.CG_OK, cg.cg_last_error(h)
        assert abs(it - ref.iters) <= max(5, math.ceil(0.1 * ref.iters)), (it, ref.iters)
        xh = x.cpu().numpy()
        assert rel <= tol and oracle.true_relres(A, b, xh) <= tol * (1 + 1e-6)
        assert np.linalg.norm(xh - ref.x) <= 1e-6 * np.linalg.norm(ref.x)
    finally:
        cg.cg_destroy(h)
