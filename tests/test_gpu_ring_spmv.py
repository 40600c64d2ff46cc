"""Refinement on 27-point stencils, whose persistent loop stages the matrix and its operand in
shared memory, at the sizes where that can go wrong: ragged last slices, windows that leave the
vector at both ends, the narrowest grid, few and many slices a warp, warps without a slice, and a
26-offset matrix without the stencil's runs (the general path).  Against the oracle.

Tolerances as in test_gpu_fsai.py: the fp64 true residual recomputed by the oracle <= tol, the
iteration count within 10 % (reliable updates decide on fp32 residuals), the solution to 1e-6.
"""
import math

import numpy as np
import pytest

import cgproblems as gen
import oracle
from helpers import to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2608_09647_gb300 as cg  # noqa: E402


def box27(nx, ny, nz, skip=()):
    """27-point couplings of uneven weight on an nx x ny x nz grid; `skip` offsets are shifted by 3."""
    import scipy.sparse as sp
    n = nx * ny * nz
    offs = sorted({dx + nx * (dy + ny * dz) for dx in (-1, 0, 1) for dy in (-1, 0, 1) for dz in (-1, 0, 1)} - {0})
    right = [o + 3 if o in skip else o for o in offs if o > 0]
    rng = np.random.default_rng(nx * ny + nz)
    U = sp.diags([-rng.uniform(0.2, 1.0, n - o) for o in right], right, shape=(n, n))
    W = U + U.T
    d = -np.asarray(W.sum(axis=1)).ravel() * 1.02 + rng.uniform(0.05, 0.5, n)
    M = (W + sp.diags(d)).tocsr()
    M.sort_indices()
    return gen.CSR(n, M.indptr.astype(np.int32), M.indices.astype(np.int32), M.data, f"box{nx}x{ny}x{nz}")


CASES = [
    # matrix, CTAs (0: automatic)
    ("cube", lambda: box27(31, 31, 31), 3),
    ("narrow", lambda: box27(4, 4, 2051), 1),
    ("flat", lambda: box27(131, 67, 3), 2),
    ("few_slices", lambda: box27(21, 17, 23), 8),       # 257 slices for 64 warps
    ("below", lambda: box27(21, 17, 23), 9),            # fewer than four slices a warp: general path
    ("no_runs", lambda: box27(31, 29, 9, skip=(29 * 31,)), 1),
    ("automatic", lambda: box27(71, 69, 67), 0),
]


@pytest.mark.parametrize("precond", [cg.CG_PRECOND_JACOBI, cg.CG_PRECOND_NONE], ids=["jacobi", "none"])
@pytest.mark.parametrize("name,make,ctas", CASES, ids=[c[0] for c in CASES])
def test_refinement_matches_oracle(name, make, ctas, precond):
    A = make()
    b = oracle.spmv(A, gen.xstar(A.n, 5))
    tol = 1e-10
    h = cg.cg_create(A.n, *to_device(A))
    try:
        if ctas:
            assert cg.cg_set_option(h, cg.CG_OPT_GRID_CTAS, ctas) == cg.CG_OK
        bd = torch.from_numpy(b).cuda()
        ref = oracle.pcg_ru(A, b, tol=tol, tol_in=0.1, precond=int(precond == cg.CG_PRECOND_JACOBI))
        for _ in range(2):  # the second solve reuses the vectors
            x = torch.zeros_like(bd)
            st, it, rel = cg.cg_solve(h, bd, x, tol, 100000, precond, cg.CG_PREC_FP32_RU)
            assert st == ref.status == cg.CG_OK, cg.cg_last_error(h)
            assert abs(it - ref.iters) <= max(5, math.ceil(0.1 * ref.iters)), (it, ref.iters)
            xh = x.cpu().numpy()
            assert rel <= tol and oracle.true_relres(A, b, xh) <= tol * (1 + 1e-6)
            assert np.linalg.norm(xh - ref.x) <= 1e-6 * np.linalg.norm(ref.x)
    finally:
        cg.cg_destroy(h)
