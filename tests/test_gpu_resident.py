"""Parity of the shared-memory form of stencil systems (a CTA per SM) at the sizes where it can
go wrong, against the oracle: a ragged last CTA, one row past a slice, the matrix in shared
memory or streamed, any number of diagonals.

Tolerances as in test_gpu_parity.py: iteration counts within max(3, 2 %), the fp64 true
residual recomputed by the oracle <= tol, the solution to 1e-4 relative of the oracle's.
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


def shifted(A, shift):
    """The matrix with its diagonal scaled by 1 + shift (fewer iterations)."""
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    vals = np.where(A.colind == rows, A.vals * (1.0 + shift), A.vals)
    return gen.CSR(A.n, A.rowptr, A.colind, vals, A.name + "_shifted")


def grid(nx, ny, points=5):
    """A non-square 5-/9-point grid graph Laplacian with a varying diagonal."""
    import scipy.sparse as sp
    def path(m):
        return sp.diags([np.ones(m - 1), np.ones(m - 1)], [1, -1]) if m > 1 else sp.csr_matrix((1, 1))
    W = sp.kron(sp.eye(ny), path(nx)) + sp.kron(path(ny), sp.eye(nx)) * 0.7
    if points == 9:
        W = W + 0.3 * sp.kron(path(ny), path(nx))
    n = nx * ny
    d = np.asarray(W.sum(axis=1)).ravel() * (1.02 + 0.05 * np.sin(np.arange(n))) + 0.05
    M = (sp.diags(d) - W).tocsr()
    M.sort_indices()
    return gen.CSR(n, M.indptr.astype(np.int32), M.indices.astype(np.int32), M.data, f"grid{points}_{nx}x{ny}")


def check(A, b, st, it, rel, x, ref, tol):
    assert st == ref.status == cg.CG_OK
    assert abs(it - ref.iters) <= max(3, math.ceil(0.02 * ref.iters)), (it, ref.iters)
    assert rel <= tol and oracle.true_relres(A, b, x) <= tol * (1 + 1e-6)
    assert np.linalg.norm(x - ref.x) <= 1e-4 * np.linalg.norm(ref.x)


RESIDENT = [
    # (matrix, precond, the matrix's rows fit in shared memory beside the vectors)
    ("5pt_small", lambda: grid(37, 13), 1),             # fewer slices than SMs, a ragged last slice
    ("9pt_one_past", lambda: grid(152 * 32 + 1, 1, 9), 1),  # one row past a slice for every SM
    ("9pt", lambda: grid(173, 211, 9), 0),
    ("7pt_3d", lambda: shifted(gen.lap3d7(45), 0.01), 1),
    ("27pt", lambda: shifted(gen.diff3d27(31, 1.0, 3), 0.01), 1),   # 26 diagonals: streamed in groups
    ("27pt_none", lambda: shifted(gen.diff3d27(52, 0.5, 4), 0.01), 0),  # too many to hold on chip
    ("5pt_streamed", lambda: shifted(gen.lap2d(1000, 5, 0.5), 0.05), 1),  # vectors on chip, matrix not
]


@pytest.mark.parametrize("name,make,precond", RESIDENT, ids=[r[0] for r in RESIDENT])
def test_shared_memory_form_matches_oracle(name, make, precond):
    A = make()
    b = oracle.spmv(A, gen.xstar(A.n, 3))
    h = cg.cg_create(A.n, *to_device(A))
    assert cg.cg_set_option(h, cg.CG_OPT_LOOP_MODE, 1) == cg.CG_OK
    bd = torch.from_numpy(b).cuda()
    x0 = 0.25 * gen.xstar(A.n, 8)
    for start in (np.zeros(A.n), x0):
        xd = torch.from_numpy(start.copy()).cuda()
        st, it, rel = cg.cg_solve(h, bd, xd, 1e-9, 5000, precond)
        info = cg.cg_get_solve_info(h)
        assert info["loop_form"] == 1 and info["grid_ctas"] <= 152
        check(A, b, st, it, rel, xd.cpu().numpy(), oracle.pcg(A, b, x0=start, tol=1e-9, maxit=5000, precond=precond), 1e-9)
    cg.cg_destroy(h)


def test_shared_memory_form_edge_cases():
    """Sudden convergence (two distinct eigenvalues), a maxit of a few steps, breakdown, b = 0."""
    A = grid(90, 190)
    h = cg.cg_create(A.n, *to_device(A))
    assert cg.cg_set_option(h, cg.CG_OPT_LOOP_MODE, 1) == cg.CG_OK
    b = oracle.spmv(A, gen.xstar(A.n, 3))
    x = torch.zeros(A.n, dtype=torch.float64, device="cuda")
    st, it, rel = cg.cg_solve(h, torch.from_numpy(b).cuda(), x, 1e-12, 7, cg.CG_PRECOND_JACOBI)
    ref = oracle.pcg(A, b, tol=1e-12, maxit=7, precond=1)
    assert st == ref.status == cg.CG_NOT_CONVERGED and it == 7
    assert abs(rel - ref.relres_true) <= 1e-9 * ref.relres_true
    assert np.linalg.norm(x.cpu().numpy() - ref.x) <= 1e-10 * np.linalg.norm(ref.x)
    st, it, rel = cg.cg_solve(h, torch.zeros_like(x), x, 1e-12, 7, cg.CG_PRECOND_JACOBI)
    assert (st, it) == (cg.CG_OK, 0) and float(x.abs().max()) == 0.0
    cg.cg_destroy(h)
    n = 20000  # 2 x 2 blocks: two eigenvalues of the scaled matrix
    import scipy.sparse as sp
    s = np.repeat(np.random.default_rng(1).uniform(0.5, 2.0, n // 2), 2)
    M = (sp.diags(s) @ sp.block_diag([sp.csr_matrix([[2.0, 1.0], [1.0, 2.0]])] * (n // 2)) @ sp.diags(s)).tocoo()
    # the coupling to the next block, zero, keeps both offsets full (the diagonal layout)
    z = np.arange(1, n - 1, 2)
    M = sp.coo_matrix((np.concatenate([M.data, np.zeros(2 * len(z))]),
                       (np.concatenate([M.row, z, z + 1]), np.concatenate([M.col, z + 1, z]))), shape=(n, n)).tocsr()
    M.sort_indices()
    A = gen.CSR(n, M.indptr.astype(np.int32), M.indices.astype(np.int32), M.data, "blocks")
    b = oracle.spmv(A, gen.xstar(n, 5))
    for sign, precond in ((1.0, 1), (-1.0, 0)):
        vals = A.vals * sign
        h = cg.cg_create(n, torch.from_numpy(A.rowptr).cuda(), torch.from_numpy(A.colind).cuda(), torch.from_numpy(vals).cuda())
        assert cg.cg_set_option(h, cg.CG_OPT_LOOP_MODE, 1) == cg.CG_OK
        x = torch.zeros(n, dtype=torch.float64, device="cuda")
        st, it, rel = cg.cg_solve(h, torch.from_numpy(b).cuda(), x, 1e-10, 100, precond)
        ref = oracle.pcg(gen.CSR(n, A.rowptr, A.colind, vals, "b"), b, tol=1e-10, maxit=100, precond=precond)
        assert st == ref.status and it == ref.iters
        assert abs(rel - ref.relres_true) <= 1e-9 * ref.relres_true + 1e-13
        cg.cg_destroy(h)
