"""cg_solve_noalloc in every form its size and row lengths choose (the cluster with the CSR in
shared memory or not, one CTA), against the oracle: iteration counts within max(3, 2 %), the
fp64 true residual recomputed by the oracle <= tol, the solution to 1e-4 relative.
"""
import math

import numpy as np
import pytest

import cgproblems as gen
import oracle
from helpers import random_graph_spd, spd_from_pattern, to_device

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


NOALLOC = [
    ("one_row", lambda: gen.CSR(1, np.array([0, 1], np.int32), np.array([0], np.int32), np.array([2.5]), "one"), 1),
    ("65_rows", lambda: grid(13, 5), 1),
    ("16_ctas_ragged", lambda: grid(41, 25, 9), 0),
    ("rows_of_many", lambda: random_graph_spd(9001, 9, 3), 1),      # rows past shared memory or not: the kernels look
    ("long_rows", lambda: spd_from_pattern(6000, 5, long_rows=[(3, 5000), (4000, 3000)], max_len=24), 1),
    ("most_rows", lambda: shifted(gen.lap3d7(32), 0.05), 1),         # 32,768 rows: 2,048 a CTA
    ("one_cta", lambda: shifted(gen.lap2d(182, 5, 0.4), 0.05), 1),   # 33,124 rows: past the cluster
]


@pytest.mark.parametrize("name,make,precond", NOALLOC, ids=[r[0] for r in NOALLOC])
def test_noalloc_forms_match_oracle(name, make, precond):
    A = make()
    b = oracle.spmv(A, gen.xstar(A.n, 2))
    bd = torch.from_numpy(b).cuda()
    xd = torch.zeros_like(bd)
    st, it, rel = cg.cg_solve_noalloc(*to_device(A), bd, xd, 1e-9, 4000, precond)
    check(A, b, st, it, rel, xd.cpu().numpy(), oracle.pcg(A, b, tol=1e-9, maxit=4000, precond=precond), 1e-9)
