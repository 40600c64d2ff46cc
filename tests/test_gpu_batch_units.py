"""Batches whose members lie at the steps of the reduction units or outnumber the teams: every
member is solved as alone, whatever the grid."""
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


@pytest.mark.parametrize("precision", ["fp64", "ru"])
def test_batch_units_and_queue(precision):
    """Members at the steps of the reduction unit (64 / 65 and 256 / 257 tiles of 256 rows), and
    far more members than teams: every member is solved as alone, bit for bit the same on
    another grid."""
    sizes = [(128, 128), (128, 129), (256, 256), (257, 256), (3, 1), (16, 16), (16, 17)]
    systems = [grid(a, b, 9 if k % 2 else 5) for k, (a, b) in enumerate(sizes)]
    systems += [grid(5 + k % 37, 3 + k % 11) for k in range(170)]
    bs = [oracle.spmv(A, gen.xstar(A.n, k)) for k, A in enumerate(systems)]
    dev = [to_device(A) for A in systems]
    h = cg.cg_batch_create(*[[d[j] for d in dev] for j in range(3)])
    prec = cg.CG_PREC_FP64 if precision == "fp64" else cg.CG_PREC_FP32_RU
    bd = [torch.from_numpy(b).cuda() for b in bs]
    outs = []
    for ctas in (0, 5, 304):
        assert cg.cg_set_option(h, cg.CG_OPT_GRID_CTAS, ctas) == cg.CG_OK
        xd = [torch.zeros_like(b) for b in bd]
        st, its, rels = cg.cg_solve_batch(h, bd, xd, 1e-9, 5000, cg.CG_PRECOND_JACOBI, prec)
        assert st == cg.CG_OK, cg.cg_last_error(h)
        outs.append((its, [x.cpu().numpy() for x in xd]))
    for its, xs in outs[1:]:
        assert its == outs[0][0] and all(np.array_equal(a, b) for a, b in zip(xs, outs[0][1]))
    for k, A in enumerate(systems):
        assert oracle.true_relres(A, bs[k], outs[0][1][k]) <= 1e-9 * (1 + 1e-6)
        if precision == "fp64":
            ref = oracle.pcg(A, bs[k], tol=1e-9, maxit=5000, precond=1)
            assert abs(outs[0][0][k] - ref.iters) <= max(3, math.ceil(0.02 * ref.iters))
    cg.cg_destroy(h)
