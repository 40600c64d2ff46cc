"""Right-hand sides so small that rho = r.z falls below 5.6e-309, where 1 / rho is infinite, in
every fp64 loop form: scaled by a power of two the solve takes the steps of the unscaled one.

Bounds: the status and the true-residual test as ever; the iteration count within max(3, 2 %) of
the unscaled solve's, as for any two solves of the same system in this suite (rho has about 30
bits left at the end); the solution to 1e-9 of the unscaled one, the tolerance being 1e-12.
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

SCALE, TOL, MAXIT = 2.0 ** -482, 1e-12, 5000  # |b| ~ 1e-143, |r|^2 ~ 1e-310 at the end
JACOBI, NONE, FSAI = cg.CG_PRECOND_JACOBI, cg.CG_PRECOND_NONE, cg.CG_PRECOND_FSAI


def shifted_grid(m):
    A = gen.lap2d(m, 9, 0.5)
    on = A.colind == np.repeat(np.arange(A.n), np.diff(A.rowptr))
    return gen.CSR(A.n, A.rowptr, A.colind, np.where(on, A.vals * 1.02, A.vals), A.name + "_shifted")


def rhs(A):
    return oracle.spmv(A, gen.xstar(A.n, 3))


def compare(A, b, one, tiny):
    (st1, it1, _), x1 = one
    (st, it, rel), x = tiny
    assert st1 == cg.CG_OK
    assert st == cg.CG_OK and rel <= TOL
    assert abs(it - it1) <= max(3, math.ceil(0.02 * it1)), (it, it1)
    assert np.linalg.norm(x / SCALE - x1) <= 1e-9 * np.linalg.norm(x1)


FORMS = {  # rows a side, options, the form that has to have run
    "cluster": (60, {}, 4),
    "shared_memory": (140, {}, 1),
    "persistent": (140, {cg.CG_OPT_GRID_CTAS: 152}, 1),
    "graph": (140, {cg.CG_OPT_LOOP_MODE: 2}, 2),
}


@pytest.mark.parametrize("precond", [JACOBI, NONE], ids=["jacobi", "none"])
@pytest.mark.parametrize("form", FORMS)
def test_tiny_rhs(form, precond):
    side, options, want = FORMS[form]
    A = shifted_grid(side)
    b = rhs(A)
    h = cg.cg_create(A.n, *to_device(A))
    for k, v in options.items():
        assert cg.cg_set_option(h, k, v) == cg.CG_OK
    got = []
    for s in (1.0, SCALE):
        x = torch.zeros(A.n, dtype=torch.float64, device="cuda")
        facts = cg.cg_solve(h, torch.from_numpy(b * s).cuda(), x, TOL, MAXIT, precond)
        assert cg.cg_get_solve_info(h)["loop_form"] == want
        got.append((facts, x.cpu().numpy()))
    cg.cg_destroy(h)
    compare(A, b, *got)


def test_tiny_rhs_noalloc():
    A = shifted_grid(60)
    b = rhs(A)
    csr = to_device(A)
    got = []
    for s in (1.0, SCALE):
        x = torch.zeros(A.n, dtype=torch.float64, device="cuda")
        got.append((cg.cg_solve_noalloc(*csr, torch.from_numpy(b * s).cuda(), x, TOL, MAXIT), x.cpu().numpy()))
    compare(A, b, *got)


def test_tiny_rhs_fsai():
    A = shifted_grid(60)
    b = rhs(A)
    h = cg.cg_create(A.n, *to_device(A))
    assert cg.cg_fsai_set_factor(h, torch.from_numpy(fsai.classic(A)).cuda()) == cg.CG_OK
    got = []
    for s in (1.0, SCALE):
        x = torch.zeros(A.n, dtype=torch.float64, device="cuda")
        got.append((cg.cg_solve(h, torch.from_numpy(b * s).cuda(), x, TOL, MAXIT, FSAI), x.cpu().numpy()))
    cg.cg_destroy(h)
    compare(A, b, *got)


@pytest.mark.parametrize("precond", [JACOBI, NONE], ids=["jacobi", "none"])
def test_tiny_rhs_batch(precond):
    systems = [shifted_grid(m) for m in (20, 60, 45)]
    bs = [rhs(A) for A in systems]
    on_device = [to_device(A) for A in systems]
    h = cg.cg_batch_create([d[0] for d in on_device], [d[1] for d in on_device], [d[2] for d in on_device])
    got = []
    for s in (1.0, SCALE):
        xs = [torch.zeros(A.n, dtype=torch.float64, device="cuda") for A in systems]
        st, its, rels = cg.cg_solve_batch(h, [torch.from_numpy(b * s).cuda() for b in bs], xs, TOL, MAXIT, precond)
        got.append([((st, int(its[k]), float(rels[k])), x.cpu().numpy()) for k, x in enumerate(xs)])
    cg.cg_destroy(h)
    for A, b, one, tiny in zip(systems, bs, *got):
        compare(A, b, one, tiny)
