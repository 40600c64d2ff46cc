"""Which slots of a symmetric diagonal layout the refinement's loop reads, by the bytes an
iteration of it must move: the right half of the slots from 16 MiB to 63 MiB of that half and
four vectors, all of them elsewhere, whatever was solved on the handle before."""
import math

import numpy as np
import pytest

import cgproblems as gen
import oracle
from helpers import to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2608_09647_gb300 as cg  # noqa: E402

VECTORS = 40  # bytes a row of the fp32 loop's vectors (constant diagonal)
JACOBI, NONE, RU, IR, FP64 = (cg.CG_PRECOND_JACOBI, cg.CG_PRECOND_NONE, cg.CG_PREC_FP32_RU, cg.CG_PREC_FP32_IR,
                              cg.CG_PREC_FP64)


def bytes_per_row(h, n, precond, precision):
    b = torch.ones(n, dtype=torch.float64, device="cuda")
    st, _, _ = cg.cg_solve(h, b, torch.zeros_like(b), 1e-6, 5, precond, precision)
    assert st >= 0, cg.cg_last_error(h)
    return cg.cg_get_solve_info(h)["kernel_bytes_per_iter"] / n


@pytest.mark.parametrize("order", [(RU, FP64, RU), (FP64, RU, FP64, IR, RU)], ids=["ru_first", "fp64_first"])
@pytest.mark.parametrize("precond", [JACOBI, NONE], ids=["jacobi", "none"])
def test_fp64_solves_leave_the_mirrored_values_on(precond, order):
    A = gen.lap3d7(96)  # whole slices: 96^3 = 32 * 27,648
    h = cg.cg_create(A.n, *to_device(A))
    for precision in order:
        got = bytes_per_row(h, A.n, precond, precision)
        if precision != FP64:
            assert got == 4 * 3 + VECTORS
    cg.cg_destroy(h)


@pytest.mark.parametrize("name", ["below", "one_sided"])
def test_all_slots_where_the_half_does_not_serve(name):
    A = gen.lap3d7(84 if name == "below" else 96)  # 84^3: 28 bytes a row are 0.3 MB short of the limit
    if name == "one_sided":
        A.vals[A.rowptr[A.n // 2 + 1] - 1] *= 1.0 + 2.0 ** -20
    h = cg.cg_create(A.n, *to_device(A))
    assert bytes_per_row(h, A.n, NONE, RU) == 4 * 6 + VECTORS
    cg.cg_destroy(h)


CASES = {  # the smallest ones past the limit, with ragged last slices, one for each number of slots
    "5pt": (lambda: gen.lap2d(841, 5, 0.5), 2),
    "7pt": (lambda: gen.lap3d7(85), 3),
    "9pt": (lambda: gen.q1aniso(729, 1.5, 1.9, 0.05, 8), 4),
}


@pytest.mark.parametrize("precond", [JACOBI, NONE], ids=["jacobi", "none"])
@pytest.mark.parametrize("name", CASES)
def test_mirrored_refinement_matches_oracle(name, precond):
    """Tolerances as in test_gpu_symmetric_slices.py: the fp64 true residual recomputed by the
    oracle <= tol, the iteration count within 10 %, the solution to 1e-6."""
    make, slots = CASES[name]
    A = make()
    on = A.colind == np.repeat(np.arange(A.n), np.diff(A.rowptr))
    A = gen.CSR(A.n, A.rowptr, A.colind, np.where(on, A.vals * 1.01, A.vals), A.name + "_shifted")
    b = oracle.spmv(A, gen.xstar(A.n, 5))
    tol = 1e-10
    h = cg.cg_create(A.n, *to_device(A))
    x = torch.zeros(A.n, dtype=torch.float64, device="cuda")
    st, it, rel = cg.cg_solve(h, torch.from_numpy(b).cuda(), x, tol, 5000, precond, RU)
    info = cg.cg_get_solve_info(h)
    cg.cg_destroy(h)
    d = A.vals[on]
    vectors = VECTORS + (4 if precond == JACOBI and d.min() != d.max() else 0)
    slices = -(-A.n // 32)
    assert info["kernel_bytes_per_iter"] == slices * 32 * slots * 4 + vectors * A.n
    ref = oracle.pcg_ru(A, b, tol=tol, tol_in=0.1, precond=int(precond == JACOBI))
    assert st == ref.status == cg.CG_OK
    assert abs(it - ref.iters) <= max(5, math.ceil(0.1 * ref.iters)), (it, ref.iters)
    xh = x.cpu().numpy()
    assert rel <= tol and oracle.true_relres(A, b, xh) <= tol * (1 + 1e-6)
    assert np.linalg.norm(xh - ref.x) <= 1e-6 * np.linalg.norm(ref.x)
