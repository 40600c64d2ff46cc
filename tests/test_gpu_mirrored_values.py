"""Which slots of a symmetric diagonal layout the refinement's loop reads, by the bytes an
iteration of it must move: the right half of the slots from about 1 MB to 63 MB of that half and
four vectors, all of them elsewhere, whatever was solved on the handle before."""
import pytest

import cgproblems as gen
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


@pytest.mark.parametrize("name", ["small", "one_sided"])
def test_all_slots_where_the_half_does_not_serve(name):
    A = gen.lap3d7(16 if name == "small" else 96)
    if name == "one_sided":
        A.vals[A.rowptr[A.n // 2 + 1] - 1] *= 1.0 + 2.0 ** -20
    h = cg.cg_create(A.n, *to_device(A))
    assert bytes_per_row(h, A.n, NONE, RU) == 4 * 6 + VECTORS
    cg.cg_destroy(h)
