"""The grid-wide rounds of a persistent fp32 refinement: two a residual (the product, its sums),
one more where the search direction is carried over, three an iteration.  Counted with the
library's fault injection: the last round skipped, the solve runs into its limit; one past the
last, it does not.  (A residual's sums may not cost rounds of their own: they would outweigh a
small system's iterations.)
"""
import pytest

import cgproblems as gen
from helpers import to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2608_09647_gb300 as cg  # noqa: E402


@pytest.mark.parametrize("precision", [cg.CG_PREC_FP32_IR, cg.CG_PREC_FP32_RU], ids=["ir", "ru"])
@pytest.mark.parametrize("precond", [cg.CG_PRECOND_JACOBI, cg.CG_PRECOND_NONE], ids=["jacobi", "none"])
def test_rounds_of_a_refinement(precond, precision):
    A = gen.lap3d7(20)  # constant diagonal: r.r follows from r.z, never a round of its own
    h = cg.cg_create(A.n, *to_device(A))
    assert cg.cg_set_option(h, cg.CG_OPT_LOOP_MODE, 1) == cg.CG_OK
    b = torch.from_numpy(gen.xstar(A.n, 3)).cuda()

    def solve():
        x = torch.zeros_like(b)
        return cg.cg_solve(h, b, x, 1e-10, 1000, precond, precision)

    st, iters, _ = solve()
    info = cg.cg_get_solve_info(h)
    assert st == cg.CG_OK and info["loop_form"] == 1 and info["grid_ctas"] > 1 and info["restarts"] >= 2
    rounds = 2 * (info["restarts"] + 1) + 3 * iters
    if precision == cg.CG_PREC_FP32_RU:
        rounds += info["restarts"] - 1
    assert cg.cg_set_option(h, cg.CG_OPT_BARRIER_TIMEOUT_MS, 50) == cg.CG_OK
    assert cg.cg_set_option(h, cg.CG_OPT_DEBUG_SKIP_ARRIVAL, rounds + 1) == cg.CG_OK
    assert solve()[:2] == (cg.CG_OK, iters)
    assert cg.cg_set_option(h, cg.CG_OPT_DEBUG_SKIP_ARRIVAL, rounds) == cg.CG_OK
    assert solve()[0] == cg.CG_ERR_TIMEOUT
    cg.cg_destroy(h)
