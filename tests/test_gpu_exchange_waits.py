"""The bounded waits of the forms whose barriers carry sums, and of the persistent kernel: with an
arrival left out (the library's fault injection on the host's request) the solve ends with
CG_ERR_TIMEOUT after the limit and says where, and the handle solves again to the same bits."""
import re

import numpy as np
import pytest

import cgproblems as gen
from helpers import to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2608_09647_gb300 as cg  # noqa: E402


def solve(h, n, precond):
    b = torch.from_numpy(gen.xstar(n, 7)).cuda()
    x = torch.zeros_like(b)
    st, it, _ = cg.cg_solve(h, b, x, 1e-8, 2000, precond)
    return st, it, x.cpu().numpy(), cg.cg_get_solve_info(h)["grid_ctas"]


# the residual's two exchanges (the first use of their scales takes further rounds), those of
# the loop: p.q, the r update's sums, the one that orders p
@pytest.mark.parametrize("arrival", [1, 2, 5, 9, 14, 15, 16, 40])
@pytest.mark.parametrize("precond", [cg.CG_PRECOND_JACOBI, cg.CG_PRECOND_NONE], ids=["jacobi", "none"])
@pytest.mark.parametrize("form", ["shared_memory", "persistent"])
def test_a_missing_arrival_runs_into_the_limit(form, precond, arrival):
    A = gen.lap2d(130, 9, 0.5)  # 16,900 rows: 529 slices, 133 CTAs in shared memory
    h = cg.cg_create(A.n, *to_device(A))
    assert cg.cg_set_option(h, cg.CG_OPT_LOOP_MODE, 1) == cg.CG_OK
    if form == "persistent":
        assert cg.cg_set_option(h, cg.CG_OPT_GRID_CTAS, 60) == cg.CG_OK
    before = solve(h, A.n, precond)
    assert before[0] == cg.CG_OK and before[3] == (60 if form == "persistent" else 133)
    assert cg.cg_set_option(h, cg.CG_OPT_BARRIER_TIMEOUT_MS, 50) == cg.CG_OK
    assert cg.cg_set_option(h, cg.CG_OPT_DEBUG_SKIP_ARRIVAL, arrival) == cg.CG_OK
    st, _, _, ctas = solve(h, A.n, precond)
    assert st == cg.CG_ERR_TIMEOUT and ctas == before[3]
    said = re.search(r"barrier (\d+), CTA (\d+)\); timed out", cg.cg_last_error(h))
    assert said and int(said.group(1)) == arrival and int(said.group(2)) < ctas
    assert cg.cg_set_option(h, cg.CG_OPT_DEBUG_SKIP_ARRIVAL, 0) == cg.CG_OK
    assert cg.cg_set_option(h, cg.CG_OPT_BARRIER_TIMEOUT_MS, 2000) == cg.CG_OK
    after = solve(h, A.n, precond)
    assert after[:2] == before[:2] and np.array_equal(after[2], before[2])
    cg.cg_destroy(h)
