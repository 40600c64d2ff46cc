"""The bounded waits of the 27-point refinement's shared-memory ring: with a copy that is never
started (the library's fault injection on the host's request) the solve ends with CG_ERR_TIMEOUT
after the limit, says where, and the handle solves again to the bits it gave before.  The
injection reaches only launches that run the ring, so it also shows which matrices do."""
import numpy as np
import pytest

import cgproblems as gen
from helpers import to_device
import test_gpu_ring_spmv
from test_gpu_ring_spmv import box27

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2608_09647_gb300 as cg  # noqa: E402

COPY = 1 << 30  # CG_OPT_DEBUG_SKIP_ARRIVAL from here on: a copy's number


def solve(h, n, precond=cg.CG_PRECOND_JACOBI):
    b = torch.from_numpy(gen.xstar(n, 7)).cuda()
    x = torch.zeros_like(b)
    st, it, _ = cg.cg_solve(h, b, x, 1e-10, 500, precond, cg.CG_PREC_FP32_RU)
    return st, it, x.cpu().numpy()


@pytest.mark.parametrize("precond", [cg.CG_PRECOND_JACOBI, cg.CG_PRECOND_NONE], ids=["jacobi", "none"])
@pytest.mark.parametrize("copy", [1, 3, 4, 10, 41])  # the first, the ring's last, refills, a later product's
def test_a_copy_that_never_starts(copy, precond):
    A = box27(31, 31, 31)  # 931 slices, 24 warps: 39 or 38 slices a warp, two copies each
    h = cg.cg_create(A.n, *to_device(A))
    assert cg.cg_set_option(h, cg.CG_OPT_GRID_CTAS, 3) == cg.CG_OK
    before = solve(h, A.n, precond)
    assert before[0] == cg.CG_OK
    assert cg.cg_set_option(h, cg.CG_OPT_BARRIER_TIMEOUT_MS, 50) == cg.CG_OK
    assert cg.cg_set_option(h, cg.CG_OPT_DEBUG_SKIP_ARRIVAL, COPY + copy) == cg.CG_OK
    st, _, _ = solve(h, A.n, precond)
    assert st == cg.CG_ERR_TIMEOUT and "timed out" in cg.cg_last_error(h)
    assert cg.cg_set_option(h, cg.CG_OPT_DEBUG_SKIP_ARRIVAL, 0) == cg.CG_OK
    assert cg.cg_set_option(h, cg.CG_OPT_BARRIER_TIMEOUT_MS, 2000) == cg.CG_OK
    after = solve(h, A.n, precond)
    assert after[:2] == before[:2] and np.array_equal(after[2], before[2])
    cg.cg_destroy(h)


FORMS = {  # matrix, CTAs (0: automatic), whether it runs the ring (from 16 slices a warp)
    "sixteen": (lambda: box27(21, 17, 23), 2, True),  # 257 slices
    "below": (lambda: box27(21, 17, 23), 3, False),
    "no_runs": (lambda: box27(31, 29, 9, skip=(29 * 31,)), 1, False),
    "automatic": (lambda: gen.diff3d27(109, 0.5, 3), 0, True),
    "automatic_below": (lambda: gen.diff3d27(60, 0.5, 3), 0, False),
}


@pytest.mark.parametrize("name", FORMS)
def test_which_matrices_run_the_ring(name):
    make, ctas, ring = FORMS[name]
    A = make()
    h = cg.cg_create(A.n, *to_device(A))
    assert cg.cg_set_option(h, cg.CG_OPT_GRID_CTAS, ctas) == cg.CG_OK
    assert cg.cg_set_option(h, cg.CG_OPT_BARRIER_TIMEOUT_MS, 50) == cg.CG_OK
    assert cg.cg_set_option(h, cg.CG_OPT_DEBUG_SKIP_ARRIVAL, COPY + 1) == cg.CG_OK
    st, _, _ = solve(h, A.n)
    assert (st == cg.CG_ERR_TIMEOUT) if ring else st >= 0
    cg.cg_destroy(h)


@pytest.mark.parametrize("precond", [cg.CG_PRECOND_JACOBI, cg.CG_PRECOND_NONE], ids=["jacobi", "none"])
def test_fewest_slices_match_oracle(precond):
    test_gpu_ring_spmv.test_refinement_matches_oracle("sixteen", FORMS["sixteen"][0], 2, precond)
