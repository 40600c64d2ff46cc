"""Solves of different sizes from two host threads, each on its own handle and stream (one
handle belongs to one thread; several handles may solve at the same time).  Every call has to
succeed and to give the result it gives alone, bit for bit: the forms' sums do not depend on
what else runs."""
import threading
import time

import numpy as np
import pytest

import cgproblems as gen
from helpers import to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2608_09647_gb300 as cg  # noqa: E402

SECONDS = 3.0  # of calls in each thread


def handle_solver(A, maxit=1):
    """A function that solves A on a handle of its own, in the form that auto takes."""
    csr = to_device(A)
    h = cg.cg_create(A.n, *csr)
    b = torch.from_numpy(gen.xstar(A.n, 3)).cuda()
    x = torch.zeros_like(b)

    def solve():
        st, it, _ = cg.cg_solve(h, b, x.zero_(), 1e-14, maxit, cg.CG_PRECOND_JACOBI)
        info = cg.cg_get_solve_info(h)
        return (st, it, info["loop_form"], info["grid_ctas"], cg.cg_last_error(h) if st < 0 else ""), x
    return solve


def noalloc_solver(A, maxit=1):
    csr = to_device(A)
    b = torch.from_numpy(gen.xstar(A.n, 3)).cuda()
    x = torch.zeros_like(b)

    def solve():
        st, it, _ = cg.cg_solve_noalloc(*csr, b, x.zero_(), 1e-14, maxit)
        return (st, it), x
    return solve


PAIRS = {
    # two systems whose vectors the SMs' shared memory holds, a small and a large one
    "shared_memory": (lambda: handle_solver(gen.lap2d(400, 9, 0.5)), lambda: handle_solver(gen.lap2d(140, 9, 0.5))),
    # two systems of the cluster form
    "cluster": (lambda: handle_solver(gen.lap2d(120)), lambda: handle_solver(gen.lap2d(24))),
    # the handle-free solve shares the cluster form's kernels
    "noalloc": (lambda: handle_solver(gen.lap2d(120)), lambda: noalloc_solver(gen.lap2d(24))),
}


@pytest.mark.parametrize("name", PAIRS)
def test_two_threads_solve_different_sizes(name):
    solvers = [make() for make in PAIRS[name]]
    alone = [(facts, x.cpu().numpy()) for facts, x in (s() for s in solvers)]
    assert all(facts[:2] == (cg.CG_NOT_CONVERGED, 1) for facts, _ in alone)
    failures = []
    start = threading.Barrier(2)

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            start.wait()
            end, calls = time.time() + SECONDS, 0
            while time.time() < end and not failures:
                facts, x = solvers[k]()
                calls += 1
                if facts != alone[k][0]:
                    failures.append((k, calls, facts))
            if not np.array_equal(x.cpu().numpy(), alone[k][1]):
                failures.append((k, calls, "result"))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
