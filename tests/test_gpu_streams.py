"""First solves on a stream of their own while another thread keeps the default stream busy:
what a handle sets up on the default stream has to be complete before the solve's stream uses
it.  The result is the one obtained alone, bit for bit."""
import threading

import numpy as np
import pytest

import cgproblems as gen
from helpers import to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2608_09647_gb300 as cg  # noqa: E402


@pytest.mark.parametrize("precision", [cg.CG_PREC_FP64, cg.CG_PREC_FP32_RU], ids=["fp64", "ru"])
def test_first_solve_beside_work_on_the_default_stream(precision):
    A = gen.lap3d7(24)
    csr = to_device(A)
    b = torch.from_numpy(gen.xstar(A.n, 3)).cuda()
    torch.cuda.synchronize()

    def first_solve():
        h = cg.cg_create(A.n, *csr)
        x = torch.zeros_like(b)
        st, it, rel = cg.cg_solve(h, b, x, 1e-10, 2000, cg.CG_PRECOND_JACOBI, precision)
        x = x.cpu().numpy()
        cg.cg_destroy(h)
        return (st, it, rel), x

    alone = first_solve()
    assert alone[0][0] == cg.CG_OK
    stop = threading.Event()

    def occupy():  # ~1 ms of work at a time
        while not stop.is_set():
            torch.cuda._sleep(2000000)
            torch.cuda.default_stream().synchronize()

    busy = threading.Thread(target=occupy)
    busy.start()
    try:
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(10):
                facts, x = first_solve()
                assert facts == alone[0]
                assert np.array_equal(x, alone[1])
    finally:
        stop.set()
        busy.join()
