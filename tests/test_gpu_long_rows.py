"""Rows of 17 to 2044 entries in the caller's CSR product: 32 chains and a fixed tree, whatever the
row's place in its block.  The value is the one a warp of 32 lanes forms (chain l of entries l, l +
32, ..., then an xor tree), bit for bit: fused multiply-adds and single additions, all exactly
rounded, are emulated on the host in extended precision."""
from fractions import Fraction

import numpy as np
import pytest

import cgproblems as gen
from helpers import adversarial, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2608_09647_gb300 as cg  # noqa: E402


def warp_sum(vals, x):
    s = [0.0] * 32
    for k, (a, b) in enumerate(zip(vals.tolist(), x.tolist())):
        s[k % 32] = float(Fraction(a) * Fraction(b) + Fraction(s[k % 32]))  # correctly rounded
    for o in (16, 8, 4, 2, 1):
        s = [s[l] + s[l ^ o] for l in range(32)]
    return s[0]


@pytest.mark.parametrize("lengths", [(17, 24, 31, 32, 33), (63, 64, 65, 200), (511, 1024, 1500), (2044,)],
                         ids=lambda v: "_".join(map(str, v)))
def test_long_rows_sum_as_a_warp(lengths):
    n = 3000
    rows = [(11 + 257 * j, L) for j, L in enumerate(lengths)]
    A = adversarial(n, 5 + lengths[0], long_rows=rows)
    x = np.random.default_rng(1).uniform(-1.0, 1.0, n)
    h = cg.cg_create(n, *to_device(A))
    y = torch.empty(n, dtype=torch.float64, device="cuda")
    assert cg.cg_spmv(h, torch.from_numpy(x).cuda(), y) == cg.CG_OK
    cg.cg_destroy(h)
    got = y.cpu().numpy()
    for r, L in rows:
        k0, k1 = A.rowptr[r], A.rowptr[r + 1]
        assert k1 - k0 == L
        assert got[r] == warp_sum(A.vals[k0:k1], x[A.colind[k0:k1]])
