"""GPU: C = alpha A + beta B has each product rounded once and one rounded sum, bit
for bit, by every path a row can take (a team's lanes, a warp's shared memory, the
slots of rows that are not strictly ascending, a CTA), with coefficients whose
products are not exact: there a fused multiply-add would differ."""
import numpy as np
import pytest

from paper_2103_11991_gb300 import inputs as I
from tests.test_gpu_spadd import _check, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [(1, 8), (9, 16), (17, 32), (33, 128), (200, 400)])
@pytest.mark.parametrize("order", ["sorted", "unsorted"])
@pytest.mark.parametrize("alpha,beta", [(1.3, -0.7), (1.0, -0.7), (1.3, 1.0), (1 / 3, 0.1)])
def test_products_are_rounded_before_the_sum(lens, order, alpha, beta):
    m, n = 150, 4 * lens[1]  # many shared columns
    A = I.random_rows(m, n, *lens, seed=lens[0], purpose="rrA")
    B = I.random_rows(m, n, *lens, seed=lens[1], purpose="rrB")
    A.vals, B.vals = (I.uniform01(s, "rr.v", M.nnz) * 2 - 1 for s, M in ((3, A), (4, B)))
    if order == "unsorted":
        for M in (A, B):
            for r in range(m):
                s, e = M.rowptr[r], M.rowptr[r + 1]
                M.colind[s:e] = M.colind[s:e][::-1].copy()
    rp, ci, va = _run(A, B, alpha, beta)
    _check(A, B, alpha, beta, rp, ci, va, exact=True)
