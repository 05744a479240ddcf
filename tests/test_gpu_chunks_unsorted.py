"""GPU: column chunks of rows of A stored in no order and with repeated columns,
with few and many products per chunk, against the oracle."""
import numpy as np
import pytest

from paper_2103_11991_gb300 import inputs as I
from tests._gpu import check_against_oracle, run_gpu

pytestmark = pytest.mark.gpu


# B's first rows are the ones whose entries lie at the start of its arrays; lens of
# B: fewer products than a CTA has threads, an odd number of steps, several of them
@pytest.mark.parametrize("lens", [(8, 20), (40, 60), (120, 200), (500, 700)])
@pytest.mark.parametrize("k", [65536, 90000, 300000])
@pytest.mark.parametrize("repeats", [False, True])
def test_rows_in_no_order(lens, k, repeats):
    m, n, per = 40, 300, 60
    B = I.random_rows(n, k, *lens, seed=k + lens[0], purpose="cuB")
    pick = np.argsort(I.uniform01(lens[1], "cu.p", m * n).reshape(m, n), axis=1)[:, :per]
    pick[:, -1] = 0  # the first row of B last
    if repeats:
        pick[:, 1::3] = pick[:, 0::3]
    A = I.ensure_csr(m, n, np.arange(m + 1) * per, pick.reshape(-1), I.uniform01(k, "cu.v", m * per) - 0.5)
    rp, ci, va, _, _ = run_gpu(A, B, force_tier=2, arith=1)
    check_against_oracle(A, B, rp, ci, va)
