"""GPU: rank-tier rows whose bits come from the compressed B of the symbolic call
while B's columns changed in place: a column of C that no product of the new B
reaches is reported (KK_ERR_STRUCTURE_MISMATCH), also without the fingerprint of
kept rows (structure_cache = 0, debug_checks = 1)."""
import numpy as np
import pytest

from paper_2103_11991_gb300 import inputs as I
from tests._gpu import check_against_oracle

pytestmark = pytest.mark.gpu


# n: rows of one warp and of two; where: which column of the row loses its product
@pytest.mark.parametrize("n", [3000, 40000])
@pytest.mark.parametrize("where", ["first", "middle", "last"])
@pytest.mark.parametrize("cache,debug", [(0, 0), (1, 1), (1, 0)])
def test_column_without_a_product_is_reported(n, where, cache, debug):
    import torch
    from paper_2103_11991_gb300 import spgemm as K
    k, m = 60, 90
    # even columns but for row 0, which holds the first, the last and an odd one
    B = I.random_rows(k, n // 2 - 2, 25, 40, seed=n, purpose="rcB")
    lens = np.diff(B.rowptr)
    cols = 2 * B.colind.astype(np.int64) + 2
    own = np.array([0, n // 2 | 1, n - 1])
    B = I.ensure_csr(k, n, np.concatenate([[0], 3 + np.cumsum(np.concatenate([[0], lens[1:]]))]),
                     np.concatenate([own, cols[lens[0]:]]), I.uniform01(n, "rc.v", 3 + int(lens[1:].sum())) - 0.5)
    A = I.random_rows(m, k - 1, 12, 20, seed=7, purpose="rcA")
    al = np.diff(A.rowptr)
    acol = np.insert(A.colind.astype(np.int64) + 1, A.rowptr[:-1], 0)  # row 0 of B in every row
    A = I.ensure_csr(m, k, np.concatenate([[0], np.cumsum(al + 1)]), acol,
                     I.uniform01(8, "rc.a", len(acol)) - 0.5)
    dA, dB = K.DeviceCSR.from_host(A), K.DeviceCSR.from_host(B)
    with K.SpGEMM(structure_cache=cache, debug_checks=debug, small_max_rows=0, arith=1) as op:
        rp, nnz = op.symbolic(dA, dB)
        st = op.stats()
        assert st["num_window_rows"] == m and st["kept_structure_rows"] == 0
        changed = B.colind.copy()
        at = {"first": 0, "middle": 1, "last": 2}[where]
        changed[at] = own[1] if at != 1 else own[0]
        dB.colind.copy_(torch.from_numpy(changed).cuda())
        with pytest.raises(K.KKError) as e:
            op.numeric(dA, dB, rp, nnz)
            op.sync()
        assert e.value.status == 4
        dB.colind.copy_(torch.from_numpy(B.colind).cuda())
        ci, va = op.numeric(dA, dB, rp, nnz)
        op.sync()
        check_against_oracle(A, B, rp.cpu().numpy(), ci.cpu().numpy(), va.cpu().numpy(), exact=True)
