"""GPU: index arrays that changed in place between the phases, on rows whose
column chunks are computed from what the symbolic phase kept: reported
(KK_ERR_STRUCTURE_MISMATCH) also where the new products fall on kept columns
only, with every index in range and the row pointers as they were."""
import numpy as np
import pytest

from paper_2103_11991_gb300 import inputs as I
from tests._gpu import check_against_oracle

pytestmark = pytest.mark.gpu


def _operands():
    # rows of A: 40 rows of B, the first of which is in all of them; then rows whose
    # span is a window's
    n, k = 200, 90000
    B = I.random_rows(n, k, 60, 90, seed=1, purpose="ccB")
    near = I.random_rows(30, 3000, 20, 30, seed=4, purpose="ccN")
    B = I.ensure_csr(n + 30, k, np.concatenate([B.rowptr, B.rowptr[-1] + near.rowptr[1:]]),
                     np.concatenate([B.colind, near.colind]), np.concatenate([B.vals, near.vals]))
    pick = np.sort(np.argsort(I.uniform01(2, "cc.p", 50 * (n - 1)).reshape(50, n - 1), axis=1)[:, :39] + 1, axis=1)
    cols = np.concatenate([np.zeros((50, 1), np.int64), pick], axis=1).reshape(-1)
    tail = n + np.tile(np.arange(0, 30, 3), 20)  # 20 rows of 10
    A = I.ensure_csr(70, n + 30, np.concatenate([np.arange(51) * 40, 2000 + np.arange(1, 21) * 10]),
                     np.concatenate([cols, tail]), I.uniform01(3, "cc.a", 2200) - 0.5)
    return A, B


# tier 2: no row of the call takes the window tier; -1: with window rows' own fingerprint
@pytest.mark.parametrize("tier", [2, -1])
@pytest.mark.parametrize("debug", [0, 1])
@pytest.mark.parametrize("which,jacobi", [("A", False), ("B", False), ("both", False), ("values", False), ("B", True)])
def test_changed_in_place_is_reported(tier, debug, which, jacobi):
    import torch
    from paper_2103_11991_gb300 import spgemm as K
    A, B = _operands()
    if jacobi:
        A = I.with_diagonal(I.ensure_csr(A.m, A.m, A.rowptr, A.colind % A.m, A.vals), 4)
        end = int(B.rowptr[A.m])
        B = I.ensure_csr(A.m, B.n, B.rowptr[:A.m + 1], B.colind[:end], B.vals[:end])
    dA, dB = K.DeviceCSR.from_host(A), K.DeviceCSR.from_host(B)
    with K.SpGEMM(force_tier=tier, debug_checks=debug, small_max_rows=0, arith=1) as op:
        rp, nnz = op.symbolic(dA, dB)
        st = op.stats()
        assert st["num_cta_rows"] + st["num_dense_rows"] >= 50
        assert jacobi or (st["sym_window_rows"] > 0) == (tier == -1)
        a, b = A.colind.copy(), B.colind.copy()
        if which in ("A", "both"):
            a[1:2000:2] = a[0:2000:2]  # pairs of entries meet in one row of B: a subset of the columns
        if which in ("B", "both"):  # B's first row repeats its first half
            half = int(B.rowptr[1]) // 2
            b[half:2 * half] = b[:half]
        dA.colind.copy_(torch.from_numpy(a).cuda())
        dB.colind.copy_(torch.from_numpy(b).cuda())
        run = (lambda: op.jacobi_numeric(dA, dB, rp, nnz, 0.5)) if jacobi else (lambda: op.numeric(dA, dB, rp, nnz))
        if which == "values":
            ci, va = run()
            op.sync()
            check_against_oracle(A, B, rp.cpu().numpy(), ci.cpu().numpy(), va.cpu().numpy())
            return
        with pytest.raises(K.KKError) as e:
            run()
            op.sync()
        assert e.value.status == 4
        # the arrays as they were: the kept rows serve them again
        dA.colind.copy_(torch.from_numpy(A.colind).cuda())
        dB.colind.copy_(torch.from_numpy(B.colind).cuda())
        ci, va = op.numeric(dA, dB, rp, nnz)
        op.sync()
        check_against_oracle(A, B, rp.cpu().numpy(), ci.cpu().numpy(), va.cpu().numpy())
