"""GPU: numeric calls whose window rows have no kept structure for their arrays (kept by
no option, or the symbolic call saw other arrays): the structure is derived again, rows
that cannot be kept go to the rank tier beside them, and other structures are reported."""
import numpy as np
import pytest

from paper_2103_11991_gb300 import inputs as I
from tests._gpu import check_against_oracle

pytestmark = pytest.mark.gpu


def _mixed():
    # stencil rows (kept), dense blocks (kept) and spread rows (more words than are kept)
    S = I.stencil_3d(9, 9, 9, 27, 26.0, -1.0)
    n = 2000
    rows = [S.colind[S.rowptr[i]:S.rowptr[i + 1]] for i in range(S.m)]
    rows += [np.arange(40) + 800 + 40 * (i // 40) for i in range(400)]
    g = np.random.default_rng(3)
    rows += [np.sort(g.choice(n, 14, replace=False)) for _ in range(n - len(rows))]
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    return I.ensure_csr(n, n, ptr, np.concatenate(rows), g.random(int(ptr[-1])) - 0.5)


def _clone(K, M):
    return K.DeviceCSR(M.m, M.n, M.rowptr.clone(), M.colind.clone(), M.vals.clone())


@pytest.mark.parametrize("cache", [0, 1])
@pytest.mark.parametrize("other", [False, True])
@pytest.mark.parametrize("arith", [0, 1, 2])
def test_structure_derived_again(cache, other, arith):
    from paper_2103_11991_gb300 import spgemm as K
    A = _mixed()
    dA = K.DeviceCSR.from_host(A)
    with K.SpGEMM(structure_cache=cache, arith=arith, small_max_rows=0) as op:
        rp, nnz = op.symbolic(dA, dA)
        st = op.stats()
        assert (st["kept_structure_rows"] > 0) == (cache == 1)
        use = _clone(K, dA) if other else dA
        for _ in range(2):
            ci, va = op.numeric(use, use, rp, nnz)
            op.sync()
            check_against_oracle(A, A, rp.cpu().numpy(), ci.cpu().numpy(), va.cpu().numpy(), exact=arith == 1)
        ci, va = op.numeric(dA, dA, rp, nnz)  # and the symbolic call's own
        op.sync()
        check_against_oracle(A, A, rp.cpu().numpy(), ci.cpu().numpy(), va.cpu().numpy(), exact=arith == 1)


@pytest.mark.parametrize("cache", [0, 1])
def test_another_structure_is_reported(cache):
    import torch
    from paper_2103_11991_gb300 import spgemm as K
    A = _mixed()
    dA = K.DeviceCSR.from_host(A)
    with K.SpGEMM(structure_cache=cache, arith=1, small_max_rows=0) as op:
        rp, nnz = op.symbolic(dA, dA)
        dB = _clone(K, dA)
        shifted = A.colind.copy()
        s = slice(int(A.rowptr[900]), int(A.rowptr[901]))  # a row of a block, one column further
        shifted[s] += 1
        dB.colind.copy_(torch.from_numpy(shifted).cuda())
        with pytest.raises(K.KKError) as e:
            op.numeric(dA, dB, rp, nnz)
            op.sync()
        assert e.value.status == 4


@pytest.mark.parametrize("cache", [0, 1])
def test_jacobi_and_learned(cache):
    from oracle import jacobi as OJ
    from paper_2103_11991_gb300 import spgemm as K
    A = I.with_diagonal(_mixed(), 5)
    dA = K.DeviceCSR.from_host(A)
    dB = _clone(K, dA)
    with K.SpGEMM(structure_cache=cache, small_max_rows=0) as op:
        rp, nnz = op.symbolic(dA, dB)
        ci, va = op.jacobi_numeric(_clone(K, dA), dB, rp, nnz, 0.7)
        op.sync()
        ref = OJ.jacobi_spgemm(A, A, 0.7)
        assert np.array_equal(ci.cpu().numpy(), ref.colind)
        assert np.all(np.abs(va.cpu().numpy() - ref.vals) <= 1e-12 * OJ.jacobi_abs(A, A, 0.7))
        rp, nnz = op.learned_symbolic(dA, dB)
        ci, va = op.learned_numeric(dA, dB, rp, nnz)
        op.sync()
        check_against_oracle(A, A, rp.cpu().numpy(), ci.cpu().numpy(), va.cpu().numpy())
