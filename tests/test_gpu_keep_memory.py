"""GPU: keeping rows for the numeric phase is optional: a product on a device with
little free memory runs without, or with as much as there is room for."""
import numpy as np
import pytest

from paper_2103_11991_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# free: room for some of the 0.84 GB that the kept rows want, and for little of it
@pytest.mark.parametrize("free_mb", [700, 160])
@pytest.mark.parametrize("learned", [False, True])
def test_product_beside_a_nearly_full_device(free_mb, learned):
    import torch
    from paper_2103_11991_gb300 import spgemm as K
    k, m, per = 300000, 20000, 30
    B = I.random_rows(m, k, per, per, seed=1, purpose="kmB")
    A = I.random_rows(m, m, per, per, seed=2, purpose="kmA")
    dA, dB = K.DeviceCSR.from_host(A), K.DeviceCSR.from_host(B)
    opts = dict(arith=1, small_max_rows=0)
    with K.SpGEMM(structure_cache=0, **opts) as op:
        rp0, nnz = op.symbolic(dA, dB)
        ci0, va0 = op.numeric(dA, dB, rp0, nnz)
        op.sync()
    with K.SpGEMM(structure_cache=0, **opts) as op:  # the bound of the values' error
        pos = [K.DeviceCSR(M.m, M.n, M.rowptr, M.colind, M.vals.abs()) for M in (dA, dB)]
        _, ab = op.numeric(*pos, *op.symbolic(*pos))
        op.sync()
    rp, ci, va = torch.empty_like(rp0), torch.empty_like(ci0), torch.empty_like(va0)
    torch.cuda.empty_cache()
    op = K.SpGEMM(**opts)
    try:
        rest = max(0, torch.cuda.mem_get_info()[0] - (free_mb << 20))
        full = torch.empty(rest, dtype=torch.uint8, device="cuda")
        if learned:
            n2 = K.kk_spgemm_learned_symbolic(op.h, dA, dB, rp)
            K.kk_spgemm_learned_numeric(op.h, dA, dB, rp, ci, va)
        else:
            n2 = K.kk_spgemm_symbolic(op.h, dA, dB, rp)
            K.kk_spgemm_numeric(op.h, dA, dB, rp, ci, va)
        op.sync()
        del full
        assert n2 == nnz and torch.equal(rp, rp0) and torch.equal(ci, ci0)
        assert bool(((va - va0).abs() <= 2e-12 * ab).all())
    finally:
        op.close()
        torch.cuda.empty_cache()
