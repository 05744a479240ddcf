"""GPU: chunked numeric phase of the wide tier's kept rows, at the edges of its
chunks, of B's index and of the kept-row budget, against the oracle."""
import numpy as np
import pytest

from oracle import jacobi as OJ
from paper_2103_11991_gb300 import inputs as I
from tests._gpu import check_against_oracle, run_gpu

pytestmark = pytest.mark.gpu


# k: one to three 2,048-word parts of the bit vector, either side of the width
# at which chunks end at coarser columns; lens: B rows without and with an index
@pytest.mark.parametrize("k", [1500, 65536, 65537, 131072, 262144, 262145, 300000])
@pytest.mark.parametrize("la,lb", [((30, 60), (40, 127)), ((4, 9), (500, 1400)), ((260, 300), (5, 40))])
def test_chunks_match_oracle(k, la, lb):
    n = 700
    A = I.random_rows(60, n, *la, seed=k + la[0], purpose="chA")
    B = I.random_rows(n, k, *lb, seed=k + lb[0], purpose="chB")
    kept = run_gpu(A, B, force_tier=2, arith=1)
    check_against_oracle(A, B, *kept[:3])
    rebuilt = run_gpu(A, B, force_tier=2, arith=1, structure_cache=0)
    assert np.array_equal(kept[0], rebuilt[0]) and np.array_equal(kept[1], rebuilt[1])
    few = run_gpu(A, B, force_tier=2, arith=1, wide_cache_mb=1)
    check_against_oracle(A, B, *few[:3])


@pytest.mark.parametrize("count", [1024, 1025, 3071, 3072, 3073, 3584, 3585, 20000])
def test_dense_columns_at_chunk_ends(count):
    # neighbouring columns: every group of columns is full, chunks end between them
    k = 70000
    lens = np.array([count, count // 2, 7])
    cols = np.concatenate([np.arange(count), np.arange(count // 2) * 2, np.arange(7) * 100]) + 300
    B = I.ensure_csr(3, k, np.concatenate([[0], np.cumsum(lens)]), cols, I.uniform01(count, "ch.b", int(lens.sum())))
    A = I.ensure_csr(4, 3, [0, 3, 5, 6, 9], [0, 1, 2, 0, 2, 0, 2, 1, 0], I.uniform01(count, "ch.a", 9) - 0.5)
    rp, ci, va, _, _ = run_gpu(A, B, force_tier=2)
    check_against_oracle(A, B, rp, ci, va)


def test_chunks_refresh_other_arrays_and_jacobi():
    import torch
    from paper_2103_11991_gb300 import spgemm as K
    A = I.with_diagonal(I.random_rows(500, 500, 30, 60, seed=3, purpose="chJ"), 4)
    B = I.random_rows(500, 90000, 80, 200, seed=5, purpose="chK")
    dA, dB = K.DeviceCSR.from_host(A), K.DeviceCSR.from_host(B)
    with K.SpGEMM(force_tier=2) as op:
        rp, nnz = op.symbolic(dA, dB)
        for seed in (6, 7):  # new values on the kept structure
            B.vals = I.uniform01(seed, "ch.v", B.nnz) - 0.5
            dB.vals.copy_(torch.from_numpy(B.vals).cuda())
            ci, va = op.numeric(dA, dB, rp, nnz)
            op.sync()
            check_against_oracle(A, B, rp.cpu().numpy(), ci.cpu().numpy(), va.cpu().numpy())
        ci, va = op.jacobi_numeric(dA, dB, rp, nnz, 2.0 / 3.0)
        op.sync()
        ref = OJ.jacobi_spgemm(A, B, 2.0 / 3.0)
        assert np.array_equal(ci.cpu().numpy(), ref.colind)
        assert np.all(np.abs(va.cpu().numpy() - ref.vals) <= 1e-12 * OJ.jacobi_abs(A, B, 2.0 / 3.0))
        # the same matrices in other arrays: nothing kept is used
        dB2 = K.DeviceCSR(B.m, B.n, dB.rowptr.clone(), dB.colind.clone(), dB.vals.clone())
        ci, va = op.numeric(dA, dB2, rp, nnz)
        op.sync()
        check_against_oracle(A, B, rp.cpu().numpy(), ci.cpu().numpy(), va.cpu().numpy())


# rows that leave the hash kernels for the chunks by their products: either side of
# that line (513 or a 512th of B's columns) and of the columns a kept row needs
@pytest.mark.parametrize("k", [65536, 65537, 98304, 131072, 262144, 262145])
@pytest.mark.parametrize("flop,count", [(511, 300), (512, 257), (513, 256), (513, 257), (767, 767),
                                        (768, 256), (768, 257), (769, 256), (769, 257), (1023, 400), (1024, 400), (1040, 520),
                                        (2047, 700), (2048, 700)])
def test_rows_beyond_the_hash_kernels(k, flop, count):
    m = 40
    full, rest = divmod(flop, count)
    lens = np.tile([count] * full + ([rest] if rest else []), m)
    per = len(lens) // m
    pick = [np.sort(np.argsort(I.uniform01(i, "ch.p%d" % flop, k))[:count]) for i in range(m)]
    cols = np.concatenate([np.concatenate([pick[i]] * full + ([pick[i][:rest]] if rest else [])) for i in range(m)])
    B = I.ensure_csr(m * per, k, np.concatenate([[0], np.cumsum(lens)]), cols,
                     I.uniform01(k, "ch.q", len(cols)) * 2 - 1)
    A = I.ensure_csr(m, m * per, np.arange(m + 1) * per, np.arange(m * per),
                     I.uniform01(flop, "ch.r", m * per) * 2 - 1)
    rp, ci, va, _, st = run_gpu(A, B, arith=1, small_max_rows=0)
    assert np.all(np.diff(rp) == count)
    early = flop >= max(513, k // 512)
    if k in (98304, 131072, 262144):  # every row's span is beyond the window tier's
        assert (st["sym_cta_rows"] + st["sym_dense_rows"] == m) == early
        assert st["num_dense_rows"] == (m if early and count > 256 else 0)
    check_against_oracle(A, B, rp, ci, va)
    few = run_gpu(A, B, arith=1, small_max_rows=0, wide_cache_mb=1)  # most rows find no slot
    check_against_oracle(A, B, *few[:3])
    plain = run_gpu(A, B, arith=1, small_max_rows=0, structure_cache=0)
    assert np.array_equal(rp, plain[0]) and np.array_equal(ci, plain[1])


# the widest B whose kept rows are computed in chunks, and the next: rows with few
# and with many columns, kept, without room to keep them, and with nothing kept
@pytest.mark.parametrize("k", [524288, 524289])
@pytest.mark.parametrize("la,lb", [((6, 9), (300, 500)), ((200, 300), (40, 80))])
def test_chunks_at_the_widest_b(k, la, lb):
    A = I.random_rows(50, 600, *la, seed=k + la[0], purpose="chX")
    B = I.random_rows(600, k, *lb, seed=k + lb[0], purpose="chY")
    kept = run_gpu(A, B, arith=1, small_max_rows=0)
    check_against_oracle(A, B, *kept[:3])
    for other in (dict(wide_cache_mb=1), dict(structure_cache=0)):
        got = run_gpu(A, B, arith=1, small_max_rows=0, **other)
        check_against_oracle(A, B, *got[:3])
        assert np.array_equal(kept[0], got[0]) and np.array_equal(kept[1], got[1])
