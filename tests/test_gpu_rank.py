"""GPU: rank tier of the numeric phase (rows without kept structure, one or two
warps per row) at the edges of its windows and slot counts, against the oracle.
Float64 sums are in A-row storage order there, for sorted and unsorted B alike,
so they equal the oracle bit for bit."""
import numpy as np
import pytest

from paper_2103_11991_gb300 import inputs as I
from tests._gpu import check_against_oracle, run_gpu

pytestmark = pytest.mark.gpu


def _shuffled(B, seed, repeats):
    """B with its rows' entries in random order; repeats stores some columns twice."""
    rows = np.repeat(np.arange(B.m), np.diff(B.rowptr))
    cols, vals = B.colind, B.vals
    if repeats:
        again = I.uniform01(seed, "rank.again", B.nnz) < 0.2
        rows, cols, vals = (np.concatenate([x, x[again]]) for x in (rows, cols, vals))
    order = np.lexsort((I.uniform01(seed, "rank.order", len(rows)), rows))
    return I._from_sorted_coo(B.m, B.n, rows[order], cols[order], vals[order])


# n: one column to either side of a window's words, and of the widest window;
# lens of A and B: few products, chunks of more than 32 A entries, long B rows
@pytest.mark.parametrize("n", [300, 4095, 4097, 8193, 16384, 32769, 65536, 65537])
@pytest.mark.parametrize("la,lb", [((3, 12), (3, 40)), ((30, 70), (4, 12)), ((2, 6), (60, 200)), ((12, 34), (12, 40))])
@pytest.mark.parametrize("order", ["sorted", "unsorted", "repeats"])
def test_rank_rows_are_exact(n, la, lb, order):
    k = 900
    A = I.random_rows(400, k, *la, seed=n + la[1], purpose="rkA")
    B = I.random_rows(k, n, *lb, seed=n + lb[1], purpose="rkB")
    if order != "sorted":
        B = _shuffled(B, n, order == "repeats")
    rp, ci, va, _, st = run_gpu(A, B, arith=1)
    if n <= 65536 and lb[1] < 60:
        assert st["num_window_rows"] > 0
    check_against_oracle(A, B, rp, ci, va, exact=st["num_team_rows"] + st["num_cta_rows"] + st["num_dense_rows"] == 0)


@pytest.mark.parametrize("count", [255, 256, 257, 511, 512, 513, 1023, 1024, 1025])
@pytest.mark.parametrize("arith", [0, 1, 2])
def test_rank_rows_at_slot_counts(count, arith):
    # every row of C has exactly `count` columns: A picks one long row of B and
    # a few short ones whose columns it holds
    n, m = 30000, 64
    step = n // count
    long_rows = np.arange(count, dtype=np.int64) * step
    cols = [long_rows + s for s in range(8)] + [np.sort((long_rows + s)[(np.arange(20) * 7 + s) % count])
                                                for s in range(8)]
    lens = np.array([len(c) for c in cols])
    B = I.ensure_csr(16, n, np.concatenate([[0], np.cumsum(lens)]), np.concatenate(cols),
                     I.uniform01(count, "rk.b", int(lens.sum())) * 2 - 1)
    acol = np.stack([np.arange(m) % 8, 8 + np.arange(m) % 8], 1).reshape(-1)
    A = I.ensure_csr(m, 16, np.arange(m + 1) * 2, acol, I.uniform01(count, "rk.a", 2 * m) * 2 - 1)
    rp, ci, va, _, st = run_gpu(A, B, arith=arith)
    assert np.all(np.diff(rp) == count)
    assert (st["num_window_rows"] == m) == (count <= 1024)
    check_against_oracle(A, B, rp, ci, va, exact=count <= 1024 and arith != 2)


# the symbolic phase of unsorted rows: word edges of its windows, the largest one,
# the first size beyond it, and products to either side of its limit
@pytest.mark.parametrize("n", [4096, 4097, 32768, 65535, 65536, 65537])
@pytest.mark.parametrize("flop", [510, 4095, 4096, 4097])
def test_unsorted_symbolic_counts(n, flop):
    lens = np.array([flop // 8] * 7 + [flop - 7 * (flop // 8)], np.int64)
    k = 8 * 24
    lb = np.tile(lens, 24)
    cols = (I.uniform01(n + flop, "rk.uc", int(lb.sum())) * n).astype(np.int64)
    cols[:2] = 0, n - 1
    B = I._from_sorted_coo(k, n, np.repeat(np.arange(k), lb), cols, I.uniform01(flop, "rk.uv", len(cols)) * 2 - 1)
    A = I.ensure_csr(24, k, np.arange(25) * 8, np.arange(k), I.uniform01(n, "rk.ua", k) * 2 - 1)
    rp, ci, va, _, st = run_gpu(A, B, arith=1, small_max_rows=0)
    want = [0] + [len(np.unique(cols[B.rowptr[8 * i]:B.rowptr[8 * i + 8]])) for i in range(24)]
    assert np.array_equal(rp, np.cumsum(want))
    check_against_oracle(A, B, rp, ci, va, exact=False)
