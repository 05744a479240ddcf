"""GPU: matrices of small dense blocks, whose rows have many products in few words
of columns, keep their window rows' structure with a narrow B too; rows whose
products are spread out leave the window for the wide tier."""
import numpy as np
import pytest

from paper_2103_11991_gb300 import inputs as I
from tests._gpu import check_against_oracle, run_gpu

pytestmark = pytest.mark.gpu


def _blocks(count, b, cols=None):
    n = count * b
    col = (np.arange(n) // b * b)[:, None] + np.arange(b)[None, :]
    return I.ensure_csr(n, cols or n, np.arange(n + 1) * b, col.reshape(-1), I.uniform01(b, "db.v", n * b) - 0.5)


def _block_stencil(nx, ny, d):
    """9-point grid with dense d x d blocks: runs of 3 d columns, nx d apart."""
    S = I.stencil_2d(nx, ny, 9, 8.0, -1.0)
    rows = np.repeat(np.arange(S.m), np.diff(S.rowptr))
    r = (rows[:, None, None] * d + np.arange(d)[None, :, None]).repeat(d, 2)
    c = (S.colind[:, None, None] * d + np.arange(d)[None, None, :]).repeat(d, 1)
    order = np.lexsort((c.reshape(-1), r.reshape(-1)))
    return I._from_sorted_coo(S.m * d, S.n * d, r.reshape(-1)[order], c.reshape(-1)[order],
                              I.uniform01(d, "db.s", r.size) - 0.5)


# blocks below and above 64 x 64 (4,096 products), k at the widest window
@pytest.mark.parametrize("make", [lambda: _blocks(12, 64), lambda: _blocks(12, 65), lambda: _blocks(9, 81),
                                  lambda: _blocks(4, 256), lambda: _blocks(9, 81, 65536),
                                  lambda: _block_stencil(14, 9, 8), lambda: _block_stencil(40, 9, 8)])
def test_block_rows_keep_their_structure(make):
    A = make()
    B = A if A.m == A.n else I.ensure_csr(A.n, A.n, np.minimum(np.arange(A.n + 1), A.m) * 81, A.colind, A.vals)
    rp, ci, va, _, st = run_gpu(A, B, arith=1, small_max_rows=0)
    assert st["sym_window_rows"] == A.m and st["kept_structure_rows"] == A.m
    check_against_oracle(A, B, rp, ci, va, exact=True)


@pytest.mark.parametrize("k", [4000, 65536, 65537])
@pytest.mark.parametrize("pairs", [4032, 4096, 4160])
def test_line_by_pairs(k, pairs):
    # one or more entries of B to a word: as many pairs, more products; A's rows of
    # 64 entries, and rows without entries for a smaller mean row length (other teams)
    per, la = pairs // 64, 64
    for dense in (1, 5, 6, 8):
        words = np.sort(np.argsort(I.uniform01(k, "db.w", 30 * 64 * 120).reshape(30 * 64, 120), 1)[:, :per], 1)
        cols = (words * (k // 120 // 32 * 32))[:, :, None] + np.arange(dense)[None, None]
        B = I.ensure_csr(30 * 64, k, np.arange(30 * 64 + 1) * cols[0].size, cols.reshape(-1),
                         I.uniform01(pairs, "db.b", cols.size) - 0.5)
        for empty in (0, 300):
            lens = np.concatenate([np.full(30, la), np.zeros(empty, int)])
            A = I.ensure_csr(30 + empty, 30 * 64, np.concatenate([[0], np.cumsum(lens)]), np.arange(30 * 64),
                             I.uniform01(la, "db.a", 30 * 64) - 0.5)
            rp, ci, va, _, st = run_gpu(A, B, arith=1, small_max_rows=0)
            window = k > 65536 or (pairs <= 4096 and (dense == 1 or dense >= 6))
            assert st["sym_window_rows"] == (30 if window else 0), (dense, empty, st)
            check_against_oracle(A, B, rp, ci, va)


# 27-point rows of a flat grid (567 products in 75 columns, a span beyond the widest
# window) and with 2 x 2 blocks (2,268 products in 150 columns)
@pytest.mark.parametrize("use_window", [1, 0])
@pytest.mark.parametrize("blocks", [1, 2])
def test_rows_of_few_columns_stay_in_the_team_tier(blocks, use_window):
    d = blocks
    S = I.stencil_3d(200, 190, 3, 27, 26.0, -1.0) if d == 1 else I.stencil_3d(150, 110, 3, 27, 26.0, -1.0)
    rows = np.repeat(np.arange(S.m, dtype=np.int64), np.diff(S.rowptr))
    pick = np.arange(S.m)[:: 37] if d == 2 else np.arange(S.m)
    r = (rows[:, None, None] * d + np.arange(d)[None, :, None]).repeat(d, 2).reshape(-1)
    c = (S.colind[:, None, None].astype(np.int64) * d + np.arange(d)[None, None, :]).repeat(d, 1).reshape(-1)
    order = np.lexsort((c, r))
    A = I._from_sorted_coo(S.m * d, S.n * d, r[order], c[order], I.uniform01(d, "db.f", r.size) - 0.5)
    A2 = A if d == 1 else I.ensure_csr(len(pick), A.n, np.concatenate([[0], np.cumsum(np.diff(A.rowptr)[pick])]),
                                       np.concatenate([A.colind[A.rowptr[i]:A.rowptr[i + 1]] for i in pick]),
                                       np.concatenate([A.vals[A.rowptr[i]:A.rowptr[i + 1]] for i in pick]))
    rp, ci, va, _, st = run_gpu(A2, A, arith=1, use_window=use_window, small_max_rows=0)
    assert st["sym_team_rows"] == A2.m
    check_against_oracle(A2, A, rp, ci, va)
