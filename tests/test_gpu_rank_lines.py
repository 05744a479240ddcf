"""GPU: rows of few columns in a wide window stay in the team tier, rows of more go to
the rank tier; the tiers either side of each line, against the oracle."""
import numpy as np
import pytest

from paper_2103_11991_gb300 import inputs as I
from tests._gpu import check_against_oracle, run_gpu

pytestmark = pytest.mark.gpu

M = 60


def _rows(columns, span, unsorted):
    """M rows of C of that many columns, spread over a window of that span, each column of two products."""
    B = I.random_rows(M * columns, span - 1, 1, 1, seed=columns + span, purpose="rlB")
    cols = B.colind.reshape(M, columns).astype(np.int64)
    for r in range(M):  # distinct columns, the first and the last of the window among them
        have = np.unique(np.concatenate([[0, span - 1], cols[r]]))
        extra = np.setdiff1d(np.arange(1, span - 1), have)[: max(0, columns - len(have))]
        inner = np.setdiff1d(np.concatenate([have, extra]), [0, span - 1])[: columns - 2]
        cols[r] = np.sort(np.concatenate([[0, span - 1], inner]))
    twice = np.repeat(cols, 2, axis=0).reshape(-1)
    if unsorted:
        twice = np.repeat(cols[:, ::-1], 2, axis=0).reshape(-1)
    B = I.ensure_csr(2 * M, 65536, np.arange(2 * M + 1) * columns, twice, I.uniform01(span, "rl.b", 2 * M * columns) - 0.5)
    A = I.ensure_csr(M, 2 * M, np.arange(M + 1) * 2, np.arange(2 * M), I.uniform01(columns, "rl.a", 2 * M) - 0.5)
    return A, B


@pytest.mark.parametrize("columns,span,rank", [(32, 4097, False), (33, 4097, True), (64, 16384, True), (64, 16385, False),
                                               (65, 16385, True), (65, 32768, True), (32, 9000, False), (40, 16384, True)])
def test_numeric_line(columns, span, rank):
    A, B = _rows(columns, span, False)
    rp, ci, va, _, st = run_gpu(A, B, arith=1, small_max_rows=0, structure_cache=0)
    assert np.all(np.diff(rp) == columns)
    assert st["num_window_rows"] == (M if rank else 0)
    check_against_oracle(A, B, rp, ci, va)


@pytest.mark.parametrize("columns,rank", [(28, False), (29, False), (32, False), (33, True), (200, True)])
def test_symbolic_line_of_an_unsorted_b(columns, rank):
    # B has 65,536 columns: rows of more than 64 products (2 to a column) and a window of 512 to a product
    A, B = _rows(columns, 60000, True)
    rp, ci, va, _, st = run_gpu(A, B, arith=1, small_max_rows=0)
    assert st["sym_window_rows"] == (M if rank and 2 * columns * 512 >= 65536 else 0)
    check_against_oracle(A, B, rp, ci, va)


def test_nine_point_rows_of_a_wide_grid():
    A = I.stencil_2d(1080, 60, 9, 8.0, -1.0)
    A.vals = I.uniform01(1, "rl.g", A.nnz) - 0.5
    rp, ci, va, _, st = run_gpu(A, A)
    assert st["num_window_rows"] == st["kept_structure_rows"]
    check_against_oracle(A, A, rp, ci, va)
