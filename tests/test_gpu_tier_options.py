"""GPU: options that say which tier takes a row do so, also for rows that the
automatic choice would give to the wide tier's column chunks."""
import numpy as np
import pytest

from paper_2103_11991_gb300 import inputs as I
from tests._gpu import check_against_oracle, run_gpu

pytestmark = pytest.mark.gpu

M = 40


def _rows(k, flop, span=None):
    # M rows of about `flop` products and columns each
    per = 30
    B = I.random_rows(M * per, span or k, flop // per, flop // per, seed=k + flop, purpose="toB")
    B = I.ensure_csr(B.m, k, B.rowptr, B.colind, B.vals)
    A = I.ensure_csr(M, B.m, np.arange(M + 1) * per, np.arange(M * per), I.uniform01(flop, "to.a", M * per) - 0.5)
    return A, B


@pytest.mark.parametrize("opts,flop,sym,num", [
    (dict(), 900, "dense", "dense"),  # the automatic choice
    (dict(force_tier=0), 900, "team", "team"),
    (dict(force_tier=0), 3600, "cta", "cta"),
    (dict(sym_team_max_flop=1536), 900, "team", "team"),
    (dict(sym_team_max_flop=1536), 1800, "dense", "dense"),
    (dict(num_team_max_nnz=512), 900, "dense", "dense"),
    (dict(num_team_max_nnz=2048), 900, "dense", "team"),
    (dict(sym_team_max_flop=1536, num_team_max_nnz=2048), 1800, "dense", "cta"),
])
def test_tiers_of_rows_of_a_wide_b(opts, flop, sym, num):
    A, B = _rows(98304, flop)
    rp, ci, va, _, st = run_gpu(A, B, arith=1, small_max_rows=0, **opts)
    tiers = {t: st["sym_%s_rows" % t] for t in ("team", "cta", "dense", "window")}
    if sym == "dense":  # a CTA per row: which of the two bins depends on the products
        assert tiers["cta"] + tiers["dense"] == M, tiers
    else:
        assert tiers[sym] == M, tiers
    assert st["num_%s_rows" % num] == M, st
    check_against_oracle(A, B, rp, ci, va)


@pytest.mark.parametrize("flop", [3000, 6000])
def test_forced_window_takes_every_row_of_a_narrow_b(flop):
    A, B = _rows(60000, flop)
    rp, ci, va, _, st = run_gpu(A, B, arith=1, force_tier=3)
    assert st["sym_window_rows"] == M
    check_against_oracle(A, B, rp, ci, va)


# beyond five pieces of 2,048 words a row's chunks pay from more products on
@pytest.mark.parametrize("k,flop,wide", [(327680, 690, True), (327681, 690, False), (400000, 1300, False),
                                         (400000, 1800, True), (520000, 2010, False), (520000, 2100, True)])
def test_line_by_columns_of_b(k, flop, wide):
    A, B = _rows(k, flop)
    rp, ci, va, _, st = run_gpu(A, B, arith=1, small_max_rows=0)
    assert st["sym_cta_rows"] + st["sym_dense_rows"] == (M if wide else 0)
    check_against_oracle(A, B, rp, ci, va)
