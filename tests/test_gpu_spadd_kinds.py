"""GPU: sums whose rows take every path of SpAdd side by side (the same columns in both
matrices, a few of them, none, rows of a team, of a warp and of a CTA, out of order,
repeated columns, empty), the numeric phase repeated with other coefficients and with
a product on the same handle in between."""
import numpy as np
import pytest

from oracle import spadd as S
from paper_2103_11991_gb300 import inputs as I
from tests._util import assert_structure_equal, assert_values_within

pytestmark = pytest.mark.gpu


def _matrices(short, kinds, m=240, n=3000):
    """Rows cycling through kinds; rows of up to `short` entries or of the lengths of their kind."""
    g = np.random.default_rng(short)
    rows = {"A": [], "B": []}
    for i in range(m):
        kind = kinds[i % len(kinds)]
        size = {"warp": 100, "cta": 700}.get(kind, int(g.integers(1, short + 1)))
        a = np.sort(g.choice(n, size, replace=False))
        b = np.sort(g.choice(n, size, replace=False))
        if kind == "same":
            b = a.copy()
        elif kind == "some":  # a few of A's columns
            b = a[::4].copy()
        elif kind == "half":
            b = np.unique(np.concatenate([a[::2], b[: size // 2]]))
        elif kind == "empty A":
            a = a[:0]
        elif kind == "empty":
            a, b = a[:0], b[:0]
        elif kind == "order":
            a, b = g.permutation(a), b[::-1].copy()
        elif kind == "repeats":
            a, b = np.concatenate([a, a[:3]]), np.concatenate([b, a[:2], b[:2]])
        rows["A"].append(a)
        rows["B"].append(b)
    out = []
    for k in "AB":
        ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows[k]])])
        out.append(I.ensure_csr(m, n, ptr, np.concatenate(rows[k]), g.random(int(ptr[-1])) * 2 - 1))
    return out


@pytest.mark.parametrize("short", [8, 16, 32])
@pytest.mark.parametrize("kinds", [("same",), ("same", "some"), ("some", "half", "other", "empty A", "empty"),
                                   ("warp",), ("cta",), ("order",),
                                   ("same", "warp", "order", "cta", "empty", "half", "some", "repeats")])
def test_every_kind_of_row(short, kinds):
    import torch
    from paper_2103_11991_gb300 import spgemm as K
    A, B = _matrices(short, kinds)
    dA, dB = K.DeviceCSR.from_host(A), K.DeviceCSR.from_host(B)
    square = K.DeviceCSR.from_host(I.stencil_2d(20, 20, 5))
    with K.SpGEMM() as op:
        rp, nnz = op.spadd_symbolic(dA, dB)
        for alpha, beta in ((1.0, 1.0), (0.3, -0.7), (0.0, 1.0)):
            ci = torch.full((nnz,), -1, dtype=torch.int32, device="cuda")
            va = torch.full((nnz,), float("nan"), dtype=torch.float64, device="cuda")
            op.spadd_numeric(alpha, dA, beta, dB, rp, nnz, ci, va)
            op.sync()
            ref = S.spadd(A, B, alpha, beta)
            assert_structure_equal(rp.cpu().numpy(), ci.cpu().numpy(), ref.rowptr, ref.colind)
            got = va.cpu().numpy()
            if "repeats" in kinds:
                assert_values_within(got, ref.vals, S.spadd_abs(A, B, alpha, beta) + 1e-300)
            else:
                assert np.array_equal(got, ref.vals)
            op(square, square)  # the handle's product state is its own
