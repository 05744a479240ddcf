"""GPU: gradient of the row-capacity network over the sample counts at which its
tiles, its clusters and its grid end, and with labels that name no class, against
the float64 formulas (float32 sums: the tolerances of the other network tests)."""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu


def _case(n, seed):
    rng = np.random.default_rng(seed)
    X = (rng.random((n, 8)) * 6).astype(np.float32)
    y = rng.integers(0, 16, size=n).astype(np.int32)
    th = np.concatenate([(rng.normal(size=s) * (0.3 if len(s) == 2 else 0.1)).reshape(-1) for s in M.SHAPES])
    return X, y, th.astype(np.float32)


def _run(X, y, th):
    import torch
    from paper_2103_11991_gb300 import spgemm as K
    g = torch.empty(M.NUM_PARAMS, dtype=torch.float32, device="cuda")
    l = torch.empty(1, dtype=torch.float32, device="cuda")
    K.kk_mlp_loss_grad(*(torch.from_numpy(a).cuda() for a in (X, y, th)), g, l)
    torch.cuda.synchronize()
    return g.cpu().numpy(), float(l.item())


def _check(X, y, th):
    g, l = _run(X, y, th)
    X, th = X.astype(np.float64), th.astype(np.float64)
    known = (y >= 0) & (y < 16)
    # a label that names no class: softmax alone in the gradient, lse in the loss
    z = M.forward(th, X)[-1]
    lse = np.log(np.exp(z - z.max(1, keepdims=True)).sum(1)) + z.max(1)
    ref_l = (lse - np.where(known, z[np.arange(len(y)), np.where(known, y, 0)], 0.0)).mean()
    n = len(y)
    ref_g = M.grad(th, X, np.where(known, y, 0))
    if not known.all():  # take the unit target of those samples out again
        out = ~known
        W1, b1, W2, b2, W3, b3 = M.unpack(th)
        a1, h1, a2, h2, _ = M.forward(th, X[out])
        dz = np.zeros((out.sum(), 16))
        dz[:, 0] = 1.0 / n
        d2 = (dz @ W3.T) * (a2 > 0)
        d1 = (d2 @ W2.T) * (a1 > 0)
        ref_g = ref_g + np.concatenate([v.reshape(-1) for v in (X[out].T @ d1, d1.sum(0), h1.T @ d2, d2.sum(0),
                                                                h2.T @ dz, dz.sum(0))])
    assert abs(l - ref_l) <= 1e-4 * max(1.0, abs(ref_l))
    np.testing.assert_allclose(g, ref_g, rtol=1e-3, atol=1e-5)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 256, 257, 19455, 19456, 19457, 40001])
def test_sample_counts(n):
    _check(*_case(n, n))


@pytest.mark.parametrize("label", [-1, 16, 35, -(2 ** 31), 2 ** 31 - 1])
@pytest.mark.parametrize("n", [1, 40, 1000])
def test_labels_that_name_no_class(label, n):
    X, y, th = _case(n, n + 7)
    y[::3] = label
    _check(X, y, th)
