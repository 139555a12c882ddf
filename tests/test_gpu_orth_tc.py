"""The standalone FP64 orthogonalisation at sizes whose products run on the tensor cores:
ragged widths, strided operands, a basis with rows of very different entries, dependent
columns.  Y = P H + Q R is checked row by row against quadruple precision."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps


def _basis(rng, q, s):
    """Leading columns of a product of Householder reflectors: entries near 1 and near 1/sqrt(q)."""
    P = np.zeros((q, s))
    P[np.arange(s), np.arange(s)] = 1.0
    for _ in range(6):
        u = rng.standard_normal(q)
        u /= np.linalg.norm(u)
        P -= 2.0 * np.outer(u, u @ P)
    return P


def _window(a, pad):
    """The same matrix as a column window of a wider one (odd leading dimension)."""
    import torch
    w = torch.zeros(a.shape[0], a.shape[1] + pad, dtype=torch.float64, device="cuda")
    v = w[:, 1:1 + a.shape[1]]
    v.copy_(torch.from_numpy(a))
    return v


@pytest.mark.parametrize("q,s,b,pad", [(6_001, 100, 33, 2), (4_000, 0, 128, 3), (20_000, 64, 16, 4), (3_000, 300, 17, 2)])
def test_factorisation_row_by_row(tsvd, q, s, b, pad):
    rng = np.random.default_rng(q + s + b)
    P = _basis(rng, q, s)
    Y = rng.standard_normal((q, b)) * np.logspace(0, -3, b) + P @ rng.standard_normal((s, b))
    Q, H, R, bd = tsvd.cgs_cqr2(_window(Y, pad), _window(P, pad))
    Q, H, R = (t.cpu().numpy() for t in (Q, H, R))
    assert bd == 0
    rows = np.r_[0:s, rng.integers(s, q, 400)]  # the spiky rows and a sample of the others
    W = np.longdouble
    res = np.abs(Y[rows].astype(W) - P[rows].astype(W) @ H.astype(W) - Q[rows].astype(W) @ R.astype(W))
    # two passes of updates of s terms and normalisations of b terms; CholeskyQR's backward
    # error mixes a row's columns, so the row's largest entry scales it
    bound = 2 * (s + b + 4) * EPS * (np.abs(P[rows]) @ np.abs(H) + np.abs(Q[rows]) @ np.abs(R)).max(1, keepdims=True)
    assert np.all(res <= bound), float((res / bound).max())
    G = np.concatenate([P, Q], 1)
    assert np.abs(G.T @ G - np.eye(s + b)).max() < 100 * EPS


def test_dependent_columns_take_the_fallback(tsvd):
    import torch
    rng = np.random.default_rng(0)
    Y = rng.standard_normal((5_000, 64))
    Y[:, 40] = Y[:, 3] - 2 * Y[:, 7]
    Q, R, bd = tsvd.cholqr2(torch.from_numpy(Y).cuda())
    Q, R = Q.cpu().numpy(), R.cpu().numpy()
    assert bd == 1
    assert np.abs(Q.T @ Q - np.eye(64)).max() < 1e-12
    assert np.abs(Q @ R - Y).max() < 1e-11
