"""FP64 products of few rows, split over more CTAs than their 256-row slabs or 32-row tiles give:
ragged rows and columns around the slab (16), region (32) and panel (4 to 128 columns) sizes, each
entry against numpy's within twice an s-term (q-term) sum's rounding bound."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = np.finfo(float).eps


@pytest.mark.parametrize("q,s,b", [(1, 1, 1), (15, 33, 16), (16, 16, 17), (255, 64, 16), (257, 31, 1), (512, 64, 16),
                                   (700, 100, 40), (1000, 7, 130), (4000, 48, 20), (33, 200, 200)])
def test_products_of_few_rows(q, s, b):
    import torch

    import paper_2403_06218_gb300 as tsvd
    rng = np.random.default_rng(q + s + b)
    P, Y, M = rng.standard_normal((q, s)), rng.standard_normal((q, b)), rng.standard_normal((s, b))
    t = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    C = tsvd.dense_mm(t(P), t(Y), trans=True).cpu().numpy()
    assert np.all(np.abs(C - P.T @ Y) <= 2 * q * EPS * (np.abs(P).T @ np.abs(Y)))
    D = tsvd.dense_mm(t(P), t(M)).cpu().numpy()
    assert np.all(np.abs(D - P @ M) <= 2 * s * EPS * (np.abs(P) @ np.abs(M)))


@pytest.mark.parametrize("n", [48, 49, 63, 64])
def test_small_svd_at_the_block_path_s_smallest_orders(n):
    import torch

    import paper_2403_06218_gb300 as tsvd
    B = np.tril(np.random.default_rng(n).standard_normal((n, n))) + 3.0 * np.eye(n)
    nv = n // 2
    U, s, V, sweeps = tsvd.small_svd(torch.from_numpy(B).cuda(), nv=nv)
    U, s, V = (x.cpu().numpy() for x in (U, s, V))
    ref = np.linalg.svd(B, compute_uv=False)
    tol = 4 * n ** 1.5 * EPS * ref[0]
    assert 1 <= sweeps < 40
    assert np.abs(s - ref).max() <= tol
    assert np.abs(B @ V[:, :nv] - U[:, :nv] * s[:nv]).max() <= tol
    assert np.abs(B.T @ U[:, :nv] - V[:, :nv] * s[:nv]).max() <= tol
