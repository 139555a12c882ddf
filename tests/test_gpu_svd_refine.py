"""The small SVD above the one-CTA size at the edges of its parts: orders around a multiple of
the 32 columns of a pair of blocks and of the clusters' row shares, spectra that its rotations of
all pairs at once can finish, spectra with equal values (left to the sweeps) and a wide range.

The sweeps' test bounds the cosine of every column pair by n eps, so a triplet's residual is a
small multiple of n eps sigma_1 (an n-term sum of such columns: sqrt(n) n eps, and 4 for the
constants); singular values of an orthogonalised B are then off by at most that."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _matrix(n, kind, rng):
    def q():
        return np.linalg.qr(rng.standard_normal((n, n)))[0]
    if kind == "gauss":
        return rng.standard_normal((n, n))
    if kind == "equal":      # every value four times
        return (q() * np.repeat(np.linspace(1.0, 0.1, (n + 3) // 4), 4)[:n]) @ q().T
    if kind == "pairs":      # values in close pairs, apart from one another
        return (q() * (np.repeat(np.linspace(1.0, 0.1, (n + 1) // 2), 2)[:n] * (1 + 1e-9 * np.arange(n)))) @ q().T
    return (q() * np.logspace(0, -6, n)) @ q().T


@pytest.mark.parametrize("n,kind", [(65, "gauss"), (95, "equal"), (96, "wide"), (97, "pairs"), (129, "gauss"),
                                    (256, "pairs"), (511, "equal"), (513, "wide"), (600, "gauss"), (1023, "pairs")])
def test_block_svd_at_edges_and_close_values(n, kind):
    import torch

    import paper_2403_06218_gb300 as tsvd
    rng = np.random.default_rng(n)
    B = _matrix(n, kind, rng)
    nv = n // 3
    U, s, V, sweeps = tsvd.small_svd(torch.from_numpy(B).cuda(), nv=nv)
    U, s, V = (x.cpu().numpy() for x in (U, s, V))
    ref = np.linalg.svd(B, compute_uv=False)
    tol = 4 * n ** 1.5 * np.finfo(float).eps * ref[0]
    assert 1 <= sweeps < 40
    assert np.abs(s - ref).max() <= tol
    assert np.abs(V[:, :nv].T @ V[:, :nv] - np.eye(nv)).max() <= 1e-12
    assert np.abs(B @ V[:, :nv] - U[:, :nv] * s[:nv]).max() <= tol
    assert np.abs(B.T @ U[:, :nv] - V[:, :nv] * s[:nv]).max() <= tol
