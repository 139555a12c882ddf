"""The small SVD's FP32 sweeps on clusters of 8, 4 and 2 CTAs: orders at the edges of the
block pairs and of the row shares, the same bits from call to call, and the exit of whole
clusters when a wait runs out."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = np.finfo(float).eps


@pytest.mark.parametrize("ctas", [8, 4, 2])
@pytest.mark.parametrize("n", [49, 64, 97, 255, 513, 1024])
def test_every_cluster_size(tsvd, n, ctas):
    import torch
    rng = np.random.default_rng(n)
    B = rng.standard_normal((n, n)) * np.logspace(0, -4, n)
    Bd = torch.from_numpy(B).cuda()
    nv = n // 2
    with tsvd.svd_cluster(ctas):
        runs = [tsvd.small_svd(Bd, nv=nv) for _ in range(3)]
    U, s, V = (x.cpu().numpy() for x in runs[0][:3])
    for other in runs[1:]:
        for x, y in zip(runs[0][:3], other[:3]):
            x, y = (x[:, :nv], y[:, :nv]) if x.dim() == 2 else (x, y)
            assert torch.equal(x, y)
    # the sweeps' test bounds the cosine of every column pair by n eps: a triplet is off by a
    # small multiple of n eps sigma_1, over an n-term sum
    ref = np.linalg.svd(B, compute_uv=False)
    tol = 4 * n ** 1.5 * EPS * ref[0]
    assert np.abs(s - ref).max() <= tol
    assert np.abs(B @ V[:, :nv] - U[:, :nv] * s[:nv]).max() <= tol
    assert np.abs(V[:, :nv].T @ V[:, :nv] - np.eye(nv)).max() <= 1e-12


def test_other_cluster_sizes_are_refused(tsvd):
    from paper_2403_06218_gb300 import _capi
    for ctas in (1, 3, 16, -8):
        with pytest.raises(tsvd.TsvdError) as e:
            with tsvd.svd_cluster(ctas):
                pass
        assert e.value.code == _capi.TSVD_ERR_INVALID_ARG


@pytest.mark.parametrize("ctas", [8, 4, 2])
@pytest.mark.parametrize("n", [100, 300])
def test_clusters_leave_when_a_wait_runs_out(tsvd, n, ctas):
    import torch

    from paper_2403_06218_gb300 import _capi
    rng = np.random.default_rng(n)
    B = torch.from_numpy(rng.standard_normal((n, n))).cuda()
    with tsvd.svd_cluster(ctas):
        with tsvd.wait_limit(2):
            with pytest.raises(tsvd.TsvdError) as e:
                tsvd.small_svd(B, nv=n // 2)
        assert e.value.code == _capi.TSVD_ERR_TIMEOUT
        s = tsvd.small_svd(B, nv=n // 2)[1].cpu().numpy()
    ref = np.linalg.svd(B.cpu().numpy(), compute_uv=False)
    assert np.abs(s - ref).max() < 1e-12 * ref[0] * n


@pytest.mark.parametrize("n,decades", [(100, 8), (256, 8), (512, 8), (100, 12), (256, 12), (512, 12)])
def test_spectra_over_many_decades(tsvd, n, decades):
    # (the sweeps finish before their limit of 40; values are held to sigma_1, as everywhere)
    import torch
    rng = np.random.default_rng(n + decades)
    q = [np.linalg.qr(rng.standard_normal((n, n)))[0] for _ in range(2)]
    B = (q[0] * np.logspace(0, -decades, n)) @ q[1].T
    nv = n // 3
    U, s, V, sweeps = tsvd.small_svd(torch.from_numpy(B).cuda(), nv=nv)
    U, s, V = (x.cpu().numpy() for x in (U, s, V))
    tol = 4 * n ** 1.5 * EPS
    assert 1 <= sweeps < 40
    assert np.abs(s - np.linalg.svd(B, compute_uv=False)).max() <= tol
    assert np.abs(B @ V[:, :nv] - U[:, :nv] * s[:nv]).max() <= tol
    assert np.abs(B.T @ U[:, :nv] - V[:, :nv] * s[:nv]).max() <= tol
    assert np.abs(V[:, :nv].T @ V[:, :nv] - np.eye(nv)).max() <= 1e-12
