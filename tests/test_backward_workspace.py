"""Scratch of the gradient: the size that its projections need on the FP64 pipe is accepted
and gives the same gradient as the tensor-core form."""

import ctypes as C

import numpy as np
import pytest

from paper_2403_06218_gb300 import _capi


def _query(lib, m, n, nnz, k, least):
    d, o, nb = _capi.TsvdMatrix(), _capi.TsvdBackwardOpts(), C.c_size_t()
    d.m, d.n, d.format, d.dtype, d.location = m, n, _capi.TSVD_CSR, _capi.TSVD_F64, _capi.TSVD_DEVICE
    d.val, d.ld, d.row_ptr, d.col_idx, d.nnz = 1, n, 1, 1, nnz
    lib.tsvd_default_backward_opts(C.byref(o))
    fn = lib.tsvd_svd_backward_workspace_min if least else lib.tsvd_svd_backward_workspace
    assert fn(C.byref(d), k, C.byref(o), C.byref(nb)) == _capi.TSVD_OK
    return nb.value


@pytest.mark.parametrize("m,n,k", [(100_001, 80_003, 32), (2_000_000, 500_000, 40), (300, 200, 4)])
def test_least_size_holds_no_digit_planes(tsvd, m, n, k):
    lib, nnz = tsvd.load(), 10 * m
    least, full = _query(lib, m, n, nnz, k, True), _query(lib, m, n, nnz, k, False)
    assert least <= full <= least + (4 << 30)
    assert (full > least) == (m > 300)
    # 5 blocks of max(m, n) x k, the two factors of 2 k columns, Y and Z, CSR(A^T) and what
    # its transposition needs, one wave of partial sums
    assert least <= 8 * k * (5 * max(m, n) + 3 * (m + n)) + 56 * nnz + 8 * (m + n) + (64 << 20)


@pytest.mark.gpu
def test_gradient_with_the_least_size(tsvd, monkeypatch):
    import scipy.sparse as sp
    import torch

    import workloads
    from paper_2403_06218_gb300 import api
    m, n, k = 24_000, 20_001, 32
    A = workloads.csr_uniform(m, n, 10, seed=3)
    A = (sp.diags(1 + 9 * (1.0 + np.arange(m)) ** -0.25) @ A).tocsr()
    Ad = tsvd.CsrMatrix.from_scipy(A)
    r = tsvd.blanczos(Ad, k, 32, 10, seed=1, tol=1e-9, max_restarts=60, restart_keep=64)
    Ub = torch.randn(m, k, generator=torch.Generator(device="cuda").manual_seed(1), dtype=torch.float64, device="cuda")
    one = torch.ones(k, dtype=torch.float64, device="cuda")
    sizes, grads = [], []

    def pick(which):
        def ws(full, least, dev):
            sizes.append((full, least)[which])
            return api._ws(sizes[-1], dev)
        return ws
    for which in (0, 1):
        monkeypatch.setattr(api, "_ws_or", pick(which))
        grads.append(tsvd.svd_backward(Ad, r.sigma, r.U, r.V, one, Ub, cg_tol=1e-12)[0])
    assert sizes[0] > sizes[1]
    # both solved to the same relative residual: the bar of the gradient's parity test
    assert float((grads[0] - grads[1]).abs().max() / grads[0].abs().max()) < 1e-8
    monkeypatch.setattr(api, "_ws_or", lambda full, least, dev: api._ws(least - 1024, dev))
    with pytest.raises(tsvd.TsvdError) as e:
        tsvd.svd_backward(Ad, r.sigma, r.U, r.V, one, Ub)
    assert e.value.code == _capi.TSVD_ERR_WORKSPACE
