"""Scratch of the standalone orthogonalisation: the size that the products need on the FP64
pipe is always accepted, FP32 blocks need no more, and the tensor-core scratch on top stays
within its limit."""

import ctypes as C

import numpy as np
import pytest

from paper_2403_06218_gb300 import _capi

EPS = np.finfo(float).eps


def _query(lib, name, *args):
    nb = C.c_size_t()
    assert getattr(lib, name)(*args, C.byref(nb)) == _capi.TSVD_OK
    return nb.value


@pytest.mark.parametrize("q,s,b", [(64, 0, 64), (5_000, 100, 33), (100_000, 512, 64), (220_000, 512, 64),
                                   (2_000_000, 1024, 128)])
def test_least_size_holds_no_copy_of_the_basis(tsvd, q, s, b):
    lib = tsvd.load()
    least, full = _query(lib, "tsvd_orth_workspace_min", q, s, b), _query(lib, "tsvd_orth_workspace", q, s, b)
    # a saved copy of the block, two columns and one wave of partial sums (152 x 7 tiles of
    # 32 x 32 in FP64, 152 x 16 in FP32), never the basis
    assert least <= 8 * q * (b + 2) + 8 * 152 * 16 * 1024 + (64 << 10) + 8 * (8 * b * b + 4 * (s + b) * b)
    assert least <= full <= least + (4 << 30)
    r = s + b
    qr = _query(lib, "tsvd_cgs_qr_workspace", q, r, b) - _query(lib, "tsvd_cgs_qr_workspace_min", q, r, b)
    # no kept planes: one layout of 8 two-byte digits at a time, and the block's
    assert qr <= 16 * (q + 16) * (r + b + 32) + 64 * 2 ** 20


def _call(tsvd, q, s, b, nbytes, f32=False):
    import torch
    g = torch.Generator(device="cuda").manual_seed(q + s + b)
    dt = torch.float32 if f32 else torch.float64
    P = torch.linalg.qr(torch.randn(q, max(s, 1), generator=g, dtype=torch.float64, device="cuda"))[0][:, :s].to(dt).contiguous()
    Y = torch.randn(q, b, generator=g, dtype=torch.float64, device="cuda").to(dt)
    Q, H, R = Y.clone(), torch.zeros(max(s, 1), b, device="cuda").double(), torch.zeros(b, b, device="cuda").double()
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    fn = tsvd.load().tsvd_cgs_cqr2_f32 if f32 else tsvd.load().tsvd_cgs_cqr2
    rep, bd = C.c_int(0), C.c_int(0)
    rc = fn(tsvd.handle(Y.device), q, s, b, P.data_ptr(), max(s, 1), Q.data_ptr(), b, H.data_ptr(), R.data_ptr(),
            C.c_uint64(0), C.byref(rep), C.byref(bd), ws.data_ptr(), nbytes, torch.cuda.current_stream().cuda_stream)
    res = (P.double() @ H[:s] + Q.double() @ R - Y.double()).norm() / Y.double().norm()
    orth = (torch.cat([P, Q], 1).double().t() @ Q.double() - torch.eye(s + b, device="cuda").double()[:, s:]).abs().max()
    return rc, float(res), float(orth)


@pytest.mark.gpu
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("q,s,b", [(20_000, 300, 64), (5_001, 100, 33), (30_000, 0, 128)])
def test_least_size_is_accepted(tsvd, q, s, b, f32):
    lib = tsvd.load()
    least, full = _query(lib, "tsvd_orth_workspace_min", q, s, b), _query(lib, "tsvd_orth_workspace", q, s, b)
    assert full > least  # the tensor cores take these sizes
    # orthogonal to the block's precision; the residual to that of the updates
    eps, orth = (2.0 ** -24, 1e-4) if f32 else (EPS, 100 * EPS)
    for nbytes in (least, (least + full) // 2, full):
        rc, res, off = _call(tsvd, q, s, b, nbytes, f32)
        assert rc == _capi.TSVD_OK and res <= 8 * (s + b) * eps and off <= orth, (nbytes, rc, res, off)
    assert _call(tsvd, q, s, b, least - 256, f32)[0] == _capi.TSVD_ERR_WORKSPACE


@pytest.mark.gpu
@pytest.mark.parametrize("r,b", [(300, 64), (160, 128), (129, 128), (130, 33), (64, 100)])
def test_cgs_qr_with_and_without_its_scratch(tsvd, r, b):
    import torch
    q, lib = 20_000, tsvd.load()
    Y = torch.randn(q, r, generator=torch.Generator(device="cuda").manual_seed(r), dtype=torch.float64, device="cuda")
    full = _query(lib, "tsvd_cgs_qr_workspace", q, r, b)
    least = _query(lib, "tsvd_cgs_qr_workspace_min", q, r, b)
    for nbytes in (least, full):
        Q, R = Y.clone(), torch.empty(r, r, dtype=torch.float64, device="cuda")
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        rep, bd = C.c_int(0), C.c_int(0)
        rc = lib.tsvd_cgs_qr(tsvd.handle(Y.device), q, r, b, Q.data_ptr(), r, R.data_ptr(), C.c_uint64(0), C.byref(rep),
                             C.byref(bd), ws.data_ptr(), nbytes, torch.cuda.current_stream().cuda_stream)
        assert rc == _capi.TSVD_OK and bd.value == 0
        assert float((Q @ R - Y).norm() / Y.norm()) <= 8 * r * EPS
        assert float((Q.t() @ Q - torch.eye(r, device="cuda").double()).abs().max()) <= 100 * EPS


def test_blocks_sized_for_the_last_one_hold_the_earlier_ones(tsvd):
    # more rows, columns or width never take less, and the size for a basis of r columns covers
    # every block of its orthogonalisation
    lib = tsvd.load()
    least = lambda *a: _query(lib, "tsvd_cgs_qr_workspace_min", *a)  # noqa: E731
    for q in (5_000, 60_000, 200_000, 2_000_000):
        for b in (16, 32, 33, 64, 100, 128):
            row = [least(q, r, b) for r in range(b, 1_025, 16)]
            assert row == sorted(row), (q, b)
            for s in range(0, 1_024 - b, b):
                assert _query(lib, "tsvd_orth_workspace_min", q, s, b) <= row[-1], (q, s, b)
    for r, b in ((64, 64), (160, 32), (512, 64)):
        row = [least(q, r, b) for q in range(1_000, 400_000, 7_001)]
        assert row == sorted(row), (r, b)


def test_python_call_takes_the_least_size_where_the_full_one_does_not_fit(monkeypatch):
    import torch

    from paper_2403_06218_gb300 import api

    def ws(nbytes, dev):
        if nbytes > 1_000:
            raise torch.cuda.OutOfMemoryError("no room")
        return nbytes
    monkeypatch.setattr(api, "_ws", ws)
    assert api._ws_or(5_000, 900, None) == 900 and api._ws_or(800, 700, None) == 800
    with pytest.raises(torch.cuda.OutOfMemoryError):
        api._ws_or(5_000, 2_000, None)
