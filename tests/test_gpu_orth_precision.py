"""Error of the standalone FP64 orthogonalisation on the tensor cores against arithmetic of
about 1e-28, next to the same call on the FP64 pipe (which the least workspace selects).

The reference cuts both operands of a product into slices of 17 bits, whose FP64 products are
exact, and adds those in double-double; the Gram matrix is factored in extended precision."""

import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


def _two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def _slices(torch, a):
    e = torch.ceil(torch.log2(a.abs().amax(0, keepdim=True).clamp_min(1e-300))) + 1
    out = []
    for i in range(6):
        c = 0.75 * torch.exp2(e + 53 - 17 * (i + 1))
        s = (a + c) - c
        out.append(s)
        a = a - s
    return out


def _tn(torch, A, B):
    """A^T B as an unevaluated sum of two matrices."""
    a, b = _slices(torch, A), _slices(torch, B)
    hi = torch.zeros(A.shape[1], B.shape[1], dtype=torch.float64, device="cuda")
    lo = torch.zeros_like(hi)
    for i in range(6):
        for j in range(6 - i):
            hi, e = _two_sum(hi, a[i].t() @ b[j])
            lo += e
    return _two_sum(hi, lo)


def _reference(torch, Y, P):
    """Q, H, R of the two passes of Alg. 5 in exact arithmetic, each as (high, low)."""
    W, H = (Y, torch.zeros_like(Y)), None
    for _ in range(2 if P.shape[1] else 0):
        h = _tn(torch, P, W[0])
        h = _two_sum(h[0], h[1] + P.t() @ W[1])
        u = _tn(torch, P.t().contiguous(), h[0])
        u = _two_sum(u[0], u[1] + P @ h[1])
        d, e = _two_sum(W[0], -u[0])
        W = _two_sum(d, e + (W[1] - u[1]))
        H = h if H is None else _two_sum(*(lambda s: (s[0], s[1] + H[1] + h[1]))(_two_sum(H[0], h[0])))
    g = _tn(torch, W[0], W[0])
    x = W[0].t() @ W[1]
    L = np.longdouble
    G = g[0].cpu().numpy().astype(L) + (g[1] + x + x.t()).cpu().numpy().astype(L)
    b = G.shape[0]
    R, M = np.zeros((b, b), L), np.zeros((b, b), L)
    for i in range(b):
        R[i, i] = np.sqrt(G[i, i] - (R[:i, i] ** 2).sum())
        R[i, i + 1:] = (G[i, i + 1:] - R[:i, i] @ R[:i, i + 1:]) / R[i, i]
    for i in range(b - 1, -1, -1):
        M[i] = ((np.arange(b) == i).astype(L) - R[i, i + 1:] @ M[i + 1:]) / R[i, i]

    def pair(X):
        hi = X.astype(np.float64)
        return torch.from_numpy(hi).cuda(), torch.from_numpy((X - hi).astype(np.float64)).cuda()
    m = pair(M)
    q = _tn(torch, W[0].t().contiguous(), m[0])
    return _two_sum(q[0], q[1] + W[1] @ m[0] + W[0] @ m[1]), H, pair(R)


def _run(tsvd, Y, P, query):
    import torch
    (q, b), s, lib, nb = Y.shape, P.shape[1], tsvd.load(), C.c_size_t()
    assert getattr(lib, query)(q, s, b, C.byref(nb)) == 0
    ws = torch.empty(nb.value, dtype=torch.uint8, device="cuda")
    Q, H, R = Y.clone(), torch.zeros(max(s, 1), b, device="cuda").double(), torch.zeros(b, b, device="cuda").double()
    rep, bd = C.c_int(0), C.c_int(0)
    assert lib.tsvd_cgs_cqr2(tsvd.handle(Y.device), q, s, b, P.data_ptr(), max(s, 1), Q.data_ptr(), b, H.data_ptr(),
                             R.data_ptr(), C.c_uint64(0), C.byref(rep), C.byref(bd), ws.data_ptr(), nb.value,
                             torch.cuda.current_stream().cuda_stream) == 0
    return Q, H[:s], R


def _error(x, ref):
    """Largest relative error of a column."""
    d = (x - ref[0]) - ref[1]
    return float((d.norm(dim=0) / ref[0].norm(dim=0)).max())


@pytest.mark.parametrize("q,s,b", [(87_413, 0, 128), (30_001, 0, 100), (66_746, 33, 33), (60_000, 64, 64),
                                   (40_000, 300, 100)])
def test_no_further_off_than_the_fp64_pipe(tsvd, q, s, b):
    import torch
    g = torch.Generator(device="cuda").manual_seed(q + s + b)
    P = torch.zeros(q, s, dtype=torch.float64, device="cuda")
    P.fill_diagonal_(1.0)
    for _ in range(8 if s else 0):
        u = torch.randn(q, generator=g, dtype=torch.float64, device="cuda")
        u /= u.norm()
        P.addr_(u, u @ P, alpha=-2.0)
    Y = torch.randn(q, b, generator=g, dtype=torch.float64, device="cuda")
    Y *= torch.logspace(0, -3, b, dtype=torch.float64, device="cuda")
    if s:
        Y += P @ torch.randn(s, b, generator=g, dtype=torch.float64, device="cuda")
    ref = _reference(torch, Y, P)
    pipe, tc = (_run(tsvd, Y, P, f"tsvd_orth_workspace{k}") for k in ("_min", ""))
    assert not torch.equal(pipe[0], tc[0])
    # two rounded triangular products of a column, and what the two roundings of R leave in it
    assert _error(tc[0], ref[0]) <= max(4 * U64, _error(pipe[0], ref[0]))
    if s:
        assert _error(tc[1], ref[1]) <= max(2 * U64, _error(pipe[1], ref[1]))
    assert _error(tc[2], ref[2]) <= max(8 * U64, _error(pipe[2], ref[2]))
