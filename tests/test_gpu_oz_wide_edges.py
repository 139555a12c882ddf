"""Edges of the sliced product with 8 digits an entry: tiles, exact accumulations, carries and
flushes (every 16,384 and 98,304 k) on integer data, and digits of -128 in the seven lower
places, whose group sums are known integers.

With 8 digits a row's entries are F = x 2^(63 - e); F = -0x80808080808080 has the digits 0,
-128, .. -128.  With one CTA share a tile, what the product keeps (p + q <= 7) is rounded to
half of 2^-62 an accumulation of 128 k (its last group) and once to FP64."""

import ctypes as C
import fractions

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _mm(tsvd, A, X, trans=False):
    import torch
    lib, h = tsvd.load(), tsvd.handle(A.device)
    (m, n), w, nb = A.shape, X.shape[1], C.c_size_t()
    assert lib.tsvd_dense_mm_f64tc_workspace(int(trans), m, n, w, C.byref(nb)) == 0
    nbytes = nb.value * 8 // 7 // 256 * 256 + (1 << 20)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    Y = torch.empty(n if trans else m, w, dtype=torch.float64, device="cuda")
    assert lib.tsvd_set_product_digits(h, 8) == 0
    try:
        rc = lib.tsvd_dense_mm_f64tc(h, int(trans), m, n, A.data_ptr(), max(n, 1), w, X.data_ptr(), max(w, 1),
                                     Y.data_ptr(), max(w, 1), ws.data_ptr(), nbytes,
                                     torch.cuda.current_stream().cuda_stream)
    finally:
        assert lib.tsvd_set_product_digits(h, 0) == 0
    assert rc == 0
    return Y


@pytest.mark.parametrize("trans", [False, True])
@pytest.mark.parametrize("K", [1, 16, 17, 128, 191, 192, 193, 256, 448, 449, 16_400])
def test_integer_products(tsvd, K, trans):
    import torch
    for M, N in ((127, 1), (128, 16), (129, 17), (1, 32), (257, 33), (300, 64), (64, 65), (640, 129)):
        rng = np.random.default_rng(K * 1000 + M + N)
        A = rng.integers(-2 ** 18, 2 ** 18 + 1, size=(M, K)).astype(np.float64)
        X = rng.integers(-2 ** 18, 2 ** 18 + 1, size=(K, N)).astype(np.float64)
        At = torch.from_numpy(np.ascontiguousarray(A.T if trans else A)).cuda()
        Y = _mm(tsvd, At, torch.from_numpy(X).cuda(), trans).cpu().numpy()
        ref = (A.astype(np.int64) @ X.astype(np.int64)).astype(np.float64)  # below 2^53
        assert np.array_equal(Y, ref), (M, N, K, trans)


def _digits(F):
    """The 8 balanced base-256 digits of F, the leading one first."""
    d = []
    for _ in range(7):
        d.append((F + 128) % 256 - 128)
        F = (F - d[-1]) // 256
    return [F] + d[::-1]


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("K", [130, 258, 450, 1_002, 18_000])
def test_extreme_digits(tsvd, K, sign):
    import torch
    a = -float(0x80808080808080) * 2.0 ** -63
    M = 152 * 128
    A = torch.full((M, K), a, dtype=torch.float64, device="cuda")
    X = torch.full((K, 40), sign * a, dtype=torch.float64, device="cuda")
    # 0.5 sets the exponent of every row and column to 0 and meets a zero
    A[:, 0], A[:, 1], X[0], X[1] = 0.5, 0.0, 0.0, 0.5
    Y = _mm(tsvd, A, X).cpu().numpy()
    assert np.all(Y == Y[0, 0])
    p, q = _digits(-0x80808080808080), _digits(-sign * 0x80808080808080)
    assert p == [0] + [-128] * 7
    kept = (K - 2) * sum(fractions.Fraction(p[i] * q[j], 2 ** 14 * 256 ** (i + j)) for i in range(8) for j in range(8 - i))
    bound = abs(kept) / 2 ** 53 + fractions.Fraction(-(-K // 128), 2 ** 63)
    assert abs(fractions.Fraction(float(Y[0, 0])) - kept) <= bound, (float(Y[0, 0]), float(kept))


def test_flush_inside_one_share(tsvd):
    import torch
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randint(-50, 51, (8, 100_000), generator=g, device="cuda").double()
    X = torch.randint(-50, 51, (100_000, 9_728), generator=g, device="cuda", dtype=torch.int8).double()
    assert bool((_mm(tsvd, A, X) == A @ X).all())


def test_leading_digit_of_128(tsvd):
    # entries just below a power of two: F rounds up to a leading digit of +128, entries just
    # above minus it to -128
    import torch
    x = np.array([np.nextafter(1.0, 0), -np.nextafter(1.0, 0), 0.999, -0.999, 127.6 / 128, -127.6 / 128, 0.5, -1e-3])
    A = torch.from_numpy(np.tile(x, (130, 4))).cuda()
    X = torch.eye(32, dtype=torch.float64, device="cuda")
    assert torch.equal(_mm(tsvd, A, X), A)
    assert torch.equal(_mm(tsvd, X, A[:32].contiguous()), A[:32])
