"""Edges of the sliced tensor-core product's tiles and exact accumulations.

Column tiles of 16, 32 and 64, row tiles of 128, K blocks of 16, exact accumulation over
128 k (p + q >= 4) and 256 k (p + q <= 3, the first one over 192 k), carries every 16,384 k
and FP64 flushes every 98,304 k.  Integer data must give numpy's bits; digits at their
extreme (-128 everywhere) drive every group sum to its bound.
"""

import fractions

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("trans", [False, True])
@pytest.mark.parametrize("K", [1, 16, 17, 128, 191, 192, 193, 256, 448, 449, 16_400])
def test_integer_products_at_the_edges(tsvd, K, trans):
    import torch
    for M, N in ((127, 1), (128, 16), (129, 17), (1, 32), (257, 33), (300, 64), (64, 65), (640, 129)):
        rng = np.random.default_rng(K * 1000 + M + N)
        A = rng.integers(-500, 501, size=(M, K)).astype(np.float64)
        X = rng.integers(-500, 501, size=(K, N)).astype(np.float64)
        # (torch's own row-major strides, also where a dimension is 1)
        At = torch.empty((K, M) if trans else (M, K), dtype=torch.float64, device="cuda")
        At.copy_(torch.from_numpy(A.T.copy() if trans else A))
        Xt = torch.empty(K, N, dtype=torch.float64, device="cuda")
        Xt.copy_(torch.from_numpy(X))
        Y = tsvd.dense_mm(At, Xt, trans=trans, tensor_cores=True).cpu().numpy()
        assert np.array_equal(Y, A @ X), (M, N, K, trans)


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("M", [130, 152 * 128])
def test_extreme_digits(tsvd, sign, M):
    # a = -(127 2^48 + 128 (256^6 - 1) / 255) 2^-55: digits -127, -128, .. (the last one
    # rounded to 53 bits), so the group sums come close to (p + q + 1) 2^14 K
    import torch
    a = -float(fractions.Fraction(127 * 2 ** 48 + 128 * (256 ** 6 - 1) // 255, 2 ** 55))
    a_exact = fractions.Fraction(a)
    for K in (128, 256, 448, 1_000):
        A = torch.full((M, K), a, dtype=torch.float64, device="cuda")
        X = torch.full((K, 40), sign * a, dtype=torch.float64, device="cuda")
        Y = tsvd.dense_mm(A, X, tensor_cores=True).cpu().numpy()
        assert np.all(Y == Y[0, 0])
        err = abs(fractions.Fraction(float(Y[0, 0])) - int(sign) * K * a_exact * a_exact)
        # the header's bound with 2^ea = 2^eb = 1: one FP64 partial sum with 152 whole tiles,
        # with two tiles one per CTA share of K, which is at least one K block of 16
        P = 1 if M == 152 * 128 else -(-K // 16)
        bound = (2 * K * -a_exact + fractions.Fraction(62 * K, 10)) / 2 ** 56 + P * K * a_exact * a_exact / 2 ** 52
        assert err <= bound, (K, float(err), float(bound))


def test_flush_inside_one_share(tsvd):
    # 152 column tiles: every CTA runs the whole K = 100,000 of its tile (more than one
    # 64-bit accumulation), with integer sums that FP64 holds exactly
    import torch
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randint(-50, 51, (8, 100_000), generator=g, device="cuda").double()
    X = torch.randint(-50, 51, (100_000, 9_728), generator=g, device="cuda", dtype=torch.int8).double()
    Y = tsvd.dense_mm(A, X, tensor_cores=True)
    assert bool((Y == A @ X).all())
