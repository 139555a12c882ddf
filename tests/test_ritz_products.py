"""The restart and Ritz products of the FP64 Lanczos method slice the basis afresh.

The kept rows-layout planes of a growing basis hold a row's exponent one above its largest
entry, so that later columns rarely raise it.  Emulated in integers, a product of 7 digits
with such exponents is about twice as far off as with fresh ones; the products whose results
leave the cycle (restart vectors, returned vectors) therefore do not read them."""

import re
from fractions import Fraction
from pathlib import Path

import numpy as np

from test_ozaki_math import DIGITS, digits, fixed_point, row_exponent

CSRC = Path(__file__).resolve().parents[1] / "paper_2403_06218_gb300" / "csrc"


def _error(A, B, above):
    """rms error of the digit products p + q <= 6 with row exponents `above` the smallest."""
    err = []
    for a in A:
        e = row_exponent(a) + above
        da = [digits(fixed_point(float(x), e)) for x in a]
        for b in B.T:
            f = row_exponent(b)
            db = [digits(fixed_point(float(x), f)) for x in b]
            s = sum(x[p] * y[q] << (8 * (DIGITS - 1 - p - q)) for x, y in zip(da, db)
                    for p in range(DIGITS) for q in range(DIGITS - p))
            exact = sum(Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b))
            err.append(float(Fraction(s) * Fraction(2) ** (e + f - 14 - 8 * (DIGITS - 1)) - exact))
    return float(np.sqrt(np.mean(np.square(err))))


def test_exponents_one_above_double_the_error():
    rng = np.random.default_rng(0)
    A, B = rng.standard_normal((24, 192)) / 50, np.linalg.qr(rng.standard_normal((192, 192)))[0][:, :12]
    assert 1.6 < _error(A, B, 1) / _error(A, B, 0) < 2.4


def test_vectors_that_leave_the_cycle_come_from_fresh_slices():
    src = (CSRC / "drivers.cu").read_text()
    for out in (r"\bdU\b", r"\bdV\b", r"\bPk\b", r"\bPbk\b", r"\bQnext\b"):
        calls = [m for m in re.finditer(r"gemm_nn<T, double, (?:double|T)>\(([^;]*?)\)\)\);", src)
                 if re.search(rf"0\.0, {out}", m.group(1)) and "1.0, B" in m.group(1) or
                 re.search(rf"1\.0, P(?:bar)?, rb, [UV]b, \w+, 0\.0, {out}", m.group(1))]
        assert calls, out
        for m in calls:
            block = src[src.rindex("{", 0, m.start()):m.start()]
            assert "OzFreshRows" in block, (out, m.group(0))
    assert "!h->oz_fresh_rows" in (CSRC / "k_dense.cu").read_text()
