"""The FP32 projections add no more rows in FP32 than the plan of 32 x 32 regions does, also
where regions of 128 columns are not full.

An FP32 sum of n random products is off by a rounding error of rms 0.425 2^-24 of the partial
sum at each step (uniform in half an ulp, the mantissa distributed as its logarithm), so by
0.425 2^-24 sqrt(n / 2) of its size; the slabs are added in FP64.  The measured rms over the
outputs scatters by 1 / sqrt(2 s b), 1.5% for the smallest shape here."""

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q,s,b", [(500_003, 96, 64), (500_003, 65, 33), (300_001, 192, 64), (500_003, 128, 64),
                                   (500_003, 128, 128), (9_999, 96, 64)])
def test_error_of_the_longest_fp32_sum(tsvd, q, s, b):
    import torch
    slabs = min(152 * 16 // (-(-s // 32) * -(-b // 32)), -(-q // 256))
    run = -(-q // slabs)
    g = torch.Generator(device="cuda").manual_seed(s + b)
    P, Y = (torch.randn(q, x, generator=g, device="cuda") for x in (s, b))
    ref = P.double().t() @ Y.double()
    err = float((tsvd.dense_mm(P, Y, trans=True).double() - ref).norm() / ref.norm())
    # with the rounding of the output
    assert err <= 1.06 * 0.425 * 2.0 ** -24 * (run / 2 + 1) ** 0.5, (err, run)
