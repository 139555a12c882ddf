"""The three-way BF16 split at the edges of its 64 x 64 tiles and of the FP32 range.

Each piece is a rounding to 8 significant bits of what the earlier ones left, so three leave at
most 2^-9 of the third, itself at most 2^-16 of the value: 2^-25, and 2^-24 is asserted.  Pieces
below the smallest normal BF16 value (2^-126) are rounded to a multiple of 2^-133, so an
absolute 2^-133 is added."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(1, 1), (63, 65), (64, 64), (65, 129), (2, 777), (777, 3)])
@pytest.mark.parametrize("trans", [False, True])
def test_split_at_tile_edges_and_range_ends(m, n, trans):
    import torch

    import paper_2403_06218_gb300 as tsvd
    rng = np.random.default_rng(m * 1000 + n)
    A = rng.standard_normal((m, n)) * 2.0 ** rng.integers(-140, 125, size=(m, n))
    A[rng.random((m, n)) < 0.1] = 0.0
    A[0, 0] = 1.0 + 2.0 ** -8 + 2.0 ** -52  # a tie of the leading piece but for the last bit
    pcs = tsvd.bf16x3_split(torch.from_numpy(A).cuda(), trans=trans).pieces().double().cpu().numpy()
    ref = A.T if trans else A
    assert pcs.shape == (3,) + ref.shape
    assert np.all(np.abs(pcs.sum(0) - ref) <= 2.0 ** -24 * np.abs(ref) + 2.0 ** -133)
    assert np.all(np.abs(pcs[1]) <= 2.0 ** -8 * np.abs(ref) + 2.0 ** -133)
