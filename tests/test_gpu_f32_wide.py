"""FP32 products P^T Y in regions of 128 x 128 and 128 x 64: ragged rows, columns at the regions'
edges, and rows that are not 16-byte aligned.  A slab's two halves are FP32 sums of at most q / 2
terms each and the rest is FP64: an entry is within q 2^-24 |P|^T |Y| of the exact product."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q,s,b,off", [(1024, 128, 64, 0), (1025, 128, 128, 0), (4099, 512, 128, 0), (2000, 127, 63, 0),
                                       (5001, 260, 130, 0), (3000, 256, 200, 0), (1500, 128, 64, 1), (40_001, 512, 64, 3),
                                       (1031, 96, 96, 0)])
def test_wide_projection(q, s, b, off):
    import torch

    import paper_2403_06218_gb300 as tsvd
    rng = np.random.default_rng(q + s + b)
    P = rng.standard_normal((q, s + off)).astype(np.float32)
    Y = rng.standard_normal((q, b + off)).astype(np.float32)
    Pt, Yt = torch.from_numpy(P).cuda()[:, off:], torch.from_numpy(Y).cuda()[:, off:]  # off: misaligned views
    C = tsvd.dense_mm(Pt, Yt, trans=True).double().cpu().numpy()
    P, Y = P[:, off:].astype(np.float64), Y[:, off:].astype(np.float64)
    assert np.all(np.abs(C - P.T @ Y) <= q * 2.0 ** -24 * (np.abs(P).T @ np.abs(Y)))
