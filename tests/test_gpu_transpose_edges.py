"""csr_transpose at the edges of its sort: one entry more or less than a tile of 4,096, one,
two and three radix passes (512, 513 and more than 2^18 columns), all entries in one
column, columns in any order within a row and repeated ones (kept in CSR order)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 511, 512, 513, 262_144, 262_145, 1_000_003])
@pytest.mark.parametrize("nnz", [0, 1, 31, 4_095, 4_096, 4_097, 70_001])
def test_transpose_matches_a_stable_sort(tsvd, n, nnz):
    import torch
    rng = np.random.default_rng(n + nnz)
    m = 1_537
    rows = np.sort(rng.integers(0, m, nnz))
    rows[: nnz // 4] = 0  # one long row
    rows.sort()
    cols = rng.integers(0, n, nnz)
    cols[rng.random(nnz) < 0.3] = n - 1  # a heavy column, repeated within rows
    val = rng.standard_normal(nnz)
    rp = np.zeros(m + 1, dtype=np.int32)
    np.cumsum(np.bincount(rows, minlength=m), out=rp[1:])
    A = tsvd.CsrMatrix(torch.from_numpy(rp).cuda(), torch.from_numpy(cols.astype(np.int32)).cuda(),
                       torch.from_numpy(val).cuda(), (m, n))
    T = tsvd.csr_transpose(A)
    order = np.argsort(cols, kind="stable")
    trp = np.zeros(n + 1, dtype=np.int32)
    np.cumsum(np.bincount(cols, minlength=n), out=trp[1:])
    assert np.array_equal(T.row_ptr.cpu().numpy(), trp)
    assert np.array_equal(T.col_idx.cpu().numpy(), rows[order])
    assert np.array_equal(T.val.cpu().numpy(), val[order])
