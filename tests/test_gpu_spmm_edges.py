"""SpMM at the edges of its batches of entries (4 gathers, as many entries as a row has lanes), of its
chunks (1,024 entries) and of its panels of columns, with Inf in rows of X that no entry reads: within
(row length + 2) roundings of |A| |X|."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LENGTHS = [0, 1, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 1023, 1024, 1025, 2049, 0, 2]


@pytest.mark.parametrize("w", [1, 2, 5, 8, 16, 31, 64, 100, 129, 260])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_spmm_at_batch_chunk_and_panel_edges(w, dtype):
    import scipy.sparse as sp
    import torch

    import paper_2403_06218_gb300 as tsvd
    rng = np.random.default_rng(w)
    n = 3000
    cols = [np.sort(rng.choice(n - 1, size=k, replace=False)) for k in LENGTHS]  # never the last column
    indptr = np.concatenate([[0], np.cumsum(LENGTHS)])
    A = sp.csr_matrix((rng.standard_normal(indptr[-1]).astype(dtype), np.concatenate(cols), indptr),
                      shape=(len(LENGTHS), n))
    X = rng.standard_normal((n, w)).astype(dtype)
    X[n - 1] = np.inf
    Y = tsvd.spmm(tsvd.CsrMatrix.from_scipy(A), torch.from_numpy(X).cuda()).double().cpu().numpy()
    A64, X64 = A.astype(np.float64)[:, :-1], X[:-1].astype(np.float64)
    u = 2.0 ** -53 if dtype == np.float64 else 2.0 ** -24
    lens = np.diff(indptr)[:, None]
    ref = (A64.astype(np.longdouble).toarray() @ X64.astype(np.longdouble)).astype(np.float64)
    assert np.all(np.abs(Y - ref) <= (lens + 2) * u * (abs(A64) @ np.abs(X64)))
