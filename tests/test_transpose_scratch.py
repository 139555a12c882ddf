"""A solve's workspace does not add the scratch of its CSR(A^T) build to the buffers that take
its place afterwards."""

import ctypes as C

import pytest

from paper_2403_06218_gb300 import _capi


def _solve(lib, m, n, nnz, method, k, a, c):
    d, o, nb = _capi.TsvdMatrix(), _capi.TsvdOpts(), C.c_size_t()
    d.m, d.n, d.format, d.dtype, d.location = m, n, _capi.TSVD_CSR, _capi.TSVD_F64, _capi.TSVD_DEVICE
    d.val, d.ld, d.row_ptr, d.col_idx, d.nnz = 1, n, 1, 1, nnz
    lib.tsvd_default_opts(C.byref(o))
    assert lib.tsvd_workspace_size(C.byref(d), method, k, a, c, C.byref(o), C.byref(nb)) == _capi.TSVD_OK
    return nb.value


@pytest.mark.parametrize("method,a,c", [(_capi.TSVD_METHOD_BLANCZOS, 16, 4), (_capi.TSVD_METHOD_RSVD, 16, 2)])
def test_scratch_is_shared_with_later_buffers(tsvd, method, a, c):
    lib = tsvd.load()
    m, n, k = 1_000_000, 800_000, 16
    few, many = 10_000_000, 300_000_000
    scratch = C.c_size_t()
    assert lib.tsvd_csr_transpose_workspace(m, n, many, C.byref(scratch)) == _capi.TSVD_OK
    # CSR(A^T) and the long rows' partial sums and descriptors (a kSpmmChunk's share each, both
    # ways) grow with the entries; the bases do not
    size = {z: _solve(lib, m, n, z, method, k, a, c) for z in (few, many)}
    assert size[many] >= 12 * many + scratch.value  # room for the build itself
    parts = lambda z: 12 * z + 4 * n  # noqa: E731  CSR(A^T)
    later = size[few] - parts(few)  # (upper bound of) what comes after it
    plans = 2 * 2 * (many // 512 + 1) * (16 + 8 * 32)
    assert size[many] <= parts(many) + max(later + plans, scratch.value) + (1 << 20), (size, scratch.value)
