"""The Cholesky kernels' reciprocal square roots (csrc/fp64_rsqrt.cuh) against extended
precision: both exponent parities, mantissas at the ends of [1, 4), the ends of the normal
range, subnormals.  The header's derivations give 0.51 and 2 ulp; CUDA's own rsqrt runs on the
same values for comparison (1 ulp by its documentation)."""

import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_2403_06218_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include "fp64_rsqrt.cuh"
__global__ void k(int n, const double* d, double* a, double* b, double* c) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    a[i] = tsvd::rsqrt_fp64_short(d[i]);
    b[i] = tsvd::rsqrt_fp64(d[i]);
    c[i] = rsqrt(d[i]);
}
extern "C" int run(int n, const double* d, double* a, double* b, double* c) {
    k<<<(n + 255) / 256, 256>>>(n, d, a, b, c);
    return (int)cudaDeviceSynchronize();
}
"""


def _values():
    rng = np.random.default_rng(0)
    m = np.concatenate([rng.uniform(1, 4, 20_000), 1 + np.arange(512) * 2.0 ** -52, 4 - np.arange(1, 513) * 2.0 ** -51,
                        2 - np.arange(1, 513) * 2.0 ** -52, 2 + np.arange(512) * 2.0 ** -51])
    scaled = [m * 2.0 ** s for s in (0, 1, -1, 7, -8, 300, -301, 1021, -1022)]
    ends = np.array([np.finfo(float).max, np.finfo(float).tiny, np.nextafter(np.finfo(float).tiny, 1)])
    sub = np.concatenate([np.arange(1, 2_000), rng.integers(1, 2 ** 52, 2_000)]).astype(np.uint64).view(np.float64)
    normal = np.concatenate(scaled + [ends])
    return normal[np.isfinite(normal) & (normal >= np.finfo(float).tiny)], sub


def test_reciprocal_square_roots(tmp_path):
    import torch
    src, so = tmp_path / "rsqrt.cu", tmp_path / "rsqrt.so"
    src.write_text(SRC)
    subprocess.run([B._nvcc(), *B.NVCC_FLAGS, "-shared", "-o", str(so), str(src)], check=True)
    lib = C.CDLL(str(so))
    for d, subnormal in zip(_values(), (False, True)):
        x = torch.from_numpy(d).cuda()
        out = [torch.empty_like(x) for _ in range(3)]
        torch.cuda.synchronize()
        assert lib.run(len(d), *(C.c_void_p(t.data_ptr()) for t in (x, *out))) == 0
        ref = 1 / np.sqrt(d.astype(np.longdouble))
        ulp = np.spacing(ref.astype(np.float64)).astype(np.longdouble)
        off = [float((np.abs(t.cpu().numpy() - ref) / ulp).max()) for t in out]
        # (subnormal values take the Newton steps)
        assert off[0] <= (2.0 if subnormal else 0.51) and off[1] <= 2.0, off
        assert off[2] <= 1.0, off
