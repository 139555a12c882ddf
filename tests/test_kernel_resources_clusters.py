"""Registers and shared memory of the cluster, wide and persistent kernels, from ptxas's report
and the sizes that their launches ask for (computed here from the constants in the source).

* The cluster Cholesky: one CTA (256 threads, its rows and the panels) on each of 8 SMs.
* The FP32 Jacobi sweeps at order 1024: clusters of 8 need two CTAs an SM on 152 SMs
  (32 block pairs), those of 4 and 2 one.
* The wide FP32 projection, the radix sort's scatter and every shape of the sliced product."""

import re

import pytest

from paper_2403_06218_gb300 import build as B
from test_kernel_resources import REGS_PER_SM, SMEM_PER_SM, _one, _resident_ctas, kernels  # noqa: F401

MAX_BLOCK_SMEM = 227 * 1024


def _const(file, name):
    m = re.search(rf"\b{name} = (\d+)\b", (B.CSRC / file).read_text())
    assert m, name
    return int(m.group(1))


def test_cluster_cholesky(kernels):  # noqa: F811
    p, c = _const("k_dense.cu", "kCholPanel"), _const("k_dense.cu", "kCholCluster")
    b = int(re.search(r"#define TSVD_MAX_BLOCK\s+(\d+)", (B.INCLUDE / "tsvd.h").read_text()).group(1))
    rows, ld, ldp = b // c, b + 4, p + 1
    # own rows of A and M, the panel's columns of L and rows of M, its block and own columns of
    # M, three pivot columns, two rows of M, the pivots' reciprocals, threshold and flag
    smem = 8 * (2 * rows * ld + b * ldp + p * ld + 2 * p * ldp + 3 * 32 + 2 * p + p + 2)
    src = (B.CSRC / "k_dense.cu").read_text()
    fields = re.search(r"struct CholSmem \{(.*?)\};", src, re.S).group(1)
    assert re.findall(r"\b(\w+)\[", fields) == ["A", "M", "Lp", "Mp", "D", "Mq", "col", "mrow", "dinv"]
    k = _one(kernels, r"chol_inv_cluster_kernel")
    assert k["regs"] * 256 <= REGS_PER_SM, k
    assert k["smem"] + smem <= MAX_BLOCK_SMEM and k["smem"] + smem < 100 * 1024, (k, smem)


@pytest.mark.parametrize("ctas,per_sm", [(8, 2), (4, 1), (2, 1)])
def test_fp32_jacobi_clusters_fit_at_order_1024(kernels, ctas, per_sm):  # noqa: F811
    ld, threads = _const("k_jacobi.cu", "kJ32Ld"), _const("k_jacobi.cu", "kJ32Threads")
    k = _one(kernels, rf"jacobi32_kernelILi{ctas}E")
    smem = 4 * ld * 2 * (1024 // ctas)
    assert k["smem"] <= 48 * 1024 and k["smem"] + smem <= MAX_BLOCK_SMEM, (k, smem)
    assert _resident_ctas(k["regs"], threads, k["smem"] + smem) >= per_sm, k
    assert 152 * per_sm >= 1024 // 32 * ctas


@pytest.mark.parametrize("nb", [64, 128])
def test_wide_projection_fits_one_cta(kernels, nb):  # noqa: F811
    f = "k_f32.cu"
    smem = 2 * _const(f, "kWideStages") * _const(f, "kWideK") * (_const(f, "kWideS") + nb) * 4
    # the exchange of the two groups' sums takes the same memory
    assert smem >= 256 * 8 * (2 * nb // 64) * 8
    hits = [v for k, v in kernels.items() if re.search(rf"gemm_tn_wide_f32_kernelILi{nb}E", k)]
    assert len(hits) == 4  # aligned or not, FP32 or FP64 output
    for k in hits:
        assert k["regs"] * 512 <= REGS_PER_SM and k["smem"] + smem <= MAX_BLOCK_SMEM, (k, smem)


def test_radix_scatter_keeps_two_ctas_an_sm(kernels):  # noqa: F811
    f = "k_sparse.cu"
    threads, per, bits = (_const(f, n) for n in ("kSortThreads", "kSortPer", "kSortMaxBits"))
    for t, size in (("d", 8), ("f", 4)):
        k = _one(kernels, rf"sort_scatter_kernelI{t}E")
        smem = (size + 8) * threads * per + 4 * threads // 32 * (1 << bits)
        assert _resident_ctas(k["regs"], threads, k["smem"] + smem) >= 2, (k, smem)


@pytest.mark.parametrize("nc,dig", [(n, d) for n in (16, 32, 64) for d in (7, 8)])
def test_sliced_product_shapes(kernels, nc, dig):  # noqa: F811
    stages = {7: {64: 5, 32: 6, 16: 7}, 8: {64: 4, 32: 5, 16: 6}}[dig][nc]
    line = re.search(r"kStages = (.*?);", (B.CSRC / "k_oz.cu").read_text()).group(1)
    assert line == "D == 7 ? (NC == 64 ? 5 : (NC == 32 ? 6 : 7)) : (NC == 64 ? 4 : (NC == 32 ? 5 : 6))"
    smem = stages * dig * 32 * (128 + nc) + 1024
    threads = 64 + 32 * (16 if nc == 64 else 8)
    k = _one(kernels, rf"oz_gemm_kernelILi{nc}ELi{dig}E")
    assert k["smem"] + smem <= MAX_BLOCK_SMEM and k["smem"] + smem + 1024 <= SMEM_PER_SM, (k, smem)
    assert _resident_ctas(k["regs"], threads, k["smem"] + smem) == 1, k
    assert dig * nc <= {64: 512, 32: 256, 16: 128}[nc]  # columns of tensor memory
