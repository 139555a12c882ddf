"""A product of the gradient or of a standalone orthogonalisation that gives up its wait is
reported as a timeout, not as a value in the caller's data, and the context stays usable."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _code(tsvd, call):
    with tsvd.wait_limit(2):
        with pytest.raises(tsvd.TsvdError) as e:
            call()
    return e.value.code


@pytest.mark.parametrize("side", ["u", "v"])
def test_gradient_reports_a_timeout(tsvd, side):
    import torch

    import workloads
    from paper_2403_06218_gb300 import _capi
    m, n, k = 24_000, 20_001, 32
    g = torch.Generator(device="cuda").manual_seed(2)
    A = tsvd.CsrMatrix.from_scipy(workloads.csr_uniform(m, n, 10, seed=3))
    # (any orthonormal columns will do: the call ends at its first check)
    U, V = (torch.linalg.qr(torch.randn(x, k, generator=g, dtype=torch.float64, device="cuda"))[0].contiguous()
            for x in (m, n))
    s = torch.linspace(20, 19, k, dtype=torch.float64, device="cuda")
    bar = {"u": (torch.randn(m, k, generator=g, dtype=torch.float64, device="cuda"), None),
           "v": (None, torch.randn(n, k, generator=g, dtype=torch.float64, device="cuda"))}[side]
    def call():
        return tsvd.svd_backward(A, s, U, V, None, *bar)
    assert _code(tsvd, call) == _capi.TSVD_ERR_TIMEOUT
    grad = call()[0]
    assert bool(torch.isfinite(grad).all())


def test_orthogonalisation_reports_a_timeout(tsvd):
    import torch

    from paper_2403_06218_gb300 import _capi
    g = torch.Generator(device="cuda").manual_seed(4)
    Y = torch.randn(20_000, 64, generator=g, dtype=torch.float64, device="cuda")
    assert _code(tsvd, lambda: tsvd.cholqr2(Y)) == _capi.TSVD_ERR_TIMEOUT
    Q, R, _ = tsvd.cholqr2(Y)
    off = (Q.t() @ Q - torch.eye(64, dtype=torch.float64, device="cuda")).abs().max()
    assert float(off) < 100 * np.finfo(float).eps
