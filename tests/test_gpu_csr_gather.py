"""The CSR pass that gathers from the scaled copy of q_i against the pass that
scales while it gathers.  Only the last step of a run has no copy, so step k of
a k-step run and of a longer run take the two paths on the same vectors: the
coefficients are bitwise the same."""
import numpy as np
import pytest

from paper_1602_02306_gb300 import evc
from paper_1602_02306_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_02306_gb300 import build
    build.build()
    evc.load()


@pytest.mark.parametrize("prec", [evc.EVC_FP64, evc.EVC_MIXED])
@pytest.mark.parametrize("n,m,shifts", [(1, 3, [0.3]), (17, 1, [0.3]), (1003, 33, [-0.5, 0.5]),
                                         (5001, 64, [-0.5, 0.5])])
@pytest.mark.parametrize("threads", [128, 256, 512])
def test_copied_and_direct_gathers_are_bitwise_the_same(prec, n, m, shifts, threads):
    csr = I.powerlaw_symmetric(n, cap=200, seed=2) if n > 1 else \
        (np.array([0, 1]), np.array([0], dtype=np.int32), np.array([1.5]))
    ncol = len(shifts) * m
    with evc.Context.csr(csr, precision=prec) as ctx:
        ctx.set_precond(evc.EVC_PREC_JACOBI, 1e-3)
        ctx.set_option(evc.EVC_OPT_CSR_THREADS, threads)
        K = min(6, n)
        ctx.count_slices(shifts, m, K, seed=3)
        al, be, _ = ctx.tridiag(ncol, K)
        for k in range(1, K):
            ctx.count_slices(shifts, m, k, seed=3)
            a, b, _ = ctx.tridiag(ncol, k)
            np.testing.assert_array_equal(a, al[:, :k])
            np.testing.assert_array_equal(b[:, :k], be[:, :k])
            np.testing.assert_array_equal(b[:, k], be[:, k])
