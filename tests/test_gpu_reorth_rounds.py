"""The number of blocks that share a row block in the reorthogonalisation kernels
follows the size of the launch; the sums do not: batches of 1, 3 and 10 chunks of
columns give the same bits, on both sides of each line at which the dot kernel's FP64
route or the number of segments of the update kernel changes, and agree with the
oracle."""
import numpy as np
import pytest

from oracle import oracle as O
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


def _chain(n):
    r = np.arange(n)
    d = np.random.default_rng(n).uniform(0.0, 4.0, size=n)
    return I.coo_to_csr(n, np.r_[r, r[1:], r[:-1]], np.r_[r, r[:-1], r[1:]],
                        np.r_[d, -np.ones(2 * (n - 1))])


@pytest.mark.parametrize("prec", [evc.EVC_FP64, evc.EVC_MIXED])
@pytest.mark.parametrize("n,K", [(8191, 20), (8192, 2), (63999, 18), (64000, 18), (131071, 10), (131072, 18),
                                 (511 * 3456, 3), (511 * 3456 + 1, 3)])
def test_batches_keep_the_coefficients(prec, n, K):
    csr, m = _chain(n), 32
    with evc.Context.csr(csr, precision=prec) as ctx:
        got = []
        for chunks in (1, 3, 10 if n < 1000000 else 4):
            ctx.count_slices([0.3], chunks * m, K, seed=3)
            got.append([x[:m] for x in ctx.tridiag(chunks * m, K)[:2]])
    for a, b in got[1:]:
        np.testing.assert_array_equal(a, got[0][0])
        np.testing.assert_array_equal(b, got[0][1])
    # ten steps (before any Ritz value converges) against the FP64 oracle: rounding of
    # 1e-16 (FP32: 6e-8) per operation, some sqrt(n) < 1400 of them in a sum, ten steps
    tol = 1e-11 if prec == evc.EVC_FP64 else 1e-3
    k = min(10, K)
    a, b, _, _ = O.lanczos(O.Problem.csr_matrix(csr, O.PREC_NONE), 0.3, O.probe_vector(3, 31, n), k)
    np.testing.assert_allclose(got[0][0][31, :k], a, rtol=0, atol=6 * tol)
    np.testing.assert_allclose(got[0][1][31, 1:k], b[1:k], rtol=0, atol=6 * tol)
