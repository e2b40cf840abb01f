"""How many blocks share a row block of the reorthogonalisation kernels depends on
the launch, its sums do not: FP64 runs of the T^-1 process and runs whose row
blocks are one or two tiles of the update kernel give a column the same bits
alone and in batches that take other numbers of blocks, and one, four and sixteen
row blocks in flight in the sums of the partials agree with the oracle."""
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


def _batches(ctx, K, chunks):
    out = []
    for c in chunks:
        ctx.count_slices([0.3], 32 * c, K, seed=3)
        out.append([x[:32] for x in ctx.tridiag(32 * c, K)[:2]])
    for a, b in out[1:]:
        np.testing.assert_array_equal(a, out[0][0])
        np.testing.assert_array_equal(b, out[0][1])
    return out[0]


@pytest.mark.parametrize("prec", [evc.EVC_FP64, evc.EVC_MIXED])
@pytest.mark.parametrize("n,chunks", [(300, (1, 2, 31)), (7000, (1, 2, 3, 4, 5)), (65000, (1, 2, 3, 4, 8))])
def test_tinv_batches_keep_the_coefficients(prec, n, chunks):
    with evc.Context.csr(_chain(n), precision=prec) as ctx:
        ctx.set_precond(evc.EVC_PREC_JACOBI, 1e-3)
        ctx.set_option(evc.EVC_OPT_TINV_LANCZOS, 1)
        _batches(ctx, 34, chunks)                      # five groups of vectors


@pytest.mark.parametrize("prec", [evc.EVC_FP64, evc.EVC_MIXED])
@pytest.mark.parametrize("n", [31, 32, 33, 63, 64, 65, 129, 256, 257, 1024, 1025, 2048, 2049, 4096, 4097])
def test_row_blocks_of_one_or_two_tiles(prec, n):
    csr, K = _chain(n), min(12, n)
    with evc.Context.csr(csr, precision=prec) as ctx:
        al, be = _batches(ctx, K, (1, 3, 40))
    # ten steps against the FP64 oracle: rounding of 1e-16 (FP32: 6e-8) per operation,
    # some sqrt(n) < 65 of them in a sum, ten steps
    tol = 1e-12 if prec == evc.EVC_FP64 else 1e-3
    k = min(10, K)
    a, b, _, _ = O.lanczos(O.Problem.csr_matrix(csr, O.PREC_NONE), 0.3, O.probe_vector(3, 31, n), k)
    np.testing.assert_allclose(al[31, :k], a, rtol=0, atol=6 * tol)
    np.testing.assert_allclose(be[31, 1:k], b[1:k], rtol=0, atol=6 * tol)
