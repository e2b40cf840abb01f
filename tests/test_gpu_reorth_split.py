"""The splits of the reorthogonalisation kernels.  The dot kernel shares a row
block's basis vectors between blocks when there are few columns, and every sum
keeps its order: a batch of many columns, which is not split, gives the same
bits.  The update kernel shares a row block's tiles below 64 x 3456 rows: both
sides of that line against the oracle.  And counts that share the GPU with others
give the bits that they give alone."""
import threading

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
@pytest.mark.parametrize("n", [5, 70, 4100, 221183, 221184])
def test_splits_keep_the_coefficients(prec, n):
    csr, K, m = _chain(n), min(20, n), 32          # K: three groups of eight vectors
    with evc.Context.csr(csr, precision=prec) as ctx:
        ctx.count_slices([0.3], m, K, seed=3)
        al, be, kd = ctx.tridiag(m, K)
        ctx.count_slices([0.3], 10 * m, K, seed=3)
        al2, be2, kd2 = ctx.tridiag(10 * m, K)
    np.testing.assert_array_equal(al, al2[:m])
    np.testing.assert_array_equal(be, be2[:m])
    # ten steps (before any Ritz value converges) against the FP64 oracle: rounding
    # of 1e-16 (FP32: 6e-8) per operation, some sqrt(n) < 500 of them in a sum, ten steps
    tol = 1e-11 if prec == evc.EVC_FP64 else 1e-3
    P = O.Problem.csr_matrix(csr, O.PREC_NONE)
    for j in (0, 31):
        a, b, _, k = O.lanczos(P, 0.3, O.probe_vector(3, j, n), min(10, K))
        np.testing.assert_allclose(al[j, :k], a, atol=tol * 6)
        np.testing.assert_allclose(be[j, 1:k], b[1:k], atol=tol * 6)


def test_counts_side_by_side_give_the_bits_of_one_alone():
    import torch
    ctxs, alone, bad = [], [], []
    for N in (40, 50, 60):
        st = torch.cuda.Stream()
        ctx = evc.Context.stencil(N, 0.3, 2, I.gaussian_wells(N, 0.3, nwells=4, seed=1),
                                  precision=evc.EVC_MIXED, stream=st.cuda_stream)
        ctxs.append((ctx, st))
        ctx.count_slices([-2.0, -1.0], 32, 30, seed=3)
        alone.append(ctx.tridiag(64, 30)[:2])

    def work(i):
        for _ in range(40):
            ctxs[i][0].count_slices([-2.0, -1.0], 32, 30, seed=3)
            bad.extend(i for x, y in zip(ctxs[i][0].tridiag(64, 30)[:2], alone[i]) if not np.array_equal(x, y))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for ctx, _ in ctxs:
        ctx.close()
    assert not bad
