"""FP64 stencil passes, whose scales and coefficients are folded into per-column
constants: the coefficients of a few Lanczos steps against the oracle, and the three
kernels (single points, patches, tensor-copied tiles) against one another, bit by bit."""
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


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("N", [5, 8, 17, 24])      # odd, tiles filled and not
@pytest.mark.parametrize("prec", ["identity", "jacobi", "tinv", "cheb"])
def test_folded_passes(order, N, prec):
    V, k, m, tau = I.gaussian_wells(N, 0.3, nwells=3, seed=1), 5, 33, -1.3
    got = []
    for patch in (1, 2, 3):
        with evc.Context.stencil(N, 0.3, order, V, precision=evc.EVC_FP64) as ctx:
            if prec == "cheb":
                ctx.set_precond(evc.EVC_PREC_CHEB_KINETIC, 6, 1.0)
            elif prec != "identity":
                ctx.set_precond(evc.EVC_PREC_JACOBI, 1e-3)
            ctx.set_option(evc.EVC_OPT_TINV_LANCZOS, 1 if prec == "tinv" else 0)
            ctx.set_option(evc.EVC_OPT_STENCIL_PATCH, patch)
            ctx.count_slices([tau], m, k, seed=3)
            got.append(ctx.tridiag(m, k)[:2])
    for a, b in got[1:]:
        np.testing.assert_array_equal(a, got[0][0])
        np.testing.assert_array_equal(b, got[0][1])
    kind = {"identity": O.PREC_NONE, "jacobi": O.PREC_JACOBI, "tinv": O.PREC_JACOBI, "cheb": O.PREC_CHEB}[prec]
    P = O.Problem.stencil(N, 0.3, order, V, kind, jac_eps=1e-3, cheb_degree=6, cheb_c=1.0)
    for j in (0, 32):
        # five steps of sums of n < 14,000 products, each off by some 1e-16 of the
        # operator's norm, which the Jacobi scales of a near-zero diagonal raise
        a, b, _, kd = O.lanczos(P, tau, O.probe_vector(3, j, N ** 3), k)
        tol = 1e-10 * max(np.abs(a).max(), np.abs(b).max())
        np.testing.assert_allclose(got[0][0][j, :kd], a, rtol=0, atol=tol)
        np.testing.assert_allclose(got[0][1][j, 1:kd], b[1:kd], rtol=0, atol=tol)
