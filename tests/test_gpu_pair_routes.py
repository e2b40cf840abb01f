"""Chebyshev passes in pairs and one by one are bitwise the same in whole counts:
several chunks, chunk groups, the last pass of M with the three-term operand and
the factor of a real root, on both sides of the line between the two.  The
reference is the passes one by one, which 2 x 2 patches run on grids of 18 to 22
points a side from some number of columns on: columns are independent, so the
same probes in a small batch (pairs) give the same bits."""
import numpy as np
import pytest

from paper_1602_02306_gb300 import evc
from paper_1602_02306_gb300 import inputs as I

pytestmark = pytest.mark.gpu
H = 0.3


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_02306_gb300 import build
    build.build()
    evc.load()


def _tridiag(N, degree, groups, patch, m, K, shifts=(-2.0,)):
    with evc.Context.stencil(N, H, 2, I.gaussian_wells(N, H, nwells=8, seed=1),
                             precision=evc.EVC_MIXED) as ctx:
        ctx.set_precond(evc.EVC_PREC_CHEB_KINETIC, degree, 1.0)
        ctx.set_option(evc.EVC_OPT_STENCIL_GROUPS, groups)
        ctx.set_option(evc.EVC_OPT_STENCIL_PATCH, patch)
        _, q, _ = ctx.count_slices(list(shifts), m, K, seed=3)
        a, b, _ = ctx.tridiag(len(shifts) * m, K)
    return a, b, q


@pytest.mark.parametrize("degree", [7, 8])                 # with a real root, without
@pytest.mark.parametrize("N", [18, 20, 22])
def test_pairs_and_single_passes_give_the_same_bits(N, degree):
    K, small = 4, 40
    many = 32 * (-(-180000 // N ** 3))                     # first size without pairs
    a1, b1, q1 = _tridiag(N, degree, 4, 2, many, K)        # one by one
    a2, b2, q2 = _tridiag(N, degree, 4, 2, many - 32, K)   # pairs, groups of chunks
    a3, b3, q3 = _tridiag(N, degree, 1, 2, small, K)       # pairs, two chunks
    for m, a, b, q in ((many - 32, a2, b2, q2), (small, a3, b3, q3)):
        np.testing.assert_array_equal(a1[:m], a)
        np.testing.assert_array_equal(b1[:m], b)
        np.testing.assert_array_equal(q1[0, :m], q[0])


@pytest.mark.parametrize("N", [12, 14, 26, 30])
def test_chunks_and_groups_give_the_same_bits(N):
    a1, b1, q1 = _tridiag(N, 8, 1, 2, 100, 5, (-2.0, -1.0))
    for groups in (2, 4):
        for patch in (2, 3):
            a, b, q = _tridiag(N, 8, groups, patch, 100, 5, (-2.0, -1.0))
            np.testing.assert_array_equal(a, a1)
            np.testing.assert_array_equal(b, b1)
            np.testing.assert_array_equal(q, q1)
