"""Quadratures of many columns, several to a warp: the same bits as one block per
column, whatever the sizes in a warp, with columns that fail among them; and the
static call's two eigensolvers, which take turns by the number of columns, agree
to rounding."""
import numpy as np
import pytest

from paper_1602_02306_gb300 import evc
from paper_1602_02306_gb300 import inputs as I

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_02306_gb300 import build
    build.build()
    evc.load()


def _static(alpha, beta, sizes=None):
    import torch
    k, ncol = alpha.shape
    a, b = torch.from_numpy(np.ascontiguousarray(alpha)).cuda(), torch.from_numpy(np.ascontiguousarray(beta)).cuda()
    kc = None if sizes is None else torch.from_numpy(np.ascontiguousarray(sizes, dtype=np.int32)).cuda()
    q = torch.zeros(ncol, dtype=torch.float64, device="cuda")
    st = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    rc, msg = evc.evc_gauss_quadrature_static(a.data_ptr(), b.data_ptr(), None if kc is None else kc.data_ptr(), k,
                                              ncol, 2.0, q.data_ptr(), st.data_ptr())
    assert rc == evc.EVC_OK, msg
    torch.cuda.synchronize()
    return q.cpu().numpy(), int(st.item())


def _matrices(k, ncol, seed):
    rng = np.random.default_rng(seed)
    alpha, beta = 0.3 * rng.standard_normal((k, ncol)), 0.7 + 0.6 * rng.random((k + 1, ncol))
    alpha[:, 3::7] = np.round(alpha[:, 3::7])                       # close poles
    beta[:, 4::7] = 10.0 ** rng.uniform(-18, 0, beta[:, 4::7].shape)   # small couplings
    beta[:, 5::7] *= -1e120
    alpha[:, 5::7] *= 1e120
    return alpha, beta


@pytest.mark.parametrize("k", [4, 5, 6, 7, 8, 9, 10, 11, 15, 16, 17, 21, 31, 32])
def test_packed_columns_have_the_bits_of_single_ones(k):
    ncol = 1500 if k <= 16 else 4096
    alpha, beta = _matrices(k, ncol, k)
    sizes = np.random.default_rng(k).integers(1, k + 1, ncol)
    alpha[0, 10], beta[1, 11], alpha[k - 1, 12] = np.nan, np.inf, -np.inf
    for kc in (None, sizes):
        q, st = _static(alpha, beta, kc)
        assert st == evc.EVC_ENUMERIC
        for lo in (0, 600, ncol - 100):
            part = slice(lo, lo + 100)                              # one block per column
            p, _ = _static(alpha[:, part], beta[:, part], None if kc is None else kc[part])
            np.testing.assert_array_equal(p, q[part])
        assert np.isnan(q[10])
    sizes[20], sizes[21] = 0, k + 1
    q, st = _static(alpha[:, 13:], beta[:, 13:], sizes[13:])
    assert st == evc.EVC_EINVAL and list(np.flatnonzero(np.isnan(q))) == [7, 8]


@pytest.mark.parametrize("k,line", [(2, 2048), (4, 2048), (5, 4096), (16, 4096), (31, 4096)])
def test_both_eigensolvers_agree(k, line):
    # 0 in a gap of every spectrum: two rows of +-4 on the diagonal keep the rest away
    rng = np.random.default_rng(k)
    alpha = np.where(rng.random((k, line + 1)) < 0.5, -4.0, 4.0) + 0.3 * rng.standard_normal((k, line + 1))
    beta = 0.7 + 0.6 * rng.random((k + 1, line + 1))
    few, _ = _static(alpha[:, :line], beta[:, :line])
    many, _ = _static(alpha, beta)
    # both within 64 k eps ||J|| / gap of the exact weights (twice vnorm2 = 2)
    J = np.zeros((line, k, k))
    i = np.arange(k)
    J[:, i, i] = alpha[:, :line].T
    J[:, i[1:], i[:-1]] = J[:, i[:-1], i[1:]] = beta[1:k, :line].T
    th = np.linalg.eigvalsh(J)
    bound = 2 * 2.0 * 64 * k * EPS * np.abs(th).max(1) / np.abs(th).min(1)
    assert np.all(np.abs(few - many[:line]) <= bound)


@pytest.mark.parametrize("prec", [evc.EVC_FP64, evc.EVC_MIXED])
@pytest.mark.parametrize("rule,K", [(evc.EVC_QUAD_GAUSS, 18), (evc.EVC_QUAD_GA, 10)])
@pytest.mark.parametrize("shifts,precond", [([1.0], evc.EVC_PREC_JACOBI), ([0.7, 1.0, 2.1], evc.EVC_PREC_IDENTITY)])
def test_counts_of_many_columns(prec, rule, K, shifts, precond):
    # columns that break down at different steps (16 rows, all steps run: the stop rule
    # looks at means, which differ between the batches), then a tolerance, with the
    # quadratures of the last three steps formed and no earlier stop allowed
    for N, k, tol in ((4, min(K, 16), 0.0), (12, K, 1e-300)):
        with evc.Context.csr(I.laplace2d_dirichlet(N), precision=prec) as ctx:
            ctx.set_precond(precond, 1e-3)
            ctx.set_option(evc.EVC_OPT_QUADRATURE, rule)
            ctx.set_option(evc.EVC_OPT_MIN_STEPS, k)
            _, few, steps = ctx.count_slices(shifts, 40, k, tol=tol, seed=3)
            _, many, steps2 = ctx.count_slices(shifts, 4200, k, tol=tol, seed=3)
        assert list(steps) == list(steps2) == [k] * len(shifts)
        np.testing.assert_array_equal(few, many[:, :40])
