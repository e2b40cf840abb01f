"""The block-per-column eigensolver behind the quadratures, against LAPACK.

The weight of the eigenvalues below a gap moves by at most 2 ||E|| / gap under
a perturbation E of the matrix; both sides are backward stable, so each test's
tolerance is 64 k eps ||J|| / gap for its own matrices (gap: the distance of
the shift, 0, from the spectrum)."""
import numpy as np
import pytest

from paper_1602_02306_gb300 import evc

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


def _quad(alpha, beta, sizes=None):
    """alpha [ncol, k], beta [ncol, k + 1] -> (quad, status, call status)."""
    import torch
    ncol, k = alpha.shape
    a = torch.from_numpy(np.ascontiguousarray(alpha.T)).cuda()
    b = torch.from_numpy(np.ascontiguousarray(beta.T)).cuda()
    kc = torch.from_numpy(np.asarray(sizes, dtype=np.int32)).cuda() if sizes is not None else None
    q = torch.zeros(ncol, dtype=torch.float64, device="cuda")
    st = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    rc, msg = evc.evc_gauss_quadrature_static(a.data_ptr(), b.data_ptr(),
                                              kc.data_ptr() if kc is not None else None, k, ncol, 2.0,
                                              q.data_ptr(), st.data_ptr())
    torch.cuda.synchronize()
    return q.cpu().numpy(), int(st.item()), rc


def _eig(a, b):
    return np.linalg.eigh(np.diag(a) + np.diag(b[1:len(a)], 1) + np.diag(b[1:len(a)], -1))


def _centre(a, b):
    """The diagonal moved so that 0 lies in the middle of the widest gap of the
    middle half of the spectrum; gap / 2 and ||J||."""
    th = _eig(a, b)[0]
    if len(th) == 1:
        return a - th[0] - 1.0, 1.0, 1.0
    lo, hi = len(th) // 4, max(len(th) // 4 + 1, 3 * len(th) // 4)
    g = np.diff(th)[lo:hi]
    i = lo + int(np.argmax(g))
    s = 0.5 * (th[i] + th[i + 1])
    return a - s, 0.5 * (th[i + 1] - th[i]), np.abs(th - s).max()


def _kinds(k, rng):
    beta = 0.7 + 0.6 * rng.random(k + 1)
    yield 0.3 * rng.standard_normal(k), beta                        # generic
    yield np.abs(np.arange(k) - k // 2).astype(float), np.ones(k + 1)   # pairs equal to rounding
    b = beta.copy()
    b[k // 2] = 0.0                                                 # two uncoupled halves
    yield 0.3 * rng.standard_normal(k), b
    b = beta.copy()
    b[1::3] *= 1e-13                                                # nearly uncoupled pieces
    yield rng.standard_normal(k), b
    yield rng.standard_normal(k), 10.0 ** rng.uniform(-18, 0, k + 1)
    yield rng.standard_normal(k) * 1e120, -beta * 1e120             # scaled, negative couplings


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33, 64, 65, 128, 129, 134, 255, 256])
def test_block_quadrature_equals_lapack(k):
    rng = np.random.default_rng(k)
    cols = [(*_centre(a, b), b) for a, b in _kinds(k, rng)]
    quad, status, rc = _quad(np.stack([c[0] for c in cols]), np.stack([c[3] for c in cols]))
    assert rc == evc.EVC_OK and status == evc.EVC_OK
    for (a, gap, norm, b), q in zip(cols, quad):
        th, Z = _eig(a, b)
        ref = 2.0 * (Z[0] ** 2)[th < 0].sum()
        assert abs(q - ref) <= 2.0 * 64 * k * EPS * norm / gap


@pytest.mark.parametrize("ncol", [3, 4097])       # one block, one thread per column
def test_column_sizes_and_non_finite_columns(ncol):
    rng = np.random.default_rng(1)
    k = 12
    alpha, beta = 0.3 * rng.standard_normal((ncol, k)), 0.7 + 0.6 * rng.random((ncol, k + 1))
    sizes = rng.integers(1, k + 1, ncol)
    centred = [_centre(alpha[c, :s], beta[c, :s + 1]) for c, s in enumerate(sizes)]
    for c, s in enumerate(sizes):
        alpha[c, :s] = centred[c][0]
    sizes[1], alpha[2, 0] = k + 1, np.inf
    quad, status, rc = _quad(alpha, beta, sizes)
    assert rc == evc.EVC_OK and status in (evc.EVC_EINVAL, evc.EVC_ENUMERIC)
    assert np.isnan(quad[1]) and np.isnan(quad[2])
    for c in [0] + list(range(3, min(ncol, 300))):
        s = sizes[c]
        th, Z = _eig(alpha[c, :s], beta[c, :s + 1])
        ref = 2.0 * (Z[0] ** 2)[th < 0].sum()
        assert abs(quad[c] - ref) <= 2.0 * 64 * s * EPS * centred[c][2] / centred[c][1]


def test_averaged_rule_of_the_longest_run():
    # 2 k - 1 = 511 rows; the extended matrix is its own mirror image
    from paper_1602_02306_gb300 import inputs as I
    csr = I.laplace2d_dirichlet(24)
    with evc.Context.csr(csr, precision=evc.EVC_FP64) as ctx:
        ctx.set_option(evc.EVC_OPT_QUADRATURE, evc.EVC_QUAD_GA)
        _, quad, _ = ctx.count_slices([2.011], 2, 256)
        al, be, kd = ctx.tridiag(2, 256)
    for c in range(2):
        k = int(kd[c])
        a, b = al[c, :k], be[c, :k + 1]
        full = np.concatenate([a, a[:-1][::-1]])
        off = np.concatenate([b[1:k], b[k:k + 1], b[1:k - 1][::-1]])
        th, Z = _eig(full, np.concatenate([[0.0], off]))
        gap = np.abs(th).min()
        ref = 576 * (Z[0] ** 2)[th < 0].sum()
        assert abs(quad[0, c] - ref) <= 576 * 64 * len(full) * EPS * np.abs(th).max() / gap
