"""The quadrature of tridiagonals with couplings far below the rounding of
their diagonals, whose squares underflow.  With equal diagonal entries on
every coupled row the matrix is, to rounding, its diagonal in another basis:
the weight below 0 is 1 when all entries are negative, and in general the
first row's share, compared with LAPACK's within 64 k eps ||J|| / gap."""
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


@pytest.mark.parametrize("k", [2, 3, 4, 5, 8, 40])
def test_vanishing_couplings(k):
    import torch
    tiny = [1e-150, 1e-162, 1e-165, 1e-200, 1e-300, 5e-324]
    alpha, beta = [], []
    for t in tiny:
        alpha.append([-1.0] * k)
        beta.append([0.0] + [t] * k)
        alpha.append(([-3.0, -3.0, 2.0, 5.0] + [1.0] * k)[:k])
        beta.append(([0.0, t, t, 0.5] + [t] * k)[:k + 1])
        alpha.append(([2.0, 2.0, -3.0, -3.0] * k)[:k])
        beta.append(([0.0, t, 3.0, t] + [t, 1.0] * k)[:k + 1])
    a = torch.tensor(alpha, dtype=torch.float64).T.contiguous().cuda()
    b = torch.tensor(beta, dtype=torch.float64).T.contiguous().cuda()
    q = torch.zeros(a.shape[1], dtype=torch.float64, device="cuda")
    st = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    rc, msg = evc.evc_gauss_quadrature_static(a.data_ptr(), b.data_ptr(), None, k, a.shape[1], 1.0,
                                              q.data_ptr(), st.data_ptr())
    assert rc == evc.EVC_OK, msg
    torch.cuda.synchronize()
    assert int(st.item()) == evc.EVC_OK
    for c, got in enumerate(q.cpu().numpy()):
        off = beta[c][1:k]
        th, Z = np.linalg.eigh(np.diag(alpha[c]) + np.diag(off, 1) + np.diag(off, -1))
        gap, norm = np.abs(th).min(), np.abs(th).max()
        assert abs(got - (Z[0] ** 2)[th < 0].sum()) <= 64 * k * EPS * norm / gap, (c, tiny[c // 3])
