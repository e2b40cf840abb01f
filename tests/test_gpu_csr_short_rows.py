"""CSR passes on rows of every length around a batch of gathers (1 to 19 entries
and empty rows but for the diagonal), of few and of many columns, and on both
sides of the row length from which a Jacobi run in FP32 keeps a scaled copy of
q_i: alpha_1 and beta_2 against the operator in numpy float64.  A row of r
products summed one by one is off by at most (r + 4) u of the sum of their
magnitudes, here below 40 u times the largest such sum of any row times the
norms; alpha_1 and beta_2 are means over n rows of such terms."""
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


def _ragged(n, longest, seed):
    """Symmetric; row r couples to r % (longest / 2 + 1) later rows."""
    rng = np.random.default_rng(seed)
    r, c = [], []
    for i in range(n):
        k = min(i % (longest // 2 + 1), n - 1 - i)
        c += list(i + 1 + rng.choice(n - 1 - i, size=k, replace=False)) if k else []
        r += [i] * k
    r, c = np.array(r, dtype=np.int64), np.array(c, dtype=np.int64)
    v, d = rng.standard_normal(r.size), rng.uniform(-5, 5, n)
    i = np.arange(n)
    return I.coo_to_csr(n, np.r_[i, r, c], np.r_[i, c, r], np.r_[d, v, v])


@pytest.mark.parametrize("prec", [evc.EVC_FP64, evc.EVC_MIXED])
@pytest.mark.parametrize("mode", ["identity", "jacobi", "tinv"])
@pytest.mark.parametrize("n,longest", [(37, 6), (501, 20), (501, 40), (1030, 4)])
@pytest.mark.parametrize("S,m", [(1, 32), (2, 20)])
def test_first_step_against_numpy(prec, mode, n, longest, S, m):
    csr = _ragged(n, longest, seed=n + longest)
    A = np.zeros((n, n))
    rows = np.repeat(np.arange(n), np.diff(csr[0]))
    np.add.at(A, (rows, csr[1]), csr[2])
    shifts = [0.3, -0.7][:S]
    with evc.Context.csr(csr, precision=prec) as ctx:
        ctx.set_precond(evc.EVC_PREC_IDENTITY if mode == "identity" else evc.EVC_PREC_JACOBI, 1e-1)
        ctx.set_option(evc.EVC_OPT_SHARED_KRYLOV, 0)
        if mode == "tinv":
            ctx.set_option(evc.EVC_OPT_TINV_LANCZOS, 1)
        ctx.count_slices(shifts, m, 3, seed=3)
        al, be, _ = ctx.tridiag(S * m, 3)
    u = 2.0 ** -53 if prec == evc.EVC_FP64 else 2.0 ** -24
    for s, tau in enumerate(shifts):
        B = A - tau * np.eye(n)
        if mode != "identity":
            M = 1.0 / np.sqrt(np.abs(np.diag(A) - tau) + 1e-1)
            B = M[:, None] * B * M[None, :]
        bound = 40 * u * np.abs(B).sum(1).max()
        for j in (0, m - 1):
            q = O.probe_vector(3, j, n) / np.sqrt(n)
            w = B @ q
            a1 = q @ w
            b2 = np.linalg.norm(w - a1 * q)
            assert abs(al[s * m + j, 0] - a1) <= bound
            assert abs(be[s * m + j, 1] - b2) <= 2 * bound
