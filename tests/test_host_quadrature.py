"""The divide and conquer eigensolver of the quadratures on the host, against
LAPACK: evc_dc.cuh compiled by the host compiler, its phases run in order.

Both solvers return the eigenvalues and first components of a matrix within
some k eps ||J|| of J, so eigenvalues are compared within 4 k eps ||J|| and the
weight below the middle of a gap of the spectrum within 8 k eps ||J|| / gap
(a perturbation E moves it by at most 2 ||E|| / gap)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1602_02306_gb300", "csrc")
EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module")
def solver(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("dc") / "dc_host.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", lib,
                           os.path.join(HERE, "dc_host.cpp")])
    return ctypes.CDLL(lib).dc_eig


def _solve(solver, diag, off):
    k = len(diag)
    a, b = np.array(diag, dtype=np.float64), np.array(list(off) + [0.0], dtype=np.float64)
    theta, first = np.full(k, np.nan), np.full(k, np.nan)
    p = [x.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for x in (a, b, theta, first)]
    solver(ctypes.c_int(k), *p)
    return theta, first


def _check(solver, diag, off):
    diag, off = np.asarray(diag, dtype=np.float64), np.asarray(off, dtype=np.float64)
    k = len(diag)
    theta, first = _solve(solver, diag, off)
    assert np.all(np.isfinite(theta)) and np.all(np.isfinite(first))
    ref, Z = np.linalg.eigh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1))
    norm = np.abs(ref).max()
    assert np.all(np.diff(theta) >= 0.0)
    np.testing.assert_allclose(theta, ref, rtol=0, atol=4 * k * EPS * norm)
    gap = np.diff(ref)
    below, exact = np.cumsum(first ** 2), np.cumsum(Z[0] ** 2)
    assert abs(below[-1] - 1.0) <= 8 * k * EPS
    for t in np.flatnonzero(gap > 1e-6 * norm):
        assert abs(below[t] - exact[t]) <= 8 * k * EPS * norm / gap[t]


@pytest.mark.parametrize("tiny", [1e-150, 1e-162, 1e-165, 1e-200, 1e-300, 5e-324])
@pytest.mark.parametrize("k", [2, 3, 4, 5, 40])
def test_equal_diagonal_entries_with_a_vanishing_coupling(solver, k, tiny):
    # the square of the coupling underflows in the rotation of two rows
    _check(solver, [-1.0] * k, [tiny] * (k - 1))
    _check(solver, [-3.0, -3.0, 2.0, 5.0][:k] + [1.0] * (k - 4), ([tiny, tiny, 0.5] + [tiny] * k)[:k - 1])
    rng = np.random.default_rng(k)
    off = np.where(rng.random(k - 1) < 0.5, tiny, 0.7)
    _check(solver, np.round(rng.standard_normal(k)), off)


@pytest.mark.parametrize("k", [1, 2, 3, 7, 16, 33, 64, 100, 255])
def test_matrices_of_every_kind(solver, k):
    rng = np.random.default_rng(k)
    a, b = 0.3 * rng.standard_normal(k), 0.7 + 0.6 * rng.random(k)
    e = b[:k - 1]
    _check(solver, a, e)
    _check(solver, np.abs(np.arange(k) - k // 2), np.ones(k - 1))
    _check(solver, np.zeros(k), np.ones(k - 1))
    _check(solver, np.ones(k), np.zeros(k - 1))
    _check(solver, np.concatenate([a, a[:-1][::-1]]), np.concatenate([e, b[k - 1:k] if k > 1 else [], e[:-1][::-1]]))
    _check(solver, a * 1e150, -e * 1e150)
    _check(solver, a * 1e-300, e * 1e-300)
    _check(solver, a, 10.0 ** rng.uniform(-20, 0, k - 1))
    # entries over the whole range: pieces far below single precision's range
    for lo in (-30, -44, -60, -150, -300):
        _check(solver, a * 10.0 ** rng.uniform(lo, 0, k), 10.0 ** rng.uniform(lo, 0, k - 1))
        _check(solver, np.concatenate([a * 10.0 ** lo, [1.0]]), np.concatenate([e * 10.0 ** lo, [10.0 ** lo] if k else []]))
