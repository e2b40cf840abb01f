"""The kernel that applies a conjugate pair of the Chebyshev preconditioner's
roots in one launch (FP32, 7-point): M q_1 of a one-step run, read from the
workspace, against the two single passes restated in numpy float32 -- the same
operations in the same order, so the bits must be the same."""
from fractions import Fraction

import numpy as np
import pytest

from paper_1602_02306_gb300 import evc
from paper_1602_02306_gb300 import inputs as I

pytestmark = pytest.mark.gpu
f32, f64 = np.float32, np.float64


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_02306_gb300 import build
    build.build()
    evc.load()


def _fma(a, b, c):
    return (np.asarray(a, f64) * np.asarray(b, f64) + np.asarray(c, f64)).astype(f32)


def _stencil(x, k1, k0, h):
    s = np.roll(x, 1, 2) + np.roll(x, -1, 2)
    for axis in (1, 0):
        s = s + np.roll(x, 1, axis)
        s = s + np.roll(x, -1, axis)
    off = f32(-0.5 / (h * h)) * s
    dg = f32(float(Fraction(k1) * Fraction(3.0 * (1.0 / (h * h))) + Fraction(k0)))
    return _fma(f32(k1), off, dg * x)


@pytest.mark.parametrize("N", [12, 14, 16, 18, 26, 40])      # every tile size, overlapping last tiles
@pytest.mark.parametrize("zb", [3, 64])
def test_pair_is_bitwise_the_two_passes(N, zb):
    import torch
    h, degree, n = 0.3, 2, N ** 3
    ch = evc.evc_cheb_kinetic(2, h, degree, 1.0, N)
    (re, im, is_pair), = ch["factors"]
    assert is_pair
    with evc.Context.stencil(N, h, 2, I.gaussian_wells(N, h, nwells=4, seed=1),
                             precision=evc.EVC_MIXED) as ctx:
        ctx.set_precond(evc.EVC_PREC_CHEB_KINETIC, degree, 1.0)
        ctx.set_option(evc.EVC_OPT_STENCIL_ZB, zb)
        need = evc.evc_workspace_bytes(ctx.h, 1, 32, 1)
        ws = torch.empty(need // 4 + 64, dtype=torch.float32, device="cuda")
        start = (-ws.data_ptr() % 256) // 4
        evc.evc_set_workspace(ctx.h, ws.data_ptr() + 4 * start, need)
        evc.evc_count_slices(ctx.h, [-2.0], 32, 1, seed=3)
        torch.cuda.synchronize()
        # two basis slots, then the work vectors: the third holds M q_1
        v = ws[start:start + 5 * n * 32].cpu().numpy().reshape(5, N, N, N, 32)
        evc.evc_set_workspace(ctx.h, None, 0)
    g, sg, scale = ch["g"], ch["sign"], 1.0 / np.sqrt(float(n))
    u = f32(scale) * _stencil(v[0], g, g * (1.0 - re), h)
    w = _stencil(u, sg * g, sg * g * (1.0 - re), h)
    np.testing.assert_array_equal(v[4], w + f32(sg * g * g * im * im * scale) * v[0])
