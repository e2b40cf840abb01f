"""The end of the pair kernel after a wait that gave up: it waits for the copies
that were issued, and only for those, and the device goes on working."""
import time

import numpy as np
import pytest

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


def _count():
    with evc.Context.stencil(12, 0.3, 2, I.gaussian_wells(12, 0.3, nwells=4, seed=1),
                             precision=evc.EVC_MIXED) as ctx:
        ctx.set_precond(evc.EVC_PREC_CHEB_KINETIC, 8, 1.0)
        return ctx.count_slices([-2.0, -1.0], 32, 8, seed=3)[1]


def test_a_missing_copy_ends_in_one_limit_and_the_device_stays_usable():
    before = _count()
    assert evc.evc_wait_selftest(1.0) == evc.EVC_ETIMEOUT
    # two waits run out, one after the other; were a copy that nobody issued
    # waited for at the kernel's end, a third would
    t0 = time.perf_counter()
    assert evc.evc_wait_selftest(400.0) == evc.EVC_ETIMEOUT
    dt = time.perf_counter() - t0
    assert 0.75 < dt < 1.1
    np.testing.assert_array_equal(_count(), before)
