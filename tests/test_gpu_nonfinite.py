"""Inputs that are not finite, without a GPU fault: every mesh index is clamped or wrapped, whatever the
position, so that a position that is not finite can only make values that are not finite.  They must be
reported."""

import numpy as np
import pytest

import pic_inputs as pi

pytestmark = pytest.mark.gpu

NAMES = ("x", "v", "P", "vprev", "phi", "psi", "rho", "A", "U")


@pytest.fixture(scope="module")
def sim(cuda_ok):
    from paper_2606_15035_gb300 import build
    build.build()
    from paper_2606_15035_gb300 import sim as s
    return s


@pytest.mark.parametrize("precision,diagnostics", [(0, 0), (0, 1), (1, 0)])
@pytest.mark.parametrize("value", [np.nan, -np.nan, np.inf, -np.inf])
def test_position_that_is_not_finite_is_reported_and_the_state_kept(sim, precision, diagnostics, value):
    w = pi.WORKLOADS["twostream-8c-8k"]
    x, v, q, m = pi.random_twostream(w.n, w.L, 2, w.v0, w.eps, 1e-3, 4100)
    cfg = sim.pic_config_default(n=w.n, L=w.L, dt=w.dt, picard_tol=1e-13, precision=precision, diagnostics=diagnostics)
    s = sim.PicSim(cfg, x, v, q, m)
    s.step(1)
    good = s.get_state()
    bad = s.get_state()
    bad.x[17, 1] = value
    s.set_state(bad)
    before = s.get_state()
    assert np.isnan(before.x[17, 1])                # (wrapping an infinity leaves a NaN)
    for call in (lambda: s.step(1), lambda: s.iterate(good.v)):
        with pytest.raises(sim.PicError) as e:
            call()
        assert e.value.status == 5                  # PIC_ERR_NONFINITE
    after = s.get_state()
    for name in NAMES:
        assert np.array_equal(getattr(after, name), getattr(before, name), equal_nan=True), name
    s.set_state(good)                               # the cause removed: the context works again
    assert s.step(1).converged
    s.close()
