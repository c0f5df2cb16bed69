"""Corner depths no water has: not land, which only SWE_LAND is, but a numeric
error of the domain, also where a fixed step never asks for the wave speed."""
import numpy as np
import pytest

from paper_1912_02457_gb300 import synth
from tests import helpers
from tests.test_gpu_parity import swe  # noqa: F401

pytestmark = pytest.mark.gpu


def _case(dtype, **params):
    wl = helpers.flat(61, 40, dtype=dtype, **params)
    wl.eta = (0.1 * np.random.default_rng(1).standard_normal((40, 61))).astype(dtype)
    return wl


@pytest.mark.parametrize("dt", [0.0, 1.0])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("prec", ["f32", "f32_kahan", "f64"])
def test_a_depth_that_is_not_finite_is_an_error(swe, prec, bad, dt):
    wl = _case(np.float64 if prec == "f64" else np.float32, dt_fixed=dt)
    wl.H[17, 30] = bad
    with swe.Domain(wl, prec) as d:
        d.step(2)
        i = d.info(check=False)
    assert i.error == swe.ERR_NUMERIC


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_land_beside_any_depth_is_land(swe, prec):
    """Cells with a LAND corner beside deep and negative ones raise nothing."""
    wl = _case(np.float64 if prec == "f64" else np.float32)
    wl.H[10:30:3, 5:50:4] = synth.LAND
    wl.H[10:30:3, 6:50:4] = 11000.0
    wl.H[11:30:3, 5:50:4] = -3.0
    with swe.Domain(wl, prec) as d:
        d.step(3)
        assert d.info().error == 0
        assert np.isfinite(d.state()[0]).all()
