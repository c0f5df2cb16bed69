"""The Kahan terms of the march arrive by asynchronous copies, a row ahead of
the row that uses them and into two slots that take turns. A column whose next
row is land must not leave a copy in flight when the slot is filled again: with
land scattered over the domain, columns that go in and out of land give the
bits, state and Kahan terms alike, of items of one row, whose columns fill a
slot once."""
import numpy as np
import pytest

from paper_1912_02457_gb300 import synth
from tests import helpers
from tests.test_gpu_parity import swe  # noqa: F401

pytestmark = pytest.mark.gpu


def _scattered(nx, ny, every):
    wl = helpers.rough(nx, ny, seed=nx + ny, land=False, min_depth=5.0, cd=0.002)
    rng = np.random.default_rng(nx * ny)
    # a LAND corner makes the (up to) four cells around it land
    wl.H[rng.random(wl.H.shape) < 1.0 / every] = synth.LAND
    wl.eta, wl.hu, wl.hv = helpers.random_state(wl, seed=5, amp=0.2, mom=0.5)
    return wl.astype(np.float32)


def _all(swe, d):
    return list(d.state()) + [d.read(k) for k in (swe.COMP_ETA, swe.COMP_HU, swe.COMP_HV)]


@pytest.mark.parametrize("every", [8, 25, 60])
@pytest.mark.parametrize("size", [(57, 64), (400, 330)])
def test_columns_with_scattered_land_agree_across_tilings(swe, size, every):
    wl = _scattered(*size, every)
    out = []
    for rows in (1, 64):
        with swe.Domain(wl, "f32_kahan") as d, swe.Batch() as b:
            b.add(d)
            b.set_rows(rows)
            b.step(9)
            b.sync()
            out.append(_all(swe, d))
    with swe.Domain(wl, "f32_kahan") as d:
        d.step(9)
        out.append(_all(swe, d))
    wet = ~wl.land_cells()
    assert np.isfinite(out[0][0][wet]).all() and out[0][3][wet].any()
    for got in out[1:]:
        for x, y in zip(got, out[0]):
            assert np.array_equal(x, y)
