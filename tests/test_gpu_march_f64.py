"""The march in FP64: work plans of one wave, whose items are packed into blocks of
equal work, against the oracle (the tolerance of the FP64 one-step checks)."""
import pytest

from tests import helpers
from tests.test_gpu_parity import swe  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(swe, oracle_mod, wl, steps):
    ref = oracle_mod.Oracle(wl).run(steps)
    with swe.Domain(wl, "f64") as d:
        d.step(steps)
        st = d.state()
    for a, b in zip(st, ref[:3]):
        assert helpers.rel(a, b) <= 1e-12


@pytest.mark.parametrize("nx,ny", [(401, 390), (600, 333), (450, 801)])
def test_balanced_plans_cover_every_row(swe, oracle_mod, nx, ny):
    wl = helpers.rough(nx, ny, seed=nx, land=True, min_depth=5.0, cd=0.002)
    wl.eta, wl.hu, wl.hv = helpers.random_state(wl, seed=ny, amp=0.2, mom=0.5)
    _check(swe, oracle_mod, wl, 2)
