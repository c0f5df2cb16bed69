"""The march in FP64: work plans of one wave, whose items are packed into blocks of
equal work, against the oracle (the tolerance of the FP64 one-step checks); the
strip edges and boundary kinds of the FP32 march; and its accesses under the bounds
checks."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from tests import helpers
from tests.test_gpu_march import SIZES, _domain
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


@pytest.mark.parametrize("kind", ["walls", "nested", "nested fine wind", "periodic"])
@pytest.mark.parametrize("size", SIZES)
def test_strip_edges_match_the_oracle(swe, oracle_mod, size, kind):
    """Within 32 spacings of the largest state component: the 16 of the FP32 march
    against an oracle of higher precision, twice, as here the oracle rounds alike."""
    wl = _domain(*size, kind).astype(np.float64)
    ref = oracle_mod.Oracle(wl).run(2)
    with swe.Domain(wl, "f64") as d:
        d.step(2)
        st = d.state()
    spacing = float(np.spacing(max(np.abs(r).max() for r in ref[:3])))
    assert max(np.abs(a - b).max() for a, b in zip(st, ref[:3])) <= 32 * spacing


def _bounds(**env):
    from paper_1912_02457_gb300 import build
    here = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, os.path.join(here, "bounds_cases_f64.py")],
                       env=dict(os.environ, SWE_LIBRARY=build.build_debug(), **env), capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_no_access_leaves_its_buffer():
    res = _bounds()
    assert len(res) >= 19
    bad = {k: v for k, v in res.items() if v[0] != 0}
    assert not bad, bad


def test_the_checks_catch_a_shrunk_extent():
    """A build told that the last row of every state plane is out of bounds (the
    allocation is untouched) reports it for every domain."""
    res = _bounds(SWE_DEBUG_SHRINK_PLANE_ROWS="1")
    assert all(v[0] == -6 and v[1] > 0 for v in res.values()), res
