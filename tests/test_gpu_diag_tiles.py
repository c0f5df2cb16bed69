"""Mass and energy on both sides of the rule for the rows of a thread and at the
edges of its tiles: blocks of 32 columns by 16 or 64 rows.

Against the same sums without rounding (math.fsum). A sum passes through at most 8
additions in a thread, 5 in a warp, 8 in a block and, over the blocks, 1 in a
thread and 8 in the last block on these sizes; a term takes some ten roundings: 64
roundings of the sum of magnitudes."""
import math

import numpy as np
import pytest

from paper_1912_02457_gb300 import synth
from tests import helpers
from tests.test_gpu_parity import swe  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1, 1), (31, 15), (32, 16), (33, 17), (64, 63), (95, 65), (385, 769), (417, 833)])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_sums_match_exact_ones(swe, prec, nx, ny):
    dtype = np.float64 if prec == "f64" else np.float32
    wl = helpers.flat(nx, ny, dtype=dtype)
    rng = np.random.default_rng(nx * ny)
    wl.H = rng.uniform(-0.05, 40.0, (ny + 1, nx + 1)).astype(dtype)
    wl.H[rng.random(wl.H.shape) < 0.02] = synth.LAND
    wl.eta, wl.hu, wl.hv = (rng.standard_normal((ny, nx)).astype(dtype) for _ in range(3))
    with swe.Domain(wl, prec) as d:
        got = d.diagnostics()
    wet = ~wl.land_cells()
    H = wl.H.astype(np.float64)
    e, u, v = (a.astype(np.float64)[wet] for a in (wl.eta, wl.hu, wl.hv))
    h = np.abs(e + (0.25 * (H[:-1, :-1] + H[:-1, 1:] + H[1:, :-1] + H[1:, 1:]))[wet])
    kappa, g = float(dtype(1e-2)), float(dtype(9.81))
    hs = np.maximum(h, np.minimum(h * h / (2 * kappa) + 0.5 * kappa, kappa))
    energy = 0.5 * (u * u + v * v) / hs + 0.5 * g * e * e
    area = wl.dx * wl.dy
    for x, terms in zip(got, (e, energy)):
        assert abs(x - area * math.fsum(terms)) <= 64 * 2.0 ** -53 * area * math.fsum(np.abs(terms))
