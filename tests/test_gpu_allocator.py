"""Buffers of a caller's allocator: addresses on 8-byte boundaries only (cells
are vectors of 16 bytes), every one given back as it was handed out."""
import numpy as np
import pytest

from paper_1912_02457_gb300 import synth
from tests import helpers
from tests.test_gpu_parity import swe  # noqa: F401

pytestmark = pytest.mark.gpu


def _domain(dtype):
    wl = helpers.rough(61, 40, seed=9, land=True, min_depth=5.0, cd=0.002)
    wl.bc = (synth.BC_NESTED, synth.BC_NESTED, synth.BC_NESTED, synth.BC_WALL)
    wl.boundary = synth.still_boundary(61, 40, eta=0.05)
    wl.wind = helpers.gridded_wind(5, 4, seed=2)
    wl.eta, wl.hu, wl.hv = helpers.random_state(wl, seed=3, amp=0.2, mom=0.5)
    return wl.astype(dtype)


@pytest.mark.parametrize("offset", [0, 8])
@pytest.mark.parametrize("prec", ["f32", "f32_kahan", "f64"])
def test_addresses_on_eight_byte_boundaries(swe, prec, offset):
    import torch
    wl = _domain(np.float64 if prec == "f64" else np.float32)

    def run():
        with swe.Domain(wl, prec) as d:
            d.step(5)
            return list(d.state()) + [np.array(d.diagnostics())]

    want = run()
    live = {}

    def alloc(nbytes, stream, ctx):
        t = torch.empty(int(nbytes) + 16, dtype=torch.uint8, device="cuda")
        ptr = t.data_ptr() + offset
        live[ptr] = t
        return ptr

    def release(ptr, stream, ctx):
        del live[ptr]

    refs = (swe.ALLOC_FN(alloc), swe.FREE_FN(release))
    assert swe.load().swe_set_allocator(refs[0], refs[1], None) == 0
    try:
        got = run()
    finally:
        swe.use_default_allocator()
    assert not live
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
