"""Device pointers at the state entry points: elements off their own boundary
(a field inside a packed record), which kernels cannot read, go through a copy;
and reads and writes of device memory can be captured into a CUDA graph."""
import ctypes as C

import numpy as np
import pytest

from tests import helpers
from tests.test_gpu_parity import swe  # noqa: F401

pytestmark = pytest.mark.gpu


def _case(prec):
    wl = helpers.rough(45, 31, seed=4, land=True, min_depth=5.0, cd=0.002)
    wl.eta, wl.hu, wl.hv = helpers.random_state(wl, seed=6, amp=0.2, mom=0.5)
    wl.f = np.full((31, 45), 1.2e-4) + 1e-6 * np.random.default_rng(1).random((31, 45))
    return wl.astype(np.float64 if prec == "f64" else np.float32)


def _room(a, off):
    """Device bytes holding `a` from byte `off` on."""
    import torch
    t = torch.zeros(a.nbytes + 16, dtype=torch.uint8, device="cuda")
    t[off:off + a.nbytes] = torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1).copy()).cuda()
    return t, t.data_ptr() + off


def _back(t, off, like):
    return t[off:off + like.nbytes].cpu().numpy().view(like.dtype).reshape(like.shape)


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("prec", ["f32", "f32_kahan", "f64"])
def test_elements_off_their_boundary(swe, prec, kernel):
    import torch
    wl = _case(prec)
    with swe.Domain(wl, prec, kernel=("fast", "reference")[kernel]) as d:
        d.step(3)
        want = d.state()
    L = swe.load()
    desc, p = swe.DomainDesc(), swe.params_from(wl.params, wl.t0, kernel)
    desc.nx, desc.ny, desc.dx, desc.dy, desc.precision = wl.nx, wl.ny, wl.dx, wl.dy, swe.PRECISIONS[prec]
    for k in range(4):
        desc.bc[k] = int(wl.bc[k])
    desc.f_const, desc.theta_const, desc.src_is_device = wl.f_const, wl.theta_const, 1
    keep = []
    for name in ("eta", "hu", "hv", "H", "f", "theta"):
        t, ptr = _room(getattr(wl, name), 2)
        keep.append(t)
        setattr(desc, name, ptr)
    h = C.c_void_p()
    swe._check(L.swe_create_domain(C.byref(desc), C.byref(p), None, C.byref(h)), "swe_create_domain")
    try:
        swe._check(L.swe_step(h, 3), "swe_step")
        out = np.empty_like(wl.eta)
        for k in range(3):
            swe._check(L.swe_read_state(h, k, out.ctypes.data, 0), "swe_read_state")
            assert np.array_equal(out, want[k])
        new = np.random.default_rng(2).standard_normal(wl.eta.shape).astype(wl.eta.dtype)
        fields = [swe.HU] + ([swe.COMP_HV] if prec == "f32_kahan" else [])
        for field in fields:
            t, ptr = _room(new, 3)
            swe._check(L.swe_write_state(h, field, C.c_void_p(ptr), 1), "swe_write_state")
            swe._check(L.swe_read_state(h, field, out.ctypes.data, 0), "swe_read_state")
            assert np.array_equal(out, new)
        if prec == "f32_kahan":
            t, ptr = _room(np.zeros_like(new), 1)
            swe._check(L.swe_read_state(h, swe.COMP_HV, C.c_void_p(ptr), 1), "swe_read_state")
            torch.cuda.synchronize()
            assert np.array_equal(_back(t, 1, new), new) and not t[:1].any() and not t[1 + new.nbytes:].any()
    finally:
        L.swe_destroy_domain(h)


def test_device_reads_and_writes_under_capture(swe):
    import torch
    wl = _case("f32")
    s = torch.cuda.Stream()
    src = torch.zeros((wl.ny, wl.nx), device="cuda")
    dst = torch.zeros_like(src)
    torch.cuda.synchronize()
    with swe.Domain(wl, "f32", stream=s.cuda_stream) as d:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            d.write_device(swe.HV, src.data_ptr())
            d.read_device(swe.HV, dst.data_ptr())
        for k in range(1, 3):
            src.fill_(float(k))
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            assert (dst == float(k)).all()
