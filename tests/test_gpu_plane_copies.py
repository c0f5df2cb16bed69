"""Fields to and from a cell's vector on planes of every shape: narrower than a
block, one cell past a power of two, more rows than a grid takes blocks of one."""
import numpy as np
import pytest

from tests import helpers
from tests.test_gpu_parity import swe  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 131), (7, 5), (8, 129), (9, 64), (33, 17), (255, 3), (256, 4), (257, 5),
                                   (3, 65536), (257, 65536), (65536, 2)])
@pytest.mark.parametrize("prec", ["f32_kahan", "f64"])
def test_fields_come_back_as_written(swe, prec, nx, ny):
    import torch
    wl = helpers.flat(nx, ny, dtype=np.float64 if prec == "f64" else np.float32)
    rng = np.random.default_rng(nx + ny)
    wl.eta, wl.hu, wl.hv = (rng.standard_normal((ny, nx)).astype(wl.H.dtype) for _ in range(3))
    with swe.Domain(wl, prec) as d:
        for a, b in zip(d.state(), (wl.eta, wl.hu, wl.hv)):
            assert np.array_equal(a, b)
        fields = [swe.ETA, swe.HV] + ([swe.COMP_HU] if prec == "f32_kahan" else [])
        for k in fields:
            new = rng.standard_normal((ny, nx)).astype(wl.H.dtype)
            src = torch.from_numpy(new).cuda()
            dst = torch.zeros(nx * ny + 8, dtype=src.dtype, device="cuda")
            d.write_device(k, src.data_ptr())
            d.read_device(k, dst.data_ptr())
            torch.cuda.synchronize()
            got = dst.cpu().numpy()
            assert np.array_equal(got[:nx * ny].reshape(ny, nx), new) and not got[nx * ny:].any()
            assert np.array_equal(d.read(k), new)
