"""Iterations of the corner bathymetry overlap: the blocks of one start while
those of the one before it still run, and the two planes of corners change
places on every iteration. They must give the bits of iterations that run one
after the other (CUDA_LAUNCH_BLOCKING: every launch ends before the next), on
planes that leave room for the blocks of several iterations at once and on one
that takes more than a wave of them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))

CODE = """
import hashlib, sys
import torch
from paper_1912_02457_gb300 import swe
for nx, ny, n_iter in ((150, 90, 40), (700, 500, 40), (1501, 1203, 25), (4100, 4090, 12)):
    g = torch.Generator().manual_seed(nx)
    Hm = (torch.rand((ny, nx), generator=g) * 100.0).cuda()
    work = torch.empty(swe.bathymetry_work_bytes(nx, ny), dtype=torch.uint8, device="cuda")
    for stats in (False, True):
        Hc = torch.zeros((ny + 1, nx + 1), device="cuda")
        out = swe.bathymetry_reconstruct(Hm.data_ptr(), nx, nx, ny, Hc.data_ptr(), nx + 1, work.data_ptr(),
                                         n_iter=n_iter, stats=stats)
        torch.cuda.synchronize()
        h = hashlib.sha256(Hc.cpu().numpy().tobytes())
        if stats:
            h.update(out.tobytes())
        print(nx, ny, stats, h.hexdigest())
"""


def _run(**env):
    from paper_1912_02457_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", CODE], env=dict(os.environ, **env), cwd=os.path.dirname(HERE),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout.splitlines()


def test_overlapping_iterations_equal_separate_ones():
    together, apart = _run(), _run(CUDA_LAUNCH_BLOCKING="1")
    assert len(apart) == 8
    assert together == apart
