"""The FP64 reciprocal and square root of the march give CUDA's correctly rounded
results, also where the argument's mantissa lies next to a power of two (an exact
value there is closest to the middle of two doubles)."""
import ctypes as C
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "swe_march.cuh"
namespace swe {
// out: results off by one spacing, by more; what 0: reciprocal, 1: square root
__global__ void compare(int what, unsigned long long seed, int per, unsigned long long *out) {
    unsigned long long s = seed + 0x9e3779b97f4a7c15ull * (blockIdx.x * blockDim.x + threadIdx.x + 1);
    for (int k = 0; k < per; k++) {
        s ^= s << 13; s ^= s >> 7; s ^= s << 17;
        unsigned long long m = s & 0xfffffffffffffull;
        // also mantissas next to a power of two, where spacings change
        if (k % 8 == 0) m &= 0xffull;
        if (k % 8 == 1) m |= 0xfffffffffff00ull;
        const long long e = 23 + (long long)((s >> 53) % 2000);
        const double x = __longlong_as_double((long long)(e << 52 | m));
        const double got = what ? sqrt_(x) : rcp_(x), want = what ? __dsqrt_rn(x) : __drcp_rn(x);
        const long long d = __double_as_longlong(got) - __double_as_longlong(want);
        if (d == 1 || d == -1) atomicAdd(out, 1ull);
        else if (d) atomicAdd(out + 1, 1ull);
        if (!what && rcp_(-x) != -got) atomicAdd(out + 1, 1ull);
    }
}
}  // namespace swe
extern "C" int swe_compare(int what, unsigned long long seed, int blocks, int per, unsigned long long *host) {
    unsigned long long *dev = nullptr;
    if (cudaMalloc(&dev, 16) != cudaSuccess) return 1;
    cudaMemset(dev, 0, 16);
    swe::compare<<<blocks, 256>>>(what, seed, per, dev);
    const int rc = cudaMemcpy(host, dev, 16, cudaMemcpyDeviceToHost) == cudaSuccess ? 0 : 2;
    cudaFree(dev);
    return rc;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1912_02457_gb300 import build
    d = tmp_path_factory.mktemp("f64")
    src, out = str(d / "f64.cu"), str(d / "f64.so")
    with open(src, "w") as fh:
        fh.write(SOURCE)
    r = subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-fmad=false", "-shared", "-cudart", "static",
                        src, "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    assert os.path.exists(out)
    return C.CDLL(out)


@pytest.mark.parametrize("what", [0, 1])
def test_rounding_of_reciprocal_and_root(lib, what):
    blocks, per = 1024, 128
    n = blocks * 256 * per
    off = (C.c_ulonglong * 2)()
    assert lib.swe_compare(what, C.c_ulonglong(12345 + what), blocks, per, off) == 0
    print(f"{'root' if what else 'reciprocal'}: {off[0]} of {n} off by one spacing, {off[1]} by more")
    assert off[0] == 0 and off[1] == 0
