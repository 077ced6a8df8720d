"""The device's reciprocal, quotient and root without a slow path against the general operations."""
import ctypes as C
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2604_13191_gb300 import _build  # noqa: E402

SOURCE = r"""
#include "vx_internal.cuh"
// every mantissa at one exponent
__global__ void k_unary(int exponent, unsigned long long* bad) {
    for (uint32_t m = blockIdx.x * blockDim.x + threadIdx.x; m < 1u << 23; m += gridDim.x * blockDim.x) {
        const float x = __uint_as_float(((uint32_t)(exponent + 127) << 23) | m);
        if (vx_rcp(x) != 1.0f / x) atomicAdd(bad, 1ull);
        if (vx_rcp(-x) != 1.0f / -x) atomicAdd(bad, 1ull);
        if (vx_sqrt(x) != sqrtf(x)) atomicAdd(bad + 1, 1ull);
    }
}
// quotients next to a midpoint: a 2^(k+1) - (2 n + 1) b = c with n of 24 bits, for every odd b and |c| <= 7
__global__ void k_quotient(int ea, int eb, unsigned long long* bad, unsigned long long* count) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < 1u << 22; i += gridDim.x * blockDim.x) {
        const unsigned long long b = (1ull << 23) + 2ull * i + 1ull;
        unsigned long long inv = b;
        for (int t = 0; t < 5; ++t) inv *= 2ull - b * inv;
        for (int k = 23; k <= 24; ++k)
            for (int c = -7; c <= 7; c += 2) {
                unsigned long long m = ((unsigned long long)(-(long long)c) * inv) & ((1ull << (k + 1)) - 1ull);
                if (k == 23) m |= 1ull << 24;
                if (m < 1ull << 24 || m >= 1ull << 25) continue;
                const long long a = (long long)(m * b + (unsigned long long)(long long)c) >> (k + 1);
                if (a < 1ll << 23 || a >= 1ll << 24) continue;
                const float fa = ldexpf((float)a, ea - 23), fb = ldexpf((float)b, eb - 23);
                if (vx_div(fa, fb) != fa / fb || vx_div(-fa, fb) != -fa / fb) atomicAdd(bad, 1ull);
                atomicAdd(count, 1ull);
            }
    }
}
extern "C" __attribute__((visibility("default"))) int check_unary(int exponent, unsigned long long* out) {
    k_unary<<<1024, 256>>>(exponent, out);
    return (int)cudaDeviceSynchronize();
}
extern "C" __attribute__((visibility("default"))) int check_quotient(int ea, int eb, unsigned long long* out) {
    k_quotient<<<1024, 256>>>(ea, eb, out, out + 1);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("arith")
    src, out = d / "arith.cu", d / "arith.so"
    src.write_text(SOURCE)
    cmd = [_build._nvcc(), *_build.ARCH, *_build.NVFLAGS, "-I", os.path.join(_build.ROOT, "include"), "-I", _build.CSRC,
           "-shared", str(src), "-o", str(out)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    so = C.CDLL(str(out))
    for f in (so.check_unary, so.check_quotient):
        f.restype = C.c_int
    so.check_unary.argtypes = [C.c_int, C.c_void_p]
    so.check_quotient.argtypes = [C.c_int, C.c_int, C.c_void_p]
    return so


@pytest.mark.parametrize("exponent", [-100, -67, -24, -2, -1, 0, 1, 2, 31, 64, 99])
def test_reciprocal_and_root_of_every_mantissa(lib, exponent):
    out = torch.zeros(2, dtype=torch.int64, device="cuda")
    assert lib.check_unary(exponent, out.data_ptr()) == 0
    assert out.tolist() == [0, 0]


@pytest.mark.parametrize("ea,eb", [(0, 0), (-80, 45), (-80, -100), (99, 99), (-20, 100), (126, 1)])
def test_quotients_next_to_a_midpoint(lib, ea, eb):
    """The pairs that a wrong rounding could come from (see test_host_arith.py), for every odd b, at the ends
    of the stated range: |a| >= 2^-80, |b| in [2^-100, 2^100], |a / b| normal."""
    out = torch.zeros(2, dtype=torch.int64, device="cuda")
    assert lib.check_quotient(ea, eb, out.data_ptr()) == 0
    bad, count = out.tolist()
    assert bad == 0 and count > 20_000_000
