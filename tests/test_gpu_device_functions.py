"""Device functions that replace conversions and square roots of the FP64 pipe by
other arithmetic, compiled by themselves and compared with what they replace:
every FP32 pattern, and square roots over the whole FP64 range."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1307_6720_gb300")

SOURCE = r"""
#include "device_util.cuh"
#include "df_bodies.cuh"

namespace {
__device__ unsigned long long bits(double d) { return (unsigned long long)__double_as_longlong(d); }

// all 2^32 patterns over the grid: bits that differ from the conversion's (NaN: any NaN)
__global__ void widen_kernel(unsigned long long* wrong) {
    unsigned long long n = 0;
    const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long q = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; q < (1ull << 32); q += step) {
        const float f = __uint_as_float(unsigned(q));
        const double a = mhs::df_widen(f), b = double(f);
        n += (a != a) ? (b == b) : bits(a) != bits(b);
    }
    if (n) atomicAdd(wrong, n);
}

// arguments m[i]: out[0] results that differ from sqrt's, out[1] the largest difference in units of the last place
__global__ void root_kernel(const double* m, long long n, unsigned long long* out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double a = mhs::sqrt_mid(m[i]), b = sqrt(m[i]);
        if (a != a && b != b) continue;
        const unsigned long long x = bits(a), y = bits(b), d = x > y ? x - y : y - x;
        if (d) {
            atomicAdd(out, 1ull);
            atomicMax(out + 1, d);
        }
    }
}
}  // namespace

extern "C" __attribute__((visibility("default"))) int widen_mismatches(unsigned long long* d) {
    widen_kernel<<<152 * 8, 256>>>(d);
    return int(cudaGetLastError());
}
extern "C" __attribute__((visibility("default"))) int root_mismatches(const double* m, long long n, unsigned long long* d) {
    root_kernel<<<152 * 8, 256>>>(m, n, d);
    return int(cudaGetLastError());
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch
    assert torch.cuda.is_available()
    from paper_1307_6720_gb300 import build
    d = tmp_path_factory.mktemp("devfn")
    src, so = d / "devfn.cu", d / "devfn.so"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), "-shared", "-o", str(so), str(src), "-I", os.path.join(PKG, "csrc"), "-I",
                    os.path.join(ROOT, "include")] + build.NVCC_FLAGS, check=True)
    lib = ctypes.CDLL(str(so))
    lib.widen_mismatches.argtypes = [ctypes.c_void_p]
    lib.root_mismatches.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_void_p]
    return lib


def test_widening_by_integer_operations_equals_the_conversion(lib):
    import torch
    out = torch.zeros(1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert lib.widen_mismatches(out.data_ptr()) == 0
    torch.cuda.synchronize()
    assert int(out[0]) == 0


def _roots(lib, m):
    import torch
    out = torch.zeros(2, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert lib.root_mismatches(m.data_ptr(), m.numel(), out.data_ptr()) == 0
    torch.cuda.synchronize()
    return int(out[0]), int(out[1])


def test_square_roots_are_correctly_rounded_but_for_ties(lib):
    """An error of 2^-80 before the last rounding changes the rounded value only
    within 2^-80 of a midpoint between doubles (2^-53 apart or more): in
    at most 2^-26 of the arguments, 4 of 2^28; 16 allowed, one unit each."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(1307)
    off = worst = 0
    for part in range(4):
        e = torch.randint(1023 - 99, 1023 + 99, (1 << 26,), generator=g, device="cuda", dtype=torch.int64)   # 1e-30 .. 1e30
        f = torch.randint(0, 1 << 52, (1 << 26,), generator=g, device="cuda", dtype=torch.int64)
        n, w = _roots(lib, ((e << 52) | f).view(torch.float64))
        off, worst = off + n, max(worst, w)
    assert off <= 16 and worst <= 1, (off, worst)


def test_square_roots_outside_the_fp32_range_are_the_library_s(lib):
    """0, -0, subnormals, both limits and their neighbours, squares of neighbouring
    doubles, infinities, NaN and negative arguments, and the whole exponent
    range: exact squares come out exact, and every value outside the limits
    equals sqrt's bit for bit."""
    import numpy as np
    import torch
    rng = np.random.default_rng(5)
    lim = [1e-30, 1e30]
    edge = [0.0, -0.0, 5e-324, 2.2250738585072014e-308, 1.7976931348623157e308, np.inf, -np.inf, np.nan, -1.0, -1e-40]
    for v in lim:
        edge += [v, np.nextafter(v, 0), np.nextafter(v, np.inf)]
    e = np.concatenate([np.arange(0, 1023 - 100), np.arange(1023 + 100, 2047)]).astype(np.uint64)
    far = ((e[:, None] << np.uint64(52)) | rng.integers(0, 1 << 52, (len(e), 256)).astype(np.uint64)).ravel().view(np.float64)
    r = rng.integers(1, 1 << 26, 1 << 20).astype(np.float64)   # 26-bit roots: exact squares
    for vals in (np.array(edge), far, r * r, (r * 2.0**-40) ** 2):
        assert _roots(lib, torch.from_numpy(vals).cuda()) == (0, 0)
