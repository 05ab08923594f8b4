"""The packed square root and quotient of exact_pair.cuh and the reciprocal of
shadow.cuh against the library's correctly rounded ones, on the device that
runs them: the root for every float of [2^-20, 2^64), the reciprocal for every
float, the quotient for 2^36 of the 2^46 pairs of mantissas (spread over all of
them) and for the mantissas at both ends against all others.

Run as a script it takes all 2^46 pairs (some minutes)."""
import ctypes
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "exact_pair.cuh"
#include "shadow.cuh"
using namespace nvc;
typedef unsigned long long u64;

__device__ void count(float got, float want, u64* bad) {
  const bool nan = got != got && want != want;
  if (!nan && __float_as_uint(got) != __float_as_uint(want)) atomicAdd(bad, 1ull);
}

__global__ void roots(u64 first, u64 n, u64* bad) {
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x) {
    const float x = __uint_as_float((uint32_t)(first + i));
    const float z = __uint_as_float((uint32_t)(first + (n - 1 - i)));
    const float2 s = xp::sqrt2_rn(make_float2(x, z), make_float2(-x, -z));
    count(s.x, __fsqrt_rn(x), bad);
    count(s.y, __fsqrt_rn(z), bad);
  }
}

__global__ void reciprocals(u64 first, u64 n, u64* bad) {
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x) {
    const float x = __uint_as_float((uint32_t)(first + i));
    count(rcp_rn(x), __fdiv_rn(1.0f, x), bad);
  }
}

// pair i of 2^46: an odd multiple modulo 2^46 visits all, and spreads a part
__global__ void quotients(u64 first, u64 n, u64* bad) {
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x) {
    const u64 j = ((first + i) * 0x1B873593A2C5ull) & ((1ull << 46) - 1);
    const float a = __uint_as_float(0x3F800000u | (uint32_t)(j & 0x7FFFFFu));
    const float b = __uint_as_float(0x3F800000u | (uint32_t)(j >> 23));
    const float2 q = xp::div2_rn(make_float2(a, 0.75f * a), make_float2(-b, -b));
    count(q.x, __fdiv_rn(a, b), bad);
    count(q.y, __fdiv_rn(0.75f * a, b), bad);
  }
}

// every numerator with the first and last 64 denominators
__global__ void ends(u64 first, u64 n, u64* bad) {
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x) {
    const uint32_t e = (uint32_t)((first + i) & 127u), m = e < 64 ? e : 0x800000u - (e - 63);
    const float a = __uint_as_float(0x3F800000u | (uint32_t)((first + i) >> 7));
    const float b = __uint_as_float(0x3F800000u | m);
    const float2 q = xp::div2_rn(make_float2(a, b), make_float2(-b, -a));
    count(q.x, __fdiv_rn(a, b), bad);
    count(q.y, __fdiv_rn(b, a), bad);
  }
}

extern "C" int run(int what, u64 first, u64 n, u64* bad) {
  const int blocks = 152 * 8;
  if (what == 0) roots<<<blocks, 256>>>(first, n, bad);
  if (what == 1) reciprocals<<<blocks, 256>>>(first, n, bad);
  if (what == 2) quotients<<<blocks, 256>>>(first, n, bad);
  if (what == 3) ends<<<blocks, 256>>>(first, n, bad);
  const int e = (int)cudaGetLastError();
  return e ? e : (int)cudaDeviceSynchronize();
}
"""

RANGES = {"root": (0, 0x35800000, 84 << 23), "reciprocal": (1, 0, 1 << 32),
          "quotient": (2, 0, 1 << 36), "quotient ends": (3, 0, 128 << 23)}


def _library(folder):
    from paper_2506_05930_gb300.build import ARCH, FLAGS, nvcc
    src, lib = os.path.join(folder, "check.cu"), os.path.join(folder, "check.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([nvcc(), *ARCH, *FLAGS, "-shared", src, "-o", lib], check=True)
    run = ctypes.CDLL(lib).run
    run.argtypes = [ctypes.c_int, ctypes.c_uint64, ctypes.c_uint64, ctypes.c_void_p]
    return run


def _wrong(run, what, first, n):
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert run(what, first, n, bad.data_ptr()) == 0
    return int(bad.item())


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    return _library(str(tmp_path_factory.mktemp("exact")))


@pytest.mark.parametrize("name", list(RANGES))
def test_correctly_rounded(run, name):
    assert _wrong(run, *RANGES[name]) == 0


if __name__ == "__main__":
    import tempfile
    import time
    sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    with tempfile.TemporaryDirectory() as folder:
        f, total, t0 = _library(folder), 0, time.time()
        for part in range(256):
            total += _wrong(f, 2, part << 38, 1 << 38)
        print(f"quotient: {total} wrong of 2^46 pairs of mantissas, {time.time() - t0:.0f} s")
        sys.exit(1 if total else 0)
