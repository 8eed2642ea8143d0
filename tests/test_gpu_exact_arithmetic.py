"""mul_int and rcp_int return the bits of the FP64 product and reciprocal.

The results that do not depend on where a reactor is evaluated rest on this, and
a lost rounding would disappear in the gross-sum bounds of the parity tests.
"""
import subprocess

import pytest

from paper_1608_05794_gb300.build import ARCH, CSRC, INCLUDE, _nvcc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include <cuda_runtime.h>
#include "ck_common.cuh"
using namespace ck;

__device__ unsigned long long hash(unsigned long long x) {  // splitmix64
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}
// sign, biased exponent, 52-bit fraction
__device__ double make(unsigned s, unsigned e, unsigned long long f) {
  return __longlong_as_double((long long)(((unsigned long long)(s & 1) << 63) | ((unsigned long long)e << 52) |
                                          (f & 0xfffffffffffffull)));
}
__device__ unsigned long long edge(int i) {  // fractions where a rounding or a carry can go wrong
  const unsigned long long t = 0xfffffffffffffull;
  switch (i) {
    case 0: return 0;
    case 1: return 1;
    case 2: return 2;
    case 3: return 3;
    case 4: return t;
    case 5: return t - 1;
    case 6: return t - 2;
    case 7: return 0x8000000000000ull;
    case 8: return 0x7ffffffffffffull;
    case 9: return 0x8000000000001ull;
    case 10: return 0x6a09e667f3bccull;  // sqrt 2
    case 11: return 0x6a09e667f3bcdull;
    case 12: return 0x00000ffffffffull;
    case 13: return 0xfffff00000000ull;
    case 14: return 0x0000100000000ull;
    default: return 0x5555555555555ull;
  }
}
constexpr int EDGES = 16;

__device__ void check(double got, double want, unsigned long long* bad) {
  if (__double_as_longlong(got) != __double_as_longlong(want)) atomicAdd(bad, 1ull);
}

// kind 0: any fractions; 1: 27 by 27 bits, every second product a tie; 2: edges
__global__ void products(unsigned long long n, int kind, unsigned long long* bad) {
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned long long h = hash(2 * i), g = hash(2 * i + 1), w = hash(h ^ g);
    unsigned long long fa = h, fb = g;
    if (kind == 1) {
      fa = (h & 0xfffffffffffffull) & ~((1ull << 26) - 1) | (1ull << 26);
      fb = (g & 0xfffffffffffffull) & ~((1ull << 26) - 1) | (1ull << 26);
      if (w & 1) fb &= ~((1ull << 27) - 1);
    }
    if (kind == 2) {
      fa = edge(i % EDGES);
      fb = edge(i / EDGES % EDGES);
    }
    // exponents whose sum leaves the product a normal number
    const int ea = 1 + (int)((w >> 8) % 2046), lo = ea - 1023 < 0 ? -1022 - (ea - 1023) : -1022;
    const int hi = ea - 1023 > 0 ? 1022 - (ea - 1023) : 1022;
    const int eb = 1023 + lo + (int)((w >> 24) % (unsigned)(hi - lo + 1));
    if (eb < 1 || eb > 2046) continue;
    const double a = make((unsigned)(w >> 60), ea, fa), b = make((unsigned)(w >> 61), eb, fb), p = __dmul_rn(a, b);
    if (!isfinite(p)) continue;
    check(mul_int(a, b), p, bad);
    check(mul_int(b, a), p, bad);
  }
}
// every exponent; fractions at random (kind 0), near 1 and 2 (1), the edges (2)
__global__ void reciprocals(unsigned long long n, int kind, unsigned long long* bad) {
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned long long h = hash(i);
    unsigned long long f = h;
    if (kind == 1) f = h & 1 ? 0xfffffffffffffull - (i >> 12) % 100000 : (i >> 12) % 100000;
    if (kind == 2) f = edge((int)((i >> 12) % EDGES));
    const double x = make((unsigned)i, (unsigned)(i >> 1) & 2047, f);
    check(rcp_int(x), __drcp_rn(x), bad);
  }
}
int main() {
  unsigned long long* bad;
  if (cudaMallocManaged(&bad, 8) != cudaSuccess) return 2;
  for (int kind = 0; kind < 3; ++kind) {
    *bad = 0;
    products<<<1024, 256>>>(kind == 2 ? 1ull << 20 : 1ull << 26, kind, bad);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    std::printf("mul %d %llu\n", kind, *bad);
    *bad = 0;
    reciprocals<<<1024, 256>>>(kind == 2 ? (unsigned long long)EDGES << 12 : 1ull << 27, kind, bad);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    std::printf("rcp %d %llu\n", kind, *bad);
  }
}
"""


def test_integer_products_and_reciprocals_round_like_fp64(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    (tmp_path / "exact.cu").write_text(PROGRAM)
    subprocess.run([_nvcc(), *ARCH, "-O2", "-std=c++17", "-I", CSRC, "-I", INCLUDE, "--expt-relaxed-constexpr",
                    str(tmp_path / "exact.cu"), "-o", str(tmp_path / "exact")], check=True)
    out = subprocess.run([str(tmp_path / "exact")], capture_output=True, text=True, check=True).stdout
    assert out.split("\n")[:-1] == [f"{op} {kind} 0" for kind in range(3) for op in ("mul", "rcp")], out
