"""The float32 reciprocal, quotient and root of the kernels equal the correctly rounded
operations bit for bit: 1/x and sqrt(x) over every value, quotients over 2^33 pairs of
significands and over those closest to a rounding boundary.  The float64 path divides: psi as
the Peng-Robinson pressure in two quotients gives it, and reciprocals of the entropic weights
equal to 1/x."""
import ctypes

import pytest

from device_ops import load

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbm_kernels.cuh"
using namespace lbm;
__device__ unsigned long long differ[5];
__device__ unsigned long long mix(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ unsigned long long halves;
__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b); }
__device__ bool same(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }
__device__ void count(int k, bool ok) { if (!ok) atomicAdd(&differ[k], 1ull); }
__global__ void every_value() {
  const unsigned step = gridDim.x * blockDim.x;
  for (unsigned long long b = blockIdx.x * blockDim.x + threadIdx.x; b <= 0x7f800000u; b += step) {
    const float x = __uint_as_float((unsigned)b);
    if (b >= 0x00800000u && b <= 0x7e800000u) {  // normal, and the reciprocal too
      count(0, same(rcp(x), 1.0f / x));
      count(0, same(rcp(-x), 1.0f / -x));
    }
    count(1, same(root(x), sqrtf(x)));
  }
}
__global__ void pairs(unsigned long long n) {
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += step) {
    const unsigned long long r = mix(i);
    const float a = __uint_as_float(0x3f800000u | (unsigned)(r & 0x7fffff));
    const float b = __uint_as_float(0x3f800000u | (unsigned)((r >> 24) & 0x7fffff));
    count(2, same(quotient(a, b), a / b));
  }
}
// x in (lo, hi) from the upper bits of r
__device__ double in(unsigned long long r, double lo, double hi) { return lo + (hi - lo) * ((double)(r >> 11) * 0x1p-53); }
__global__ void float64(unsigned long long n) {
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += step) {
    double x[9], r[9];
    for (int k = 0; k < 9; ++k) x[k] = in(mix(16 * i + k), k % 3 == 1 ? 0.4 : 0.05, k % 3 == 1 ? 0.8 : 0.4);
    weight_rcp<9>(x, r);
    for (int k = 0; k < 9; ++k) count(3, same(r[k], 1.0 / x[k]));
    DevDomain d;
    d.eos = 1;
    Phys<double>& p = d.pd;
    p.RT = in(mix(16 * i + 9), 0.003, 0.2);
    p.b = 0.095;
    p.aalpha = in(mix(16 * i + 10), 0.003, 1.0);
    p.band_lo = 0.1;
    p.band_hi = 9.0;
    const double rho = in(mix(16 * i + 11), 1e-3, 9.5);
    const double P = rho * p.RT / (1.0 - p.b * rho) - p.aalpha * rho * rho / (1.0 + 2.0 * p.b * rho - p.b * p.b * rho * rho);
    count(4, same(psi_of<double>(d, rho), sqrt(fabs(P - rho * (1.0 / 3.0)))));
  }
}
// the pairs whose quotient lies closest to half way between two floats: a 2^s = b m + k with m
// odd, of 25 bits, and |k| <= 4
__global__ void near_halves() {
  const unsigned step = gridDim.x * blockDim.x;
  for (unsigned b = 0x800000u + blockIdx.x * blockDim.x + threadIdx.x; b < 0x1000000u; b += step)
    for (int s = 24; s <= 25; ++s)
      for (int k = -4; k <= 4; ++k) {
        int e = 0;
        while (!(((b >> e) | (unsigned)(k >> e)) & 1u) && e < 3) ++e;
        const unsigned odd = b >> e, mod = (1u << (s - e)) - 1u;
        if (k == 0 || !(odd & 1u) || k != (k >> e) * (1 << e)) continue;
        unsigned inv = odd;
        for (int i = 0; i < 5; ++i) inv *= 2u - odd * inv;
        for (unsigned m = (inv * (unsigned)-(k >> e)) & mod; m < 0x2000000u; m += mod + 1u) {
          const long long a = ((long long)b * m + k) >> s;
          if (m < 0x1000000u || !(m & 1u) || a < 0x800000 || a >= 0x1000000 || (a << s) != (long long)b * m + k) continue;
          count(2, same(quotient((float)a, (float)b), (float)a / (float)b));
          atomicAdd(&halves, 1ull);
        }
      }
}
extern "C" int run(unsigned long long* out) {
  every_value<<<1216, 256>>>();
  pairs<<<1216, 256>>>(1ull << 33);
  near_halves<<<1216, 256>>>();
  float64<<<1216, 256>>>(1ull << 24);
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  unsigned long long n = 0;
  if (cudaMemcpyFromSymbol(&n, halves, sizeof(n)) != cudaSuccess || n < 1000000) return 2;
  return cudaMemcpyFromSymbol(out, differ, sizeof(differ)) != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def differ(tmp_path_factory):
    lib = load(str(tmp_path_factory.mktemp("ops")), SOURCE)
    out = (ctypes.c_ulonglong * 5)()
    assert lib.run(out) == 0
    return list(out)


@pytest.mark.parametrize("k,name", list(enumerate(["reciprocal", "root", "quotient", "weights64", "psi64"])))
def test_equal_to_the_rounded_operation(differ, k, name):
    assert differ[k] == 0, (name, differ)
