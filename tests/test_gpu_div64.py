"""The FP64 sweeps' quotients (csrc/div64.cuh) against IEEE division, bit by bit:
random mantissas, quotients next to the midpoint of two neighbouring values
(where a division is hardest to round: a 2^53 - m b = +-k for odd m and small k),
divisors near a power of two and near twice one, and exponents at and beyond
the range that is written out."""
import random
import subprocess

import numpy as np
import pytest

from paper_1004_1680_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "div64.cuh"
using namespace mhd;
__device__ double quotient(double a, double r) {
  return plain_divisor(r) && plain_exponent(a) ? ddiv_by(a, r, reciprocal(r)) : __ddiv_rn(a, r);
}
__device__ double limiter(double a, double b) {
  const double ab = __dmul_rn(a, b);
  return ab > 0.0 ? __ddiv_rn(ab, __dadd_rn(a, b)) : 0.0;
}
__device__ bool same(double x, double y) {
  return __double_as_longlong(x) == __double_as_longlong(y) || (x != x && y != y);
}
__global__ void pairs(const double* p, long long n, unsigned long long* bad) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double a = p[2 * i], b = p[2 * i + 1];
    if (!same(quotient(a, b), __ddiv_rn(a, b)) || !same(quotient(b, a), __ddiv_rn(b, a)) || !same(quotient(-a, b), __ddiv_rn(-a, b)))
      atomicAdd(bad, 1ull);
    if (!same(vl_half(a, b), limiter(a, b)) || !same(vl_half(-a, b), limiter(-a, b))) atomicAdd(bad + 1, 1ull);
  }
}
__device__ unsigned long long mix(unsigned long long x) {  // splitmix64 (Steele, Lea, Flood 2014)
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}
__global__ void randoms(int turns, unsigned long long* bad) {
  unsigned long long s = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) << 20;
  for (int t = 0; t < turns; t++) {
    const unsigned long long x = mix(s++), y = mix(s++);
    // mantissas in [1, 2); every fourth pair with exponents all over the place
    const unsigned long long m = (1ull << 52) - 1, one = 1023ull << 52;
    const double a = __longlong_as_double(t & 3 ? (x & m) | one : x & ~(1ull << 63));
    const double b = __longlong_as_double(t & 3 ? (y & m) | one : y & ~(1ull << 63));
    if (!same(quotient(a, b), __ddiv_rn(a, b))) atomicAdd(bad, 1ull);
    if (!same(vl_half(a, b), limiter(a, b))) atomicAdd(bad + 1, 1ull);
  }
}
int main(int argc, char** argv) {
  FILE* f = fopen(argv[1], "rb");
  const long long n = atoll(argv[2]);
  double* p;
  unsigned long long* bad;
  if (!f || cudaMallocManaged(&p, n * 16) || cudaMallocManaged(&bad, 16)) return 1;
  if (fread(p, 16, n, f) != (size_t)n) return 2;
  bad[0] = bad[1] = 0;
  pairs<<<152, 256>>>(p, n, bad);
  randoms<<<152 * 8, 256>>>(1000, bad);
  if (cudaDeviceSynchronize() != cudaSuccess) return 3;
  printf("%llu %llu\n", bad[0], bad[1]);
  return 0;
}
"""


def near_midpoints(count, rng):
    """Pairs (a, b) of 53-bit integers whose quotient, in [1, 2), lies k / (2^53 b)
    from a midpoint m / 2^53 (m odd, 54 bits)."""
    one = 1 << 53
    out = []
    while len(out) < count:
        kind = rng.randrange(3)
        if kind == 0:
            b = rng.randrange(1 << 52, one) | 1
        else:  # near twice a power of two, near a power of two
            d = rng.randrange(1, 1 << rng.randrange(2, 36)) | 1
            b = one - d if kind == 1 else (1 << 52) + d
        k = rng.choice([1, -1]) * (2 * rng.randrange(4) + 1) << rng.randrange(2)
        # a 2^53 = m b + k with m odd: k odd, or even for a doubled numerator
        m = -k * pow(b, -1, one) % one
        m += one
        if m % 2 == 0:
            continue
        a, rest = divmod(m * b + k, one)
        assert rest == 0
        while a % 2 == 0 and a >= one:
            a //= 2
        if a < one:
            out.append((float(a), float(b)))
    return out


def edges(rng):
    exps = [-1074, -1060, -1022, -1000, -501, -500, -499, -250, -1, 0, 1, 250, 499, 500, 501, 1000, 1023]
    mants = [1.0, 1.0 + 2.0 ** -52, 1.5, 2.0 - 2.0 ** -52, 2.0 - 2.0 ** -20, 2.0 - 2.0 ** -20 - 2.0 ** -52, 2.0 - 2.0 ** -21,
             2.0 - 2.0 ** -19, 1.0 + rng.random()]
    vals = [np.ldexp(m, e) for e in exps for m in mants] + [0.0, -0.0, np.inf, -np.inf, np.nan]
    return [(x, y) for x in vals for y in vals]


def test_quotients_are_ieee_division(tmp_path):
    rng = random.Random(17)
    data = np.array(near_midpoints(200000, rng) + edges(rng), dtype=np.float64)
    data.tofile(tmp_path / "pairs")
    (tmp_path / "div.cu").write_text(PROGRAM)
    exe = str(tmp_path / "div")
    subprocess.check_call([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I", build.CSRC, str(tmp_path / "div.cu"), "-o", exe])
    out = subprocess.run([exe, str(tmp_path / "pairs"), str(len(data))], check=True, capture_output=True, text=True).stdout
    assert out.split() == ["0", "0"]
