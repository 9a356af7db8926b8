// Reductions over the whole box and device-side step control:
//   - CFL signal rate (Section II.B: the fastest wave may cross at most a
//     fraction `cfl` of a cell per sweep): per-cell rate, warp-shuffle max,
//     one atomicMax per warp on the float bits (rates are >= 0, so the
//     unsigned order of the bits is the float order; invalid cells are +inf).
//   - the per-step control kernel that turns the rate into the sweep step
//     on the device, so a run of many steps needs no host round trip;
//   - FP64 diagnostics: compensated (Neumaier) sums of the 8 fields, the
//     max |div b| and the min pressure, reduced in a fixed order (bitwise
//     reproducible).
#include <cfloat>
#include <cstdint>

#include "fp32_sums.cuh"
#include "mhd_device.cuh"
#include "mhd_launch.h"

namespace mhd {

// COPY: also writes the fields to out (a state that arrives is copied and
// rated in one pass: 64 bytes per cell moved instead of 96, one launch instead
// of nine).
struct FieldCopy {
  float* out[8];
};
template <bool COPY>
__global__ void __launch_bounds__(256) cfl_rate_kernel(const float* __restrict__ rho, const float* __restrict__ mx,
                                                       const float* __restrict__ my, const float* __restrict__ mz,
                                                       const float* __restrict__ en, const float* __restrict__ bx,
                                                       const float* __restrict__ by, const float* __restrict__ bz,
                                                       Box box, float gamma, unsigned* rate, CellRange r, FieldCopy d) {
  // a warp walks whole x rows, 32 cells at a time; rows are stepped without
  // a division per row or cell (64-bit integer division is emulated)
  const int nx = box.n[0], ny = box.n[1], nz = box.n[2];
  const int lane = threadIdx.x & 31;
  const long long rows = (long long)ny * nz;
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  long long row = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  int j = (int)(row % ny);
  long long k = row / ny;
  const int dj = (int)(nwarps % ny);
  const long long dk = nwarps / ny;
  float rmax = 0.f;
  for (; row < rows; row += nwarps) {
    const bool rated = j >= r.lo[1] && j < r.hi[1] && k >= r.lo[2] && k < r.hi[2];
    if (rated || COPY) {
      const long long rowbase = j * box.stride[1] + k * box.stride[2];
      const long long yoff = (j + 1 < ny) ? box.stride[1] : -(long long)(ny - 1) * box.stride[1];
      const long long zoff = (k + 1 < nz) ? box.stride[2] : -(long long)(nz - 1) * box.stride[2];
#pragma unroll 2
      for (int i = (COPY ? 0 : r.lo[0]) + lane; i < (COPY ? nx : r.hi[0]); i += 32) {
        const long long c = rowbase + i;  // x is the contiguous axis (checked at launch)
        float m[3] = {__ldg(mx + c), __ldg(my + c), __ldg(mz + c)};
        const float b0 = __ldg(bx + c), b1 = __ldg(by + c), b2 = __ldg(bz + c);
        const float rr = __ldg(rho + c), ee = __ldg(en + c);
        float b[3];
        b[0] = 0.5f * (b0 + __ldg(bx + (i + 1 < nx ? c + 1 : c - (nx - 1))));
        b[1] = 0.5f * (b1 + __ldg(by + c + yoff));
        b[2] = 0.5f * (b2 + __ldg(bz + c + zoff));
        if constexpr (COPY) {
          d.out[RHO][c] = rr;
          d.out[MX][c] = m[0];
          d.out[MY][c] = m[1];
          d.out[MZ][c] = m[2];
          d.out[EN][c] = ee;
          d.out[BX][c] = b0;
          d.out[BY][c] = b1;
          d.out[BZ][c] = b2;
        }
        if (!COPY || (rated && i >= r.lo[0] && i < r.hi[0])) rmax = fmaxf(rmax, cell_rate(rr, m, ee, b, gamma, box.ih));
      }
    }
    j += dj;
    k += dk;
    if (j >= ny) {
      j -= ny;
      k++;
    }
  }
  for (int o = 16; o > 0; o >>= 1) rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
  if (lane == 0) atomicMax(rate, __float_as_uint(rmax));
}

cudaError_t launch_cfl_rate(const float* const f[8], const Box& box, float gamma, unsigned* rate,
                            cudaStream_t s, const CellRange* range, float* const copy[8]) {
  if (box.stride[0] != 1) return cudaErrorInvalidValue;
  const long long N = (long long)box.n[0] * box.n[1] * box.n[2];
  long long blocks = (N + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  CellRange r;
  for (int d = 0; d < 3; d++) {
    r.lo[d] = range ? range->lo[d] : 0;
    r.hi[d] = range ? range->hi[d] : box.n[d];
  }
  FieldCopy c = {};
  if (copy)
    for (int q = 0; q < 8; q++) c.out[q] = copy[q];
  auto* kernel = copy ? cfl_rate_kernel<true> : cfl_rate_kernel<false>;
  kernel<<<(unsigned)blocks, 256, 0, s>>>(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], box, gamma, rate, r, c);
  return cudaGetLastError();
}

// The 8 fields of N cells from one place on this device to another, in one
// launch (8 copies take 8 launches of about 2 us for a small box).  W = 4:
// 16-byte accesses (aligned fields).
template <int W>
__global__ void __launch_bounds__(256) copy_fields_kernel(const __grid_constant__ CopyArgs a, long long N) {
  const long long n = N / W;
  const long long step = (long long)gridDim.x * 256;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += step) {
    if constexpr (W == 4) {
      float4 v[8];
#pragma unroll
      for (int q = 0; q < 8; q++) v[q] = __ldg(reinterpret_cast<const float4*>(a.in[q]) + i);
#pragma unroll
      for (int q = 0; q < 8; q++) reinterpret_cast<float4*>(a.out[q])[i] = v[q];
    } else {
#pragma unroll
      for (int q = 0; q < 8; q++) a.out[q][i] = __ldg(a.in[q] + i);
    }
  }
  if (W == 4 && blockIdx.x == 0 && threadIdx.x < N % 4)
#pragma unroll
    for (int q = 0; q < 8; q++) a.out[q][n * 4 + threadIdx.x] = __ldg(a.in[q] + n * 4 + threadIdx.x);
}

cudaError_t launch_copy_fields(const float* const in[8], float* const out[8], long long N, cudaStream_t s) {
  CopyArgs a;
  bool vec = true;
  for (int q = 0; q < 8; q++) {
    a.in[q] = in[q];
    a.out[q] = out[q];
    vec = vec && reinterpret_cast<uintptr_t>(in[q]) % 16 == 0 && reinterpret_cast<uintptr_t>(out[q]) % 16 == 0;
  }
  const long long n = vec ? N / 4 : N;
  long long blocks = (n + 255) / 256;
  blocks = blocks < 1 ? 1 : (blocks > 152 * 8 ? 152 * 8 : blocks);
  if (vec) copy_fields_kernel<4><<<(unsigned)blocks, 256, 0, s>>>(a, N);
  else copy_fields_kernel<1><<<(unsigned)blocks, 256, 0, s>>>(a, N);
  return cudaGetLastError();
}

// Whether a kernel of the current device can copy between a box that lives on
// device `home` and the 8 fields directly (another device's memory, or the
// host's, goes through cudaMemcpyAsync).
bool local_fields(const void* const f[8], int home) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  return all_on_device(dev, home, [&](int q) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, f[q]) != cudaSuccess) {
      cudaGetLastError();
      return -1;
    }
    return at.type == cudaMemoryTypeDevice ? at.device : -1;
  });
}

__global__ void step_control_kernel(StepControl c) {
  wait_for_previous();
  step_begin(c, step_tau(c));
}

cudaError_t launch_step_control(const StepControl& c, int split, cudaStream_t s) {
  return launch_after(true, split, step_control_kernel, dim3(1), dim3(1), 0, s, c);
}

__global__ void ens_control_kernel(const unsigned* rate_cur, unsigned* rate_next, float* tau,
                                   double* time, int nbox, double cfl) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nbox) return;
  const float r = __uint_as_float(rate_cur[b]);
  const double t = (r > 0.f && r <= FLT_MAX) ? cfl / (double)r : 0.0;  // invalid state: stand still
  const float tf = (float)t;
  tau[b] = tf;
  time[b] += 2.0 * (double)tf;
  rate_next[b] = 0u;
}

cudaError_t launch_ens_control(const unsigned* rate_cur, unsigned* rate_next, float* tau,
                               double* time, int nbox, double cfl, cudaStream_t s) {
  ens_control_kernel<<<(nbox + 127) / 128, 128, 0, s>>>(rate_cur, rate_next, tau, time, nbox, cfl);
  return cudaGetLastError();
}

__global__ void set_tau_kernel(float* tau, float value) { *tau = value; }

cudaError_t launch_set_tau(float* tau, double value, cudaStream_t s) {
  set_tau_kernel<<<1, 1, 0, s>>>(tau, (float)value);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP64 compensated sums (Neumaier): a value is the pair (s, c), total s + c.

struct KB {
  double s, c;
};

__device__ __forceinline__ KB kb_merge(KB a, KB b) {
  const double t = a.s + b.s;
  const double err = (fabs(a.s) >= fabs(b.s)) ? (a.s - t) + b.s : (b.s - t) + a.s;
  return KB{t, a.c + b.c + err};
}

constexpr int kDiagThreads = 256;

// Order-preserving integer image of a float (atomic minima and maxima).
__device__ __forceinline__ int float_key(float x) {
  const int i = __float_as_int(x);
  return i < 0 ? i ^ 0x7fffffff : i;
}
__device__ __forceinline__ float key_float(int k) { return __int_as_float(k < 0 ? k ^ 0x7fffffff : k); }

// The FP64 values of one cell (the formulas the diagnostics define), out of
// line: the filters below reach them for a few cells only.
__device__ __noinline__ double cell_div64(float bxl, float bxh, float byl, float byh, float bzl, float bzh,
                                          int nx, int ny, int nz) {
  return ((double)bxh - bxl) * nx + ((double)byh - byl) * ny + ((double)bzh - bzl) * nz;
}

__device__ __noinline__ double cell_p64(float rho, float m1, float m2, float m3, float e, float bxl,
                                        float bxh, float byl, float byh, float bzl, float bzh, double gamma) {
  const double b0 = 0.5 * ((double)bxl + bxh), b1 = 0.5 * ((double)byl + byh), b2 = 0.5 * ((double)bzl + bzh);
  const double kin = 0.5 * ((double)m1 * m1 + (double)m2 * m2 + (double)m3 * m3) / rho;
  return (gamma - 1.0) * ((double)e - kin - 0.5 * (b0 * b0 + b1 * b1 + b2 * b2));
}

// Float-float estimate of |div b| of two cells on packed FP32.  Each difference
// is exact (TwoSum), times n_d (product error by FMA), summed by TwoSum: the
// estimate is within 2^-44 dT of div, dT = sum |(b_high - b_low) n_d|; err
// covers it with a margin of 16.  (An FP32 estimate in front rules nothing
// out: the field is divergence-free up to rounding, so max |div b| is of the
// size of that estimate's own error.)
__device__ __forceinline__ void div_ff2(float2 xl, float2 xh, float2 yl, float2 yh, float2 zl, float2 zh, float2 nx,
                                        float2 ny, float2 nz, float2& dabs, float2& err, float2& dT) {
  float2 s0, e0, s1, e1, s2, e2;
  two_sum2(xh, neg2(xl), s0, e0);
  two_sum2(yh, neg2(yl), s1, e1);
  two_sum2(zh, neg2(zl), s2, e2);
  const float2 p0 = __fmul2_rn(s0, nx), p1 = __fmul2_rn(s1, ny), p2 = __fmul2_rn(s2, nz);
  const float2 q0 = __ffma2_rn(s0, nx, neg2(p0)), q1 = __ffma2_rn(s1, ny, neg2(p1)), q2 = __ffma2_rn(s2, nz, neg2(p2));
  float2 h01, r01, dh, r2;
  two_sum2(p0, p1, h01, r01);
  two_sum2(h01, p2, dh, r2);
  float2 dl = __fadd2_rn(__fadd2_rn(q0, q1), q2);
  dl = __ffma2_rn(e0, nx, __ffma2_rn(e1, ny, __ffma2_rn(e2, nz, dl)));
  dl = __fadd2_rn(dl, __fadd2_rn(r01, r2));
  const float2 d = __fadd2_rn(dh, dl);
  dabs = make_float2(fabsf(d.x), fabsf(d.y));
  dT = make_float2(fabsf(p0.x) + fabsf(p1.x) + fabsf(p2.x), fabsf(p0.y) + fabsf(p1.y) + fabsf(p2.y));
  err = __ffma2_rn(f2(0x1p-22f), dabs, __ffma2_rn(f2(0x1p-40f), dT, f2(1e-37f)));
}

// What an estimate of p may lose to underflow: the momenta's squares and their
// error words, a dozen terms that may each be off by 2^-149, over rho (at densities
// and momenta of 1e-25 that is most of p), and the other terms.
__device__ __forceinline__ float2 underflow2(float2 rr, float g_hi) {
  return __ffma2_rn(f2(0x1p-142f * g_hi), abs2(rr), f2(1e-37f));
}

// Float-float estimate ph + pl of the pressure of two cells on packed FP32,
// within 2^-42 (gamma - 1) U of p (U below) and what underflows (underflow2); err
// covers it with a margin of 16.  rr: an approximate reciprocal of rho.
__device__ __forceinline__ void p_ff2(float2 rho, float2 m1, float2 m2, float2 m3, float2 e, float2 xl, float2 xh,
                                      float2 yl, float2 yh, float2 zl, float2 zh, float2 rr, float g_hi, float g_lo,
                                      float2 U, float2& ph, float2& pl, float2& err) {
  float2 a0, ae0, a1, ae1, a2, ae2, sa, ra, sh, rb;
  two_prod2(m1, m1, a0, ae0);
  two_prod2(m2, m2, a1, ae1);
  two_prod2(m3, m3, a2, ae2);
  two_sum2(a0, a1, sa, ra);
  two_sum2(sa, a2, sh, rb);
  const float2 sl = __fadd2_rn(__fadd2_rn(__fadd2_rn(ae0, ae1), ae2), __fadd2_rn(ra, rb));
  // k1 within a few ulp of S / rho; the FMA remainder S - k1 rho corrects it
  // to about 2^-43 S / rho
  const float2 k1 = __fmul2_rn(sh, rr);
  const float2 k2 = __fmul2_rn(__fadd2_rn(__ffma2_rn(neg2(k1), rho, sh), sl), rr);  // kin = (k1 + k2) / 2
  float2 c0h, c0l, c1h, c1l, c2h, c2l;
  two_sum2(xl, xh, c0h, c0l);
  two_sum2(yl, yh, c1h, c1l);
  two_sum2(zl, zh, c2h, c2l);  // 2 b_c = c_h + c_l exactly
  float2 w0, we0, w1, we1, w2, we2, sw, rw, mh, rm;
  two_prod2(c0h, c0h, w0, we0);
  two_prod2(c1h, c1h, w1, we1);
  two_prod2(c2h, c2h, w2, we2);
  we0 = __ffma2_rn(__fadd2_rn(c0h, c0h), c0l, we0);
  we1 = __ffma2_rn(__fadd2_rn(c1h, c1h), c1l, we1);
  we2 = __ffma2_rn(__fadd2_rn(c2h, c2h), c2l, we2);
  two_sum2(w0, w1, sw, rw);
  two_sum2(sw, w2, mh, rm);  // 4 |b_c|^2 = mh + ml
  const float2 ml = __fadd2_rn(__fadd2_rn(__fadd2_rn(we0, we1), we2), __fadd2_rn(rw, rm));
  float2 d1, de1, d2, de2;
  two_sum2(e, __fmul2_rn(f2(-0.5f), k1), d1, de1);
  two_sum2(d1, __fmul2_rn(f2(-0.125f), mh), d2, de2);
  float2 dlo = __ffma2_rn(f2(-0.5f), k2, __fadd2_rn(de1, de2));
  dlo = __ffma2_rn(f2(-0.125f), ml, dlo);
  float2 phe;
  two_prod2(f2(g_hi), d2, ph, phe);
  pl = __fadd2_rn(phe, __ffma2_rn(f2(g_hi), dlo, __fmul2_rn(f2(g_lo), d2)));
  err = __ffma2_rn(f2(0x1p-38f * g_hi), U, underflow2(rr, g_hi));
}

// n / d for 0 <= n < 2^31 by a multiplication: the quotient rounded down (Granlund
// and Montgomery, "Division by invariant integers using multiplication", 1994).
struct FastDiv {
  unsigned mul, shift, d;
};
FastDiv fast_div(unsigned d) {
  FastDiv f{0, 0, d};
  while ((1ull << f.shift) < d) f.shift++;
  f.mul = (unsigned)(((1ull << 32) * ((1ull << f.shift) - d)) / d + 1);
  return f;
}
__device__ __forceinline__ unsigned quotient(unsigned n, const FastDiv& f) {
  return (unsigned)(((unsigned long long)__umulhi(n, f.mul) + n) >> f.shift);
}

// One pass over the box: the compensated sums of the 8 fields, max |div b|
// (the face differences of each cell) and min p, in FP64 as defined by the
// formulas above.  The extrema are exact FP64 values of those formulas: a
// cell's FP64 value is only evaluated when an estimate with an error bound
// (and a margin of 4 or more) does not rule it out against the running
// extremum.  The estimates sit behind warp votes, a warp's lanes share their
// new thresholds right after, and the block's warps share theirs through
// shared memory (a threshold only rules cells out, so the extrema do not
// depend on when it arrives).
//
// A lane takes W = 2 consecutive cells per turn (8-byte loads; nx even and
// aligned fields) or one, and every operation runs on two cells at once (packed
// FP32; with 4 cells the windows and values spill).  At 256^3, pressures
// tied to FP32 rounding (a uniform initial pressure: every cell takes the
// float-float estimate): 381 -> 255 us, 431 -> 288 instructions per cell,
// and 512^3 of evolved turbulence 2.12 -> 1.63 ms with the final reduction.
// Instruction issue and its latencies at 16 warps per SM bound it.  An FP64
// instruction occupies an SM's pipe for 16 cycles a warp, so the grid is what
// fits at once (2 blocks per SM: few blocks meet their extremum from
// nothing), thresholds come from the estimates, the lowest pressure of a lane
// is evaluated once at the end, and FP64 sums appear once per block or window.
template <int W>
__global__ void __launch_bounds__(kDiagThreads, 2)
diag_partial_kernel(const float* __restrict__ rho, const float* __restrict__ mx,
                    const float* __restrict__ my, const float* __restrict__ mz,
                    const float* __restrict__ en, const float* __restrict__ bx,
                    const float* __restrict__ by, const float* __restrict__ bz, int nx, int ny, int nz,
                    FastDiv row_div, FastDiv ny_div, double gamma, double* __restrict__ partial) {
  const float* f[8] = {rho, mx, my, mz, en, bx, by, bz};
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __shared__ int sh_p, sh_div;  // the block's thresholds (float_key)
  __shared__ double sacc[kDiagThreads / 32][8];
  __shared__ float2 sw[kDiagThreads / 32][8][3];
  __shared__ double sx[kDiagThreads / 32][2];
  FWin2 win[8];
#pragma unroll
  for (int q = 0; q < 8; q++) win[q].h = win[q].l = win[q].t = f2(0.f);
  double divmax = 0.0, pmin = DBL_MAX;
  float best_h = 3e38f, best_l = 0.f, best_e = 0.f;       // the lane's lowest pressure so far, to be evaluated at the end
  unsigned best_c = 0;
  float div_thr = 0.f;                                    // <= the block's running max |div b|
  float pt_hi = __int_as_float(0x7f800000), pt_lo = 0.f;  // >= the block's running min p
  const float2 n0 = f2((float)nx), n1 = f2((float)ny), n2 = f2((float)nz);
  const float g_hi = (float)(gamma - 1.0), g_lo = (float)((gamma - 1.0) - (double)g_hi);
  if (threadIdx.x == 0) {
    sh_p = float_key(pt_hi);
    sh_div = float_key(0.f);
  }
  if (lane == 0)
    for (int q = 0; q < 8; q++) sacc[wid][q] = 0.0;
  __syncthreads();
  const unsigned rowlen = (unsigned)nx / W;            // turns of a row
  const unsigned turns = rowlen * (unsigned)ny * (unsigned)nz;  // < 2^31
  const unsigned plane = (unsigned)nx * (unsigned)ny;
  bool seeded = false;
  int it = 0;
  // a warp's window words into its FP64 accumulators
  auto flush = [&] {
#pragma unroll
    for (int q = 0; q < 8; q++) {
      double a0 = 0.0, a1 = 0.0;
      fwin_flush(win[q], a0, a1);
      a0 += a1;
      for (int o = 16; o > 0; o >>= 1) a0 += __shfl_xor_sync(0xffffffffu, a0, o);
      if (lane == 0) sacc[wid][q] += a0;
    }
  };
  for (unsigned base = (blockIdx.x * kDiagThreads + wid * 32); base < turns; base += gridDim.x * kDiagThreads) {
    const unsigned g = min(base + lane, turns - 1);
    const bool valid = base + lane < turns;
    const unsigned row = quotient(g, row_div), i = (g - row * rowlen) * W, k = quotient(row, ny_div), j = row - k * ny;
    const unsigned c = row * (unsigned)nx + i;
    const unsigned cy = j + 1 == (unsigned)ny ? c - (unsigned)(ny - 1) * nx : c + nx;
    const unsigned cz = k + 1 == (unsigned)nz ? c - (unsigned)(nz - 1) * plane : c + plane;
    float v[8][2], hy[2], hz[2];
    auto load = [&](const float* p, float (&d)[2]) {
      if constexpr (W == 2) {
        const float2 x = __ldg(reinterpret_cast<const float2*>(p));
        d[0] = x.x, d[1] = x.y;
      } else {
        d[0] = __ldg(p);
        d[1] = 0.f;
      }
    };
#pragma unroll
    for (int q = 0; q < 8; q++) load(f[q] + c, v[q]);
    load(by + cy, hy);
    load(bz + cz, hz);
    const float bx_next = __ldg(bx + (i + W == (unsigned)nx ? c - i : c + W));
    if (!valid)
#pragma unroll
      for (int q = 0; q < 8; q++)
        v[q][0] = v[q][1] = 0.f;
#pragma unroll
    for (int q = 0; q < 8; q++) fwin_add(win[q], make_float2(v[q][0], v[q][1]));
    // high x face of cell e
    auto hx = [&](int e) { return e + 1 < W ? v[5][1] : bx_next; };
    auto pair = [&](int q) { return make_float2(v[q][0], v[q][1]); };
    const float2 xh = make_float2(hx(0), hx(1)), yh = make_float2(hy[0], hy[1]), zh = make_float2(hz[0], hz[1]);
    // thresholds that other warps have found since
    div_thr = fmaxf(div_thr, key_float(*reinterpret_cast<volatile int*>(&sh_div)));
    {
      const float sp = key_float(*reinterpret_cast<volatile int*>(&sh_p));
      if (sp < pt_hi) {
        pt_hi = sp;
        pt_lo = 0.f;
      }
    }
    // p = (gamma - 1)(e - |m|^2 / (2 rho) - |b_c|^2 / 2), U = |e| + |kin| +
    // sum ((|b| + |b_high|) / 2)^2 / 2.  FP32: |error| <= 2^-19 (gamma - 1) U.
    float2 dabs, derr, dT;
    div_ff2(pair(5), xh, pair(6), yh, pair(7), zh, n0, n1, n2, dabs, derr, dT);
    const float2 rr = make_float2(fast_rcp(v[0][0]), fast_rcp(v[0][1]));
    const float2 kin = __fmul2_rn(__ffma2_rn(pair(1), pair(1), __ffma2_rn(pair(2), pair(2), __fmul2_rn(pair(3), pair(3)))),
                                  __fmul2_rn(f2(0.5f), rr));
    const float2 bc0 = __fadd2_rn(pair(5), xh), bc1 = __fadd2_rn(pair(6), yh), bc2 = __fadd2_rn(pair(7), zh);  // 2 b_c
    const float2 b2 = __ffma2_rn(bc0, bc0, __ffma2_rn(bc1, bc1, __fmul2_rn(bc2, bc2)));
    const float2 a0 = __fadd2_rn(abs2(pair(5)), abs2(xh)), a1 = __fadd2_rn(abs2(pair(6)), abs2(yh)),
                 a2 = __fadd2_rn(abs2(pair(7)), abs2(zh));
    const float2 U = __ffma2_rn(f2(0.125f), __ffma2_rn(a0, a0, __ffma2_rn(a1, a1, __fmul2_rn(a2, a2))),
                                __fadd2_rn(abs2(pair(4)), abs2(kin)));
    const float2 perr = __ffma2_rn(f2(0x1p-17f * g_hi), U, underflow2(rr, g_hi));
    const float2 p32 = __fmul2_rn(f2(g_hi), sub2(__ffma2_rn(f2(-0.125f), b2, pair(4)), kin));
    auto el = [](const float2& x, int e) { return e & 1 ? x.y : x.x; };
    if (!seeded) {  // the block's first thresholds
      seeded = true;
#pragma unroll
      for (int e = 0; e < W; e++) {
        const float lo = el(dabs, e) - el(derr, e), hi = el(p32, e) + el(perr, e);
        if (valid && lo > div_thr && lo < 3e38f) div_thr = lo;
        if (valid && hi < pt_hi && fabsf(hi) < 3e38f) pt_hi = hi, pt_lo = 0.f;
      }
      if (div_thr > 0.f) atomicMax(&sh_div, float_key(div_thr));
      if (fabsf(pt_hi) < 3e38f) atomicMin(&sh_p, float_key(pt_hi));
      __syncwarp();
      div_thr = key_float(*reinterpret_cast<volatile int*>(&sh_div));
      pt_hi = key_float(*reinterpret_cast<volatile int*>(&sh_p));
    }
    // cells that the estimates do not rule out; a NaN always goes on, and a
    // cell whose three differences are zero (uniform fields) has div b = 0
    const float pt_up = pt_hi + (pt_lo + 0x1p-22f * fabsf(pt_hi));  // >= the threshold, rounded
    unsigned cd = 0, cp = 0;
#pragma unroll
    for (int e = 0; e < W; e++) {
      if (valid && el(dT, e) != 0.f && !(el(dabs, e) + el(derr, e) < div_thr)) cd |= 1u << e;
      if (valid && !(__fsub_rn(el(p32, e), el(perr, e)) > pt_up)) cp |= 1u << e;
    }
    if (__any_sync(0xffffffffu, cd != 0)) {
#pragma unroll
      for (int e = 0; e < W; e++) {
        if (cd >> e & 1) {
          const double div = cell_div64(v[5][e], hx(e), v[6][e], hy[e], v[7][e], hz[e], nx, ny, nz);
          divmax = fmax(divmax, fabs(div));
          div_thr = fmaxf(div_thr, __double2float_rd(divmax));
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) div_thr = fmaxf(div_thr, __shfl_xor_sync(0xffffffffu, div_thr, o));
      if (lane == 0) atomicMax(&sh_div, float_key(div_thr));
    }
    if (__any_sync(0xffffffffu, cp != 0)) {
      float2 ph, pl, pe;
      p_ff2(pair(0), pair(1), pair(2), pair(3), pair(4), pair(5), xh, pair(6), yh, pair(7), zh, rr, g_hi, g_lo, U, ph, pl,
            pe);
      // new upper bounds of the minimum: over the lane's cells, then the warp
      bool lower = false;
#pragma unroll
      for (int e = 0; e < W; e++) {
        const float h = el(ph, e), l = __fadd_ru(el(pl, e), el(pe, e));
        if ((cp >> e & 1) && fabsf(h) < 1e38f && !(__fadd_rn(__fsub_rn(h, pt_hi), __fsub_rn(l, pt_lo)) >= 0.f)) {
          pt_hi = h;
          pt_lo = l;
          lower = true;
        }
      }
      if (__any_sync(0xffffffffu, lower)) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const float oh = __shfl_xor_sync(0xffffffffu, pt_hi, o), ol = __shfl_xor_sync(0xffffffffu, pt_lo, o);
          if (__fadd_rn(__fsub_rn(oh, pt_hi), __fsub_rn(ol, pt_lo)) < 0.f) {
            pt_hi = oh;
            pt_lo = ol;
          }
        }
        if (lane == 0 && fabsf(pt_hi) < 1e38f) atomicMin(&sh_p, float_key(__fadd_ru(pt_hi, pt_lo)));
      }
      // candidates against the new bound: the lane keeps the lowest one for the
      // end (its FP64 value is needed only if it still stands then); one that
      // cannot be told from it, or that FP32 cannot hold, is evaluated now
#pragma unroll
      for (int e = 0; e < W; e++) {
        const float h = el(ph, e), l = el(pl, e), er = el(pe, e);
        const bool far = !(fabsf(h) < 1e38f) || !(fabsf(er) < 1e38f);
        if ((cp >> e & 1) && (far || !(__fadd_rn(__fsub_rn(h, pt_hi), __fsub_rn(__fsub_rn(l, pt_lo), er)) > 0.f))) {
          const float diff = __fadd_rn(__fsub_rn(h, best_h), __fsub_rn(l, best_l)), tol = 1.125f * (er + best_e);
          if (!far && diff < -tol) {
            best_h = h;
            best_l = l;
            best_e = er;
            best_c = c + e;
          } else if (far || !(diff > tol)) {
            pmin = fmin(pmin, cell_p64(v[0][e], v[1][e], v[2][e], v[3][e], v[4][e], v[5][e], hx(e), v[6][e], hy[e],
                                       v[7][e], hz[e], gamma));
          }
        }
      }
    }
    if (++it == kWin) {
      it = 0;
      flush();
    }
  }
  // the lanes' kept candidates that the block's final threshold leaves
  __syncthreads();
  {
    const float sp = key_float(sh_p);
    if (best_h < 3e38f && !(best_h + (best_l - best_e) - 0x1p-22f * fabsf(best_h) > sp)) {
      const unsigned c = best_c, row = c / (unsigned)nx, i = c - row * nx, k = row / (unsigned)ny, j = row - k * ny;
      const unsigned cx = i + 1 == (unsigned)nx ? c - i : c + 1;
      const unsigned cy = j + 1 == (unsigned)ny ? c - (unsigned)(ny - 1) * nx : c + nx;
      const unsigned cz = k + 1 == (unsigned)nz ? c - (unsigned)(nz - 1) * plane : c + plane;
      pmin = fmin(pmin, cell_p64(rho[c], mx[c], my[c], mz[c], en[c], bx[c], bx[cx], by[c], by[cy], bz[c], bz[cz], gamma));
    }
  }
  // windows whose block total could leave FP32's range go on in FP64
  bool large = false;
#pragma unroll
  for (int q = 0; q < 8; q++) large = large || !(fabsf(win[q].h.x) + fabsf(win[q].h.y) < 1e35f);
  if (__syncthreads_or(large)) flush();
  // the block's totals in a fixed order: the words over the lanes by a shuffle
  // tree and over the warps in order, in FP32, then in FP64 with the windows
  // flushed before; one warp per extremum
#pragma unroll
  for (int q = 0; q < 8; q++) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) fwin_merge(win[q], shfl_down2(win[q].h, o), shfl_down2(win[q].l, o), shfl_down2(win[q].t, o));
    if (lane == 0) {
      sw[wid][q][0] = win[q].h;
      sw[wid][q][1] = win[q].l;
      sw[wid][q][2] = win[q].t;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    divmax = fmax(divmax, __shfl_down_sync(0xffffffffu, divmax, o));
    pmin = fmin(pmin, __shfl_down_sync(0xffffffffu, pmin, o));
  }
  if (lane == 0) {
    sx[wid][0] = divmax;
    sx[wid][1] = pmin;
  }
  __syncthreads();
  double* out = partial + (long long)blockIdx.x * kDiagSlots;
  if (threadIdx.x < 8) {
    const int q = threadIdx.x;
    FWin2 t{sw[0][q][0], sw[0][q][1], sw[0][q][2]};
    for (int w = 1; w < kDiagThreads / 32; w++) fwin_merge(t, sw[w][q][0], sw[w][q][1], sw[w][q][2]);
    double a0 = 0.0, a1 = 0.0;
    fwin_flush(t, a0, a1);
    KB s{a0 + a1, 0.0};
    for (int w = 0; w < kDiagThreads / 32; w++) s = kb_merge(s, KB{sacc[w][q], 0.0});
    out[2 * q] = s.s;
    out[2 * q + 1] = s.c;
  } else if (threadIdx.x == 32) {
    double m = sx[0][0];
    for (int w = 1; w < kDiagThreads / 32; w++) m = fmax(m, sx[w][0]);
    out[16] = m;
  } else if (threadIdx.x == 64) {
    double m = sx[0][1];
    for (int w = 1; w < kDiagThreads / 32; w++) m = fmin(m, sx[w][1]);
    out[17] = m;
  }
}

// The blocks' partials in a fixed order: a block per quantity, each lane
// merging every 96th partial (with compensation for the sums), then the lanes
// by a shuffle tree and the 3 warps in order.  (One lane per quantity over 1216
// partials took 537 us, a chain of dependent FP64 operations; all quantities
// on one SM are bound by its FP64 pipe, 23 us.)
constexpr int kFinalWarps = 3;
__global__ void __launch_bounds__(32 * kFinalWarps)
diag_final_kernel(const double* __restrict__ partial, int nblk, double hmin, double* __restrict__ out) {
  __shared__ double sm[kFinalWarps][2];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, q = blockIdx.x;
  KB t{0.0, 0.0};
  double m = q == 9 ? DBL_MAX : 0.0;
  for (int b = threadIdx.x; b < nblk; b += 32 * kFinalWarps) {
    const double* p = partial + (long long)b * kDiagSlots;
    if (q < 8) t = kb_merge(t, KB{p[2 * q], p[2 * q + 1]});
    else m = q == 8 ? fmax(m, p[16]) : fmin(m, p[17]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (q < 8) {
      t = kb_merge(t, KB{__shfl_down_sync(0xffffffffu, t.s, o), __shfl_down_sync(0xffffffffu, t.c, o)});
    } else {
      const double x = __shfl_down_sync(0xffffffffu, m, o);
      m = q == 8 ? fmax(m, x) : fmin(m, x);
    }
  }
  if (lane == 0) {
    sm[w][0] = q < 8 ? t.s : m;
    sm[w][1] = t.c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    KB s{sm[0][0], sm[0][1]};
    for (int i = 1; i < kFinalWarps; i++) {
      if (q < 8) s = kb_merge(s, KB{sm[i][0], sm[i][1]});
      else s.s = q == 8 ? fmax(s.s, sm[i][0]) : fmin(s.s, sm[i][0]);
    }
    out[q] = q < 8 ? s.s + s.c : (q == 8 ? s.s * hmin : s.s);
  }
}

int diag_blocks(const Box& box) {
  const long long N = (long long)box.n[0] * box.n[1] * box.n[2];
  long long b = (N + 4LL * kDiagThreads - 1) / (4LL * kDiagThreads);
  if (b > kDiagGrid) b = kDiagGrid;
  if (b < 1) b = 1;
  return (int)b;
}

cudaError_t launch_diagnostics(const float* const f[8], const Box& box, double gamma, double* partial,
                               double* out, cudaStream_t s) {
  if (box.stride[0] != 1) return cudaErrorInvalidValue;
  const int nblk = diag_blocks(box);
  bool vec = box.n[0] % 2 == 0;
  for (int q = 0; q < 8; q++) vec = vec && reinterpret_cast<uintptr_t>(f[q]) % 8 == 0;
  const int W = vec ? 2 : 1;
  const FastDiv row_div = fast_div(box.n[0] / W), ny_div = fast_div(box.n[1]);
  auto* kernel = vec ? diag_partial_kernel<2> : diag_partial_kernel<1>;
  kernel<<<nblk, kDiagThreads, 0, s>>>(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], box.n[0], box.n[1], box.n[2],
                                       row_div, ny_div, gamma, partial);
  int nmax = box.n[0] > box.n[1] ? box.n[0] : box.n[1];
  nmax = nmax > box.n[2] ? nmax : box.n[2];
  diag_final_kernel<<<10, 32 * kFinalWarps, 0, s>>>(partial, nblk, 1.0 / nmax, out);
  return cudaGetLastError();
}

}  // namespace mhd
