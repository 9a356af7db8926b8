// Element-wise and stencil kernels of the learned coarse-grid correction
// (everything around the convolutions): restriction of a fine state to a
// coarse grid, input normalisation, projection of the network output onto a
// conservative, divergence-free correction (and its exact adjoint for
// training), the loss, the clipped application of a correction to a state,
// and the Adam update.  Fields are SoA FP32 (8 arrays of nx*ny*nz, as in the
// solver); network tensors are channels-last [cell][8].
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "fp32_sums.cuh"
#include "mhd.h"
#include "mhd_launch.h"

namespace mhd {
namespace {

struct F8 {
  float v[8];
};
struct P8 {
  float* p[8];
};
struct CP8 {
  const float* p[8];
};

// coarse cell (I, J, K) <- fine r^3 block; face fields: mean of the r^2 fine
// faces tiling the coarse low face (flux preserving, so div b stays 0).  A
// thread sums one coarse cell: in the three FP32 words of fp32_sums.cuh for
// windows of up to 64 values (their error, 64^3 2^-72 of the largest partial
// sum, is below an FP64 sum's), the windows of larger blocks in FP64.  With
// FP64 additions per fine value the kernel took 407 us for 256^3 -> 64^3; now
// it is bound by reading the fine state (89 us).
struct FSum {
  FWin2 w;
  double acc;
  __device__ __forceinline__ void init() {
    w.h = w.l = w.t = f2(0.f);
    acc = 0.0;
  }
  __device__ __forceinline__ void flush() {
    double a1 = 0.0;
    fwin_flush(w, acc, a1);
    acc += a1;
  }
  // the sum over n (exact in FP32): the words as a float-float value over n,
  // rounded once more than the exact quotient
  __device__ __forceinline__ float mean(float n) const {
    float h, l, e;
    two_sum(w.h.x, w.h.y, h, l);
    two_sum(h, __fadd_rn(__fadd_rn(l, __fadd_rn(w.l.x, w.l.y)), __fadd_rn(w.t.x, w.t.y)), h, l);
    const float q = __fdiv_rn(h, n);
    e = __fadd_rn(__fmaf_rn(-q, n, h), l);  // remainder of the quotient
    return __fadd_rn(q, __fdiv_rn(e, n));
  }
};

// The FP64 mean of an n0 x n1 x n2 block of values (strides 1, s1, s2), for
// blocks that the FP32 words cannot hold: infinities, and sums past FP32's range.
__device__ __noinline__ float mean_f64(const float* p, int n0, int n1, int n2, long long s0, long long s1,
                                       long long s2) {
  double a = 0.0;
  for (int k = 0; k < n2; k++)
    for (int j = 0; j < n1; j++)
      for (int i = 0; i < n0; i++) a += p[i * s0 + j * s1 + k * s2];
  return (float)(a / ((double)n0 * n1 * n2));
}

// R: the ratio (2 or 4: vector loads, one window per cell) or 0 (any r).
template <int R>
__global__ void __launch_bounds__(128) restrict_kernel(CP8 f, int nx, int ny, int nz, int rr, P8 c) {
  const int r = R ? R : rr;
  const int NX = nx / r, NY = ny / r, NZ = nz / r;
  const long long N = (long long)NX * NY * NZ;
  const bool wide = !R && (long long)r * r * r > 64;  // several windows: FP64 across them
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < N;
       idx += (long long)gridDim.x * blockDim.x) {
    const int I = (int)(idx % NX), J = (int)((idx / NX) % NY), K = (int)(idx / ((long long)NX * NY));
    const int i0 = I * r;
    FSum s[5], b[3];
    for (int q = 0; q < 5; q++) s[q].init();
    for (int q = 0; q < 3; q++) b[q].init();
    int in_window = 0, in_face = 0;
    for (int kk = 0; kk < r; kk++) {
#pragma unroll(R ? R : 1)
      for (int jj = 0; jj < r; jj++) {
        const long long row = i0 + (long long)nx * ((J * r + jj) + (long long)ny * (K * r + kk));
        if constexpr (R == 4) {
#pragma unroll
          for (int q = 0; q < 5; q++) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(f.p[q] + row));
            fwin_add(s[q].w, make_float2(v.x, v.y));
            fwin_add(s[q].w, make_float2(v.z, v.w));
          }
        } else if constexpr (R == 2) {
#pragma unroll
          for (int q = 0; q < 5; q++) fwin_add(s[q].w, __ldg(reinterpret_cast<const float2*>(f.p[q] + row)));
        } else {
          for (int ii = 0; ii < r; ii++) {
            for (int q = 0; q < 5; q++) fwin_add(s[q].w, make_float2(__ldg(f.p[q] + row + ii), 0.f));
            if (wide && ++in_window == 64) {
              in_window = 0;
              for (int q = 0; q < 5; q++) s[q].flush();
            }
          }
        }
        // the low x face takes every (jj, kk); kk and jj double as the y and
        // z faces' second index
        const long long fy = i0 + jj + (long long)nx * ((J * r) + (long long)ny * (K * r + kk));
        const long long fz = i0 + jj + (long long)nx * ((J * r + kk) + (long long)ny * (K * r));
        fwin_add(b[0].w, make_float2(__ldg(f.p[BX] + row), 0.f));
        fwin_add(b[1].w, make_float2(__ldg(f.p[BY] + fy), 0.f));
        fwin_add(b[2].w, make_float2(__ldg(f.p[BZ] + fz), 0.f));
        if (wide && ++in_face == 64) {
          in_face = 0;
          for (int q = 0; q < 3; q++) b[q].flush();
        }
      }
    }
    const long long corner = i0 + (long long)nx * (J * r + (long long)ny * (K * r)), plane = (long long)nx * ny;
    for (int q = 0; q < 5; q++) {
      if (wide) s[q].flush();
      float m = wide ? (float)(s[q].acc / ((double)r * r * r)) : s[q].mean((float)(r * r * r));
      if (!isfinite(m)) m = mean_f64(f.p[q] + corner, r, r, r, 1, nx, plane);
      c.p[q][idx] = m;
    }
    for (int q = 0; q < 3; q++) {
      if (wide) b[q].flush();
      float m = wide ? (float)(b[q].acc / ((double)r * r)) : b[q].mean((float)(r * r));
      if (!isfinite(m))
        m = mean_f64(f.p[BX + q] + corner, q == 0 ? 1 : r, q == 1 ? 1 : r, q == 2 ? 1 : r, 1, nx, plane);
      c.p[BX + q][idx] = m;
    }
  }
}

// 8 channels of a cell: one 16-byte access where the tensor is aligned (vec)
__device__ __forceinline__ void store_cell(__nv_bfloat16* x, int c, const float (&v)[8], bool vec) {
  if (vec) {
    __nv_bfloat162 p[4];
#pragma unroll
    for (int q = 0; q < 4; q++) p[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
    *reinterpret_cast<uint4*>(x + (size_t)c * 8) = *reinterpret_cast<const uint4*>(p);
  } else {
#pragma unroll
    for (int q = 0; q < 8; q++) x[(size_t)c * 8 + q] = __float2bfloat16_rn(v[q]);
  }
}
__device__ __forceinline__ void load_cell(const float* __restrict__ y, int c, float (&v)[8], bool vec) {
  if (vec) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(y + (size_t)c * 8));
    const float4 b = __ldg(reinterpret_cast<const float4*>(y + (size_t)c * 8 + 4));
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
    v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
  } else {
#pragma unroll
    for (int q = 0; q < 8; q++) v[q] = __ldg(y + (size_t)c * 8 + q);
  }
}

__global__ void normalize_kernel(CP8 s, int N, F8 mu, F8 isig, __nv_bfloat16* x, bool vec) {
  wait_for_previous();
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
    float v[8];
#pragma unroll
    for (int q = 0; q < 8; q++) v[q] = (s.p[q][c] - mu.v[q]) * isig.v[q];
    store_cell(x, c, v, vec);
  }
}

// Totals over a block of n quantities, from each thread's FP32 windows (pairs
// of quantities), added to sums[0 .. n-1] with one FP64 atomic each: the words
// are merged over lanes and warps in FP32, so FP64 appears once per block.
// (An FP64 sum and shuffle tree per warp and an atomic per warp took 58 us on
// a 64^3 grid.)  A block with infinities or sums near the end of FP32's range
// takes the threads' FP64 totals `exact(q)` instead.
template <int NP, class Exact>
__device__ __forceinline__ void block_totals(FWin2 (&w)[NP], int n, double* sums, Exact exact) {
  __shared__ float2 sm[kSumThreads / 32][NP][3];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  bool fits = true;
#pragma unroll
  for (int k = 0; k < NP; k++) {
    const float m = fmaxf(fabsf(w[k].h.x), fabsf(w[k].h.y));
    // (an infinity turns the error words into NaNs)
    fits = fits && m < 1e35f && w[k].l.x == w[k].l.x && w[k].l.y == w[k].l.y;
  }
  if (__syncthreads_or(!fits)) {
    for (int q = 0; q < n; q++) {
      double v = exact(q);
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) atomicAdd(&sums[q], v);
    }
    return;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < NP; k++) fwin_merge(w[k], shfl_down2(w[k].h, o), shfl_down2(w[k].l, o), shfl_down2(w[k].t, o));
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < NP; k++) {
      sm[wid][k][0] = w[k].h;
      sm[wid][k][1] = w[k].l;
      sm[wid][k][2] = w[k].t;
    }
  __syncthreads();
  if (threadIdx.x < NP) {
    const int k = threadIdx.x;
    FWin2 t{sm[0][k][0], sm[0][k][1], sm[0][k][2]};
    for (int i = 1; i < kSumThreads / 32; i++) fwin_merge(t, sm[i][k][0], sm[i][k][1], sm[i][k][2]);
    double a0 = 0.0, a1 = 0.0;
    fwin_flush(t, a0, a1);
    atomicAdd(&sums[2 * k], a0);
    if (2 * k + 1 < n) atomicAdd(&sums[2 * k + 1], a1);
  }
}

// Box totals of d_q = s_q y_q (q < 5), for the mean removal.
__global__ void __launch_bounds__(kSumThreads) project_sums_kernel(const float* __restrict__ y, int N, F8 sc,
                                                                   double* sums, bool vec) {
  wait_for_previous();
  FWin2 w[3];
  for (int k = 0; k < 3; k++) w[k].h = w[k].l = w[k].t = f2(0.f);
  for (unsigned c = blockIdx.x * kSumThreads + threadIdx.x; c < (unsigned)N; c += gridDim.x * kSumThreads) {
    float v[8];
    load_cell(y, c, v, vec);
    fwin_add(w[0], make_float2(__fmul_rn(sc.v[0], v[0]), __fmul_rn(sc.v[1], v[1])));
    fwin_add(w[1], make_float2(__fmul_rn(sc.v[2], v[2]), __fmul_rn(sc.v[3], v[3])));
    fwin_add(w[2], make_float2(__fmul_rn(sc.v[4], v[4]), 0.f));
  }
  block_totals(w, 5, sums, [&](int q) {
    double a = 0.0;
    for (unsigned c = blockIdx.x * kSumThreads + threadIdx.x; c < (unsigned)N; c += gridDim.x * kSumThreads)
      a += __fmul_rn(sc.v[q], y[(size_t)c * 8 + q]);
    return a;
  });
}

// Network output y[cell][8] -> correction d: d_q = s_q y_q less its box mean
// for q < 5 (cell quantities), and b = curl of the edge potential A_c = s_A
// y_{5+c} (A_x on x-edges (i, j-1/2, k-1/2), A_y on (i-1/2, j, k-1/2), A_z on
// (i-1/2, j-1/2, k)): the discrete divergence of d_b vanishes identically.
// The means are formed once per block (an FP64 division per cell and quantity
// took 28 us on a 64^3 grid).
__global__ void __launch_bounds__(256) project_kernel(const float* __restrict__ y, int nx, int ny, int nz, F8 sc,
                                                      P8 d, const double* __restrict__ sums, bool vec) {
  wait_for_previous();
  __shared__ float mean[5];
  const int N = nx * ny * nz;
  if (threadIdx.x < 5) mean[threadIdx.x] = (float)(sums[threadIdx.x] / N);
  __syncthreads();
  const float sA = sc.v[5];
  auto pot = [&](int c, float (&A)[3]) {  // y_5 .. y_7 of a cell
    A[0] = __ldg(y + (size_t)c * 8 + 5);
    A[1] = __ldg(y + (size_t)c * 8 + 6);
    A[2] = __ldg(y + (size_t)c * 8 + 7);
  };
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
    const int i = c % nx, r = c / nx, j = r % ny, k = r / ny;
    const int ip = i + 1 == nx ? c - i : c + 1, jp = j + 1 == ny ? c - j * nx : c + nx,
              kp = k + 1 == nz ? c - k * nx * ny : c + nx * ny;
    float v[8];
    load_cell(y, c, v, vec);
#pragma unroll
    for (int q = 0; q < 5; q++) d.p[q][c] = __fsub_rn(__fmul_rn(sc.v[q], v[q]), mean[q]);
    float I[3], J[3], K[3];
    pot(ip, I);
    pot(jp, J);
    pot(kp, K);
    const float Ax = v[5], Ay = v[6], Az = v[7];
    d.p[BX][c] = sA * ((J[2] - Az) * ny - (K[1] - Ay) * nz);
    d.p[BY][c] = sA * ((K[0] - Ax) * nz - (I[2] - Az) * nx);
    d.p[BZ][c] = sA * ((I[1] - Ay) * nx - (J[0] - Ax) * ny);
  }
}

// loss = sum_q w_q sum_cells (d_q - t_q)^2 ; g_q = 2 w_q (d_q - t_q).  The
// squares are summed exactly (product and its error) in FP32 words per
// field, and weighted once per block in FP64 (weighting and adding every
// square in FP64 took 26 us on a 64^3 grid).  A field's differences are scaled
// by a power of two, scale_q, that brings those the weight expects near 1, so
// that their squares keep clear of FP32's range; w2_q = w_q / scale_q^2.
struct LossWeights {
  float w[8], scale[8];
  double w2[8];
};
__global__ void __launch_bounds__(kSumThreads) loss_kernel(CP8 d, CP8 t, int N, LossWeights w, double* loss, P8 g) {
  wait_for_previous();
  __shared__ double tot[8];
  if (threadIdx.x < 8) tot[threadIdx.x] = 0.0;
  FWin2 s[4];
  for (int k = 0; k < 4; k++) s[k].h = s[k].l = s[k].t = f2(0.f);
  bool small = false;  // squares that underflow, or whose error words would
  for (unsigned c = blockIdx.x * kSumThreads + threadIdx.x; c < (unsigned)N; c += gridDim.x * kSumThreads) {
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const float2 diff = make_float2(d.p[2 * k][c] - t.p[2 * k][c], d.p[2 * k + 1][c] - t.p[2 * k + 1][c]);
      if (g.p[0]) {
        g.p[2 * k][c] = 2.f * w.w[2 * k] * diff.x;
        g.p[2 * k + 1][c] = 2.f * w.w[2 * k + 1] * diff.y;
      }
      const float2 x = __fmul2_rn(diff, make_float2(w.scale[2 * k], w.scale[2 * k + 1]));
      const float2 p = __fmul2_rn(x, x);
      const float2 e = __ffma2_rn(x, x, make_float2(-p.x, -p.y));
      fwin_add(s[k], p);
      float2 l, e2;
      two_sum2(s[k].l, e, l, e2);
      s[k].l = l;
      s[k].t = __fadd2_rn(s[k].t, e2);
    }
  }
  // (a field whose squares add up to nothing is looked through once more for a
  // difference that is not zero; kept in the loop above, that cost 3 us on a 64^3 grid)
  auto check = [&](int q, float h) {
    if (h > 0.f) small = small || h < 1e-20f;
    else if (h == 0.f)
      for (unsigned c = blockIdx.x * kSumThreads + threadIdx.x; c < (unsigned)N && !small; c += gridDim.x * kSumThreads)
        small = d.p[q][c] - t.p[q][c] != 0.f;
  };
#pragma unroll
  for (int k = 0; k < 4; k++) {
    check(2 * k, s[k].h.x);
    check(2 * k + 1, s[k].h.y);
  }
  if (small) s[0].h.x = __int_as_float(0x7f800000);  // the block takes the FP64 totals
  __syncthreads();
  block_totals(s, 8, tot, [&](int q) {
    double a = 0.0;
    for (unsigned c = blockIdx.x * kSumThreads + threadIdx.x; c < (unsigned)N; c += gridDim.x * kSumThreads) {
      const double x = (double)(d.p[q][c] - t.p[q][c]) * w.scale[q];
      a += x * x;
    }
    return a;
  });
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int q = 0; q < 8; q++) v += w.w2[q] * tot[q];
    atomicAdd(loss, v);
  }
}

__global__ void __launch_bounds__(kSumThreads) grad_sums_kernel(CP8 g, int N, double* sums) {
  wait_for_previous();
  FWin2 w[3];
  for (int k = 0; k < 3; k++) w[k].h = w[k].l = w[k].t = f2(0.f);
  for (unsigned c = blockIdx.x * kSumThreads + threadIdx.x; c < (unsigned)N; c += gridDim.x * kSumThreads) {
    fwin_add(w[0], make_float2(g.p[0][c], g.p[1][c]));
    fwin_add(w[1], make_float2(g.p[2][c], g.p[3][c]));
    fwin_add(w[2], make_float2(g.p[4][c], 0.f));
  }
  block_totals(w, 5, sums, [&](int q) {
    double a = 0.0;
    for (unsigned c = blockIdx.x * kSumThreads + threadIdx.x; c < (unsigned)N; c += gridDim.x * kSumThreads) a += g.p[q][c];
    return a;
  });
}

// adjoint of project + mean removal: gy_q = s_q (g_q - mean g_q) for q < 5;
// gy_{5+c} = s_A (curl^T g_b)_c
__global__ void __launch_bounds__(256) project_backward_kernel(CP8 g, int nx, int ny, int nz, F8 sc,
                                                               const double* __restrict__ sums, __nv_bfloat16* gy,
                                                               bool vec) {
  wait_for_previous();
  __shared__ float mean[5];
  const int N = nx * ny * nz;
  if (threadIdx.x < 5) mean[threadIdx.x] = (float)(sums[threadIdx.x] / N);
  __syncthreads();
  const float sA = sc.v[5];
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
    const int i = c % nx, r = c / nx, j = r % ny, k = r / ny;
    float v[8];
#pragma unroll
    for (int q = 0; q < 5; q++) v[q] = sc.v[q] * (g.p[q][c] - mean[q]);
    const int im = i == 0 ? c + nx - 1 : c - 1, jm = j == 0 ? c + (ny - 1) * nx : c - nx,
              km = k == 0 ? c + (nz - 1) * nx * ny : c - nx * ny;
    const float* gx = g.p[BX];
    const float* gyf = g.p[BY];
    const float* gz = g.p[BZ];
    v[5] = sA * (nz * (gyf[km] - gyf[c]) + ny * (gz[c] - gz[jm]));
    v[6] = sA * (nz * (gx[c] - gx[km]) + nx * (gz[im] - gz[c]));
    v[7] = sA * (ny * (gx[jm] - gx[c]) + nx * (gyf[c] - gyf[im]));
    store_cell(gy, c, v, vec);
  }
}

// Clipped application, pass 1 (cells): density clipped at -rho/2 and the whole
// cell correction scaled by the largest of 1, 1/2, 1/4, 0 that keeps the
// thermal energy, evaluated with the corrected faces, above half its value in
// the uncorrected state; if even 0 does not (the field correction raised the
// magnetic energy), e is raised to that bound.  The faces are read
// uncorrected and corrected on the fly; pass 2 writes them.
__global__ void __launch_bounds__(256) add_cells_kernel(P8 s, CP8 d, int nx, int ny, int nz, int* nclip) {
  wait_for_previous_in_place();
  const int N = nx * ny * nz;
  int clipped = 0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
    const int i = c % nx, r = c / nx, j = r % ny, k = r / ny;
    const int up[3] = {i + 1 == nx ? c - i : c + 1, j + 1 == ny ? c - j * nx : c + nx,
                       k + 1 == nz ? c - k * nx * ny : c + nx * ny};
    float b0[3], b1[3];  // cell-centred field, uncorrected and corrected
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const float lo = s.p[BX + a][c], hi = s.p[BX + a][up[a]];
      b0[a] = 0.5f * (lo + hi);
      b1[a] = 0.5f * (__fadd_rn(lo, d.p[BX + a][c]) + __fadd_rn(hi, d.p[BX + a][up[a]]));
    }
    const float mag0 = 0.5f * (b0[0] * b0[0] + b0[1] * b0[1] + b0[2] * b0[2]);
    const float mag = 0.5f * (b1[0] * b1[0] + b1[1] * b1[1] + b1[2] * b1[2]);
    float u0[5], du[5];
#pragma unroll
    for (int q = 0; q < 5; q++) {
      u0[q] = s.p[q][c];
      du[q] = d.p[q][c];
    }
    const float kin0 = 0.5f * (u0[1] * u0[1] + u0[2] * u0[2] + u0[3] * u0[3]) / u0[0];
    const float floor_e = 0.5f * (u0[4] - kin0 - mag0);
    const float drho = du[0];
    du[0] = fmaxf(drho, -0.5f * u0[0]);
    float u[5];
    bool done = false;
    for (int t = 0; t < 4 && !done; t++) {
      const float a = t == 0 ? 1.f : (t == 1 ? 0.5f : (t == 2 ? 0.25f : 0.f));
      for (int q = 0; q < 5; q++) u[q] = u0[q] + a * du[q];
      const float kin = 0.5f * (u[1] * u[1] + u[2] * u[2] + u[3] * u[3]) / u[0];
      if (u[4] - kin - mag >= floor_e) {
        done = true;
        clipped += t > 0;
      }
    }
    if (!done) {  // u holds the uncorrected cell quantities (a = 0)
      const float kin = 0.5f * (u[1] * u[1] + u[2] * u[2] + u[3] * u[3]) / u[0];
      u[4] = kin + mag + floor_e;
      clipped += 1;
    }
    if (du[0] != drho) clipped += 1;
    for (int q = 0; q < 5; q++) s.p[q][c] = u[q];
  }
  if (nclip && clipped) atomicAdd(nclip, clipped);
}

// pass 2: faces b += d_b (divergence-free, never scaled)
__global__ void add_field_kernel(P8 s, CP8 d, int N) {
  wait_for_previous_in_place();
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x)
    for (int q = 5; q < 8; q++) s.p[q][c] += d.p[q][c];
}

__global__ void adam_kernel(float* p, const float* g, float* m, float* v, int n, float lr, float b1, float b2,
                            float eps, float bc1, float bc2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
  }
}

int blocks(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b > 152 * 32 ? 152 * 32 : (b < 1 ? 1 : b));
}

bool vec16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

CP8 cp8(const float* const f[8]) {
  CP8 r;
  for (int q = 0; q < 8; q++) r.p[q] = f[q];
  return r;
}
P8 p8(float* const f[8]) {
  P8 r;
  for (int q = 0; q < 8; q++) r.p[q] = f ? f[q] : nullptr;
  return r;
}
F8 f8(const float* v, int n) {
  F8 r;
  for (int q = 0; q < 8; q++) r.v[q] = q < n ? v[q] : 0.f;
  return r;
}

int check_launch(const char* where) {
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? MHD_OK : set_error(MHD_E_CUDA, where, cudaGetErrorString(e));
}

bool bad_ptrs(const float* const f[8]) {
  if (!f) return true;
  for (int q = 0; q < 8; q++)
    if (!f[q]) return true;
  return false;
}

}  // namespace
}  // namespace mhd

using namespace mhd;

extern "C" {

int mhd_restrict(int nx, int ny, int nz, int r, const float* const fine[8], float* const coarse[8], void* stream) {
  if (r < 1 || nx % r || ny % r || nz % r || bad_ptrs(fine) || !coarse)
    return set_error(MHD_E_ARG, "mhd_restrict", "dims must be divisible by r; non-null fields");
  const long long N = (long long)(nx / r) * (ny / r) * (nz / r);
  // vector loads of a coarse cell's row: aligned fields (rows of nx = r NX
  // cells then start on a multiple of r cells)
  const auto aligned = [&](size_t bytes) {
    for (int q = 0; q < 5; q++)
      if (reinterpret_cast<uintptr_t>(fine[q]) % bytes) return false;
    return true;
  };
  const int grid = (int)std::max<long long>(1, std::min<long long>((N + 127) / 128, 152 * 64));  // (1: no cells)
  cudaStream_t st = (cudaStream_t)stream;
  if (r == 4 && aligned(16)) restrict_kernel<4><<<grid, 128, 0, st>>>(cp8(fine), nx, ny, nz, r, p8(coarse));
  else if (r == 2 && aligned(8)) restrict_kernel<2><<<grid, 128, 0, st>>>(cp8(fine), nx, ny, nz, r, p8(coarse));
  else restrict_kernel<0><<<grid, 128, 0, st>>>(cp8(fine), nx, ny, nz, r, p8(coarse));
  return check_launch("mhd_restrict");
}

int mhd_cnn_normalize(int nx, int ny, int nz, const float* const s[8], const float mu[8], const float inv_sigma[8],
                      void* x_bf16, void* stream) {
  if (bad_ptrs(s) || !mu || !inv_sigma || !x_bf16) return set_error(MHD_E_ARG, "mhd_cnn_normalize", "null argument");
  const int N = nx * ny * nz;
  launch_after(true, normalize_kernel, dim3(blocks(N)), dim3(256), 0, (cudaStream_t)stream, cp8(s), N, f8(mu, 8),
               f8(inv_sigma, 8), static_cast<__nv_bfloat16*>(x_bf16), vec16(x_bf16));
  return check_launch("mhd_cnn_normalize");
}

int mhd_cnn_project(int nx, int ny, int nz, const float* y, const float scale[6], float* const d[8], double* sums,
                    void* stream) {
  if (!y || !scale || !d || !sums) return set_error(MHD_E_ARG, "mhd_cnn_project", "null argument");
  const int N = nx * ny * nz;
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaMemsetAsync(sums, 0, sizeof(double) * 5, s);
  if (e != cudaSuccess) return set_error(MHD_E_CUDA, "mhd_cnn_project", cudaGetErrorString(e));
  launch_after(true, project_sums_kernel, dim3(sum_blocks(N)), dim3(kSumThreads), 0, s, y, N, f8(scale, 6), sums,
               vec16(y));
  launch_after(true, project_kernel, dim3(blocks(N)), dim3(256), 0, s, y, nx, ny, nz, f8(scale, 6), p8(d),
               static_cast<const double*>(sums), vec16(y));
  return check_launch("mhd_cnn_project");
}

int mhd_cnn_loss(int nx, int ny, int nz, const float* const d[8], const float* const t[8], const float weight[8],
                 double* loss, float* const g[8], void* stream) {
  if (bad_ptrs(d) || bad_ptrs(t) || !weight || !loss) return set_error(MHD_E_ARG, "mhd_cnn_loss", "null argument");
  const int N = nx * ny * nz;
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaMemsetAsync(loss, 0, sizeof(double), s);
  if (e != cudaSuccess) return set_error(MHD_E_CUDA, "mhd_cnn_loss", cudaGetErrorString(e));
  LossWeights lw;
  for (int q = 0; q < 8; q++) {
    // 1 / (8 w N) is the mean square that makes the field's share of the loss 1/8
    int ex = 0;
    const double ms = 8.0 * std::fabs((double)weight[q]) * N;
    if (ms > 0.0 && std::isfinite(ms)) ex = std::max(-60, std::min(60, (int)std::lround(0.5 * std::log2(ms))));
    lw.w[q] = weight[q];
    lw.scale[q] = (float)std::ldexp(1.0, ex);
    lw.w2[q] = std::ldexp((double)weight[q], -2 * ex);
  }
  launch_after(true, loss_kernel, dim3(sum_blocks(N)), dim3(kSumThreads), 0, s, cp8(d), cp8(t), N, lw, loss, p8(g));
  return check_launch("mhd_cnn_loss");
}

int mhd_cnn_project_backward(int nx, int ny, int nz, const float* const g[8], const float scale[6], double* sums,
                             void* gy_bf16, void* stream) {
  if (bad_ptrs(g) || !scale || !sums || !gy_bf16)
    return set_error(MHD_E_ARG, "mhd_cnn_project_backward", "null argument");
  const int N = nx * ny * nz;
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaMemsetAsync(sums, 0, sizeof(double) * 5, s);
  if (e != cudaSuccess) return set_error(MHD_E_CUDA, "mhd_cnn_project_backward", cudaGetErrorString(e));
  launch_after(true, grad_sums_kernel, dim3(sum_blocks(N)), dim3(kSumThreads), 0, s, cp8(g), N, sums);
  launch_after(true, project_backward_kernel, dim3(blocks(N)), dim3(256), 0, s, cp8(g), nx, ny, nz, f8(scale, 6),
               static_cast<const double*>(sums), static_cast<__nv_bfloat16*>(gy_bf16), vec16(gy_bf16));
  return check_launch("mhd_cnn_project_backward");
}

int mhd_correct(int nx, int ny, int nz, float* const s[8], const float* const d[8], float* scratch, int* nclip,
                void* stream) {
  if (!s || bad_ptrs(d) || !scratch) return set_error(MHD_E_ARG, "mhd_correct", "null argument");
  for (int q = 0; q < 8; q++)
    if (!s[q]) return set_error(MHD_E_ARG, "mhd_correct", "null field");
  const int N = nx * ny * nz;
  cudaStream_t st = (cudaStream_t)stream;
  launch_after(true, add_cells_kernel, dim3(blocks(N)), dim3(256), 0, st, p8(s), cp8(d), nx, ny, nz, nclip);
  launch_after(true, add_field_kernel, dim3(blocks(N)), dim3(256), 0, st, p8(s), cp8(d), N);
  return check_launch("mhd_correct");
}

int mhd_adam(float* p, const float* g, float* m, float* v, int count, float lr, float beta1, float beta2, float eps,
             int step, void* stream) {
  if (!p || !g || !m || !v || count < 0 || step < 1) return set_error(MHD_E_ARG, "mhd_adam", "bad arguments");
  const float bc1 = 1.f - powf(beta1, (float)step), bc2 = 1.f - powf(beta2, (float)step);
  adam_kernel<<<blocks(count), 256, 0, (cudaStream_t)stream>>>(p, g, m, v, count, lr, beta1, beta2, eps, bc1, bc2);
  return check_launch("mhd_adam");
}

}  // extern "C"
