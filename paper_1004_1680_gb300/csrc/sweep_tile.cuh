// Tile sweeps (Section II.B), FP32: sweeps along any axis in which a block
// holds its pencils' whole stencil on chip and every thread updates 4
// consecutive cells, for boxes whose pencils are too few or too short for the
// marching sweeps.
//
// A marching thread carries its pencil through one position after another:
// about 0.5 us per position of dependent arithmetic and loads, 39 positions
// for a 32-cell pencil, however idle the chip is.  Here the positions of a
// pencil are spread over threads, all loads of a sweep go out at once and the
// chain is that of 4 cells, with three exchanges between neighbouring threads
// (fluid) or two passes over shared memory (magnetic).  Time per step, marching
// -> tile: 32^3 302 -> 78 us, 64^3 308 -> 111, 96^3 432 -> 217, 236 x 150 x 98
// (x sweeps without transposes) 1043 -> 800 us (all sweeps by tiles, before
// the later changes; now 41, 68, 174 and 567).  Small boxes are bound by the
// launches (about 2.5 us each) and one chain of loads, arithmetic and stores
// (2 to 5 us); once the chip is full a fluid tile sweep runs at 17 (x) or 21 ps
// per cell, twice the marching sweep's 8.3 ps on a 512^3 box: its phases are
// separated by barriers at 16 warps per SM (resident blocks that copy the next
// tile's fields ahead only added instructions: 200^3 along x 141 -> 167 us).
// The dispatch (tile_choice in mhd_api.cu) leaves large boxes to the marching
// and row sweeps.
//
// The arithmetic of a cell is that of FluidPipe and MagPipe (mhd_device.cuh),
// operation for operation, so a tile sweep gives bitwise the result of the
// register-load marching sweep (FSQ = false), and agrees with it to FP32
// rounding with the hardware square root (FSQ = true, as in the staged
// sweeps).
#pragma once
#include "mhd_device.cuh"
#include "mhd_launch.h"
#include "sweep_row.cuh"
#include "tma.cuh"

namespace mhd {

// Periodic image of a position anywhere (a modulo only where one period is
// not enough: pencils of a few cells).
__device__ __forceinline__ int wrap_any(int i, int n) {
  i = i < 0 ? i + n : i;
  i = i >= n ? i - n : i;
  return (unsigned)i < (unsigned)n ? i : wrapi(i, n);
}

// ---------------------------------------------------------------------------
// Fluid tile sweep.  A block takes `np` consecutive pencils (row order of the
// other two axes, the contiguous one fastest) and `out` positions of them,
// `td` threads of 4 cells along each pencil.  Pencils of a multiple of 4
// cells that fit in the block are taken whole (`whole`: the end threads are
// neighbours across the periodic wrap); others in segments with one thread of
// 4 halo cells at each end (3 are needed), which stores nothing.
// (FluidTile and fluid_tile_split are declared in mhd_launch.h: the host
// builds the grid with the same split.)
constexpr int kTileSlots = 6;  // exchanged V5 values per thread (slot 0 is used twice)

__host__ __device__ constexpr size_t fluid_tile_smem(int threads) {
  return (size_t)threads * (5 * 16 + kTileSlots * 20);  // U of the 4 cells, the slots
}

// 128 registers: 2 blocks of 256 threads (or 4 of 128) per SM.  4 cells per
// thread: with 2 the exchanges cost more than the extra warps hide (128^3
// along y 57 us against 44).
template <int D, bool RATE, bool FLOOR, int LIM, int FRZ, bool FSQ>
__global__ void __launch_bounds__(kTileThreads, 2) fluid_tile_kernel(const __grid_constant__ FluidArgs a) {
  static_assert(FRZ != 2, "the per-pencil freezing speed keeps the pencil sweeps");
  constexpr int K = kTileCells;
  constexpr int A = (D == 0) ? 1 : 0, O = (D == 2) ? 1 : 2, T1 = (D + 1) % 3, T2 = (D + 2) % 3;
  extern __shared__ float4 tile_dyn[];
  const int nA = a.box.n[A], nO = a.box.n[O], nD = a.box.n[D];
  const int T = blockDim.x, tid = threadIdx.x;
  const FluidTile s = fluid_tile_split(D, nD, a.tile);
  const int np = s.np, td = s.td;
  // thread -> (pencil of the block, group of 4 cells): along x the groups of a
  // pencil are neighbouring threads (16 contiguous bytes each), else the
  // pencils are
  const int pp = D == 0 ? tid / td : tid % np, l = D == 0 ? tid - pp * td : tid / np;
  const int P = blockIdx.x * np + pp;
  const bool live = pp < np && l < td && P < nA * nO;
  RowSlots X;
  X.A = tile_dyn;
  X.E = reinterpret_cast<float*>(X.A + kTileSlots * T);
  X.T = T;
  float4* park = reinterpret_cast<float4*>(X.E + kTileSlots * T) + tid;  // U, [field][thread]
  const int lm = l > 0 ? l - 1 : (s.whole ? td - 1 : 0), lp = l + 1 < td ? l + 1 : (s.whole ? 0 : l);
  const int im = D == 0 ? tid + lm - l : tid + (lm - l) * np, ip = D == 0 ? tid + lp - l : tid + (lp - l) * np;

  const int pb = P / nA, pa = P - pb * nA;
  const int sA = (int)a.box.stride[A], sO = (int)a.box.stride[O], sD = (int)a.box.stride[D];
  unsigned base = (unsigned)(pa * sA + pb * sO);
  unsigned baseA1 = base + (unsigned)((pa + 1 == nA ? 1 - nA : 1) * sA);  // pencil +1 along A
  unsigned baseO1 = base + (unsigned)((pb + 1 == nO ? 1 - nO : 1) * sO);  // pencil +1 along O
  // the first of the thread's cells, before wrapping
  int p0 = blockIdx.z * s.out + K * (l - (s.whole ? 0 : 1));
  unsigned off[K + 1];  // of the cells p0 .. p0+4 along the pencil
#pragma unroll
  for (int j = 0; j <= K; j++) {
    off[j] = (D == 0 && j > 0 && j < K) ? 0u : (unsigned)(wrap_any(p0 + j, nD) * sD);
    settle(off[j]);
  }
  settled(base, baseA1, baseO1, p0);
  wait_for_previous();
  const float gamma = a.gamma;
  const bool begins = D == 0 && !RATE && a.control.rate;
  __shared__ float own_tau;
  float tau = 0.f;
  if (!begins) {
    tau = *a.tau;
  } else if (tid == 0) {
    tau = step_tau(a.control);
    own_tau = tau;
    if (blockIdx.x == 0 && blockIdx.z == 0) step_begin(a.control, tau);
  }

  V5 f1[K + 1];  // flux1 at p0-1/2 .. p0+7/2
  V5 FR3, FL0;
  B3 B[K];
  if (live) {
    // every load of the sweep, before the first use
    const float* __restrict__ f[8];
#pragma unroll
    for (int q = 0; q < 8; q++) f[q] = a.in[q];
    const unsigned baseT1 = (T1 == A) ? baseA1 : baseO1, baseT2 = (T2 == A) ? baseA1 : baseO1;
    constexpr int kField[5] = {RHO, MX + D, MX + T1, MX + T2, EN};
    float u[5][K], bd[K + 1], b1[K], b1n[K], b2[K], b2n[K];
    if constexpr (D == 0) {
      const unsigned c = base + off[0];  // p0 and nx are multiples of 4
      auto ld4 = [](const float* p, float (&d)[K]) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p));
#pragma unroll
        for (int j = 0; j < K; j++) d[j] = (&v.x)[j];
      };
      const unsigned w = c - base;
#pragma unroll
      for (int q = 0; q < 5; q++) ld4(f[kField[q]] + c, u[q]);
      float t[K];
      ld4(f[BX + D] + c, t);
#pragma unroll
      for (int j = 0; j < K; j++) bd[j] = t[j];
      bd[K] = __ldg(f[BX + D] + (base + off[K]));
      ld4(f[BX + T1] + c, b1);
      ld4(f[BX + T1] + (baseT1 + w), b1n);
      ld4(f[BX + T2] + c, b2);
      ld4(f[BX + T2] + (baseT2 + w), b2n);
    } else {
#pragma unroll
      for (int j = 0; j < K; j++) {
#pragma unroll
        for (int q = 0; q < 5; q++) u[q][j] = __ldg(f[kField[q]] + (base + off[j]));
        bd[j] = __ldg(f[BX + D] + (base + off[j]));
        b1[j] = __ldg(f[BX + T1] + (base + off[j]));
        b1n[j] = __ldg(f[BX + T1] + (baseT1 + off[j]));
        b2[j] = __ldg(f[BX + T2] + (base + off[j]));
        b2n[j] = __ldg(f[BX + T2] + (baseT2 + off[j]));
      }
      bd[K] = __ldg(f[BX + D] + (base + off[K]));
    }
    // U waits in the thread's own shared memory between its three uses
#pragma unroll
    for (int q = 0; q < 5; q++) {
      float4 v;
#pragma unroll
      for (int j = 0; j < K; j++) (&v.x)[j] = u[q][j];
      park[q * T] = v;
    }
    // stage 1: first-order fluxes
    V5 FRp;
#pragma unroll
    for (int j = 0; j < K; j++) {
      B[j] = {{face_mean(bd[j], bd[j + 1]), face_mean(b1[j], b1n[j]), face_mean(b2[j], b2n[j])}};
      const V5 U = {make_float2(u[0][j], u[1][j]), make_float2(u[2][j], u[3][j]), u[4][j]};
      V5 FR, FL;
      split_flux<FRZ, FSQ>(U, B[j].v[0], make_float2(B[j].v[1], B[j].v[2]), gamma, FR, FL);
      if (j == 0) FL0 = FL;
      else f1[j] = v5_sub(FRp, FL);
      FRp = FR;
    }
    FR3 = FRp;
    X.put(0, tid, FR3);
    X.put(1, tid, FL0);
  }
  __syncthreads();
  if (begins) tau = own_tau;
  const float c_full = tau * a.box.ih[D];  // tau / h_D
  const float c_half = 0.5f * c_full;
  V5 Rh[K], Lh[K];
  auto parked = [&](V5 (&U)[K]) {
    float4 v[5];
#pragma unroll
    for (int q = 0; q < 5; q++) v[q] = park[q * T];
#pragma unroll
    for (int j = 0; j < K; j++)
      U[j] = {make_float2((&v[0].x)[j], (&v[1].x)[j]), make_float2((&v[2].x)[j], (&v[3].x)[j]), (&v[4].x)[j]};
  };
  if (live) {
    f1[0] = v5_sub(X.get(0, im), FL0);          // FR(p0-1) - FL(p0)
    f1[K] = v5_sub(FR3, X.get(1, ip));  // FR(p0+3) - FL(p0+4)
    V5 U[K];
    parked(U);
#pragma unroll
    for (int j = 0; j < K; j++) {
      const V5 Uh = v5_fma(-c_half, v5_sub(f1[j + 1], f1[j]), U[j]);
      // stage 2
      split_flux<FRZ, FSQ>(Uh, B[j].v[0], make_float2(B[j].v[1], B[j].v[2]), gamma, Rh[j], Lh[j]);
    }
    X.put(2, tid, Rh[K - 1]);
    X.put(3, tid, Rh[0]);
    X.put(4, tid, Lh[0]);
    X.put(5, tid, Lh[1]);
  }
  __syncthreads();
  V5 F2[K];
  if (live) {
    // interface j+1/2: Rh(j-1..j+1), Lh(j..j+2)
    auto flux2 = [&](int j, const V5& Rl, const V5& Rr, const V5& L1, const V5& L2) {
      const V5 right = v5_add(Rh[j], half_limited5<LIM>(v5_sub(Rh[j], Rl), v5_sub(Rr, Rh[j])));
      const V5 left = v5_sub(L1, half_limited5<LIM>(v5_sub(L1, Lh[j]), v5_sub(L2, L1)));
      return v5_sub(right, left);
    };
    const V5 Rp = X.get(3, ip), Lp0 = X.get(4, ip), Lp1 = X.get(5, ip);
    F2[K - 1] = flux2(K - 1, Rh[K - 2], Rp, Lp0, Lp1);
    X.put(0, tid, F2[K - 1]);
    F2[2] = flux2(2, Rh[1], Rh[3], Lh[3], Lp0);
    F2[1] = flux2(1, Rh[0], Rh[2], Lh[2], Lh[3]);
    F2[0] = flux2(0, X.get(2, im), Rh[1], Lh[1], Lh[2]);
  }
  __syncthreads();
  float rmax = 0.f;
  // cells of this block's own positions (halo threads and the cells past the
  // pencil's end store nothing)
  const int first = blockIdx.z * s.out, pend = min(nD, first + s.out);
  if (live && p0 >= first && p0 < pend) {
    float* __restrict__ o[5];
    constexpr int kField[5] = {RHO, MX + D, MX + T1, MX + T2, EN};
#pragma unroll
    for (int q = 0; q < 5; q++) o[q] = a.out[kField[q]];
    V5 U[K];
    parked(U);
    const V5 Fm = X.get(0, im);
    const bool rate_pencil =
        RATE && pa >= a.rate_lo[A] && pa < a.rate_hi[A] && pb >= a.rate_lo[O] && pb < a.rate_hi[O];
    float r[K][5];
    bool clear = true;  // FLOOR: every cell above the floor
#pragma unroll
    for (int j = 0; j < K; j++) {
      const V5 v = v5_fma(-c_full, v5_sub(F2[j], j ? F2[j ? j - 1 : 0] : Fm), U[j]);
      r[j][0] = v.p0.x;
      r[j][1] = v.p0.y;
      r[j][2] = v.p1.x;
      r[j][3] = v.p1.y;
      r[j][4] = v.e;
      if (FLOOR) clear &= above_floor(r[j], square3(B[j].v), a.e_floor);
    }
    if (FLOOR && !clear)
#pragma unroll
      for (int j = 0; j < K; j++) r[j][4] = floored_energy(r[j], square3(B[j].v), a.e_floor);
    if (RATE && rate_pencil)
#pragma unroll
      for (int j = 0; j < K; j++) {
        const int p = p0 + j;
        if (p < pend && p >= a.rate_lo[D] && p < a.rate_hi[D]) {
          float m[3], bg[3];
          m[D] = r[j][1]; m[T1] = r[j][2]; m[T2] = r[j][3];
          bg[D] = B[j].v[0]; bg[T1] = B[j].v[1]; bg[T2] = B[j].v[2];
          rmax = fmaxf(rmax, cell_rate(r[j][0], m, r[j][4], bg, gamma, a.box.ih));
        }
      }
    if constexpr (D == 0) {
#pragma unroll
      for (int q = 0; q < 5; q++) {
        float4 v;
#pragma unroll
        for (int j = 0; j < K; j++) (&v.x)[j] = r[j][q];
        *reinterpret_cast<float4*>(o[q] + (base + (unsigned)p0)) = v;
      }
    } else {
#pragma unroll
      for (int j = 0; j < K; j++)
        if (p0 + j < pend)
#pragma unroll
          for (int q = 0; q < 5; q++) o[q][base + (unsigned)((p0 + j) * sD)] = r[j][q];
    }
  }
  if (RATE) {
    for (int k = 16; k > 0; k >>= 1) rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, k));
    if ((tid & 31) == 0 && rmax > 0.f) atomicMax(a.rate, __float_as_uint(rmax));
  }
}

// ---------------------------------------------------------------------------
// Magnetic tile sweep.  A block takes a tile of LX (lane axis A) x R (row
// axis O) pencils and `out` positions of them, and holds in shared memory,
// with the positions' halo at each end (periodic images):
//   v  = m_D / rho of the tile's pencils and of the ones next to them,
//   b_A of columns 0 .. LX and b_O of rows 0 .. R (LX and R: the halo pencils
//   whose edge flux the tile's b_D takes), b_D of the tile's pencils.
// All of it arrives by asynchronous 16-byte copies, issued at once.  Then every
// (pencil, group of 4 edges) is one independent task: 9 cells of b_A, b_O and
// the velocities around them give the 4 limited edge fluxes of both fields on
// packed FP32 (one of the two is unused in a halo pencil), with the half step of
// 3 cells at the group's ends repeated by both neighbours (which needs no
// exchange between threads).  After a barrier the cells are finished from the
// fluxes.  Along y and z it executes 232 instructions per cell (318 with a task
// per field and 4-byte copies; the marching sweep 144), and what bounds it is
// the latency of its phases at the blocks that shared memory lets in: 2 per
// SM, of 384 threads so that a tile's tasks take two whole rounds (96^3 along
// y 19.7 -> 16.4 us, a step 217 -> 181 us with the launches overlapped).
template <int LX, int R>
struct MTile {
  static constexpr int T = LX * R >= 64 ? 384 : 128;     // threads
  static constexpr int Tasks = (R + 1) * (LX + 1) - 1;   // pencils with a flux (not the far corner)
  static constexpr int C = LX * R;                       // cells of a plane
};
__host__ __device__ constexpr int mag_tile_halo(int D) { return D == 0 ? 4 : 3; }  // 4: 16-byte copies along x

// positions held per pencil: `out`, the halos and what the last group of edges
// may touch past them; along x an odd number of 16-byte pieces
__host__ __device__ constexpr int mag_tile_positions(int D, int out) {
  const int n = out + 2 * mag_tile_halo(D) + 4;
  return D == 0 ? (n + 3) / 8 * 8 + 4 : n;
}

__device__ __forceinline__ void copy16_async(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ float4& at4(float* p) { return *reinterpret_cast<float4*>(p); }
__device__ __forceinline__ float4 v_div4(const float4& m, const float4& r) {
  return make_float4(v_div(m.x, r.x), v_div(m.y, r.y), v_div(m.z, r.z), v_div(m.w, r.w));
}

// The 4 limited edge fluxes of a group from 9 cells of (b_A, b_O) and of their
// face velocities (MagPipe's arithmetic, each element rounded as there): edge k
// lies between cells k + 2 and k + 3.
template <int LIM>
__device__ __forceinline__ void edge_fluxes2(const float2 (&q)[9], const float2 (&u)[9], float c_half, float2 (&f)[4]) {
  auto sel = [](float2 w, float2 a, float2 b) { return make_float2(w.x >= 0.f ? a.x : b.x, w.y >= 0.f ? a.y : b.y); };
  float2 ub[8], g[8], h[7], d[6];
#pragma unroll
  for (int k = 0; k < 8; k++) {
    ub[k] = __fmul2_rn(f2(0.5f), __fadd2_rn(u[k], u[k + 1]));
    g[k] = __fmul2_rn(ub[k], sel(ub[k], q[k], q[k + 1]));
  }
#pragma unroll
  for (int k = 0; k < 7; k++) h[k] = __ffma2_rn(f2(-c_half), sub2(g[k + 1], g[k]), q[k + 1]);
#pragma unroll
  for (int k = 0; k < 6; k++) d[k] = sub2(h[k + 1], h[k]);
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const float2 w = ub[k + 2];
    const float2 lim = half_limited2<LIM>(sel(w, d[k], d[k + 1]), sel(w, d[k + 1], d[k + 2]));
    // base + lim upwind from below, base - lim from above (the product is exact)
    f[k] = __fmul2_rn(w, __ffma2_rn(sel(w, f2(1.f), f2(-1.f)), lim, sel(w, h[k + 1], h[k + 2])));
  }
}

// Along y and z: planes of pencils, one per position.  NP = 2 (whole pencils
// only): two sweeps with the same step; the first one's result stays in
// shared memory.  SHORT: pencils of 1 or 2 cells, which have several periodic
// images on a side of the halo (a kernel of their own: 32^3 39.4 us per step,
// 39.9 with the loops over images in the one that it runs).
template <int LX, int R>
struct MPlane {  // offsets of a plane's arrays (floats) and its size
  static constexpr int VW = LX + 8, V = (R + 2) * VW;  // v: rows -1 .. R, columns -4 .. LX + 3
  static constexpr int AW = LX + 4, A = R * AW;        // b_A: columns 0 .. LX + 3
  static constexpr int O = (R + 1) * LX;               // b_O: rows 0 .. R
  static constexpr int B = LX * R;                     // b_D
  static constexpr int F = (2 * MTile<LX, R>::Tasks + 3) / 4 * 4;  // (f_A, f_O) of the tasks; first holds rho
  static constexpr int Size = V + A + O + B + (F > V ? F : V);
  static constexpr int Pieces = (2 * V + A + O + B) / 4;
};

template <int D, int LX, int R, int LIM, int NP, bool SHORT = false>
__global__ void __launch_bounds__(MTile<LX, R>::T) mag_tile_kernel(const __grid_constant__ MagArgs a) {
  static_assert(D != 0, "x sweeps use mag_tile_x_kernel");
  constexpr int A = 0, O = (D == 2) ? 1 : 2, T1 = (D + 1) % 3;
  using M = MTile<LX, R>;
  using L = MPlane<LX, R>;
  constexpr int H = mag_tile_halo(D), T = M::T, Sv = L::V, Sa = L::A, So = L::O, Sb = L::B, Sf = L::F > L::V ? L::F : L::V;
  extern __shared__ __align__(16) float mt_dyn[];
  const int nA = a.box.n[A], nO = a.box.n[O], nD = a.box.n[D];
  const MagTile sp = mag_tile_split(nD);
  const int a0 = (int)blockIdx.x * LX, b0 = (int)blockIdx.y * R;
  const int s0 = (int)blockIdx.z * sp.out, S = min(sp.out, nD - s0);  // this block's positions s0 .. s0 + S - 1
  const int PN = mag_tile_positions(D, sp.out);
  float* sv = mt_dyn;
  float* sa = sv + Sv * PN;
  float* so = sa + Sa * PN;
  float* sb = so + So * PN;
  float* sf = sb + Sb * PN;
  const int tid = threadIdx.x;
  const int sO = (int)a.box.stride[O], sD = (int)a.box.stride[D];

  // A thread keeps its 16-byte piece of the plane and walks the positions.  The
  // lanes are contiguous and nA a multiple of 4, so pieces never straddle the
  // periodic wrap; rho waits in sf.
  {
    constexpr int kSlots = L::Pieces <= 64 ? 64 : 128, kStep = T / kSlots;
    static_assert(L::Pieces <= kSlots && T % kSlots == 0, "pieces of a plane");
    int piece = tid % kSlots;
    if (piece < L::Pieces) {
      const float* src;
      float* dst;
      int row, col, plane;
      auto place = [&](float* arr, int size, int width, int r0, int c0, const float* field) {
        const int q = piece * 4;
        row = q / width + r0;
        col = q % width + c0;
        dst = arr + q;
        plane = size;
        src = field;
      };
      if (piece < Sv / 4) {
        place(sv, Sv, L::VW, -1, -4, a.in[MX + D]);
      } else if ((piece -= Sv / 4) < Sv / 4) {
        place(sf, Sf, L::VW, -1, -4, a.in[RHO]);
      } else if ((piece -= Sv / 4) < Sa / 4) {
        place(sa, Sa, L::AW, 0, 0, a.in[BX + A]);
      } else if ((piece -= Sa / 4) < So / 4) {
        place(so, So, LX, 0, 0, a.in[BX + O]);
      } else {
        piece -= So / 4;
        place(sb, Sb, LX, 0, 0, a.in[BX + D]);
      }
      int at = wrap_any(a0 + col, nA) + wrap_any(b0 + row, nO) * sO;
      settled(at, plane);
      src += at;
      wait_for_previous();
      for (int p = tid / kSlots; p < S + 2 * H; p += kStep)
        copy16_async(dst + p * plane, src + (unsigned)(wrap_any(s0 - H + p, nD) * sD));
    } else {
      wait_for_previous();
    }
    copies_wait();
    __syncthreads();
    constexpr int kQuads = Sv / 4;
    for (int t = tid; t < kQuads * (S + 2 * H); t += T) {
      const int p = t / kQuads, q = 4 * (t - p * kQuads);
      at4(sv + p * Sv + q) = v_div4(at4(sv + p * Sv + q), at4(sf + p * Sf + q));
    }
  }
  const float tau = *a.tau;
  const float c_full = tau * a.box.ih[D];  // tau / h_D
  const float c_half = 0.5f * c_full;
  const float kA = tau * a.box.ih[A];      // tau / h_A
  const float kO = tau * a.box.ih[O];      // tau / h_O
  // edge e lies between local cells e - 1 and e: edges 0 .. S are needed; of a
  // whole pencil 1 .. S (edge 0 is edge S)
  const int e0 = sp.whole ? 1 : 0;
  const int groups = (S + 1 - e0 + 3) / 4;
  auto flux = [&](int task, int e) -> float2& { return *reinterpret_cast<float2*>(sf + e * Sf + 2 * task); };
#pragma unroll 1
  for (int pass = 0; pass < NP; pass++) {
    __syncthreads();
    for (int t = tid; t < M::Tasks * groups; t += T) {
      const int g = t / M::Tasks, ts = t - g * M::Tasks, row = ts / (LX + 1), col = ts - row * (LX + 1);
      const int e = e0 + 4 * g;  // edges e .. e + 3; cells e - 3 .. e + 5
      const float* pv = sv + (e - 3 + H) * Sv + (row + 1) * L::VW + col + 4;
      const float* pa = sa + (e - 3 + H) * Sa + row * L::AW + col;  // (past the array in row R: unused)
      const float* po = so + (e - 3 + H) * So + row * LX + col;     // (the next row's in column LX: unused)
      float2 q[9], u[9], f[4];
#pragma unroll
      for (int k = 0; k < 9; k++) {
        const float v = pv[k * Sv];
        q[k] = make_float2(pa[k * Sa], po[k * So]);
        // v_D on the b_A and the b_O face
        u[k] = __fmul2_rn(f2(0.5f), __fadd2_rn(f2(v), make_float2(pv[k * Sv - 1], pv[k * Sv - L::VW])));
      }
      edge_fluxes2<LIM>(q, u, c_half, f);
#pragma unroll
      for (int k = 0; k < 4; k++) flux(ts, e + k) = f[k];
    }
    __syncthreads();
    if (pass + 1 == NP) {
      // finish the tile's cells
      float* __restrict__ oA = a.out[A];
      float* __restrict__ oO = a.out[O];
      float* __restrict__ oD = a.out[D];
      static_assert(T % M::C == 0, "a thread keeps its pencil");
      const int c = tid % M::C, row = c / LX, col = c - row * LX, ts = row * (LX + 1) + col;
      if (a0 + col < nA && b0 + row < nO) {
        const unsigned ob = (unsigned)((a0 + col) + (b0 + row) * sO + s0 * sD);
        for (int p = tid / M::C; p < S; p += T / M::C) {
          const int el = sp.whole && p == 0 ? S : p;  // the edge below cell p
          const float2 lo = flux(ts, el), hi = flux(ts, p + 1);
          const unsigned o = ob + (unsigned)(p * sD);
          oA[o] = __fmaf_rn(-c_full, __fsub_rn(hi.x, lo.x), sa[(p + H) * Sa + row * L::AW + col]);
          oO[o] = __fmaf_rn(-c_full, __fsub_rn(hi.y, lo.y), so[(p + H) * So + c]);
          oD[o] = constrain(sb[(p + H) * Sb + c], kA, lo.x, flux(ts + 1, el).x, kO, lo.y, flux(ts + LX + 1, el).y, T1 == A);
        }
      }
    } else {
      // the first pass's result back into shared memory (whole pencils): the
      // advected fields with their periodic images, and b_D
      for (int t = tid; t < M::Tasks * S; t += T) {
        const int p = t / M::Tasks, ts = t - p * M::Tasks, row = ts / (LX + 1), col = ts - row * (LX + 1);
        const float2 lo = flux(ts, p == 0 ? S : p), hi = flux(ts, p + 1);
        auto update = [&](float* z, int plane, float fl, float fh) {
          const float v = __fmaf_rn(-c_full, __fsub_rn(fh, fl), z[p * plane]);
          z[p * plane] = v;
          if (p < H) z[(p + S) * plane] = v;
          if (p >= S - H) z[(p - S) * plane] = v;
          if constexpr (SHORT) {
            for (int m = p + S; m < S + H; m += S) z[m * plane] = v;
            for (int m = p - S; m >= -H; m -= S) z[m * plane] = v;
          }
        };
        if (row < R) update(sa + H * Sa + row * L::AW + col, Sa, lo.x, hi.x);
        if (col < LX) update(so + H * So + row * LX + col, So, lo.y, hi.y);
        if (row < R && col < LX) {
          float* z = sb + (p + H) * Sb + row * LX + col;
          const int el = p == 0 ? S : p;
          *z = constrain(*z, kA, lo.x, flux(ts + 1, el).x, kO, lo.y, flux(ts + LX + 1, el).y, T1 == A);
        }
      }
    }
  }
}

// Along x: a pencil's positions are contiguous, everything moves in 16-byte
// pieces of 4 positions (an odd number of pieces per pencil keeps the pencils
// of a quarter warp in different banks).  A task is one field's edge flux: the
// packed pairs of the other axes, whose operands come from separate 16-byte
// reads here, executed as many instructions (358 per cell against 354) and ran
// slower (128^3: 33 us against 31).
template <int LX, int R>
struct MRows {
  static constexpr int VC = LX + 2, V = (R + 2) * VC;      // pencils of v: rows -1 .. R, columns -1 .. LX
  static constexpr int QA = R * (LX + 1), Q = QA + (R + 1) * LX;  // edge-flux rows: b_A, then b_O
  static constexpr int C = LX * R;
  static constexpr int Size = V + 2 * Q + C;
  // v pencils of edge-flux row ts's pencil and of the one across its faces
  static __device__ __forceinline__ void rows(int ts, int& own, int& nbr) {
    if (ts < QA) {
      const int row = ts / (LX + 1), col = ts - row * (LX + 1);
      own = (row + 1) * VC + col + 1;
      nbr = own - 1;
    } else {
      const int o = ts - QA, row = o / LX, col = o - row * LX;
      own = (row + 1) * VC + col + 1;
      nbr = own - VC;
    }
  }
};

// The 4 limited edge fluxes of a group from 9 cells of q and face velocity u
// (MagPipe's arithmetic): edge k lies between cells k + 2 and k + 3.
template <int LIM>
__device__ __forceinline__ void edge_fluxes(const float (&q)[9], const float (&u)[9], float c_half, float (&f)[4]) {
  float ub[8], g[8], h[7], d[6];
#pragma unroll
  for (int k = 0; k < 8; k++) {
    ub[k] = __fmul_rn(0.5f, __fadd_rn(u[k], u[k + 1]));
    g[k] = __fmul_rn(ub[k], ub[k] >= 0.f ? q[k] : q[k + 1]);
  }
#pragma unroll
  for (int k = 0; k < 7; k++) h[k] = __fmaf_rn(-c_half, __fsub_rn(g[k + 1], g[k]), q[k + 1]);
#pragma unroll
  for (int k = 0; k < 6; k++) d[k] = __fsub_rn(h[k + 1], h[k]);
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const float w = ub[k + 2];
    const bool pos = w >= 0.f;
    const float lim = half_limited<LIM>(pos ? d[k] : d[k + 1], pos ? d[k + 1] : d[k + 2]);
    f[k] = __fmul_rn(w, pos ? __fadd_rn(h[k + 1], lim) : __fsub_rn(h[k + 2], lim));
  }
}

template <int LX, int R, int LIM>
__global__ void __launch_bounds__(MTile<LX, R>::T) mag_tile_x_kernel(const __grid_constant__ MagArgs a) {
  using M = MRows<LX, R>;
  constexpr int H = mag_tile_halo(0), T = MTile<LX, R>::T;
  extern __shared__ __align__(16) float mt_dyn[];
  const int nA = a.box.n[1], nO = a.box.n[2], nD = a.box.n[0];
  const MagTile sp = mag_tile_split(nD);
  const int a0 = (int)blockIdx.x * LX, b0 = (int)blockIdx.y * R;
  const int s0 = (int)blockIdx.z * sp.out, S = min(sp.out, nD - s0);  // multiples of 4
  const int PN = mag_tile_positions(0, sp.out);
  float* sv = mt_dyn;
  float* sq = sv + M::V * PN;
  float* sf = sq + M::Q * PN;
  float* sb = sf + M::Q * PN;
  const int tid = threadIdx.x;
  const int sA = (int)a.box.stride[1], sO = (int)a.box.stride[2];
  // (pencil, piece) pairs, stepped without a division per piece; a thread
  // forms v of the pieces it has copied itself
  const int pieces = (S + 2 * H) / 4;
  int dslot = T / pieces, dpiece = T - dslot * pieces, slot0 = tid / pieces, piece0 = tid - slot0 * pieces;
  settled(dslot, dpiece, slot0, piece0);
  wait_for_previous();
  for (int half = 0; half < 2; half++) {
    int slot = slot0, g = piece0;
    while (slot < M::V) {
      const int row = slot / M::VC, col = slot - row * M::VC;
      const bool rin = row >= 1 && row <= R, cin = col >= 1 && col <= LX;
      if (rin || cin) {
        float* v = sv + slot * PN + 4 * g;
        float* r = sf + slot * PN + 4 * g;
        if (half == 0) {
          const unsigned c = (unsigned)(wrap_any(a0 + col - 1, nA) * sA + wrap_any(b0 + row - 1, nO) * sO +
                                        wrap_any(s0 - H + 4 * g, nD));
          copy16_async(v, a.in[MX] + c);
          copy16_async(r, a.in[RHO] + c);
          if (rin && col >= 1) copy16_async(sq + ((row - 1) * (LX + 1) + col - 1) * PN + 4 * g, a.in[BY] + c);
          if (cin && row >= 1) copy16_async(sq + (M::QA + (row - 1) * LX + col - 1) * PN + 4 * g, a.in[BZ] + c);
          if (rin && cin) copy16_async(sb + ((row - 1) * LX + col - 1) * PN + 4 * g, a.in[BX] + c);
        } else {
          at4(v) = v_div4(at4(v), at4(r));
        }
      }
      slot += dslot;
      g += dpiece;
      if (g >= pieces) {
        g -= pieces;
        slot++;
      }
    }
    if (half == 0) copies_wait();
  }
  const float tau = *a.tau;
  const float c_full = tau * a.box.ih[0];  // tau / h_x
  const float c_half = 0.5f * c_full;
  const float kA = tau * a.box.ih[1];      // tau / h_y
  const float kO = tau * a.box.ih[2];      // tau / h_z
  const int e0 = sp.whole ? 1 : 0;         // edges e0 .. S, edge e at position e - e0 of sf
  const int groups = (S + 1 - e0 + 3) / 4;
  __syncthreads();
  for (int t = tid; t < M::Q * groups; t += T) {
    const int g = t / M::Q, ts = t - g * M::Q;
    int vo, vn;
    M::rows(ts, vo, vn);
    // cells e - 3 .. e + 5, e = e0 + 4 g: positions 4 g + 1 + e0 .. of the
    // three pieces from 4 g
    auto cells = [&](float* s, float (&x)[9]) {
      float w[12];
#pragma unroll
      for (int k = 0; k < 3; k++) {
        const float4 z = at4(s + 4 * k);
        w[4 * k] = z.x;
        w[4 * k + 1] = z.y;
        w[4 * k + 2] = z.z;
        w[4 * k + 3] = z.w;
      }
#pragma unroll
      for (int k = 0; k < 9; k++) x[k] = e0 ? w[k + 2] : w[k + 1];
    };
    float q[9], u[9], un[9], f[4];
    cells(sv + vo * PN + 4 * g, u);
    cells(sv + vn * PN + 4 * g, un);
#pragma unroll
    for (int k = 0; k < 9; k++) u[k] = __fmul_rn(0.5f, __fadd_rn(u[k], un[k]));  // v_x on the face
    cells(sq + ts * PN + 4 * g, q);
    edge_fluxes<LIM>(q, u, c_half, f);
    at4(sf + ts * PN + 4 * g) = make_float4(f[0], f[1], f[2], f[3]);
  }
  __syncthreads();
  // finish: 4 cells per thread and pencil
  const int quads = S / 4;
  for (int t = tid; t < M::C * quads; t += T) {
    const int c = t / quads, g = t - c * quads;
    const int row = c / LX, col = c - row * LX;
    if (a0 + col >= nA || b0 + row >= nO) continue;
    // edges below the 4 cells and above the last: F[0..4]
    auto edges = [&](int ts, float (&F)[5]) {
      float* s = sf + ts * PN;
      const float4 z = at4(s + 4 * g);
      if (e0) {
        F[0] = s[g ? 4 * g - 1 : S - 1];
        F[1] = z.x, F[2] = z.y, F[3] = z.z, F[4] = z.w;
      } else {
        F[0] = z.x, F[1] = z.y, F[2] = z.z, F[3] = z.w;
        F[4] = s[4 * g + 4];
      }
    };
    const int qa = row * (LX + 1) + col, qo = M::QA + row * LX + col;
    float fa[5], fo[5], fa1[5], fo1[5], rA[4], rO[4], rD[4];
    edges(qa, fa);
    edges(qo, fo);
    edges(qa + 1, fa1);
    edges(qo + LX, fo1);
    const float4 bA = at4(sq + qa * PN + H + 4 * g), bO = at4(sq + qo * PN + H + 4 * g),
                 bD = at4(sb + c * PN + H + 4 * g);
#pragma unroll
    for (int k = 0; k < 4; k++) {
      rA[k] = __fmaf_rn(-c_full, __fsub_rn(fa[k + 1], fa[k]), (&bA.x)[k]);
      rO[k] = __fmaf_rn(-c_full, __fsub_rn(fo[k + 1], fo[k]), (&bO.x)[k]);
      rD[k] = constrain((&bD.x)[k], kA, fa[k], fa1[k], kO, fo[k], fo1[k], true);
    }
    const unsigned o = (unsigned)((a0 + col) * sA + (b0 + row) * sO + s0 + 4 * g);
    at4(a.out[1] + o) = make_float4(rA[0], rA[1], rA[2], rA[3]);
    at4(a.out[2] + o) = make_float4(rO[0], rO[1], rO[2], rO[3]);
    at4(a.out[0] + o) = make_float4(rD[0], rD[1], rD[2], rD[3]);
  }
}

template <int LX, int R>
__host__ __device__ constexpr size_t mag_tile_smem(int D, int out) {
  return sizeof(float) * (D == 0 ? MRows<LX, R>::Size : MPlane<LX, R>::Size) * mag_tile_positions(D, out);
}

// ---------------------------------------------------------------------------
// Launches: a block per run of pencils (fluid) or tile (magnetic) and segment.
template <int LIM, int FRZ, bool FSQ>
cudaError_t launch_fluid_tile(int axis, bool rate, const FluidArgs& a, cudaStream_t s) {
  if constexpr (FRZ == 2) {
    return cudaErrorInvalidValue;
  } else {
    const int A = (axis == 0) ? 1 : 0, O = (axis == 2) ? 1 : 2;
    const FluidTile t = fluid_tile_split(axis, a.box.n[axis], a.tile);
    const int threads = (t.np * t.td + 31) / 32 * 32;
    const long long pencils = (long long)a.box.n[A] * a.box.n[O];
    const dim3 grid((unsigned)((pencils + t.np - 1) / t.np), 1, t.segs);
    const size_t smem = fluid_tile_smem(threads);
    const int split = shared_split(pencils * a.box.n[axis]);
    const bool floor = a.p_floor > 0.f;
    // (blocks of more than 224 threads need their limit raised; done here for the one
    // kernel that runs: raised for all 96 of them whenever a box is created, the first
    // box of a process took 50 ms instead of 29, every other one 0.16 instead of 0.12)
    auto launch = [&](auto* kernel) {
      const cudaError_t e =
          smem > 47 * 1024 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                           : cudaSuccess;
      return e == cudaSuccess ? launch_after(true, split, kernel, grid, dim3(threads), smem, s, a) : e;
    };
#define FLUID_TILE_CASE(DD, RR, FF) \
  if (axis == DD && rate == RR && floor == FF) return launch(fluid_tile_kernel<DD, RR, FF, LIM, FRZ, FSQ>);
    FLUID_TILE_CASE(0, false, false) FLUID_TILE_CASE(0, true, false) FLUID_TILE_CASE(0, false, true)
    FLUID_TILE_CASE(0, true, true) FLUID_TILE_CASE(1, false, false) FLUID_TILE_CASE(1, true, false)
    FLUID_TILE_CASE(1, false, true) FLUID_TILE_CASE(1, true, true) FLUID_TILE_CASE(2, false, false)
    FLUID_TILE_CASE(2, true, false) FLUID_TILE_CASE(2, false, true) FLUID_TILE_CASE(2, true, true)
#undef FLUID_TILE_CASE
    return cudaErrorInvalidValue;
  }
}

template <int LIM, int LX, int R>
cudaError_t launch_mag_tile_shape(int axis, const MagArgs& a, cudaStream_t s) {
  const int A = (axis == 0) ? 1 : 0, O = (axis == 2) ? 1 : 2;
  const MagTile t = mag_tile_split(a.box.n[axis]);
  const dim3 grid((a.box.n[A] + LX - 1) / LX, (a.box.n[O] + R - 1) / R, t.segs);
  const size_t smem = mag_tile_smem<LX, R>(axis, t.out);
  constexpr int T = MTile<LX, R>::T;
  auto* pair = a.box.n[2] < mag_tile_halo(2) ? mag_tile_kernel<2, LX, R, LIM, 2, true> : mag_tile_kernel<2, LX, R, LIM, 2>;
  auto* kernel = axis == 0   ? mag_tile_x_kernel<LX, R, LIM>
                 : axis == 1 ? mag_tile_kernel<1, LX, R, LIM, 1>
                             : (a.passes == 2 ? pair : mag_tile_kernel<2, LX, R, LIM, 1>);
  return launch_after(true, shared_split((long long)a.box.n[0] * a.box.n[1] * a.box.n[2]), kernel, grid, dim3(T), smem, s,
                      a);
}

template <int LIM>
cudaError_t launch_mag_tile(int axis, const MagArgs& a, cudaStream_t s) {
  return a.tile == 1 ? launch_mag_tile_shape<LIM, 8, 2>(axis, a, s) : launch_mag_tile_shape<LIM, 16, 4>(axis, a, s);
}

// Shared-memory limits of the magnetic tile kernels that need more than 48 KB,
// raised when a box is created, before any launch.
template <int LIM>
cudaError_t prepare_mag_tile() {
  constexpr int LX = 16, R = 4;
  static_assert(mag_tile_smem<8, 2>(0, kMTileWhole) < 48 * 1024 && mag_tile_smem<8, 2>(1, kMTileWhole) < 48 * 1024);
  cudaError_t e = cudaSuccess;
  auto set = [&](auto* k, int axis) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)mag_tile_smem<LX, R>(axis, kMTileWhole));
  };
  set(mag_tile_x_kernel<LX, R, LIM>, 0);
  set(mag_tile_kernel<1, LX, R, LIM, 1>, 1);
  set(mag_tile_kernel<2, LX, R, LIM, 1>, 2);
  set(mag_tile_kernel<2, LX, R, LIM, 2>, 2);
  set(mag_tile_kernel<2, LX, R, LIM, 2, true>, 2);
  return e;
}

}  // namespace mhd
