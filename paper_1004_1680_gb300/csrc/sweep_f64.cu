// FP64 path of the grid update (an ablation: the paper computes in FP32,
// Section III).  The same scheme as the FP32 kernels (Section II.B: relaxing
// TVD fluid sweeps, advection-constraint magnetic sweeps, xyz then zyx),
// FP64 runs at a small fraction of the FP32 rate on this GPU, so the
// arithmetic, not memory traffic, bounds these kernels.
//  * Every operation is an IEEE double operation rounded once (__dadd_rn,
//    __dmul_rn, __dsqrt_rn, the quotients of div64.cuh; no multiply-add
//    contraction).
//  * Fluid sweep: one thread per cell, the intermediate values of a block's
//    pencils exchanged through shared memory.
//  * Magnetic sweep: the velocity of every cell; a flux kernel that advects
//    each transverse component (one thread per cell and component) and
//    stores its edge flux; a constraint kernel that updates b_d of every
//    cell from the stored fluxes of its pencil and the neighbouring pencils.
//  * Launched with programmatic dependent launch (24 launches a step: 16^3 292 ->
//    243 us, 64^3 1416 -> 1358).
//  * CFL rate: the largest (|v_d| + c_f*) / h_d over cells, as double bits
//    reduced with an atomic maximum (rates are >= 0).
#include <cstdint>

#include "div64.cuh"
#include "mhd_launch.h"

namespace mhd {
namespace {

__device__ __forceinline__ bool negative(double x) { return __double2hiint(x) < 0; }

// Right and left movers FR = (c u + F) / 2, FL = (c u - F) / 2 of Eq. 1-3
// projected on the sweep axis (u = rho, m_d, m_t1, m_t2, e; b = cell-centred
// b_d, b_t1, b_t2), with the freezing speed c = |v_d| + sqrt((gamma p + b^2) / rho).
__device__ __forceinline__ void movers64(const double u[5], const double b[3], double gamma, double FR[5],
                                         double FL[5]) {
  const double y = reciprocal(u[0]);
  const bool rho_ok = plain_divisor(u[0]);
  auto over_rho = [&](double x) { return rho_ok && plain_exponent(x) ? ddiv_by(x, u[0], y) : ddiv(x, u[0]); };
  const double vd = over_rho(u[1]), v1 = over_rho(u[2]), v2 = over_rho(u[3]);
  const double bb = dadd(dadd(dmul(b[0], b[0]), dmul(b[1], b[1])), dmul(b[2], b[2]));
  const double kin = dmul(0.5, dadd(dadd(dmul(u[1], vd), dmul(u[2], v1)), dmul(u[3], v2)));
  const double p = dmul(gamma - 1.0, dsub(dsub(u[4], kin), dmul(0.5, bb)));
  const double ps = dadd(p, dmul(0.5, bb));
  const double bv = dadd(dadd(dmul(b[0], vd), dmul(b[1], v1)), dmul(b[2], v2));
  double F[5];
  F[0] = u[1];
  F[1] = dsub(dadd(dmul(u[1], vd), ps), dmul(b[0], b[0]));
  F[2] = dsub(dmul(u[2], vd), dmul(b[0], b[1]));
  F[3] = dsub(dmul(u[3], vd), dmul(b[0], b[2]));
  F[4] = dsub(dmul(dadd(u[4], ps), vd), dmul(b[0], bv));
  const double c = dadd(fabs(vd), __dsqrt_rn(over_rho(dadd(dmul(gamma, p), bb))));
#pragma unroll
  for (int q = 0; q < 5; q++) {
    FR[q] = dmul(0.5, dadd(dmul(c, u[q]), F[q]));
    FL[q] = dmul(0.5, dsub(dmul(c, u[q]), F[q]));
  }
}

// Threads of a block and split of a pencil of nD cells: one thread per cell,
// np pencils, the whole periodic pencil (`whole`, up to 512 cells) or a segment of
// `out` cells with 3 halo cells at each end (the reach of both sweeps' stencils).
// Few pencils per block, down to one, cost less across the contiguous axis (their
// 8 np-byte pieces come from L2, which has time) than halo cells do in the FP64
// pipe: with at least 4 pencils a block, and segments beyond 128 cells, 256^3 took
// 106 ms per step, now 82, 384^3 336 and 282, 512^3 827 and 671 (a thread per pencil,
// marching: 106, 321, 740), 132^3 14.6 and 12.2.
constexpr int kThreads64 = 512;
struct Tile64 {
  int threads, np, td, out, segs;
  bool whole;
};
__host__ __device__ inline Tile64 tile64(int nD) {
  Tile64 t;
  t.whole = nD <= kThreads64;
  t.segs = t.whole ? 1 : (nD + kThreads64 - 7) / (kThreads64 - 6);
  t.out = (nD + t.segs - 1) / t.segs;
  t.td = t.out + (t.whole ? 0 : 6);
  t.np = (t.td <= 64 ? 256 : kThreads64) / t.td;
  t.threads = (t.np * t.td + 31) / 32 * 32;
  return t;
}

// This thread's cell: pencil (pa, pb) of the two other axes, position p along
// D (periodic), whether it exists and whether it is written; im, ip, ip2: the
// threads of cells p - 1, p + 1, p + 2 (their own thread past a segment's end:
// only halo cells read those).
struct Cell64 {
  int pa, pb, p, im, ip, ip2;
  bool live, own;
};
template <int D>
__device__ __forceinline__ Cell64 cell64(const int n[3]) {
  constexpr int A = (D == 0) ? 1 : 0, O = (D == 2) ? 1 : 2;
  const Tile64 t = tile64(n[D]);
  const int tid = threadIdx.x;
  // along x neighbouring threads take neighbouring cells, else neighbouring pencils
  const int pp = D == 0 ? tid / t.td : tid % t.np, i = D == 0 ? tid - pp * t.td : tid / t.np;
  const int step = D == 0 ? 1 : t.np;
  Cell64 c;
  const unsigned pencils = (unsigned)n[A] * (unsigned)n[O], runs = (pencils + t.np - 1) / t.np;
  const unsigned seg = blockIdx.x / runs, P = (blockIdx.x - seg * runs) * t.np + pp;
  c.live = pp < t.np && i < t.td && P < pencils;
  c.pb = (int)(P / (unsigned)n[A]);
  c.pa = (int)(P - (unsigned)c.pb * (unsigned)n[A]);
  const int off = t.whole ? i : i - 3, s0 = (int)seg * t.out;
  c.own = c.live && off >= 0 && off < t.out && s0 + off < n[D];
  c.p = wrapi(s0 + off, n[D]);
  auto nb = [&](int d) {
    int k = i + d;
    if (t.whole) k = wrapi(k, t.td);
    else k = k < 0 || k >= t.td ? i : k;
    return tid + (k - i) * step;
  };
  c.im = nb(-1);
  c.ip = nb(1);
  c.ip2 = nb(2);
  return c;
}

// Fluid sweep, one thread per cell.  FP64 arithmetic bounds it (350 operations
// per cell, 16 cycles of an SM per warp instruction: its pipe is 83 % busy), so nothing is
// computed twice but a few subtractions: the movers of both stages and the
// limited values are exchanged through shared memory, [component][thread], in
// two alternating sets.  (Marching whole pencils with one thread each left
// the FP64 pipe idle below about 150,000 pencils: 64^3 1050 us a sweep, now
// 180; at 512^3 740 ms a step, now 671.)
template <int D>
__global__ void __launch_bounds__(kThreads64, 1) fluid64_kernel(const __grid_constant__ Fluid64Args a) {
  wait_for_previous();
  constexpr int A = (D == 0) ? 1 : 0, O = (D == 2) ? 1 : 2, T1 = (D + 1) % 3, T2 = (D + 2) % 3;
  extern __shared__ double sm64[];
  const int T = blockDim.x;
  double* x0 = sm64;                     // FR, FL, then the limited right and left values
  double* x1 = sm64 + 10 * T;   // Rh, Lh
  const long long st[3] = {1, a.n[0], (long long)a.n[0] * a.n[1]};
  const Cell64 c = cell64<D>(a.n);
  const int tid = threadIdx.x;
  const double c_full = dmul(a.tau, a.ih[D]), c_half = dmul(0.5, c_full);
  const long long cell = c.pa * st[A] + c.pb * st[O] + c.p * st[D];
  double U[5], b[3], FR[5], FL[5];
  if (c.live) {
    auto up = [&](int d, int x) { return cell + (x + 1 == a.n[d] ? -(long long)x : 1) * st[d]; };
    const long long cD = up(D, c.p), cA = up(A, c.pa), cO = up(O, c.pb);
    const long long c1 = T1 == A ? cA : cO, c2 = T2 == A ? cA : cO;
    U[0] = a.in[RHO][cell], U[1] = a.in[MX + D][cell], U[2] = a.in[MX + T1][cell], U[3] = a.in[MX + T2][cell];
    U[4] = a.in[EN][cell];
    b[0] = dmul(0.5, dadd(a.in[BX + D][cell], a.in[BX + D][cD]));
    b[1] = dmul(0.5, dadd(a.in[BX + T1][cell], a.in[BX + T1][c1]));
    b[2] = dmul(0.5, dadd(a.in[BX + T2][cell], a.in[BX + T2][c2]));
    movers64(U, b, a.gamma, FR, FL);
#pragma unroll
    for (int q = 0; q < 5; q++) {
      x0[q * T + tid] = FR[q];
      x0[(5 + q) * T + tid] = FL[q];
    }
  }
  __syncthreads();
  if (c.live) {
    double Uh[5];
#pragma unroll
    for (int q = 0; q < 5; q++) {  // first-order fluxes at p +- 1/2, half step
      const double hi = dsub(FR[q], x0[(5 + q) * T + c.ip]);
      const double lo = dsub(x0[q * T + c.im], FL[q]);
      Uh[q] = dsub(U[q], dmul(c_half, dsub(hi, lo)));
    }
    movers64(Uh, b, a.gamma, FR, FL);
#pragma unroll
    for (int q = 0; q < 5; q++) {
      x1[q * T + tid] = FR[q];
      x1[(5 + q) * T + tid] = FL[q];
    }
  }
  __syncthreads();
  if (c.live) {
#pragma unroll
    for (int q = 0; q < 5; q++) {  // the right mover extrapolated to p + 1/2, the left one to p - 1/2
      const double *R = x1 + q * T, *L = x1 + (5 + q) * T;
      FR[q] = dadd(FR[q], vl_half(dsub(FR[q], R[c.im]), dsub(R[c.ip], FR[q])));
      FL[q] = dsub(FL[q], vl_half(dsub(FL[q], L[c.im]), dsub(L[c.ip], FL[q])));
      x0[q * T + tid] = FR[q];
      x0[(5 + q) * T + tid] = FL[q];
    }
  }
  __syncthreads();
  if (c.own) {
    double o[5];
#pragma unroll
    for (int q = 0; q < 5; q++) {
      const double hi = dsub(FR[q], x0[(5 + q) * T + c.ip]);  // second-order flux at p + 1/2
      const double lo = dsub(x0[q * T + c.im], FL[q]);        // and at p - 1/2
      o[q] = dsub(U[q], dmul(c_full, dsub(hi, lo)));
    }
    a.out[RHO][cell] = o[0];
    a.out[MX + D][cell] = o[1];
    a.out[MX + T1][cell] = o[2];
    a.out[MX + T2][cell] = o[3];
    a.out[EN][cell] = o[4];
  }
}

// v_D of every cell, once per magnetic sweep.
__global__ void __launch_bounds__(256) velocity64_kernel(const double* __restrict__ m, const double* __restrict__ rho,
                                                         double* __restrict__ v, long long N) {
  wait_for_previous();
  for (long long c = (long long)blockIdx.x * 256 + threadIdx.x; c < N; c += (long long)gridDim.x * 256)
    v[c] = ddiv(m[c], rho[c]);
}

// (with the flux kernel and the constraint below: 64^3 218 us a sweep, now 51)
//
// Advection of b_t along D for one transverse axis t (blockIdx.z: 0 -> T1,
// 1 -> T2), one thread per cell: new b_t into out[BX + t], edge fluxes into
// E[blockIdx.z] (the flux of edge i + 1/2 of a pencil stored at its cell i).
template <int D>
__global__ void __launch_bounds__(kThreads64) mag64_flux_kernel(const __grid_constant__ Mag64Args a) {
  wait_for_previous();
  constexpr int A = (D == 0) ? 1 : 0, O = (D == 2) ? 1 : 2;
  __shared__ double su[kThreads64], sq[kThreads64], sh[kThreads64], sf[kThreads64];
  const long long st[3] = {1, a.n[0], (long long)a.n[0] * a.n[1]};
  const Cell64 c = cell64<D>(a.n);
  const int tid = threadIdx.x;
  const int t = (blockIdx.z == 0) ? (D + 1) % 3 : (D + 2) % 3;
  const double c_full = dmul(a.tau, a.ih[D]), c_half = dmul(0.5, c_full);
  const long long cell = c.pa * st[A] + c.pb * st[O] + c.p * st[D];
  double q = 0.0, u = 0.0;
  if (c.live) {
    // the pencil one cell down along t (the other side of the b_t face)
    const long long down = cell + (t == A ? (c.pa ? -1 : a.n[A] - 1) * st[A] : (c.pb ? -1 : a.n[O] - 1) * st[O]);
    q = a.in[BX + t][cell];
    u = dmul(0.5, dadd(a.v[cell], a.v[down]));  // v_D on the b_t face
    su[tid] = u;
    sq[tid] = q;
  }
  __syncthreads();
  double ub = 0.0, h = 0.0;
  if (c.live) {
    ub = dmul(0.5, dadd(u, su[c.ip]));                                   // edge velocity at p + 1/2
    const double um = dmul(0.5, dadd(su[c.im], u));                      // and at p - 1/2
    const double g = dmul(ub, negative(ub) ? sq[c.ip] : q), gm = dmul(um, negative(um) ? q : sq[c.im]);  // upwind fluxes
    h = dsub(q, dmul(c_half, dsub(g, gm)));                              // half step
    sh[tid] = h;
  }
  __syncthreads();
  double f = 0.0;
  if (c.live) {
    const double hm = sh[c.im], hp = sh[c.ip], hpp = sh[c.ip2];
    const bool pos = !negative(ub);
    const double base = pos ? h : hp;  // the upwind cell and the ones below and above it
    const double lim = vl_half(dsub(base, pos ? hm : h), dsub(pos ? hp : hpp, base));
    f = dmul(ub, pos ? dadd(base, lim) : dsub(base, lim));
    sf[tid] = f;
  }
  __syncthreads();
  if (c.own) {
    a.out[BX + t][cell] = dsub(q, dmul(c_full, dsub(f, sf[c.im])));
    a.E[blockIdx.z][cell] = f;  // edge p + 1/2
  }
}

// b_D of every cell (low face i along D) takes the edge fluxes of edge
// i - 1/2 of its pencil and of the next pencil along each transverse axis:
// b_D += tau/h_t (E_t(pencil + e_t) - E_t(pencil)), t = T1 then T2.
template <int D>
__global__ void __launch_bounds__(256) mag64_constraint_kernel(Mag64Args a) {
  wait_for_previous();
  const int N = a.n[0] * a.n[1] * a.n[2];
  const int s[3] = {1, a.n[0], a.n[0] * a.n[1]};
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
    int x[3] = {c % a.n[0], (c / a.n[0]) % a.n[1], c / (a.n[0] * a.n[1])};
    int em[3] = {x[0], x[1], x[2]};
    em[D] = wrapi(x[D] - 1, a.n[D]);  // the cell whose edge flux is edge i - 1/2
    const int ce = em[0] * s[0] + em[1] * s[1] + em[2] * s[2];
    double b = a.in[BX + D][c];
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const int t = (D + 1 + k) % 3;
      int ep[3] = {em[0], em[1], em[2]};
      ep[t] = wrapi(em[t] + 1, a.n[t]);
      const int cp = ep[0] * s[0] + ep[1] * s[1] + ep[2] * s[2];
      b = dadd(b, dmul(dmul(a.tau, a.ih[t]), dsub(a.E[k][cp], a.E[k][ce])));
    }
    a.out[BX + D][c] = b;
  }
}

__global__ void __launch_bounds__(256) cfl64_kernel(const double* __restrict__ rho, const double* __restrict__ mx,
                                                    const double* __restrict__ my, const double* __restrict__ mz,
                                                    const double* __restrict__ en, const double* __restrict__ bx,
                                                    const double* __restrict__ by, const double* __restrict__ bz,
                                                    int nx, int ny, int nz, double ihx, double ihy, double ihz,
                                                    double gamma, unsigned long long* rate) {
  wait_for_previous();
  const int N = nx * ny * nz;
  double rmax = 0.0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
    const int i = c % nx, j = (c / nx) % ny, k = c / (nx * ny);
    const int cx = c - i + wrapi(i + 1, nx), cy = c + (wrapi(j + 1, ny) - j) * nx, cz = c + (wrapi(k + 1, nz) - k) * nx * ny;
    const double b[3] = {dmul(0.5, dadd(bx[c], bx[cx])), dmul(0.5, dadd(by[c], by[cy])), dmul(0.5, dadd(bz[c], bz[cz]))};
    const double m[3] = {mx[c], my[c], mz[c]};
    const double r = rho[c];
    const double y = reciprocal(r);
    const bool r_ok = plain_divisor(r);
    auto over_rho = [&](double x) { return r_ok && plain_exponent(x) ? ddiv_by(x, r, y) : ddiv(x, r); };
    double v[3], bb = 0.0, kin = 0.0;
#pragma unroll
    for (int d = 0; d < 3; d++) {
      v[d] = over_rho(m[d]);
      bb = dadd(bb, dmul(b[d], b[d]));
      kin = dadd(kin, dmul(0.5, dmul(m[d], v[d])));
    }
    const double p = dmul(gamma - 1.0, dsub(dsub(en[c], kin), dmul(0.5, bb)));
    const double cf = __dsqrt_rn(over_rho(dadd(dmul(gamma, p), bb)));
    double rc = fmax(fmax(dmul(dadd(fabs(v[0]), cf), ihx), dmul(dadd(fabs(v[1]), cf), ihy)),
                     dmul(dadd(fabs(v[2]), cf), ihz));
    if (!(r > 0.0) || !(p > 0.0) || !(rc <= 1.0e300)) rc = __longlong_as_double(0x7ff0000000000000LL);
    rmax = fmax(rmax, rc);
  }
  for (int o = 16; o > 0; o >>= 1) rmax = fmax(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
  if ((threadIdx.x & 31) == 0) atomicMax(rate, (unsigned long long)__double_as_longlong(rmax));
}

}  // namespace

namespace {
dim3 grid64(int axis, const int n[3], int z) {
  const int A = (axis == 0) ? 1 : 0, O = (axis == 2) ? 1 : 2;
  const Tile64 t = tile64(n[axis]);
  const long long pencils = (long long)n[A] * n[O];
  return dim3((unsigned)((pencils + t.np - 1) / t.np * t.segs), 1, z);  // segment by segment
}
int fluid64_smem(int threads) { return 20 * threads * (int)sizeof(double); }
}  // namespace

cudaError_t prepare_f64_kernels() {
  cudaError_t e = cudaSuccess;
  for (auto* k : {fluid64_kernel<0>, fluid64_kernel<1>, fluid64_kernel<2>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                      fluid64_smem(kThreads64));
  return e;
}

cudaError_t launch_fluid64(int axis, const Fluid64Args& a, cudaStream_t s) {
  const dim3 grid = grid64(axis, a.n, 1);
  const int threads = tile64(a.n[axis]).threads, smem = fluid64_smem(threads);
  auto* kernel = axis == 0 ? fluid64_kernel<0> : (axis == 1 ? fluid64_kernel<1> : fluid64_kernel<2>);
  return launch_after(true, kernel, grid, dim3(threads), smem, s, a);
}

cudaError_t launch_mag64(int axis, const Mag64Args& a, cudaStream_t s) {
  const dim3 grid = grid64(axis, a.n, 2);
  const int threads = tile64(a.n[axis]).threads;
  const long long N = (long long)a.n[0] * a.n[1] * a.n[2];
  const int cblocks = (int)((N + 255) / 256 < 152 * 16 ? (N + 255) / 256 : 152 * 16);
  auto* flux = axis == 0 ? mag64_flux_kernel<0> : (axis == 1 ? mag64_flux_kernel<1> : mag64_flux_kernel<2>);
  auto* constraint =
      axis == 0 ? mag64_constraint_kernel<0> : (axis == 1 ? mag64_constraint_kernel<1> : mag64_constraint_kernel<2>);
  cudaError_t e = launch_after(true, velocity64_kernel, dim3(cblocks), dim3(256), 0, s,
                               static_cast<const double*>(a.in[MX + axis]), static_cast<const double*>(a.in[RHO]), a.v, N);
  if (e == cudaSuccess) e = launch_after(true, flux, grid, dim3(threads), 0, s, a);
  if (e == cudaSuccess) e = launch_after(true, constraint, dim3(cblocks), dim3(256), 0, s, a);
  return e;
}

cudaError_t launch_cfl64(const double* const f[8], const int n[3], const double ih[3], double gamma,
                         unsigned long long* rate, cudaStream_t s) {
  const long long N = (long long)n[0] * n[1] * n[2];
  const int blocks = (int)((N + 255) / 256 < 152 * 8 ? (N + 255) / 256 : 152 * 8);
  cfl64_kernel<<<blocks, 256, 0, s>>>(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], n[0], n[1], n[2], ih[0],
                                      ih[1], ih[2], gamma, rate);
  return cudaGetLastError();
}

}  // namespace mhd
