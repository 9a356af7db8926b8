// Kernel argument blocks and host-side launchers shared by the library's
// translation units (internal; the public interface is include/mhd.h).
#pragma once
#include <cuda.h>  // CUtensorMap (the maps are encoded through the runtime's driver entry point)
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "mhd_device.cuh"

namespace mhd {

constexpr int kMagWarps = 8;  // interior rows of a magnetic-sweep tile
// Rows per tile of the magnetic row sweep: 4 for rows of up to 512 cells (5
// groups of nx/4 threads, 640 threads), 3 below 640 (4 groups of 160, 640 again:
// two rows leave 480 threads on an SM; sweep of 528^3 1.73 -> 1.24 ms, of 560 x
// 300 x 200 412 -> 279 us), 2 up to 1024 cells (3 groups of 256 threads, 768).
__host__ __device__ constexpr int mag_row_tile(int nx) { return nx <= 512 ? 4 : (nx < 640 ? 3 : 2); }
// Estimated microseconds of the magnetic row sweep of a box (sweep_mag.cu).
double mag_rows_us(const int n[3], int sms);

// One box of an ensemble: physical extents, first cell in the concatenated
// field arrays (a multiple of 32), and pencil segment length per axis of its
// fluid and magnetic sweeps (the last segment of a pencil may be shorter).
struct EnsBox {
  int n[3];
  int offset;
  int seg[2][3];
  int pad[2];
};

// Ensemble launches (items != nullptr): block b of the grid works on
// items[b] = (box, block x, block y, block z) of that box; the box geometry
// comes from boxes[box] (exchanged x and y when layout == 1), its sweep step
// from tau_arr[box] and its CFL accumulator is rate_arr[box].
struct EnsArgs {
  const int4* items = nullptr;
  const EnsBox* boxes = nullptr;
  const float* tau_arr = nullptr;
  unsigned* rate_arr = nullptr;
  int layout = 0;
  int kind = 0;  // 0: fluid sweep, 1: magnetic
  int phys_axis = 0;
};

// Programmatic dependent launch of the sweeps of a step (single boxes): a
// sweep may be launched while the one before it drains, so the launch itself
// (about 2 us between dependent kernels otherwise) is hidden; it waits here,
// before its first access to device memory, until the kernels before it in the
// stream have completed and their writes are visible.  It lets its own
// dependent launch only after that wait, so at most two sweeps are on the chip
// and no block of a third can have cached what the second one writes.  Nor may
// the second one itself: a kernel that lets the next one in reads nothing that
// it writes, other than past L1 (step_begin, the floor of the marching sweeps);
// kernels that update in place let it in when they have completed.
// (The network's kernels as well: the gradients of one 64^3 pair, 18 launches,
// 342 -> 306 us.  Not the ensembles' launches, which a graph replays: 3 boxes 234
// us per step, 314 with it; the blocks of a small launch, let in early, pile up
// on the SMs that are free first.)
// 20 steps of 32^3 (13 launches each) 1.65 -> 1.00 ms, 40 steps of a 512 x 8 x
// 8 tube with open ends 6.19 -> 3.79 ms, 10 steps of 128^3 3.51 -> 3.34 ms.
__device__ __forceinline__ void wait_for_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// The tile sweeps and the ghost fill form their indexes before that wait, while
// the kernel before them still runs (several integer divisions, 0.3 us of a
// 3.3 us sweep: 32^3 43.6 -> 40.6 us per step, 64^3 91 -> 85.5, the tube 78 ->
// 72.5); `settled` keeps the compiler from moving them behind it.  The marching
// sweeps wait first: values live across the wait spill there (256^3 along y
// 172 -> 180 us).
__device__ __forceinline__ void settle(int& v) { asm volatile("" : "+r"(v)); }
__device__ __forceinline__ void settle(unsigned& v) { asm volatile("" : "+r"(v)); }
template <class... V>
__device__ __forceinline__ void settled(V&... v) {
  (settle(v), ...);
}
// For kernels that write in place what they may have cached: the dependent
// launches when they have completed.
__device__ __forceinline__ void wait_for_previous_in_place() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch a kernel that begins with one of the two; `early` = false gives an
// ordinary launch (the wait then has nothing to wait for).
//
// `split`: the share of an SM's memory (in percent) to be shared memory, 0 for the
// driver's choice.  A kernel that asks for another split than the one before
// cannot start beside it, and in small boxes that beginning is a good part of a
// sweep; left alone, the fluid tiles get 132 KB, the magnetic ones 196.  132 KB
// hold a block of 16 x 4 magnetic tiles or four fluid blocks (64^3 86 -> 68 us
// per step, 48^3 70 -> 57, 40^3 61 -> 48, 128 x 64 x 32 82 -> 64), 164 KB two
// magnetic blocks, which larger boxes need (68^3 115 -> 95, 72^3 119 -> 97; with
// 132 KB 105 and 108).  Beyond that a sweep takes so long that its beginning
// counts less than L1 or a second block (76^3 111 either way, 96^3 174 and 184).
inline int shared_split(long long cells) { return cells <= 280000 ? 50 : (cells <= 450000 ? 65 : 0); }
template <class... P>
inline cudaError_t launch_after(bool early, int split, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                                cudaStream_t s, P... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at[2] = {};
  if (early) {
    at[c.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[c.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (split) {
    at[c.numAttrs].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    at[c.numAttrs++].val.sharedMemCarveout = (unsigned)split;
  }
  c.attrs = at;
  return cudaLaunchKernelEx(&c, kernel, args...);
}
template <class... P>
inline cudaError_t launch_after(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                P... args) {
  return launch_after(early, 0, kernel, grid, block, smem, s, args...);
}

// Split of a fluid tile sweep (sweep_tile.cuh) along a pencil of nD cells for
// blocks of `threads` threads: td threads of 4 cells per pencil, np pencils
// per block, segs segments of `out` positions.  `whole`: one segment that is
// the whole periodic pencil; otherwise a segment has one thread of halo cells
// at each end.  At least 8 pencils per block (32-byte sectors of neighbouring
// pencils); used on the host for grids.
constexpr int kTileThreads = 256;
constexpr int kTileCells = 4;  // cells per thread
struct FluidTile {
  int td, np, segs, out;
  bool whole;
};
__host__ __device__ inline FluidTile fluid_tile_split(int axis, int nD, int threads) {
  constexpr int K = kTileCells;
  FluidTile s;
  const int tmax = threads / (axis == 0 ? 2 : 8);
  s.whole = nD % K == 0 && nD / K <= tmax;
  if (s.whole) {
    s.segs = 1;
    s.out = nD;
    s.td = nD / K;
  } else {
    const int most = K * (tmax - 2);
    s.segs = (nD + most - 1) / most;
    s.out = ((nD + s.segs - 1) / s.segs + 3) / 4 * 4;
    s.segs = (nD + s.out - 1) / s.out;
    s.td = s.out / K + 2;
  }
  s.np = threads / s.td;
  if (s.np > 4) s.np &= ~3;
  return s;
}
// Split of a magnetic tile sweep along a pencil of nD cells: segs segments
// of `out` positions (a multiple of 4 unless whole), whole pencils of up to
// kMTileWhole cells.
constexpr int kMTileWhole = 40, kMTileOut = 32;
struct MagTile {
  int segs, out;
  bool whole;
};
__host__ __device__ inline MagTile mag_tile_split(int nD) {
  MagTile s;
  s.whole = nD <= kMTileWhole;
  s.segs = s.whole ? 1 : (nD + kMTileOut - 1) / kMTileOut;
  s.out = s.whole ? nD : ((nD + s.segs - 1) / s.segs + 3) / 4 * 4;
  s.segs = (nD + s.out - 1) / s.out;
  return s;
}
// Positions that a tile sweep along a pencil of nD cells computes per cell of
// it: the fluid sweep's groups of 4 cells and halo threads (12 for a pencil of
// one cell, 1 for whole pencils of a multiple of 4), the magnetic sweep's groups
// of 4 edges of a whole pencil.
inline double fluid_tile_padding(int axis, int nD, int threads) {
  const FluidTile t = fluid_tile_split(axis, nD, threads);
  return (double)t.td * kTileCells * t.segs / nD;
}
inline double mag_tile_padding(int nD) { return nD <= kMTileWhole ? (nD + 3) / 4 * 4.0 / nD : 1.0; }

// What a step begins with: its sweep step tau = cfl / rate (0 for an invalid
// state: stand still), or tau_host where cfl <= 0, the time, and the next CFL
// accumulator.  A launch of its own, or done by the step's first sweep: every
// block of a fluid tile sweep along x forms tau from the rate, and one writes it
// for the sweeps that follow (32^3 40.8 -> 40.0 us per
// step, 64^3 67.6 -> 65.7, 96^3 173.8 -> 171.4).
struct StepControl {
  const unsigned* rate = nullptr;
  unsigned* rate_next = nullptr;
  float* tau = nullptr;
  double* time = nullptr;
  double cfl = 0.0, tau_host = 0.0;
};
#ifdef __CUDACC__
__device__ __forceinline__ float step_tau(const StepControl& c) {
  double t = c.tau_host;
  if (c.cfl > 0.0) {
    const float r = __uint_as_float(__ldcg(c.rate));
    t = (r > 0.f && r <= 3.402823466e+38f) ? c.cfl / (double)r : 0.0;  // invalid state: stand still
  }
  return (float)t;
}
__device__ __forceinline__ void step_begin(const StepControl& c, float tau) {
  *c.tau = tau;
  *c.time = __ldcg(c.time) + 2.0 * (double)tau;
  *c.rate_next = 0u;
}
#endif

struct FluidArgs {
  const float* in[8];  // current fields
  float* out[8];       // destinations of fields 0..4 (others unused)
  Box box;
  float gamma;
  float p_floor = 0.f; // optional floor on the gas pressure of the output (0: off)
  float e_floor = 0.f; // its internal energy, p_floor / (gamma - 1)
  const float* tau;    // device scalar: step of this sweep
  unsigned* rate;      // fused CFL rate accumulator (float bits), or nullptr
  int seg;             // pencil segment length along the sweep axis
  EnsArgs ens;         // ensemble launches only
  int nblocks = 0;     // ensemble launches: number of work items
  int lim = 0;         // slope limiter: 0 van Leer (the paper's), 1 minmod, 2 superbee
  int fast = 0;        // freezing speed: 0 the bound, 1 the fast magnetosonic speed, 2 per pencil
  const float* pencil_c = nullptr;  // fast == 2: per-pencil speeds, stage 1 then stage 2 (nA * nO each)
  // cells [rate_lo, rate_hi) per kernel axis enter the fused rate (the
  // interior of a box with ghost layers; every cell by default)
  int rate_lo[3] = {0, 0, 0};
  int rate_hi[3] = {1 << 30, 1 << 30, 1 << 30};
  int tma = 0;              // 1: stage chunks with tensor-tile copies where the sweep qualifies
  unsigned* err = nullptr;  // set to 1 (atomicOr) if a staged chunk did not arrive within the bound
  int* tma_used = nullptr;  // host: set to 1 when the launch was TMA-staged
  StepControl control;      // rate != nullptr: the first sweep of a step begins it (tile sweeps along x)
  int tile = 0;             // > 0: tile sweep with blocks of up to that many threads
};

// Tensor maps of a TMA-staged fluid sweep (kernel axes 1 and 2), dimensions
// ordered (lane axis A, row axis O, sweep axis D).  full[]: one chunk of 4
// positions, for rho, m_d, m_t1, m_t2, e, b_A, b_O (32 x 4 x 4), b_d
// (32 x 4 x 5), b_A of the next block's first 4 lanes (4 x 4 x 4; only its
// row form is used) and b_O of its first row (32 x 1 x 4); row[]: the same
// boxes one position long.
// A 3-D tensor map of FP32 elements: tensor extents dim (the first
// contiguous), byte strides st of dimensions 1 and 2, box b0 x b1 x b2;
// out-of-range elements read as zero.  False if the driver's encoder is
// unavailable or rejects the map (tma_maps.cu).
bool tma_encode_f32(CUtensorMap* m, const float* p, const cuuint64_t dim[3], const cuuint64_t st[2], cuuint32_t b0,
                    cuuint32_t b1, cuuint32_t b2);

constexpr int kFluidMaps = 10;
struct FluidMaps {
  CUtensorMap full[kFluidMaps];
  CUtensorMap row[kFluidMaps];
};
// Encode the maps of a sweep along kernel axis 1 or 2; false if the box does
// not qualify (rows not a multiple of 16 bytes, unaligned fields, pencils
// shorter than 16 cells) or the driver's encoder is unavailable.  Lane and
// row extents need not fill the 32 x 4 tiles.
bool make_fluid_maps(int axis, const FluidArgs& a, FluidMaps* m);
bool fluid_chunks_qualify(int axis, const FluidArgs& a);  // the box's part of that

struct MagArgs {
  const float* in[8];
  float* out[3];       // destinations of b_x, b_y, b_z
  Box box;
  const float* tau;
  int seg;
  EnsArgs ens;
  int nblocks = 0;
  int lim = 0;         // slope limiter (as FluidArgs::lim)
  int passes = 1;      // 2: two sweeps with the same step in one launch (kernel axis 2 only)
  int tma = 0;              // 1: stage chunks with tensor-tile copies where the sweep qualifies
  unsigned* err = nullptr;  // set to 1 (atomicOr) if a staged chunk did not arrive within the bound
  int* tma_used = nullptr;  // host: set to 1 when the launch was TMA-staged
  int tile = 0;             // 1: tile sweep
};

// Ghost layers of the non-periodic axes (boundary.cu) of the fields as stored
// in `box`: mode per kernel axis k (0 periodic, 1 outflow, 2 reflecting), whose
// normal momentum and face field are f[1 + k] and f[5 + k].
constexpr int kGhost = 4;
enum { kGhostFluid = 1, kGhostField = 2, kGhostAll = 3 };  // rho, m, e; b
struct GhostArgs {
  float* f[8];
  int parts;  // the fields to fill
  int n[3], mode[3];
  long long stride[3];
  long long first[4];  // elements (or groups of them) of the axes' ghost layers, accumulated
};
cudaError_t launch_ghost_fill(float* const f[8], const Box& box, const int mode[3], int parts, cudaStream_t s);

struct TransposeArgs {
  const float* in[8];
  float* out[8];
  int n[3];  // input extents, fastest first; the output has n[1] fastest
  EnsArgs ens;   // ensemble: items = (box, tile i, tile j, k); layout = input layout
  int nblocks = 0;
};

// A box of nx x ny x nz cells, x fastest, on the periodic unit cube.
inline Box make_box(int nx, int ny, int nz) {
  Box b;
  b.n[0] = nx;
  b.n[1] = ny;
  b.n[2] = nz;
  b.stride[0] = 1;
  b.stride[1] = nx;
  b.stride[2] = (long long)nx * ny;
  b.ih[0] = (float)nx;
  b.ih[1] = (float)ny;
  b.ih[2] = (float)nz;
  return b;
}

// Resolved geometry of the block a kernel is running: the box as the kernel
// sees it, the block's coordinates, segment, step and CFL accumulator, and
// the offset of the box in the field arrays.
struct BlockGeom {
  Box box;
  int bx, by, bz;
  int seg;
  int off;
  float tau;
  unsigned* rate;
};

__device__ __forceinline__ BlockGeom block_geom(const EnsArgs& e, const Box& box, int seg,
                                                const float* tau, unsigned* rate) {
  BlockGeom g;
  if (e.items) {
    const int4 it = e.items[blockIdx.x];
    const EnsBox eb = e.boxes[it.x];
    const int n0 = e.layout ? eb.n[1] : eb.n[0];
    const int n1 = e.layout ? eb.n[0] : eb.n[1];
    g.box.n[0] = n0;
    g.box.n[1] = n1;
    g.box.n[2] = eb.n[2];
    g.box.stride[0] = 1;
    g.box.stride[1] = n0;
    g.box.stride[2] = (long long)n0 * n1;
    g.box.ih[0] = (float)n0;  // ensemble boxes are periodic unit boxes
    g.box.ih[1] = (float)n1;
    g.box.ih[2] = (float)eb.n[2];
    g.bx = it.y;
    g.by = it.z;
    g.bz = it.w;
    g.seg = eb.seg[e.kind][e.phys_axis];
    g.off = eb.offset;
    g.tau = tau ? e.tau_arr[it.x] : 0.f;
    g.rate = e.rate_arr ? e.rate_arr + it.x : nullptr;
  } else {
    g.box = box;
    g.bx = blockIdx.x;
    g.by = blockIdx.y;
    g.bz = blockIdx.z;
    g.seg = seg;
    g.off = 0;
    g.tau = tau ? *tau : 0.f;
    g.rate = rate;
  }
  return g;
}

// Record "<where>: <what>" as this thread's last error (mhd_last_error) and
// return code.
int set_error(int code, const char* where, const char* what);

// 3x3x3 periodic convolution on the tensor cores (conv3d.cu).
struct ConvArgs {
  const __nv_bfloat16* x;     // input, channels-last [cell][cin] BF16
  const uint16_t* wpack;      // packed weight image (launch_conv_pack)
  const float* bias;          // [cout] or nullptr
  __nv_bfloat16* y;           // output [cell][cout] BF16, or nullptr
  float* y32;                 // output [cell][cout] FP32, or nullptr
  const __nv_bfloat16* mask;  // zero outputs where mask[cell][co] <= 0 (ReLU backward), or nullptr
  int n[3];
  int cin;                    // input channels per cell (8 or 32)
  int cout;                   // channels written per cell
  int npad, kchunks;          // MMA N and number of 32-wide k chunks
  int relu;
  int flip;                   // 1: input gradient (the mirrored taps come with the transposed pack)
  int* err;                   // set to 1 if a bounded wait gives up
};
int conv_npad(int n);
int conv_kchunks(int c);
size_t conv_image_bytes(int rows, int cols);
size_t conv_smem_bytes(int npad, int kchunks, int cin, int ty);
cudaError_t prepare_conv_kernels();
cudaError_t launch_conv_pack(const float* w, int cin, int cout, int transpose, uint16_t* img, cudaStream_t s);
cudaError_t launch_conv3d(const ConvArgs& a, cudaStream_t s);
cudaError_t launch_conv_wgrad(const __nv_bfloat16* x, const __nv_bfloat16* gy, const int n[3], int cin, int cout,
                              float* gw, float* gb, int* err, cudaStream_t s);
cudaError_t launch_conv_wgrad_cuda_cores(const __nv_bfloat16* x, const __nv_bfloat16* gy, const int n[3], int cin,
                                         int cout, float* gw, float* gb, cudaStream_t s);

// FP64 path (sweep_f64.cu): kernels on the plain layout, a thread per cell
struct Fluid64Args {
  const double* in[8];
  double* out[8];  // fields 0..4 written
  int n[3];
  double ih[3];    // cells per unit length
  double gamma;
  double tau;
};
struct Mag64Args {
  const double* in[8];
  double* out[8];  // fields 5..7 written
  double* E[2];    // edge fluxes of the transverse axes (D+1)%3, (D+2)%3 (N each)
  double* v;       // scratch: v_D of every cell (N)
  int n[3];
  double ih[3];
  double tau;
};
cudaError_t prepare_f64_kernels();  // once per device before any launch
cudaError_t launch_fluid64(int axis, const Fluid64Args& a, cudaStream_t s);
cudaError_t launch_mag64(int axis, const Mag64Args& a, cudaStream_t s);
cudaError_t launch_cfl64(const double* const f[8], const int n[3], const double ih[3], double gamma,
                         unsigned long long* rate, cudaStream_t s);

// launchers (return cudaGetLastError of the launch)
cudaError_t launch_transpose01(const TransposeArgs& a, cudaStream_t s);
cudaError_t launch_transpose02(const TransposeArgs& a, cudaStream_t s);  // single box only
// ensemble step control: for every box b < nbox, tau[b] = cfl / rate_cur[b]
// (0 for an invalid state), time[b] += 2 tau[b], rate_next[b] = 0
cudaError_t launch_ens_control(const unsigned* rate_cur, unsigned* rate_next, float* tau,
                               double* time, int nbox, double cfl, cudaStream_t s);
cudaError_t launch_fluid(int axis, bool rate, const FluidArgs& a, cudaStream_t s);
cudaError_t launch_mag(int axis, const MagArgs& a, cudaStream_t s);
// one instantiation per scheme variant, each in its own translation unit
template <int LIM, int FRZ>
cudaError_t launch_fluid_t(int axis, bool rate, const FluidArgs& a, cudaStream_t s);
// per-pencil freezing speeds of a fluid sweep along kernel axis `axis`
// (sweep_pencil.cu): c[pencil] = largest bound along the pencil for U, then
// c[nA nO + pencil] for the stage-1 half-step state built with it
cudaError_t launch_pencil_speeds(int axis, const FluidArgs& a, float* c, cudaStream_t s);
template <int LIM>
cudaError_t launch_mag_t(int axis, const MagArgs& a, cudaStream_t s);
template <int LIM>
cudaError_t prepare_mag_t();
extern template cudaError_t launch_fluid_t<0, 0>(int, bool, const FluidArgs&, cudaStream_t);
extern template cudaError_t launch_fluid_t<1, 0>(int, bool, const FluidArgs&, cudaStream_t);
extern template cudaError_t launch_fluid_t<2, 0>(int, bool, const FluidArgs&, cudaStream_t);
extern template cudaError_t launch_fluid_t<0, 1>(int, bool, const FluidArgs&, cudaStream_t);
extern template cudaError_t launch_fluid_t<0, 2>(int, bool, const FluidArgs&, cudaStream_t);
extern template cudaError_t launch_mag_t<0>(int, const MagArgs&, cudaStream_t);
extern template cudaError_t launch_mag_t<1>(int, const MagArgs&, cudaStream_t);
extern template cudaError_t launch_mag_t<2>(int, const MagArgs&, cudaStream_t);
extern template cudaError_t prepare_mag_t<0>();
extern template cudaError_t prepare_mag_t<1>();
extern template cudaError_t prepare_mag_t<2>();
// one-time per-device kernel attributes (call on the current device before launching)
cudaError_t prepare_sweep_kernels();
// Tensor maps of a TMA-staged magnetic sweep (kernel axes 1 and 2), dimensions
// ordered (lane axis A, row axis O, sweep axis D): rho, m_D, b_A, b_O, b_D
// over the 32 x 8 tile (32 x 8 x 4), rho, m_D, b_O one row (32 x 1 x 4) and
// rho, m_D, b_A four columns (4 x 8 x 4) of the neighbouring pencils; row[]:
// the same boxes one position long.
constexpr int kMagMaps = 11;
struct MagMaps {
  CUtensorMap full[kMagMaps];
  CUtensorMap row[kMagMaps];
};
// false if the box does not qualify (lane extent not a multiple of 32, row
// extent not a multiple of 8, unaligned fields) or the encoder is unavailable
bool make_mag_maps(int axis, const MagArgs& a, MagMaps* m);
bool mag_chunks_qualify(int axis, const MagArgs& a);  // the box's part of that
// cells [lo, hi) per kernel axis (the interior of a box with ghost layers)
struct CellRange {
  int lo[3], hi[3];
};
cudaError_t launch_cfl_rate(const float* const f[8], const Box& box, float gamma, unsigned* rate,
                            cudaStream_t s, const CellRange* range = nullptr,
                            float* const copy[8] = nullptr);  // copy: also write the fields there
struct CopyArgs {
  const float* in[8];
  float* out[8];
};
cudaError_t launch_copy_fields(const float* const in[8], float* const out[8], long long N, cudaStream_t s);
// Whether a kernel on the current device `dev` can copy between a box of device
// `home` and 8 fields, field q on device device_of(q) (-1: host or managed
// memory): only where all of it is memory of that device.
template <class DeviceOf>
inline bool all_on_device(int dev, int home, DeviceOf device_of) {
  bool local = dev == home;
  for (int q = 0; q < 8 && local; q++) local = device_of(q) == dev;
  return local;
}
bool local_fields(const void* const f[8], int home);
// device-side step control: tau = cfl / rate_cur (or the given tau if cfl<0),
// time += 2 tau, rate_next = 0
cudaError_t launch_step_control(const StepControl& c, int split, cudaStream_t s);
// set the device sweep step to a host value (no time advance)
cudaError_t launch_set_tau(float* tau, double value, cudaStream_t s);
// FP64 diagnostics: per-block partials into `partial` (nblk*kDiagSlots
// doubles), then a fixed-order final reduction into out[10] (device).
constexpr int kDiagSlots = 20;  // 8 (sum, compensation) pairs + max|div b| + min p
constexpr int kDiagGrid = 152 * 2;       // cap of the diagnostics grid (diag_blocks): the blocks that fit at once
int diag_blocks(const Box& box);
cudaError_t launch_diagnostics(const float* const f[8], const Box& box, double gamma, double* partial,
                               double* out, cudaStream_t s);

}  // namespace mhd
