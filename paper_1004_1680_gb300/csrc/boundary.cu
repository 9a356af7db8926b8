// Ghost layers of non-periodic axes (an extension: the paper's runs are
// periodic).  A non-periodic axis of n cells keeps kGhost = 4 ghost cells at
// each end inside the box: interior cells kGhost .. n-kGhost-1, wall faces
// kGhost (low) and n-kGhost (the low face of the first high ghost cell).
// The library refills them before every sweep and before every CFL rate; the
// sweeps are the periodic ones (a cell reads at most 3 cells along the sweep
// and 1 pencil across, all inside the ghost layers).
//   outflow (mode 1):    a ghost cell copies the nearest interior cell; ghost
//                        faces of the normal field copy the wall face;
//   reflecting (mode 2): a ghost cell copies its mirror image in the wall with
//                        the normal momentum negated; ghost faces of the
//                        normal field copy their mirror faces, negated.
// Tangential face fields are cell-like along the axis.  The axes are filled one
// after another (x, y, z over the whole extent of the other axes), which defines
// the edge and corner ghosts; since each axis maps a ghost position to one that
// is not, and leaves the other coordinates alone, the value that ends up in a
// cell is that of the position mapped along every axis at once, negated once
// per axis that asks for it.  So one launch fills all axes: every source is an
// interior value that nobody writes (a cell that is a ghost of two axes is
// written twice, with the same value).  One launch per axis cost 2 to 3 us more
// per axis and sweep (236 x 150 x 98, two open axes: 5.12 -> 4.98 ms for 6 steps).
//
// The time beyond the launch is index arithmetic and 16 memory instructions per
// element.  Across the contiguous axis a thread therefore takes 4 cells (V = 4,
// rows of a multiple of 4 cells), and a step asks only for the fields that the
// sweep before has written (`parts`): the same
// walls 3.91 -> 3.55 ms, 40 steps of a 512 x 8 x 8 tube 3.67 -> 3.18 ms.
#include <cstdint>

#include "mhd_launch.h"

namespace mhd {

// I: the index type of the element and plane counters (unsigned 32-bit when
// they fit, which avoids emulated 64-bit division per element).  V: cells per
// thread in the layers across the contiguous axis; with 4, cells that are also
// ghosts of the contiguous axis are left to that axis's threads.
template <typename I, int V>
__global__ void __launch_bounds__(256) ghost_fill_kernel(const __grid_constant__ GhostArgs a) {
  const I total = (I)a.first[3];
  bool waited = false;  // the first element's indexes are formed while the sweep before still runs
  for (I id = (I)blockIdx.x * blockDim.x + threadIdx.x; id < total; id += (I)gridDim.x * blockDim.x) {
    // the ghost layers of axis k: elements (groups of V cells for k > 0)
    // first[k] .. first[k + 1] - 1
    const int k = id >= (I)a.first[2] ? 2 : (id >= (I)a.first[1] ? 1 : 0);
    const I e = id - (I)a.first[k];
    const int t1 = k == 0 ? 1 : 0, t2 = k == 2 ? 1 : 2;
    // along the contiguous axis the 2 x kGhost ghost cells of a row are
    // neighbouring threads (16 contiguous bytes per side); across it,
    // neighbouring threads take neighbouring rows (contiguous along x)
    I p;
    int layer, side;
    if (k == 0) {
      layer = (int)(e % kGhost);
      side = (int)((e / kGhost) & 1);
      p = e / (2 * kGhost);
    } else {
      // (t1 is the contiguous axis: a.n[0] / V groups per row)
      const I plane = (I)(a.n[0] / V) * (I)a.n[t2], q = e / plane;
      p = e - q * plane;
      layer = (int)(q % kGhost);
      side = (int)(q / kGhost);
    }
    int x[3];
    x[k] = side ? a.n[k] - 1 - layer : layer;
    const I row = k == 0 ? (I)a.n[t1] : (I)(a.n[0] / V);
    x[t2] = (int)(p / row);
    x[t1] = (int)(p - (I)x[t2] * row);
    if (V > 1 && k > 0) {
      x[0] *= V;
      if (a.mode[0] && (x[0] < kGhost || x[0] >= a.n[0] - kGhost)) continue;
    }
    // per axis: where cell-like fields and the axis's own face field come from
    long long di = 0, cell = 0, face[3];
    bool neg_m[3], neg_b[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
      const int n = a.n[d], lo = kGhost, hi = n - kGhost, c = x[d];
      int s = c, f = c;
      neg_m[d] = neg_b[d] = false;
      if (a.mode[d]) {
        if (c < lo) {
          s = a.mode[d] == 1 ? lo : 2 * lo - 1 - c;
          f = a.mode[d] == 1 ? lo : 2 * lo - c;
        } else if (c >= hi) {
          s = a.mode[d] == 1 ? hi - 1 : 2 * hi - 1 - c;
          f = a.mode[d] == 1 || c == hi ? hi : 2 * hi - c;  // (the wall face itself is an interior unknown)
        }
        neg_m[d] = a.mode[d] == 2 && s != c;
        neg_b[d] = a.mode[d] == 2 && f != c;
      }
      di += (long long)c * a.stride[d];
      cell += (long long)s * a.stride[d];
      face[d] = (long long)(f - s) * a.stride[d];
    }
    if (!waited) {
      int moves = di != cell;
      settled(moves, x[0]);
      wait_for_previous_in_place();
      waited = true;
    }
#pragma unroll
    for (int q = 0; q < 8; q++) {
      if (!(a.parts & (q >= 5 ? kGhostField : kGhostFluid))) continue;
      const long long si = q >= 5 ? cell + face[q >= 5 ? q - 5 : 0] : cell;
      if (si == di) continue;
      const bool neg = q >= 5 ? neg_b[q >= 5 ? q - 5 : 0] : (q >= 1 && q <= 3 && neg_m[q >= 1 && q <= 3 ? q - 1 : 0]);
      if (V == 1 || k == 0) {
        const float v = a.f[q][si];
        a.f[q][di] = neg ? -v : v;
      } else {  // (along x the cells map to themselves)
        float4 v = *reinterpret_cast<const float4*>(a.f[q] + si);
        if (neg) v = make_float4(-v.x, -v.y, -v.z, -v.w);
        *reinterpret_cast<float4*>(a.f[q] + di) = v;
      }
    }
  }
  if (!waited) wait_for_previous_in_place();
}

cudaError_t launch_ghost_fill(float* const f[8], const Box& box, const int mode[3], int parts, cudaStream_t s) {
  GhostArgs a;
  a.parts = parts;
  bool wide = box.n[0] % 4 == 0 && box.stride[0] == 1 && box.stride[1] % 4 == 0 && box.stride[2] % 4 == 0;
  for (int q = 0; q < 8; q++) {
    a.f[q] = f[q];
    wide = wide && reinterpret_cast<uintptr_t>(f[q]) % 16 == 0;
  }
  const int V = wide ? 4 : 1;
  a.first[0] = 0;
  for (int k = 0; k < 3; k++) {
    a.n[k] = box.n[k];
    a.stride[k] = box.stride[k];
    a.mode[k] = mode[k];
    const int t1 = k == 0 ? 1 : 0, t2 = k == 2 ? 1 : 2;
    a.first[k + 1] = a.first[k] + (mode[k] ? 2LL * kGhost * (k ? box.n[t1] / V : box.n[t1]) * box.n[t2] : 0);
  }
  const long long total = a.first[3];
  long long blocks = (total + 255) / 256;
  if (blocks > 65535LL * 16) blocks = 65535LL * 16;
  // 32-bit counters while the element count and the last id + stride fit
  const bool narrow = total + blocks * 256 < (1LL << 32);
  auto* kernel = narrow ? (wide ? ghost_fill_kernel<unsigned, 4> : ghost_fill_kernel<unsigned, 1>)
                        : (wide ? ghost_fill_kernel<unsigned long long, 4> : ghost_fill_kernel<unsigned long long, 1>);
  const int split = shared_split((long long)box.n[0] * box.n[1] * box.n[2]);
  return launch_after(true, split, kernel, dim3((unsigned)blocks), dim3(256), 0, s, a);
}

}  // namespace mhd
