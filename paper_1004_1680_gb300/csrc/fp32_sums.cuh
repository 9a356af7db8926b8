// Sums of FP32 values to FP64 accuracy and beyond without FP64 arithmetic per
// value: FP64 runs at a small fraction of the FP32 rate on this GPU (a warp
// instruction occupies its pipe for 16 cycles).
#pragma once
#include "mhd_device.cuh"

namespace mhd {

// Error-free FP32 transformations (Knuth's TwoSum; the FMA product error):
// s + e == a + b and p + e == a * b exactly (round to nearest, no overflow).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

// FP32 window sums without FP64 arithmetic per value (FP64 runs at a small
// fraction of the FP32 rate on this GPU): three FP32 words h + l + t.  Each
// value goes into h by TwoSum; its error goes into l by TwoSum; that error
// into t by a plain add.  With P the largest partial sum of a window of K
// values, |error of h + l| <= K 2^-24 P, so |t's errors| <= K^3 2^-72 P:
// 2^-48 P for K = kWin = 256.  Infinities and NaNs make the sum NaN, as in
// FP64.
// Two fields at a time, on packed FP32 (each element rounded as the scalar
// operation would round it): 13 instructions for two values.
constexpr int kWin = 256;
// Grid of the kernels whose threads add their share of n < 2^31 values into one
// window each (block_totals): enough blocks to read at full rate and few FP64
// atomics, but no thread with more than kWin values (beyond 39.8 M).
constexpr int kSumThreads = 256;
inline int sum_blocks(long long n) {
  const long long all = (n + kSumThreads - 1) / kSumThreads, most = 152 * 4, least = (all + kWin - 1) / kWin;
  return (int)(all < 1 ? 1 : (all < most ? all : (least > most ? least : most)));
}
struct FWin2 {
  float2 h, l, t;
};

__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
  s = __fadd2_rn(a, b);
  const float2 bp = sub2(s, a);
  e = __fadd2_rn(sub2(a, sub2(s, bp)), sub2(b, bp));
}

__device__ __forceinline__ void two_prod2(float2 a, float2 b, float2& p, float2& e) {
  p = __fmul2_rn(a, b);
  e = __ffma2_rn(a, b, neg2(p));
}

__device__ __forceinline__ void fwin_add(FWin2& w, float2 x) {
  float2 s, e, s2, e2;
  two_sum2(w.h, x, s, e);
  two_sum2(w.l, e, s2, e2);
  w.h = s;
  w.l = s2;
  w.t = __fadd2_rn(w.t, e2);
}

// A lane's windows add up in a plain FP64 sum (a few windows per lane: their
// roundings stay near 2^-53 of the field's absolute sum); the compensated
// sum starts at the warps' totals.
__device__ __forceinline__ void fwin_flush(FWin2& w, double& a0, double& a1) {
  a0 += ((double)w.h.x + (double)w.l.x) + (double)w.t.x;
  a1 += ((double)w.h.y + (double)w.l.y) + (double)w.t.y;
  w.h = w.l = w.t = f2(0.f);
}

// Add another window's words.
__device__ __forceinline__ void fwin_merge(FWin2& w, float2 h, float2 l, float2 t) {
  float2 s, e, m, e2, m2, e3;
  two_sum2(w.h, h, s, e);
  two_sum2(w.l, l, m, e2);
  two_sum2(m, e, m2, e3);
  w.h = s;
  w.l = m2;
  w.t = __fadd2_rn(__fadd2_rn(w.t, t), __fadd2_rn(e2, e3));
}
__device__ __forceinline__ float2 shfl_down2(float2 x, int o) {
  return make_float2(__shfl_down_sync(0xffffffffu, x.x, o), __shfl_down_sync(0xffffffffu, x.y, o));
}

}  // namespace mhd
