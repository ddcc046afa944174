// Device helpers of the matrix-free operators (uniform mesh and octree): one
// line of N1 nodes along an axis and its traces at the two ends.
#pragma once

#include "dg_internal.h"

namespace dg {

// Every product and sum is written out with its rounding (mad, mul), so that the
// instances of a kernel round alike: a source's result depends neither on the
// work split nor, with it, on the number of sources in the call.
__device__ __forceinline__ float mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }

// Slots (of `lines` threads) per block, at most 320 threads, that leave the
// fewest idle lanes in the last warp; among equals the largest block of at most
// `small` threads
constexpr int best_bpb(int lines, int small) {
  int best = 1;
  for (int b = 2; b * lines <= 320; ++b) {
    const int tb = (b * lines + 31) / 32 * 32, t0 = (best * lines + 31) / 32 * 32;
    if (b * t0 > best * tb || (b * t0 == best * tb && tb <= small)) best = b;
  }
  return best;
}

// Shared-memory layout of elements of N1^3 nodes: node (a, b, c) of element e at
// a + PB b + PZ c + ES e: the strides with the fewest wavefronts of the three
// passes, counted over the warps of a block (1.4 to 1.9 per access; odd strides
// alone gave 1.9 to 2.5, and the FP32 operator was bound by them at p = 7: 86 %
// of the data pipe)
template <int N1>
struct LineLayout {
  static constexpr int PB = N1 == 8 ? 9 : N1;
  static constexpr int PZ = N1 == 2 ? 4 : N1 == 3 ? 9 : N1 == 4 ? 19 : N1 == 5 ? 25 : N1 == 6 ? 41 : N1 == 7 ? 52
                                                                                          : N1 == 8 ? 72 : 81;
  static constexpr int ES = N1 == 2 ? 10 : N1 == 3 ? 41 : N1 == 4 ? 80 : N1 == 5 ? 153 : N1 == 6 ? 260
                                                          : N1 == 7 ? 369 : N1 == 8 ? 575 : 736;
  static_assert(PZ >= PB * (N1 - 1) + N1 && ES >= (PZ + PB + 1) * (N1 - 1) + 1, "element layout overlaps");
};

// value and derivative at the left end of a line (RIGHT: at the right end, the
// derivative into the line, that is of the reversed line), from the basis values tl
// and derivatives dl at the left end
template <typename T, int N1, bool RIGHT>
__device__ __forceinline__ void end_inward(const T* tl, const T* dl, const T* v, T& val, T& der) {
  T a = mul(tl[RIGHT ? N1 - 1 : 0], v[0]), b = mul(dl[RIGHT ? N1 - 1 : 0], v[0]);
#pragma unroll
  for (int i = 1; i < N1; ++i) {
    const int k = RIGHT ? N1 - 1 - i : i;
    a = mad(tl[k], v[i], a);
    b = mad(dl[k], v[i], b);
  }
  val = a;
  der = b;
}
// the same with the derivative along the axis
template <typename T, int N1, bool RIGHT>
__device__ __forceinline__ void end_trace(const T* tl, const T* dl, const T* v, T& val, T& der) {
  end_inward<T, N1, RIGHT>(tl, dl, v, val, der);
  if (RIGHT) der = -der;
}

// line of N1 values at p with stride SD, reversed where rev is set; contiguous
// lines that are a multiple of 16 bytes are read with 16-byte loads where the
// field is aligned (vec)
template <typename T, int N1, int SD>
__device__ __forceinline__ void load_line(const T* __restrict__ p, bool rev, bool vec, T* v) {
  constexpr int W = 16 / (int)sizeof(T);
  if constexpr (SD == 1 && N1 % W == 0) {
    if (vec) {
      T q[N1];
#pragma unroll
      for (int w = 0; w < N1 / W; ++w) {
        if constexpr (sizeof(T) == 4) {
          const float4 t = __ldg(reinterpret_cast<const float4*>(p) + w);
          q[4 * w] = t.x;
          q[4 * w + 1] = t.y;
          q[4 * w + 2] = t.z;
          q[4 * w + 3] = t.w;
        } else {
          const double2 t = __ldg(reinterpret_cast<const double2*>(p) + w);
          q[2 * w] = t.x;
          q[2 * w + 1] = t.y;
        }
      }
#pragma unroll
      for (int i = 0; i < N1; ++i) v[i] = rev ? q[N1 - 1 - i] : q[i];
      return;
    }
  }
  const T* q = rev ? p + (N1 - 1) * SD : p;
  const int st = rev ? -SD : SD;
#pragma unroll
  for (int i = 0; i < N1; ++i) v[i] = __ldg(q + i * st);
}

}  // namespace dg
