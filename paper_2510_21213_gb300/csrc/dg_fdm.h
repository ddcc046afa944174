// Device helpers of the fast-diagonalisation solves (Schwarz patches, octree leaf
// blocks): transforms of lines held in registers with a mode table in shared
// memory, row q of the table = mode q at the nodes.
#pragma once

#include "dg_internal.h"

namespace dg {

// N values of a table row (16-byte aligned)
template <typename T, int N>
__device__ __forceinline__ void sw_row(const T* __restrict__ p, T* r) {
  constexpr int W = 16 / (int)sizeof(T);
#pragma unroll
  for (int w = 0; w < (N + W - 1) / W; ++w) {
    if constexpr (sizeof(T) == 4) {
      const float4 q = reinterpret_cast<const float4*>(p)[w];
      const float t[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (4 * w + k < N) r[4 * w + k] = t[k];
    } else {
      const double2 q = reinterpret_cast<const double2*>(p)[w];
      r[2 * w] = q.x;
      if (2 * w + 1 < N) r[2 * w + 1] = q.y;
    }
  }
}

// sums and differences of mirrored nodes in place: v[i] (i < HE) the even part,
// v[HE + i] the odd part
template <typename T, int MP>
__device__ __forceinline__ void sw_fold(T* v) {
  constexpr int HO = MP / 2, HE = MP - HO;
  T o[HO];
#pragma unroll
  for (int i = 0; i < HO; ++i) {
    o[i] = v[i] - v[MP - 1 - i];
    v[i] = v[i] + v[MP - 1 - i];
  }
#pragma unroll
  for (int i = 0; i < HO; ++i) v[HE + i] = o[i];
}
// the reverse: node values from the even and odd parts
template <typename T, int MP>
__device__ __forceinline__ void sw_unfold(T* v) {
  constexpr int HO = MP / 2, HE = MP - HO;
  T o[HO];
#pragma unroll
  for (int i = 0; i < HO; ++i) o[i] = v[HE + i];
#pragma unroll
  for (int i = 0; i < HO; ++i) {
    v[MP - 1 - i] = v[i] - o[i];
    v[i] = v[i] + o[i];
  }
}

// Transforms of LPT lines with the table tb (row q: mode q at the nodes, halved
// rows where SYM: the first HE even, the rest odd). A half H of the modes works
// on the values v[O .. O + N).
// forward: put(s, q, sum_i S[i][q] v[s][i])
template <typename T, int MP, int LPT, int N, int O, int Q0, int Q1, typename P>
__device__ __forceinline__ void sw_fwd_half(const T* tb, int RP, const T (*v)[MP], P&& put) {
#pragma unroll 2
  for (int q = Q0; q < Q1; ++q) {
    T r[N], a[LPT];
    sw_row<T, N>(tb + q * RP, r);
#pragma unroll
    for (int s = 0; s < LPT; ++s) a[s] = r[0] * v[s][O];
#pragma unroll
    for (int i = 1; i < N; ++i)
#pragma unroll
      for (int s = 0; s < LPT; ++s) a[s] += r[i] * v[s][O + i];
#pragma unroll
    for (int s = 0; s < LPT; ++s) put(s, q, a[s]);
  }
}
template <typename T, int MP, int LPT, typename P>
__device__ __forceinline__ void sw_fwd(bool sym, const T* tb, int RP, T (*v)[MP], P&& put) {
  constexpr int HO = MP / 2, HE = MP - HO;
  if (sym) {
#pragma unroll
    for (int s = 0; s < LPT; ++s) sw_fold<T, MP>(v[s]);
    sw_fwd_half<T, MP, LPT, HE, 0, 0, HE>(tb, RP, v, put);
    sw_fwd_half<T, MP, LPT, HO, HE, HE, MP>(tb, RP, v, put);
  } else {
    sw_fwd_half<T, MP, LPT, MP, 0, 0, MP>(tb, RP, v, put);
  }
}
// backward: v[s][i] = sum_q S[i][q] get(s, q)
template <typename T, int MP, int LPT, int N, int O, int Q0, int Q1, typename G>
__device__ __forceinline__ void sw_bwd_half(const T* tb, int RP, T (*v)[MP], G&& get) {
#pragma unroll
  for (int s = 0; s < LPT; ++s)
#pragma unroll
    for (int i = 0; i < N; ++i) v[s][O + i] = (T)0;
#pragma unroll 2
  for (int q = Q0; q < Q1; ++q) {
    T r[N], c[LPT];
#pragma unroll
    for (int s = 0; s < LPT; ++s) c[s] = get(s, q);
    sw_row<T, N>(tb + q * RP, r);
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int s = 0; s < LPT; ++s) v[s][O + i] += r[i] * c[s];
  }
}
template <typename T, int MP, int LPT, typename G>
__device__ __forceinline__ void sw_bwd(bool sym, const T* tb, int RP, T (*v)[MP], G&& get) {
  constexpr int HO = MP / 2, HE = MP - HO;
  if (sym) {
    sw_bwd_half<T, MP, LPT, HE, 0, 0, HE>(tb, RP, v, get);
    sw_bwd_half<T, MP, LPT, HO, HE, HE, MP>(tb, RP, v, get);
#pragma unroll
    for (int s = 0; s < LPT; ++s) sw_unfold<T, MP>(v[s]);
  } else {
    sw_bwd_half<T, MP, LPT, MP, 0, 0, MP>(tb, RP, v, get);
  }
}
// both, with the scaling between: v[s] <- S diag(scale(s, q, .)) S^T v[s]
template <typename T, int MP, int LPT, int N, int O, int Q0, int Q1, typename F>
__device__ __forceinline__ void sw_mid_half(const T* tb, int RP, const T (*v)[MP], T (*w)[MP], F&& scale) {
#pragma unroll
  for (int s = 0; s < LPT; ++s)
#pragma unroll
    for (int i = 0; i < N; ++i) w[s][O + i] = (T)0;
#pragma unroll 1
  for (int q = Q0; q < Q1; ++q) {
    T r[N], a[LPT];
    sw_row<T, N>(tb + q * RP, r);
#pragma unroll
    for (int s = 0; s < LPT; ++s) a[s] = r[0] * v[s][O];
#pragma unroll
    for (int i = 1; i < N; ++i)
#pragma unroll
      for (int s = 0; s < LPT; ++s) a[s] += r[i] * v[s][O + i];
#pragma unroll
    for (int s = 0; s < LPT; ++s) a[s] = scale(s, q, a[s]);
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int s = 0; s < LPT; ++s) w[s][O + i] += r[i] * a[s];
  }
}
template <typename T, int MP, int LPT, typename F>
__device__ __forceinline__ void sw_mid(bool sym, const T* tb, int RP, T (*v)[MP], T (*w)[MP], F&& scale) {
  constexpr int HO = MP / 2, HE = MP - HO;
  if (sym) {
#pragma unroll
    for (int s = 0; s < LPT; ++s) sw_fold<T, MP>(v[s]);
    sw_mid_half<T, MP, LPT, HE, 0, 0, HE>(tb, RP, v, w, scale);
    sw_mid_half<T, MP, LPT, HO, HE, HE, MP>(tb, RP, v, w, scale);
#pragma unroll
    for (int s = 0; s < LPT; ++s) sw_unfold<T, MP>(w[s]);
  } else {
    sw_mid_half<T, MP, LPT, MP, 0, 0, MP>(tb, RP, v, w, scale);
  }
}

}  // namespace dg
