// Matrix-free SIPDG operator (Sec. 3.4 eq. sip_bilinear with the penalty of
// Sec. 3.5 and Nitsche boundary faces) on the element-blocked layout.
//
// For an element the operator needs its own (p+1)^3 values and, for each of its
// six faces, the neighbour's trace and reference normal derivative there (the
// off-diagonal blocks of the 1-D operator are rank 2). Output node (a, b, c):
//   (Au) = My_b Mz_c [sum_i Kx[a,i] u_ibc + cL.x(-x traces) + cR.x(+x traces)]
//        + Mx_a Mz_c [ ... y ... ] + Mx_a My_b [ ... z ... ]
//
// Arithmetic of one line (N1 = p + 1 values along the direction). The GL nodes
// are symmetric about the element's middle, so the interior element's 1-D block
// K and the pair of couplings are invariant under reversing the line. With
// e_i = v_i + v_(N1-1-i) and o_i = v_i - v_(N1-1-i) the line splits into an even
// and an odd half of size N1/2: K costs N1^2/2 multiply-adds instead of N1^2,
// the couplings to both neighbours 2 N1 instead of 4 N1. A boundary face is a
// face whose neighbour has the traces
//   value = -t,  derivative = d -+ sigma h t   (- left, + right)
// with t, d the element's own trace and derivative there: inserted into the
// interior coupling they turn it into the Nitsche terms, so every element of an
// axis has the same tables and no element type is distinguished. 41 operations
// a node instead of 52 (p = 7).
//
// Work split. A brick of 2 x 2 x 2 elements of one source (or a single element)
// per slot; in the pass along a direction a thread owns the lines of the two
// elements that are neighbours along it, so the traces across their common face
// stay in registers, and a brick reads 24 outer neighbours instead of the 48 of
// eight single elements. Own elements and the outer neighbours' lines (reduced to
// traces at once) are read before the barrier ahead of the x pass, the operand of a
// residual in the z pass. The tables are kernel parameters: every product takes its constant
// from the constant bank, so shared memory carries only the field.
//
// Measured (GB300; before: one element per slot, dense blocks and tables in
// shared memory): FP32 16^3, p = 7, 42 fields 0.720 -> 0.279 ms (2.5 TB/s of the
// 0.70 GB in and out), 8^3, p = 6, 56 fields 0.100 -> 0.042 ms; bound by
// shared-memory wavefronts, then by the neighbours' reads. FP64, at the rate of
// its pipe before and after: 7.86 -> 7.01 ms and 0.954 -> 0.793 ms, p = 3 and 1 (16^3,
// 42 fields) 0.828 -> 0.820 and 0.087 -> 0.054 ms.
#include "dg_line.h"

namespace dg {


// 1-D tables of one level, folded into even and odd halves (host-built, passed
// by value). HE = ceil(N1/2) even and HO = floor(N1/2) odd rows.
//
// N1 = 2 is not folded (two sums and differences per line cost what the halves
// save): there Ke, Ko hold K[0][0], K[0][1], and likewise the couplings their
// entries 0 and 1.
template <typename T, int N1>
struct ApplyTab {
  static constexpr int HO = N1 / 2, HE = N1 - HO;
  // FP64 with few nodes: neighbours enter by their values (see line_direct)
  static constexpr bool DIRECT = sizeof(T) == 8 && N1 <= 3;
  static constexpr int DN = DIRECT ? N1 : 1;
  T Ke[3][HE][HE], Ko[3][HO][HO];                          // K on the even and the odd part
  T cve[3][HE], cde[3][HE], cvo[3][HO], cdo[3][HO];        // couplings (neighbour value / derivative)
  T tl[N1], dl[N1];                                        // trace and derivative at a line's left end
  T gam[3];                                                // sigma h
  T mm[3][N1 * N1];                                        // products of the two other axes' masses, by line
  int n[3], nb[3];                                         // elements and bricks per axis
  long long Nq, items;                                     // nodes of a source; bricks of all sources
  T K[3][DN][DN], C[3][DN][DN], B[3][DN][DN];  // own block, coupling to the right neighbour, right boundary face
};

template <typename T, int N1>
static void fill_tab(ApplyTab<T, N1>& t, const LevelOp& op) {
  constexpr int HO = N1 / 2, HE = N1 - HO;
  for (int d = 0; d < 3; ++d) {
    const AxisOp& A = op.ax[d];
    // K[a][i], averaged with its mirror image (equal up to round-off)
    auto K = [&](int a, int i) {
      return 0.5 * (A.Kd[0][a * N1 + i] + A.Kd[0][(N1 - 1 - a) * N1 + (N1 - 1 - i)]);
    };
    for (int a = 0; a < HE; ++a)
      for (int i = 0; i < HE; ++i)
        t.Ke[d][a][i] = (T)(i < HO ? 0.5 * (K(a, i) + K(a, N1 - 1 - i)) : K(a, i));
    for (int a = 0; a < HO; ++a)
      for (int i = 0; i < HO; ++i) t.Ko[d][a][i] = (T)(0.5 * (K(a, i) - K(a, N1 - 1 - i)));
    const AxisOp &B = op.ax[d == 0 ? 1 : 0], &C = op.ax[d == 2 ? 1 : 2];
    for (int l = 0; l < N1 * N1; ++l) t.mm[d][l] = (T)(B.m[l % N1] * C.m[l / N1]);
    for (int a = 0; a < HE; ++a) {
      t.cve[d][a] = (T)(0.5 * (A.cLv[a] + A.cLv[N1 - 1 - a]));
      t.cde[d][a] = (T)(0.5 * (A.cLd[a] + A.cLd[N1 - 1 - a]));
    }
    for (int a = 0; a < HO; ++a) {
      t.cvo[d][a] = (T)(0.5 * (A.cLv[a] - A.cLv[N1 - 1 - a]));
      t.cdo[d][a] = (T)(0.5 * (A.cLd[a] - A.cLd[N1 - 1 - a]));
    }
    t.gam[d] = (T)(A.sigma * A.h);
    t.n[d] = op.n[d];
  }
  if constexpr (ApplyTab<T, N1>::DIRECT) {
    for (int d = 0; d < 3; ++d) {
      const AxisOp& A = op.ax[d];
      for (int a = 0; a < N1; ++a)
        for (int i = 0; i < N1; ++i) {
          t.K[d][a][i] = (T)(0.5 * (A.Kd[0][a * N1 + i] + A.Kd[0][(N1 - 1 - a) * N1 + (N1 - 1 - i)]));
          t.C[d][a][i] = (T)(A.cRv[a] * op.tl[i] + A.cRd[a] * op.dl[i]);
          t.B[d][a][i] = (T)(A.cRd[a] * (op.dr[i] + A.sigma * A.h * op.tr[i]) - A.cRv[a] * op.tr[i]);
        }
    }
  } else if (N1 == 2) {
    for (int d = 0; d < 3; ++d) {
      const AxisOp& A = op.ax[d];
      t.Ke[d][0][0] = (T)A.Kd[0][0];
      t.Ko[d][0][0] = (T)A.Kd[0][1];
      t.cve[d][0] = (T)A.cLv[0];
      t.cvo[d][0] = (T)A.cLv[1];
      t.cde[d][0] = (T)A.cLd[0];
      t.cdo[d][0] = (T)A.cLd[1];
    }
  }
  for (int a = 0; a < N1; ++a) {
    t.tl[a] = (T)op.tl[a];
    t.dl[a] = (T)op.dl[a];
  }
  t.Nq = op.Nq;
}

// Launch shape. BR: elements of a brick along each axis (2 or 1); BPB: bricks of a
// block. FP64 at p = 2: 126 of 128 lanes at work, instead of 288 of 288 in blocks that
// are too large for a few thousand elements.
template <typename T, int N1, int BR>
constexpr int apply_bpb() {
  return sizeof(T) == 8 && N1 == 3 ? 14 : best_bpb(BR * BR * N1 * N1, sizeof(T) == 4 ? 128 : 64);
}
// smaller blocks for FP64 where the full ones are large (288 and 256 threads)
template <int N1>
constexpr int apply_few() {
  return N1 == 6 ? 5 : N1 == 7 ? 3 : apply_bpb<double, N1, 1>();
}
template <typename T, int N1, int BR, int BPB_ = apply_bpb<T, N1, BR>()>
struct ApplyCfg {
  static constexpr int NPE = N1 * N1 * N1, NF = N1 * N1;
  static constexpr int EB = BR * BR * BR;        // elements of a brick
  static constexpr int LINES = BR * BR * NF;     // threads of a brick: one (pair of) line(s) each
  static constexpr int PB = LineLayout<N1>::PB, PZ = LineLayout<N1>::PZ, ES = LineLayout<N1>::ES;
  static constexpr int BPB = BPB_;
  static constexpr int THREADS = (BPB * LINES + 31) / 32 * 32;
  static constexpr size_t SMEM = sizeof(T) * 2 * (size_t)BPB * EB * ES;
  // resident threads per SM asked of ptxas (register cap 65536 / that)
  static constexpr int WANT = sizeof(T) == 4 ? 768 : 640;
  static constexpr int MINB = WANT / THREADS < 1 ? 1 : WANT / THREADS;
};

// What lies beyond the two ends of a line (pair), 0: left of the first, 1: right of the
// last line: ov, od the traces there (value, derivative), or with DIRECT ov[end N1 + i]
// the values of the neighbour's line (at a boundary face of the own line). The left
// neighbour's derivative is kept along the axis in FP32 and against it in FP64, where a
// change of sign is an operation of the pipe that bounds the kernel.
template <typename T>
constexpr bool left_inward() {
  return sizeof(T) == 8;
}
template <typename T, int N1>
constexpr int outer_vals() {
  return ApplyTab<T, N1>::DIRECT ? 2 * N1 : 2;
}
template <typename T, int N1>
__device__ __forceinline__ void left_end(const ApplyTab<T, N1>& tab, const T* v, T& val, T& der) {
  if constexpr (left_inward<T>())
    end_inward<T, N1, true>(tab.tl, tab.dl, v, val, der);
  else
    end_trace<T, N1, true>(tab.tl, tab.dl, v, val, der);
}

// The pass of line_op for FP64 at p = 1 and 2, bound by the FP64 pipe: the coupling
// block of a neighbour has N1^2 entries, no more than a trace and its lifting take
// (4 N1), and nothing is folded: 12 and 27 multiply-adds a line instead of 20 and 34
// operations. The left neighbour's and the left boundary's blocks are the right ones'
// mirror images. Which block an end takes is selected, not branched on: lanes at the
// boundary would double the products of their warp. The own block comes last: its
// error against 64-bit exact lines is then no larger than with traces.
// Measured (GB300, 16^3, 20 fields; with traces, folded at p = 2, and before those): p =
// 1 45 / 53 -> 27 us, p = 2 150 / 172 -> 122 us.
template <typename T, int N1, int D>
__device__ __forceinline__ void line_direct(const ApplyTab<T, N1>& tab, T* v, const T* ov, bool in0, bool in1) {
  T r[N1];
#pragma unroll
  for (int a = 0; a < N1; ++a) {
    const int m = N1 - 1 - a;
    T acc = mul(in0 ? tab.C[D][m][N1 - 1] : tab.B[D][m][N1 - 1], ov[0]);
#pragma unroll
    for (int i = 1; i < N1; ++i)
      acc = mad(in0 ? tab.C[D][m][N1 - 1 - i] : tab.B[D][m][N1 - 1 - i], ov[i], acc);
#pragma unroll
    for (int i = 0; i < N1; ++i) acc = mad(in1 ? tab.C[D][a][i] : tab.B[D][a][i], ov[N1 + i], acc);
#pragma unroll
    for (int i = 0; i < N1; ++i) acc = mad(tab.K[D][a][i], v[i], acc);
    r[a] = acc;
  }
#pragma unroll
  for (int a = 0; a < N1; ++a) v[a] = r[a];
}

// one pass along direction D for this thread's line (pair): on entry v[s] holds
// the line values, ov/od what is beyond its two ends (in0, in1: a neighbour). On exit
// v[s] holds the unscaled result.
template <typename T, int N1, int BR, int D>
__device__ __forceinline__ void line_op(const ApplyTab<T, N1>& tab, T (*v)[N1], const T* ov, const T* od,
                                        bool second, bool in0, bool in1) {
  constexpr int HO = N1 / 2, HE = N1 - HO;
  if constexpr (ApplyTab<T, N1>::DIRECT) {
    static_assert(BR == 1, "bricks are FP32's");
    line_direct<T, N1, D>(tab, v[0], ov, in0, in1);
    return;
  }
  T e[BR][HE], o[BR][HO == 0 ? 1 : HO];
  T tv[BR], td[BR];  // the pair's traces on their common face
#pragma unroll
  for (int s = 0; s < BR; ++s) {
    if (BR == 2) {
      if (s == 0)
        left_end(tab, v[s], tv[s], td[s]);
      else
        end_trace<T, N1, false>(tab.tl, tab.dl, v[s], tv[s], td[s]);
    }
    if constexpr (N1 > 2) {
#pragma unroll
      for (int i = 0; i < HO; ++i) {
        e[s][i] = v[s][i] + v[s][N1 - 1 - i];
        o[s][i] = v[s][i] - v[s][N1 - 1 - i];
      }
      if (HE > HO) e[s][HE - 1] = v[s][HO];
    }
  }
#pragma unroll
  for (int s = 0; s < BR; ++s) {
    T nl, dl, nr, dr;  // the neighbours' traces, left and right
    if (BR == 2) {
      nl = s == 0 ? ov[0] : tv[0];
      dl = s == 0 ? od[0] : td[0];
      nr = s == 0 && second ? tv[BR - 1] : ov[1];
      dr = s == 0 && second ? td[BR - 1] : od[1];
    } else {
      nl = ov[0];
      dl = od[0];
      nr = ov[1];
      dr = od[1];
    }
    if constexpr (N1 == 2) {
      const T v0 = v[s][0], v1 = v[s][1];
      T x = mul(tab.cve[D][0], nl), y = mul(tab.cvo[D][0], nl);
      x = mad(tab.cde[D][0], dl, x);
      y = mad(tab.cdo[D][0], dl, y);
      x = mad(tab.cvo[D][0], nr, x);
      y = mad(tab.cve[D][0], nr, y);
      x = mad(-tab.cdo[D][0], dr, x);
      y = mad(-tab.cde[D][0], dr, y);
      x = mad(tab.Ke[D][0][0], v0, x);
      y = mad(tab.Ko[D][0][0], v0, y);
      v[s][0] = mad(tab.Ko[D][0][0], v1, x);
      v[s][1] = mad(tab.Ke[D][0][0], v1, y);
      continue;
    }
    constexpr bool NEG = left_inward<T>();
    const T vp = nl + nr, vm = nl - nr, dm = NEG ? dl + dr : dl - dr, dp = NEG ? dr - dl : dl + dr;
    T O[HO == 0 ? 1 : HO];
#pragma unroll
    for (int a = 0; a < HO; ++a) {
      T acc = mad(tab.cdo[D][a], dp, mul(tab.cvo[D][a], vm));
#pragma unroll
      for (int i = 0; i < HO; ++i) acc = mad(tab.Ko[D][a][i], o[s][i], acc);
      O[a] = acc;
    }
#pragma unroll
    for (int a = 0; a < HE; ++a) {
      T acc = mad(NEG ? -tab.cde[D][a] : tab.cde[D][a], dm, mul(tab.cve[D][a], vp));
#pragma unroll
      for (int i = 0; i < HE; ++i) acc = mad(tab.Ke[D][a][i], e[s][i], acc);
      if (a < HO) {
        v[s][a] = acc + O[a];
        v[s][N1 - 1 - a] = acc - O[a];
      } else {
        v[s][a] = acc;
      }
    }
  }
}

// what lies beyond the ends of this thread's line (pair) along D: the outer
// neighbours' where there are any (out0, out1), else what the boundary stands for,
// from the line's own values. Read reversed, the own line looks like the
// neighbour's: value t and derivative -d at the common face. ue points at the
// brick's first element, es is the element stride along D (elements).
template <typename T, int N1, int BR, int D>
__device__ __forceinline__ void outer_traces(const ApplyTab<T, N1>& tab, const T* __restrict__ ue, long long pair,
                                             int l1, int l2, long long es, bool second, bool out0, bool out1,
                                             bool vec, T* ov, T* od) {
  constexpr int NF = N1 * N1, NPE = NF * N1;
  constexpr int SD = D == 0 ? 1 : (D == 1 ? N1 : NF);
  const int base = D == 0 ? N1 * l1 + NF * l2 : (D == 1 ? l1 + NF * l2 : l1 + N1 * l2);
  const T* p = ue + pair * NPE + base;
  if constexpr (ApplyTab<T, N1>::DIRECT) {
    load_line<T, N1, SD>(out0 ? p - es * NPE : p, false, vec, ov);
    load_line<T, N1, SD>(out1 ? p + es * NPE : p, false, vec, ov + N1);
    return;
  }
  const T gam = tab.gam[D];
  T v[N1];
  load_line<T, N1, SD>(out0 ? p - es * NPE : p, !out0, vec, v);
  left_end(tab, v, ov[0], od[0]);
  if (!out0) {
    od[0] = mad(left_inward<T>() ? gam : -gam, ov[0], -od[0]);
    ov[0] = -ov[0];
  }
  const int last = BR == 2 && second ? 1 : 0;
  load_line<T, N1, SD>(p + (last + (out1 ? 1 : 0)) * es * NPE, !out1, vec, v);
  end_trace<T, N1, false>(tab.tl, tab.dl, v, ov[1], od[1]);
  if (!out1) {
    od[1] = mad(gam, ov[1], -od[1]);
    ov[1] = -ov[1];
  }
}

template <typename T, int N1, int BR, int BPB>
__global__ void __launch_bounds__(ApplyCfg<T, N1, BR, BPB>::THREADS, ApplyCfg<T, N1, BR, BPB>::MINB)
    k_apply(const __grid_constant__ ApplyTab<T, N1> tab, const T* __restrict__ u, T* __restrict__ out,
            const T* __restrict__ rin, const int* __restrict__ act, int mode, int vec_i) {
  using C = ApplyCfg<T, N1, BR, BPB>;
  constexpr int NPE = C::NPE, NF = C::NF, EB = C::EB, LINES = C::LINES;
  constexpr int PB = C::PB, PZ = C::PZ, ES = C::ES;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* su = reinterpret_cast<T*>(smem_raw);
  T* sacc = su + BPB * EB * ES;
  __shared__ long long sbase[BPB];  // first value of the brick's first element, -1: no brick
  __shared__ int sflag[BPB];        // bits d: second element along d; 3 + 2 d + side: outer neighbour
  const int tid = threadIdx.x;
  const bool vec = vec_i != 0;
  const int nx = tab.n[0], ny = tab.n[1];
  const long long est[3] = {1, nx, (long long)nx * ny};
  if (tid < BPB) {
    const long long it = (long long)blockIdx.x * BPB + tid;
    long long base = -1;
    int flag = 0;
    if (it < tab.items) {
      const unsigned nbr = (unsigned)(tab.nb[0] * tab.nb[1]) * (unsigned)tab.nb[2];
      const unsigned k = (unsigned)(it / nbr), r = (unsigned)(it - (long long)k * nbr);
      const unsigned bx = r % tab.nb[0], q = r / tab.nb[0], by = q % tab.nb[1], bz = q / tab.nb[1];
      const int e[3] = {(int)bx * BR, (int)by * BR, (int)bz * BR};
      base = (long long)act[k] * tab.Nq + (e[0] + est[1] * e[1] + est[2] * e[2]) * NPE;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const bool sec = BR == 2 && e[d] + 1 < tab.n[d];
        if (sec) flag |= 1 << d;
        if (e[d] > 0) flag |= 8 << (2 * d);
        if (e[d] + (sec ? 2 : 1) < tab.n[d]) flag |= 16 << (2 * d);
      }
    }
    sbase[tid] = base;
    sflag[tid] = flag;
  }
  __syncthreads();
  const int slot = tid / LINES, lt = tid - slot * LINES;
  const int pr = lt / NF, l = lt - pr * NF, l1 = l % N1, l2 = l / N1;
  const int p1 = pr & 1, p2 = pr >> 1;  // the pair's position along the lower and the higher other axis
  const bool on = slot < BPB && sbase[slot < BPB ? slot : 0] >= 0;
  const int flag = on ? sflag[slot] : 0;
  const long long b0 = on ? sbase[slot] : 0;
  const T* ue = u + b0;
  // a pair is there if its position along both other axes is
  bool have[3];
  have[0] = on && (!p1 || (flag & 2)) && (!p2 || (flag & 4));
  have[1] = on && (!p1 || (flag & 1)) && (!p2 || (flag & 4));
  have[2] = on && (!p1 || (flag & 1)) && (!p2 || (flag & 2));
  const long long pe[3] = {est[1] * p1 + est[2] * p2, est[0] * p1 + est[2] * p2, est[0] * p1 + est[1] * p2};
  const int sb = (slot < BPB ? slot : 0) * EB * ES;
  const int zat = sb + (p1 + 2 * p2) * ES + l1 + PB * l2;  // this thread's z line (pair): shared and global
  const long long g0 = b0 + pe[2] * NPE + l;
  T v[BR][N1];
  // own elements, a z line (pair) per thread: coalesced, and no index arithmetic per value
  if (have[2]) {
#pragma unroll
    for (int s = 0; s < BR; ++s)
      if (s == 0 || (flag & 4)) {
#pragma unroll
        for (int i = 0; i < N1; ++i) v[s][i] = __ldg(u + g0 + s * est[2] * NPE + i * NF);
#pragma unroll
        for (int i = 0; i < N1; ++i) su[zat + 4 * s * ES + i * PZ] = v[s][i];
      }
  }
  T ov[3][outer_vals<T, N1>()], od[3][2];
#define DG_OUT(d, s) ((flag & ((8 << (s)) << (2 * (d)))) != 0)
  if (have[0])
    outer_traces<T, N1, BR, 0>(tab, ue, pe[0], l1, l2, est[0], flag & 1, DG_OUT(0, 0), DG_OUT(0, 1), vec, ov[0], od[0]);
  if (have[1])
    outer_traces<T, N1, BR, 1>(tab, ue, pe[1], l1, l2, est[1], flag & 2, DG_OUT(1, 0), DG_OUT(1, 1), vec, ov[1], od[1]);
  if (have[2])
    outer_traces<T, N1, BR, 2>(tab, ue, pe[2], l1, l2, est[2], flag & 4, DG_OUT(2, 0), DG_OUT(2, 1), vec, ov[2], od[2]);
  __syncthreads();
  // x: line (b, c) = (l1, l2)
  if (have[0]) {
    const int at = sb + (2 * p1 + 4 * p2) * ES + PB * l1 + PZ * l2;
    const bool sec = flag & 1;
#pragma unroll
    for (int s = 0; s < BR; ++s)
#pragma unroll
      for (int i = 0; i < N1; ++i) v[s][i] = s == 0 || sec ? su[at + s * ES + i] : (T)0;
    line_op<T, N1, BR, 0>(tab, v, ov[0], od[0], sec, DG_OUT(0, 0), DG_OUT(0, 1));
    const T sc = tab.mm[0][l];
#pragma unroll
    for (int s = 0; s < BR; ++s)
      if (s == 0 || sec) {
#pragma unroll
        for (int i = 0; i < N1; ++i) sacc[at + s * ES + i] = mul(sc, v[s][i]);
      }
  }
  __syncthreads();
  // y: line (a, c)
  if (have[1]) {
    const int at = sb + (p1 + 4 * p2) * ES + l1 + PZ * l2;
    const bool sec = flag & 2;
#pragma unroll
    for (int s = 0; s < BR; ++s)
#pragma unroll
      for (int i = 0; i < N1; ++i) v[s][i] = s == 0 || sec ? su[at + 2 * s * ES + i * PB] : (T)0;
    line_op<T, N1, BR, 1>(tab, v, ov[1], od[1], sec, DG_OUT(1, 0), DG_OUT(1, 1));
    const T sc = tab.mm[1][l];
#pragma unroll
    for (int s = 0; s < BR; ++s)
      if (s == 0 || sec) {
#pragma unroll
        for (int i = 0; i < N1; ++i) {
          T* p = sacc + at + 2 * s * ES + i * PB;
          *p = mad(sc, v[s][i], *p);
        }
      }
  }
  __syncthreads();
  // z: line (a, b), straight to the result
  if (have[2]) {
    const bool sec = flag & 4;
    T r[BR][N1];
    if (mode != 0) {
      const T* rp = mode == 1 ? rin : out;
#pragma unroll
      for (int s = 0; s < BR; ++s)
        if (s == 0 || sec) {
#pragma unroll
          for (int i = 0; i < N1; ++i) r[s][i] = rp[g0 + s * est[2] * NPE + i * NF];
        }
    }
#pragma unroll
    for (int s = 0; s < BR; ++s)
#pragma unroll
      for (int i = 0; i < N1; ++i) v[s][i] = s == 0 || sec ? su[zat + 4 * s * ES + i * PZ] : (T)0;
    line_op<T, N1, BR, 2>(tab, v, ov[2], od[2], sec, DG_OUT(2, 0), DG_OUT(2, 1));
    const T sc = tab.mm[2][l];
#pragma unroll
    for (int s = 0; s < BR; ++s)
      if (s == 0 || sec) {
#pragma unroll
        for (int i = 0; i < N1; ++i) {
          const T Au = mad(sc, v[s][i], sacc[zat + 4 * s * ES + i * PZ]);
          if constexpr (sizeof(T) == 8)
            v[s][i] = Au;
          else
            out[g0 + s * est[2] * NPE + i * NF] = mode == 0 ? Au : r[s][i] - Au;
        }
        if constexpr (sizeof(T) == 8) {  // a branch: the FP64 pipe would pay for a select's difference
          if (mode == 0) {
#pragma unroll
            for (int i = 0; i < N1; ++i) out[g0 + s * est[2] * NPE + i * NF] = v[s][i];
          } else {
#pragma unroll
            for (int i = 0; i < N1; ++i) out[g0 + s * est[2] * NPE + i * NF] = r[s][i] - v[s][i];
          }
        }
      }
  }
#undef DG_OUT
}

// The operator where there are too few elements to fill the chip: one element per
// block and a group of threads per direction, which work at the same time (a warp
// issues an FP64 operation every 67 cycles whatever else it has to do, so the chain
// that a thread runs is the kernel's time). The three results are scaled and added
// in the order of k_apply: the same bits.
// Measured (GB300, FP64, in a graph; the passes one after the other before): 4^3, p =
// 4, 4 fields 10.3 -> 6.2 us, 5 x 7 x 3, p = 5, 3 fields 24.0 -> 15.7 us, 4^3, p = 8, 1
// field 31.6 -> 14.3 us.
template <int N1>
struct ApplySmall {
  static constexpr int GROUP = (N1 * N1 + 31) / 32 * 32;  // whole warps per direction
  static constexpr int THREADS = 3 * GROUP;
};

template <typename T, int N1, int D>
__device__ __forceinline__ void small_pass(const ApplyTab<T, N1>& tab, const T* su, T* res, int l1, int l2, const T* ov,
                                           const T* od, bool in0, bool in1) {
  using Y = LineLayout<N1>;
  constexpr int ST = D == 0 ? 1 : (D == 1 ? Y::PB : Y::PZ);
  const int at = D == 0 ? Y::PB * l1 + Y::PZ * l2 : (D == 1 ? l1 + Y::PZ * l2 : l1 + Y::PB * l2);
  T v[1][N1];
#pragma unroll
  for (int i = 0; i < N1; ++i) v[0][i] = su[at + ST * i];
  line_op<T, N1, 1, D>(tab, v, ov, od, false, in0, in1);
#pragma unroll
  for (int i = 0; i < N1; ++i) res[at + ST * i] = v[0][i];
}

template <typename T, int N1>
__global__ void __launch_bounds__(ApplySmall<N1>::THREADS)
    k_apply_small(const __grid_constant__ ApplyTab<T, N1> tab, const T* __restrict__ u, T* __restrict__ out,
                  const T* __restrict__ rin, const int* __restrict__ act, int mode, int vec_i) {
  using Y = LineLayout<N1>;
  constexpr int NF = N1 * N1, NPE = NF * N1, GROUP = ApplySmall<N1>::GROUP, NT = ApplySmall<N1>::THREADS;
  __shared__ T su[Y::ES], sr[3][Y::ES];
  const int nx = tab.n[0], ny = tab.n[1], E = nx * ny * tab.n[2];
  const int k = blockIdx.x / E, e = blockIdx.x - k * E;
  const int ex = e % nx, eq = e / nx, ey = eq % ny, ez = eq / ny;
  const long long g0 = (long long)act[k] * tab.Nq + (long long)e * NPE;
  const T* ue = u + g0;
  for (int t = threadIdx.x; t < NPE; t += NT) su[t % N1 + Y::PB * ((t / N1) % N1) + Y::PZ * (t / NF)] = __ldg(ue + t);
  const int d = threadIdx.x / GROUP, l = threadIdx.x - d * GROUP, l1 = l % N1, l2 = l / N1;
  const bool on = l < NF, vec = vec_i != 0;
  T ov[outer_vals<T, N1>()], od[2];
  const bool in0 = (d == 0 ? ex : d == 1 ? ey : ez) > 0;
  const bool in1 = d == 0 ? ex < nx - 1 : d == 1 ? ey < ny - 1 : ez < tab.n[2] - 1;
  if (on) {
    if (d == 0)
      outer_traces<T, N1, 1, 0>(tab, ue, 0, l1, l2, 1, false, in0, in1, vec, ov, od);
    else if (d == 1)
      outer_traces<T, N1, 1, 1>(tab, ue, 0, l1, l2, nx, false, in0, in1, vec, ov, od);
    else
      outer_traces<T, N1, 1, 2>(tab, ue, 0, l1, l2, (long long)nx * ny, false, in0, in1, vec, ov, od);
  }
  __syncthreads();
  if (on) {
    if (d == 0)
      small_pass<T, N1, 0>(tab, su, sr[0], l1, l2, ov, od, in0, in1);
    else if (d == 1)
      small_pass<T, N1, 1>(tab, su, sr[1], l1, l2, ov, od, in0, in1);
    else
      small_pass<T, N1, 2>(tab, su, sr[2], l1, l2, ov, od, in0, in1);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < NPE; t += NT) {
    const int a = t % N1, b = (t / N1) % N1, c = t / NF, at = a + Y::PB * b + Y::PZ * c;
    T Au = mul(tab.mm[0][b + N1 * c], sr[0][at]);
    Au = mad(tab.mm[1][a + N1 * c], sr[1][at], Au);
    Au = mad(tab.mm[2][a + N1 * b], sr[2][at], Au);
    out[g0 + t] = mode == 0 ? Au : (mode == 1 ? rin : out)[g0 + t] - Au;
  }
}

template <typename T, int N1>
static cudaError_t apply_small(const LevelOp& hop, int mode, const T* u, T* out, const T* rin, const int* act, int nact,
                               cudaStream_t s) {
  ApplyTab<T, N1> tab;
  fill_tab<T, N1>(tab, hop);
  const int vec = ((uintptr_t)u & 15) == 0 && (N1 * N1 * N1 * sizeof(T)) % 16 == 0 && (hop.Nq * sizeof(T)) % 16 == 0;
  count_launch();
  k_apply_small<T, N1><<<(unsigned)(hop.E * nact), ApplySmall<N1>::THREADS, 0, s>>>(tab, u, out, rin, act, mode, vec);
  return cudaGetLastError();
}

template <typename T, int N1, int BR, int BPB = apply_bpb<T, N1, BR>()>
static cudaError_t apply_br(const LevelOp& hop, int mode, const T* u, T* out, const T* rin, const int* act, int nact,
                            cudaStream_t s) {
  using C = ApplyCfg<T, N1, BR, BPB>;
  ApplyTab<T, N1> tab;
  fill_tab<T, N1>(tab, hop);
  long long per = 1;
  for (int d = 0; d < 3; ++d) {
    tab.nb[d] = (hop.n[d] + BR - 1) / BR;
    per *= tab.nb[d];
  }
  tab.items = per * nact;
  const long long blocks = (tab.items + C::BPB - 1) / C::BPB;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  // 16-byte reads of an element's values: the field and every element of it aligned
  const int vec = ((uintptr_t)u & 15) == 0 && (C::NPE * sizeof(T)) % 16 == 0 && (hop.Nq * sizeof(T)) % 16 == 0;
  auto kern = k_apply<T, N1, BR, BPB>;
  if (C::SMEM > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e != cudaSuccess) return e;
  }
  count_launch();
  kern<<<(unsigned)blocks, C::THREADS, C::SMEM, s>>>(tab, u, out, rin, act, mode, vec);
  return cudaGetLastError();
}

// Few elements: one group of threads per direction, while its warps are at most 24 per
// SM in FP64 (16 at p = 5, where 36 lines leave half of a group's lanes idle) and 13 in
// FP32 and at p <= 3. Measured around the line (us, small / single elements): FP64 p = 1
// 512 elements 3.4 / 3.6, 2048 6.8 / 3.7; p = 2 512 4.9 / 5.8, 1024 7.5 / 6.0; p = 3 512
// 7.5 / 7.6, 2048 22 / 14; p = 4 512 9.4 / 10.0, 1024 15.1 / 16.5, 4096 51 / 45; p = 5 375
// 15.6 / 16.0, 512 19.9 / 16.1; p = 6 512 23.5 / 23.4, 2048 75 / 65; p = 8 250 24.8 / 31.3;
// FP32 p = 5 315 3.7 / 4.2, 1260 6.3 / 5.1; p = 4 256 2.9 / 3.3, 1024 3.9 / 3.6; p = 8 64
// 4.0 / 4.4, 256 5.4 / 4.5.
// Then bricks of eight elements in FP32, where reading the neighbours is what bounds
// the kernel (single elements / bricks: p = 6 4096 elements 10.7 / 8.2 us, 512 4.1 /
// 4.5; p = 5 2880 6.5 / 6.3, 960 4.3 / 4.9), with two blocks for every SM and, on odd
// meshes, at least half of the elements that the bricks have room for; single
// elements otherwise and in FP64 (bound by the FP64 pipe, to which a brick saves
// nothing), in blocks of the size that leaves the busiest SM fewer warps (small /
// full blocks: p = 5 512 elements 16.1 / 23.1, 1372 29.1 / 42.8, 20480 362 / 342; p = 6
// 1536 55 / 65, 2048 68 / 65).
template <typename T, int N1>
static cudaError_t apply_n1(const LevelOp& hop, int mode, const T* u, T* out, const T* rin, const int* act, int nact,
                            cudaStream_t s) {
  if (nact == 0) return cudaSuccess;
  const long long items = (long long)nact * hop.E;
  constexpr int warps = sizeof(T) == 4 || N1 <= 4 ? 13 : N1 == 6 ? 16 : 24;
  if (items * (ApplySmall<N1>::THREADS / 32) <= 152 * warps)
    return apply_small<T, N1>(hop, mode, u, out, rin, act, nact, s);
  if constexpr (sizeof(T) == 4) {
    long long br = nact;
    for (int d = 0; d < 3; ++d) br *= (hop.n[d] + 1) / 2;
    if (br / ApplyCfg<T, N1, 2>::BPB >= 2 * 152 && 8 * br <= 2 * items)
      return apply_br<T, N1, 2>(hop, mode, u, out, rin, act, nact, s);
  } else if constexpr (apply_few<N1>() != apply_bpb<T, N1, 1>()) {
    using F = ApplyCfg<T, N1, 1>;
    using S = ApplyCfg<T, N1, 1, apply_few<N1>()>;
    auto busiest = [&](long long bpb, int threads) { return ((items + bpb - 1) / bpb + 151) / 152 * (threads / 32); };
    if (busiest(S::BPB, S::THREADS) < busiest(F::BPB, F::THREADS))
      return apply_br<T, N1, 1, S::BPB>(hop, mode, u, out, rin, act, nact, s);
  }
  return apply_br<T, N1, 1>(hop, mode, u, out, rin, act, nact, s);
}

template <typename T>
cudaError_t launch_apply(const LevelOp& hop, int mode, const T* u, T* out, const T* rin, const int* act, int nact,
                         cudaStream_t s) {
  switch (hop.n1) {
    case 2: return apply_n1<T, 2>(hop, mode, u, out, rin, act, nact, s);
    case 3: return apply_n1<T, 3>(hop, mode, u, out, rin, act, nact, s);
    case 4: return apply_n1<T, 4>(hop, mode, u, out, rin, act, nact, s);
    case 5: return apply_n1<T, 5>(hop, mode, u, out, rin, act, nact, s);
    case 6: return apply_n1<T, 6>(hop, mode, u, out, rin, act, nact, s);
    case 7: return apply_n1<T, 7>(hop, mode, u, out, rin, act, nact, s);
    case 8: return apply_n1<T, 8>(hop, mode, u, out, rin, act, nact, s);
    case 9: return apply_n1<T, 9>(hop, mode, u, out, rin, act, nact, s);
    default: return cudaErrorInvalidValue;
  }
}

// Jacobi diagonal of the Kronecker sum: Kx[a,a] My Mz + Mx Ky[b,b] Mz + Mx My Kz[c,c].
template <typename T>
__global__ void k_inv_diag(const LevelOp* __restrict__ op, T* __restrict__ invD) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= op->Nq) return;
  const int n1 = op->n1, npe = n1 * n1 * n1;
  const int e = (int)(i / npe), loc = (int)(i % npe);
  const int a = loc % n1, b = (loc / n1) % n1, c = loc / (n1 * n1);
  const int nx = op->n[0], ny = op->n[1], nz = op->n[2];
  const int ex = e % nx, ey = (e / nx) % ny, ez = e / (nx * ny);
  const int tyx = (ex == 0 ? 1 : 0) | (ex == nx - 1 ? 2 : 0);
  const int tyy = (ey == 0 ? 1 : 0) | (ey == ny - 1 ? 2 : 0);
  const int tyz = (ez == 0 ? 1 : 0) | (ez == nz - 1 ? 2 : 0);
  const double mx = op->ax[0].m[a], my = op->ax[1].m[b], mz = op->ax[2].m[c];
  const double dval = op->ax[0].Kd[tyx][a * n1 + a] * my * mz + mx * op->ax[1].Kd[tyy][b * n1 + b] * mz +
                      mx * my * op->ax[2].Kd[tyz][c * n1 + c];
  invD[i] = (T)(1.0 / dval);
}

template <typename T>
cudaError_t launch_inv_diag(const LevelOp& hop, const LevelOp* dop, T* invD, cudaStream_t s) {
  const long long n = hop.Nq;
  count_launch();
  k_inv_diag<T><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(dop, invD);
  return cudaGetLastError();
}

template cudaError_t launch_apply<double>(const LevelOp&, int, const double*, double*, const double*, const int*, int,
                                          cudaStream_t);
template cudaError_t launch_apply<float>(const LevelOp&, int, const float*, float*, const float*, const int*, int,
                                         cudaStream_t);
template cudaError_t launch_inv_diag<double>(const LevelOp&, const LevelOp*, double*, cudaStream_t);
template cudaError_t launch_inv_diag<float>(const LevelOp&, const LevelOp*, float*, cudaStream_t);

}  // namespace dg
