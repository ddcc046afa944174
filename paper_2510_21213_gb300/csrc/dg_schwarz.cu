// Overlapping Schwarz smoother for the hp-multigrid of Sec. 6.4.
//
// The paper does not specify the smoother. With the penalty of Sec. 3.5
// (eps = 1/8, i.e. eight times the coercivity bound) point- and element-block
// Jacobi smoothers leave continuous high-order modes undamped, so each
// multigrid level uses additive Schwarz over element patches with one node of
// overlap, accelerated by Chebyshev iteration. Each patch problem is solved
// exactly by fast diagonalisation (the patch operator is a Kronecker sum of
// restricted 1-D matrices; tables built at setup):
//   k_schwarz_patch:  zp_e = A_P(e)^-1 R_P(e) r
//   k_schwarz_gather: z = sum_e R_P(e)^T zp_e          (each node gathers the
//                     at most 8 patches covering it; no atomics), fused with
//                     the Chebyshev update d = c1 d + c2 z, x += d
//
// Patch kernel. FP64 is bound by the FP64 pipe, so what counts is the number of
// operations; FP32 by shared-memory accesses, so what counts is how often a
// value goes through shared memory and how many products share a table load.
//   - A patch whose two ends look alike (all but the two elements next to either
//     boundary) has a 1-D matrix that is invariant under reversal: its modes are
//     even or odd, and on the sums and differences of mirrored nodes each half
//     costs a quarter of the dense product. m^2 / 2 + m multiply-adds per line
//     instead of m^2 (m = p + 3).
//   - z forward on the values as they come from global memory; y forward; the
//     whole x direction in registers (transform, division by the eigenvalue sum,
//     transform back, each table row loaded once for both); y backward; z
//     backward straight to global memory, consecutive threads on consecutive
//     values. 8 shared-memory accesses a node instead of 16.
//   - FP64 multiplies by a tabulated reciprocal of the eigenvalue sum (a division
//     costs about ten operations of the FP64 pipe).
//   - A thread owns LPT lines of one patch in every pass and reads table rows
//     with 16-byte loads, so one load serves 4 LPT products. The tables of the at
//     most five position classes of an axis stay in shared memory, loaded once
//     by each block of a persistent grid.
// Measured (GB300; before: all six passes through shared memory, dense
// transforms, a division per node, tables per patch): FP64 16^3, p = 7, 42
// sources 22.0 -> 15.6 ms, 8^3, p = 6, 56 sources 2.33 -> 1.91 ms; FP32 8^3, p = 6, 56
// sources 150 -> 98 us, 16^3, p = 3, 42 sources 271 -> 137 us, p = 1 86 -> 37 us, 6 x 10
// x 8, p = 5, 21 sources 49 -> 20 us (in a graph; 2 to 3 us more by single launches).
// FP64 runs at the rate of its pipe; FP32 issues in 55 % of the cycles with a quarter of
// the warps resident (96 registers).
#include "dg_fdm.h"
#include "dg_swtc.h"

namespace dg {

constexpr int GATHER_WAVE = 8;  // gather grid: at most this many blocks per SM per source list (16: the same to 1 %)

template <typename T, int N1>
struct SwCfg {
  static constexpr int MP = N1 + 2, MP2 = MP * MP, MP3 = MP2 * MP;
  static constexpr int HO = MP / 2, HE = MP - HO;
  static constexpr int W = 16 / (int)sizeof(T);           // values of a 16-byte load
  static constexpr int RP = (MP + W - 1) / W * W;         // padded table row
  static constexpr int TB = (MP + 1) * RP;                // one table: MP rows and the eigenvalues
  // lines per thread: FP32 as many as keep the lanes of a patch busy; FP64 one
  // (bound by its pipe, and short chains matter on small problems)
  static constexpr int LPT = sizeof(T) == 8 ? 1 : MP == 4 ? 4 : MP == 5 ? 5 : MP == 7 || MP == 8 ? 2 : MP == 10 ? 4 : 3;
  static constexpr int TPE = (MP2 + LPT - 1) / LPT;       // threads of a patch
  // node (i, j, k) of a slot at i + SJ j + SK k + SE slot: the strides with the
  // fewest shared-memory wavefronts of the passes in FP32, counted over the
  // warps of a block (1.0 to 1.8 per access; the dense layout takes up to 8);
  // FP64 keeps the dense layout
  static constexpr int SJ = sizeof(T) == 8 ? MP : MP == 4 ? 5 : MP == 5 ? 6 : MP == 6 ? 9 : MP == 7 ? 8 : MP == 8 ? 9
                                                  : MP == 9 ? 9 : MP == 10 ? 13 : 12;
  static constexpr int SK = sizeof(T) == 8 ? MP2 : MP == 4 ? 19 : MP == 5 ? 30 : MP == 6 ? 70 : MP == 7 ? 71
                                                  : MP == 8 ? 72 : MP == 9 ? 111 : MP == 10 ? 138 : 139;
  static constexpr int SE = sizeof(T) == 8 ? MP3 : MP == 4 ? 76 : MP == 5 ? 165 : MP == 6 ? 428 : MP == 7 ? 505
                                                  : MP == 8 ? 575 : MP == 9 ? 987 : MP == 10 ? 1369 : 1545;
  static_assert(SK >= SJ * (MP - 1) + MP && SE >= (SK + SJ + 1) * (MP - 1) + 1, "patch layout overlaps");
  // slots of a block: the fewest idle lanes in its last warp (as best_bpb of the operator)
  static constexpr int slots(int small) {
    int best = 1;
    for (int b = 2; b * TPE <= 320; ++b) {
      const int tb = (b * TPE + 31) / 32 * 32, t0 = (best * TPE + 31) / 32 * 32;
      if (b * t0 > best * tb || (b * t0 == best * tb && tb <= small)) best = b;
    }
    return best;
  }
};

template <typename T, int N1, int EPB_ = SwCfg<T, N1>::slots(sizeof(T) == 4 ? 128 : 64)>
struct SwShape {
  using C = SwCfg<T, N1>;
  static constexpr int EPB = EPB_;
  static constexpr int THREADS = (EPB * C::TPE + 31) / 32 * 32;
  // resident threads per SM asked of ptxas (p = 6, 8^3, 56 sources: 101 us at 640, 104 at 768, 147 at 1024; two or
  // one line per thread instead of three 105 to 117)
  static constexpr int WANT = sizeof(T) == 4 && C::MP < 10 ? 640 : 512;
  static constexpr int MINB = WANT / THREADS < 1 ? 1 : WANT / THREADS > 32 ? 32 : WANT / THREADS;
  static constexpr size_t SMEM = sizeof(T) * ((size_t)SW_MAXCLS * 3 * C::TB + (size_t)EPB * C::SE);
};

template <typename T, int N1, int EPB>
__global__ void __launch_bounds__(SwShape<T, N1, EPB>::THREADS, SwShape<T, N1, EPB>::MINB)
    k_schwarz_patch(const __grid_constant__ SwGeom g, const unsigned char* __restrict__ blob, const T* __restrict__ r,
                    T* __restrict__ zp, const int* __restrict__ act, int nact) {
  using C = SwCfg<T, N1>;
  using H = SwShape<T, N1, EPB>;
  constexpr int MP = C::MP, MP2 = C::MP2, MP3 = C::MP3, NF = N1 * N1, NPE = NF * N1;
  constexpr int SJ = C::SJ, SK = C::SK, SE = C::SE, RP = C::RP, TB = C::TB, TPE = C::TPE, LPT = C::LPT;
  constexpr int NT = H::THREADS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tabs = reinterpret_cast<T*>(smem_raw);
  T* buf = tabs + SW_MAXCLS * 3 * TB;
  __shared__ int spos[EPB][3];   // per axis: table | patch size | left halo | symmetric
  __shared__ int selem[EPB];     // element, -1: none
  __shared__ long long ssrc[EPB];
  const int nx = g.n[0], ny = g.n[1];
  const long long E = (long long)nx * ny * g.n[2], Nq = E * NPE, items = E * nact;
  const int* pos = reinterpret_cast<const int*>(blob + g.pos_off);
  const T* gt = reinterpret_cast<const T*>(blob + g.tab_off);
  for (int t = threadIdx.x; t < g.ntab * TB / C::W; t += NT)
    reinterpret_cast<uint4*>(tabs)[t] = reinterpret_cast<const uint4*>(gt)[t];
  const int slot = threadIdx.x / TPE, lt = threadIdx.x - slot * TPE;
  const int sl = slot < EPB ? slot : 0;
  T* b = buf + sl * SE;
  const long long groups = (items + EPB - 1) / EPB;
  for (long long grp = blockIdx.x; grp < groups; grp += gridDim.x) {
    if (threadIdx.x < EPB) {
      const long long it = grp * EPB + threadIdx.x;
      const bool v = it < items;
      const int k = v ? (int)(it / E) : 0, e = v ? (int)(it - k * E) : 0;
      const int ex = e % nx, q = e / nx, ey = q % ny, ez = q / ny;
      selem[threadIdx.x] = v ? e : -1;
      spos[threadIdx.x][0] = pos[ex];
      spos[threadIdx.x][1] = pos[nx + ey];
      spos[threadIdx.x][2] = pos[nx + ny + ez];
      ssrc[threadIdx.x] = act[k];
    }
    __syncthreads();  // slots (and, the first time, tables) ready; the previous group's reads of them are done
    const int e = selem[sl];
    const bool on = slot < EPB && e >= 0;
    const int px = spos[sl][0], py = spos[sl][1], pz = spos[sl][2];
    const long long src = ssrc[sl];
    const T *tx = tabs + sw_tab(px) * TB, *ty = tabs + sw_tab(py) * TB, *tz = tabs + sw_tab(pz) * TB;
    T v[LPT][MP];
    if (on) {
      // z forward, lines (i, j): the patch residual (own element plus one node
      // layer of each neighbour), zero outside the domain
      const int oLx = sw_halo(px), oLy = sw_halo(py), oLz = sw_halo(pz);
      const int mx = sw_size(px), my = sw_size(py), mz = sw_size(pz);
      const T* rr = r + src * Nq;
      const long long pe = (long long)nx * ny * NPE;  // values of a z layer of elements
#pragma unroll
      for (int s = 0; s < LPT; ++s) {
        const int l = lt + TPE * s, i = l % MP, j = l / MP;
        const bool in = l < MP2 && i < mx && j < my;
        int a = i - oLx, bb = j - oLy, ee = e;
        if (a < 0) {
          a = N1 - 1;
          ee -= 1;
        } else if (a >= N1) {
          a = 0;
          ee += 1;
        }
        if (bb < 0) {
          bb = N1 - 1;
          ee -= nx;
        } else if (bb >= N1) {
          bb = 0;
          ee += nx;
        }
        const T* p = rr + (long long)ee * NPE + (a + N1 * bb);
        const T *below = p - pe + (N1 - 1) * NF, *own = p - oLz * NF, *above = p + pe;
        v[s][0] = in ? __ldg(oLz ? below : own) : (T)0;
#pragma unroll
        for (int k = 1; k < N1; ++k) v[s][k] = in ? __ldg(own + NF * k) : (T)0;
        v[s][N1] = in && N1 < mz ? __ldg(oLz ? own + NF * N1 : above) : (T)0;
        v[s][N1 + 1] = in && N1 + 1 < mz ? __ldg(above) : (T)0;
      }
      sw_fwd<T, MP, LPT>(sw_sym(pz), tz, RP, v, [&](int s, int q, T a) {
        const int l = lt + TPE * s;
        if (MP2 % LPT == 0 || l < MP2) b[l % MP + SJ * (l / MP) + SK * q] = a;
      });
    }
    __syncthreads();
    if (on) {
      // y forward, lines (i, k)
      int at[LPT];
#pragma unroll
      for (int s = 0; s < LPT; ++s) {
        const int l = lt + TPE * s;
        at[s] = MP2 % LPT == 0 || l < MP2 ? l % MP + SK * (l / MP) : 0;
#pragma unroll
        for (int j = 0; j < MP; ++j) v[s][j] = b[at[s] + SJ * j];
      }
      sw_fwd<T, MP, LPT>(sw_sym(py), ty, RP, v, [&](int s, int q, T a) {
        if (MP2 % LPT == 0 || lt + TPE * s < MP2) b[at[s] + SJ * q] = a;
      });
    }
    __syncthreads();
    if (on) {
      // x, lines (j, k)
      T w[LPT][MP];
      const T* lx = tx + MP * RP;
      T lyz[LPT];
      const T* inv[LPT];
#pragma unroll
      for (int s = 0; s < LPT; ++s) {
        const int l = lt + TPE * s, ll = MP2 % LPT == 0 || l < MP2 ? l : 0, j = ll % MP, k = ll / MP;
        const int at = SJ * j + SK * k;
#pragma unroll
        for (int i = 0; i < MP; ++i) v[s][i] = b[at + i];
        if constexpr (sizeof(T) == 8) {
          inv[s] = reinterpret_cast<const T*>(blob + g.inv_off) +
                   (((long long)sw_cls(pz) * SW_MAXCLS + sw_cls(py)) * SW_MAXCLS + sw_cls(px)) * MP3 + ll;
          lyz[s] = (T)0;
        } else {
          inv[s] = nullptr;
          lyz[s] = ty[MP * RP + j] + tz[MP * RP + k];
        }
      }
      sw_mid<T, MP, LPT>(sw_sym(px), tx, RP, v, w, [&](int s, int q, T a) -> T {
        if constexpr (sizeof(T) == 8)
          return a * __ldg(inv[s] + q * MP2);
        else
          return __fdividef(a, lx[q] + lyz[s]);  // within 2 ulp; the sums are positive and far from the range limits
      });
#pragma unroll
      for (int s = 0; s < LPT; ++s) {
        const int l = lt + TPE * s, at = SJ * (l % MP) + SK * (l / MP);
        if (MP2 % LPT == 0 || l < MP2) {
#pragma unroll
          for (int i = 0; i < MP; ++i) b[at + i] = w[s][i];
        }
      }
    }
    __syncthreads();
    if (on) {
      // y backward, lines (i, k)
      int at[LPT];
#pragma unroll
      for (int s = 0; s < LPT; ++s) {
        const int l = lt + TPE * s;
        at[s] = MP2 % LPT == 0 || l < MP2 ? l % MP + SK * (l / MP) : 0;
      }
      sw_bwd<T, MP, LPT>(sw_sym(py), ty, RP, v, [&](int s, int q) -> T { return b[at[s] + SJ * q]; });
#pragma unroll
      for (int s = 0; s < LPT; ++s)
        if (MP2 % LPT == 0 || lt + TPE * s < MP2) {
#pragma unroll
          for (int j = 0; j < MP; ++j) b[at[s] + SJ * j] = v[s][j];
        }
    }
    __syncthreads();
    if (on) {
      // z backward, lines (i, j), to the patch buffer: node (i, j, k) at i + MP j + MP^2 k
      sw_bwd<T, MP, LPT>(sw_sym(pz), tz, RP, v, [&](int s, int q) -> T {
        const int l = lt + TPE * s, ll = MP2 % LPT == 0 || l < MP2 ? l : 0;
        return b[ll % MP + SJ * (ll / MP) + SK * q];
      });
      T* out = zp + (src * E + e) * MP3;
#pragma unroll
      for (int s = 0; s < LPT; ++s) {
        const int l = lt + TPE * s;
        if (MP2 % LPT == 0 || l < MP2) {
#pragma unroll
          for (int k = 0; k < MP; ++k) out[l + MP2 * k] = v[s][k];
        }
      }
    }
    __syncthreads();  // everybody is done with the slots and the buffer
  }
}

// The same patch solves where there are too few patches to fill the chip: one
// patch per block and two lanes per line, so that the chain of operations that a
// thread runs is half as long (a warp issues an FP64 operation every 67 cycles
// whatever else it has to do, so at 4^3 elements and p = 4 that chain is the
// kernel's time). Lane h = 0 takes the even modes (of a patch without symmetry the
// first half of the modes, and of the nodes on the way back), h = 1 the rest; even
// and odd parts of the nodes change hands by a shuffle. Each sum is that of
// k_schwarz_patch, so the results are the same bits. Only the patch's own three
// tables are staged, and the reciprocals are loaded up front.
// Measured (GB300, FP64, 4^3, 4 sources; k_schwarz_patch with one patch per block, and
// with the several that are used for many patches): p = 4 13.3 us (14.1, 22.4), p = 2 5.9
// (8.9, 10.1).
template <typename T, int N1>
struct SwSmall {
  using C = SwCfg<T, N1>;
  static constexpr int THREADS = (2 * C::MP2 + 31) / 32 * 32;
  static constexpr size_t SMEM = sizeof(T) * (3 * C::TB + (size_t)C::SE);
};

// modes h HE + t of the line v: put(t, sum_i S[i][q] v[i])
template <typename T, int MP, int RP, typename P>
__device__ __forceinline__ void sw_fwd2(bool sym, const T* tb, int h, const T* v, P&& put) {
  constexpr int HO = MP / 2, HE = MP - HO;
  const T* row = tb + h * HE * RP;
  const int n = h ? HO : HE;
  if (sym) {
    T x[HE];
#pragma unroll
    for (int i = 0; i < HO; ++i) x[i] = h ? v[i] - v[MP - 1 - i] : v[i] + v[MP - 1 - i];
    if (HE > HO) x[HE - 1] = h ? (T)0 : v[HO];  // the odd rows are zero there
#pragma unroll
    for (int t = 0; t < HE; ++t)
      if (t < n) {
        T a = row[t * RP] * x[0];
#pragma unroll
        for (int i = 1; i < HE; ++i) a += row[t * RP + i] * x[i];
        put(t, a);
      }
  } else {
#pragma unroll
    for (int t = 0; t < HE; ++t)
      if (t < n) {
        T a = row[t * RP] * v[0];
#pragma unroll
        for (int i = 1; i < MP; ++i) a += row[t * RP + i] * v[i];
        put(t, a);
      }
  }
}
// nodes from the modes at line + st q: put(node, value) for this lane's nodes (the
// first HE with h = 0, the others with h = 1), after every lane has read its modes.
// Every lane of the warp takes part.
template <typename T, int MP, int RP, typename P>
__device__ __forceinline__ void sw_bwd2(bool sym, const T* tb, int h, const T* line, int st, P&& put) {
  constexpr int HO = MP / 2, HE = MP - HO;
  T x[HE];
#pragma unroll
  for (int t = 0; t < HE; ++t) x[t] = (T)0;
  if (sym) {
    const int n = h ? HO : HE;
#pragma unroll
    for (int t = 0; t < HE; ++t)
      if (t < n) {
        const int q = h * HE + t;
        const T c = line[st * q];
#pragma unroll
        for (int i = 0; i < HE; ++i) x[i] += tb[q * RP + i] * c;
      }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < HO; ++i) {
      const T y = __shfl_xor_sync(0xffffffffu, x[i], 1);
      if (h == 0)
        put(i, x[i] + y);
      else
        put(MP - 1 - i, y - x[i]);
    }
    if (HE > HO && h == 0) put(HO, x[HE - 1]);
  } else {
#pragma unroll
    for (int q = 0; q < MP; ++q) {
      const T c = line[st * q];
#pragma unroll
      for (int t = 0; t < HE; ++t)
        if (t < HO || h == 0) x[t] += tb[q * RP + h * HE + t] * c;
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < HE; ++t)
      if (t < HO || h == 0) put(h * HE + t, x[t]);
  }
}

template <typename T, int N1>
__global__ void __launch_bounds__(SwSmall<T, N1>::THREADS)
    k_schwarz_patch_small(const __grid_constant__ SwGeom g, const unsigned char* __restrict__ blob,
                          const T* __restrict__ r, T* __restrict__ zp, const int* __restrict__ act) {
  using C = SwCfg<T, N1>;
  constexpr int MP = C::MP, MP2 = C::MP2, MP3 = C::MP3, NF = N1 * N1, NPE = NF * N1, HE = C::HE, HO = C::HO;
  constexpr int SJ = C::SJ, SK = C::SK, RP = C::RP, TB = C::TB, NT = SwSmall<T, N1>::THREADS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tabs = reinterpret_cast<T*>(smem_raw);
  T* b = tabs + 3 * TB;
  const int nx = g.n[0], ny = g.n[1], E = nx * ny * g.n[2];
  const int k = blockIdx.x / E, e = blockIdx.x - k * E;
  const int ex = e % nx, eq = e / nx, ey = eq % ny, ez = eq / ny;
  const int* pos = reinterpret_cast<const int*>(blob + g.pos_off);
  const int px = __ldg(pos + ex), py = __ldg(pos + nx + ey), pz = __ldg(pos + nx + ny + ez);
  const long long src = act[k], Nq = (long long)E * NPE;
  const T* gt = reinterpret_cast<const T*>(blob + g.tab_off);
  const int from[3] = {sw_tab(px), sw_tab(py), sw_tab(pz)};
#pragma unroll
  for (int d = 0; d < 3; ++d)
    for (int t = threadIdx.x; t < TB / C::W; t += NT)
      reinterpret_cast<uint4*>(tabs + d * TB)[t] = __ldg(reinterpret_cast<const uint4*>(gt + from[d] * TB) + t);
  const T *tx = tabs, *ty = tabs + TB, *tz = tabs + 2 * TB;
  const int h = threadIdx.x & 1, l0 = threadIdx.x >> 1;
  const bool on = l0 < MP2;
  const int l = on ? l0 : 0, l1 = l % MP, l2 = l / MP;
  // z line (i, j) = (l1, l2) of the patch residual, zero outside the domain
  T v[MP], inv[HE];
  {
    const int oLx = sw_halo(px), oLy = sw_halo(py), oLz = sw_halo(pz);
    const int mz = sw_size(pz);
    const bool in = on && l1 < sw_size(px) && l2 < sw_size(py);
    int a = l1 - oLx, bb = l2 - oLy, ee = e;
    if (a < 0) {
      a = N1 - 1;
      ee -= 1;
    } else if (a >= N1) {
      a = 0;
      ee += 1;
    }
    if (bb < 0) {
      bb = N1 - 1;
      ee -= nx;
    } else if (bb >= N1) {
      bb = 0;
      ee += nx;
    }
    const T* p = r + src * Nq + (long long)ee * NPE + (a + N1 * bb);
    const long long pe = (long long)nx * ny * NPE;
    const T *below = p - pe + (N1 - 1) * NF, *own = p - oLz * NF, *above = p + pe;
    v[0] = in ? __ldg(oLz ? below : own) : (T)0;
#pragma unroll
    for (int c = 1; c < N1; ++c) v[c] = in ? __ldg(own + NF * c) : (T)0;
    v[N1] = in && N1 < mz ? __ldg(oLz ? own + NF * N1 : above) : (T)0;
    v[N1 + 1] = in && N1 + 1 < mz ? __ldg(above) : (T)0;
  }
  if constexpr (sizeof(T) == 8) {
    const T* ip = reinterpret_cast<const T*>(blob + g.inv_off) +
                  (((long long)sw_cls(pz) * SW_MAXCLS + sw_cls(py)) * SW_MAXCLS + sw_cls(px)) * MP3 + l;
#pragma unroll
    for (int t = 0; t < HE; ++t) inv[t] = t < HO || h == 0 ? __ldg(ip + (h * HE + t) * MP2) : (T)0;
  }
  __syncthreads();
  const int az = l1 + SJ * l2, ay = l1 + SK * l2, ax = SJ * l1 + SK * l2;
  sw_fwd2<T, MP, RP>(sw_sym(pz), tz, h, v, [&](int t, T a) {
    if (on) b[az + SK * (h * HE + t)] = a;
  });
  __syncthreads();
#pragma unroll
  for (int j = 0; j < MP; ++j) v[j] = b[ay + SJ * j];
  __syncwarp();
  sw_fwd2<T, MP, RP>(sw_sym(py), ty, h, v, [&](int t, T a) {
    if (on) b[ay + SJ * (h * HE + t)] = a;
  });
  __syncthreads();
#pragma unroll
  for (int i = 0; i < MP; ++i) v[i] = b[ax + i];
  __syncwarp();
  const T lyz = ty[MP * RP + l1] + tz[MP * RP + l2];
  sw_fwd2<T, MP, RP>(sw_sym(px), tx, h, v, [&](int t, T a) {
    if constexpr (sizeof(T) == 8)
      a *= inv[t];
    else
      a = __fdividef(a, tx[MP * RP + h * HE + t] + lyz);
    if (on) b[ax + h * HE + t] = a;
  });
  __syncwarp();
  // back: the values of a line's other lane are read before any of its nodes is written
  auto back = [&](bool sym, const T* tb, int at, int st, auto&& put) {
    sw_bwd2<T, MP, RP>(sym, tb, h, b + at, st, put);
  };
  back(sw_sym(px), tx, ax, 1, [&](int i, T a) {
    if (on) b[ax + i] = a;
  });
  __syncthreads();
  back(sw_sym(py), ty, ay, SJ, [&](int j, T a) {
    if (on) b[ay + SJ * j] = a;
  });
  __syncthreads();
  T* out = zp + (src * E + e) * MP3 + l;
  back(sw_sym(pz), tz, az, SK, [&](int kk, T a) {
    if (on) out[MP2 * kk] = a;
  });
}

template <typename T, int N1, typename H = SwShape<T, N1>>
static cudaError_t patch_fill(const SwTables& tb, const T* r, T* zp, const int* act, int nact, cudaStream_t s) {
  const SwGeom& g = tb.geom;
  const long long items = (long long)g.n[0] * g.n[1] * g.n[2] * nact;
  const long long groups = (items + H::EPB - 1) / H::EPB;
  auto kern = k_schwarz_patch<T, N1, H::EPB>;
  if (H::SMEM > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)H::SMEM);
    if (e != cudaSuccess) return e;
  }
  // persistent grid: the blocks that shared memory and the thread limit let an SM hold
  constexpr int BY_SMEM = (int)(227 * 1024 / (H::SMEM + 1024)), BY_THREADS = 2048 / H::THREADS;
  const long long cap = 152LL * (BY_SMEM < BY_THREADS ? BY_SMEM : BY_THREADS);
  count_launch();
  kern<<<(unsigned)(groups < cap ? groups : cap), H::THREADS, H::SMEM, s>>>(g, (const unsigned char*)tb.blob, r, zp, act,
                                                                         nact);
  return cudaGetLastError();
}

// Few patches (the warps of k_schwarz_patch_small at most 24 per SM, at p = 8 8): one
// patch per block and two lanes per line; otherwise several per block, so that warps
// are full.
// Measured around the line (us, small / several): FP64 p = 4 256 patches 13.3 / 22.4,
// 1024 41.3 / 41.5, 4096 152 / 119; p = 6 512 54 / 68, 1024 103 / 100; p = 8 64 28.1 /
// 29.7, 256 53.7 / 50.1; p = 1 512 4.2 / 6.6, 4096 14.6 / 14.1; FP32 p = 6 512 6.2 /
// 7.9, 1024 9.2 / 8.0; p = 4 256 3.2 / 4.4, 1024 5.6 / 5.0; p = 2 1024 3.5 / 5.7.
// In FP64 large blocks leave the SM that gets one more than the others alone for long: at
// p = 7 (three patches, 320 threads) the kernel whose busiest SM has less to do, at p = 6
// (three patches, 256 threads) blocks of one patch up to ten per SM, but not where blocks
// of three are two for every SM. us, one patch and two lanes per line / three patches: p =
// 7 540 68 / 99, 1050 118 / 147, 2400 256 / 275; one patch / three: p = 6 686 59 / 67, 875
// 91 / 79, 1296 112 / 123, 1536 115 / 119, 3430 257 / 240.
template <typename T, int N1>
static cudaError_t patch_n1(const SwTables& tb, const T* r, T* zp, const int* act, int nact, cudaStream_t s) {
  const long long items = (long long)tb.geom.n[0] * tb.geom.n[1] * tb.geom.n[2] * nact;
  bool small = items * (SwSmall<T, N1>::THREADS / 32) <= 152 * (N1 < 9 ? 24 : 8);
  if constexpr (sizeof(T) == 8 && N1 == 8) {
    // the busier SM's warps, of which the small kernel's do half the work each
    using H = SwShape<T, N1>;
    auto busiest = [&](long long blocks, int threads) { return (blocks + 151) / 152 * threads; };
    small |= items <= 152 * 24 && busiest(items, SwSmall<T, N1>::THREADS) / 2 <
                                      busiest((items + H::EPB - 1) / H::EPB, H::THREADS);
  }
  if constexpr (sizeof(T) == 8 && N1 == 7) {
    const bool even = items > 152 * 5 && items <= 152 * 6;  // two blocks of three on every SM
    if (!small && items <= 152 * 10 && !even) return patch_fill<T, N1, SwShape<T, N1, 1>>(tb, r, zp, act, nact, s);
  }
  if (!small) return patch_fill<T, N1>(tb, r, zp, act, nact, s);
  using S = SwSmall<T, N1>;
  static_assert(S::SMEM <= 48 * 1024, "one patch and its tables");
  count_launch();
  k_schwarz_patch_small<T, N1><<<(unsigned)items, S::THREADS, S::SMEM, s>>>(tb.geom, (const unsigned char*)tb.blob, r,
                                                                           zp, act);
  return cudaGetLastError();
}

// Gather block shape: GE elements of NPE nodes per block (several small
// elements per block on the coarse levels), one thread per node.
#ifndef DG_GATHER_THREADS
#define DG_GATHER_THREADS 256  // thread budget of a gather block (at least one element)
#endif
template <int N1>
struct GatherCfg {
  static constexpr int NPE = N1 * N1 * N1;
  static constexpr int GE = DG_GATHER_THREADS / NPE < 1 ? 1 : DG_GATHER_THREADS / NPE;
  static constexpr int THREADS = GE * NPE;
};

// mode 0: z = M r; 1: d = c1 M r, x = d; 2: d = c1 M r, x += d; 3: d = c1 d + c2 M r, x += d
// (d is passed in z). GE elements per block and iteration (grid-stride), one thread per node,
// GS sources per thread (the node's position, neighbour tests and offsets shared by them).
// All loads of the group are issued before the first sum: the contributions of one
// source at a time left too few bytes in flight. At most 4 in FP32, 2 in FP64
// (registers; 4 is 1 % slower); gather_n1 chooses.
// Measured (GB300, FP32, d and x not touched): 16^3, p = 7, 42 sources 0.516 ->
// 0.262 ms for 1.04 GB, 8^3, p = 6, 56 sources 66 -> 36 us.
template <typename T, int N1, int MODE, int GS>
__global__ void __launch_bounds__(GatherCfg<N1>::THREADS)
    k_schwarz_gather(const LevelOp* __restrict__ op, const T* __restrict__ zp, T* __restrict__ z, T* __restrict__ x,
                     T c1, T c2, const int* __restrict__ act, int nact) {
  constexpr int MP = N1 + 2, MP2 = MP * MP, MP3 = MP2 * MP, NPE = N1 * N1 * N1, GE = GatherCfg<N1>::GE;
  const int nx = op->n[0], ny = op->n[1], nz = op->n[2];
  const int E = op->E;
  const long long Nq = op->Nq;
  // this block's sources (GS consecutive entries of the active list)
  const int k0 = blockIdx.y * GS;
  const int ns = min(GS, nact - k0);
  long long zoff[GS], foff[GS];  // of each source in the patch buffer and in the fields
#pragma unroll
  for (int j = 0; j < GS; ++j) {
    const long long rhs = act[k0 + min(j, ns - 1)];
    zoff[j] = rhs * E * MP3;
    foff[j] = rhs * Nq;
  }
  const int slot = threadIdx.x / NPE, loc = threadIdx.x % NPE;
  const int a = loc % N1, bb = (loc / N1) % N1, c = loc / (N1 * N1);
  // element position, advanced by the grid stride without runtime divisions
  const int g = gridDim.x * GE, sx = g % nx, sy = (g / nx) % ny, sz = g / (nx * ny);
  const int e0 = blockIdx.x * GE + slot;
  int ex = e0 % nx, ey = (e0 / nx) % ny, ez = e0 / (nx * ny);
  for (int e = e0; e < E; e += g) {
    const int ix = a + (ex > 0), iy = bb + (ey > 0), iz = c + (ez > 0);
    // neighbour along each axis whose patch also covers this node, if any
    int dx = 0, jx = 0, dy = 0, jy = 0, dz = 0, jz = 0;
    if (a == 0 && ex > 0) {
      dx = -1;
      jx = N1 + (ex > 1);
    } else if (a == N1 - 1 && ex < nx - 1) {
      dx = 1;
    }
    if (bb == 0 && ey > 0) {
      dy = -nx;
      jy = N1 + (ey > 1);
    } else if (bb == N1 - 1 && ey < ny - 1) {
      dy = nx;
    }
    if (c == 0 && ez > 0) {
      dz = -nx * ny;
      jz = N1 + (ez > 1);
    } else if (c == N1 - 1 && ez < nz - 1) {
      dz = nx * ny;
    }
    // offsets (values, within one source's patch buffer) of every contribution;
    // a source's patch buffer holds E MP^3 < 2^31 values
    const int o0 = e * MP3 + ix + MP * iy + MP2 * iz;
    const int ox = (e + dx) * MP3 + jx + MP * iy + MP2 * iz;
    const int oy = (e + dy) * MP3 + ix + MP * jy + MP2 * iz;
    const int oz = (e + dz) * MP3 + ix + MP * iy + MP2 * jz;
    const int oxy = (e + dx + dy) * MP3 + jx + MP * jy + MP2 * iz;
    const int oxz = (e + dx + dz) * MP3 + jx + MP * iy + MP2 * jz;
    const int oyz = (e + dy + dz) * MP3 + ix + MP * jy + MP2 * jz;
    const int oxyz = (e + dx + dy + dz) * MP3 + jx + MP * jy + MP2 * jz;
    const int gi = e * NPE + loc;
    // every load of the group is issued before the first sum, contributions in a
    // fixed order; sources past the end repeat the last one and are not stored
    T acc[GS], v[7][GS], dv[GS], xv[GS];
#pragma unroll
    for (int j = 0; j < GS; ++j) {
      const T* zs = zp + zoff[j];
      acc[j] = zs[o0];
      v[0][j] = dx ? zs[ox] : (T)0;
      v[1][j] = dy ? zs[oy] : (T)0;
      v[2][j] = dz ? zs[oz] : (T)0;
      v[3][j] = dx && dy ? zs[oxy] : (T)0;
      v[4][j] = dx && dz ? zs[oxz] : (T)0;
      v[5][j] = dy && dz ? zs[oyz] : (T)0;
      v[6][j] = dx && dy && dz ? zs[oxyz] : (T)0;
      if (MODE == 3) dv[j] = z[foff[j] + gi];
      if (MODE >= 2) xv[j] = x[foff[j] + gi];
    }
#pragma unroll
    for (int c = 0; c < 7; ++c)
#pragma unroll
      for (int j = 0; j < GS; ++j) acc[j] += v[c][j];
#pragma unroll
    for (int j = 0; j < GS; ++j) {
      if (j >= ns) break;
      T* zg = z + foff[j] + gi;
      T* xg = x + foff[j] + gi;
      if (MODE == 0) {
        *zg = acc[j];
      } else if (MODE == 1) {
        const T w = c1 * acc[j];
        *zg = w;
        *xg = w;
      } else if (MODE == 2) {
        const T w = c1 * acc[j];
        *zg = w;
        *xg = xv[j] + w;
      } else {
        const T w = c1 * dv[j] + c2 * acc[j];
        *zg = w;
        *xg = xv[j] + w;
      }
    }
    ex += sx;
    int carry = ex >= nx;
    ex -= carry ? nx : 0;
    ey += sy + carry;
    carry = ey >= ny;
    ey -= carry ? ny : 0;
    ez += sz + carry;
  }
}

// z = M r from the patch solutions (the second kernel of the smoother)
template <typename T, int N1, int GS>
static cudaError_t gather_gs(const LevelOp& hop, const LevelOp* dop, const T* zp, T* z, T* x, int mode, double c1,
                             double c2, const int* act, int nact, cudaStream_t s) {
  constexpr int GT = GatherCfg<N1>::THREADS;
  // the gather indexes one source's patch buffer with 32-bit offsets
  if ((long long)hop.E * (N1 + 2) * (N1 + 2) * (N1 + 2) >= (1LL << 31)) return cudaErrorInvalidValue;
  long long gx = (hop.E + GatherCfg<N1>::GE - 1) / GatherCfg<N1>::GE;
  const long long ngroups = (nact + GS - 1) / GS;
  const long long cap = 152LL * GATHER_WAVE / ngroups + 1;
  if (gx > cap) gx = cap;
  const dim3 grid((unsigned)gx, (unsigned)ngroups);
  count_launch();
  switch (mode) {
    case 0: k_schwarz_gather<T, N1, 0, GS><<<grid, GT, 0, s>>>(dop, zp, z, x, (T)c1, (T)c2, act, nact); break;
    case 1: k_schwarz_gather<T, N1, 1, GS><<<grid, GT, 0, s>>>(dop, zp, z, x, (T)c1, (T)c2, act, nact); break;
    case 2: k_schwarz_gather<T, N1, 2, GS><<<grid, GT, 0, s>>>(dop, zp, z, x, (T)c1, (T)c2, act, nact); break;
    default: k_schwarz_gather<T, N1, 3, GS><<<grid, GT, 0, s>>>(dop, zp, z, x, (T)c1, (T)c2, act, nact); break;
  }
  return cudaGetLastError();
}

// As few groups as the largest size allows, all of about one size: a thread of a group
// with fewer sources than its size repeats the loads of the last one. Smoother, FP32, us,
// groups of 1 / 2 / 3 / 4: 16^3, p = 7, 1 source 71 / 77 / 77 / 80, 2 sources 106 / 101 /
// 102 / 105, 5 sources 191 / 185 / 173 / 180; p = 6, 1 source 29.7 / 31.6 / 33.5 / 36.9, 3
// sources 67 / 64 / 57 / 61, 9 sources 191 / 174 / 162 / 171.
template <typename T, int N1>
static cudaError_t gather_n1(const LevelOp& hop, const LevelOp* dop, const T* zp, T* z, T* x, int mode, double c1,
                             double c2, const int* act, int nact, cudaStream_t s) {
  constexpr int MAXGS = sizeof(T) == 4 ? 4 : 2;
  const int groups = (nact + MAXGS - 1) / MAXGS, gs = (nact + groups - 1) / groups;
  if constexpr (MAXGS == 4) {
    if (gs == 4) return gather_gs<T, N1, 4>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s);
    if (gs == 3) return gather_gs<T, N1, 3>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s);
  }
  return gs == 2 ? gather_gs<T, N1, 2>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s)
                 : gather_gs<T, N1, 1>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s);
}

template <typename T>
cudaError_t launch_schwarz_patch(const LevelOp& hop, const LevelOp* dop, const SwTables& tabs, const T* r, T* zp,
                                 const int* act, int nact, cudaStream_t s, const SwTcPlan* tc) {
  if (nact == 0) return cudaSuccess;
  if (sizeof(T) == 4 && tc && tc->blob)
    return launch_schwarz_patch_tc(hop, dop, *tc, (const float*)r, (float*)zp, act, nact, s);
  switch (hop.n1) {
    case 2: return patch_n1<T, 2>(tabs, r, zp, act, nact, s);
    case 3: return patch_n1<T, 3>(tabs, r, zp, act, nact, s);
    case 4: return patch_n1<T, 4>(tabs, r, zp, act, nact, s);
    case 5: return patch_n1<T, 5>(tabs, r, zp, act, nact, s);
    case 6: return patch_n1<T, 6>(tabs, r, zp, act, nact, s);
    case 7: return patch_n1<T, 7>(tabs, r, zp, act, nact, s);
    case 8: return patch_n1<T, 8>(tabs, r, zp, act, nact, s);
    case 9: return patch_n1<T, 9>(tabs, r, zp, act, nact, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t launch_schwarz(const LevelOp& hop, const LevelOp* dop, const SwTables& tabs, const T* r, T* zp, T* z,
                           T* x, int mode, double c1, double c2, const int* act, int nact, cudaStream_t s,
                           const SwTcPlan* tc) {
  if (nact == 0) return cudaSuccess;
  const cudaError_t e = launch_schwarz_patch<T>(hop, dop, tabs, r, zp, act, nact, s, tc);
  if (e != cudaSuccess) return e;
  switch (hop.n1) {
    case 2: return gather_n1<T, 2>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s);
    case 3: return gather_n1<T, 3>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s);
    case 4: return gather_n1<T, 4>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s);
    case 5: return gather_n1<T, 5>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s);
    case 6: return gather_n1<T, 6>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s);
    case 7: return gather_n1<T, 7>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s);
    case 8: return gather_n1<T, 8>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s);
    case 9: return gather_n1<T, 9>(hop, dop, zp, z, x, mode, c1, c2, act, nact, s);
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_schwarz_patch<double>(const LevelOp&, const LevelOp*, const SwTables&, const double*,
                                                  double*, const int*, int, cudaStream_t, const SwTcPlan*);
template cudaError_t launch_schwarz_patch<float>(const LevelOp&, const LevelOp*, const SwTables&, const float*, float*,
                                                 const int*, int, cudaStream_t, const SwTcPlan*);
template cudaError_t launch_schwarz<double>(const LevelOp&, const LevelOp*, const SwTables&, const double*, double*,
                                            double*, double*, int, double, double, const int*, int, cudaStream_t,
                                            const SwTcPlan*);
template cudaError_t launch_schwarz<float>(const LevelOp&, const LevelOp*, const SwTables&, const float*, float*,
                                           float*, float*, int, double, double, const int*, int, cudaStream_t,
                                           const SwTcPlan*);

}  // namespace dg
