// Adaptive octree auxiliary mesh, host side (Sec. 6.2): the uniform root grid
// refined where the density's quadrature indicator exceeds a threshold, kept
// 2:1 balanced across faces, and the face connectivity the operator on it
// needs (same-size, larger or smaller neighbours, boundary).
//
// Readings: isotropic 8-child splits; indicator Q = |I_K(rho) - sum over the
// children of I_C(rho)| with the degree-p tensor Gauss-Legendre rule of the
// leaf and of each child; a leaf is split while Q > delta and its level is
// below the maximum level.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <map>
#include <set>
#include <vector>

#include "dg_ctx.h"
#include "dg_line.h"
#include "dg_octree.h"
#include "dg_setup.h"

namespace dg {

using Leaf = std::array<int, 4>;  // level, ix, iy, iz

struct Octree {
  double lo[3], H[3];
  int n[3], p;
  std::set<Leaf> leaves;

  double h(int level, int d) const { return H[d] / double(1 << level); }
  long long extent(int level, int d) const { return (long long)n[d] << level; }

  void refine(const std::vector<Leaf>& ks) {
    for (const Leaf& k : ks) {
      if (!leaves.erase(k)) continue;
      for (int c = 0; c < 8; ++c)
        leaves.insert({k[0] + 1, 2 * k[1] + (c & 1), 2 * k[2] + ((c >> 1) & 1), 2 * k[3] + (c >> 2)});
    }
  }

  // leaf containing the cell (level, x, y, z) unless finer leaves cover it
  bool covering(int level, int x, int y, int z, Leaf& out) const {
    for (int lv = level; lv >= 0; --lv) {
      const int s = level - lv;
      const Leaf k{lv, x >> s, y >> s, z >> s};
      if (leaves.count(k)) {
        out = k;
        return true;
      }
    }
    return false;
  }

  // same-level cell across face (d, side); false at the domain boundary
  bool neighbour(const Leaf& k, int d, int side, Leaf& out) const {
    out = k;
    out[1 + d] += side;
    return out[1 + d] >= 0 && out[1 + d] < extent(k[0], d);
  }

  void balance() {
    for (;;) {
      std::set<Leaf> split;
      for (const Leaf& k : leaves)
        for (int d = 0; d < 3; ++d)
          for (int side = -1; side <= 1; side += 2) {
            Leaf nb, L;
            if (!neighbour(k, d, side, nb)) continue;
            if (covering(nb[0], nb[1], nb[2], nb[3], L) && L[0] < k[0] - 1) split.insert(L);
          }
      if (split.empty()) return;
      refine(std::vector<Leaf>(split.begin(), split.end()));
    }
  }

  // element order: root cell (x fastest), then level, z, y, x
  std::vector<Leaf> ordered() const {
    std::vector<Leaf> v(leaves.begin(), leaves.end());
    auto key = [&](const Leaf& k) {
      const int lv = k[0];
      const long long r = (k[1] >> lv) + (long long)n[0] * ((k[2] >> lv) + (long long)n[1] * (k[3] >> lv));
      return std::array<long long, 5>{r, lv, k[3], k[2], k[1]};
    };
    std::sort(v.begin(), v.end(), [&](const Leaf& a, const Leaf& b) { return key(a) < key(b); });
    return v;
  }
};

// integral of rho over the box [o, o + h] by the degree-p tensor GL rule
static double gl_integral(const double* o, const double* h, int n1, const double* xi, const double* w,
                          dg_density_fn rho, void* user, std::vector<double>& pts, std::vector<double>& val) {
  const int np = n1 * n1 * n1;
  pts.resize(3 * (size_t)np);
  val.resize(np);
  for (int c = 0; c < n1; ++c)
    for (int b = 0; b < n1; ++b)
      for (int a = 0; a < n1; ++a) {
        const int q = a + n1 * (b + n1 * c);
        pts[3 * q + 0] = o[0] + (xi[a] + 1.0) * h[0] / 2.0;
        pts[3 * q + 1] = o[1] + (xi[b] + 1.0) * h[1] / 2.0;
        pts[3 * q + 2] = o[2] + (xi[c] + 1.0) * h[2] / 2.0;
      }
  rho(pts.data(), np, val.data(), user);
  double s = 0.0;
  for (int c = 0; c < n1; ++c)
    for (int b = 0; b < n1; ++b)
      for (int a = 0; a < n1; ++a) s += w[a] * w[b] * w[c] * val[a + n1 * (b + n1 * c)];
  return s * h[0] * h[1] * h[2] / 8.0;
}

// Face connectivity of a leaf set (see dg_octree_faces); false for a bad mesh
// or leaf set.
bool octree_faces(const dg_mesh_desc* root, const int32_t* leaves, int32_t n_leaves, int32_t* kind,
                         int32_t* nb, int32_t* pos) {
  if (!root || !leaves || n_leaves < 1 || !kind || !nb || !pos) return false;
  Octree t;
  for (int d = 0; d < 3; ++d) {
    if (root->n[d] < 1 || !(root->hi[d] > root->lo[d])) return false;
    t.lo[d] = root->lo[d];
    t.n[d] = root->n[d];
    t.H[d] = (root->hi[d] - root->lo[d]) / root->n[d];
  }
  t.p = root->p;
  std::map<Leaf, int> index;
  for (int e = 0; e < n_leaves; ++e) {
    const Leaf k{leaves[4 * e], leaves[4 * e + 1], leaves[4 * e + 2], leaves[4 * e + 3]};
    if (k[0] < 0 || k[0] > 20) return false;
    for (int d = 0; d < 3; ++d)
      if (k[1 + d] < 0 || k[1 + d] >= t.extent(k[0], d)) return false;
    if (!index.emplace(k, e).second) return false;
    t.leaves.insert(k);
  }
  // a partition: no leaf may lie inside another leaf of the set
  for (int e = 0; e < n_leaves; ++e) {
    const Leaf k{leaves[4 * e], leaves[4 * e + 1], leaves[4 * e + 2], leaves[4 * e + 3]};
    for (int lv = k[0] - 1; lv >= 0; --lv) {
      const int sh = k[0] - lv;
      if (index.count(Leaf{lv, k[1] >> sh, k[2] >> sh, k[3] >> sh})) return false;
    }
  }
  for (int e = 0; e < n_leaves; ++e) {
    const Leaf k{leaves[4 * e], leaves[4 * e + 1], leaves[4 * e + 2], leaves[4 * e + 3]};
    for (int d = 0; d < 3; ++d)
      for (int sd = 0; sd < 2; ++sd) {
        const int f = 2 * d + sd, side = sd ? 1 : -1;
        const long long o = 6LL * e + f;
        for (int j = 0; j < 4; ++j) nb[4 * o + j] = -1;
        pos[o] = -1;
        Leaf c, L;
        if (!t.neighbour(k, d, side, c)) {
          kind[o] = 0;  // boundary
          continue;
        }
        const int t0 = d == 0 ? 1 : 0, t1 = d == 2 ? 1 : 2;
        if (t.covering(c[0], c[1], c[2], c[3], L)) {
          if (L[0] == k[0]) {
            kind[o] = 1;
          } else if (L[0] == k[0] - 1) {
            kind[o] = 2;  // this face is a quarter of L's face: its two tangential bits
            pos[o] = (k[1 + t0] & 1) | ((k[1 + t1] & 1) << 1);
          } else {
            return false;  // not 2:1 balanced
          }
          nb[4 * o] = index.at(L);
          continue;
        }
        // four smaller neighbours: the level + 1 cells touching this face
        kind[o] = 3;
        for (int j = 0; j < 4; ++j) {
          Leaf sl{k[0] + 1, 2 * k[1], 2 * k[2], 2 * k[3]};
          sl[1 + d] = sd ? 2 * k[1 + d] + 2 : 2 * k[1 + d] - 1;
          sl[1 + t0] += j & 1;
          sl[1 + t1] += j >> 1;
          auto it = index.find(sl);
          if (it == index.end()) return false;  // not 2:1 balanced or not a leaf set
          nb[4 * o + j] = it->second;
        }
      }
  }
  return true;
}


// ---------------------------------------------------------------------------
// SIPDG operator on the octree leaves (Sec. 3.4 eq. sip_bilinear with the
// Nitsche boundary terms of Sec. 6.3), matrix-free. Volume term: the element's
// Kronecker sum (GL-collocated mass, exact 1-D stiffness). Face terms: traces
// and normal derivatives of this leaf and of its neighbour(s) at Gauss points of
// the smaller face (a hanging face is integrated on each of its four quarters),
// fluxes
//   v-trace:      -{d_n u} + sigma [u]     (boundary: -d_n u + sigma u)
//   d_n v:        -1/2 [u]                 (boundary: -u)
// with [u] = u_K - u_L along K's outward normal, sigma = (p+1)^2/(eps h) of
// the smaller leaf, and the test-side contraction back onto the leaf's nodes.
//
// The Gauss points of a face are the leaf's own face nodes, so between leaves of
// one size (and at the boundary) no interpolation is needed: the flux at a face
// node takes the two lines that meet there, and a leaf is worked like an element
// of the uniform operator (k_oct_apply: a thread owns a line along each
// direction in turn, folded into even and odd halves, tables in the constant
// bank; lengths enter as one factor per axis). Only hanging faces interpolate:
// k_oct_hang takes each of them once per source, for both sides: the larger
// leaf's traces to its four quarters (two sum-factorised steps), the fluxes
// there, and their projection back onto the larger face; k_oct_apply reads the
// result in place of a neighbour's traces.
//
// Measured (GB300, density-refined chain octree, 715 leaves, p = 6, 8 fields; one
// block per leaf with every face interpolated to Gauss points and back before):
// FP32 396 -> 20 us (5 us of it the hanging faces), FP64 974 -> 255 us; the V-cycle of
// the FP64 solve, three degrees of this operator and the leaf-block inverse, 9.8 ->
// 4.2 ms; a mixed solve of 8 sources to 1e-12 238 -> 84 ms by this alone (42 ms with
// the fused leaf-block inverse and the 16-row boundary GEMM).
// ---------------------------------------------------------------------------

// tables of k_oct_apply: 1-D stiffness and end traces, folded (see dg_apply.cu)
template <typename V, int N1>
struct OctLine {
  static constexpr int HO = N1 / 2, HE = N1 - HO;
  V Se[HE][HE], So[HO][HO];
  V te[HE], de[HE], to[HO], dO[HO];  // value and derivative at the left end
  V tl[N1], dl[N1];                  // the same unfolded
  V ww[N1 * N1];                     // w_i w_j by line
  V g0;                              // (p+1)^2 / (2 eps): sigma h / 2 (times 1/h for penalty form 1)
  long long Nq, items;
  int E, k0, nslots;                 // leaves, first source of this launch, hanging slots per source
};

template <typename V, int N1, bool FILL>
struct OctShape {
  static constexpr int LINES = N1 * N1;
  static constexpr int BPB = FILL ? best_bpb(LINES, sizeof(V) == 4 ? 128 : 64) : 1;
  static constexpr int THREADS = (BPB * LINES + 31) / 32 * 32;
  static constexpr size_t SMEM = sizeof(V) * 2 * (size_t)BPB * LineLayout<N1>::ES;
  static constexpr int WANT = sizeof(V) == 4 ? 768 : 512;
  static constexpr int MINB = WANT / THREADS < 1 ? 1 : WANT / THREADS > 32 ? 32 : WANT / THREADS;
};

// traces beyond the ends of a line: of the neighbour leaf (face code fc >= 0), or
// those that the boundary stands for (fc = -1; the own line read reversed looks
// like a neighbour's), nothing for a hanging face (fc < -1)
template <typename V, int N1, int D>
__device__ __forceinline__ void oct_outer(const OctLine<V, N1>& tab, const V* __restrict__ us, int e, int l, int fl,
                                          int fr, V gam, bool vec, V* ov, V* od) {
  constexpr int NF = N1 * N1, NPE = NF * N1;
  constexpr int SD = D == 0 ? 1 : (D == 1 ? N1 : NF);
  const int l1 = l % N1, l2 = l / N1;
  const int base = D == 0 ? N1 * l : (D == 1 ? l1 + NF * l2 : l);
  V v[N1];
  ov[0] = od[0] = ov[1] = od[1] = (V)0;
  if (fl >= -1) {
    load_line<V, N1, SD>(us + (long long)(fl < 0 ? e : fl) * NPE + base, fl < 0, vec, v);
    end_trace<V, N1, true>(tab.tl, tab.dl, v, ov[0], od[0]);
    if (fl < 0) {
      od[0] = mad((V)-2 * gam, ov[0], -od[0]);
      ov[0] = -ov[0];
    }
  }
  if (fr >= -1) {
    load_line<V, N1, SD>(us + (long long)(fr < 0 ? e : fr) * NPE + base, fr < 0, vec, v);
    end_trace<V, N1, false>(tab.tl, tab.dl, v, ov[1], od[1]);
    if (fr < 0) {
      od[1] = mad((V)2 * gam, ov[1], -od[1]);
      ov[1] = -ov[1];
    }
  }
}

// S v plus the face terms of a line; hL/hR: hanging, then ov/od hold the
// projected fluxes instead of a neighbour's traces
template <typename V, int N1>
__device__ __forceinline__ void oct_line(const OctLine<V, N1>& tab, V* v, const V* ov, const V* od, bool hL, bool hR,
                                         V gam) {
  constexpr int HO = N1 / 2, HE = N1 - HO;
  V e[HE], o[HO];
#pragma unroll
  for (int i = 0; i < HO; ++i) {
    e[i] = v[i] + v[N1 - 1 - i];
    o[i] = v[i] - v[N1 - 1 - i];
  }
  if (HE > HO) e[HE - 1] = v[HO];
  V a = mul(tab.te[0], e[0]), b = mul(tab.to[0], o[0]), c = mul(tab.de[0], e[0]), d = mul(tab.dO[0], o[0]);
#pragma unroll
  for (int i = 1; i < HE; ++i) {
    a = mad(tab.te[i], e[i], a);
    c = mad(tab.de[i], e[i], c);
  }
#pragma unroll
  for (int i = 1; i < HO; ++i) {
    b = mad(tab.to[i], o[i], b);
    d = mad(tab.dO[i], o[i], d);
  }
  const V h = (V)0.5;
  const V jL = (a + b) - ov[0], jR = (a - b) - ov[1];  // jumps
  const V gL1 = hL ? ov[0] : mad(gam, jL, mul(h, (c + d) + od[0])), gL2 = hL ? od[0] : mul(-h, jL);
  const V gR1 = hR ? ov[1] : mad(gam, jR, mul(-h, (d - c) + od[1])), gR2 = hR ? od[1] : mul(-h, jR);
  const V p1 = gL1 + gR1, m1 = gL1 - gR1, p2 = gL2 + gR2, m2 = gL2 - gR2;
  V O[HO];
#pragma unroll
  for (int k = 0; k < HO; ++k) {
    V acc = mad(-tab.dO[k], m2, mul(tab.to[k], m1));
#pragma unroll
    for (int i = 0; i < HO; ++i) acc = mad(tab.So[k][i], o[i], acc);
    O[k] = acc;
  }
#pragma unroll
  for (int k = 0; k < HE; ++k) {
    V acc = mad(-tab.de[k], p2, mul(tab.te[k], p1));
#pragma unroll
    for (int i = 0; i < HE; ++i) acc = mad(tab.Se[k][i], e[i], acc);
    if (k < HO) {
      v[k] = acc + O[k];
      v[N1 - 1 - k] = acc - O[k];
    } else {
      v[k] = acc;
    }
  }
}

// out = A u (rin null) or rin - A u, one slot per leaf and source. fac [E][6]: h_t0 h_t1 / (2 h_d) per
// axis, then 1 (penalty form 0) or 1 / h_d; hslot [E][6]: hanging slot of a
// face, -1 for the others; gbuf [source - k0][slot][2][N1^2]: k_oct_hang's
// projected fluxes.
template <typename V, int N1, bool FILL>
__global__ void __launch_bounds__(OctShape<V, N1, FILL>::THREADS, OctShape<V, N1, FILL>::MINB)
    k_oct_apply(const __grid_constant__ OctLine<V, N1> tab, const double* __restrict__ fac,
                const int* __restrict__ kind, const int* __restrict__ nbr, const int* __restrict__ hslot,
                const V* __restrict__ gbuf, const V* __restrict__ u, V* __restrict__ out,
                const V* __restrict__ rin, const int* __restrict__ act, int vec_i) {
  using H = OctShape<V, N1, FILL>;
  using Y = LineLayout<N1>;
  constexpr int NF = N1 * N1, NPE = NF * N1, BPB = H::BPB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* su = reinterpret_cast<V*>(smem_raw);
  V* sacc = su + BPB * Y::ES;
  __shared__ int sleaf[BPB], ssrc[BPB], skk[BPB], sface[BPB][6];
  __shared__ V sfac[BPB][6];
  const int tid = threadIdx.x;
  if (tid < BPB) {
    const long long it = (long long)blockIdx.x * BPB + tid;
    const bool in = it < tab.items;
    const int kk = in ? (int)(it / tab.E) : 0, e = in ? (int)(it - (long long)kk * tab.E) : -1;
    sleaf[tid] = e;
    skk[tid] = kk;
    ssrc[tid] = act ? act[tab.k0 + kk] : tab.k0 + kk;
  }
  __syncthreads();
  for (int t = tid; t < BPB * 6; t += H::THREADS) {
    const int sl = t / 6, f = t - 6 * sl, e = sleaf[sl];
    if (e < 0) continue;
    const long long o = 6LL * e + f;
    const int kd = kind[o];
    sface[sl][f] = kd == 0 ? -1 : kd == 1 ? nbr[4 * o] : -2 - hslot[o];
    sfac[sl][f] = (V)fac[o] * (f >= 3 ? tab.g0 : (V)1);
  }
  __syncthreads();
  const int slot = tid / NF, l = tid - slot * NF, l1 = l % N1, l2 = l / N1;
  const bool on = slot < BPB && sleaf[slot < BPB ? slot : 0] >= 0;
  const int sl = on ? slot : 0, e = on ? sleaf[sl] : 0;
  const bool vec = vec_i != 0;
  const V* us = u + (long long)ssrc[sl] * tab.Nq;
  const long long g0 = (long long)ssrc[sl] * tab.Nq + (long long)e * NPE;
  const int* fc = sface[sl];
  const int sb = sl * Y::ES, zat = sb + l1 + Y::PB * l2;
  V v[N1], ov[3][2], od[3][2], gam[3];
  if (on) {
#pragma unroll
    for (int i = 0; i < N1; ++i) v[i] = __ldg(us + (long long)e * NPE + l + NF * i);
#pragma unroll
    for (int i = 0; i < N1; ++i) su[zat + Y::PZ * i] = v[i];
#pragma unroll
    for (int d = 0; d < 3; ++d) gam[d] = sfac[sl][3 + d];
    oct_outer<V, N1, 0>(tab, us, e, l, fc[0], fc[1], gam[0], vec, ov[0], od[0]);
    oct_outer<V, N1, 1>(tab, us, e, l, fc[2], fc[3], gam[1], vec, ov[1], od[1]);
    oct_outer<V, N1, 2>(tab, us, e, l, fc[4], fc[5], gam[2], vec, ov[2], od[2]);
#pragma unroll
    for (int f = 0; f < 6; ++f)
      if (fc[f] < -1) {
        const V* g = gbuf + (((long long)skk[sl] * tab.nslots + (-2 - fc[f])) * 2) * NF + l;
        ov[f >> 1][f & 1] = g[0];
        od[f >> 1][f & 1] = g[NF];
      }
  }
  __syncthreads();
  if (on) {
    const int at = sb + Y::PB * l1 + Y::PZ * l2;
#pragma unroll
    for (int i = 0; i < N1; ++i) v[i] = su[at + i];
    oct_line<V, N1>(tab, v, ov[0], od[0], fc[0] < -1, fc[1] < -1, gam[0]);
    const V sc = mul(sfac[sl][0], tab.ww[l]);
#pragma unroll
    for (int i = 0; i < N1; ++i) sacc[at + i] = mul(sc, v[i]);
  }
  __syncthreads();
  if (on) {
    const int at = sb + l1 + Y::PZ * l2;
#pragma unroll
    for (int i = 0; i < N1; ++i) v[i] = su[at + Y::PB * i];
    oct_line<V, N1>(tab, v, ov[1], od[1], fc[2] < -1, fc[3] < -1, gam[1]);
    const V sc = mul(sfac[sl][1], tab.ww[l]);
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      V* p = sacc + at + Y::PB * i;
      *p = mad(sc, v[i], *p);
    }
  }
  __syncthreads();
  if (on) {
#pragma unroll
    for (int i = 0; i < N1; ++i) v[i] = su[zat + Y::PZ * i];
    oct_line<V, N1>(tab, v, ov[2], od[2], fc[4] < -1, fc[5] < -1, gam[2]);
    const V sc = mul(sfac[sl][2], tab.ww[l]);
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      const V Au = mad(sc, v[i], sacc[zat + Y::PZ * i]);
      out[g0 + l + NF * i] = rin ? rin[g0 + l + NF * i] - Au : Au;
    }
  }
}

// tables of k_oct_hang
template <typename V, int N1>
struct OctHang {
  V Lh[2][N1 * N1];  // [c][i][a]: the larger leaf's basis a at point i of its half c
  V tl[N1], dl[N1], w[N1];
  V g0;
  long long Nq;
  int k0, nI;
};

// Fluxes of a hanging face in units of 2 / h of the side that they are for, with
// the side's weights w_i w_j and lengths divided out: record [leaf of the larger
// side, its face, the four smaller leaves]; slot 5 i of gbuf is the larger side's,
// 5 i + 1 + j the j-th smaller one's. 4 N1^2 threads a face: one per quarter and
// point.
template <typename V, int N1>
struct HangShape {
  static constexpr int T4 = 4 * N1 * N1;
  static constexpr int HPB = T4 >= 96 ? 1 : 128 / T4;
  static constexpr int THREADS = (HPB * T4 + 31) / 32 * 32;
};
template <typename V, int N1>
__global__ void __launch_bounds__(HangShape<V, N1>::THREADS)
    k_oct_hang(const __grid_constant__ OctHang<V, N1> tab, const int* __restrict__ rec, const double* __restrict__ fac,
               const V* __restrict__ u, V* __restrict__ gbuf, const int* __restrict__ act) {
  using H = HangShape<V, N1>;
  constexpr int NF = N1 * N1, NPE = NF * N1, T4 = H::T4, HPB = H::HPB;
  __shared__ V sL[2][NF], sw[N1];
  __shared__ V sX[HPB][2][NF];      // larger side: value, derivative at its face nodes
  __shared__ V sR[HPB][2][2][NF];   // [quantity][half along t0]
  __shared__ V sF[HPB][2][4][NF];   // weighted fluxes per quarter
  const int tid = threadIdx.x;
  for (int i = tid; i < 2 * NF; i += H::THREADS) sL[i / NF][i % NF] = tab.Lh[i / NF][i % NF];
  for (int i = tid; i < N1; i += H::THREADS) sw[i] = tab.w[i];
  const int hs = tid / T4, t = tid - hs * T4;
  const int ifc = blockIdx.x * HPB + hs;
  const bool on = hs < HPB && ifc < tab.nI;
  const int src = act ? act[tab.k0 + blockIdx.y] : tab.k0 + (int)blockIdx.y;
  const V* us = u + (long long)src * tab.Nq;
  const int* rc = rec + 6LL * (on ? ifc : 0);
  const int big = rc[0], f = rc[1], d = f >> 1, r = f & 1;
  const int st[3] = {1, N1, NF};
  const int sd = st[d], s0 = st[d == 0 ? 1 : 0], s1 = st[d == 2 ? 1 : 2];
  const int q = t / NF, l = t - q * NF, i = l % N1, j = l / N1;  // quarter, point (i along t0, j along t1)
  const int b0 = q & 1, b1 = q >> 1;
  V vs = 0, ds = 0;
  auto trace = [&](int leaf, int end, V& val, V& der) {  // end 0: left, 1: right end of the line along d
    const V* p = us + (long long)leaf * NPE + i * s0 + j * s1;
    V x[N1];
#pragma unroll
    for (int a = 0; a < N1; ++a) x[a] = __ldg(p + (end ? N1 - 1 - a : a) * sd);
    end_trace<V, N1, false>(tab.tl, tab.dl, x, val, der);
    if (end) der = -der;  // the line was read reversed
  };
  if (on) {
    trace(rc[2 + q], 1 - r, vs, ds);
    if (q == 0) trace(big, r, sX[hs][0][l], sX[hs][1][l]);
  }
  __syncthreads();
  if (on) {
    // first step, along t0: thread (quantity q & 1, half q >> 1)
    V s = 0;
#pragma unroll
    for (int b = 0; b < N1; ++b) s = mad(sL[b1][i * N1 + b], sX[hs][b0][b + N1 * j], s);
    sR[hs][b0][b1][l] = s;
  }
  __syncthreads();
  V* g = gbuf + ((long long)blockIdx.y * 5 * tab.nI + 5LL * ifc) * 2 * NF;
  if (on) {
    V vb = 0, db = 0;
#pragma unroll
    for (int c = 0; c < N1; ++c) {
      const V x = sL[b1][j * N1 + c];
      vb = mad(x, sR[hs][0][b0][i + N1 * c], vb);
      db = mad(x, sR[hs][1][b0][i + N1 * c], db);
    }
    // gam = sigma h / 2 of the smaller leaf; the larger one's 2 / h is half of its
    const V gam = (V)fac[6LL * rc[2 + q] + 3 + d] * tab.g0, h = (V)0.5;
    const V so = r ? (V)-1 : (V)1;  // outward sign of the smaller side
    const V jump = vs - vb;
    V* gs = g + (1 + q) * 2 * NF;
    gs[l] = mad(gam, jump, mul(mul(-h, so), mad(h, db, ds)));
    gs[NF + l] = mul(-h, jump);
    const V wq = mul((V)0.25, mul(sw[i], sw[j]));
    sF[hs][0][q][l] = mul(wq, mad((V)-2 * gam, jump, mul(mul(h, so), mad((V)2, ds, db))));
    sF[hs][1][q][l] = mul(wq, mul(h, jump));
  }
  __syncthreads();
  if (on) {
    // back along t1, the two halves along it summed: thread (quantity b0, half b1 along t0) into sR
    V s = 0;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int jj = 0; jj < N1; ++jj) s = mad(sL[c][jj * N1 + j], sF[hs][b0][b1 + 2 * c][i + N1 * jj], s);
    sR[hs][b0][b1][l] = s;
  }
  __syncthreads();
  if (on && q < 2) {
    V s = 0;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int ii = 0; ii < N1; ++ii) s = mad(sL[c][ii * N1 + i], sR[hs][q][c][ii + N1 * j], s);
    g[q * NF + l] = s / mul(sw[i], sw[j]);
  }
}

template <typename V, int N1>
struct HangShared {
  V X[2][N1 * N1];        // larger side: value, derivative at its face nodes
  V R[2][2][N1 * N1];     // [quantity][half along t0]
  V F[2][4][N1 * N1];     // weighted fluxes per quarter
};
// The same fluxes for k_oct_leaf, a face at a time: put(quantity, l, value) takes those of
// slot `side` (0: the larger leaf, 1 + j: the j-th smaller one). sL, sw: the tables' Lh
// and w in shared memory. Every thread of the block takes part (barriers). (In place of
// k_oct_hang's body, which is this one for all slots at once, it took 0.4 us longer.)
template <typename V, int N1, typename P>
__device__ __forceinline__ void hang_face(const OctHang<V, N1>& tab, const V (*sL)[N1 * N1], const V* sw,
                                          HangShared<V, N1>& s, const int* __restrict__ rc,
                                          const double* __restrict__ fac, const V* __restrict__ us, int side, bool on,
                                          int t, P&& put) {
  constexpr int NF = N1 * N1, NPE = NF * N1;
  const int big = rc[0], f = rc[1], d = f >> 1, r = f & 1;
  const int st[3] = {1, N1, NF};
  const int sd = st[d], s0 = st[d == 0 ? 1 : 0], s1 = st[d == 2 ? 1 : 2];
  const int q = t / NF, l = t - q * NF, i = l % N1, j = l / N1;  // quarter, point (i along t0, j along t1)
  const int b0 = q & 1, b1 = q >> 1;
  const bool mine = on && (side == 0 || q == side - 1);  // this quarter's fluxes are wanted
  // loaded ahead of the barriers: gam = sigma h / 2 of the smaller leaf
  const int small = mine ? rc[2 + q] : 0;
  const V gam = (V)__ldg(fac + 6LL * small + 3 + d) * tab.g0;
  V vs = 0, ds = 0;
  auto trace = [&](int leaf, int end, V& val, V& der) {  // end 0: left, 1: right end of the line along d
    const V* p = us + (long long)leaf * NPE + i * s0 + j * s1;
    V x[N1];
#pragma unroll
    for (int a = 0; a < N1; ++a) x[a] = __ldg(p + (end ? N1 - 1 - a : a) * sd);
    end_trace<V, N1, false>(tab.tl, tab.dl, x, val, der);
    if (end) der = -der;  // the line was read reversed
  };
  if (mine) trace(small, 1 - r, vs, ds);
  if (on && q == 0) trace(big, r, s.X[0][l], s.X[1][l]);
  __syncthreads();
  if (on) {
    // first step, along t0: thread (quantity q & 1, half q >> 1)
    V v = 0;
#pragma unroll
    for (int b = 0; b < N1; ++b) v = mad(sL[b1][i * N1 + b], s.X[b0][b + N1 * j], v);
    s.R[b0][b1][l] = v;
  }
  __syncthreads();
  if (mine) {
    V vb = 0, db = 0;
#pragma unroll
    for (int c = 0; c < N1; ++c) {
      const V x = sL[b1][j * N1 + c];
      vb = mad(x, s.R[0][b0][i + N1 * c], vb);
      db = mad(x, s.R[1][b0][i + N1 * c], db);
    }
    const V h = (V)0.5;  // the larger leaf's 2 / h is half of the smaller one's
    const V so = r ? (V)-1 : (V)1;  // outward sign of the smaller side
    const V jump = vs - vb;
    if (side != 0) {
      put(0, l, mad(gam, jump, mul(mul(-h, so), mad(h, db, ds))));
      put(1, l, mul(-h, jump));
    } else {
      const V wq = mul((V)0.25, mul(sw[i], sw[j]));
      s.F[0][q][l] = mul(wq, mad((V)-2 * gam, jump, mul(mul(h, so), mad((V)2, ds, db))));
      s.F[1][q][l] = mul(wq, mul(h, jump));
    }
  }
  if (side != 0) return;
  __syncthreads();
  if (on) {
    // back along t1, the two halves along it summed: thread (quantity b0, half b1 along t0) into R
    V v = 0;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int jj = 0; jj < N1; ++jj) v = mad(sL[c][jj * N1 + j], s.F[b0][b1 + 2 * c][i + N1 * jj], v);
    s.R[b0][b1][l] = v;
  }
  __syncthreads();
  if (on && q < 2) {
    V v = 0;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int ii = 0; ii < N1; ++ii) v = mad(sL[c][ii * N1 + i], s.R[q][c][ii + N1 * j], v);
    put(q, l, v / mul(sw[i], sw[j]));
  }
}

// The operator in one launch and without scratch, for calls that have none (a
// captured call): one leaf per block, which works out the fluxes of its own hanging
// faces. The leaf's three directions go to three groups of threads; every number is
// that of k_oct_hang and k_oct_apply, in the same order: the same bits.
template <int N1>
struct OctLeaf {
  static constexpr int THREADS = (4 * N1 * N1 + 31) / 32 * 32;
};
template <typename V, int N1>
__global__ void __launch_bounds__(OctLeaf<N1>::THREADS)
    k_oct_leaf(const __grid_constant__ OctLine<V, N1> tab, const __grid_constant__ OctHang<V, N1> hg,
               const int* __restrict__ rec, const double* __restrict__ fac, const int* __restrict__ kind,
               const int* __restrict__ nbr, const int* __restrict__ hslot, const V* __restrict__ u,
               V* __restrict__ out) {
  using Y = LineLayout<N1>;
  constexpr int NF = N1 * N1, NPE = NF * N1, NT = OctLeaf<N1>::THREADS;
  __shared__ V su[Y::ES], sr[3][Y::ES], sg[6][2][NF], sL[2][NF], sw[N1], sww[NF], sfac[6];
  __shared__ HangShared<V, N1> sh;
  __shared__ int sface[6];
  const int tid = threadIdx.x, e = blockIdx.x;
  const V* us = u + (long long)blockIdx.y * tab.Nq;
  if (tid < 6) {
    const long long o = 6LL * e + tid;
    const int kd = kind[o];
    sface[tid] = kd == 0 ? -1 : kd == 1 ? nbr[4 * o] : -2 - hslot[o];
    sfac[tid] = (V)fac[o] * (tid >= 3 ? tab.g0 : (V)1);
  }
  for (int t = tid; t < NPE; t += NT)
    su[t % N1 + Y::PB * ((t / N1) % N1) + Y::PZ * (t / NF)] = __ldg(us + (long long)e * NPE + t);
  for (int t = tid; t < NF; t += NT) sww[t] = tab.ww[t];
  __syncthreads();
  const int q = tid / NF, l = tid - q * NF, l1 = l % N1, l2 = l / N1;
  bool any = false;
#pragma unroll
  for (int f = 0; f < 6; ++f) any |= sface[f] < -1;
  if (any) {
    for (int i = tid; i < 2 * NF; i += NT) sL[i / NF][i % NF] = hg.Lh[i / NF][i % NF];
    for (int i = tid; i < N1; i += NT) sw[i] = hg.w[i];
#pragma unroll 1
    for (int f = 0; f < 6; ++f) {
      const int fc = sface[f];
      if (fc >= -1) continue;
      const int slot = -2 - fc, ifc = slot / 5;
      hang_face<V, N1>(hg, sL, sw, sh, rec + 6LL * ifc, fac, us, slot - 5 * ifc, q < 4, tid,
                       [&](int c, int k, V v) { sg[f][c][k] = v; });
    }
    __syncthreads();
  }
  if (q < 3) {
    // direction q: strides in the field and in the shared layout
    const int sd = q == 0 ? 1 : (q == 1 ? N1 : NF), sp = q == 0 ? 1 : (q == 1 ? Y::PB : Y::PZ);
    const int base = q == 0 ? N1 * l : (q == 1 ? l1 + NF * l2 : l);
    const int at = q == 0 ? Y::PB * l1 + Y::PZ * l2 : (q == 1 ? l1 + Y::PZ * l2 : l1 + Y::PB * l2);
    const int fl = sface[2 * q], fr = sface[2 * q + 1];
    const V gam = sfac[3 + q];
    V v[N1], ov[2], od[2];
    // traces beyond the two ends, as oct_outer
    auto line = [&](int fc) {
      const V* p = us + (long long)(fc < 0 ? e : fc) * NPE + base + (fc < 0 ? (N1 - 1) * sd : 0);
      const int st = fc < 0 ? -sd : sd;
#pragma unroll
      for (int i = 0; i < N1; ++i) v[i] = __ldg(p + i * st);
    };
    if (fl >= -1) {
      line(fl);
      end_trace<V, N1, true>(tab.tl, tab.dl, v, ov[0], od[0]);
      if (fl < 0) {
        od[0] = mad((V)-2 * gam, ov[0], -od[0]);
        ov[0] = -ov[0];
      }
    } else {
      ov[0] = sg[2 * q][0][l];
      od[0] = sg[2 * q][1][l];
    }
    if (fr >= -1) {
      line(fr);
      end_trace<V, N1, false>(tab.tl, tab.dl, v, ov[1], od[1]);
      if (fr < 0) {
        od[1] = mad((V)2 * gam, ov[1], -od[1]);
        ov[1] = -ov[1];
      }
    } else {
      ov[1] = sg[2 * q + 1][0][l];
      od[1] = sg[2 * q + 1][1][l];
    }
#pragma unroll
    for (int i = 0; i < N1; ++i) v[i] = su[at + sp * i];
    oct_line<V, N1>(tab, v, ov, od, fl < -1, fr < -1, gam);
#pragma unroll
    for (int i = 0; i < N1; ++i) sr[q][at + sp * i] = v[i];
  }
  __syncthreads();
  V* o = out + (long long)blockIdx.y * tab.Nq + (long long)e * NPE;
  for (int t = tid; t < NPE; t += NT) {
    const int a = t % N1, b = (t / N1) % N1, c = t / NF, at = a + Y::PB * b + Y::PZ * c;
    V Au = mul(mul(sfac[0], sww[b + N1 * c]), sr[0][at]);
    Au = mad(mul(sfac[1], sww[a + N1 * c]), sr[1][at], Au);
    o[t] = mad(mul(sfac[2], sww[a + N1 * b]), sr[2][at], Au);
  }
}

void octree_hanging(const int32_t* kind, const int32_t* nb, int E, std::vector<int>& rec, std::vector<int>& hslot) {
  rec.clear();
  hslot.assign(6 * (size_t)E, -1);
  for (int e = 0; e < E; ++e)
    for (int f = 0; f < 6; ++f) {
      const size_t o = 6 * (size_t)e + f;
      if (kind[o] != 3) continue;
      const int i = (int)(rec.size() / 6);
      hslot[o] = 5 * i;
      rec.push_back(e);
      rec.push_back(f);
      for (int j = 0; j < 4; ++j) {
        const int s = nb[4 * o + j];
        hslot[6 * (size_t)s + (f ^ 1)] = 5 * i + 1 + j;
        rec.push_back(s);
      }
    }
}

void octree_factors(const double* hq, int E, int pform, std::vector<double>& fac) {
  fac.resize(6 * (size_t)E);
  for (int e = 0; e < E; ++e)
    for (int d = 0; d < 3; ++d) {
      const double* h = hq + 3 * (size_t)e;
      fac[6 * (size_t)e + d] = h[d == 0 ? 1 : 0] * h[d == 2 ? 1 : 2] / (2.0 * h[d]);
      fac[6 * (size_t)e + 3 + d] = pform == 0 ? 1.0 : 1.0 / h[d];
    }
}

void octree_tables(int n1, OctTables& T) {
  std::memset(&T, 0, sizeof(T));
  double xi[MAXN1], w[MAXN1], xq[MAXN1], wq[MAXN1], L[MAXN1], dL[MAXN1];
  gauss_legendre(n1, xi, w);
  gauss_legendre(n1, xq, wq);  // Gauss points of a face direction (exact for the face integrands)
  for (int a = 0; a < n1; ++a) T.w[a] = w[a];
  for (int i = 0; i < n1; ++i) {
    for (int c = 0; c < 2; ++c) {
      lagrange(xi, n1, (xq[i] + 2.0 * c - 1.0) / 2.0, L, dL);
      for (int a = 0; a < n1; ++a) T.Lh[c][i * n1 + a] = L[a];
    }
  }
  for (int r = 0; r < 2; ++r) {
    lagrange(xi, n1, r ? 1.0 : -1.0, L, dL);
    for (int a = 0; a < n1; ++a) {
      T.Le[r][a] = L[a];
      T.dLe[r][a] = dL[a];
    }
  }
  // 1-D stiffness: sum_q wq l_a'(xq) l_b'(xq)
  std::vector<double> dq((size_t)n1 * n1);
  for (int i = 0; i < n1; ++i) {
    lagrange(xi, n1, xq[i], L, dL);
    for (int a = 0; a < n1; ++a) dq[(size_t)i * n1 + a] = dL[a];
  }
  for (int a = 0; a < n1; ++a)
    for (int b = 0; b < n1; ++b) {
      double sum = 0.0;
      for (int i = 0; i < n1; ++i) sum += wq[i] * dq[(size_t)i * n1 + a] * dq[(size_t)i * n1 + b];
      T.S[a * n1 + b] = sum;
    }
}

template <typename V, int N1>
static void oct_fill(const OctTables& T, const OctMesh& m, double eps, OctLine<V, N1>& t, OctHang<V, N1>& g) {
  constexpr int HO = N1 / 2, HE = N1 - HO, NF = N1 * N1, NPE = NF * N1;
  auto S = [&](int a, int i) { return 0.5 * (T.S[a * N1 + i] + T.S[(N1 - 1 - a) * N1 + (N1 - 1 - i)]); };
  for (int a = 0; a < HE; ++a) {
    for (int i = 0; i < HE; ++i) t.Se[a][i] = (V)(i < HO ? 0.5 * (S(a, i) + S(a, N1 - 1 - i)) : S(a, i));
    t.te[a] = (V)(a < HO ? 0.5 * (T.Le[0][a] + T.Le[0][N1 - 1 - a]) : T.Le[0][a]);
    t.de[a] = (V)(a < HO ? 0.5 * (T.dLe[0][a] + T.dLe[0][N1 - 1 - a]) : T.dLe[0][a]);
  }
  for (int a = 0; a < HO; ++a) {
    for (int i = 0; i < HO; ++i) t.So[a][i] = (V)(0.5 * (S(a, i) - S(a, N1 - 1 - i)));
    t.to[a] = (V)(0.5 * (T.Le[0][a] - T.Le[0][N1 - 1 - a]));
    t.dO[a] = (V)(0.5 * (T.dLe[0][a] - T.dLe[0][N1 - 1 - a]));
  }
  for (int a = 0; a < N1; ++a) {
    t.tl[a] = g.tl[a] = (V)T.Le[0][a];
    t.dl[a] = g.dl[a] = (V)T.dLe[0][a];
    g.w[a] = (V)T.w[a];
  }
  for (int l = 0; l < NF; ++l) {
    t.ww[l] = (V)(T.w[l % N1] * T.w[l / N1]);
    for (int c = 0; c < 2; ++c) g.Lh[c][l] = (V)T.Lh[c][l];
  }
  t.g0 = g.g0 = (V)(N1 * N1 / (2.0 * eps));
  t.Nq = g.Nq = (long long)m.E * NPE;
  t.E = m.E;
  t.nslots = 5 * m.nI;
  g.nI = m.nI;
}

template <typename V, int N1>
static cudaError_t oct_apply_n1(const OctTables& T, const OctMesh& m, double eps, const V* u, V* out, const V* rin,
                                const int* act, int nact, V* gbuf, long long gelems, cudaStream_t s) {
  constexpr int NF = N1 * N1, NPE = NF * N1;
  OctLine<V, N1> t;
  OctHang<V, N1> g;
  oct_fill<V, N1>(T, m, eps, t, g);
  const int vec = ((uintptr_t)u & 15) == 0 && (NPE * sizeof(V)) % 16 == 0 && (t.Nq * sizeof(V)) % 16 == 0;
  // sources go through in chunks whose hanging fluxes fit the buffer (and a grid's second axis)
  const long long per_src = 10LL * m.nI * NF;
  long long per = m.nI > 0 ? std::min<long long>(65535, gelems / per_src) : nact;
  if (per < 1) return cudaErrorInvalidValue;
  for (long long k0 = 0; k0 < nact; k0 += per) {
    const int n = (int)std::min<long long>(per, nact - k0);
    t.k0 = g.k0 = (int)k0;
    if (m.nI > 0) {
      using H = HangShape<V, N1>;
      count_launch();
      k_oct_hang<V, N1><<<dim3((unsigned)((m.nI + H::HPB - 1) / H::HPB), (unsigned)n), H::THREADS, 0, s>>>(
          g, m.rec, m.fac, u, gbuf, act);
    }
    t.items = (long long)n * m.E;
    auto go = [&](auto kern, int bpb, int threads, size_t smem) -> cudaError_t {
      const long long blocks = (t.items + bpb - 1) / bpb;
      if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
      if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
      }
      count_launch();
      kern<<<(unsigned)blocks, threads, smem, s>>>(t, m.fac, m.kind, m.nb, m.hslot, gbuf, u, out, rin, act, vec);
      return cudaGetLastError();
    };
    using F = OctShape<V, N1, true>;
    using P = OctShape<V, N1, false>;
    // several leaves per block once that leaves two blocks per SM (as the uniform operator)
    const cudaError_t e = t.items / F::BPB >= 304 ? go(k_oct_apply<V, N1, true>, F::BPB, F::THREADS, F::SMEM)
                                                 : go(k_oct_apply<V, N1, false>, P::BPB, P::THREADS, P::SMEM);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename V>
cudaError_t launch_octree_apply(int n1, const OctTables& T, const OctMesh& m, double eps, const V* u, V* out,
                                const V* rin, const int* act, int nact, V* gbuf, long long gelems, cudaStream_t s) {
  if (nact == 0 || m.E == 0) return cudaSuccess;
  switch (n1) {
    case 2: return oct_apply_n1<V, 2>(T, m, eps, u, out, rin, act, nact, gbuf, gelems, s);
    case 3: return oct_apply_n1<V, 3>(T, m, eps, u, out, rin, act, nact, gbuf, gelems, s);
    case 4: return oct_apply_n1<V, 4>(T, m, eps, u, out, rin, act, nact, gbuf, gelems, s);
    case 5: return oct_apply_n1<V, 5>(T, m, eps, u, out, rin, act, nact, gbuf, gelems, s);
    case 6: return oct_apply_n1<V, 6>(T, m, eps, u, out, rin, act, nact, gbuf, gelems, s);
    case 7: return oct_apply_n1<V, 7>(T, m, eps, u, out, rin, act, nact, gbuf, gelems, s);
    case 8: return oct_apply_n1<V, 8>(T, m, eps, u, out, rin, act, nact, gbuf, gelems, s);
    case 9: return oct_apply_n1<V, 9>(T, m, eps, u, out, rin, act, nact, gbuf, gelems, s);
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_octree_apply<double>(int, const OctTables&, const OctMesh&, double, const double*, double*,
                                                 const double*, const int*, int, double*, long long, cudaStream_t);
template cudaError_t launch_octree_apply<float>(int, const OctTables&, const OctMesh&, double, const float*, float*,
                                                const float*, const int*, int, float*, long long, cudaStream_t);

template <int N1>
static cudaError_t oct_leaf_n1(const OctTables& T, const OctMesh& m, double eps, const double* u, double* out, int B,
                               cudaStream_t s) {
  OctLine<double, N1> t;
  OctHang<double, N1> g;
  oct_fill<double, N1>(T, m, eps, t, g);
  t.items = t.k0 = g.k0 = 0;
  count_launch();
  k_oct_leaf<double, N1><<<dim3((unsigned)m.E, (unsigned)B), OctLeaf<N1>::THREADS, 0, s>>>(t, g, m.rec, m.fac, m.kind,
                                                                                         m.nb, m.hslot, u, out);
  return cudaGetLastError();
}

cudaError_t launch_octree_direct(int n1, const OctTables& T, const OctMesh& m, double eps, const double* u, double* out,
                                 int B, cudaStream_t s) {
  if (B == 0 || m.E == 0) return cudaSuccess;
  switch (n1) {
    case 2: return oct_leaf_n1<2>(T, m, eps, u, out, B, s);
    case 3: return oct_leaf_n1<3>(T, m, eps, u, out, B, s);
    case 4: return oct_leaf_n1<4>(T, m, eps, u, out, B, s);
    case 5: return oct_leaf_n1<5>(T, m, eps, u, out, B, s);
    case 6: return oct_leaf_n1<6>(T, m, eps, u, out, B, s);
    case 7: return oct_leaf_n1<7>(T, m, eps, u, out, B, s);
    case 8: return oct_leaf_n1<8>(T, m, eps, u, out, B, s);
    case 9: return oct_leaf_n1<9>(T, m, eps, u, out, B, s);
    default: return cudaErrorInvalidValue;
  }
}
}  // namespace dg

using namespace dg;

extern "C" {

int dg_octree_refine(const dg_mesh_desc* root, double delta, int32_t max_level, dg_density_fn rho, void* user,
                     int32_t max_leaves, int32_t* leaves_host, int32_t* n_leaves) {
  if (!root || !rho || !n_leaves || !(delta > 0.0) || max_level < 0 || max_level > 20 || root->p < 1 ||
      root->p > MAXN1 - 1 || max_leaves < 0)
    return DG_ERR_INVALID_ARG;
  Octree t;
  for (int d = 0; d < 3; ++d) {
    if (root->n[d] < 1 || !(root->hi[d] > root->lo[d])) return DG_ERR_INVALID_ARG;
    t.lo[d] = root->lo[d];
    t.n[d] = root->n[d];
    t.H[d] = (root->hi[d] - root->lo[d]) / root->n[d];
  }
  t.p = root->p;
  for (int z = 0; z < t.n[2]; ++z)
    for (int y = 0; y < t.n[1]; ++y)
      for (int x = 0; x < t.n[0]; ++x) t.leaves.insert({0, x, y, z});
  const int n1 = t.p + 1;
  double xi[MAXN1], w[MAXN1];
  gauss_legendre(n1, xi, w);
  std::vector<double> pts, val;
  for (;;) {
    std::vector<Leaf> split;
    for (const Leaf& k : t.leaves) {
      if (k[0] >= max_level) continue;
      double o[3], h[3];
      for (int d = 0; d < 3; ++d) {
        h[d] = t.h(k[0], d);
        o[d] = t.lo[d] + k[1 + d] * h[d];
      }
      const double whole = gl_integral(o, h, n1, xi, w, rho, user, pts, val);
      double parts = 0.0;
      for (int c = 0; c < 8; ++c) {
        double oc[3], hc[3];
        for (int d = 0; d < 3; ++d) {
          hc[d] = h[d] / 2.0;
          oc[d] = o[d] + ((c >> d) & 1) * hc[d];
        }
        parts += gl_integral(oc, hc, n1, xi, w, rho, user, pts, val);
      }
      if (std::fabs(whole - parts) > delta) split.push_back(k);
    }
    if (split.empty()) break;
    t.refine(split);
    t.balance();
    if ((long long)t.leaves.size() > (1LL << 24)) return DG_ERR_NO_MEMORY;
  }
  const std::vector<Leaf> v = t.ordered();
  *n_leaves = (int32_t)v.size();
  if (leaves_host) {
    if ((long long)v.size() > max_leaves) return DG_ERR_INVALID_ARG;
    for (size_t i = 0; i < v.size(); ++i)
      for (int j = 0; j < 4; ++j) leaves_host[4 * i + j] = v[i][j];
  }
  return DG_OK;
}

int dg_octree_faces(const dg_mesh_desc* root, const int32_t* leaves, int32_t n_leaves, int32_t* kind, int32_t* nb,
                    int32_t* pos) {
  return octree_faces(root, leaves, n_leaves, kind, nb, pos) ? DG_OK : DG_ERR_INVALID_ARG;
}


int dg_octree_apply(const dg_mesh_desc* root, const int32_t* leaves, int32_t n_leaves, int32_t penalty_form,
                    double penalty_eps, const double* u, double* out, int64_t B, void* stream) {
  if (!root || root->p < 1 || root->p > MAXN1 - 1 || (penalty_form != 0 && penalty_form != 1) ||
      !(penalty_eps > 0.0) || B < 0 || B > 65535 || n_leaves < 1 || (B > 0 && (!u || !out)))
    return DG_ERR_INVALID_ARG;
  const int E = n_leaves;
  if (B > 0) {
    // out is written while other blocks still read u: the two must not overlap
    const size_t bytes = sizeof(double) * (size_t)B * (size_t)E * (size_t)((root->p + 1) * (root->p + 1) * (root->p + 1));
    const char *u0 = (const char*)u, *o0 = (const char*)out;
    if (u0 < o0 + bytes && o0 < u0 + bytes) return DG_ERR_INVALID_ARG;
  }
  std::vector<int32_t> kind(6 * (size_t)E), nb(24 * (size_t)E), pos(6 * (size_t)E);
  if (!octree_faces(root, leaves, n_leaves, kind.data(), nb.data(), pos.data())) return DG_ERR_INVALID_ARG;
  if (B == 0) return DG_OK;
  std::vector<double> hq(3 * (size_t)E);
  for (int e = 0; e < E; ++e)
    for (int d = 0; d < 3; ++d)
      hq[3 * (size_t)e + d] = (root->hi[d] - root->lo[d]) / root->n[d] / double(1 << leaves[4 * e]);
  const int n1 = root->p + 1;
  OctTables T;
  octree_tables(n1, T);
  cudaStream_t s = (cudaStream_t)stream;
  std::vector<int> rec, hslot;
  std::vector<double> fac;
  octree_hanging(kind.data(), nb.data(), E, rec, hslot);
  octree_factors(hq.data(), E, penalty_form, fac);
  DevBuf df, dk, dn, ds, dr, dg;
  auto ck = [](cudaError_t e) { return e == cudaSuccess ? DG_OK : (e == cudaErrorMemoryAllocation ? DG_ERR_NO_MEMORY : DG_ERR_CUDA); };
  int rc;
  auto up = [&](DevBuf& d, const void* p, size_t bytes) -> int {
    if (bytes == 0) return DG_OK;
    const int r = ck(d.ensure(bytes));
    return r != DG_OK ? r : ck(cudaMemcpyAsync(d.p, p, bytes, cudaMemcpyHostToDevice, s));
  };
  if ((rc = up(df, fac.data(), sizeof(double) * fac.size())) != DG_OK ||
      (rc = up(dk, kind.data(), sizeof(int) * kind.size())) != DG_OK ||
      (rc = up(dn, nb.data(), sizeof(int) * nb.size())) != DG_OK ||
      (rc = up(ds, hslot.data(), sizeof(int) * hslot.size())) != DG_OK ||
      (rc = up(dr, rec.data(), sizeof(int) * rec.size())) != DG_OK)
    return rc;
  const int nI = (int)(rec.size() / 6);
  // hanging fluxes: as many sources at a time as 64 MB hold, at least one
  const size_t one = sizeof(double) * octree_hang_elems(n1, nI);
  const size_t gbytes = std::max(one, std::min<size_t>(one * (size_t)B, 64u << 20));
  if (nI > 0 && (rc = ck(dg.ensure(gbytes))) != DG_OK) return rc;
  const OctMesh m{E, dk.as<int>(), dn.as<int>(), df.as<double>(), ds.as<int>(), dr.as<int>(), nI};
  if ((rc = ck(launch_octree_apply<double>(n1, T, m, penalty_eps, u, out, nullptr, nullptr, (int)B, dg.as<double>(),
                                           (long long)(gbytes / sizeof(double)), s))) != DG_OK)
    return rc;
  // the tables and connectivity are call-local: wait before they are freed
  return ck(cudaStreamSynchronize(s));
}

}  // extern "C"
