// Per-element 3-D convolutional network for the learned initial guess (not in
// the paper; the learned form of the exchange-build solves).
//
// Network: per element, two input channels on the (p+1)^3 nodes (scaled
// source, scaled coarse-grid solution) -> conv 3x3x3 (2 -> 32) -> ReLU ->
// conv 3x3x3 (32 -> 32) -> ReLU -> conv 3x3x3 (32 -> 2), zero padding at the
// element border. Weights are kept in FP32 (master copy, Adam) and used in
// BF16; activations are stored in BF16; every sum accumulates in FP32.
//
// Layouts: nodes of an element x-fastest, channels last: act[e][node][C].
// Tap t = (dz+1)*9 + (dy+1)*3 + (dx+1). Parameter vector (FP32):
//   W1 [27][2][32] | b1 [32] | W2 [27][32][32] (tap, ci, co) | b2 [32] |
//   W3 [27][32][2] | b3 [2]
// BF16 copies of W2: W2t [27][32 co][32 ci] (forward) and W2o [27][32 ci][32 co]
// (gradient with respect to the layer input).
//
// The 32 -> 32 layer and its two gradients run on the tensor cores with
// mma.sync m16n8k16 (BF16 in, FP32 accumulate); A tiles come from
// channel-last shared memory with ldmatrix (16 nodes x 16 channels), the
// convolution taps are row offsets into a zero-bordered (p+3)^3 grid.
#include <cuda_bf16.h>

#include "dg_internal.h"

namespace dg {

constexpr int NN_OW1 = 0, NN_OB1 = 1728, NN_OW2 = 1760, NN_OB2 = 29408, NN_OW3 = 29440, NN_OB3 = 31168;
static_assert(NN_NPARAM == 31170, "parameter layout");
constexpr int NN_H = 32;

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void ldsm_x4(unsigned addr, unsigned& r0, unsigned& r1, unsigned& r2, unsigned& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(unsigned addr, unsigned& r0, unsigned& r1, unsigned& r2, unsigned& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void mma16816(float* d, unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                         unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

template <int N1>
struct NNCfg {
  static constexpr int P = N1 + 2;
  static constexpr int P3 = P * P * P;
  static constexpr int NPE = N1 * N1 * N1;
  // elements that a block works on at once, each with its own border
  static constexpr int GROUP = N1 == 2 ? 12 : (N1 == 3 ? 7 : (N1 == 4 ? 4 : (N1 == 5 ? 2 : 1)));
};

template <int N1>
__device__ __forceinline__ int pad_index(int n) {
  constexpr int P = N1 + 2;
  const int x = n % N1, y = (n / N1) % N1, z = n / (N1 * N1);
  return (z + 1) * P * P + (y + 1) * P + (x + 1);
}
// the same for node n of a group of elements
template <int N1>
__device__ __forceinline__ int group_index(int n) {
  using C = NNCfg<N1>;
  if constexpr (C::GROUP == 1) return pad_index<N1>(n);
  return n / C::NPE * C::P3 + pad_index<N1>(n % C::NPE);
}
template <int N1>
__device__ __forceinline__ int tap_offset(int t) {
  constexpr int P = N1 + 2;
  return (t / 9 - 1) * P * P + ((t / 3) % 3 - 1) * P + (t % 3 - 1);
}

// pair i of a two-channel field of the caller's: 8-byte loads where its address allows (vec)
__device__ __forceinline__ float2 load_pair(const float* __restrict__ p, long long i, bool vec) {
  return vec ? ((const float2*)p)[i] : make_float2(p[2 * i], p[2 * i + 1]);
}
static int pairs_aligned(const void* a, const void* b) { return (((uintptr_t)a | (uintptr_t)b) & 7) == 0; }

// ---------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------
// Shared-memory activations: row p (padded node) holds 32 BF16 channels as four
// 16-byte chunks; chunk c of row p is stored at position c ^ ((p >> 1) & 3), so
// the eight consecutive rows an ldmatrix phase reads fall into distinct banks.
__device__ __forceinline__ int swz(int p, int ch) {
  return p * NN_H + ((((ch >> 3) ^ ((p >> 1) & 3)) << 3) | (ch & 7));
}

// shared-memory index of entry (row, ch) of a staged copy of W2 (rows of 32 channels)
__device__ __forceinline__ int swz_w2(int row, int ch) {
  return row * 32 + ((((ch >> 3) ^ ((row >> 1) & 3)) << 3) | (ch & 7));
}

// Forward kernel: one block per SM, 16 warps, a group of elements at a time.
// Layer 1: a thread computes 4 channels of a line of nodes along x, a warp (mostly)
// lines of the same channels: per row of taps it loads p + 3 inputs (row strides free of
// bank conflicts) and 6 broadcast float4 of weights for 48 (p + 1) products; one
// node and 8 channels per thread before, 5 loads for 16 products. Products and sums
// per output are in the same order: the same bits.
// Layer 2 (tensor cores): a warp owns two 16-node tiles and loads the operand tiles
// of W2 with ldmatrix (8 scalar loads per 8 MMAs before); same bits.
// Layer 3: a thread sums 4 input channels for a line of nodes, eight lanes are one
// line; their sums are added by halving shuffles (one thread per node before: half
// of the warps' issue slots idle, 20 loads for 64 products).
// Measured (GB300, with activations stored): 16384 elements at p = 7 4.92 -> 2.91 ms,
// 2000 at p = 6 0.57 -> 0.39, 200 at p = 4 0.061 -> 0.049, 4000 at p = 1 0.306 -> 0.060.
constexpr int NN_FWD_THREADS = 512;

// ldmatrix address of chunk c (8 channels) of row p, and of chunk c ^ 2 (16 channels on)
__device__ __forceinline__ unsigned row_addr(unsigned base, int p, int c) {
  return base + 64u * p + (((p << 3) & 0x30) ^ (c << 4));
}
__device__ __forceinline__ unsigned row_addr2(unsigned base, int p, int c) {
  return base + 64u * p + (((p << 3) & 0x30) ^ (c << 4) ^ 32);
}

template <int N1>
struct FwdCfg {
  using C = NNCfg<N1>;
  // strides of the rows and planes of the two-channel fields, in float2, by which 16
  // lanes on lines of neighbouring planes read distinct banks: odd rows and planes 8
  // modulo 16, or, where P is twice an odd number (p = 7, which has no room for more),
  // rows as they are and odd planes
  static constexpr bool TWO = C::P % 4 == 2;
  static constexpr int YS = TWO ? C::P : C::P | 1, ZS = TWO ? C::P * C::P + 1 : (C::P * YS + 7) / 16 * 16 + 8;
  static constexpr int IS = C::P * ZS;
  static constexpr int ROWS = C::P3 * C::GROUP;
  static constexpr size_t SMEM = 2 * sizeof(__nv_bfloat16) * ROWS * NN_H + sizeof(__nv_bfloat16) * 27 * 32 * 32 +
                                 sizeof(float2) * C::GROUP * IS + sizeof(float) * (1760 + 1728 + 32);
};

template <int N1>
__global__ void __launch_bounds__(NN_FWD_THREADS, 1)
    k_nn_forward(const float* __restrict__ prm, const __nv_bfloat16* __restrict__ W2t, const float* __restrict__ in,
                 float* __restrict__ out, __nv_bfloat16* __restrict__ a1_out, __nv_bfloat16* __restrict__ a2_out,
                 long long ne, int ng, int vec) {
  using C = NNCfg<N1>;
  using F = FwdCfg<N1>;
  constexpr int ROWS = F::ROWS, P = C::P, NT = NN_FWD_THREADS, NW = NT / 32, LPE = N1 * N1;
  extern __shared__ __align__(16) unsigned char smem[];
  __nv_bfloat16* sA1 = (__nv_bfloat16*)smem;                           // [ROWS][32] swizzled
  __nv_bfloat16* sA2 = sA1 + ROWS * NN_H;                               // [ROWS][32] swizzled
  __nv_bfloat16* sW2 = sA2 + ROWS * NN_H;                               // [27 * 32 co][32 ci] swizzled
  float* sW1 = (float*)(sW2 + 27 * 32 * 32);                           // [27][2][32] + b1
  float* sW3 = sW1 + 1728 + 32;                                        // [27][2][8 groups][2 ci][2 co]
  float* sb2 = sW3 + 1728;                                             // [32]
  float2* sIn = (float2*)(sb2 + 32);                                   // [GROUP][P][P][.]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < C::GROUP * F::IS; i += NT) sIn[i] = make_float2(0.f, 0.f);
  for (int i = tid; i < ROWS * NN_H; i += NT) ((unsigned*)sA1)[i] = 0u;  // sA1 and sA2
  for (int i = tid; i < 27 * 32 * 4; i += NT)
    *(uint4*)(sW2 + swz_w2(i >> 2, (i & 3) * 8)) = ((const uint4*)W2t)[i];
  for (int i = tid; i < 1760; i += NT) sW1[i] = prm[NN_OW1 + i];
  for (int i = tid; i < 1728; i += NT) {  // channel 4 g + 2 k + c of tap t
    const int t = i / 64, ci = i / 2 % 32;
    sW3[t * 64 + (ci >> 1 & 1) * 32 + (ci >> 2) * 4 + (i & 3)] = prm[NN_OW3 + i];
  }
  for (int i = tid; i < 32; i += NT) sb2[i] = prm[NN_OB2 + i];
  const float b30 = prm[NN_OB3], b31 = prm[NN_OB3 + 1];
  __syncthreads();
  const int g = lane >> 2, c4 = lane & 3, j = lane >> 3, r = lane & 7;
  for (long long e0 = (long long)blockIdx.x * ng; e0 < ne; e0 += (long long)gridDim.x * ng) {
    const long long nb0 = e0 * C::NPE;  // first node of the pass; np nodes on nl lines
    const int nel = (int)(ne - e0 < ng ? ne - e0 : ng), np = nel * C::NPE, nl = nel * LPE, MT = (np + 15) / 16;
    for (int i = tid; i < np; i += NT) {
      const int l = i / N1, y = l % N1, z = l / N1 % N1;
      sIn[l / LPE * F::IS + (z + 1) * F::ZS + (y + 1) * F::YS + i % N1 + 1] = load_pair(in, nb0 + i, vec);
    }
    __syncthreads();
    // layer 1 (2 -> 32)
    for (int w = tid; w < nl * 8; w += NT) {
      const int cg = w / nl * 4, l = w % nl;
      const int y = l % N1, z = l / N1 % N1;
      const float2* src = sIn + l / LPE * F::IS + z * F::ZS + y * F::YS;
      float acc[N1][4];
#pragma unroll
      for (int i = 0; i < N1; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[i][c] = sW1[1728 + cg + c];
#pragma unroll 1
      for (int d = 0; d < 9; ++d) {
        const float2* row = src + d / 3 * F::ZS + d % 3 * F::YS;
        float2 v[P];
#pragma unroll
        for (int i = 0; i < P; ++i) v[i] = row[i];
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          const float4 wa = *(const float4*)(sW1 + (3 * d + dx) * 64 + cg);
          const float4 wb = *(const float4*)(sW1 + (3 * d + dx) * 64 + 32 + cg);
          const float w0[4] = {wa.x, wa.y, wa.z, wa.w}, w1[4] = {wb.x, wb.y, wb.z, wb.w};
#pragma unroll
          for (int i = 0; i < N1; ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[i][c] += v[i + dx].x * w0[c] + v[i + dx].y * w1[c];
        }
      }
      const int p0 = l / LPE * C::P3 + (z + 1) * P * P + (y + 1) * P + 1;
#pragma unroll
      for (int i = 0; i < N1; ++i) {
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(fmaxf(acc[i][0], 0.f), fmaxf(acc[i][1], 0.f));
        const __nv_bfloat162 h1 = __floats2bfloat162_rn(fmaxf(acc[i][2], 0.f), fmaxf(acc[i][3], 0.f));
        *(uint2*)(sA1 + swz(p0 + i, cg)) = make_uint2(*(const unsigned*)&h0, *(const unsigned*)&h1);
      }
    }
    __syncthreads();
    // layer 2 (32 -> 32) on the tensor cores: warp owns node tiles warp, warp + NW, ...
    for (int mt0 = warp; mt0 < MT; mt0 += 2 * NW) {
      float acc[2][4][4];
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.f;
      int rowp[2];
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const int node = (mt0 + NW * a) * 16 + r + 8 * (j & 1);
        rowp[a] = node < np ? group_index<N1>(node) : -1;  // rows past the nodes read the zero corner
      }
      // B tiles: matrix j = input channels 8 j .. 8 j + 7 of the 8 rows co of column tile nt
      unsigned wa = smem_u32(sW2 + swz_w2(r, 8 * j));
      const unsigned ab = smem_u32(sA1);
#pragma unroll 1
      for (int d = 0; d < 9; ++d) {
        const int od = (d / 3 - 1) * P * P + (d % 3 - 1) * P - 1;
#pragma unroll 1
        for (int dx = 0; dx < 3; ++dx, wa += 2048) {
          unsigned b[4][4];
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) ldsm_x4(wa + nt * 512, b[nt][0], b[nt][1], b[nt][2], b[nt][3]);
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            if (mt0 + NW * a >= MT) continue;
            const int q = rowp[a] >= 0 ? rowp[a] + od + dx : 0;
#pragma unroll
            for (int kh = 0; kh < 2; ++kh) {
              unsigned a0, a1, a2, a3;
              ldsm_x4(kh ? row_addr2(ab, q, j >> 1) : row_addr(ab, q, j >> 1), a0, a1, a2, a3);
#pragma unroll
              for (int nt = 0; nt < 4; ++nt) mma16816(acc[a][nt], a0, a1, a2, a3, b[nt][2 * kh], b[nt][2 * kh + 1]);
            }
          }
        }
      }
      // epilogue: bias, ReLU, BF16 into sA2 (rows g and g+8, columns 2c4, 2c4+1 of each n tile)
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int node = (mt0 + NW * a) * 16 + g + 8 * h;
          if (node >= np) continue;
          const int p = group_index<N1>(node);
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            const int co = nt * 8 + 2 * c4;
            const float v0 = fmaxf(acc[a][nt][2 * h] + sb2[co], 0.f);
            const float v1 = fmaxf(acc[a][nt][2 * h + 1] + sb2[co + 1], 0.f);
            *(__nv_bfloat162*)(sA2 + swz(p, co)) = __floats2bfloat162_rn(v0, v1);
          }
        }
    }
    __syncthreads();
    // layer 3 (32 -> 2): lane r of eight sums channels 4 r .. 4 r + 3 of a line
    for (int w = warp; w < (nl + 3) / 4; w += NW) {
      const int l = w * 4 + j, ll = l < nl ? l : 0;
      const int y = ll % N1, z = ll / N1 % N1;
      const int p0 = ll / LPE * C::P3 + z * P * P + y * P;
      float acc[8][2];
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = 0.f;
#pragma unroll 1
      for (int d = 0; d < 9; ++d) {
        const int q = p0 + d / 3 * P * P + d % 3 * P;
        float4 wa[3], wb[3];  // (ci, co) = (0, 0), (0, 1), (1, 0), (1, 1) and the next two channels
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          wa[dx] = *(const float4*)(sW3 + (3 * d + dx) * 64 + 4 * r);
          wb[dx] = *(const float4*)(sW3 + (3 * d + dx) * 64 + 32 + 4 * r);
        }
#pragma unroll
        for (int i = 0; i < P; ++i) {
          const uint2 raw = *(const uint2*)(sA2 + swz(q + i, 4 * r));
          const float v0 = __uint_as_float(raw.x << 16), v1 = __uint_as_float(raw.x & 0xffff0000u);
          const float v2 = __uint_as_float(raw.y << 16), v3 = __uint_as_float(raw.y & 0xffff0000u);
#pragma unroll
          for (int dx = 0; dx < 3; ++dx) {
            const int x = i - dx;
            if (x < 0 || x >= N1) continue;
            acc[x][0] = fmaf(v3, wb[dx].z, fmaf(v2, wb[dx].x, fmaf(v1, wa[dx].z, fmaf(v0, wa[dx].x, acc[x][0]))));
            acc[x][1] = fmaf(v3, wb[dx].w, fmaf(v2, wb[dx].y, fmaf(v1, wa[dx].w, fmaf(v0, wa[dx].y, acc[x][1]))));
          }
        }
      }
      // add the eight lanes' sums; lane r is left with node r of the line
#pragma unroll
      for (int h = 4; h > 0; h >>= 1) {
        const bool up = r & h;
#pragma unroll
        for (int i = 0; i < h; ++i)
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const float give = up ? acc[i][c] : acc[i + h][c], keep = up ? acc[i + h][c] : acc[i][c];
            acc[i][c] = keep + __shfl_xor_sync(0xffffffffu, give, h);
          }
      }
      if (l < nl && r < N1) {
        const long long o = nb0 + l * N1 + r;
        const float2 v = make_float2(acc[0][0] + b30, acc[0][1] + b31);
        if (vec) {
          ((float2*)out)[o] = v;
        } else {
          out[2 * o] = v.x;
          out[2 * o + 1] = v.y;
        }
      }
    }
    if (a1_out) {
      for (int i = tid; i < np * 4; i += NT) {
        const int n = i >> 2, c = i & 3;
        const int q = swz(group_index<N1>(n), 8 * c);
        ((uint4*)(a1_out + (nb0 + n) * NN_H))[c] = *(const uint4*)(sA1 + q);
        ((uint4*)(a2_out + (nb0 + n) * NN_H))[c] = *(const uint4*)(sA2 + q);
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// backward: per-block partial gradients, reduced in a fixed order afterwards
//
// One block per SM, 16 warps. All four weight contractions are matrix products
// on the tensor cores (mma.sync BF16, FP32 accumulate):
//   dW2[t] (ci x co)  += a1[n + t]^T g_a2[n]           K = nodes
//   g_a1[n]           = sum_t g_a2[n - t] W2[t]^T      K = channels
//   dW3[t] (ci x co)  += a2[n]^T g3[n - t]             K = nodes
//   dW1[t] (co x ci)  += g_a1[n]^T in[n + t]           K = nodes
// The last two have an FP32 operand (g3, in) with two channels: each value is
// split exactly into three BF16 numbers (24 bits), so the two channels fill six
// of the eight columns of one MMA tile and the products are those of the FP32
// values; an element's sums are added up and joined to a compensated running sum,
// and so are the blocks' partials (the error against float64 sums of the same
// operands stays below that of the FP32 chains before).
// In SIMT form these two took 885 k products per element at two shared-memory
// loads each, most of the kernel's time. Shared-memory activations are swizzled
// as in the forward kernel (unswizzled rows put an ldmatrix phase on four banks),
// W2 stays in shared memory, and operand tiles are loaded once for all taps of a
// warp. g_a2 (FP32 weights and inputs, K = 54) stays on the FP32 pipe, two channels
// of a line per thread. Tap offsets are outside the loops, a tile's second half is
// 32 bytes off by an exclusive or, and all operand loads stand before the products:
// address arithmetic and load latency, not the MMAs, set the time of the tile loops.
// Measured (GB300, 16384 elements, p = 7): 28.8 -> 5.9 ms (7.1 with addresses worked
// out at each load and g_a2 by nodes); cycles per element now: loads 7 k, dW3 13 k,
// g_a2 22 k, dW2 28 k, g_a1 24 k, dW1 18 k. 2000 elements at p = 6 6.7 -> 0.82 ms.
// Elements with few nodes go through in groups (p = 1: up to 12), since one of them
// fills neither the warps nor an MMA row tile: 2000 elements at p = 1 0.173 -> 0.090 ms,
// 500 at p = 4 0.588 -> 0.130 ms. What is slower: p = 1 with at most 152 elements, by 1 to
// 5 % of a call (49.6 -> 51.7 us at 8: staging W2).
// ---------------------------------------------------------------------------
constexpr int NN_BWD_THREADS = 512;

__device__ __forceinline__ void ldsm_x2_t(unsigned addr, unsigned& r0, unsigned& r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}

// x = hi + mid + lo exactly (8 bits each, truncated); what is not finite stays in hi
__device__ __forceinline__ void split3(float x, __nv_bfloat16* o) {
  const unsigned b = __float_as_uint(x);
  const bool fin = (b & 0x7f800000u) != 0x7f800000u;
  const float hi = fin ? __uint_as_float(b & 0xffff0000u) : x;
  const float r1 = fin ? x - hi : 0.f;
  const float mid = __uint_as_float(__float_as_uint(r1) & 0xffff0000u);
  o[0] = __float2bfloat16(hi);
  o[1] = __float2bfloat16(mid);
  o[2] = __float2bfloat16(r1 - mid);
}

// s + c <- s + c + v (TwoSum); the carry of an overflow would be NaN and is left out
__device__ __forceinline__ void nn_two_sum(float& s, float& c, float v) {
  const float t = s + v, b = t - s;
  if (isfinite(t)) c += (s - (t - b)) + (v - b);
  s = t;
}

// Adds one element's tile sums (rows g, g + 8; columns = three split parts of two
// channels) to the running sum, compensated (TwoSum): lane c4 keeps row g + 8 (c4 >> 1), channel c4 & 1.
__device__ __forceinline__ void join3(const float* d, int c4, float& run, float& car) {
  float x[4];
  // lane c4's share of the quad's sums x, added up; x[c4] is this lane's
  auto quad = [&]() {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      x[k] += __shfl_xor_sync(0xffffffffu, x[k], 1);
      x[k] += __shfl_xor_sync(0xffffffffu, x[k], 2);
    }
    return c4 == 0 ? x[0] : c4 == 1 ? x[1] : c4 == 2 ? x[2] : x[3];
  };
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float p = d[2 * h] + d[2 * h + 1];
    x[2 * h] = c4 == 0 ? p : (c4 == 1 ? d[2 * h] : 0.f);
    x[2 * h + 1] = c4 == 2 ? p : (c4 == 1 ? d[2 * h + 1] : 0.f);
  }
  float v = quad();
  if (__any_sync(0xffffffffu, !isfinite(v))) {
    // an overflowed activation gradient times a remainder part that is zero is
    // NaN: what is not finite is the leading part's sum
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      x[2 * h] = c4 == 0 ? d[2 * h] : 0.f;
      x[2 * h + 1] = c4 == 1 ? d[2 * h + 1] : 0.f;
    }
    const float hi = quad();
    if (!isfinite(v)) v = hi;
  }
  nn_two_sum(run, car, v);
}

// per-tap contraction over the nodes of the element with split columns:
// acc[a] (32 rows x 8 columns) = sum_n act[n]^T col[n + sgn off(tap a)] for this
// warp's taps, joined to run[a][m] every JOIN node tiles. The tensor core rounds
// its accumulator toward zero: dW1 is 4.5e-7 off its float64 sums at 16384 elements
// with one chain over the element (JOIN 32), 2.0e-7 with 16, 1.1e-7 with 8 (0.4 ms
// slower); the FP32 chains before were 4.4e-7 off. dW3: 0.4e-7, 2.9e-7.
template <int N1, int JOIN>
__device__ __forceinline__ void split_grad(const __nv_bfloat16* act, const __nv_bfloat16* col, int sgn, int np,
                                           int warp, int lane, float (*run)[2], float (*car)[2]) {
  constexpr int NW = NN_BWD_THREADS / 32;
  constexpr bool FULL = NNCfg<N1>::NPE % 16 == 0;  // no row tile reaches past the nodes
  const int MT = (np + 15) / 16;
  const int j = lane >> 3, r = lane & 7, c4 = lane & 3;
  const unsigned ab = smem_u32(act), cb = smem_u32(col);
  const bool two = warp + NW < 27;  // this warp's taps: warp, warp + NW
  int off[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) off[a] = sgn * 16 * tap_offset<N1>(a == 0 || two ? warp + NW * a : warp);
#pragma unroll 1
  for (int k0 = 0; k0 < MT; k0 += JOIN) {
    const int k1 = k0 + JOIN < MT ? k0 + JOIN : MT;
    float acc[2][2][4];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][m][c] = 0.f;
#pragma unroll 2
    for (int kt = k0; kt < k1; ++kt) {
      const int na = kt * 16 + r + 8 * (j >> 1), nb = kt * 16 + (lane & 15);
      const bool okb = FULL || nb < np;
      const int pA = FULL || na < np ? group_index<N1>(na) : 0;
      const unsigned bb = cb + 16 * (okb ? group_index<N1>(nb) : 0);
      unsigned A[2][4], b[2][2];  // all loads before the first product
      ldsm_x4_t(row_addr(ab, pA, j & 1), A[0][0], A[0][1], A[0][2], A[0][3]);
      ldsm_x4_t(row_addr2(ab, pA, j & 1), A[1][0], A[1][1], A[1][2], A[1][3]);
#pragma unroll
      for (int a = 0; a < 2; ++a) ldsm_x2_t(bb + (okb ? off[a] : 0), b[a][0], b[a][1]);
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int m = 0; m < 2; ++m) mma16816(acc[a][m], A[m][0], A[m][1], A[m][2], A[m][3], b[a][0], b[a][1]);
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int m = 0; m < 2; ++m)
        if (a == 0 || two) join3(acc[a][m], c4, run[a][m], car[a][m]);
  }
}

template <int N1>
__global__ void __launch_bounds__(NN_BWD_THREADS, 1)
    k_nn_backward(const float* __restrict__ prm, const __nv_bfloat16* __restrict__ W2o, const float* __restrict__ in,
                  const __nv_bfloat16* __restrict__ a1g, const __nv_bfloat16* __restrict__ a2g,
                  const float* __restrict__ gout, float* __restrict__ part, long long ne, int ng, int vec) {
  using C = NNCfg<N1>;
  using F = FwdCfg<N1>;
  constexpr int P3 = C::P3 * C::GROUP, P = C::P, NT = NN_BWD_THREADS, NW = NT / 32, LPE = N1 * N1;
  extern __shared__ __align__(16) unsigned char smem[];
  // sA1 holds a1 until the layer-2 weight gradient is done, then g_a1 (masked)
  __nv_bfloat16* sA1 = (__nv_bfloat16*)smem;                           // [P3][32] swizzled
  __nv_bfloat16* sA2 = sA1 + P3 * NN_H;                                 // [P3][32] swizzled -> g_a2 (masked)
  __nv_bfloat16* sGs = sA2 + P3 * NN_H;                                 // [P3][8] g3 split
  __nv_bfloat16* sIs = sGs + P3 * 8;                                    // [P3][8] in split
  __nv_bfloat16* sW2 = sIs + P3 * 8;                                    // [27 * 32 ci][32 co] swizzled
  float* sW3 = (float*)(sW2 + 27 * 32 * 32);                           // [27][32][2]
  float* sred = sW3 + 1728;                                            // [NW][32]
  float2* sG3 = (float2*)(sred + NW * 32);                             // [GROUP][P][P][.], rows as in FwdCfg
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the borders stay zero; only the rows of the elements that this launch groups are used
  const int rows = C::P3 * ng;
  for (int i = tid; i < rows * NN_H / 8; i += NT) ((uint4*)sA1)[i] = ((uint4*)sA2)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < rows; i += NT) ((uint4*)sGs)[i] = ((uint4*)sIs)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < ng * F::IS; i += NT) sG3[i] = make_float2(0.f, 0.f);
  for (int i = tid; i < 1728; i += NT) sW3[i] = prm[NN_OW3 + i];
#pragma unroll
  for (int k = 0; k < (27 * 32 * 4 + NT - 1) / NT; ++k) {  // every load ahead of the first store
    const int i = tid + k * NT;
    if (i < 27 * 32 * 4) *(uint4*)(sW2 + swz_w2(i >> 2, (i & 3) * 8)) = __ldg((const uint4*)W2o + i);
  }
  // dW2 accumulators: warp owns taps warp, warp + 16 (< 27); per tap 32 (ci) x 32 (co) = 2 x 4 mma tiles
  float accW[2][2][4][4], run1[2][2], run3[2][2], car1[2][2], car3[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      run1[a][m] = run3[a][m] = car1[a][m] = car3[a][m] = 0.f;
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int c = 0; c < 4; ++c) accW[a][m][n][c] = 0.f;
    }
  float db1 = 0.f, db2 = 0.f, db3 = 0.f;  // of thread (channel) < 32, < 32, < 2
  __syncthreads();
  const int j = lane >> 3, r = lane & 7, g = lane >> 2, c4 = lane & 3;
  // sum over the nodes of a masked gradient's channels: 16 partial sums per channel, joined by join_bias
  auto bias_part = [&](const __nv_bfloat16* A, int np) {
    float acc = 0.f;
    for (int n = warp; n < np; n += NW) acc += __bfloat162float(A[swz(group_index<N1>(n), lane)]);
    sred[warp * 32 + lane] = acc;
  };
  auto g3_index = [](int n) {
    const int l = n / N1;
    return l / LPE * F::IS + (l / N1 % N1 + 1) * F::ZS + (l % N1 + 1) * F::YS + n % N1 + 1;
  };
  auto bias_join = [&](float& db) {
    if (tid < 32) {
      float acc = 0.f;
#pragma unroll
      for (int w = 0; w < NW; ++w) acc += sred[w * 32 + tid];
      db += acc;
    }
  };
  for (long long e0 = (long long)blockIdx.x * ng; e0 < ne; e0 += (long long)gridDim.x * ng) {
    const long long nb0 = e0 * C::NPE;  // first node of the pass; np nodes
    const int np = (int)(ne - e0 < ng ? ne - e0 : ng) * C::NPE, MT = (np + 15) / 16;
    for (int i = tid; i < np; i += NT) {
      const int p = group_index<N1>(i);
      const float2 x = load_pair(in, nb0 + i, vec), y = load_pair(gout, nb0 + i, vec);
      sG3[g3_index(i)] = y;
      split3(x.x, sIs + 8 * p);
      split3(x.y, sIs + 8 * p + 3);
      split3(y.x, sGs + 8 * p);
      split3(y.y, sGs + 8 * p + 3);
    }
    for (int i = tid; i < np * 4; i += NT) {
      const int n = i >> 2, c = i & 3;
      const int q = swz(group_index<N1>(n), 8 * c);
      *(uint4*)(sA1 + q) = ((const uint4*)(a1g + (nb0 + n) * NN_H))[c];
      *(uint4*)(sA2 + q) = ((const uint4*)(a2g + (nb0 + n) * NN_H))[c];
    }
    __syncthreads();
    // layer 3 weights and bias
    split_grad<N1, 32>(sA2, sGs, -1, np, warp, lane, run3, car3);
    {
      float x = 0.f, y = 0.f;
      for (int i = tid; i < np; i += NT) {
        const float2 v = sG3[g3_index(i)];
        x += v.x;
        y += v.y;
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, d);
        y += __shfl_xor_sync(0xffffffffu, y, d);
      }
      if (lane == 0) {
        sred[warp * 32] = x;
        sred[warp * 32 + 1] = y;
      }
    }
    __syncthreads();
    if (tid < 2) {
      float acc = 0.f;
#pragma unroll
      for (int w = 0; w < NW; ++w) acc += sred[w * 32 + tid];
      db3 += acc;
    }
    // g_a2[n][ci] = (sum_t sum_co W3[t][ci][co] g3[n - t][co]) * (a2[n][ci] > 0), in place of a2:
    // thread = line along x and two channels (mostly the same for a warp: weights are broadcast reads)
    const int nl = np / N1;
    for (int w = tid; w < nl * 16; w += NT) {
      const int cg = w / nl * 2, l = w % nl;
      const int y = l % N1, z = l / N1 % N1;
      const float2* src = sG3 + l / LPE * F::IS + (z + 2) * F::ZS + (y + 2) * F::YS;
      float acc[N1][2];
#pragma unroll
      for (int i = 0; i < N1; ++i) acc[i][0] = acc[i][1] = 0.f;
#pragma unroll 1
      for (int d = 0; d < 9; ++d) {
        const float2* row = src - d / 3 * F::ZS - d % 3 * F::YS;
        float2 v[P];
#pragma unroll
        for (int i = 0; i < P; ++i) v[i] = row[i];
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          const float4 wt = *(const float4*)(sW3 + (3 * d + dx) * 64 + cg * 2);
#pragma unroll
          for (int i = 0; i < N1; ++i) {
            const float g0 = v[i + 2 - dx].x, g1 = v[i + 2 - dx].y;
            acc[i][0] += wt.x * g0 + wt.y * g1;
            acc[i][1] += wt.z * g0 + wt.w * g1;
          }
        }
      }
      const int p0 = l / LPE * C::P3 + (z + 1) * P * P + (y + 1) * P + 1;
#pragma unroll
      for (int i = 0; i < N1; ++i) {
        __nv_bfloat162* dst = (__nv_bfloat162*)(sA2 + swz(p0 + i, cg));
        const float2 v = __bfloat1622float2(*dst);
        *dst = __floats2bfloat162_rn(v.x > 0.f ? acc[i][0] : 0.f, v.y > 0.f ? acc[i][1] : 0.f);
      }
    }
    __syncthreads();
    bias_part(sA2, np);
    // layer 2 weights: dW2[t] (ci x co) += sum_n a1[n + t][ci] g_a2[n][co]
    {
      constexpr bool FULL = C::NPE % 16 == 0;
      const unsigned b1 = smem_u32(sA1), b2 = smem_u32(sA2);
      const bool two = warp + NW < 27;
      int off[2];
#pragma unroll
      for (int a = 0; a < 2; ++a) off[a] = tap_offset<N1>(a == 0 || two ? warp + NW * a : warp);
#pragma unroll 1
      for (int kt = 0; kt < MT; ++kt) {
        // k = 16 nodes of tile kt; lane row address: node kt*16 + r + 8*(j>>1)
        const int node = kt * 16 + r + 8 * (j >> 1);
        const bool ok = FULL || node < np;
        const int p = ok ? group_index<N1>(node) : 0;
        unsigned b[2][4];
        ldsm_x4_t(row_addr(b2, p, j & 1), b[0][0], b[0][1], b[0][2], b[0][3]);
        ldsm_x4_t(row_addr2(b2, p, j & 1), b[1][0], b[1][1], b[1][2], b[1][3]);
        unsigned A[2][2][4];  // all loads before the first product
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          const int pA = ok ? p + off[a] : 0;
          ldsm_x4_t(row_addr(b1, pA, j & 1), A[a][0][0], A[a][0][1], A[a][0][2], A[a][0][3]);
          ldsm_x4_t(row_addr2(b1, pA, j & 1), A[a][1][0], A[a][1][1], A[a][1][2], A[a][1][3]);
        }
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          if (a == 1 && !two) continue;
#pragma unroll
          for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int nh = 0; nh < 2; ++nh) {
              mma16816(accW[a][m][2 * nh], A[a][m][0], A[a][m][1], A[a][m][2], A[a][m][3], b[nh][0], b[nh][2]);
              mma16816(accW[a][m][2 * nh + 1], A[a][m][0], A[a][m][1], A[a][m][2], A[a][m][3], b[nh][1], b[nh][3]);
            }
        }
      }
    }
    __syncthreads();
    bias_join(db2);
    // layer 2 input gradient: g_a1[n][ci] = mask * sum_t sum_co g_a2[n - t][co] W2[t][ci][co], written over a1
    // (each lane reads the mask of exactly the entries it writes); two node tiles per warp share the W2 tiles
    for (int mt0 = warp; mt0 < MT; mt0 += 2 * NW) {
      float acc[2][4][4];
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.f;
      int prow[2];
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const int node = (mt0 + NW * a) * 16 + r + 8 * (j & 1);
        prow[a] = node < np ? group_index<N1>(node) : -1;
      }
      // W2 tiles: matrices j = (kh, 8-column half) of the 8 rows ci of column tile nt
      unsigned wa = smem_u32(sW2 + swz_w2(r, 8 * j));
      const unsigned ab = smem_u32(sA2);
#pragma unroll 1
      for (int d = 0; d < 9; ++d) {
        const int od = (d / 3 - 1) * P * P + (d % 3 - 1) * P - 1;
#pragma unroll 1
        for (int dx = 0; dx < 3; ++dx, wa += 2048) {
          unsigned w2[4][4];
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) ldsm_x4(wa + nt * 512, w2[nt][0], w2[nt][1], w2[nt][2], w2[nt][3]);
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            if (mt0 + NW * a >= MT) continue;
            const int q = prow[a] >= 0 ? prow[a] - od - dx : 0;
            unsigned A[2][4];
            ldsm_x4(row_addr(ab, q, j >> 1), A[0][0], A[0][1], A[0][2], A[0][3]);
            ldsm_x4(row_addr2(ab, q, j >> 1), A[1][0], A[1][1], A[1][2], A[1][3]);
#pragma unroll
            for (int kh = 0; kh < 2; ++kh)
#pragma unroll
              for (int nt = 0; nt < 4; ++nt)
                mma16816(acc[a][nt], A[kh][0], A[kh][1], A[kh][2], A[kh][3], w2[nt][2 * kh], w2[nt][2 * kh + 1]);
          }
        }
      }
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int nn = (mt0 + NW * a) * 16 + g + 8 * h;
          if (nn >= np) continue;
          const int p = group_index<N1>(nn);
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            __nv_bfloat162* dst = (__nv_bfloat162*)(sA1 + swz(p, nt * 8 + 2 * c4));
            const float2 a1v = __bfloat1622float2(*dst);
            *dst = __floats2bfloat162_rn(a1v.x > 0.f ? acc[a][nt][2 * h] : 0.f,
                                         a1v.y > 0.f ? acc[a][nt][2 * h + 1] : 0.f);
          }
        }
    }
    __syncthreads();
    // layer 1 weights and bias
    split_grad<N1, 16>(sA1, sIs, 1, np, warp, lane, run1, car1);
    bias_part(sA1, np);
    __syncthreads();
    bias_join(db1);
    // a1 and a2 were overwritten by their gradients at interior nodes only;
    // the zero borders stay, the interiors are reloaded for the next element
  }
  // write this block's partial gradients in parameter order
  float* pb = part + (long long)blockIdx.x * NN_NPARAM;
  if (tid < 32) {
    pb[NN_OB1 + tid] = db1;
    pb[NN_OB2 + tid] = db2;
  }
  if (tid < 2) pb[NN_OB3 + tid] = db3;
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int t = warp + NW * a;
    if (t >= 27) continue;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const int row = m * 16 + g + 8 * (c4 >> 1), ch = c4 & 1;
      pb[NN_OW3 + t * 64 + row * 2 + ch] = run3[a][m] + car3[a][m];
      pb[NN_OW1 + t * 64 + ch * 32 + row] = run1[a][m] + car1[a][m];
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int ci = m * 16 + g + 8 * h, co = n * 8 + 2 * c4;
          pb[NN_OW2 + (t * 32 + ci) * 32 + co] = accW[a][m][n][2 * h];
          pb[NN_OW2 + (t * 32 + ci) * 32 + co + 1] = accW[a][m][n][2 * h + 1];
        }
    }
  }
}

// The blocks' partials added up, compensated: NN_RSL threads take a stretch of the
// blocks each, the stretches are joined in order. Bound by the 4 bytes per partial
// (19 MB at 152 blocks). In FP64 the additions and conversions took 26 us there (the
// FP64 pipe), one thread per parameter 8.9 us (too few bytes in flight).
constexpr int NN_RSL = 8;
__global__ void __launch_bounds__(32 * NN_RSL) k_nn_reduce(const float* __restrict__ part, int nblk,
                                                           float* __restrict__ grad) {
  __shared__ float sh[NN_RSL][2][32];
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  const int per = (nblk + NN_RSL - 1) / NN_RSL, b0 = sl * per, b1 = min(nblk, b0 + per);
  float sum = 0.f, car = 0.f;
  if (i < NN_NPARAM) {
#pragma unroll 4
    for (int b = b0; b < b1; ++b) nn_two_sum(sum, car, part[(long long)b * NN_NPARAM + i]);
  }
  sh[sl][0][lane] = sum;
  sh[sl][1][lane] = car;
  __syncthreads();
  if (sl > 0 || i >= NN_NPARAM) return;
#pragma unroll
  for (int k = 1; k < NN_RSL; ++k) {
    nn_two_sum(sum, car, sh[k][0][lane]);
    car += sh[k][1][lane];
  }
  grad[i] = sum + car;
}

// BF16 copies of W2 in both layouts
__global__ void k_nn_prep(const float* __restrict__ prm, __nv_bfloat16* __restrict__ W2t,
                          __nv_bfloat16* __restrict__ W2o) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 27 * 32 * 32) return;
  const int t = i / 1024, ci = (i / 32) % 32, co = i % 32;
  const __nv_bfloat16 v = __float2bfloat16(prm[NN_OW2 + i]);
  W2o[i] = v;
  W2t[(t * 32 + co) * 32 + ci] = v;
}

__global__ void k_nn_adam(float* __restrict__ prm, const float* __restrict__ grad, float* __restrict__ m,
                          float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NN_NPARAM) return;
  const float gi = grad[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  prm[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

template <int N1>
static constexpr size_t bwd_smem() {
  using C = NNCfg<N1>;
  constexpr size_t sm = sizeof(__nv_bfloat16) * (2 * C::P3 * C::GROUP * (NN_H + 8) + 27 * 32 * 32) +
                        sizeof(float2) * C::GROUP * FwdCfg<N1>::IS + sizeof(float) * (1728 + NN_BWD_THREADS);
  static_assert(sm <= 227 * 1024, "shared memory of a block");
  return sm;
}

static int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// resident blocks of a kernel per SM at its dynamic shared memory (at least 1)
template <typename K>
static int blocks_per_sm(K kern, size_t smem, int threads = 256) {
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, threads, smem) != cudaSuccess || b < 1) b = 1;
  return b;
}

// elements at once: no more than the share of each of blocks blocks
template <int N1>
static int nn_group(long long ne, long long blocks) {
  const long long per = (ne + blocks - 1) / blocks;
  return (int)(per < 1 ? 1 : (per < NNCfg<N1>::GROUP ? per : NNCfg<N1>::GROUP));
}

template <int N1>
static cudaError_t nn_fwd_n1(const float* prm, const __nv_bfloat16* W2t, const float* in, float* out,
                             __nv_bfloat16* a1, __nv_bfloat16* a2, long long ne, cudaStream_t s) {
  constexpr size_t sm = FwdCfg<N1>::SMEM;
  static_assert(sm <= 227 * 1024, "shared memory of a block");
  static int bps = 0;
  if (!bps) {
    cudaError_t e = cudaFuncSetAttribute(k_nn_forward<N1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    bps = blocks_per_sm(k_nn_forward<N1>, sm, NN_FWD_THREADS);
  }
  if (ne < 1) return cudaSuccess;
  const long long cap = (long long)sm_count() * bps;
  const int ng = nn_group<N1>(ne, cap);
  const long long grid = (ne + ng - 1) / ng;
  count_launch();
  k_nn_forward<N1><<<(unsigned)(grid < cap ? grid : cap), NN_FWD_THREADS, sm, s>>>(prm, W2t, in, out, a1, a2, ne, ng,
                                                                                      pairs_aligned(in, out));
  return cudaGetLastError();
}

template <int N1>
static int nn_bwd_blocks(long long ne) {
  static int bps = 0;
  if (!bps) {
    const size_t sm = bwd_smem<N1>();
    if (cudaFuncSetAttribute(k_nn_backward<N1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
      return 0;
    bps = blocks_per_sm(k_nn_backward<N1>, sm, NN_BWD_THREADS);
  }
  const long long cap = (long long)sm_count() * bps;
  return (int)(ne < cap ? (ne < 1 ? 1 : ne) : cap);
}

template <int N1>
static cudaError_t nn_bwd_n1(const float* prm, const __nv_bfloat16* W2o, const float* in, const __nv_bfloat16* a1,
                             const __nv_bfloat16* a2, const float* gout, float* part, int nblk, long long ne,
                             cudaStream_t s) {
  count_launch();
  k_nn_backward<N1><<<nblk, NN_BWD_THREADS, bwd_smem<N1>(), s>>>(prm, W2o, in, a1, a2, gout, part, ne,
                                                                    nn_group<N1>(ne, nblk), pairs_aligned(in, gout));
  return cudaGetLastError();
}

cudaError_t nn_prep(const float* prm, void* W2t, void* W2o, cudaStream_t s) {
  count_launch();
  k_nn_prep<<<(27 * 1024 + 255) / 256, 256, 0, s>>>(prm, (__nv_bfloat16*)W2t, (__nv_bfloat16*)W2o);
  return cudaGetLastError();
}

cudaError_t nn_forward(int n1, const float* prm, const void* W2tv, const float* in, float* out, void* a1v, void* a2v,
                       long long ne, cudaStream_t s) {
  const __nv_bfloat16* W2t = (const __nv_bfloat16*)W2tv;
  __nv_bfloat16* a1 = (__nv_bfloat16*)a1v;
  __nv_bfloat16* a2 = (__nv_bfloat16*)a2v;
  switch (n1) {
    case 2: return nn_fwd_n1<2>(prm, W2t, in, out, a1, a2, ne, s);
    case 3: return nn_fwd_n1<3>(prm, W2t, in, out, a1, a2, ne, s);
    case 4: return nn_fwd_n1<4>(prm, W2t, in, out, a1, a2, ne, s);
    case 5: return nn_fwd_n1<5>(prm, W2t, in, out, a1, a2, ne, s);
    case 6: return nn_fwd_n1<6>(prm, W2t, in, out, a1, a2, ne, s);
    case 7: return nn_fwd_n1<7>(prm, W2t, in, out, a1, a2, ne, s);
    case 8: return nn_fwd_n1<8>(prm, W2t, in, out, a1, a2, ne, s);
    default: return cudaErrorInvalidValue;
  }
}

// blocks (and gradient partials) of the backward kernel for ne elements; 0 on error
int nn_backward_blocks(int n1, long long ne) {
  switch (n1) {
    case 2: return nn_bwd_blocks<2>(ne);
    case 3: return nn_bwd_blocks<3>(ne);
    case 4: return nn_bwd_blocks<4>(ne);
    case 5: return nn_bwd_blocks<5>(ne);
    case 6: return nn_bwd_blocks<6>(ne);
    case 7: return nn_bwd_blocks<7>(ne);
    case 8: return nn_bwd_blocks<8>(ne);
    default: return 0;
  }
}

cudaError_t nn_backward(int n1, const float* prm, const void* W2ov, const float* in, const void* a1v, const void* a2v,
                        const float* gout, float* part, float* grad, long long ne, cudaStream_t s) {
  const __nv_bfloat16* W2o = (const __nv_bfloat16*)W2ov;
  const __nv_bfloat16* a1 = (const __nv_bfloat16*)a1v;
  const __nv_bfloat16* a2 = (const __nv_bfloat16*)a2v;
  const int nblk = nn_backward_blocks(n1, ne);
  if (nblk < 1) return cudaErrorInvalidValue;
  cudaError_t e;
  switch (n1) {
    case 2: e = nn_bwd_n1<2>(prm, W2o, in, a1, a2, gout, part, nblk, ne, s); break;
    case 3: e = nn_bwd_n1<3>(prm, W2o, in, a1, a2, gout, part, nblk, ne, s); break;
    case 4: e = nn_bwd_n1<4>(prm, W2o, in, a1, a2, gout, part, nblk, ne, s); break;
    case 5: e = nn_bwd_n1<5>(prm, W2o, in, a1, a2, gout, part, nblk, ne, s); break;
    case 6: e = nn_bwd_n1<6>(prm, W2o, in, a1, a2, gout, part, nblk, ne, s); break;
    case 7: e = nn_bwd_n1<7>(prm, W2o, in, a1, a2, gout, part, nblk, ne, s); break;
    case 8: e = nn_bwd_n1<8>(prm, W2o, in, a1, a2, gout, part, nblk, ne, s); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  count_launch();
  k_nn_reduce<<<(NN_NPARAM + 31) / 32, 32 * NN_RSL, 0, s>>>(part, nblk, grad);
  return cudaGetLastError();
}

cudaError_t nn_adam(float* prm, const float* grad, float* m, float* v, float lr, float b1, float b2, float eps,
                    int step, cudaStream_t s) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  count_launch();
  k_nn_adam<<<(NN_NPARAM + 255) / 256, 256, 0, s>>>(prm, grad, m, v, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

}  // namespace dg
