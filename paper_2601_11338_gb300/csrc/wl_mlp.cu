// Learned warm start for the walk-degree solve (the paper has no learned
// part; this network only supplies the CG starting guess of D_f = phi 1).
//
// Node features (all from the graph alone, FP64, stored FP32):
//   f0 = log(1 + d_i), f1 = log(1 + (A d)_i), f2 = log(1 + t_i),
//   f3 = log(1 + (A d - d)_i)
// with t_i the triangles through i (degree-ordered intersection) and
// A d - d the nonbacktracking 2-walk count (p_2(A) 1 with p_2 = A^2 - D).
//
// The guess is x0 = x_an * exp(y): x_an = 1 + B 1 + B^2 1 is the two-term
// Neumann series of D_f = sum_k B^k 1, B = (alpha A - alpha^2 mu D) / a,
// a = 1 - mu^2 alpha^2 (Sec. 4.2, the resolvent's series), and y the output
// of a 4 -> 64 -> 64 -> 1 tanh perceptron on the standardised features,
// trained on log(D_f / x_an).
//
// Parameter vector (floats): mean[4], std[4], W1[64][4], b1[64],
// W2[64][64], b2[64], W3[64], b3 (4553 values).
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "wl.h"
#include "wl_df.cuh"
#include "wl_host.h"

namespace wl {

constexpr int kH = 64;
constexpr int kIn = 4;
constexpr int kOffMean = 0, kOffStd = 4, kOffW1 = 8, kOffB1 = kOffW1 + kH * kIn, kOffW2 = kOffB1 + kH,
              kOffB2 = kOffW2 + kH * kH, kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH;
constexpr int kParams = kOffB3 + 1;        // 4553
constexpr int kTrain = kParams - kOffW1;   // 4545 trainable values (after the standardisation)
constexpr int kRowsCTA = 128;              // rows per tile of the network kernels

// ------------------------------------------------------------------ features
// Row passes of the features: a warp takes a row of up to kFeatLong entries,
// the CTA's eight warps a longer one together. The rows of a CTA lie a grid
// apart, so that the hubs, which the relabelling puts first, spread over the
// chip (R-MAT scale 18: 64 and 80 us for the two passes; with one warp per row the
// longest row held each of them: 313 and 314 us).
constexpr int kFeatLong = 512;
constexpr int kFeatBlock = 256;

// rank order for the triangle orientation: (degree, index)
__device__ __forceinline__ bool ranks_above(int dj, int j, int di, int i) { return dj > di || (dj == di && j > i); }

// calls f(row, beg, end, lane, lanes, whole) for every row: by a warp (lanes =
// 32), or for a long row by the whole CTA (lanes = kFeatBlock, whole = true)
template <typename F>
__device__ __forceinline__ void feat_rows(const int32_t* __restrict__ rp, int64_t n, F f) {
  constexpr int NW = kFeatBlock / 32;
  __shared__ int s_long[NW];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t base = blockIdx.x; base < n; base += (int64_t)gridDim.x * NW) {
    const int64_t i = base + (int64_t)w * gridDim.x;
    int is_long = 0;
    if (i < n) {
      const int beg = rp[i], end = rp[i + 1];
      is_long = end - beg > kFeatLong;
      if (!is_long) f(i, beg, end, lane, 32, false);
    }
    if (lane == 0) s_long[w] = is_long;
    if (__syncthreads_or(is_long)) {
      for (int q = 0; q < NW; ++q) {
        if (!s_long[q]) continue;
        const int64_t r = base + (int64_t)q * gridDim.x;
        f(r, rp[r], rp[r + 1], (int)threadIdx.x, kFeatBlock, true);
      }
    }
    __syncthreads();
  }
}

// (A d)_i and, for the triangle orientation (OUT), the number of neighbours
// of higher rank; nodes with more than kTriWarpDeg of them go to `big`
constexpr int kTriWarpDeg = 128;

template <bool OUT>
__global__ void __launch_bounds__(kFeatBlock) k_feat_ad(const int32_t* __restrict__ rp,
                                                        const int32_t* __restrict__ col, int64_t n,
                                                        double* __restrict__ ad, int64_t* __restrict__ outdeg,
                                                        int32_t* __restrict__ big, int* __restrict__ nbig) {
  __shared__ long long s_sum;
  __shared__ int s_cnt;
  feat_rows(rp, n, [&](int64_t i, int beg, int end, int lane, int lanes, bool whole) {
    const int di = end - beg;
    long long s = 0;  // exact: at most 2^31 neighbours of degree below 2^31
    int c = 0;
#pragma unroll 4
    for (int e = beg + lane; e < end; e += lanes) {
      const int j = __ldg(col + e);
      const int dj = __ldg(rp + j + 1) - __ldg(rp + j);
      s += dj;
      if (OUT) c += ranks_above(dj, j, di, (int)i) ? 1 : 0;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, off);
      if (OUT) c += __shfl_xor_sync(0xffffffffu, c, off);
    }
    if (whole) {  // integer sums: the order does not matter
      __syncthreads();
      if (threadIdx.x == 0) {
        s_sum = 0;
        s_cnt = 0;
      }
      __syncthreads();
      if ((threadIdx.x & 31) == 0) {
        atomicAdd((unsigned long long*)&s_sum, (unsigned long long)s);
        if (OUT) atomicAdd(&s_cnt, c);
      }
      __syncthreads();
      s = s_sum;
      c = s_cnt;
    }
    if (lane == 0) {
      ad[i] = (double)s;
      if (OUT) {
        outdeg[i] = c;
        if (c > kTriWarpDeg) big[atomicAdd(nbig, 1)] = (int32_t)i;
      }
    }
  });
}

// oriented lists N+(i), in no particular order
__global__ void __launch_bounds__(kFeatBlock) k_feat_orient(const int32_t* __restrict__ rp,
                                                            const int32_t* __restrict__ col, int64_t n,
                                                            const int64_t* __restrict__ orp,
                                                            int32_t* __restrict__ ocol) {
  __shared__ int s_pos;
  feat_rows(rp, n, [&](int64_t i, int beg, int end, int lane, int lanes, bool whole) {
    const int di = end - beg;
    const int64_t o = orp[i];
    const int wl = threadIdx.x & 31;
    if (whole) {
      __syncthreads();
      if (threadIdx.x == 0) s_pos = 0;
      __syncthreads();
    }
    int pos = 0;
    for (int e0 = beg; e0 < end; e0 += lanes) {
      const int e = e0 + lane;
      bool keep = false;
      int j = 0;
      if (e < end) {
        j = __ldg(col + e);
        keep = ranks_above(__ldg(rp + j + 1) - __ldg(rp + j), j, di, (int)i);
      }
      const unsigned m = __ballot_sync(0xffffffffu, keep);
      if (whole) {
        if (wl == 0) pos = atomicAdd(&s_pos, __popc(m));
        pos = __shfl_sync(0xffffffffu, pos, 0);
      }
      if (keep) ocol[o + pos + __popc(m & ((1u << wl) - 1u))] = j;
      if (!whole) pos += __popc(m);
    }
  });
}

// Every triangle once: for each i, N+(i) goes into a hash table in shared
// memory, and the w of every N+(j), j in N+(i), are looked up in it. A hit is
// one triangle (i, j, w): t_w is counted in the table's slot, t_j in a
// register of the warp that walks N+(j), t_i beside it, and the global
// counters see one atomic per node of N+(i) instead of one per triangle. The
// table is at most a quarter full, so a look-up reads 1.2 words on average:
// the pass is bound by shared-memory reads, one for each wedge (i, j, w)
// (6.6e8 on R-MAT scale 18), and not by the dependent global reads of a
// merge or binary search per edge. R-MAT scale 18, 7.6e6 entries: 2.19 ms (eight lanes to a
// list, four lists a warp: 2.98 ms; a
// merge or binary search by one lane per edge, a global atomic per triangle:
// 20.4 ms).
// A warp takes a node of up to kTriWarpDeg out-neighbours, a CTA a longer
// one, in pieces of kTriPiece that fit its table.
constexpr int kTriWarpTab = 4 * kTriWarpDeg;
constexpr int kTriPiece = 1024;
constexpr int kTriTab = 4 * kTriPiece;
constexpr int kTriBlock = 256;
constexpr int kTriTicket = 8;  // nodes a warp takes at a time
constexpr int kTriUnroll = 4;  // look-ups in flight per lane

__device__ __forceinline__ unsigned tri_hash(int key, int shift) { return ((unsigned)key * 0x9E3779B1u) >> shift; }

// slot of key in the table, or -1 (empty slots hold -1; never full)
__device__ __forceinline__ int tri_find(const int* tab, unsigned mask, int shift, int key) {
  unsigned s = tri_hash(key, shift);
  for (;;) {
    const int v = tab[s];
    if (v == key) return (int)s;
    if (v < 0) return -1;
    s = (s + 1) & mask;
  }
}

template <int T, int PIECE, typename Sync>
__device__ __forceinline__ void tri_node(int64_t i, const int64_t* __restrict__ orp, const int32_t* __restrict__ ocol,
                                         unsigned long long* __restrict__ t, int* tab, int* cnt, int tid, Sync sync) {
  constexpr int NW = T / 32;
  const int ib = (int)orp[i];  // at most 2^30 oriented entries
  const int len = (int)(orp[i + 1] - ib);
  if (len < 2) return;
  const int w = tid / 32, lane = tid & 31;
  unsigned long long ti = 0;
  for (int p0 = 0; p0 < len; p0 += PIECE) {
    const int pl = min(PIECE, len - p0);
    const int lg = max(5, 34 - __clz(pl - 1 > 0 ? pl - 1 : 1));  // log2 of the table: 4 x the next power of two
    const int S = 1 << lg, shift = 32 - lg;
    const unsigned mask = (unsigned)S - 1u;
    for (int s = tid; s < S; s += T) {
      tab[s] = -1;
      cnt[s] = 0;
    }
    sync();
    for (int p = tid; p < pl; p += T) {
      const int key = ocol[ib + p0 + p];
      unsigned s = tri_hash(key, shift);
      while (atomicCAS(tab + s, -1, key) != -1) s = (s + 1) & mask;
    }
    sync();
    // 32 members j of N+(i) at a time, their list bounds one per lane; then the
    // warp walks one N+(j) after the other
    for (int q0 = w; q0 < len; q0 += 32 * NW) {
      const int q = q0 + lane * NW;
      int j = 0, jb = 0, je = 0;
      if (q < len) {
        j = __ldg(ocol + ib + q);
        jb = (int)__ldg(orp + j);
        je = (int)__ldg(orp + j + 1);
      }
      const int nj = min(32, (len - q0 + NW - 1) / NW);
      int mine = 0;  // triangles with this lane's j
      for (int u = 0; u < nj; ++u) {
        const int b0 = __shfl_sync(0xffffffffu, jb, u), b1 = __shfl_sync(0xffffffffu, je, u);
        int tj = 0;
        for (int b = b0 + lane; b - lane < b1; b += 32 * kTriUnroll) {
          int key[kTriUnroll];
#pragma unroll
          for (int v = 0; v < kTriUnroll; ++v) key[v] = b + 32 * v < b1 ? __ldg(ocol + b + 32 * v) : -1;
#pragma unroll
          for (int v = 0; v < kTriUnroll; ++v) {
            if (key[v] < 0) continue;
            const int s = tri_find(tab, mask, shift, key[v]);
            if (s >= 0) {
              atomicAdd(cnt + s, 1);
              ++tj;
            }
          }
        }
        tj = __reduce_add_sync(0xffffffffu, tj);
        if (lane == u) mine = tj;
      }
      if (mine) {
        atomicAdd(t + j, (unsigned long long)mine);
        ti += mine;
      }
    }
    sync();
    for (int p = tid; p < pl; p += T) {
      const int key = ocol[ib + p0 + p];
      const int c = cnt[tri_find(tab, mask, shift, key)];
      if (c) atomicAdd(t + key, (unsigned long long)c);
    }
    sync();
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) ti += __shfl_xor_sync(0xffffffffu, ti, off);
  if (lane == 0 && ti) atomicAdd(t + i, ti);
}

__global__ void __launch_bounds__(kTriBlock) k_feat_tri_warp(const int64_t* __restrict__ orp,
                                                             const int32_t* __restrict__ ocol, int64_t n,
                                                             unsigned long long* __restrict__ t,
                                                             unsigned long long* __restrict__ ticket) {
  __shared__ int s_tab[kTriBlock / 32][kTriWarpTab];
  __shared__ int s_cnt[kTriBlock / 32][kTriWarpTab];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (;;) {
    unsigned long long i0 = 0;
    if (lane == 0) i0 = atomicAdd(ticket, (unsigned long long)kTriTicket);
    i0 = __shfl_sync(0xffffffffu, i0, 0);
    if (i0 >= (unsigned long long)n) return;
    const int64_t i1 = min((int64_t)i0 + kTriTicket, n);
    for (int64_t i = (int64_t)i0; i < i1; ++i) {
      if (orp[i + 1] - orp[i] > kTriWarpDeg) continue;
      tri_node<32, kTriWarpDeg>(i, orp, ocol, t, s_tab[w], s_cnt[w], lane, [] { __syncwarp(); });
      __syncwarp();
    }
  }
}

__global__ void __launch_bounds__(kTriBlock) k_feat_tri_cta(const int64_t* __restrict__ orp,
                                                            const int32_t* __restrict__ ocol,
                                                            const int32_t* __restrict__ big,
                                                            const int* __restrict__ nbig,
                                                            unsigned long long* __restrict__ t) {
  __shared__ int s_tab[kTriTab];
  __shared__ int s_cnt[kTriTab];
  const int nb = *nbig;
  for (int b = blockIdx.x; b < nb; b += gridDim.x)
    tri_node<kTriBlock, kTriPiece>(big[b], orp, ocol, t, s_tab, s_cnt, (int)threadIdx.x, [] { __syncthreads(); });
}

// features (FP32) and the analytic guess x_an (FP64), written at position
// perm[i] (perm == NULL: i)
__global__ void k_feat_out(const int32_t* __restrict__ rp, const double* __restrict__ ad,
                           const unsigned long long* __restrict__ t, int64_t n, double alpha, double mu,
                           const int32_t* __restrict__ perm, float* __restrict__ F, double* __restrict__ xan) {
  const double a = 1.0 - mu * mu * alpha * alpha;
  const double c1 = (alpha - alpha * alpha * mu) / a;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double d = (double)(rp[i + 1] - rp[i]);
    const double adi = ad[i];
    const int64_t o = perm ? (int64_t)perm[i] : i;
    if (F) {
      F[o * 4 + 0] = (float)log1p(d);
      F[o * 4 + 1] = (float)log1p(adi);
      F[o * 4 + 2] = (float)log1p((double)t[i]);
      F[o * 4 + 3] = (float)log1p(adi - d);
    }
    if (xan) xan[o] = 1.0 + c1 * d + c1 * (alpha * adi - alpha * alpha * mu * d * d) / a;
  }
}

// ------------------------------------------------------------------ network
// Both network kernels take kRowsCTA rows at a time as small matrix products
// in shared memory (rows x 64 by 64 x 64) with eight rows and four units per
// thread in packed FP32 pairs (fma.rn.f32x2: two IEEE fused multiply-adds an
// instruction), so that a k step costs 16 packed products for three vector
// reads; the FP32 pipe bounds them. FP32 throughout, as the parity tests ask
// (TF32 tensor cores would drop 13 bits).
constexpr int kMlpThreads = 256;
constexpr int kMlpPitch = kRowsCTA + 4;  // unit-major tiles [64][kMlpPitch]: 16-byte rows, distinct banks
constexpr int kWPitch = kH + 4;

typedef unsigned long long f2x;  // two FP32 values, the lower address in the lower half
__device__ __forceinline__ f2x f2_pack(float lo, float hi) {
  f2x r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 f2_unpack(f2x v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2x f2_fma(f2x a, f2x b, f2x c) {
  f2x d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

struct alignas(16) MlpTile {
  float h1[kH * kMlpPitch];   // tanh of layer 1, [unit][row]
  float w2t[kH * kWPitch];    // W2 transposed, [k][j]
  float x[kRowsCTA * kIn];    // standardised inputs
  float head[kOffW2 + 8];     // mean, std, W1, b1
  float b2[kH], w3[kH];
  float b3;
};
static_assert(sizeof(MlpTile) % 16 == 0, "vector access to what follows it");

__device__ __forceinline__ void mlp_load(const float* __restrict__ P, MlpTile& t) {
  for (int i = threadIdx.x; i < kOffW2; i += kMlpThreads) t.head[i] = P[i];
  for (int i = threadIdx.x; i < kH * kH; i += kMlpThreads) t.w2t[(i % kH) * kWPitch + i / kH] = P[kOffW2 + i];
  if (threadIdx.x < kH) {
    t.b2[threadIdx.x] = P[kOffB2 + threadIdx.x];
    t.w3[threadIdx.x] = P[kOffW3 + threadIdx.x];
  }
  if (threadIdx.x == 0) t.b3 = P[kOffB3];
  __syncthreads();
}

// Forward pass of rows [r0, r0 + kRowsCTA) below `rows`: thread (ty, tx) =
// (tid / 16, tid % 16) gets h2 of rows 8 ty .. 8 ty + 7 and units 4 tx .. 4 tx
// + 3. Rows past the end are computed on zero inputs.
__device__ __forceinline__ void mlp_forward(const float* __restrict__ F, int64_t r0, int64_t rows, MlpTile& t,
                                            float (&h2)[8][4]) {
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  {
    // layer 1: two threads per row, 32 units each
    const int rr = tid & (kRowsCTA - 1), half = tid / kRowsCTA;
    float x[kIn] = {0.f, 0.f, 0.f, 0.f};
    if (r0 + rr < rows) {
#pragma unroll
      for (int c = 0; c < kIn; ++c) x[c] = (F[(r0 + rr) * 4 + c] - t.head[kOffMean + c]) / t.head[kOffStd + c];
    }
    if (half == 0)
#pragma unroll
      for (int c = 0; c < kIn; ++c) t.x[rr * kIn + c] = x[c];
#pragma unroll 4
    for (int k = half * (kH / 2); k < (half + 1) * (kH / 2); ++k) {
      float z = t.head[kOffB1 + k];
#pragma unroll
      for (int c = 0; c < kIn; ++c) z = fmaf(t.head[kOffW1 + k * kIn + c], x[c], z);
      t.h1[k * kMlpPitch + rr] = tanhf(z);
    }
  }
  __syncthreads();
  f2x acc[4][4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float b = t.b2[4 * tx + c];
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[p][c] = f2_pack(b, b);
  }
#pragma unroll 4
  for (int k = 0; k < kH; ++k) {
    const ulonglong2 a01 = *reinterpret_cast<const ulonglong2*>(&t.h1[k * kMlpPitch + 8 * ty]);
    const ulonglong2 a23 = *reinterpret_cast<const ulonglong2*>(&t.h1[k * kMlpPitch + 8 * ty + 4]);
    const float4 w = *reinterpret_cast<const float4*>(&t.w2t[k * kWPitch + 4 * tx]);
    const f2x av[4] = {a01.x, a01.y, a23.x, a23.y};
    const f2x wv[4] = {f2_pack(w.x, w.x), f2_pack(w.y, w.y), f2_pack(w.z, w.z), f2_pack(w.w, w.w)};
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[p][c] = f2_fma(av[p], wv[c], acc[p][c]);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const float2 z = f2_unpack(acc[p][c]);
      h2[2 * p][c] = tanhf(z.x);
      h2[2 * p + 1][c] = tanhf(z.y);
    }
}

// h2 into a unit-major tile
__device__ __forceinline__ void mlp_store_h2(const float (&h2)[8][4], float* tile) {
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    float4* o = reinterpret_cast<float4*>(tile + (4 * tx + c) * kMlpPitch + 8 * ty);
    o[0] = make_float4(h2[0][c], h2[1][c], h2[2][c], h2[3][c]);
    o[1] = make_float4(h2[4][c], h2[5][c], h2[6][c], h2[7][c]);
  }
}

// y of one row from the h2 tile, the units in order
__device__ __forceinline__ float mlp_output(const MlpTile& t, const float* tile, int row) {
  float y = t.b3;
#pragma unroll 16
  for (int j = 0; j < kH; ++j) y = fmaf(t.w3[j], tile[j * kMlpPitch + row], y);
  return y;
}

// y (per row) of the perceptron; x0 = exp(y) * xan (xan may be NULL: x0 = y).
// 200003 rows: 57 us (a thread per row reading one weight per product
// from shared memory: 112 us).
__global__ void __launch_bounds__(kMlpThreads, 3) k_mlp_predict(const float* __restrict__ P,
                                                                const float* __restrict__ F, int64_t rows,
                                                                const double* __restrict__ xan,
                                                                double* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MlpTile& t = *reinterpret_cast<MlpTile*>(smem_raw);
  mlp_load(P, t);
  for (int64_t r0 = (int64_t)blockIdx.x * kRowsCTA; r0 < rows; r0 += (int64_t)gridDim.x * kRowsCTA) {
    float h2[8][4];
    mlp_forward(F, r0, rows, t, h2);
    __syncthreads();  // h1 has been read
    mlp_store_h2(h2, t.h1);
    __syncthreads();
    const int64_t r = r0 + threadIdx.x;
    if (threadIdx.x < kRowsCTA && r < rows) {
      const double v = (double)mlp_output(t, t.h1, threadIdx.x);
      out[r] = xan ? xan[r] * exp(v) : v;
    }
    __syncthreads();  // h1 is rewritten by the next tile
  }
}

// Forward and backward over the rows [row0, row0 + rows) in tiles of
// kRowsCTA, `tiles` consecutive tiles per CTA (at most kGradTiles); writes
// the CTA's gradient (kTrain values, layout of the trainable parameters) and
// its sum of squared errors, FP64, to part[blockIdx.x * (kTrain + 1) ...].
// Loss L = (1/B) sum (y - t)^2 over the B rows of the batch.
// Three products per tile: z2 = h1 W2^T, dL/dh1 = g2 W2 and dW2 = g2^T h1 (g2 =
// dL/dz2). dW2 is summed in FP32 over a tile and in double-float across the
// CTA's tiles; the other gradients are summed per thread in FP32 over its 8
// rows of each tile (at most 128 rows) and in double-float over the threads.
// 200003 rows: 172 us for this and the reduction (a thread per row with
// its activations in shared memory, four warps per SM, and a partial per 128
// rows: 602 us and 224 us for the reduction of the partials).
constexpr int kGradTiles = 16;

// A running sum (s, c) as FP64. One that has left FP32's range is infinite, as in
// a plain sum, though its error term is not a number then.
__device__ __forceinline__ double df_sum_f64(float s, float c) {
  return isfinite(s) ? (double)s + (double)c : (double)s;
}

struct alignas(16) MlpGradSmem {
  MlpTile t;
  float g2[kH * kMlpPitch];  // dL/dz2, [unit][row]
  float w2[kH * kWPitch];    // [j][k]
  float sq[kRowsCTA], gy[kRowsCTA];
};

__global__ void __launch_bounds__(kMlpThreads, 2) k_mlp_grad(const float* __restrict__ P, const float* __restrict__ F,
                                                             const float* __restrict__ T, int64_t row0, int64_t rows,
                                                             int tiles, double inv_b, double* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MlpGradSmem& s = *reinterpret_cast<MlpGradSmem*>(smem_raw);
  MlpTile& t = s.t;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  for (int i = tid; i < kH * kH; i += kMlpThreads) s.w2[(i / kH) * kWPitch + i % kH] = P[kOffW2 + i];
  mlp_load(P, t);
  F += row0 * 4;
  T += row0;
  float dw2h[4][4], dw2l[4][4];  // j = ty + 16 a, k = tx + 16 b
  float dw1[4][4], db1[4];       // k = 4 tx + a, input b
  float db2[4], dw3[4];          // unit 4 tx + a
  float db3 = 0.f;
  double sq = 0.0;               // thread 0
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    db1[a] = db2[a] = dw3[a] = 0.f;
#pragma unroll
    for (int b = 0; b < 4; ++b) dw2h[a][b] = dw2l[a][b] = dw1[a][b] = 0.f;
  }
  const int64_t tile0 = (int64_t)blockIdx.x * tiles;
  for (int q = 0; q < tiles; ++q) {
    const int64_t r0 = (tile0 + q) * kRowsCTA;
    if (r0 >= rows) break;
    {
      float h2[8][4];
      mlp_forward(F, r0, rows, t, h2);
      mlp_store_h2(h2, s.g2);
      __syncthreads();
      if (tid < kRowsCTA) {
        const float e = r0 + tid < rows ? mlp_output(t, s.g2, tid) - T[r0 + tid] : 0.f;
        s.sq[tid] = e * e;
        s.gy[tid] = (float)(2.0 * inv_b) * e;
      }
      __syncthreads();
      if (tid == 0) {  // the tile's squared error, its rows in order
        float v = 0.f;
#pragma unroll 16
        for (int r = 0; r < kRowsCTA; ++r) v += s.sq[r];
        sq += (double)v;
      }
      float gy[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        gy[r] = s.gy[8 * ty + r];
        db3 += gy[r];
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float w = t.w3[4 * tx + c];
        float g[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          dw3[c] = fmaf(gy[r], h2[r][c], dw3[c]);
          g[r] = gy[r] * w * (1.f - h2[r][c] * h2[r][c]);
          db2[c] += g[r];
        }
        float4* o = reinterpret_cast<float4*>(&s.g2[(4 * tx + c) * kMlpPitch + 8 * ty]);
        o[0] = make_float4(g[0], g[1], g[2], g[3]);
        o[1] = make_float4(g[4], g[5], g[6], g[7]);
      }
    }
    __syncthreads();
    {  // dL/dh1 = g2 W2, then dL/dz1, dW1 and db1
      f2x acc[4][4];
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[p][c] = 0ull;
#pragma unroll 4
      for (int j = 0; j < kH; ++j) {
        const ulonglong2 a01 = *reinterpret_cast<const ulonglong2*>(&s.g2[j * kMlpPitch + 8 * ty]);
        const ulonglong2 a23 = *reinterpret_cast<const ulonglong2*>(&s.g2[j * kMlpPitch + 8 * ty + 4]);
        const float4 w = *reinterpret_cast<const float4*>(&s.w2[j * kWPitch + 4 * tx]);
        const f2x av[4] = {a01.x, a01.y, a23.x, a23.y};
        const f2x wv[4] = {f2_pack(w.x, w.x), f2_pack(w.y, w.y), f2_pack(w.z, w.z), f2_pack(w.w, w.w)};
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[p][c] = f2_fma(av[p], wv[c], acc[p][c]);
      }
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float4 x0 = *reinterpret_cast<const float4*>(&t.x[(8 * ty + 2 * p) * kIn]);
        const float4 x1 = *reinterpret_cast<const float4*>(&t.x[(8 * ty + 2 * p + 1) * kIn]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float2 gh = f2_unpack(acc[p][c]);
          const float2 h = *reinterpret_cast<const float2*>(&t.h1[(4 * tx + c) * kMlpPitch + 8 * ty + 2 * p]);
          const float g0 = gh.x * (1.f - h.x * h.x), g1 = gh.y * (1.f - h.y * h.y);
          db1[c] += g0 + g1;
          dw1[c][0] = fmaf(g1, x1.x, fmaf(g0, x0.x, dw1[c][0]));
          dw1[c][1] = fmaf(g1, x1.y, fmaf(g0, x0.y, dw1[c][1]));
          dw1[c][2] = fmaf(g1, x1.z, fmaf(g0, x0.z, dw1[c][2]));
          dw1[c][3] = fmaf(g1, x1.w, fmaf(g0, x0.w, dw1[c][3]));
        }
      }
    }
    {  // dW2 = g2^T h1: even and odd rows in the halves of each pair
      f2x acc[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0ull;
#pragma unroll 2
      for (int r = 0; r < kRowsCTA; r += 4) {
        ulonglong2 g[4], hh[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          g[a] = *reinterpret_cast<const ulonglong2*>(&s.g2[(ty + 16 * a) * kMlpPitch + r]);
          hh[a] = *reinterpret_cast<const ulonglong2*>(&t.h1[(tx + 16 * a) * kMlpPitch + r]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] = f2_fma(g[a].y, hh[b].y, f2_fma(g[a].x, hh[b].x, acc[a][b]));
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const float2 v = f2_unpack(acc[a][b]);
          df_acc(dw2h[a][b], dw2l[a][b], v.x + v.y);
        }
    }
    __syncthreads();  // h1, g2 and x are rewritten by the next tile
  }
  double* out = part + (size_t)blockIdx.x * (kTrain + 1);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b)
      out[kOffW2 - kOffW1 + (ty + 16 * a) * kH + tx + 16 * b] = df_sum_f64(dw2h[a][b], dw2l[a][b]);
  // the other gradients: 16 threads (ty) hold parts of each; red[v][ty][tx]
  float* red = s.g2;
  constexpr int NV = 29;
  static_assert(NV * kMlpThreads <= kH * kMlpPitch, "reduction fits in g2");
  auto put = [&](int v, float x) { red[v * kMlpThreads + tid] = x; };
#pragma unroll
  for (int a = 0; a < 4; ++a) {
#pragma unroll
    for (int b = 0; b < 4; ++b) put(a * 4 + b, dw1[a][b]);
    put(16 + a, db1[a]);
    put(20 + a, db2[a]);
    put(24 + a, dw3[a]);
  }
  put(28, db3);
  __syncthreads();
  for (int e = tid; e < NV * 16; e += kMlpThreads) {
    const int v = e / 16, u = e % 16;  // u: tx
    float h = 0.f, l = 0.f;
    for (int g = 0; g < 16; ++g) df_acc(h, l, red[v * kMlpThreads + g * 16 + u]);
    const double d = df_sum_f64(h, l);
    if (v < 16)
      out[(4 * u + v / 4) * kIn + v % 4] = d;
    else if (v < 20)
      out[kOffB1 - kOffW1 + 4 * u + v - 16] = d;
    else if (v < 24)
      out[kOffB2 - kOffW1 + 4 * u + v - 20] = d;
    else if (v < 28)
      out[kOffW3 - kOffW1 + 4 * u + v - 24] = d;
    else if (u == 0)  // every tx holds the same rows
      out[kOffB3 - kOffW1] = d;
  }
  if (tid == 0) out[kTrain] = sq;
}

// Sums the CTA partials in a fixed order (FP64), eight threads per value. mode
// 0: write the gradient and loss; mode 1: Adam update of the trainable
// parameters (m, v state).
__global__ void __launch_bounds__(256) k_mlp_reduce(const double* __restrict__ part, int nblk, double inv_b,
                                                    float* __restrict__ P, float* __restrict__ m,
                                                    float* __restrict__ v, float lr, float b1, float b2, float eps,
                                                    double bc1, double bc2, int mode, float* __restrict__ grad,
                                                    double* __restrict__ loss) {
  __shared__ double red[8][32];
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
  const int q = blockIdx.x * 32 + lane;
  double g = 0.0;
  if (q <= kTrain) {
#pragma unroll 4
    for (int c = sl; c < nblk; c += 8) g += part[(size_t)c * (kTrain + 1) + q];
  }
  red[sl][lane] = g;
  __syncthreads();
  if (sl != 0 || q > kTrain) return;
#pragma unroll
  for (int c = 1; c < 8; ++c) g += red[c][lane];
  if (q == kTrain) {
    if (loss) *loss = g * inv_b;
    return;
  }
  if (mode == 0) {
    grad[q] = (float)g;
    return;
  }
  const float gf = (float)g;
  const float mm = b1 * m[q] + (1.f - b1) * gf;
  const float vv = b2 * v[q] + (1.f - b2) * gf * gf;
  m[q] = mm;
  v[q] = vv;
  const double mh = (double)mm / bc1, vh = (double)vv / bc2;
  P[kOffW1 + q] = (float)((double)P[kOffW1 + q] - (double)lr * mh / (sqrt(vh) + (double)eps));
}
constexpr int kReduceBlocks = (kTrain + 1 + 31) / 32;

// feature means and standard deviations (FP64 partial sums per CTA)
__global__ void k_mlp_stats_part(const float* __restrict__ F, int64_t rows, double* __restrict__ part) {
  double s[2 * kIn] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (int64_t)gridDim.x * blockDim.x)
#pragma unroll
    for (int c = 0; c < kIn; ++c) {
      const double x = F[r * 4 + c];
      s[c] += x;
      s[kIn + c] += x * x;
    }
  __shared__ double sh[2 * kIn][256];
#pragma unroll
  for (int c = 0; c < 2 * kIn; ++c) sh[c][threadIdx.x] = s[c];
  __syncthreads();
  if (threadIdx.x < 2 * kIn) {
    double t = 0.0;
    for (int i = 0; i < (int)blockDim.x; ++i) t += sh[threadIdx.x][i];
    part[blockIdx.x * 2 * kIn + threadIdx.x] = t;
  }
}

__global__ void k_mlp_stats_fin(const double* __restrict__ part, int nblk, int64_t rows, float* __restrict__ P) {
  const int c = threadIdx.x;
  if (c >= kIn) return;
  double s = 0.0, s2 = 0.0;
  for (int b = 0; b < nblk; ++b) {
    s += part[b * 2 * kIn + c];
    s2 += part[b * 2 * kIn + kIn + c];
  }
  const double mean = s / (double)rows;
  const double var = fmax(s2 / (double)rows - mean * mean, 0.0);
  P[kOffMean + c] = (float)mean;
  P[kOffStd + c] = (float)fmax(sqrt(var), 1e-6);
}

// training target log(D_f / x_an)
__global__ void k_log_ratio(const double* __restrict__ Df, const double* __restrict__ xan, int64_t rows,
                            float* __restrict__ t) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (int64_t)gridDim.x * blockDim.x)
    t[r] = (float)log(Df[r] / xan[r]);
}

cudaError_t mlp_setup() {
  static PerDevice attr;
  return attr.once([] {
    cudaError_t r = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(MlpGradSmem));
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(k_mlp_predict, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlpTile));
    return r;
  });
}

// CTAs of a gradient pass: up to two per SM, each with at most kGradTiles tiles
int grad_tiles(int64_t rows) {
  const int64_t tiles = (rows + kRowsCTA - 1) / kRowsCTA;
  return (int)std::min<int64_t>(kGradTiles, std::max<int64_t>(1, (tiles + 2 * 152 - 1) / (2 * 152)));
}
int grad_blocks(int64_t rows) {
  const int64_t tiles = (rows + kRowsCTA - 1) / kRowsCTA;
  return (int)((tiles + grad_tiles(rows) - 1) / grad_tiles(rows));
}

// ------------------------------------------------------------------ launchers (wl_host.h)
cudaError_t launch_features(const int32_t* rp, const int32_t* col, int64_t n, int64_t nnz, double alpha, double mu,
                            const int32_t* perm, float* F, double* xan, void* tmp, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  // tmp: ad (n doubles), t (n u64), ticket (u64) and number of long lists (int) in 16 bytes, outdeg / orp (n + 1
  // int64 each), scan scratch, ocol (nnz / 2 + 1 int32), the nodes with long lists (n int32)
  double* ad = (double*)tmp;
  unsigned long long* t = (unsigned long long*)(ad + n);
  unsigned long long* ticket = t + n;
  int* nbig = (int*)(ticket + 1);
  int64_t* outdeg = (int64_t*)(ticket + 2);
  int64_t* orp = outdeg + n + 1;
  int64_t* sc = orp + n + 1;
  int32_t* ocol = (int32_t*)(sc + n / 1024 + 64);
  int32_t* big = ocol + nnz / 2 + 1;
  constexpr int NW = kFeatBlock / 32;
  const unsigned gw = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + NW - 1) / NW, 152 * 8));
  const unsigned g1 = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 32));
  if (F) {  // triangles only for the network's inputs (x_an needs d and A d alone)
    cudaError_t e = cudaMemsetAsync(t, 0, sizeof(unsigned long long) * (n + 2), s);
    if (e != cudaSuccess) return e;
    k_feat_ad<true><<<gw, kFeatBlock, 0, s>>>(rp, col, n, ad, outdeg, big, nbig);
    e = launch_scan(outdeg, n, orp, sc, s);  // orp[0..n]: exclusive prefix, orp[n] = total
    if (e != cudaSuccess) return e;
    k_feat_orient<<<gw, kFeatBlock, 0, s>>>(rp, col, n, orp, ocol);
    // long lists first (one CTA each, the heaviest work), then the rest of the nodes by warps
    const unsigned gb = (unsigned)std::max<int64_t>(1, std::min<int64_t>(n, 152 * 6));
    k_feat_tri_cta<<<gb, kTriBlock, 0, s>>>(orp, ocol, big, nbig, t);
    const unsigned gt = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + NW - 1) / NW, 152 * 6));
    k_feat_tri_warp<<<gt, kTriBlock, 0, s>>>(orp, ocol, n, t, ticket);
  } else {
    k_feat_ad<false><<<gw, kFeatBlock, 0, s>>>(rp, col, n, ad, nullptr, nullptr, nullptr);
  }
  k_feat_out<<<g1, 256, 0, s>>>(rp, ad, t, n, alpha, mu, perm, F, xan);
  return cudaGetLastError();
}

size_t features_tmp_bytes(int64_t n, int64_t nnz) {
  return (size_t)n * 8 * 2 + 16 + (size_t)(n + 1) * 8 * 2 + (size_t)(n / 1024 + 64) * 8 + (size_t)(nnz / 2 + 1) * 4 +
         (size_t)n * 4 + 256;
}

cudaError_t launch_mlp_predict(const float* P, const float* F, int64_t rows, const double* xan, double* out,
                               cudaStream_t s) {
  if (rows == 0) return cudaSuccess;
  const cudaError_t e = mlp_setup();
  if (e != cudaSuccess) return e;
  const unsigned g = (unsigned)std::min<int64_t>((rows + kRowsCTA - 1) / kRowsCTA, 152 * 3);
  k_mlp_predict<<<g, kMlpThreads, sizeof(MlpTile), s>>>(P, F, rows, xan, out);
  return cudaGetLastError();
}

}  // namespace wl

using namespace wl;

namespace {

int mlp_err(cudaError_t e, const char* where) { return report_cuda_error(e, where); }

#define ML_CU(call)                                       \
  do {                                                    \
    cudaError_t e__ = (call);                             \
    if (e__ != cudaSuccess) return mlp_err(e__, #call);   \
  } while (0)

// staging and scratch of one synchronous call: released after the call's
// stream has been synchronised (or, on an early error, after a device sync)
struct DevBuf {
  void* p = nullptr;
  ~DevBuf() {
    if (p) {
      cudaDeviceSynchronize();
      pool_free(p);
    }
  }
  cudaError_t alloc(size_t b) { return pool_malloc(&p, b ? b : 16); }
};

bool dev_ptr(const void* p) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

// device copy of a caller array (host or device); `own` keeps a copy alive
int stage(const void* src, size_t bytes, DevBuf& own, const void** dev, cudaStream_t s) {
  if (dev_ptr(src)) {
    *dev = src;
    return WL_OK;
  }
  ML_CU(own.alloc(bytes));
  ML_CU(cudaMemcpyAsync(own.p, src, bytes, cudaMemcpyHostToDevice, s));
  *dev = own.p;
  return WL_OK;
}

// gradient partials over rows [row0, row0 + rows)
int grad_pass(const float* P, const float* F, const float* T, int64_t row0, int64_t rows, double* part,
              cudaStream_t s) {
  ML_CU(mlp_setup());
  k_mlp_grad<<<grad_blocks(rows), kMlpThreads, sizeof(MlpGradSmem), s>>>(P, F, T, row0, rows, grad_tiles(rows),
                                                                       1.0 / (double)rows, part);
  ML_CU(cudaGetLastError());
  return WL_OK;
}

}  // namespace

extern "C" {

int wl_mlp_loss_grad(const float* params, const float* feats, const float* target, int64_t rows, double* loss,
                     float* grad, void* stream) {
  if (!params || !feats || !target || rows <= 0 || rows > (int64_t)1 << 30) return WL_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  DevBuf bp, bf, bt, bpart, bg, bl;
  const void *P, *F, *T;
  int rc;
  if ((rc = stage(params, sizeof(float) * kParams, bp, &P, s)) != WL_OK) return rc;
  if ((rc = stage(feats, sizeof(float) * 4 * rows, bf, &F, s)) != WL_OK) return rc;
  if ((rc = stage(target, sizeof(float) * rows, bt, &T, s)) != WL_OK) return rc;
  const int nb = grad_blocks(rows);
  ML_CU(bpart.alloc(sizeof(double) * (size_t)nb * (kTrain + 1)));
  ML_CU(bg.alloc(sizeof(float) * kTrain));
  ML_CU(bl.alloc(sizeof(double)));
  if ((rc = grad_pass((const float*)P, (const float*)F, (const float*)T, 0, rows, (double*)bpart.p, s)) != WL_OK)
    return rc;
  k_mlp_reduce<<<kReduceBlocks, 256, 0, s>>>((const double*)bpart.p, nb, 1.0 / (double)rows, nullptr,
                                                       nullptr, nullptr, 0.f, 0.f, 0.f, 0.f, 1.0, 1.0, 0,
                                                       (float*)bg.p, (double*)bl.p);
  ML_CU(cudaGetLastError());
  // grad layout follows the parameter vector: zeros for the standardisation
  std::vector<float> gh(kParams, 0.f);
  ML_CU(cudaMemcpyAsync(gh.data() + kOffW1, bg.p, sizeof(float) * kTrain, cudaMemcpyDeviceToHost, s));
  double l = 0.0;
  ML_CU(cudaMemcpyAsync(&l, bl.p, sizeof(double), cudaMemcpyDeviceToHost, s));
  ML_CU(cudaStreamSynchronize(s));
  if (grad) ML_CU(cudaMemcpy(grad, gh.data(), sizeof(float) * kParams, cudaMemcpyDefault));
  if (loss) *loss = l;
  return WL_OK;
}

int wl_mlp_train(float* params, const float* feats, const float* target, int64_t rows, int steps, int64_t batch,
                 float lr, int standardize, double* final_loss, void* stream) {
  if (!params || !feats || !target || rows <= 0 || steps < 0 || rows > (int64_t)1 << 30) return WL_ERR_INVALID_ARG;
  if (batch <= 0 || batch > rows) batch = rows;
  cudaStream_t s = (cudaStream_t)stream;
  DevBuf bf, bt, bP, bpart, bm, bv, bl, bst;
  const void *F, *T;
  int rc;
  if ((rc = stage(feats, sizeof(float) * 4 * rows, bf, &F, s)) != WL_OK) return rc;
  if ((rc = stage(target, sizeof(float) * rows, bt, &T, s)) != WL_OK) return rc;
  ML_CU(bP.alloc(sizeof(float) * kParams));
  ML_CU(cudaMemcpyAsync(bP.p, params, sizeof(float) * kParams, cudaMemcpyDefault, s));
  float* P = (float*)bP.p;
  if (standardize) {
    const int sb = 152 * 4;
    ML_CU(bst.alloc(sizeof(double) * sb * 2 * kIn));
    k_mlp_stats_part<<<sb, 256, 0, s>>>((const float*)F, rows, (double*)bst.p);
    k_mlp_stats_fin<<<1, 32, 0, s>>>((const double*)bst.p, sb, rows, P);
    ML_CU(cudaGetLastError());
  }
  ML_CU(bpart.alloc(sizeof(double) * (size_t)std::max(grad_blocks(batch), grad_blocks(rows)) * (kTrain + 1)));
  ML_CU(bm.alloc(sizeof(float) * kTrain));
  ML_CU(bv.alloc(sizeof(float) * kTrain));
  ML_CU(bl.alloc(sizeof(double)));
  ML_CU(cudaMemsetAsync(bm.p, 0, sizeof(float) * kTrain, s));
  ML_CU(cudaMemsetAsync(bv.p, 0, sizeof(float) * kTrain, s));
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  int64_t off = 0;
  for (int it = 1; it <= steps; ++it) {
    if (off + batch > rows) off = 0;
    if ((rc = grad_pass(P, (const float*)F, (const float*)T, off, batch, (double*)bpart.p, s)) != WL_OK) return rc;
    const int nb = grad_blocks(batch);
    k_mlp_reduce<<<kReduceBlocks, 256, 0, s>>>((const double*)bpart.p, nb, 1.0 / (double)batch, P,
                                                         (float*)bm.p, (float*)bv.p, lr, b1, b2, eps,
                                                         1.0 - std::pow((double)b1, it), 1.0 - std::pow((double)b2, it),
                                                         1, nullptr, (double*)bl.p);
    ML_CU(cudaGetLastError());
    off += batch;
  }
  // loss of the trained network over all rows
  if ((rc = grad_pass(P, (const float*)F, (const float*)T, 0, rows, (double*)bpart.p, s)) != WL_OK) return rc;
  k_mlp_reduce<<<kReduceBlocks, 256, 0, s>>>((const double*)bpart.p, grad_blocks(rows),
                                                       1.0 / (double)rows, nullptr, nullptr, nullptr, 0.f, 0.f, 0.f,
                                                       0.f, 1.0, 1.0, 0, (float*)bm.p, (double*)bl.p);
  ML_CU(cudaGetLastError());
  double l = 0.0;
  ML_CU(cudaMemcpyAsync(&l, bl.p, sizeof(double), cudaMemcpyDeviceToHost, s));
  ML_CU(cudaMemcpyAsync(params, P, sizeof(float) * kParams, cudaMemcpyDefault, s));
  ML_CU(cudaStreamSynchronize(s));
  if (final_loss) *final_loss = l;
  return WL_OK;
}

int wl_mlp_predict(const float* params, const float* feats, int64_t rows, const double* xan, double* out,
                   void* stream) {
  if (!params || !feats || !out || rows < 0) return WL_ERR_INVALID_ARG;
  if (rows == 0) return WL_OK;
  cudaStream_t s = (cudaStream_t)stream;
  DevBuf bp, bf, bx, bo;
  const void *P, *F, *X = nullptr;
  int rc;
  if ((rc = stage(params, sizeof(float) * kParams, bp, &P, s)) != WL_OK) return rc;
  if ((rc = stage(feats, sizeof(float) * 4 * rows, bf, &F, s)) != WL_OK) return rc;
  if (xan && (rc = stage(xan, sizeof(double) * rows, bx, &X, s)) != WL_OK) return rc;
  double* o = out;
  const bool dev_out = dev_ptr(out);
  if (!dev_out) {
    ML_CU(bo.alloc(sizeof(double) * rows));
    o = (double*)bo.p;
  }
  ML_CU(launch_mlp_predict((const float*)P, (const float*)F, rows, (const double*)X, o, s));
  if (!dev_out) ML_CU(cudaMemcpyAsync(out, o, sizeof(double) * rows, cudaMemcpyDeviceToHost, s));
  ML_CU(cudaStreamSynchronize(s));
  return WL_OK;
}

int wl_mlp_param_count(void) { return kParams; }

// Checkpoint file of the network: a 32-byte header (magic "WLMLP001",
// uint32 inputs, hidden width, output width, parameter count, FNV-1a hash of
// the parameter bytes, uint32 zero) followed by the parameter vector as
// little-endian FP32 in the order of the parameter layout above.
namespace {
constexpr char kMlpMagic[8] = {'W', 'L', 'M', 'L', 'P', '0', '0', '1'};

uint32_t fnv1a(const unsigned char* p, size_t n) {
  uint32_t h = 2166136261u;
  for (size_t i = 0; i < n; ++i) {
    h ^= p[i];
    h *= 16777619u;
  }
  return h;
}

void put_u32(unsigned char* p, uint32_t v) {
  for (int i = 0; i < 4; ++i) p[i] = (unsigned char)(v >> (8 * i));
}

uint32_t get_u32(const unsigned char* p) {
  uint32_t v = 0;
  for (int i = 0; i < 4; ++i) v |= (uint32_t)p[i] << (8 * i);
  return v;
}
}  // namespace

int wl_mlp_save(const char* path, const float* params) {
  if (!path || !params) return WL_ERR_INVALID_ARG;
  std::vector<unsigned char> buf(32 + (size_t)kParams * 4);
  memcpy(buf.data(), kMlpMagic, 8);
  for (int i = 0; i < kParams; ++i) {
    uint32_t bits;
    memcpy(&bits, params + i, 4);
    put_u32(buf.data() + 32 + (size_t)i * 4, bits);
  }
  put_u32(buf.data() + 8, kIn);
  put_u32(buf.data() + 12, kH);
  put_u32(buf.data() + 16, 1);
  put_u32(buf.data() + 20, kParams);
  put_u32(buf.data() + 24, fnv1a(buf.data() + 32, (size_t)kParams * 4));
  put_u32(buf.data() + 28, 0);
  FILE* f = fopen(path, "wb");
  if (!f) return WL_ERR_INVALID_ARG;
  const size_t w = fwrite(buf.data(), 1, buf.size(), f);
  const int rc = fclose(f);
  return (w == buf.size() && rc == 0) ? WL_OK : WL_ERR_INVALID_ARG;
}

int wl_mlp_load(const char* path, float* params) {
  if (!path || !params) return WL_ERR_INVALID_ARG;
  FILE* f = fopen(path, "rb");
  if (!f) return WL_ERR_INVALID_ARG;
  std::vector<unsigned char> buf(32 + (size_t)kParams * 4);
  const size_t r = fread(buf.data(), 1, buf.size(), f);
  unsigned char extra;
  const bool trailing = fread(&extra, 1, 1, f) == 1;
  fclose(f);
  if (r != buf.size() || trailing || memcmp(buf.data(), kMlpMagic, 8) != 0) return WL_ERR_INVALID_ARG;
  if (get_u32(buf.data() + 8) != (uint32_t)kIn || get_u32(buf.data() + 12) != (uint32_t)kH ||
      get_u32(buf.data() + 16) != 1u || get_u32(buf.data() + 20) != (uint32_t)kParams)
    return WL_ERR_INVALID_ARG;
  if (get_u32(buf.data() + 24) != fnv1a(buf.data() + 32, (size_t)kParams * 4)) return WL_ERR_NONFINITE;
  for (int i = 0; i < kParams; ++i) {
    const uint32_t bits = get_u32(buf.data() + 32 + (size_t)i * 4);
    memcpy(params + i, &bits, 4);
  }
  return WL_OK;
}

int wl_mlp_targets(const double* Df, const double* xan, int64_t rows, float* target, void* stream) {
  if (!Df || !xan || !target || rows < 0) return WL_ERR_INVALID_ARG;
  if (rows == 0) return WL_OK;
  cudaStream_t s = (cudaStream_t)stream;
  DevBuf bd, bx, bt;
  const void *D, *X;
  int rc;
  if ((rc = stage(Df, sizeof(double) * rows, bd, &D, s)) != WL_OK) return rc;
  if ((rc = stage(xan, sizeof(double) * rows, bx, &X, s)) != WL_OK) return rc;
  float* T = target;
  const bool dev_out = dev_ptr(target);
  if (!dev_out) {
    ML_CU(bt.alloc(sizeof(float) * rows));
    T = (float*)bt.p;
  }
  const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((rows + 255) / 256, 152 * 16));
  k_log_ratio<<<g, 256, 0, s>>>((const double*)D, (const double*)X, rows, T);
  ML_CU(cudaGetLastError());
  if (!dev_out) ML_CU(cudaMemcpyAsync(target, T, sizeof(float) * rows, cudaMemcpyDeviceToHost, s));
  ML_CU(cudaStreamSynchronize(s));
  return WL_OK;
}

}  // extern "C"
