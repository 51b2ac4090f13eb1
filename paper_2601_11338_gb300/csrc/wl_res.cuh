// Residual of the iterative refinement (refined form, Sec. 4.2 solves) in
// double-float arithmetic: FP64-accurate, FP32 instructions only.
//
// The refined solve of M x = b keeps b, the residual r and the iterate x as
// double-float vectors (two FP32 arrays each) and corrects x with FP32 CG
// solves M d = fl32(r). The residual is updated, not recomputed:
//     r <- r - M d ,  x <- x + d
// which equals b - M x up to the double-float rounding of each step (about
// 2^-46 of |r| + |M d|), so the gathered operand is the 4-byte correction d
// instead of an 8-byte iterate. Only a warm start needs the full form
//     r = b - M x   (x = xh + xl gathered as two FP32 terms).
// M = ca I + cA A + cD D; the neighbour sum A y is accumulated with the
// error-free two-sum, M y and the subtraction in double-float.
//
// Each kernel ends in the deterministic last-CTA reduction of |r|^2 per
// column (from the FP32 leading terms: the convergence test needs a few
// digits of the norm, not all of them) into st->gamma.
#pragma once
#include "wl_cg2.cuh"
#include "wl_df.cuh"

namespace wl {

struct DfResArgs {
  PhaseGraph g;
  const float* yh;  // gathered operand: the correction d, or (FULL) the iterate's leading term
  const float* yl;  // FULL: the iterate's trailing term
  const float* bh;  // r_in: the previous residual, or (FULL) the right-hand side b
  const float* bl;
  float* rh;        // r_out (may alias r_in)
  float* rl;
  float* xh;        // iterate, updated x += d in place (not FULL)
  float* xl;
  df ca, cA, cD;
  double* part;     // gridDim.x * K partials
  CgState* st;      // st->gamma[c] = |r_out[:, c]|^2
  int x_zero;       // the iterate is zero on entry: x = d
  // optional per-row diagonal added to M as a double-float pair (shifted
  // solves); NULL: none. bh == NULL (FULL only): b = 0, r_out = -M x
  const float* dsh_h = nullptr;
  const float* dsh_l = nullptr;
};

// (s, c, l): neighbour sum of the leading terms with its rounding errors,
// and the plain sum of the trailing terms (FULL only)
template <int K, int VW, bool FULL>
__device__ __forceinline__ void df_row_gather(const int32_t* __restrict__ col, int beg, int end, int step,
                                              const float* YH, const float* YL, int lane_off, float (&s)[VW],
                                              float (&c)[VW], float (&l)[VW]) {
  constexpr int U = kGatherU;  // predicated batches, as in row_gather
  for (int e = beg; e < end; e += U * step) {
    int j[U];
#pragma unroll
    for (int u = 0; u < U; ++u) j[u] = (e + u * step < end) ? __ldg(col + e + u * step) : -1;
    Pack<float, VW> hh[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j[u] >= 0) {
        hh[u] = ld_plain<float, VW>(YH + (size_t)j[u] * K + lane_off);
      } else {
#pragma unroll
        for (int v = 0; v < VW; ++v) hh[u].v[v] = 0.f;
      }
    }
    if constexpr (FULL) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (j[u] >= 0) {
          const Pack<float, VW> l0 = ld_plain<float, VW>(YL + (size_t)j[u] * K + lane_off);
#pragma unroll
          for (int v = 0; v < VW; ++v) l[v] += l0.v[v];
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int v = 0; v < VW; ++v) df_acc(s[v], c[v], hh[u].v[v]);
  }
}

// SH: the solve's M carries the per-row diagonal (dsh_h, dsh_l); a separate
// instance, so that the unshifted kernel carries no trace of it
template <int K, bool FULL, bool SH = false>
__global__ void __launch_bounds__(kPhaseBlock, 4) df_res(DfResArgs a) {
  using C = Cfg<float, K>;
  constexpr int VW = C::VW, G = C::G, RPB = kPhaseBlock / G;
  __shared__ float s_red[3][kPhaseBlock / 32 * K];
  __shared__ double s_tmp[kPhaseBlock];
  __shared__ double s_out[K];
  const int tid = threadIdx.x, sl = tid % G, lane_off = sl * VW;
  float nacc[VW];
#pragma unroll
  for (int v = 0; v < VW; ++v) nacc[v] = 0.f;

  auto fin = [&](int64_t row, int deg, const float (&s)[VW], const float (&c)[VW], const float (&l)[VW]) {
    const size_t o = (size_t)row * K + lane_off;
    df crow = df_add(a.ca, df_mul_f(a.cD, (float)deg));
    if constexpr (SH) crow = df_add(crow, df{a.dsh_h[row], a.dsh_l[row]});
    const Pack<float, VW> yh = ld_plain<float, VW>(a.yh + o);
    Pack<float, VW> yl;
    if constexpr (FULL) yl = ld_plain<float, VW>(a.yl + o);
    Pack<float, VW> bh, bl;
    if (!FULL || a.bh) {
      bh = ld_plain<float, VW>(a.bh + o);
      bl = ld_plain<float, VW>(a.bl + o);
    } else {
#pragma unroll
      for (int v = 0; v < VW; ++v) bh.v[v] = bl.v[v] = 0.f;
    }
    Pack<float, VW> xh, xl;
    if constexpr (!FULL) {
      if (!a.x_zero) {
        xh = ld_plain<float, VW>(a.xh + o);
        xl = ld_plain<float, VW>(a.xl + o);
      }
    }
    Pack<float, VW> rh, rl;
#pragma unroll
    for (int v = 0; v < VW; ++v) {
      const df nb = two_sum(s[v], c[v] + l[v]);
      const df y{yh.v[v], FULL ? yl.v[v] : 0.f};
      const df My = df_add(df_mul(crow, y), df_mul(a.cA, nb));
      const df r = df_sub(df{bh.v[v], bl.v[v]}, My);
      rh.v[v] = r.hi;
      rl.v[v] = r.lo;
      nacc[v] = __fmaf_rn(r.hi, r.hi, nacc[v]);
      if constexpr (!FULL) {
        if (a.x_zero) {
          xh.v[v] = yh.v[v];
          xl.v[v] = 0.f;
        } else {
          const df t = two_sum(xh.v[v], yh.v[v]);
          const df u = quick_two_sum(t.hi, t.lo + xl.v[v]);
          xh.v[v] = u.hi;
          xl.v[v] = u.lo;
        }
      }
    }
    stp<float, VW>(a.rh + o, rh);
    stp<float, VW>(a.rl + o, rl);
    if constexpr (!FULL) {
      stp<float, VW>(a.xh + o, xh);
      stp<float, VW>(a.xl + o, xl);
    }
  };

  auto fold = [](float (&s)[VW], float (&c)[VW], float (&l)[VW], int off, unsigned mask) {
#pragma unroll
    for (int v = 0; v < VW; ++v) {
      const float so = __shfl_xor_sync(mask, s[v], off);
      const float co = __shfl_xor_sync(mask, c[v], off);
      const float lo = __shfl_xor_sync(mask, l[v], off);
      const df t = two_sum(s[v], so);
      s[v] = t.hi;
      c[v] += t.lo + co;
      l[v] += lo;
    }
  };
  if ((int)blockIdx.x < a.g.nhub) {
    // one hub row per CTA: RPB lane groups stride over the entries
    const int64_t row = a.g.hubs[blockIdx.x];
    const int beg = a.g.row_ptr[row], end = a.g.row_ptr[row + 1];
    float s[VW], c[VW], l[VW];
#pragma unroll
    for (int v = 0; v < VW; ++v) s[v] = c[v] = l[v] = 0.f;
    df_row_gather<K, VW, FULL>(a.g.col, beg + tid / G, end, RPB, a.yh, a.yl, lane_off, s, c, l);
    // the lane groups' sums: within each warp by shuffles, then the warps
#pragma unroll
    for (int off = G; off < 32; off <<= 1) fold(s, c, l, off, 0xffffffffu);
    if ((tid & 31) < G)
#pragma unroll
      for (int v = 0; v < VW; ++v) {
        const int q = (tid >> 5) * K + lane_off + v;
        s_red[0][q] = s[v];
        s_red[1][q] = c[v];
        s_red[2][q] = l[v];
      }
    __syncthreads();
    if (tid < G) {
      for (int w = 1; w < kPhaseBlock / 32; ++w)
#pragma unroll
        for (int v = 0; v < VW; ++v) {
          const int q = w * K + lane_off + v;
          const df t = two_sum(s[v], s_red[0][q]);
          s[v] = t.hi;
          c[v] += t.lo + s_red[1][q];
          l[v] += s_red[2][q];
        }
      fin(row, end - beg, s, c, l);
    }
  } else if ((int)blockIdx.x < a.g.nhub + a.g.nmid_blk) {
    // mid rows, one warp each (as in the CG S kernel)
    const int lane = tid & 31;
    constexpr int WPB = kPhaseBlock / 32;
    for (int r = ((int)blockIdx.x - a.g.nhub) * WPB + (tid >> 5); r < a.g.nmid; r += a.g.nmid_blk * WPB) {
      const int64_t row = a.g.mids[r];
      const int beg = a.g.row_ptr[row], end = a.g.row_ptr[row + 1];
      float s[VW], c[VW], l[VW];
#pragma unroll
      for (int v = 0; v < VW; ++v) s[v] = c[v] = l[v] = 0.f;
      df_row_gather<K, VW, FULL>(a.g.col, beg + lane / G, end, 32 / G, a.yh, a.yl, lane_off, s, c, l);
#pragma unroll
      for (int off = G; off < 32; off <<= 1) fold(s, c, l, off, 0xffffffffu);
      if (lane < G) fin(row, end - beg, s, c, l);
    }
  } else {
    const int nlist = a.g.nhub + a.g.nmid_blk;
    const int lim = a.g.nmid_blk > 0 ? kMidDeg : kHubDeg;  // longer rows: hub CTAs or mid warps
    const int64_t nblk = (int64_t)gridDim.x - nlist;
    // E lane groups per row where a row has few lanes (K <= 2)
    constexpr int E = G >= 4 ? 1 : 4 / G, LPR = G * E, RPP = kPhaseBlock / LPR;
    const int e = (tid / G) % E;
    for (int64_t row = ((int64_t)blockIdx.x - nlist) * RPP + tid / LPR; row < a.g.n; row += nblk * RPP) {
      const int beg = a.g.row_ptr[row], end = a.g.row_ptr[row + 1];
      if (end - beg > lim) continue;
      float s[VW], c[VW], l[VW];
#pragma unroll
      for (int v = 0; v < VW; ++v) s[v] = c[v] = l[v] = 0.f;
      df_row_gather<K, VW, FULL>(a.g.col, beg + e, end, E, a.yh, a.yl, lane_off, s, c, l);
      if constexpr (E > 1) {
        const unsigned m = ((1u << LPR) - 1u) << (tid & 31 & ~(LPR - 1));
#pragma unroll
        for (int off = G; off < LPR; off <<= 1) fold(s, c, l, off, m);
      }
      if (e == 0) fin(row, end - beg, s, c, l);
    }
  }
  if (!block_partials_last<float, K>(nacc, a.part, &a.st->ticket)) return;
  sum_partials<K>(a.part, gridDim.x, s_tmp, s_out);
  if (tid < K) a.st->gamma[tid] = s_out[tid];
  if (tid == 0) a.st->ticket = 0;
}

// b (n x K FP64, contiguous) -> (bh, bl), |b|^2 per column (from bh) -> b2[c]
template <int K>
__global__ void __launch_bounds__(kPhaseBlock) df_from_f64(const double* b, int64_t n, float* bh,
                                                           float* bl, double* part, CgState* st,
                                                           double* b2) {
  using C = Cfg<float, K>;
  constexpr int VW = C::VW;
  __shared__ double s_tmp[kPhaseBlock];
  __shared__ double s_out[K];
  const int tid = threadIdx.x;
  float acc[VW];
#pragma unroll
  for (int v = 0; v < VW; ++v) acc[v] = 0.f;
  const size_t nv = (size_t)n * K / VW;
  for (size_t e = (size_t)blockIdx.x * kPhaseBlock + tid; e < nv; e += (size_t)gridDim.x * kPhaseBlock) {
    Pack<float, VW> hh, ll;
#pragma unroll
    for (int v = 0; v < VW; ++v) {
      const df x = split_f64(b[e * VW + v]);
      hh.v[v] = x.hi;
      ll.v[v] = x.lo;
      acc[v] = __fmaf_rn(x.hi, x.hi, acc[v]);
    }
    stp<float, VW>(bh + e * VW, hh);
    stp<float, VW>(bl + e * VW, ll);
  }
  if (!block_partials_last<float, K>(acc, part, &st->ticket)) return;
  sum_partials<K>(part, gridDim.x, s_tmp, s_out);
  if (tid < K) b2[tid] = s_out[tid];
  if (tid == 0) st->ticket = 0;
}

}  // namespace wl
