// Lockstep conjugate gradients on M = ca I + cA A + cD D for K columns as
// high-occupancy phase kernels (Sec. 4.2: each application of the resolvent
// walk Laplacian is one CG solve with the deformed Laplacian, positive
// definite for alpha < 1 / rho(Z), Prop. CGworks).
//
// The gather of neighbour vectors is latency bound, so these kernels keep
// the SMs full of warps (G lanes per row, one 16-byte slice each, rows
// spread over a grid-stride loop) instead of persisting with few warps.
// Hub rows (the graph's list of them) are gathered by one CTA each; when the
// graph carries a list of mid rows (kMidDeg < deg, not hubs), the S kernel
// spends a share of its CTAs (proportional to those rows' entries) on them,
// one warp per row, so that no lane group walks a long row alone, and the
// remaining CTAs take the short rows; the grid stays one wave. Where the line
// between mid rows and hubs lies is the caller's: kHubDeg entries in a handle's own
// lists, kPhaseHubDeg (wl_api.cu) in those of its solves.
//
// One iteration = two kernels:
//   S: s = M r ; q = s + beta q ; delta = (r, q)
//   U: r' = r - alpha q ; gamma' = (r', r')
// with r' in a buffer of its own, and x (and p, every kHist iterations) formed
// from the kept residuals by a third kernel (cg_x_phase). In the X form, which
// keeps none, S also makes x += alpha p and p = r + beta p, and delta = (p, q).
// Each kernel ends with a last-CTA reduction (fixed order, deterministic)
// that derives the next scalars and the per-column convergence on the
// device; a kernel finding the solve inactive returns at once, so the host
// launches iterations in chunks and reads one flag between chunks.
// Vector traffic per iteration, besides the gathers, 4 nnz and 4 (n + 1) bytes: 6 n K s
// bytes (r, q read, q written; r, q read, r' written) and n K s for x at the end;
// 10 n K s in the X form.
#pragma once
#include "wl_common.cuh"
#include "wl_df.cuh"

namespace wl {

constexpr int kHubDeg = 256;       // rows with more entries are on a handle's list of hubs
constexpr int kMidDeg = 30;        // rows with more entries (not hubs) get a warp each in the S kernels
constexpr int kPhaseBlock = 256;   // threads per CTA of the phase kernels
#ifndef WL_PHASE_MINB
#define WL_PHASE_MINB 3
#endif
constexpr int kPhaseMinBlocks = WL_PHASE_MINB;  // CTAs per SM the S kernel's registers are sized for
// FP32 CG kernels: 5 CTAs per SM (48 registers) hold the eight predicated
// gathers per lane; measured 139 us per K = 16 S phase on the Chung-Lu 1e6
// graph (6 CTAs: 147 us; 4 CTAs: the same, and U 3% slower)
#ifndef WL_PHASE_MINB_F32
#define WL_PHASE_MINB_F32 5
#endif
constexpr int kPhaseMinBlocksF32 = WL_PHASE_MINB_F32;
template <typename T>
constexpr int phase_min_blocks() { return sizeof(T) == 4 ? kPhaseMinBlocksF32 : kPhaseMinBlocks; }


// Per-solve device state (written by the last CTA of each kernel).
struct CgState {
  double gamma[64], alpha[64], beta[64], b2[64];
  int done[64], status[64];
  int active;  // 1 while some column iterates and iters < max_iter
  int iters;   // S phases executed
  unsigned ticket;
  int stiff;   // some column's p has grown beyond PhaseArgs::stiff
  double pi[64];  // |p|^2 by recurrence
};

struct PhaseGraph {
  const int32_t* row_ptr;
  const int32_t* col;
  int64_t n;
  const int32_t* hubs;  // rows with more entries than the line of the list (kHubDeg, kPhaseHubDeg)
  int nhub;
  const int32_t* mids = nullptr;  // rows with more than kMidDeg entries that are not hubs
  int nmid = 0;
  int nmid_blk = 0;               // CTAs (after the hub CTAs) that walk the mid rows; 0: no mid path
};

constexpr int kHist = 16;  // residuals kept before p and x are formed from them, at most

// Per column the step sizes of the kept iterations: x += sum alpha_i p_i with
// p_i = r_i + beta_i p_{i-1}
struct CgHist {
  double alpha[kHist][64], beta[kHist][64];
};

template <typename T>
struct PhaseArgs {
  PhaseGraph g;
  T* x;
  const T* r;  // r_j
  T* rn;       // r_{j+1} (r_j itself where x and p are updated in each S phase)
  T* p;
  T* q;
  double ca, cA, cD;
  const double* bnorm2;  // K or NULL (then ||r_0||^2)
  const int* skip;       // K or NULL
  double* part;          // gridDim.x * K partials
  CgState* st;
  int max_iter;
  double tol2;
  // optional per-row diagonal added to M (the shifted solves of the
  // shift-and-invert Lanczos: M - a (D_f + sigma I)^{-1}); NULL: none
  const T* dshift = nullptr;
  CgHist* hist = nullptr;  // where the iteration's alpha and beta go, at `slot` (NULL: x and p are updated in S)
  int slot = 0;
  // > 0: CgState::stiff is set once some column's next p has |p|^2 > stiff |r|^2
  // (|p_j|^2 = |r_j|^2 + beta^2 |p_{j-1}|^2, as r_j is orthogonal to p_{j-1}), and the solve
  // stops there (active 0) unless x and p are updated in S
  double stiff = 0.0;
};

// ---------------------------------------------------------------- helpers
template <typename T, int VW>
__device__ __forceinline__ Pack<T, VW> ld_plain(const T* p) {
  return *reinterpret_cast<const Pack<T, VW>*>(p);
}
// the last read of a value for a while: its line may leave L2 first
template <typename T, int VW>
__device__ __forceinline__ Pack<T, VW> ld_last(const T* p) {
  Pack<T, VW> o;
  if constexpr (sizeof(T) * VW == 16) {
    const int4 t = __ldcs(reinterpret_cast<const int4*>(p));
    o = *reinterpret_cast<const Pack<T, VW>*>(&t);
  } else {
#pragma unroll
    for (int v = 0; v < VW; ++v) o.v[v] = __ldcs(p + v);
  }
  return o;
}

// Gathers per lane in flight in row_gather (unrolled batches of four with the tail
// walked entry by entry: 252 us where these take 240, per K = 16 FP32 iteration)
constexpr int kGatherU = 8;
// acc + sum of N = 8 or 4 FP64 values, the values added as integers. GB300 adds two
// FP64 lanes per clock and SM, so a neighbour sum of doubles is bound by its
// additions; here each value costs about 15 integer instructions (64 lanes
// per clock) instead, and a batch two FP64 ones. The values are aligned to the
// largest exponent among them with seven guard bits and summed exactly from
// there on (53 + 7 + 3 bits), rounded once at the end: the error is below 2^-4
// units in the last place of the largest value plus that rounding, less than
// that of eight FP64 additions in sequence. Chung-Lu 3e5, K = 16: 257 -> 198 us
// an S phase (FP64 additions alone, four values in flight), 159 -> 157 us with four
// values summed so too where a row's last batch has no more (three FP64 additions
// before; R-MAT scale 18, K = 8: 3% of a call). Batches with non-finite or tiny
// values (exponent field below 64) are added in FP64.
template <int N>
__device__ __forceinline__ double add_aligned(double acc, const double (&v)[N]) {
  static_assert(N <= 8, "three bits of headroom");
  int m = 0;
#pragma unroll
  for (int u = 0; u < N; ++u) m = max(m, __double2hiint(v[u]) & 0x7fffffff);
  const int em = m >> 20;
  if (em < 64 || em == 0x7ff) {
    int any = 0;
#pragma unroll
    for (int u = 0; u < N; ++u) any |= (__double2hiint(v[u]) & 0x7fffffff) | __double2loint(v[u]);
    if (any != 0) {
#pragma unroll
      for (int u = 0; u < N; ++u) acc += v[u];
    }
    return acc;
  }
  unsigned long long sum = 0;
  int neg = 0;
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const int hi = __double2hiint(v[u]), e = (hi & 0x7fffffff) >> 20, s = hi >> 31;
    unsigned long long x = ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 |
                            (unsigned)__double2loint(v[u])) << 7;
    const unsigned d = (unsigned)(em - e);
    asm("shr.u64 %0, %0, %1;" : "+l"(x) : "r"(d));  // 0 from 64 on (a zero has e = 0, d >= 64)
    sum += x ^ (unsigned long long)(long long)s;     // -x = ~x + 1 for the negative ones
    neg -= s;
  }
  const long long total = (long long)(sum + (unsigned)neg);
  return fma((double)total, __hiloint2double((em - 59) << 20, 0), acc);
}

// Sum of X over entries [beg, end) with stride `step`. Every batch of kGatherU
// entries, the last one too, issues its index loads and then its gathers
// together (predicated on the row end), so a short row costs one index latency
// and one gather latency per batch instead of a dependent pair per entry of its
// tail.
template <typename T, int K, int VW>
__device__ __forceinline__ void row_gather(const int32_t* __restrict__ col, int beg, int end, int step,
                                           const T* X, int lane_off, T (&acc)[VW]) {
  constexpr int U = kGatherU;
  for (int e = beg; e < end; e += U * step) {
    int j[U];
#pragma unroll
    for (int u = 0; u < U; ++u) j[u] = (e + u * step < end) ? __ldg(col + e + u * step) : -1;
    Pack<T, VW> a[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j[u] >= 0) {
        a[u] = ld_plain<T, VW>(X + (size_t)j[u] * K + lane_off);
      } else {
#pragma unroll
        for (int v = 0; v < VW; ++v) a[u].v[v] = T(0);
      }
    }
    if constexpr (sizeof(T) == 8) {
      if (end - e > 4 * step) {
#pragma unroll
        for (int v = 0; v < VW; ++v) {
          const double x[8] = {a[0].v[v], a[1].v[v], a[2].v[v], a[3].v[v], a[4].v[v], a[5].v[v], a[6].v[v], a[7].v[v]};
          acc[v] = add_aligned<8>(acc[v], x);
        }
      } else {
#pragma unroll
        for (int v = 0; v < VW; ++v) {
          const double x[4] = {a[0].v[v], a[1].v[v], a[2].v[v], a[3].v[v]};
          acc[v] = add_aligned<4>(acc[v], x);
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < VW; ++v) acc[v] += a[u].v[v];
    }
  }
}

// the same sums in FP64
template <int K, int VW>
__device__ __noinline__ void block_colsum_f64(const double* val, double* s_w, double* out) {
  constexpr int G = K / VW, NW = kPhaseBlock / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int v = 0; v < VW; ++v) {
    double a = val[v];
    for (int off = G; off < 32; off <<= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    if (lane < G) s_w[warp * K + lane * VW + v] = a;
  }
  __syncthreads();
  if (tid < K) {
    double t = s_w[tid];
    for (int w = 1; w < NW; ++w) t += s_w[w * K + tid];
    out[tid] = t;
  }
}

// CTA column sums of per-thread values (thread t owns columns (t % G) VW + v),
// column c at out[c]. FP32 values (or their double-float sums) are added in
// double-float, since the FP64 adds of a butterfly over 256 threads hold the
// SM's FP64 pipe for a thousand clocks; in FP64 where one of them is so large
// that the sum might leave FP32's range.
template <typename T, int K>
__device__ __forceinline__ void block_colsum_store(const typename CoopSum<T>::S (&val)[Cfg<T, K>::VW], double* out) {
  using C = Cfg<T, K>;
  using SM = CoopSum<T>;
  using S = typename SM::S;
  constexpr int VW = C::VW, G = C::G, NW = kPhaseBlock / 32;
  static_assert(sizeof(S) == 8, "the FP64 sums reuse the array");
  __shared__ __align__(8) S s_w[NW * K];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  S a[VW];
#pragma unroll
  for (int v = 0; v < VW; ++v) a[v] = val[v];
#pragma unroll
  for (int off = G; off < 32; off <<= 1)
#pragma unroll
    for (int v = 0; v < VW; ++v) a[v] = SM::add(a[v], SM::shfl(a[v], off));
  if (lane < G)
#pragma unroll
    for (int v = 0; v < VW; ++v) s_w[warp * K + lane * VW + v] = a[v];
  if constexpr (sizeof(T) == 4) {
    bool big = false;
#pragma unroll
    for (int v = 0; v < VW; ++v) big |= !(fabsf(SM::lead(val[v])) < 1e35f);
    if (__syncthreads_or(big)) {
      double d[VW];
#pragma unroll
      for (int v = 0; v < VW; ++v) d[v] = SM::out(val[v]);
      block_colsum_f64<K, VW>(d, reinterpret_cast<double*>(s_w), out);
      return;
    }
  } else {
    __syncthreads();
  }
  if (tid < K) {
    S t = s_w[tid];
#pragma unroll
    for (int w = 1; w < NW; ++w) t = SM::add(t, s_w[w * K + tid]);
    out[tid] = SM::out(t);
  }
}

// CTA column sums of per-thread partials written to part[blockIdx.x * K + c];
// then the last CTA to finish returns true (all partials visible to it).
template <typename T, int K>
__device__ __forceinline__ bool block_partials_last(const T (&val)[Cfg<T, K>::VW], double* part, unsigned* ticket) {
  constexpr int VW = Cfg<T, K>::VW;
  __shared__ int s_last;
  const int tid = threadIdx.x;
  typename CoopSum<T>::S a[VW];
#pragma unroll
  for (int v = 0; v < VW; ++v) a[v] = CoopSum<T>::from(val[v]);
  block_colsum_store<T, K>(a, part + (size_t)blockIdx.x * K);
  if (tid < K) __threadfence();
  __syncthreads();
  if (tid == 0) s_last = (atomicAdd(ticket, 1u) == gridDim.x - 1) ? 1 : 0;
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}

// Fixed-order sum over all CTAs' partials, by the last CTA: out[c] (shared).
// 16 loads in flight per thread and added pairwise: this tail is waited for by
// the whole grid (one dependent FP64 add takes some fifty clocks).
template <int K>
__device__ __forceinline__ void sum_partials(const double* part, int nblk, double* s_tmp, double* out) {
  constexpr int J = kPhaseBlock / K, W = 16;
  const int tid = threadIdx.x, c = tid % K, j = tid / K;
  double s = 0.0;
  for (int b = j; b < nblk; b += W * J) {
    double v[W];
#pragma unroll
    for (int u = 0; u < W; ++u) v[u] = b + u * J < nblk ? __ldcg(part + (size_t)(b + u * J) * K + c) : 0.0;
#pragma unroll
    for (int h = W / 2; h >= 1; h >>= 1)
#pragma unroll
      for (int u = 0; u < h; ++u) v[u] += v[u + h];
    s += v[0];
  }
  s_tmp[tid] = s;
  __syncthreads();
#pragma unroll
  for (int h = J / 2; h >= 1; h >>= 1) {
    if (j < h) s_tmp[tid] += s_tmp[tid + h * K];
    __syncthreads();
  }
  if (tid < K) out[tid] = s_tmp[tid];
  __syncthreads();
}

// ---------------------------------------------------------------- S phase
// SH: the solve carries the per-row diagonal a.dshift (a separate instance,
// so that the unshifted kernel carries no trace of it)
// X: x and p are updated here, in place (four vectors and no more: the entry
// that allocates nothing, and what is left of a stiff solve). Otherwise the residuals r_j of up to kHist
// iterations stay where they are, each in its own buffer, and x and p are formed
// from them afterwards (cg_x_phase): the pass then reads r and q and writes q,
// where it read and wrote x and p too (192 MB of vectors for 1e6 x 16 floats, not
// 448). Chung-Lu 1e6 x 16, shifted: S 165 -> 134 us, and 85 us per solve of nine
// iterations for x; what is left is the gathers, 24e6 sectors from L2 and L1.
// 3e5 x 16 doubles: 198 -> 159 us; R-MAT scale 17 x 64 floats: 176 -> 162 us. (With
// a CTA per row of more than 256 entries; with rows of up to 1400 by a warp each
// the three take 116, 144 and 102 us.)
// delta is (r, q) then, which is (p, q) as q = M p and p_{j-1} is M-orthogonal
// to p_j. Rounding leaves them so only while p is not much longer than r. Where M is
// close to singular (alpha rho near 1, a small shift) p grows, and (r, q) costs
// iterations that (p, q) does not: simulated in FP32 to 4e-6 on four graph
// families, at most a half more with |p|^2 below 1000 |r|^2 (11 -> 15, Chung-Lu, alpha rho =
// 0.99, right-hand side 1), beyond it two to ten times as many or no end (78 -> 508, Chung-Lu,
// 0.999, shift 0.01). So a solve that gets there goes on in the X form, and the next
// of its kind begins so (PhaseArgs::stiff, run_cg). The shift-and-invert solves of
// the 1e6-node graph at alpha = 1 / (1 + rho) stay below.
template <typename T, int K, bool SH = false, bool X = false>
__global__ void __launch_bounds__(kPhaseBlock, phase_min_blocks<T>()) cg_s_phase(PhaseArgs<T> a) {
  using C = Cfg<T, K>;
  constexpr int VW = C::VW, G = C::G, RPB = kPhaseBlock / G;  // rows per CTA pass
  __shared__ T s_red[kPhaseBlock / 32 * K];
  __shared__ double s_tmp[kPhaseBlock];
  __shared__ double s_out[K];
  CgState* st = a.st;
  if (!*(volatile int*)&st->active) return;
  const int tid = threadIdx.x, sl = tid % G, lane_off = sl * VW;
  const bool first = (st->iters == 0);
  const T ca = (T)a.ca, cA = (T)a.cA, cD = (T)a.cD;
  __shared__ T s_ab[2][K];
  if (tid < K) {
    s_ab[0][tid] = (T)st->alpha[tid];
    s_ab[1][tid] = (T)st->beta[tid];
  }
  __syncthreads();
  T dacc[VW];  // per-thread partials in the working precision (FP64 adds are scarce on this GPU)
#pragma unroll
  for (int v = 0; v < VW; ++v) dacc[v] = T(0);

  T* __restrict__ px = a.x;
  T* __restrict__ pp_ = a.p;
  T* __restrict__ pq = a.q;
  const T* __restrict__ pr = a.r;
  struct Own {
    Pack<T, VW> r, x, p, q;
  };
  // own-row r, loaded before the row's gathers so the two overlap
  auto own = [&](int64_t row) {
    Own o;
    const size_t off = (size_t)row * K + lane_off;
    o.r = ld_plain<T, VW>(pr + off);
    return o;
  };
  auto fin = [&](int64_t row, int deg, const T (&nb)[VW], const Own& w0) {
    const size_t o = (size_t)row * K + lane_off;
    Own w = w0;
    // the shift diagonal is loaded with x, p, q after the gathers: held
    // across them it costs the gather loop a register
    T dx = T(0);
    if constexpr (SH) dx = __ldg(a.dshift + row);
    if (!first) {
      if constexpr (X) {
        w.x = ld_plain<T, VW>(px + o);
        w.p = ld_plain<T, VW>(pp_ + o);
      }
      w.q = ld_last<T, VW>(pq + o);
    }
    const Pack<T, VW>& rr = w.r;
    Pack<T, VW> pp, qq;  // p, or r where p is not formed
    const T dg = (T)deg;
    // (M r) of column v; FP64: the row's diagonal first (one product fewer per column)
    T crow = T(0);
    if constexpr (sizeof(T) == 8) crow = SH ? ca + cD * dg + dx : ca + cD * dg;
    auto mr = [&](int v) {
      if constexpr (sizeof(T) == 8) {
        return crow * rr.v[v] + cA * nb[v];
      } else {
        T s = ca * rr.v[v] + cA * nb[v] + cD * dg * rr.v[v];
        if constexpr (SH) s += dx * rr.v[v];
        return s;
      }
    };
    if (first) {
#pragma unroll
      for (int v = 0; v < VW; ++v) {
        pp.v[v] = rr.v[v];
        qq.v[v] = mr(v);
      }
    } else {
#pragma unroll
      for (int v = 0; v < VW; ++v) {
        const T s = mr(v);
        const T be = s_ab[1][lane_off + v];
        pp.v[v] = rr.v[v];
        if constexpr (X) pp.v[v] += be * w.p.v[v];
        qq.v[v] = s + be * w.q.v[v];
      }
      if constexpr (X) {
        Pack<T, VW> xx = w.x;
#pragma unroll
        for (int v = 0; v < VW; ++v) xx.v[v] += s_ab[0][lane_off + v] * w.p.v[v];
        stp<T, VW>(px + o, xx);
      }
    }
#pragma unroll
    for (int v = 0; v < VW; ++v) dacc[v] += pp.v[v] * qq.v[v];
    if constexpr (X) stp<T, VW>(pp_ + o, pp);
    stp<T, VW>(pq + o, qq);
  };

  if ((int)blockIdx.x < a.g.nhub) {
    // one hub row per CTA: RPB lane groups stride over the entries
    const int64_t row = a.g.hubs[blockIdx.x];
    const int beg = a.g.row_ptr[row], end = a.g.row_ptr[row + 1];
    T acc[VW];
#pragma unroll
    for (int v = 0; v < VW; ++v) acc[v] = T(0);
    row_gather<T, K, VW>(a.g.col, beg + tid / G, end, RPB, a.r, lane_off, acc);
    // the lane groups' sums: within each warp by shuffles, then the warps
#pragma unroll
    for (int off = G; off < 32; off <<= 1)
#pragma unroll
      for (int v = 0; v < VW; ++v) acc[v] += __shfl_xor_sync(0xffffffffu, acc[v], off);
    if ((tid & 31) < G)
#pragma unroll
      for (int v = 0; v < VW; ++v) s_red[(tid >> 5) * K + lane_off + v] = acc[v];
    __syncthreads();
    if (tid < G) {
      const Own w = own(row);
      for (int wq = 1; wq < kPhaseBlock / 32; ++wq)
#pragma unroll
        for (int v = 0; v < VW; ++v) acc[v] += s_red[wq * K + lane_off + v];
      fin(row, end - beg, acc, w);
    }
  } else if ((int)blockIdx.x < a.g.nhub + a.g.nmid_blk) {
    // mid rows, one warp each: the 32 / G lane groups stride over the entries
    // and are combined by shuffles; lane group 0 finishes the row
    const int lane = tid & 31;
    constexpr int WPB = kPhaseBlock / 32;
    for (int r = ((int)blockIdx.x - a.g.nhub) * WPB + (tid >> 5); r < a.g.nmid; r += a.g.nmid_blk * WPB) {
      const int64_t row = a.g.mids[r];
      const int beg = a.g.row_ptr[row], end = a.g.row_ptr[row + 1];
      Own w;
      if (lane < G) w = own(row);
      T acc[VW];
#pragma unroll
      for (int v = 0; v < VW; ++v) acc[v] = T(0);
      row_gather<T, K, VW>(a.g.col, beg + lane / G, end, 32 / G, a.r, lane_off, acc);
#pragma unroll
      for (int off = G; off < 32; off <<= 1)
#pragma unroll
        for (int v = 0; v < VW; ++v) acc[v] += __shfl_xor_sync(0xffffffffu, acc[v], off);
      if (lane < G) fin(row, end - beg, acc, w);
    }
  } else {
    const int nlist = a.g.nhub + a.g.nmid_blk;
    const int lim = a.g.nmid_blk > 0 ? kMidDeg : kHubDeg;  // longer rows: hub CTAs or mid warps
    const int64_t nblk = (int64_t)gridDim.x - nlist;
    // E lane groups per row where a row has few lanes (K <= 2); not in FP64, where a
    // warp's operations of the row's end cost the same for eight rows as for 32
    constexpr int E = G >= 4 || sizeof(T) == 8 ? 1 : 4 / G, LPR = G * E, RPP = kPhaseBlock / LPR;
    const int e = (tid / G) % E;
    for (int64_t row = ((int64_t)blockIdx.x - nlist) * RPP + tid / LPR; row < a.g.n; row += nblk * RPP) {
      const int beg = a.g.row_ptr[row], end = a.g.row_ptr[row + 1];
      if (end - beg > lim) continue;
      Own w;
      if (e == 0) w = own(row);
      T acc[VW];
#pragma unroll
      for (int v = 0; v < VW; ++v) acc[v] = T(0);
      row_gather<T, K, VW>(a.g.col, beg + e, end, E, a.r, lane_off, acc);
      if constexpr (E > 1) {
        const unsigned m = ((1u << LPR) - 1u) << (tid & 31 & ~(LPR - 1));
#pragma unroll
        for (int off = G; off < LPR; off <<= 1)
#pragma unroll
          for (int v = 0; v < VW; ++v) acc[v] += __shfl_xor_sync(m, acc[v], off);
      }
      if (e == 0) fin(row, end - beg, acc, w);
    }
  }
  if (!block_partials_last<T, K>(dacc, a.part, &st->ticket)) return;
  // last CTA: delta -> alpha, breakdown checks
  sum_partials<K>(a.part, gridDim.x, s_tmp, s_out);
  if (tid < K) {
    const double delta = s_out[tid];
    if (!st->done[tid]) {
      if (!isfinite(delta)) {
        st->status[tid] = WL_ERR_NONFINITE; st->done[tid] = 1; st->alpha[tid] = 0.0;
      } else if (delta <= 0.0) {
        st->status[tid] = WL_ERR_NOT_SPD; st->done[tid] = 1; st->alpha[tid] = 0.0;
      } else {
        st->alpha[tid] = st->gamma[tid] / delta;
      }
    } else {
      st->alpha[tid] = 0.0;
    }
    if constexpr (!X) {
      a.hist->alpha[a.slot][tid] = st->alpha[tid];
      a.hist->beta[a.slot][tid] = st->beta[tid];
    }
  }
  if (tid == 0) {
    st->iters += 1;
    st->ticket = 0;
  }
}

// ---------------------------------------------------------------- U phase (and init)
// init = 1: gamma_0 = (r, r), convergence reference and flags, no update.
template <typename T, int K>
__global__ void __launch_bounds__(kPhaseBlock, phase_min_blocks<T>()) cg_u_phase(PhaseArgs<T> a, int init) {
  using C = Cfg<T, K>;
  constexpr int VW = C::VW, G = C::G;
  __shared__ double s_tmp[kPhaseBlock];
  __shared__ double s_out[K];
  CgState* st = a.st;
  if (!init && !*(volatile int*)&st->active) return;
  const int tid = threadIdx.x;
  const int mycol = (tid % G) * VW;  // kPhaseBlock * VW is a multiple of K
  T al[VW];
#pragma unroll
  for (int v = 0; v < VW; ++v) al[v] = init ? T(0) : (T)st->alpha[mycol + v];
  T acc[VW];
#pragma unroll
  for (int v = 0; v < VW; ++v) acc[v] = T(0);
  const size_t nv = (size_t)a.g.n * K / VW;
#pragma unroll 4
  for (size_t e = (size_t)blockIdx.x * kPhaseBlock + tid; e < nv; e += (size_t)gridDim.x * kPhaseBlock) {
    Pack<T, VW> rr;
    if (init) {
      rr = ld_plain<T, VW>(a.r + e * VW);
    } else {
      rr = ld_last<T, VW>(a.r + e * VW);
      const Pack<T, VW> qq = ld_plain<T, VW>(a.q + e * VW);
#pragma unroll
      for (int v = 0; v < VW; ++v) rr.v[v] -= al[v] * qq.v[v];
      stp<T, VW>(a.rn + e * VW, rr);
    }
#pragma unroll
    for (int v = 0; v < VW; ++v) acc[v] += rr.v[v] * rr.v[v];
  }
  if (!block_partials_last<T, K>(acc, a.part, &st->ticket)) return;
  __shared__ int s_stiff;
  if (tid == 0) s_stiff = 0;
  sum_partials<K>(a.part, gridDim.x, s_tmp, s_out);
  if (tid < K) {
    const double gn = s_out[tid];
    if (init) {
      st->pi[tid] = gn;
      const double b2 = a.bnorm2 ? a.bnorm2[tid] : gn;
      st->gamma[tid] = gn;
      st->b2[tid] = b2;
      st->alpha[tid] = 0.0;
      st->beta[tid] = 0.0;
      st->status[tid] = 0;
      int done = (b2 <= 0.0) || (gn <= a.tol2 * b2) || (a.skip && a.skip[tid]);
      if (!isfinite(gn)) { done = 1; st->status[tid] = WL_ERR_NONFINITE; }
      st->done[tid] = done;
    } else if (!st->done[tid]) {
      if (!isfinite(gn)) {
        st->status[tid] = WL_ERR_NONFINITE; st->done[tid] = 1; st->beta[tid] = 0.0;
      } else {
        const double be = gn / st->gamma[tid], pi = gn + be * be * st->pi[tid];
        st->beta[tid] = be;
        st->gamma[tid] = gn;
        st->pi[tid] = pi;
        if (gn <= a.tol2 * st->b2[tid]) {
          st->done[tid] = 1;
          st->beta[tid] = 0.0;
        } else if (a.stiff > 0.0 && pi > a.stiff * gn) {
          s_stiff = 1;
        }
      }
    } else {
      st->beta[tid] = 0.0;
    }
  }
  __syncthreads();
  if (tid == 0) {
    if (init) st->iters = 0;
    int any = 0;
    for (int c = 0; c < K; ++c) any |= !st->done[c];
    const int go = (any && st->iters < a.max_iter) ? 1 : 0;
    if (init) st->stiff = 0;
    if (go && s_stiff) st->stiff = 1;
    st->active = go && !(s_stiff && a.hist);
    st->ticket = 0;
  }
}

// x += alpha p: the deferred update of the last U phase
template <typename T, int K>
__global__ void __launch_bounds__(kPhaseBlock) cg_f_phase(PhaseArgs<T> a) {
  using C = Cfg<T, K>;
  constexpr int VW = C::VW, G = C::G;
  CgState* st = a.st;
  if (st->iters == 0) return;
  const int tid = threadIdx.x;
  const int mycol = (tid % G) * VW;
  T al[VW];
#pragma unroll
  for (int v = 0; v < VW; ++v) al[v] = (T)st->alpha[mycol + v];
  const size_t nv = (size_t)a.g.n * K / VW;
  for (size_t e = (size_t)blockIdx.x * kPhaseBlock + tid; e < nv; e += (size_t)gridDim.x * kPhaseBlock) {
    Pack<T, VW> xx = ld_plain<T, VW>(a.x + e * VW);
    const Pack<T, VW> pp = ld_plain<T, VW>(a.p + e * VW);
#pragma unroll
    for (int v = 0; v < VW; ++v) xx.v[v] += al[v] * pp.v[v];
    stp<T, VW>(a.x + e * VW, xx);
  }
}

// x and p from the kept residuals r[0..m): with p_i = r_i + beta_i p_{i-1},
//   sum_i alpha_i p_i = sum_i g_i r_i + beta_0 g_0 p_{-1},  g_i = alpha_i + beta_{i+1} g_{i+1}
// and p_{m-1} likewise with h_i = beta_{i+1} h_{i+1}, h_{m-1} = 1. One pass over
// them per kHist iterations or at the end of the solve, where x and p were read
// and written in every iteration.
template <typename T>
struct CgXArgs {
  const T* r[kHist];
  T* x;
  T* p;  // p_{-1} in (has_p), p_{m-1} out (flush)
  const CgHist* hist;
  const CgState* st;
  int64_t n;
  int m;
  int has_p;  // 0: p_{-1} = 0
  int add_x;  // 0: x is written, not read
  int flush;  // 1: the solve goes on: p too, nothing to do if it does not; 2: p too, without that look
};

template <typename T, int K>
__global__ void __launch_bounds__(kPhaseBlock) cg_x_phase(CgXArgs<T> a) {
  using C = Cfg<T, K>;
  constexpr int VW = C::VW, G = C::G;
  __shared__ T s_g[kHist + 1][K], s_h[kHist + 1][K];
  if (a.flush == 1 && !*(volatile const int*)&a.st->active) return;
  const int tid = threadIdx.x, m = a.m;
  if (tid < K) {
    T g = T(0), h = T(1), be = T(0);
    for (int i = m - 1; i >= 0; --i) {
      g = (T)a.hist->alpha[i][tid] + be * g;
      if (i < m - 1) h *= be;
      be = (T)a.hist->beta[i][tid];
      s_g[i][tid] = g;
      s_h[i][tid] = h;
    }
    s_g[kHist][tid] = be * g;
    s_h[kHist][tid] = be * h;
  }
  __syncthreads();
  const int mycol = (tid % G) * VW;
  const size_t nv = (size_t)a.n * K / VW;
  for (size_t e = (size_t)blockIdx.x * kPhaseBlock + tid; e < nv; e += (size_t)gridDim.x * kPhaseBlock) {
    Pack<T, VW> xx, pp;
#pragma unroll
    for (int v = 0; v < VW; ++v) xx.v[v] = pp.v[v] = T(0);
    if (a.add_x) xx = ld_last<T, VW>(a.x + e * VW);
    if (a.has_p) {
      const Pack<T, VW> p0 = ld_last<T, VW>(a.p + e * VW);
#pragma unroll
      for (int v = 0; v < VW; ++v) {
        xx.v[v] += s_g[kHist][mycol + v] * p0.v[v];
        pp.v[v] = s_h[kHist][mycol + v] * p0.v[v];
      }
    }
    for (int i0 = 0; i0 < m; i0 += 4) {
      Pack<T, VW> rr[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + u < m) rr[u] = ld_last<T, VW>(a.r[i0 + u] + e * VW);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + u < m) {
#pragma unroll
          for (int v = 0; v < VW; ++v) {
            xx.v[v] += s_g[i0 + u][mycol + v] * rr[u].v[v];
            if (a.flush) pp.v[v] += s_h[i0 + u][mycol + v] * rr[u].v[v];
          }
        }
    }
    stp<T, VW>(a.x + e * VW, xx);
    if (a.flush) stp<T, VW>(a.p + e * VW, pp);
  }
}

// ---------------------------------------------------------------- FP64 residual
// Start of an FP64-form solve from a warm start x: r = b - M x, column norms
// ||r||^2 -> st->gamma and ||b||^2 -> st->b2 (last CTA).
struct ResPhaseArgs {
  PhaseGraph g;
  const double* x;
  const double* b;  // NULL: b = 0 (then r = -M x)
  double* r;
  double ca, cA, cD;
  double* part;  // 2 * gridDim.x * K
  CgState* st;
};

template <int K>
__global__ void __launch_bounds__(kPhaseBlock, kPhaseMinBlocks) res_phase(ResPhaseArgs a) {
  using C = Cfg<double, K>;
  constexpr int VW = C::VW, G = C::G, RPB = kPhaseBlock / G;
  __shared__ double s_red[kPhaseBlock / 32 * K];
  __shared__ double s_tmp[kPhaseBlock];
  __shared__ double s_out[K];
  const int tid = threadIdx.x, sl = tid % G, lane_off = sl * VW;
  const double ca = a.ca, cA = a.cA, cD = a.cD;
  double racc[2 * VW];  // (r, r) then (b, b)
#pragma unroll
  for (int v = 0; v < 2 * VW; ++v) racc[v] = 0.0;
  auto fin = [&](int64_t row, int deg, const double (&nb)[VW]) {
    const size_t o = (size_t)row * K + lane_off;
    const Pack<double, VW> xx = ld_plain<double, VW>(a.x + o);
    Pack<double, VW> bb;
    if (a.b) {
      bb = ld_plain<double, VW>(a.b + o);
    } else {
#pragma unroll
      for (int v = 0; v < VW; ++v) bb.v[v] = 0.0;
    }
    Pack<double, VW> rr;
#pragma unroll
    for (int v = 0; v < VW; ++v) {
      rr.v[v] = bb.v[v] - (ca * xx.v[v] + cA * nb[v] + cD * (double)deg * xx.v[v]);
      racc[v] += rr.v[v] * rr.v[v];
      racc[VW + v] += bb.v[v] * bb.v[v];
    }
    stp<double, VW>(a.r + o, rr);
  };
  if ((int)blockIdx.x < a.g.nhub) {
    const int64_t row = a.g.hubs[blockIdx.x];
    const int beg = a.g.row_ptr[row], end = a.g.row_ptr[row + 1];
    double acc[VW];
#pragma unroll
    for (int v = 0; v < VW; ++v) acc[v] = 0.0;
    row_gather<double, K, VW>(a.g.col, beg + tid / G, end, RPB, a.x, lane_off, acc);
#pragma unroll
    for (int off = G; off < 32; off <<= 1)
#pragma unroll
      for (int v = 0; v < VW; ++v) acc[v] += __shfl_xor_sync(0xffffffffu, acc[v], off);
    if ((tid & 31) < G)
#pragma unroll
      for (int v = 0; v < VW; ++v) s_red[(tid >> 5) * K + lane_off + v] = acc[v];
    __syncthreads();
    if (tid < G) {
      for (int wq = 1; wq < kPhaseBlock / 32; ++wq)
#pragma unroll
        for (int v = 0; v < VW; ++v) acc[v] += s_red[wq * K + lane_off + v];
      fin(row, end - beg, acc);
    }
  } else {
    const int64_t nblk = (int64_t)gridDim.x - a.g.nhub;
    for (int64_t row = ((int64_t)blockIdx.x - a.g.nhub) * RPB + tid / G; row < a.g.n; row += nblk * RPB) {
      const int beg = a.g.row_ptr[row], end = a.g.row_ptr[row + 1];
      if (end - beg > kHubDeg) continue;
      double acc[VW];
#pragma unroll
      for (int v = 0; v < VW; ++v) acc[v] = 0.0;
      row_gather<double, K, VW>(a.g.col, beg, end, 1, a.x, lane_off, acc);
      fin(row, end - beg, acc);
    }
  }
  double rp[VW], bp[VW];
#pragma unroll
  for (int v = 0; v < VW; ++v) {
    rp[v] = racc[v];
    bp[v] = racc[VW + v];
  }
  // two partial sets: (r, r) in part[0 .. G K), (b, b) in part[G K .. 2 G K)
  double* part_b = a.part + (size_t)gridDim.x * K;
  {
    using CC = Cfg<double, K>;
    constexpr int NW = kPhaseBlock / 32;
    __shared__ double s_w[2 * NW * K];
    const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int off = CC::G; off < 32; off <<= 1)
#pragma unroll
      for (int v = 0; v < VW; ++v) {
        rp[v] += __shfl_xor_sync(0xffffffffu, rp[v], off);
        bp[v] += __shfl_xor_sync(0xffffffffu, bp[v], off);
      }
    if (lane < CC::G)
#pragma unroll
      for (int v = 0; v < VW; ++v) {
        s_w[warp * K + lane * VW + v] = rp[v];
        s_w[NW * K + warp * K + lane * VW + v] = bp[v];
      }
    __syncthreads();
    if (tid < K) {
      double t = 0.0, u = 0.0;
      for (int w = 0; w < NW; ++w) {
        t += s_w[w * K + tid];
        u += s_w[NW * K + w * K + tid];
      }
      a.part[(size_t)blockIdx.x * K + tid] = t;
      part_b[(size_t)blockIdx.x * K + tid] = u;
      __threadfence();
    }
    __syncthreads();
  }
  __shared__ int s_last;
  if (tid == 0) s_last = (atomicAdd(&a.st->ticket, 1u) == gridDim.x - 1) ? 1 : 0;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  sum_partials<K>(a.part, gridDim.x, s_tmp, s_out);
  if (tid < K) a.st->gamma[tid] = s_out[tid];
  sum_partials<K>(part_b, gridDim.x, s_tmp, s_out);
  if (tid < K) a.st->b2[tid] = s_out[tid];
  if (tid == 0) a.st->ticket = 0;
}

}  // namespace wl
