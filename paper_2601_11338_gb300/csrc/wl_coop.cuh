// Lockstep conjugate gradients as one cooperative kernel per solve, for
// problems whose CG vectors fit in the SMs' shared memory (Sec. 4.2, the
// iteration of wl_cg2.cuh). A solve of this size is bound by latency: by the
// launches, the reductions and the host reads between the phase kernels, not
// by its traffic. Here every row belongs to one CTA for the whole solve;
// x, p, q and r of the CTA's rows stay in its shared memory and only r is
// also written to global memory, where the gathers read it (through L2: other
// SMs rewrite it between grid barriers). One iteration is
//   s = M r ; p = r + beta p ; q = s + beta q ; delta = (p, q) | barrier
//   x += alpha p ; r -= alpha q ; gamma' = (r, r)              | barrier
// with the column sums of all CTAs added by every CTA in the same fixed order
// after each barrier (deterministic, no broadcast), and no host read until
// the solve has ended.
//
// Rows: LPR = G * E lanes per row of up to kMidDeg entries (G lanes of 16
// bytes, E of them along the entries, E > 1 where G is small so that a
// quarter of a warp works on each row), a warp per row of the mid list, and a
// warp or, for very long rows, the CTA per row of the hub list.
//
// Measured per call against the phase kernels (start -> here): walk degrees and
// four columns in FP64, n = 2000: 1390 -> 428 us; 13 refined columns, n = 20011:
// 2520 -> 947 us; walk degrees of R-MAT scale 20 (refined): 4.1 -> 2.9 ms; 132
// refined shifted solves of 62500 x 32: 377 -> 214 ms. An iteration of the last
// takes 25 us; the phase kernels' two launches took 43.
#pragma once
#include <algorithm>

#include "wl_cg2.cuh"
#include "wl_df.cuh"

namespace wl {

constexpr int kCoopHubWarp = 2048;  // hub rows of up to this many entries are taken by a warp

template <typename T, int K>
struct CoopCfg {
  using C = Cfg<T, K>;
  static constexpr int VW = C::VW, G = C::G;
  static constexpr int E = G >= 4 ? 1 : 4 / G;
  static constexpr int LPR = G * E;
  static constexpr int SLOT = VW * (int)sizeof(T);                          // bytes of one lane's part of a vector
  static constexpr int CH = (32 / (K * (int)sizeof(T))) > 1 ? 32 / (K * (int)sizeof(T)) : 1;  // consecutive rows of a CTA
  static constexpr int U = sizeof(T) == 4 ? 8 : 4;                          // gathers in flight per lane
  // most threads of a CTA (one per SM); FP64: its sums hold the FP64 pipe for a microsecond at 512 already
  static constexpr int TMAX = sizeof(T) == 4 ? 1024 : 512;
  // shared memory left for the vectors: 227 KB less the static arrays
  static constexpr size_t SMEM = 227 * 1024 - (32 * K * 8 + K * (24 + 2 * (int)sizeof(T) + 8) + 256);
};

// Arrivals counted up over the launch (cleared before it) and an error word.
// A barrier is one release-add and a poll: no reset, no generation word and
// no second look at memory (the general grid_sync reads, adds and reads again:
// 4 us against 1.5 us here). Bounded like it.
struct CoopBar {
  unsigned count;
  int err;
};

template <typename T>
struct CoopArgs {
  PhaseArgs<T> a;  // a.g carries the mid list (nmid > 0: rows above kMidDeg are on it)
  CoopBar* bar;
  int nhead;             // K = 1: leading entries of r kept in shared memory
  const T* r0;           // the starting residual (a.r itself, or read only: a.r is then scratch)
  const double* gamma0;  // its column norms |r0|^2; NULL: computed here
  int add_x;             // 1: x holds a start value, the correction is added to it; 0: x is written
};

// slots (lane parts) of one vector in a CTA's shared memory
__host__ __device__ inline int64_t coop_rows_local(int64_t n, int grid, int ch) {
  return ((n + ch - 1) / ch + grid - 1) / grid * ch;
}

// sum type of the reductions: double-float for FP32 (error-free adds with
// FP32 instructions; FP64 adds run at 1/64 of their rate), FP64 for FP64
template <typename T>
struct CoopSum;
template <>
struct CoopSum<float> {
  using S = float2;
  static __device__ __forceinline__ S from(float v) { return make_float2(v, 0.f); }
  static __device__ __forceinline__ S add(S a, S b) {
    const df t = df_add(df{a.x, a.y}, df{b.x, b.y});
    return make_float2(t.hi, t.lo);
  }
  static __device__ __forceinline__ S shfl(S a, int off) {
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, off), __shfl_xor_sync(0xffffffffu, a.y, off));
  }
  static __device__ __forceinline__ S zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ double out(S a) { return (double)a.x + (double)a.y; }
};
template <>
struct CoopSum<double> {
  using S = double;
  static __device__ __forceinline__ S from(double v) { return v; }
  static __device__ __forceinline__ S add(S a, S b) { return a + b; }
  static __device__ __forceinline__ S shfl(S a, int off) { return __shfl_xor_sync(0xffffffffu, a, off); }
  static __device__ __forceinline__ S zero() { return 0.0; }
  static __device__ __forceinline__ double out(S a) { return a; }
};

__device__ __forceinline__ bool coop_sync(CoopBar* b, unsigned target) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&b->count) : "memory");
    uint64_t t0 = 0;
    for (unsigned polls = 1; (int)(ld_acquire(&b->count) - target) < 0; ++polls) {
      if ((polls & 1023u) != 0u) continue;
      if (t0 == 0) t0 = globaltimer_ns();
      if (*(volatile int*)&b->err != 0) {  // another CTA gave up: leave too
        ok = 0;
        break;
      }
      if (globaltimer_ns() - t0 > kWaitLimitNs) {
        atomicExch(&b->err, WL_ERR_TIMEOUT);
        ok = 0;
        break;
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Sum of X over entries [beg, end) with stride `step`. The loads may hit L1:
// the barrier's acquire orders them after the other SMs' writes. K = 1:
// entries below nhead come from their copy in shared memory.
template <typename T, int K, int VW, int U>
__device__ __forceinline__ void coop_gather(const int32_t* __restrict__ col, int beg, int end, int step, const T* X,
                                            const T* head, int nhead, int lane_off, T (&acc)[VW]) {
  for (int e = beg; e < end; e += U * step) {
    int j[U];
#pragma unroll
    for (int u = 0; u < U; ++u) j[u] = (e + u * step < end) ? __ldg(col + e + u * step) : -1;
    Pack<T, VW> v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (K == 1 && (unsigned)j[u] < (unsigned)nhead) {
        v[u].v[0] = head[j[u]];
      } else if (j[u] >= 0) {
        v[u] = ld_plain<T, VW>(X + (size_t)j[u] * K + lane_off);
      } else {
#pragma unroll
        for (int w = 0; w < VW; ++w) v[u].v[w] = T(0);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int w = 0; w < VW; ++w) acc[w] += v[u].v[w];
  }
}

template <typename T, int K, bool SH>
__global__ void __launch_bounds__(CoopCfg<T, K>::TMAX, 1) cg_coop(CoopArgs<T> ca_) {
  using CC = CoopCfg<T, K>;
  using SM = CoopSum<T>;
  using S = typename SM::S;
  constexpr int VW = CC::VW, G = CC::G, E = CC::E, LPR = CC::LPR, CH = CC::CH, U = CC::U;
  using P = Pack<T, VW>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ S s_w[32 * K];
  __shared__ double s_sum[K];
  __shared__ T s_al[K], s_be[K];
  __shared__ double s_gamma[K], s_b2[K];
  __shared__ int s_done[K], s_stat[K];
  __shared__ int s_any;
  const PhaseArgs<T>& a = ca_.a;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
  const int b = blockIdx.x, grid = gridDim.x;
  const int sl = tid % G, lane_off = sl * VW;
  const int nloc = (int)coop_rows_local(a.g.n, grid, CH);
  const int lim = a.g.nmid > 0 ? kMidDeg : kHubDeg;
  const int nmid_l = a.g.nmid > b ? (a.g.nmid - b + grid - 1) / grid : 0;
  const int nhub_l = a.g.nhub > b ? (a.g.nhub - b + grid - 1) / grid : 0;
  // slots: short rows, mid rows, hub rows
  const int mid0 = nloc * G;
  const int hub0 = mid0 + (a.g.nmid + grid - 1) / grid * G;
  const int nslot = hub0 + (a.g.nhub + grid - 1) / grid * G;
  P* sx = reinterpret_cast<P*>(smem_raw);
  P* sp = sx + nslot;
  P* sq = sp + nslot;
  P* sr = sq + nslot;
  T* s_head = reinterpret_cast<T*>(sr + nslot);
  const int nhead = K == 1 ? ca_.nhead : 0;
  const int32_t* __restrict__ rp = a.g.row_ptr;
  const int32_t* __restrict__ col = a.g.col;
  auto row_of = [&](int lr) -> int64_t { return ((int64_t)(lr / CH) * grid + b) * CH + lr % CH; };
  // f(slot, row) for every slot of this thread's columns
  auto for_slots = [&](auto f) {
    for (int s = tid; s < mid0; s += nthr) {
      const int64_t row = row_of(s / G);
      if (row >= a.g.n) continue;
      if (__ldg(rp + row + 1) - __ldg(rp + row) > lim) continue;
      f(s, row);
    }
    for (int s = tid; s < nmid_l * G; s += nthr) f(mid0 + s, (int64_t)__ldg(a.g.mids + (s / G) * grid + b));
    for (int s = tid; s < nhub_l * G; s += nthr) f(hub0 + s, (int64_t)__ldg(a.g.hubs + (s / G) * grid + b));
  };
  S* part = reinterpret_cast<S*>(a.part);
  unsigned target = 0;  // arrivals at the next barrier
  if (*(volatile int*)&ca_.bar->err != 0) return;  // set before the launch: every CTA leaves
  // sums the threads' values over the grid: column c in s_sum[c] on return;
  // `half` alternates the buffers of successive calls
  auto grid_sum = [&](const T (&val)[VW], int half) -> bool {
    S v[VW];
#pragma unroll
    for (int w = 0; w < VW; ++w) v[w] = SM::from(val[w]);
#pragma unroll
    for (int off = G; off < 32; off <<= 1)
#pragma unroll
      for (int w = 0; w < VW; ++w) v[w] = SM::add(v[w], SM::shfl(v[w], off));
    if (lane < G)
#pragma unroll
      for (int w = 0; w < VW; ++w) s_w[warp * K + lane * VW + w] = v[w];
    __syncthreads();
    S* p = part + (size_t)half * grid * K;
    if (tid < (K * 4 < 32 ? 32 : K * 4)) {  // four lanes per column add the warps' sums (whole warps shuffle)
      S t = SM::zero();
      if (tid < K * 4)
        for (int w = tid & 3; w < nwarp; w += 4) t = SM::add(t, s_w[w * K + (tid >> 2)]);
      t = SM::add(t, SM::shfl(t, 1));
      t = SM::add(t, SM::shfl(t, 2));
      if ((tid & 3) == 0 && tid < K * 4) {
        p[(size_t)b * K + (tid >> 2)] = t;
      }
    }
    target += grid;
    if (!coop_sync(ca_.bar, target)) return false;
    // J consecutive lanes per column over the CTAs' sums
    int J = 32;
    while (J * K > nthr) J >>= 1;
    const int c = tid / J, j = tid % J;
    if (tid < K * J) {
      S t = SM::zero();
#pragma unroll 4
      for (int g = j; g < grid; g += J) t = SM::add(t, __ldcg(p + (size_t)g * K + c));
      for (int off = 1; off < J; off <<= 1) t = SM::add(t, SM::shfl(t, off));
      if (j == 0) s_sum[c] = SM::out(t);
    }
    __syncthreads();
    return true;
  };
  const T ca = (T)a.ca, cA = (T)a.cA, cD = (T)a.cD;
  CgState* st = a.st;
  T acc[VW];
  auto zero_acc = [&] {
#pragma unroll
    for (int w = 0; w < VW; ++w) acc[w] = T(0);
  };
  // start: r into shared memory, x = 0, norms
  zero_acc();
  for_slots([&](int s, int64_t row) {
    const P r = ldp<T, VW>(ca_.r0 + (size_t)row * K + lane_off);
    sr[s] = r;
    P z;
#pragma unroll
    for (int w = 0; w < VW; ++w) {
      z.v[w] = T(0);
      acc[w] += r.v[w] * r.v[w];
    }
    sx[s] = z;
  });
  int half = 0;
  if (!ca_.gamma0) {
    if (!grid_sum(acc, half)) return;
    half ^= 1;
  } else {
    if (tid < K) s_sum[tid] = ca_.gamma0[tid];
    __syncthreads();
  }
  if (tid == 0) s_any = 0;
  __syncthreads();
  if (tid < K) {
    const double gn = s_sum[tid], b2 = !ca_.gamma0 && a.bnorm2 ? a.bnorm2[tid] : gn;
    int done = !(b2 > 0.0) || (!ca_.gamma0 && gn <= a.tol2 * b2) || (a.skip && a.skip[tid]), status = 0;
    if (!isfinite(gn)) { done = 1; status = WL_ERR_NONFINITE; }
    s_gamma[tid] = gn;
    s_b2[tid] = b2;
    s_done[tid] = done;
    s_stat[tid] = status;
    s_be[tid] = T(0);
    if (!done) s_any = 1;
  }
  __syncthreads();
  int iters = 0;
  bool active = s_any != 0 && a.max_iter > 0;
  while (active) {
    // ---- S: s = M r, p, q, delta
    const bool first = iters == 0;
    const T* rsrc = first ? ca_.r0 : a.r;
    zero_acc();
    if (K == 1 && nhead > 0) {
      for (int i = tid; i < nhead; i += nthr) s_head[i] = ldp<T, 1>(rsrc + i).v[0];
      __syncthreads();
    }
    auto fin = [&](int s, int64_t row, int deg, const T (&nb)[VW]) {
      const P r = sr[s];
      P pp, qq;
      if (!first) {
        pp = sp[s];
        qq = sq[s];
      }
      const T dg = (T)deg;
      T dx = T(0);
      if constexpr (SH) dx = __ldg(a.dshift + row);
#pragma unroll
      for (int w = 0; w < VW; ++w) {
        T v = ca * r.v[w] + cA * nb[w] + cD * dg * r.v[w];
        if constexpr (SH) v += dx * r.v[w];
        if (first) {
          pp.v[w] = r.v[w];
          qq.v[w] = v;
        } else {
          const T be = s_be[lane_off + w];
          pp.v[w] = r.v[w] + be * pp.v[w];
          qq.v[w] = v + be * qq.v[w];
        }
        acc[w] += pp.v[w] * qq.v[w];
      }
      sp[s] = pp;
      sq[s] = qq;
    };
    // long hub rows by the whole CTA
    for (int h = 0; h < nhub_l; ++h) {
      const int64_t row = __ldg(a.g.hubs + h * grid + b);
      const int beg = __ldg(rp + row), end = __ldg(rp + row + 1);
      if (end - beg <= kCoopHubWarp) continue;
      T nb[VW];
#pragma unroll
      for (int w = 0; w < VW; ++w) nb[w] = T(0);
      coop_gather<T, K, VW, U>(col, beg + tid / G, end, nthr / G, rsrc, s_head, nhead, lane_off, nb);
#pragma unroll
      for (int off = G; off < 32; off <<= 1)
#pragma unroll
        for (int w = 0; w < VW; ++w) nb[w] += __shfl_xor_sync(0xffffffffu, nb[w], off);
      T* s_t = reinterpret_cast<T*>(s_w);  // one value per warp and column fits
      __syncthreads();
      if (lane < G)
#pragma unroll
        for (int w = 0; w < VW; ++w) s_t[warp * K + lane_off + w] = nb[w];
      __syncthreads();
      if (tid < G) {
#pragma unroll
        for (int w = 0; w < VW; ++w) {
          nb[w] = T(0);
          for (int q = 0; q < nwarp; ++q) nb[w] += s_t[q * K + lane_off + w];
        }
        fin(hub0 + h * G + sl, row, end - beg, nb);
      }
      __syncthreads();  // s_w is free again
    }
    // mid rows and shorter hub rows, a warp each
    for (int m = warp; m < nmid_l + nhub_l; m += nwarp) {
      const bool hub = m >= nmid_l;
      const int64_t row = hub ? __ldg(a.g.hubs + (m - nmid_l) * grid + b) : __ldg(a.g.mids + m * grid + b);
      const int beg = __ldg(rp + row), end = __ldg(rp + row + 1);
      if (hub && end - beg > kCoopHubWarp) continue;
      T nb[VW];
#pragma unroll
      for (int w = 0; w < VW; ++w) nb[w] = T(0);
      coop_gather<T, K, VW, U>(col, beg + lane / G, end, 32 / G, rsrc, s_head, nhead, lane_off, nb);
#pragma unroll
      for (int off = G; off < 32; off <<= 1)
#pragma unroll
        for (int w = 0; w < VW; ++w) nb[w] += __shfl_xor_sync(0xffffffffu, nb[w], off);
      if (lane < G) fin((hub ? hub0 + (m - nmid_l) * G : mid0 + m * G) + sl, row, end - beg, nb);
    }
    // short rows, LPR lanes each (whole warps stay in the loop for the shuffles)
    for (int u0 = warp * 32; u0 < nloc * LPR; u0 += nthr) {
      const int u = u0 + lane, lr = u / LPR, e = (u / G) % E;
      const int64_t row = row_of(lr);
      int beg = 0, end = 0;
      bool live = lr < nloc && row < a.g.n;
      if (live) {
        beg = __ldg(rp + row);
        end = __ldg(rp + row + 1);
        live = end - beg <= lim;
      }
      T nb[VW];
#pragma unroll
      for (int w = 0; w < VW; ++w) nb[w] = T(0);
      if (live) coop_gather<T, K, VW, U>(col, beg + e, end, E, rsrc, s_head, nhead, lane_off, nb);
      if constexpr (E > 1) {
#pragma unroll
        for (int off = G; off < LPR; off <<= 1)
#pragma unroll
          for (int w = 0; w < VW; ++w) nb[w] += __shfl_xor_sync(0xffffffffu, nb[w], off);
      }
      if (live && e == 0) fin(lr * G + sl, row, end - beg, nb);
    }
    if (!grid_sum(acc, half)) return;
    half ^= 1;
    ++iters;
    if (tid < K) {
      const double delta = s_sum[tid];
      double al = 0.0;
      if (!s_done[tid]) {
        if (!isfinite(delta)) {
          s_stat[tid] = WL_ERR_NONFINITE; s_done[tid] = 1;
        } else if (delta <= 0.0) {
          s_stat[tid] = WL_ERR_NOT_SPD; s_done[tid] = 1;
        } else {
          al = s_gamma[tid] / delta;
        }
      }
      s_al[tid] = (T)al;
    }
    if (tid == 0) s_any = 0;
    __syncthreads();
    // ---- U: x += alpha p, r -= alpha q, gamma'
    zero_acc();
    for_slots([&](int s, int64_t row) {
      const P pp = sp[s], qq = sq[s];
      P xx = sx[s], rr = sr[s];
#pragma unroll
      for (int w = 0; w < VW; ++w) {
        const T al = s_al[lane_off + w];
        xx.v[w] += al * pp.v[w];
        rr.v[w] -= al * qq.v[w];
        acc[w] += rr.v[w] * rr.v[w];
      }
      sx[s] = xx;
      sr[s] = rr;
      stp<T, VW>(a.r + (size_t)row * K + lane_off, rr);
    });
    if (!grid_sum(acc, half)) return;
    half ^= 1;
    if (tid < K) {
      const double gn = s_sum[tid];
      double be = 0.0;
      if (!s_done[tid]) {
        if (!isfinite(gn)) {
          s_stat[tid] = WL_ERR_NONFINITE; s_done[tid] = 1;
        } else {
          be = gn / s_gamma[tid];
          s_gamma[tid] = gn;
          if (gn <= a.tol2 * s_b2[tid]) {
            s_done[tid] = 1;
            be = 0.0;
          }
        }
      }
      s_be[tid] = (T)be;
      if (!s_done[tid]) s_any = 1;
    }
    __syncthreads();
    active = s_any != 0 && iters < a.max_iter;
  }
  // x, and the solve's state for the host
  for_slots([&](int s, int64_t row) {
    T* px = a.x + (size_t)row * K + lane_off;
    P xx = sx[s];
    if (ca_.add_x) {
      const P x0 = ldp<T, VW>(px);
#pragma unroll
      for (int w = 0; w < VW; ++w) xx.v[w] += x0.v[w];
    }
    stp<T, VW>(px, xx);
    if (iters == 0 && ca_.r0 != a.r) stp<T, VW>(a.r + (size_t)row * K + lane_off, sr[s]);
  });
  if (b == 0) {
    if (tid < K) {
      st->gamma[tid] = s_gamma[tid];
      st->b2[tid] = s_b2[tid];
      st->done[tid] = s_done[tid];
      st->status[tid] = s_stat[tid];
    }
    if (tid == 0) {
      st->iters = iters;
      st->active = 0;
    }
  }
}

// ---------------------------------------------------------------- launch shape
struct CoopShape {
  int grid = 0, threads = 0, nhead = 0;
  size_t smem = 0;
};

// The launch of a solve with K columns, or false where its vectors don't fit.
template <typename T, int K>
bool cgc_shape(const PhaseGraph& g, int64_t nnz, int sms, CoopShape* sh) {
  using CC = CoopCfg<T, K>;
  // 256 lane units (rows x LPR) per CTA until every SM has one (each CTA adds
  // to the reductions), then more threads, evenly over the passes of the row loop
  const int64_t units = g.n * CC::LPR;
  sh->grid = (int)std::max<int64_t>(1, std::min<int64_t>(sms, (units + 255) / 256));
  const int64_t rows = coop_rows_local(g.n, sh->grid, CC::CH);
  const int64_t passes = (rows * CC::LPR + CC::TMAX - 1) / CC::TMAX;
  sh->threads = (int)std::max<int64_t>(std::max(256, 4 * K), (rows * CC::LPR / passes + 31) / 32 * 32);
  const int64_t nslot = (rows + (g.nmid + sh->grid - 1) / sh->grid + (g.nhub + sh->grid - 1) / sh->grid) * CC::G;
  if (nslot > (int64_t)(CC::SMEM / (4 * CC::SLOT))) return false;
  sh->smem = (size_t)nslot * 4 * CC::SLOT;
  // K = 1: the leading entries of r (the hubs, when the nodes are ordered by
  // degree) as far as they fit and are worth their load
  sh->nhead = 0;
  if (K == 1) {
    sh->nhead = (int)std::min<int64_t>({g.n, nnz / (4 * sh->grid), (int64_t)((CC::SMEM - sh->smem) / sizeof(T))});
    sh->smem += (size_t)sh->nhead * sizeof(T);
  }
  return true;
}

template <typename T, int K, bool SH>
cudaError_t cgc_launch(CoopArgs<T> a, const CoopShape& sh, cudaStream_t s) {
  static const cudaError_t attr =
      cudaFuncSetAttribute(cg_coop<T, K, SH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)CoopCfg<T, K>::SMEM);
  if (attr != cudaSuccess) return attr;
  a.nhead = sh.nhead;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel((const void*)cg_coop<T, K, SH>, dim3(sh.grid), dim3(sh.threads), args, sh.smem, s);
}

}  // namespace wl
