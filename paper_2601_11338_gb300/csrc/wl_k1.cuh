// Products with A for one column (K = 1): walk degrees, spectral searches.
//
// A gathered value of one column is 4 or 8 bytes of a 32-byte sector, and an SM
// takes scattered sectors from L2 at about one in two clocks whatever is read
// of them (measured: 0.52 per clock and SM, occupancy and bytes in flight
// changed nothing), so these kernels are bound by the number of gathers that
// leave the SM. One CTA per SM therefore spends its shared memory on the
// leading entries of the gathered vector (the hubs, when the nodes are ordered
// by degree: 48000 of R-MAT's million nodes take three quarters of the
// gathers) and keeps everything else in global memory, where it is streamed.
// Index reads are coalesced: a warp takes 32 consecutive short rows, whose
// entries lie one after the other, a lane per entry, and adds the rows up from
// shared memory; rows of the mid list take eight lanes each, hub rows a warp,
// the longest the CTA.
// R-MAT scale 20, FP32 CG: 875 -> 770 us a solve against the kernel that keeps the
// vectors in shared memory (wl_coop.cuh) and its residual 257 -> 147 us; FP64,
// where they don't fit, 5.2 -> 2.2 ms a call against the phase kernels. Smaller
// graphs gain less from the head than the streamed vectors cost.
#pragma once
#include "wl_coop.cuh"
#include "wl_res.cuh"

namespace wl {

// threads of the one CTA per SM: as many as the registers of eight gathers in flight allow
template <typename V>
__host__ __device__ constexpr int k1_threads() { return sizeof(V) == 4 ? 1024 : 640; }
constexpr int kK1Chunk = 128;      // entries a warp stages at a time
constexpr int kK1Long = 4096;      // longer rows: the whole CTA
constexpr int kK1MaxLong = 64;     // of them per CTA; further ones by a warp
constexpr int kK1Lim = kMidDeg;    // longest row of the streamed groups when there is a mid list
constexpr size_t kK1Smem = 227 * 1024 - 4096;

template <typename V>
__host__ inline size_t k1_smem(int nhead) {
  return ((size_t)nhead + (size_t)(k1_threads<V>() / 32) * kK1Chunk) * sizeof(V);
}

// CTAs of a launch: one per SM, fewer where a CTA would get less than eight groups of 32 rows
__host__ inline int k1_grid(int64_t n, int sms) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(((n + 31) / 32 + 7) / 8, sms));
}
// entries of the gathered vector that fit beside the stage and are worth their
// load: it takes a CTA as long as a tenth of its gathers when it has a quarter of their number
template <typename V>
__host__ inline int k1_head(int64_t n, int64_t nnz, int grid) {
  const size_t stage = (size_t)(k1_threads<V>() / 32) * kK1Chunk * sizeof(V);
  return (int)std::min<int64_t>({n, nnz / (4 * grid), (int64_t)((kK1Smem - stage) / sizeof(V))}) & ~3;
}

// the head of X into shared memory, 16 bytes at a time (X 16-byte aligned)
template <typename V>
__device__ __forceinline__ void k1_load_head(const V* X, V* head, int nhead) {
  const int4* src = reinterpret_cast<const int4*>(X);
  int4* dst = reinterpret_cast<int4*>(head);
  const int n4 = (int)((size_t)nhead * sizeof(V) / 16);
#pragma unroll 4
  for (int i = threadIdx.x; i < n4; i += blockDim.x) dst[i] = __ldcg(src + i);
  __syncthreads();
}

// Rows of the CTA that all its warps take together: hub-list entries above
// kK1Long (hub m belongs to CTA m % grid), the first kK1MaxLong of them.
struct K1Long {
  int n, last;  // count; the hub-list index after which long rows go to warps
  int idx[kK1MaxLong];
};
__device__ __forceinline__ void k1_find_long(const PhaseGraph& g, int b, int grid, K1Long& L) {
  __shared__ int s_cnt[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x, nwarp = nthr >> 5;
  int cnt = 0;
  for (int64_t m0 = b; m0 < g.nhub && cnt < kK1MaxLong; m0 += (int64_t)nthr * grid) {
    const int64_t m = m0 + (int64_t)tid * grid;
    bool lg = false;
    if (m < g.nhub) {
      const int row = __ldg(g.hubs + m);
      lg = __ldg(g.row_ptr + row + 1) - __ldg(g.row_ptr + row) > kK1Long;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, lg);
    if (lane == 0) s_cnt[warp] = __popc(bal);
    __syncthreads();
    int pos = cnt;
    for (int w = 0; w < nwarp; ++w) {
      if (w < warp) pos += s_cnt[w];
      cnt += s_cnt[w];
    }
    pos += __popc(bal & ((1u << lane) - 1u));
    if (lg && pos < kK1MaxLong) L.idx[pos] = (int)m;
    __syncthreads();
  }
  if (tid == 0) {
    L.n = cnt < kK1MaxLong ? cnt : kK1MaxLong;
    L.last = cnt < kK1MaxLong ? 0x7fffffff : L.idx[kK1MaxLong - 1];
  }
  __syncthreads();
}

// One pass over all rows of the grid. A::V is the gathered value, A the sum of
// a row's values (add, fold over lanes), fetch(col) reads a value, pre(row) what
// the row's end needs (issued before its gathers), fin(row, deg, sum, pre) ends
// a row. Every thread of the CTA calls it.
template <typename A, typename Fetch, typename Pre, typename Fin>
__device__ __forceinline__ void k1_rows(const PhaseGraph& g, int b, int grid, const K1Long& L, typename A::V* s_val,
                                        A* s_acc, Fetch fetch, Pre pre, Fin fin) {
  using V = typename A::V;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x, nwarp = nthr >> 5;
  const int32_t* __restrict__ rp = g.row_ptr;
  const int32_t* __restrict__ col = g.col;
  // sum of the entries [beg, end) with stride `step`, eight gathers in flight
  auto gather = [&](int beg, int end, int step, A& acc) {
    for (int e = beg; e < end; e += 8 * step) {
      int j[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) j[u] = e + u * step < end ? __ldg(col + e + u * step) : -1;
      V v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (j[u] >= 0) v[u] = fetch(j[u]);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (j[u] >= 0) acc.add(v[u]);
    }
  };
  // long rows by the whole CTA
  for (int h = 0; h < L.n; ++h) {
    const int row = __ldg(g.hubs + L.idx[h]);
    const int beg = __ldg(rp + row), end = __ldg(rp + row + 1);
    A acc;
    gather(beg + tid, end, nthr, acc);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc.fold(off);
    if (lane == 0) s_acc[warp] = acc;
    __syncthreads();
    if (warp == 0) {
      acc = A();
      if (lane < nwarp) acc = s_acc[lane];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) acc.fold(off);
      if (lane == 0) fin((int64_t)row, end - beg, acc, pre((int64_t)row));
    }
    __syncthreads();
  }
  // the other hub rows, a warp each
  for (int64_t m = (int64_t)warp * grid + b; m < g.nhub; m += (int64_t)nwarp * grid) {
    const int row = __ldg(g.hubs + m);
    const int beg = __ldg(rp + row), end = __ldg(rp + row + 1);
    if (end - beg > kK1Long && m <= L.last && L.n > 0) continue;
    A acc;
    gather(beg + lane, end, 32, acc);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc.fold(off);
    if (lane == 0) fin((int64_t)row, end - beg, acc, pre((int64_t)row));
  }
  // mid rows, eight lanes each (whole warps stay in the loop for the shuffles)
  for (int64_t m0 = ((int64_t)warp * grid + b) * 4; m0 < g.nmid; m0 += (int64_t)nwarp * grid * 4) {
    const int64_t m = m0 + (lane >> 3);
    const bool live = m < g.nmid;
    const int row = live ? __ldg(g.mids + m) : 0;
    const int beg = live ? __ldg(rp + row) : 0, end = live ? __ldg(rp + row + 1) : 0;
    A acc;
    gather(beg + (lane & 7), end, 8, acc);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) acc.fold(off);
    if (live && (lane & 7) == 0) fin((int64_t)row, end - beg, acc, pre((int64_t)row));
  }
  // short rows, 32 at a time
  const int lim = g.nmid > 0 ? kK1Lim : kHubDeg;
  V* val = s_val + warp * kK1Chunk;
  const int64_t ngrp = (g.n + 31) / 32;
  for (int64_t gr = (int64_t)warp * grid + b; gr < ngrp; gr += (int64_t)nwarp * grid) {
    const int64_t row = gr * 32 + lane;
    const int beg = __ldg(rp + (row < g.n ? row : g.n)), end = __ldg(rp + (row < g.n ? row + 1 : g.n));
    const bool live = row < g.n && end - beg <= lim;
    const int len = live ? end - beg : 0;
    decltype(pre((int64_t)0)) own{};
    if (live) own = pre(row);
    int pos = len;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, pos, off);
      if (lane >= off) pos += t;
    }
    const int total = __shfl_sync(0xffffffffu, pos, 31);
    pos -= len;
    const int b0 = __shfl_sync(0xffffffffu, beg, 0), b1 = __shfl_sync(0xffffffffu, end, 31);
    A acc;
    if (b1 - b0 == total) {  // no listed row between them: the entries lie together
      for (int t0 = 0; t0 < total; t0 += kK1Chunk) {
        int j[kK1Chunk / 32];
#pragma unroll
        for (int u = 0; u < kK1Chunk / 32; ++u) {
          const int i = t0 + 32 * u + lane;
          j[u] = i < total ? __ldg(col + b0 + i) : -1;
        }
        V v[kK1Chunk / 32];
#pragma unroll
        for (int u = 0; u < kK1Chunk / 32; ++u)
          if (j[u] >= 0) v[u] = fetch(j[u]);
#pragma unroll
        for (int u = 0; u < kK1Chunk / 32; ++u)
          if (j[u] >= 0) val[32 * u + lane] = v[u];
        __syncwarp();
        const int k0 = max(pos, t0) - t0, k1 = min(pos + len, t0 + kK1Chunk) - t0;
        for (int k = k0; k < k1; ++k) acc.add(val[k]);
        __syncwarp();
      }
    } else {
      gather(beg, beg + len, 1, acc);
    }
    __syncwarp();
    if (live) fin(row, len, acc, own);
  }
}

// sums of a row's values
template <typename T>
struct K1Sum {
  using V = T;
  T s = T(0);
  __device__ __forceinline__ void add(T v) { s += v; }
  __device__ __forceinline__ void fold(int off) { s += __shfl_xor_sync(0xffffffffu, s, off); }
};
// values of one FP32 term, error-free sum
struct K1SumDf {
  using V = float;
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float v) { df_acc(s, c, v); }
  __device__ __forceinline__ void fold(int off) {
    const float so = __shfl_xor_sync(0xffffffffu, s, off), co = __shfl_xor_sync(0xffffffffu, c, off);
    const df t = two_sum(s, so);
    s = t.hi;
    c += t.lo + co;
  }
};
// double-float values: error-free sum of the leading terms, plain sum of the trailing ones
struct K1SumDf2 {
  using V = float2;
  float s = 0.f, c = 0.f, l = 0.f;
  __device__ __forceinline__ void add(float2 v) {
    df_acc(s, c, v.x);
    l += v.y;
  }
  __device__ __forceinline__ void fold(int off) {
    const float so = __shfl_xor_sync(0xffffffffu, s, off), co = __shfl_xor_sync(0xffffffffu, c, off);
    l += __shfl_xor_sync(0xffffffffu, l, off);
    const df t = two_sum(s, so);
    s = t.hi;
    c += t.lo + co;
  }
};

// Sum over the grid of one value per thread, in *s_out (shared) of every CTA.
// step counts the launch's barriers; part: 2 x grid sums.
template <typename T>
struct K1GridSum {
  using SM = CoopSum<T>;
  using S = typename SM::S;
  S* part;
  CoopBar* bar;
  unsigned step = 0;
  __device__ __forceinline__ bool operator()(S v, S* s_w, S* s_out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5, grid = gridDim.x;
    S* p = part + (size_t)(step & 1u) * grid;
    ++step;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = SM::add(v, SM::shfl(v, off));
    if (lane == 0) s_w[warp] = v;
    __syncthreads();
    if (warp == 0) {
      v = lane < nwarp ? s_w[lane] : SM::zero();
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) v = SM::add(v, SM::shfl(v, off));
      if (lane == 0) p[blockIdx.x] = v;
    }
    if (!coop_sync(bar, step * (unsigned)grid)) return false;
    if (warp == 0) {
      v = SM::zero();
#pragma unroll 8
      for (int g = lane; g < grid; g += 32) v = SM::add(v, __ldcg(p + g));
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) v = SM::add(v, SM::shfl(v, off));
      if (lane == 0) *s_out = v;
    }
    __syncthreads();
    return true;
  }
};

// ---------------------------------------------------------------- CG, one column
// The iteration of cg_coop with the vectors in global memory.
template <typename T, bool SH>
__global__ void __launch_bounds__(k1_threads<T>(), 1) cg_k1(CoopArgs<T> ca_) {
  using SM = CoopSum<T>;
  using S = typename SM::S;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ S s_w[32], s_sum;
  __shared__ K1Sum<T> s_acc[32];
  __shared__ K1Long s_long;
  __shared__ T s_a, s_b;
  const PhaseArgs<T>& a = ca_.a;
  if (*(volatile int*)&ca_.bar->err != 0) return;
  const int tid = threadIdx.x, nthr = blockDim.x, b = blockIdx.x, grid = gridDim.x;
  T* s_head = reinterpret_cast<T*>(smem_raw);
  T* s_val = s_head + ca_.nhead;
  const int nhead = ca_.nhead;
  k1_find_long(a.g, b, grid, s_long);
  K1GridSum<T> sum{reinterpret_cast<S*>(a.part), ca_.bar};
  // FP32: scaled by a power of two to a starting norm near 1, as in cg_coop
  int e2 = 0;
  if (sizeof(T) == 4 && ca_.gamma0) {
    const double g0 = ca_.gamma0[0];
    if (g0 > 0.0 && isfinite(g0)) e2 = max(-120, min(120, ilogb(g0) >> 1));
  }
  const T sig = (T)ldexp(1.0, -e2), isig = (T)ldexp(1.0, e2);
  // r = scaled r0
  T acc = T(0);
  for (int64_t i = (int64_t)b * nthr + tid; i < a.g.n; i += (int64_t)grid * nthr) {
    const T r = ldp<T, 1>(ca_.r0 + i).v[0] * sig;
    a.rn[i] = r;
    acc += r * r;
  }
  if (!sum(SM::from(acc), s_w, &s_sum)) return;
  const double sig2 = (double)sig * (double)sig;
  S gamma = ca_.gamma0 ? SM::in(ca_.gamma0[0] * sig2) : s_sum;
  const double gn0 = SM::out(gamma), b2 = !ca_.gamma0 && a.bnorm2 ? a.bnorm2[0] : gn0;
  const S limit = SM::in(a.tol2 * b2);
  int done = !(b2 > 0.0) || (!ca_.gamma0 && gn0 <= a.tol2 * b2) || (a.skip && a.skip[0]), status = 0;
  if (!isfinite(gn0)) { done = 1; status = WL_ERR_NONFINITE; }
  const T ca = (T)a.ca, cA = (T)a.cA, cD = (T)a.cD;
  const T* r = a.rn;
  T beta = T(0);
  int iters = 0;
  struct Own {
    T r, p, q, d;
  };
  auto fetch = [&](int j) -> T { return j < nhead ? s_head[j] : ld_plain<T, 1>(r + j).v[0]; };
  while (!done && iters < a.max_iter) {
    const bool first = iters == 0;
    k1_load_head(r, s_head, nhead);
    acc = T(0);
    auto pre = [&](int64_t row) {
      Own o;
      o.r = ldp<T, 1>(r + row).v[0];
      o.p = first ? T(0) : ldp<T, 1>(a.p + row).v[0];
      o.q = first ? T(0) : ldp<T, 1>(a.q + row).v[0];
      o.d = T(0);
      if constexpr (SH) o.d = __ldg(a.dshift + row);
      return o;
    };
    auto fin = [&](int64_t row, int deg, const K1Sum<T>& nb, const Own& o) {
      T crow = ca + cD * (T)deg;
      if constexpr (SH) crow += o.d;
      const T p = o.r + beta * o.p, q = crow * o.r + cA * nb.s + beta * o.q;
      a.p[row] = p;
      a.q[row] = q;
      acc += p * q;
    };
    k1_rows<K1Sum<T>>(a.g, b, grid, s_long, s_val, s_acc, fetch, pre, fin);
    if (!sum(SM::from(acc), s_w, &s_sum)) return;
    ++iters;
    const S delta = s_sum;
    T al = T(0);
    if (!isfinite(SM::lead(delta))) {
      status = WL_ERR_NONFINITE;
      done = 1;
    } else if (SM::lead(delta) <= 0) {
      status = WL_ERR_NOT_SPD;
      done = 1;
    } else {
      if (tid == 0) s_a = SM::quot(gamma, delta);
      __syncthreads();
      al = s_a;
    }
    const T ax = al * isig;
    const bool x_zero = first && !ca_.add_x;
    acc = T(0);
#pragma unroll 2
    for (int64_t i = (int64_t)b * nthr + tid; i < a.g.n; i += (int64_t)grid * nthr) {
      const T p = ldp<T, 1>(a.p + i).v[0], q = ldp<T, 1>(a.q + i).v[0], r0 = ldp<T, 1>(r + i).v[0];
      const T x0 = x_zero ? T(0) : ldp<T, 1>(a.x + i).v[0];
      const T rn = r0 - al * q;
      a.x[i] = x0 + ax * p;
      a.rn[i] = rn;
      acc += rn * rn;
    }
    if (!sum(SM::from(acc), s_w, &s_sum)) return;
    const S gn = s_sum;
    if (!done) {
      if (!isfinite(SM::lead(gn))) {
        status = WL_ERR_NONFINITE;
        done = 1;
      } else {
        if (tid == 0) s_b = SM::quot(gn, gamma);
        __syncthreads();
        beta = s_b;
        gamma = gn;
        if (SM::le(gn, limit)) done = 1;
      }
    }
  }
  if (iters == 0 && !ca_.add_x)
    for (int64_t i = (int64_t)b * nthr + tid; i < a.g.n; i += (int64_t)grid * nthr) a.x[i] = T(0);
  if (b == 0 && tid == 0) {
    CgState* st = a.st;
    st->gamma[0] = SM::out(gamma) / sig2;
    st->b2[0] = b2 / sig2;
    st->done[0] = done;
    st->status[0] = status;
    st->iters = iters;
    st->active = 0;
  }
}

// ---------------------------------------------------------------- residual, one column
// df_res of wl_res.cuh for K = 1 (not FULL): r <- r - M d, x <- x + d, |r|^2.
// Every CTA's partial, the last one's sum.
template <bool SH>
__global__ void __launch_bounds__(k1_threads<float>(), 1) df_res_k1(DfResArgs a, int nhead) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ K1SumDf s_acc[32];
  __shared__ K1Long s_long;
  __shared__ double s_w[32];
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5, b = blockIdx.x,
            grid = gridDim.x;
  float* s_head = reinterpret_cast<float*>(smem_raw);
  float* s_val = s_head + nhead;
  const float* d = a.yh;
  k1_find_long(a.g, b, grid, s_long);
  k1_load_head(d, s_head, nhead);
  struct Own {
    float d, bh, bl, xh, xl;
    df sh;
  };
  float nacc = 0.f;
  auto fetch = [&](int j) -> float { return j < nhead ? s_head[j] : ld_plain<float, 1>(d + j).v[0]; };
  auto pre = [&](int64_t row) {
    Own o;
    o.d = ldp<float, 1>(d + row).v[0];
    o.bh = ldp<float, 1>(a.bh + row).v[0];
    o.bl = ldp<float, 1>(a.bl + row).v[0];
    o.xh = a.x_zero ? 0.f : ldp<float, 1>(a.xh + row).v[0];
    o.xl = a.x_zero ? 0.f : ldp<float, 1>(a.xl + row).v[0];
    o.sh = df{0.f, 0.f};
    if constexpr (SH) o.sh = df{a.dsh_h[row], a.dsh_l[row]};
    return o;
  };
  auto fin = [&](int64_t row, int deg, const K1SumDf& s, const Own& o) {
    df crow = df_add(a.ca, df_mul_f(a.cD, (float)deg));
    if constexpr (SH) crow = df_add(crow, o.sh);
    const df My = df_add(df_mul(crow, df{o.d, 0.f}), df_mul(a.cA, two_sum(s.s, s.c)));
    const df r = df_sub(df{o.bh, o.bl}, My);
    a.rh[row] = r.hi;
    a.rl[row] = r.lo;
    nacc = __fmaf_rn(r.hi, r.hi, nacc);
    if (a.x_zero) {
      a.xh[row] = o.d;
      a.xl[row] = 0.f;
    } else {
      const df t = two_sum(o.xh, o.d);
      const df u = quick_two_sum(t.hi, t.lo + o.xl);
      a.xh[row] = u.hi;
      a.xl[row] = u.lo;
    }
  };
  k1_rows<K1SumDf>(a.g, b, grid, s_long, s_val, s_acc, fetch, pre, fin);
  double t = (double)nacc;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
  if (lane == 0) s_w[warp] = t;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < nwarp; ++w) t += s_w[w];
    a.part[b] = t;
    __threadfence();
    s_last = atomicAdd(&a.st->ticket, 1u) == (unsigned)grid - 1u;
  }
  __syncthreads();
  if (!s_last || warp != 0) return;
  __threadfence();
  t = 0.0;
  for (int g = lane; g < grid; g += 32) t += __ldcg(a.part + g);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
  if (lane == 0) {
    a.st->gamma[0] = t;
    a.st->ticket = 0;
  }
}

}  // namespace wl
