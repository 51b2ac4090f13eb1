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
// bytes, E of them along the entries, E > 1 where G is small), a warp per row of
// the mid and hub lists, the CTA for the longest of these.
//
// Measured per call against the phase kernels (before -> here): walk degrees and
// four columns in FP64, n = 2000: 1385 -> 420 us; 13 refined columns, n = 20011:
// 2530 -> 451 us; R-MAT scale 14, 64 refined columns: 1140 -> 754 us (1520 with its
// hub rows by warps); R-MAT scale 19, one FP64 column: 4.8 -> 1.25 ms; 132 refined
// shifted solves of 62500 x 32: 377 -> 160 ms, an iteration 26 us where the phase
// kernels' two launches took 43.
#pragma once
#include <algorithm>
#include <atomic>

#include "wl_cg2.cuh"
#include "wl_df.cuh"

namespace wl {

constexpr int kCoopLong = 64;  // rows of a CTA that all its warps take together, at most

template <typename T, int K>
struct CoopCfg {
  using C = Cfg<T, K>;
  static constexpr int VW = C::VW, G = C::G;
  static constexpr int E = G >= 4 ? 1 : 4 / G;
  static constexpr int LPR = G * E;
  static constexpr int SLOT = VW * (int)sizeof(T);  // bytes of one lane's part of a vector
  static constexpr int SECTOR = 32 / (K * (int)sizeof(T));
  static constexpr int CHMIN = SECTOR > 1 ? SECTOR : 1;  // consecutive rows of a CTA: a 32-byte sector at least
  // K = 1: two short rows per lane group at once, and half a warp per listed
  // row, since one row's few loads leave the lanes waiting
  static constexpr int N = K == 1 ? 2 : 1;
  static constexpr int LW = K == 1 ? 16 : 32;
  // gathers in flight per lane and row: four, and all the threads that their
  // registers leave room for (a row's few entries leave half of eight unused); FP64 from K = 4 on: the eight
  // values of an integer sum
  static constexpr int U = sizeof(T) == 8 && K >= 4 ? 8 : 4;
  static constexpr int UL = sizeof(T) == 8 || K == 1 ? 8 : 4;  // the same for listed rows
  // a listed row of more entries goes to the whole CTA: beyond eight rounds of its lanes' gathers of eight
  // (K = 1: 32 rounds; twice as many rows run side by side there, and a CTA takes three barriers for one);
  // of fewer where a warp's share of all the entries is smaller than such a row (cgc_shape)
  static constexpr int LONG = K == 1 ? 4096 : 64 * (LW / G);
  // most threads of a CTA (one per SM); FP64: its sums hold the FP64 pipe for a microsecond at 512 already
  static constexpr int TMAX = sizeof(T) == 4 ? 896 : 512;
  // shared memory left for the vectors: 227 KB less the static arrays
  static constexpr size_t SMEM = 227 * 1024 - (32 * K * 8 + K * (48 + 4 * (int)sizeof(T) + 8) + 4 * kCoopLong + 512);
};

constexpr int kCoopCluster = 16;  // CTAs of the smallest solves: one cluster
constexpr int kCoopGroups = 16;   // groups of CTAs in a two-level sum, at most

// Arrivals counted up over the launch (cleared before it) and an error word.
// A barrier is one release-add and a poll: no reset, no generation word and
// no second look at memory (the general grid_sync reads, adds and reads again:
// 4 us against 1.5 us here). Bounded like it.
struct CoopBar {
  unsigned count;
  unsigned grp[kCoopGroups];  // arrivals per group of CTAs
  int err;
};

template <typename T>
struct CoopArgs {
  PhaseArgs<T> a;  // a.g carries the mid list (nmid > 0: rows above kMidDeg are on it)
  CoopBar* bar;
  const T* r0;           // the starting residual (a.rn itself, or read only: a.rn is then scratch; FP64: a.rn is the
                         // final residual on return)
  const double* gamma0;  // its column norms |r0|^2; NULL: computed here
  int add_x;             // 1: x holds a start value, the correction is added to it; 0: x is written
  // set by the launch
  int long_min;          // listed rows of more entries go to the whole CTA
  int nhead;             // K = 1: leading entries of r kept in shared memory
  int ch_log;            // log2 of a CTA's consecutive rows
  int col_cap;           // column indices of short rows that fit in shared memory (0: none kept)
  int x_global;          // x stays in global memory (it is touched once an iteration)
  int cluster;           // the grid is one cluster
  int group;             // > 0: two-level sums over groups of this many CTAs
};

// slots (lane parts) of one vector in a CTA's shared memory
__host__ __device__ inline int64_t coop_rows_local(int64_t n, int grid, int ch) {
  return ((n + ch - 1) / ch + grid - 1) / grid * ch;
}

__device__ __forceinline__ bool coop_sync(CoopBar* b, unsigned target, bool arrive = true) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    if (arrive)
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

// Sums of X over the entries [beg[i], end[i]) with stride `step` of N rows at
// once. The loads of X may hit L1: the barrier's acquire orders them after the
// other SMs' writes (CG: one cluster, whose barrier gives no order to L1: L2
// only). K = 1: entries below nhead come from their copy in shared memory.
template <typename T, int K, int VW, int U, int N>
__device__ __forceinline__ void coop_gather(const int32_t* col, int (&beg)[N], const int (&end)[N], int step,
                                            const T* X, const T* head, int nhead, bool l2, int lane_off,
                                            T (&acc)[N][VW]) {
  for (;;) {
    bool any = false;
#pragma unroll
    for (int i = 0; i < N; ++i) any |= beg[i] < end[i];
    if (!any) break;
    int j[N][U];
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int u = 0; u < U; ++u) j[i][u] = beg[i] + u * step < end[i] ? col[beg[i] + u * step] : -1;
    Pack<T, VW> v[N][U];
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q = j[i][u];
        if (K == 1 && (unsigned)q < (unsigned)nhead) {
          v[i][u].v[0] = head[q];
        } else if (q >= 0) {
          const T* p = X + (size_t)q * K + lane_off;
          v[i][u] = l2 ? ldp<T, VW>(p) : ld_plain<T, VW>(p);
        } else {
#pragma unroll
          for (int w = 0; w < VW; ++w) v[i][u].v[w] = T(0);
        }
      }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if constexpr (sizeof(T) == 8 && U == 8) {
        if (end[i] - beg[i] > 4 * step) {
#pragma unroll
          for (int w = 0; w < VW; ++w) {
            double x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = v[i][u].v[w];
            acc[i][w] = add_aligned<8>(acc[i][w], x);
          }
        } else {
#pragma unroll
          for (int w = 0; w < VW; ++w) {
            double x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = v[i][u].v[w];
            acc[i][w] = add_aligned<4>(acc[i][w], x);
          }
        }
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (sizeof(T) == 4 || j[i][u] >= 0)  // (no FP64 addition of a zero)
#pragma unroll
            for (int w = 0; w < VW; ++w) acc[i][w] += v[i][u].v[w];
      }
      beg[i] += U * step;
    }
  }
}

// All threads of the cluster. Without .aligned: that form wants every warp
// converged, and the callers' branches (four lanes a column, tid < K) leave
// that to the compiler. The wait ends whatever the other CTAs do: a cluster's
// CTAs start together, and a CTA that has exited counts as arrived.
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// 8 bytes at the same shared-memory place of CTA `rank` of the cluster
__device__ __forceinline__ unsigned long long ld_peer64(const void* p, unsigned rank) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
  unsigned long long v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(r) : "memory");
  return v;
}

template <typename T, int K, bool SH>
__global__ void __launch_bounds__(CoopCfg<T, K>::TMAX, 1) cg_coop(CoopArgs<T> ca_) {
  using CC = CoopCfg<T, K>;
  using SM = CoopSum<T>;
  using S = typename SM::S;
  static_assert(sizeof(S) == 8, "sums travel as 8 bytes");
  constexpr int VW = CC::VW, G = CC::G, E = CC::E, LPR = CC::LPR, U = CC::U, N = CC::N, LW = CC::LW;
  constexpr int kNone = 0xFFFF;
  using P = Pack<T, VW>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ S s_w[32 * K], s_part[2][K];
  __shared__ S s_sum[K], s_gamma[K], s_lim[K];  // column sums, gamma, and the gamma of convergence
  __shared__ T s_al[K], s_ax[K], s_be[K], s_sig[K];
  __shared__ double s_b2[K];
  __shared__ int s_done[K], s_stat[K];
  __shared__ int s_any, s_last, s_long[kCoopLong], s_cnt[32];
  const PhaseArgs<T>& a = ca_.a;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
  const int b = blockIdx.x, grid = gridDim.x;
  const int sl = tid % G, lane_off = sl * VW;
  const int chl = ca_.ch_log;
  const int nloc = (int)coop_rows_local(a.g.n, grid, 1 << chl);
  const int lim = a.g.nmid > 0 ? kMidDeg : kHubDeg;
  // listed rows of this CTA: hubs, then mid rows
  const int nhub_l = a.g.nhub > b ? (a.g.nhub - b + grid - 1) / grid : 0;
  const int nlist = nhub_l + (a.g.nmid > b ? (a.g.nmid - b + grid - 1) / grid : 0);
  const int cap_list = (a.g.nhub + grid - 1) / grid + (a.g.nmid + grid - 1) / grid;
  // shared memory: the vectors' slots (short rows, then listed rows), the
  // copied head of r, and the rows' places in the CSR, kept here because every
  // barrier empties L1
  const int list0 = nloc * G, nslot = list0 + cap_list * G;
  P* sp = reinterpret_cast<P*>(smem_raw);
  P* sq = sp + nslot;
  P* sr = sq + nslot;
  P* sx = sr + nslot;
  T* s_head = reinterpret_cast<T*>(ca_.x_global ? sx : sx + nslot);
  const int nhead = K == 1 ? ca_.nhead : 0;
  int* s_lrow = reinterpret_cast<int*>(s_head + nhead);
  int* s_lbeg = s_lrow + cap_list;
  int* s_llen = s_lbeg + cap_list;
  int* s_beg = s_llen + cap_list;
  int* s_col = s_beg + nloc;
  unsigned short* s_len = reinterpret_cast<unsigned short*>(s_col + ca_.col_cap);
  const int32_t* __restrict__ rp = a.g.row_ptr;
  const int32_t* __restrict__ col = a.g.col;
  auto row_of = [&](int lr) -> int64_t {
    return (((int64_t)(lr >> chl) * grid + b) << chl) + (lr & ((1 << chl) - 1));
  };
  if (*(volatile int*)&ca_.bar->err != 0) return;  // set before the launch: every CTA leaves
  for (int m = tid; m < nlist; m += nthr) {
    const int row = m < nhub_l ? __ldg(a.g.hubs + m * grid + b) : __ldg(a.g.mids + (m - nhub_l) * grid + b);
    const int beg = __ldg(rp + row);
    s_lrow[m] = row;
    s_lbeg[m] = beg;
    s_llen[m] = __ldg(rp + row + 1) - beg;
  }
  // entries of the short rows before each of them (the place of its indices in s_col)
  int ncol = 0;
  for (int l0 = 0; l0 < nloc; l0 += nthr) {
    const int lr = l0 + tid;
    const int64_t row = row_of(lr);
    int beg = 0, len = kNone;
    if (lr < nloc && row < a.g.n) {
      beg = __ldg(rp + row);
      const int d = __ldg(rp + row + 1) - beg;
      if (d <= lim) len = d;
    }
    int sum = len == kNone ? 0 : len;
    const int own = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, sum, off);
      if (lane >= off) sum += t;
    }
    if (lane == 31) s_cnt[warp] = sum;
    __syncthreads();
    int base = ncol;
    for (int w = 0; w < nwarp; ++w) {
      if (w < warp) base += s_cnt[w];
      ncol += s_cnt[w];
    }
    const int at = base + sum - own;
    if (lr < nloc) {
      s_len[lr] = (unsigned short)len;
      s_beg[lr] = beg;
      if (len != kNone && at + len <= ca_.col_cap)
        for (int e = 0; e < len; ++e) s_col[at + e] = __ldg(col + beg + e);
    }
    __syncthreads();
  }
  const bool kept = ncol <= ca_.col_cap;
  if (kept) {  // every short row's indices are in s_col, one row after the other
    int base = 0;
    for (int l0 = 0; l0 < nloc; l0 += nthr) {
      const int lr = l0 + tid;
      const int own = lr < nloc && s_len[lr] != kNone ? s_len[lr] : 0;
      int sum = own;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, sum, off);
        if (lane >= off) sum += t;
      }
      if (lane == 31) s_cnt[warp] = sum;
      __syncthreads();
      int at = base + sum - own;
      for (int w = 0; w < nwarp; ++w) {
        if (w < warp) at += s_cnt[w];
        base += s_cnt[w];
      }
      if (lr < nloc) s_beg[lr] = at;
      __syncthreads();
    }
  }
  const int32_t* scol = kept ? s_col : col;
  // the first kCoopLong long listed rows go to the whole CTA
  int nlong = 0;
  for (int m0 = 0; m0 < nlist && nlong < kCoopLong; m0 += nthr) {
    const int m = m0 + tid;
    const bool lg = m < nlist && s_llen[m] > ca_.long_min;
    const unsigned bal = __ballot_sync(0xffffffffu, lg);
    if (lane == 0) s_cnt[warp] = __popc(bal);
    __syncthreads();
    int pos = nlong;
    for (int w = 0; w < nwarp; ++w) {
      if (w < warp) pos += s_cnt[w];
      nlong += s_cnt[w];
    }
    pos += __popc(bal & ((1u << lane) - 1u));
    if (lg && pos < kCoopLong) s_long[pos] = m;
    __syncthreads();
  }
  if (nlong > kCoopLong) nlong = kCoopLong;
  const int long_last = nlong == kCoopLong ? s_long[kCoopLong - 1] : nlist;
  // f(slot, row) for every slot of this thread's columns
  auto for_slots = [&](auto f) {
    for (int s = tid; s < list0; s += nthr)
      if (s_len[s / G] != kNone) f(s, row_of(s / G));
    for (int s = tid; s < nlist * G; s += nthr) f(list0 + s, (int64_t)s_lrow[s / G]);
  };
  S* part = reinterpret_cast<S*>(a.part);
  unsigned step = 0;  // barriers passed
  // J consecutive lanes per column add n sums given by get(i, column) into s_sum
  auto add_all = [&](int n, auto get, S* to) {
    int J = 32;
    while (J * K > nthr) J >>= 1;
    const int c = tid / J, j = tid % J;
    if (tid < K * J) {
      S t = SM::zero();
#pragma unroll 8
      for (int g = j; g < n; g += J) t = SM::add(t, get(g, c));
      for (int off = 1; off < J; off <<= 1) t = SM::add(t, SM::shfl(t, off));
      if (j == 0) to[c] = t;
    }
  };
  // sums the threads' values over the grid: column c in s_sum[c] on return.
  // One cluster: from the peers' shared memory. Otherwise every CTA adds all
  // CTAs' sums, or, with many columns, the last CTA to arrive of each group adds
  // the group's and every CTA the groups' (152 SMs reading 152 x 16 sums each
  // took 6 us).
  auto grid_sum = [&](const T (&val)[VW]) -> bool {
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
    const int half = (int)(step & 1u);
    ++step;
    S* p = part + (size_t)half * grid * K;
    if (tid < (K * 4 < 32 ? 32 : K * 4)) {  // four lanes per column add the warps' sums (whole warps shuffle)
      S t = SM::zero();
      if (tid < K * 4)
        for (int w = tid & 3; w < nwarp; w += 4) t = SM::add(t, s_w[w * K + (tid >> 2)]);
      t = SM::add(t, SM::shfl(t, 1));
      t = SM::add(t, SM::shfl(t, 2));
      if ((tid & 3) == 0 && tid < K * 4) {
        if (ca_.cluster)
          s_part[half][tid >> 2] = t;
        else
          p[(size_t)b * K + (tid >> 2)] = t;
      }
    }
    if (ca_.cluster) {
      cluster_sync_all();
      add_all(grid, [&](int g, int c) {
        union {
          unsigned long long u;
          S s;
        } x;
        x.u = ld_peer64(&s_part[half][c], (unsigned)g);
        return x.s;
      }, s_sum);
      __syncthreads();
      return true;
    }
    int n = grid;
    const S* src = p;
    unsigned target = step * (unsigned)grid;
    if (ca_.group > 0) {
      const int gi = b / ca_.group, g0 = gi * ca_.group, gn = min(ca_.group, grid - g0);
      n = (grid + ca_.group - 1) / ca_.group;
      S* q = part + (size_t)2 * grid * K + (size_t)half * kCoopGroups * K;
      src = q;
      target = step * (unsigned)n;
      __syncthreads();
      if (tid == 0) {
        unsigned old;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;"
                     : "=r"(old)
                     : "l"(&ca_.bar->grp[gi])
                     : "memory");
        s_last = old + 1u == step * (unsigned)gn;
      }
      __syncthreads();
      if (s_last) add_all(gn, [&](int g, int c) { return __ldcg(p + (size_t)(g0 + g) * K + c); }, q + (size_t)gi * K);
    }
    if (!coop_sync(ca_.bar, target, ca_.group == 0 || s_last)) return false;
    add_all(n, [&](int g, int c) { return __ldcg(src + (size_t)g * K + c); }, s_sum);
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
  // FP32: every column is solved scaled by the power of two that brings its
  // starting norm near 1 (exact), so that its sums stay in the range of FP32
  // whatever the scale of the right-hand side
  if (tid < K) {
    int e = 0;
    if (sizeof(T) == 4 && ca_.gamma0) {
      const double g0 = ca_.gamma0[tid];
      if (g0 > 0.0 && isfinite(g0)) e = max(-120, min(120, ilogb(g0) >> 1));
    }
    s_sig[tid] = (T)ldexp(1.0, -e);
  }
  __syncthreads();
  // start: r into shared memory, x = 0, norms
  zero_acc();
  for_slots([&](int s, int64_t row) {
    P r = ldp<T, VW>(ca_.r0 + (size_t)row * K + lane_off);
    if constexpr (sizeof(T) == 4)
#pragma unroll
      for (int w = 0; w < VW; ++w) r.v[w] *= s_sig[lane_off + w];
    sr[s] = r;
    P z;
#pragma unroll
    for (int w = 0; w < VW; ++w) {
      z.v[w] = T(0);
      acc[w] += r.v[w] * r.v[w];
    }
    if (!ca_.x_global) sx[s] = z;
  });
  if (!ca_.gamma0) {
    if (!grid_sum(acc)) return;
  } else {
    if (tid < K) s_sum[tid] = SM::in(ca_.gamma0[tid] * ((double)s_sig[tid] * (double)s_sig[tid]));
    __syncthreads();
  }
  if (tid == 0) s_any = 0;
  __syncthreads();
  if (tid < K) {
    const double gn = SM::out(s_sum[tid]), b2 = !ca_.gamma0 && a.bnorm2 ? a.bnorm2[tid] : gn;
    int done = !(b2 > 0.0) || (!ca_.gamma0 && gn <= a.tol2 * b2) || (a.skip && a.skip[tid]), status = 0;
    if (!isfinite(gn)) { done = 1; status = WL_ERR_NONFINITE; }
    s_gamma[tid] = s_sum[tid];
    s_b2[tid] = b2;
    s_lim[tid] = SM::in(a.tol2 * b2);
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
    const T* rsrc = first ? ca_.r0 : a.rn;
    const bool l2 = ca_.cluster != 0;
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
      T crow = ca + cD * (T)deg;
      if constexpr (SH) crow += __ldg(a.dshift + row);
#pragma unroll
      for (int w = 0; w < VW; ++w) {
        // the first neighbour sums come from r0, unscaled
        const T nbw = sizeof(T) == 4 && first ? nb[w] * s_sig[lane_off + w] : nb[w];
        const T v = crow * r.v[w] + cA * nbw;
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
    auto fold = [&](T (&v)[VW], int from, int to) {
      for (int off = from; off < to; off <<= 1)
#pragma unroll
        for (int w = 0; w < VW; ++w) v[w] += __shfl_xor_sync(0xffffffffu, v[w], off);
    };
    // long listed rows by the whole CTA
    for (int h = 0; h < nlong; ++h) {
      const int m = s_long[h];
      int beg[1] = {s_lbeg[m] + tid / G};
      const int end[1] = {s_lbeg[m] + s_llen[m]};
      T nb[1][VW];
#pragma unroll
      for (int w = 0; w < VW; ++w) nb[0][w] = T(0);
      coop_gather<T, K, VW, CC::UL, 1>(col, beg, end, nthr / G, rsrc, s_head, nhead, l2, lane_off, nb);
      fold(nb[0], G, 32);
      T* s_t = reinterpret_cast<T*>(s_w);  // one value per warp and column fits
      __syncthreads();
      if (lane < G)
#pragma unroll
        for (int w = 0; w < VW; ++w) s_t[warp * K + lane_off + w] = nb[0][w];
      __syncthreads();
      if (tid < G) {
#pragma unroll
        for (int w = 0; w < VW; ++w) {
          nb[0][w] = T(0);
          for (int q = 0; q < nwarp; ++q) nb[0][w] += s_t[q * K + lane_off + w];
        }
        fin(list0 + m * G + sl, s_lrow[m], s_llen[m], nb[0]);
      }
      __syncthreads();  // s_w is free again
    }
    // the other listed rows, LW lanes each (whole warps stay in the loop for the shuffles)
    for (int m0 = warp * (32 / LW); m0 < nlist; m0 += nwarp * (32 / LW)) {
      const int m = m0 + lane / LW;
      const bool live = m < nlist && !(s_llen[m] > ca_.long_min && m <= long_last);
      int beg[1] = {live ? s_lbeg[m] + (lane % LW) / G : 0};
      const int end[1] = {live ? s_lbeg[m] + s_llen[m] : 0};
      T nb[1][VW];
#pragma unroll
      for (int w = 0; w < VW; ++w) nb[0][w] = T(0);
      coop_gather<T, K, VW, CC::UL, 1>(col, beg, end, LW / G, rsrc, s_head, nhead, l2, lane_off, nb);
      fold(nb[0], G, LW);
      if (live && lane % LW < G) fin(list0 + m * G + sl, s_lrow[m], s_llen[m], nb[0]);
    }
    // short rows, LPR lanes each, N at once
    for (int u0 = warp * 32; u0 < nloc * LPR; u0 += nthr * N) {
      int lr[N], len[N], beg[N], end[N];
      const int e = (lane / G) % E;
      T nb[N][VW];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        lr[i] = (u0 + i * nthr + lane) / LPR;
        len[i] = lr[i] < nloc ? s_len[lr[i]] : kNone;
        beg[i] = end[i] = 0;
        if (len[i] != kNone) {
          beg[i] = s_beg[lr[i]] + e;
          end[i] = s_beg[lr[i]] + len[i];
        }
#pragma unroll
        for (int w = 0; w < VW; ++w) nb[i][w] = T(0);
      }
      coop_gather<T, K, VW, U, N>(scol, beg, end, E, rsrc, s_head, nhead, l2, lane_off, nb);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        if constexpr (E > 1) fold(nb[i], G, LPR);
        if (len[i] != kNone && e == 0) fin(lr[i] * G + sl, row_of(lr[i]), len[i], nb[i]);
      }
    }
    if (!grid_sum(acc)) return;
    ++iters;
    if (tid < K) {
      const S delta = s_sum[tid];
      T al = T(0);
      if (!s_done[tid]) {
        if (!isfinite(SM::lead(delta))) {
          s_stat[tid] = WL_ERR_NONFINITE; s_done[tid] = 1;
        } else if (SM::lead(delta) <= 0) {
          s_stat[tid] = WL_ERR_NOT_SPD; s_done[tid] = 1;
        } else {
          al = SM::quot(s_gamma[tid], delta);
        }
      }
      s_al[tid] = al;
      s_ax[tid] = sizeof(T) == 4 && ca_.x_global ? al / s_sig[tid] : al;  // x in global memory is not scaled
    }
    if (tid == 0) s_any = 0;
    __syncthreads();
    // ---- U: x += alpha p, r -= alpha q, gamma'
    zero_acc();
    for_slots([&](int s, int64_t row) {
      const P pp = sp[s], qq = sq[s];
      P rr = sr[s], xx;
      T* px = a.x + (size_t)row * K + lane_off;
      if (!ca_.x_global) {
        xx = sx[s];
      } else if (!first || ca_.add_x) {
        xx = ldp<T, VW>(px);
      } else {
#pragma unroll
        for (int w = 0; w < VW; ++w) xx.v[w] = T(0);
      }
#pragma unroll
      for (int w = 0; w < VW; ++w) {
        xx.v[w] += s_ax[lane_off + w] * pp.v[w];
        rr.v[w] -= s_al[lane_off + w] * qq.v[w];
        acc[w] += rr.v[w] * rr.v[w];
      }
      if (ca_.x_global)
        stp<T, VW>(px, xx);
      else
        sx[s] = xx;
      sr[s] = rr;
      stp<T, VW>(a.rn + (size_t)row * K + lane_off, rr);
    });
    if (!grid_sum(acc)) return;
    if (tid < K) {
      const S gn = s_sum[tid];
      T be = T(0);
      if (!s_done[tid]) {
        if (!isfinite(SM::lead(gn))) {
          s_stat[tid] = WL_ERR_NONFINITE; s_done[tid] = 1;
        } else {
          be = SM::quot(gn, s_gamma[tid]);
          s_gamma[tid] = gn;
          if (SM::le(gn, s_lim[tid])) {
            s_done[tid] = 1;
            be = T(0);
          }
        }
      }
      s_be[tid] = be;
      if (!s_done[tid]) s_any = 1;
    }
    __syncthreads();
    active = s_any != 0 && iters < a.max_iter;
  }
  // x, and the solve's state for the host
  for_slots([&](int s, int64_t row) {
    T* px = a.x + (size_t)row * K + lane_off;
    if (!ca_.x_global) {
      P xx = sx[s];
      if constexpr (sizeof(T) == 4)
#pragma unroll
        for (int w = 0; w < VW; ++w) xx.v[w] /= s_sig[lane_off + w];
      if (ca_.add_x) {
        const P x0 = ldp<T, VW>(px);
#pragma unroll
        for (int w = 0; w < VW; ++w) xx.v[w] += x0.v[w];
      }
      stp<T, VW>(px, xx);
    } else if (iters == 0 && !ca_.add_x) {
      P z;
#pragma unroll
      for (int w = 0; w < VW; ++w) z.v[w] = T(0);
      stp<T, VW>(px, z);
    }
    // FP64: a.rn ends as the solve's residual, also of one that took no iteration
    if (sizeof(T) == 8 && iters == 0 && ca_.r0 != a.rn) stp<T, VW>(a.rn + (size_t)row * K + lane_off, sr[s]);
  });
  if (b == 0) {
    if (tid < K) {
      const double is = 1.0 / (double)s_sig[tid];
      st->gamma[tid] = SM::out(s_gamma[tid]) * is * is;
      st->b2[tid] = s_b2[tid] * is * is;
      st->done[tid] = s_done[tid];
      st->status[tid] = s_stat[tid];
    }
    if (tid == 0) {
      st->iters = iters;
      st->active = 0;
    }
  }
  if (ca_.cluster) cluster_sync_all();  // the peers may still read this CTA's sums
}

// ---------------------------------------------------------------- launch shape
struct CoopShape {
  int grid = 0, threads = 0, long_min = 0, nhead = 0, ch_log = 0, col_cap = 0, x_global = 0, cluster = 0, group = 0;
  size_t smem = 0;
};

// The launch of a solve with K columns, or false where its vectors don't fit.
// clusters: the device can place the kernel's clusters.
template <typename T, int K>
bool cgc_shape(const PhaseGraph& g, int64_t nnz, int sms, bool clusters, CoopShape* sh) {
  using CC = CoopCfg<T, K>;
  // 256 lane units (rows x LPR) per CTA until every SM has one (each CTA adds
  // to the reductions), then more threads, evenly over the passes of the row
  // loop. Up to 32 such CTAs are 16 of twice the threads in one cluster, whose
  // barrier and sums don't leave the cluster (FP64 only up to 4096 elements: 16
  // SMs' FP64 pipes take longer over 8000 than the grid's barrier costs).
  const int64_t units = g.n * CC::LPR, ctas = std::max<int64_t>(1, (units + 255) / 256);
  sh->cluster = clusters && ctas <= 2 * kCoopCluster && (sizeof(T) == 4 || g.n * K <= 4096);
  if (sh->cluster) {
    sh->grid = 1;
    while (sh->grid < kCoopCluster && sh->grid < ctas) sh->grid *= 2;
  } else {
    sh->grid = (int)std::min<int64_t>(sms, ctas);
  }
  // runs of up to 32 consecutive rows per CTA (neighbours of neighbouring rows
  // meet in one L1) as long as every CTA gets sixteen
  while ((1 << sh->ch_log) < CC::CHMIN) ++sh->ch_log;
  while (sh->ch_log < 5 && (g.n >> (sh->ch_log + 1)) >= (int64_t)16 * sh->grid) ++sh->ch_log;
  const int64_t rows = coop_rows_local(g.n, sh->grid, 1 << sh->ch_log);
  const int64_t passes = (rows * CC::LPR + CC::TMAX * CC::N - 1) / (CC::TMAX * CC::N);
  const int64_t per = (rows * CC::LPR + passes * CC::N - 1) / (passes * CC::N);
  sh->threads = (int)std::min<int64_t>(CC::TMAX, std::max<int64_t>(std::max(128, 4 * K), (per + 31) / 32 * 32));
  const int64_t share_w = nnz / ((int64_t)sh->grid * (sh->threads / CC::LW));  // entries per (half) warp
  sh->long_min = (int)std::min<int64_t>(CC::LONG, std::max<int64_t>(512, share_w));
  const int64_t nlist = (g.nmid + sh->grid - 1) / sh->grid + (g.nhub + sh->grid - 1) / sh->grid;
  const int64_t nslot = (rows + nlist) * CC::G;
  const size_t meta = (size_t)rows * 6 + (size_t)nlist * 12 + 16;
  const size_t vec = (size_t)nslot * CC::SLOT;
  // four vectors, or three with x in global memory
  const bool skewed = K == 1 && g.nhub > 0;
  if (!skewed && vec * 4 + meta <= CC::SMEM) {
    sh->x_global = 0;
  } else if (vec * 3 + meta <= CC::SMEM) {
    sh->x_global = 1;
  } else {
    return false;
  }
  size_t left = CC::SMEM - meta - vec * (sh->x_global ? 3 : 4);
  sh->smem = CC::SMEM - left;
  // K = 1 with hubs: the leading entries of r (the hubs, when the nodes are
  // ordered by degree) as far as they fit and are worth their load. Otherwise
  // the short rows' indices, with room for an uneven share.
  sh->nhead = sh->col_cap = 0;
  if (skewed) {
    sh->nhead = (int)std::min<int64_t>({g.n, nnz / (4 * sh->grid), (int64_t)(left / sizeof(T))}) & ~1;
    sh->smem += (size_t)sh->nhead * sizeof(T);
  } else {
    const int64_t share = nnz / sh->grid;
    sh->col_cap = (int)std::min<int64_t>(share + share / 4 + 64, (int64_t)(left / 4)) & ~1;
    sh->smem += (size_t)sh->col_cap * 4;
  }
  // two-level sums where every CTA would read tens of kilobytes
  sh->group = !sh->cluster && sh->grid > 32 && K >= 8 ? (sh->grid + 11) / 12 : 0;
  return true;
}

template <typename T, int K, bool SH>
cudaError_t cgc_attributes() {
  static PerDevice attr;
  return attr.once([] {
    cudaError_t e = cudaFuncSetAttribute(cg_coop<T, K, SH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)CoopCfg<T, K>::SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cg_coop<T, K, SH>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
  });
}

// Whether the current device can place a cluster of the kernel at its largest
// (16 CTAs, one per SM, is more than the portable size: a part of a GPU may have
// no 16 free SMs that form one). Asked once per device.
template <typename T, int K, bool SH>
bool cgc_clusters() {
  static PerDevice asked;
  static std::atomic<uint64_t> yes{0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64) return false;
  const cudaError_t e = asked.once([dev] {
    cudaError_t ce = cgc_attributes<T, K, SH>();
    if (ce != cudaSuccess) return ce;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kCoopCluster);
    cfg.blockDim = dim3(CoopCfg<T, K>::TMAX);
    cfg.dynamicSmemBytes = CoopCfg<T, K>::SMEM;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kCoopCluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int num = 0;
    if (cudaOccupancyMaxActiveClusters(&num, cg_coop<T, K, SH>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      num = 0;
    }
    if (num > 0) yes.fetch_or(uint64_t(1) << dev);
    return cudaSuccess;
  });
  if (e != cudaSuccess) (void)cudaGetLastError();
  return (yes.load() >> dev & 1) != 0;
}

// the shape of a solve on the current device
template <typename T, int K>
bool cgc_device_shape(const PhaseGraph& g, int64_t nnz, int sms, bool shifted, bool clusters, CoopShape* sh) {
  clusters = clusters && (shifted ? cgc_clusters<T, K, true>() : cgc_clusters<T, K, false>());
  return cgc_shape<T, K>(g, nnz, sms, clusters, sh);
}

template <typename T, int K, bool SH>
cudaError_t cgc_launch(CoopArgs<T> a, const CoopShape& sh, cudaStream_t s) {
  const cudaError_t ae = cgc_attributes<T, K, SH>();
  if (ae != cudaSuccess) return ae;
  a.long_min = sh.long_min;
  a.nhead = sh.nhead;
  a.ch_log = sh.ch_log;
  a.col_cap = sh.col_cap;
  a.x_global = sh.x_global;
  a.cluster = sh.cluster;
  a.group = sh.group;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sh.grid);
  cfg.blockDim = dim3(sh.threads);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  if (sh.cluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = sh.grid;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, cg_coop<T, K, SH>, a);
}

}  // namespace wl
