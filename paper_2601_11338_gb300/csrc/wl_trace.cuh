// XNysTrace of phi (Alg. 1, step "XNysTrace(Y, Omega)") on the device.
//
//  philox_sketch : Omega (n x M, bfloat16) from Philox4x32-10 (Salmon et al.,
//                  SC'11): element e = i M + j uses counter block e / 4 with key
//                  = seed; words (x0, x1) and (x2, x3) give two Box-Muller pairs
//                  r = sqrt(-2 ln u_a), (r cos 2 pi u_b, r sin 2 pi u_b),
//                  u = (x + 0.5) 2^-32, evaluated in FP64 and rounded to bf16
//                  to nearest even.
//  sketch_rhs    : B = a Omega as FP32 n x K (zero-padded columns), the
//                  right-hand side of Y = phi Omega = M^{-1} (a Omega).
//  gram_cc       : per-CTA partial Grams H = Omega^T Y and G = Y^T Y over a
//                  contiguous row chunk (FP32 products and sums inside a
//                  chunk, FP64 across chunks in gram_reduce).
//  nys_factor, nys_core : with P = H^{-1} (LDL^T, FP64), the leave-one-out
//                  estimates t_i = tr(P G) + (1 - (P G P)_ii) / P_ii, which
//                  equal tr(A_hat_(i)) + w_i^T (A - A_hat_(i)) w_i for the
//                  Nystrom approximation A_hat_(i) = Y_-i (Omega_-i^T Y_-i)^{-1}
//                  Y_-i^T built without column i (Schur-complement identities
//                  for (H_-i)^{-1}); estimate mean(t), error std(t)/sqrt(M).
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "wl_common.cuh"

namespace wl {

constexpr int kMaxSketch = 64;
constexpr int kCoreDoubles = 512;  // results and scratch of the leave-one-out core

__device__ __forceinline__ void philox4x32_10(uint32_t (&c)[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c[0]), lo0 = 0xD2511F53u * c[0];
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c[2]), lo1 = 0xCD9E8D57u * c[2];
    const uint32_t n0 = hi1 ^ c[1] ^ k0;
    const uint32_t n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0;
    c[1] = lo1;
    c[2] = n2;
    c[3] = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
}

// FP64 -> bfloat16 bits, round to nearest even, for finite normal-range inputs
__device__ __forceinline__ uint16_t f64_to_bf16_rne(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned sign = (unsigned)(b >> 63);
  int e = (int)((b >> 52) & 0x7FF);
  const unsigned long long m = b & ((1ull << 52) - 1);
  if (e == 0) return (uint16_t)(sign << 15);  // zero (and FP64 subnormals) -> signed zero
  unsigned long long keep = m >> 45;
  const unsigned long long rest = m & ((1ull << 45) - 1), half = 1ull << 44;
  if (rest > half || (rest == half && (keep & 1ull))) ++keep;
  if (keep == 128ull) {
    keep = 0;
    ++e;
  }
  int fe = e - 1023 + 127;
  if (fe <= 0) return (uint16_t)(sign << 15);
  if (fe >= 255) return (uint16_t)((sign << 15) | 0x7F80u);
  return (uint16_t)((sign << 15) | ((unsigned)fe << 7) | (unsigned)keep);
}

__device__ __forceinline__ float bf16_to_f32(uint16_t h) { return __uint_as_float(((uint32_t)h) << 16); }

#ifdef WL_TRACE_KERNELS
// FP64 Box-Muller pair of the words (xa, xb)
__device__ __forceinline__ void box_muller_f64(uint32_t xa, uint32_t xb, uint16_t* z0, uint16_t* z1) {
  const double s = 1.0 / 4294967296.0;
  const double u0 = ((double)xa + 0.5) * s, u1 = ((double)xb + 0.5) * s;
  const double two_pi = 6.283185307179586;
  const double r = sqrt(-2.0 * log(u0));
  *z0 = f64_to_bf16_rne(r * cos(two_pi * u1));
  *z1 = f64_to_bf16_rne(r * sin(two_pi * u1));
}

// the bfloat16 that every number within eps of z rounds to; false if there is none
__device__ __forceinline__ bool bf16_if_certain(float z, float eps, uint16_t* out) {
  const uint16_t lo = __bfloat16_as_ushort(__float2bfloat16_rn(z - eps));
  const uint16_t hi = __bfloat16_as_ushort(__float2bfloat16_rn(z + eps));
  *out = lo;
  return lo == hi;
}

// The sketch is defined by FP64 Box-Muller rounded to bfloat16, eight bits of
// mantissa, and this GPU's FP64 pipe (1/64 of FP32) made its logarithm and
// sine the whole cost. So a pair is computed in FP32 with an error bound, and
// only where the bound leaves the rounding open (0.3% of the pairs) in FP64:
// bit for bit the same Omega. The open pairs are queued and done together, a
// thread each, when the CTA has finished its share. Bound: r = sqrt(-2 ln u)
// to 4.6e-7 relative (u near 1 through log1p of the exact 1 - u; FP32 rounding
// of u, logf, sqrtf), the sine and cosine to 3.1e-7 absolute (argument
// rounded to 2^-24 half turns, sincospif): together below 8e-7 r; 1e-6 r is
// used. 131072 x 64: 30 us (all in FP64: 637 us).
constexpr int kPhiloxQueue = 512;
constexpr int kPhiloxBlock = 256;

__global__ void __launch_bounds__(kPhiloxBlock) philox_sketch(uint16_t* omega, int64_t total, uint64_t seed) {
  __shared__ int64_t s_q[kPhiloxQueue];  // open pairs: 2 x block + (0 or 1)
  __shared__ int s_n;
  const int64_t nblk = (total + 3) / 4;
  const uint32_t k0 = (uint32_t)(seed & 0xFFFFFFFFull), k1 = (uint32_t)(seed >> 32);
  if (threadIdx.x == 0) s_n = 0;
  __syncthreads();
  auto words = [&](int64_t b, uint32_t (&c)[4]) {
    c[0] = (uint32_t)((uint64_t)b & 0xFFFFFFFFull);
    c[1] = (uint32_t)((uint64_t)b >> 32);
    c[2] = c[3] = 0u;
    philox4x32_10(c, k0, k1);
  };
  for (int64_t b = (int64_t)blockIdx.x * kPhiloxBlock + threadIdx.x; b < nblk;
       b += (int64_t)gridDim.x * kPhiloxBlock) {
    uint32_t c[4];
    words(b, c);
    uint16_t z[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t xa = c[2 * h], xb = c[2 * h + 1];
      const float s32 = 2.3283064365386963e-10f;  // 2^-32
      const float lnu = xa >= 0x80000000u ? log1pf(-(((float)(~xa) + 0.5f) * s32)) : logf(((float)xa + 0.5f) * s32);
      const float r = sqrtf(-2.0f * lnu);
      float sn, cs;
      sincospif(((float)(int)xb + 0.5f) * (2.0f * s32), &sn, &cs);
      const float eps = 1e-6f * r;
      const bool ok0 = bf16_if_certain(r * cs, eps, &z[2 * h]);
      const bool ok1 = bf16_if_certain(r * sn, eps, &z[2 * h + 1]);
      if (!(ok0 && ok1)) {
        const int q = atomicAdd(&s_n, 1);
        if (q < kPhiloxQueue)
          s_q[q] = 2 * b + h;
        else
          box_muller_f64(xa, xb, &z[2 * h], &z[2 * h + 1]);
      }
    }
    if (b * 4 + 3 < total) {
      *reinterpret_cast<uint2*>(omega + b * 4) =
          make_uint2((uint32_t)z[0] | ((uint32_t)z[1] << 16), (uint32_t)z[2] | ((uint32_t)z[3] << 16));
    } else {
      for (int q = 0; q < 4; ++q)
        if (b * 4 + q < total) omega[b * 4 + q] = z[q];
    }
  }
  __syncthreads();
  const int nq = min(s_n, kPhiloxQueue);
  for (int q = threadIdx.x; q < nq; q += kPhiloxBlock) {
    const int64_t b = s_q[q] >> 1;
    const int h = (int)(s_q[q] & 1);
    uint32_t c[4];
    words(b, c);
    uint16_t z0, z1;
    box_muller_f64(h ? c[2] : c[0], h ? c[3] : c[1], &z0, &z1);
    const int64_t e = b * 4 + 2 * h;
    if (e < total) omega[e] = z0;
    if (e + 1 < total) omega[e + 1] = z1;
  }
}

// B[i, j] = a * Omega[i, j] (j < M), 0 for M <= j < K
__global__ void sketch_rhs(const uint16_t* omega, int64_t n, int M, int K, float a, float* B) {
  const int64_t total = n * K;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / K;
    const int j = (int)(e % K);
    B[e] = (j < M) ? a * bf16_to_f32(omega[i * M + j]) : 0.0f;
  }
}

// Omega as an FP64 n x K block (zero-padded columns): the start block of the
// return-probability Lanczos
__global__ void sketch_block_f64(const uint16_t* omega, int64_t n, int M, int K, double* B) {
  const int64_t total = n * K;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / K;
    const int j = (int)(e % K);
    B[e] = (j < M) ? (double)bf16_to_f32(omega[i * M + j]) : 0.0;
  }
}

// FP64 -> FP32 (the Gram of the estimator takes FP32 Y)
__global__ void to_f32(const double* X, int64_t total, float* Y) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x)
    Y[e] = (float)X[e];
}

// ---------------------------------------------------------------- Gram on CUDA cores
// Grid of G CTAs of kGramThreads, CTA g sums rows [g * chunk, min(n, (g+1) *
// chunk)) of the 2M x M block [Omega Y]^T Y (M <= 64). Thread (tr, tc) =
// (t / 8, t % 8) owns the 8 x 8 outputs of X columns 8 tr .. 8 tr + 7 (X =
// [Omega Y], 128 columns) and Y columns 8 tc .. 8 tc + 7: per staged row it
// reads two float4 of X and two of Y from shared memory for 64 FMAs. Tiles
// of kGramRows rows alternate between two buffers; the next tile's loads are
// issued into registers before the current tile's products.
constexpr int kGramRows = 32;     // rows staged per tile
constexpr int kGramThreads = 128;
constexpr int kGramLoads = kGramRows * kMaxSketch / kGramThreads;  // elements of Omega (and of Y) per thread and tile

__global__ void __launch_bounds__(kGramThreads) gram_cc(const uint16_t* omega, const float* Y, int64_t n, int M,
                                                        int K, int64_t chunk, float* partial /* G x 2M x M */) {
  __shared__ __align__(16) float sX[2][kGramRows][2 * kMaxSketch];  // [Omega_i, Y_i]
  const int tid = threadIdx.x;
  const int tr = tid >> 3, tc = tid & 7;
  const int64_t r0 = (int64_t)blockIdx.x * chunk;
  const int64_t r1 = min(n, r0 + chunk);
  float acc[8][8];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) acc[a][b] = 0.f;
  float po[kGramLoads], py[kGramLoads];  // the next tile, in flight
  auto fetch = [&](int64_t base) {
#pragma unroll
    for (int u = 0; u < kGramLoads; ++u) {
      const int e = tid + u * kGramThreads, i = e / kMaxSketch, j = e % kMaxSketch;
      const int64_t r = base + i;
      float om = 0.f, y = 0.f;
      if (r < r1 && j < M) {
        om = bf16_to_f32(omega[r * M + j]);
        y = Y[r * K + j];
      }
      po[u] = om;
      py[u] = y;
    }
  };
  auto stash = [&](int buf) {
#pragma unroll
    for (int u = 0; u < kGramLoads; ++u) {
      const int e = tid + u * kGramThreads, i = e / kMaxSketch, j = e % kMaxSketch;
      sX[buf][i][j] = po[u];
      sX[buf][i][kMaxSketch + j] = py[u];
    }
  };
  if (r0 < r1) fetch(r0);
  int buf = 0;
  for (int64_t base = r0; base < r1; base += kGramRows) {
    const int rows = (int)min((int64_t)kGramRows, r1 - base);
    stash(buf);
    __syncthreads();
    if (base + kGramRows < r1) fetch(base + kGramRows);
    for (int i = 0; i < rows; ++i) {
      const float4 x0 = *reinterpret_cast<const float4*>(&sX[buf][i][8 * tr]);
      const float4 x1 = *reinterpret_cast<const float4*>(&sX[buf][i][8 * tr + 4]);
      const float4 y0 = *reinterpret_cast<const float4*>(&sX[buf][i][kMaxSketch + 8 * tc]);
      const float4 y1 = *reinterpret_cast<const float4*>(&sX[buf][i][kMaxSketch + 8 * tc + 4]);
      const float xv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
      const float yv[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) acc[a][b] = fmaf(xv[a], yv[b], acc[a][b]);
    }
    buf ^= 1;  // the other buffer is written next: no barrier needed before it
  }
  // rows of the 2M block: index rr in [0, 128): rr < 64 -> Omega column rr, else Y column rr - 64
  float* out = partial + (size_t)blockIdx.x * (2 * kMaxSketch) * kMaxSketch;
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) out[(8 * tr + a) * kMaxSketch + (8 * tc + b)] = acc[a][b];
}

// out[r * 64 + c] = sum_g partial[g][r][c] in FP64, fixed order
__global__ void gram_reduce(const float* partial, int G, double* out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 2 * kMaxSketch * kMaxSketch) return;
  double s = 0.0;
  for (int g = 0; g < G; ++g) s += (double)partial[(size_t)g * 2 * kMaxSketch * kMaxSketch + e];
  out[e] = s;
}

// ---------------------------------------------------------------- Gram in FP64 (CUDA cores)
// The same block [Omega Y]^T Y from an FP64 Y (the FP64 and refined forms of
// the estimators), FP64 products and sums throughout. Bound by the FP64 pipe
// (2 lanes per clock and SM: a warp's DFMA holds its scheduler's pipe for 64
// cycles, so shared-memory reads and loads hide behind it). So the work is
// cut to what the M columns need: 4 x 4 output tiles of H = Omega^T Y (all)
// and of G = Y^T Y (the upper triangle), one tile per thread, and the rows of
// a staged tile dealt to `groups` copies of the tile set where it is small.
// One CTA per SM over the whole chip, however few the rows. Measured with 131072 x 64:
// 1550 us (a fixed 128 x 64 block per CTA of 4096 rows, 32 CTAs: 8766 us);
// with 62500 x 30: 195 us (16 CTAs and the block padded to 64 columns: 8283 us).
constexpr int kGramRows64 = 32;       // rows staged per tile
constexpr int kGramThreads64 = 512;   // most threads of a CTA
constexpr int kGramGroups64 = 16;     // most copies of the tile set in a CTA
__host__ __device__ constexpr int gram64_tiles(int M) {  // 4 x 4 tiles of H and of G's upper triangle
  const int nb = (M + 3) / 4;
  return nb * nb + nb * (nb + 1) / 2;
}
__host__ __device__ constexpr int gram64_groups(int M) {
  const int g = kGramThreads64 / gram64_tiles(M);
  return g < 1 ? 1 : (g > kGramGroups64 ? kGramGroups64 : g);
}
// tile t -> (ti, tj): H tiles row by row, then G tiles with ti <= tj
__device__ __forceinline__ void gram64_tile(int t, int nb, bool* is_g, int* ti, int* tj) {
  *is_g = t >= nb * nb;
  if (!*is_g) {
    *ti = t / nb;
    *tj = t % nb;
    return;
  }
  int q = t - nb * nb, r = 0;
  while (q >= nb - r) {
    q -= nb - r;
    ++r;
  }
  *ti = r;
  *tj = r + q;
}

// partial: gridDim.x blocks of gram64_tiles(M) x 16 doubles
__global__ void __launch_bounds__(kGramThreads64) gram_f64(const uint16_t* omega, const double* Y, int64_t n, int M,
                                                           int K, int64_t chunk, double* partial) {
  // [Omega_i, Y_i] of the staged rows; the groups' accumulators at the end
  __shared__ __align__(16) double sX[kGramRows64][2 * kMaxSketch];
  const int nb = (M + 3) / 4, W = 4 * nb, nt = gram64_tiles(M), groups = gram64_groups(M);
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int grp = tid / nt, t = tid % nt;
  const bool live = grp < groups;
  bool is_g;
  int ti, tj;
  gram64_tile(t, nb, &is_g, &ti, &tj);
  const int xo = (is_g ? kMaxSketch : 0) + 4 * ti, yo = kMaxSketch + 4 * tj;
  const int64_t r0 = (int64_t)blockIdx.x * chunk;
  const int64_t r1 = min(n, r0 + chunk);
  double acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
  for (int64_t base = r0; base < r1; base += kGramRows64) {
    const int rows = (int)min((int64_t)kGramRows64, r1 - base);
    __syncthreads();
    for (int e = tid; e < kGramRows64 * W; e += nthr) {
      const int i = e / W, j = e % W;
      double om = 0.0, y = 0.0;
      if (i < rows && j < M) {
        om = (double)bf16_to_f32(omega[(base + i) * M + j]);
        y = Y[(base + i) * K + j];
      }
      sX[i][j] = om;
      sX[i][kMaxSketch + j] = y;
    }
    __syncthreads();
    if (live) {
      for (int i = grp; i < rows; i += groups) {
        const double2 x01 = *reinterpret_cast<const double2*>(&sX[i][xo]);
        const double2 x23 = *reinterpret_cast<const double2*>(&sX[i][xo + 2]);
        const double2 y01 = *reinterpret_cast<const double2*>(&sX[i][yo]);
        const double2 y23 = *reinterpret_cast<const double2*>(&sX[i][yo + 2]);
        const double xv[4] = {x01.x, x01.y, x23.x, x23.y};
        const double yv[4] = {y01.x, y01.y, y23.x, y23.y};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] = fma(xv[a], yv[b], acc[a][b]);
      }
    }
  }
  double* out = partial + ((size_t)blockIdx.x * nt + t) * 16;
  if (groups > 1) {  // the groups' sums added in order, 16 doubles per tile at a time
    // sX holds 4096 doubles: nt * 16 <= 512 / 2 * 16 of them, as groups > 1
    double* s = &sX[0][0];
    for (int g = 0; g < groups; ++g) {
      __syncthreads();
      if (live && grp == g) {
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            if (g > 0) acc[a][b] += s[t * 16 + a * 4 + b];
            s[t * 16 + a * 4 + b] = acc[a][b];
          }
      }
    }
    if (!live || grp != groups - 1) return;
  } else if (!live) {
    return;
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) out[a * 4 + b] = acc[a][b];
}

// out (128 x 64, zeroed): H in rows 0..63, G in rows 64..127, both triangles;
// 8 threads per entry add the CTAs' partials in a fixed order
__global__ void __launch_bounds__(256) gram_reduce_f64(const double* partial, int G, int M, double* out) {
  __shared__ double s[8][32];
  const int nb = (M + 3) / 4, nt = gram64_tiles(M);
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  double v = 0.0;
  if (e < nt * 16) {
#pragma unroll 4
    for (int g = sl; g < G; g += 8) v += partial[(size_t)g * nt * 16 + e];
  }
  s[sl][lane] = v;
  __syncthreads();
  if (sl != 0 || e >= nt * 16) return;
#pragma unroll
  for (int q = 1; q < 8; ++q) v += s[q][lane];
  bool is_g;
  int ti, tj;
  gram64_tile(e / 16, nb, &is_g, &ti, &tj);
  const int r = 4 * ti + (e % 16) / 4, c = 4 * tj + e % 4;
  if (r >= M || c >= M) return;
  if (!is_g) {
    out[r * kMaxSketch + c] = v;
  } else {
    out[(kMaxSketch + r) * kMaxSketch + c] = v;
    if (ti != tj) out[(kMaxSketch + c) * kMaxSketch + r] = v;
  }
}

// ---------------------------------------------------------------- FP64 leave-one-out core
// gram: 128 x 64 doubles, rows 0..63 = Omega^T Y (H), rows 64..127 = Y^T Y (G).
// out[0] = estimate, out[1] = error estimate, out[2] = status (0 ok, 1 not PD), out[8 + i] = t_i;
// out holds kCoreDoubles, the rest is scratch.
//
// An FP64 operation waits about a hundred clocks for the one before it, and
// one SM does two a clock, so the core is split: nys_factor (one CTA)
// brings H = L D L^T and L^{-1} out of the same M elimination steps, all
// rows at once with one reciprocal per step; nys_core (one CTA per column i
// of P = H^{-1}) then needs two products with M terms a thread. Measured at
// M = 64: 97 + 33 us (one CTA for all of it, a thread per column of P and two
// triangular solves in sequence: 440 us).
constexpr int kFactorThreads = 512;
constexpr int kCoreAux = 8 + kMaxSketch;  // out[kCoreAux + 3 i ..]: (G P)_ii, (P G P)_ii, P_ii; then the ticket

// gram rows 0..63 become L^{-1} (unit lower triangle) with 1 / D_j on the diagonal
__global__ void __launch_bounds__(kFactorThreads) nys_factor(double* gram, int M, double* out) {
  extern __shared__ double sm[];
  constexpr int LD = kMaxSketch + 1;
  double* H = sm;                          // lower triangle, eliminated in place
  double* R = H + kMaxSketch * LD;         // L^{-1}
  double* s_l = R + kMaxSketch * LD;       // column k of L
  double* s_rd = s_l + kMaxSketch;         // 1 / D_k
  const int tid = threadIdx.x;
  for (int e = tid; e < M * M; e += kFactorThreads) {
    const int r = e / M, c = e % M;
    if (c <= r) H[r * LD + c] = 0.5 * (gram[r * kMaxSketch + c] + gram[c * kMaxSketch + r]);
    R[r * LD + c] = r == c ? 1.0 : 0.0;
  }
  int bad = 0;
  __syncthreads();
  for (int k = 0; k < M; ++k) {
    if (tid < kMaxSketch) {
      const double d = H[k * LD + k];
      if (!(d > 0.0)) bad = 1;
      const double rd = 1.0 / fmax(d, 1e-300);
      if (tid == 0) s_rd[k] = rd;
      if (tid > k && tid < M) s_l[tid] = H[tid * LD + k] * rd;
    }
    __syncthreads();
    // row i loses l_ik times row k: columns 0..k of L^{-1}, columns k + 1..i of H
    for (int i = k + 1 + (tid >> 4); i < M; i += kFactorThreads / 16) {
      const double l = s_l[i];
      for (int c = tid & 15; c <= i; c += 16) {
        if (c <= k)
          R[i * LD + c] = fma(-l, R[k * LD + c], R[i * LD + c]);
        else
          H[i * LD + c] = fma(-l, H[c * LD + k], H[i * LD + c]);
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < M * M; e += kFactorThreads) {
    const int r = e / M, c = e % M;
    gram[r * kMaxSketch + c] = r == c ? s_rd[r] : R[r * LD + c];
  }
  if (tid == 0) {
    out[2] = bad ? 1.0 : 0.0;
    *reinterpret_cast<unsigned long long*>(out + kCoreAux + 3 * kMaxSketch) = 0ull;  // nys_core's ticket
  }
}

// CTA i: column i of P = L^{-T} D^{-1} L^{-1}, (G P)_ii and (P G P)_ii; the
// last CTA forms t_i = tr(P G) + (1 - (P G P)_ii) / P_ii and its statistics
__global__ void __launch_bounds__(kMaxSketch) nys_core(const double* gram, int M, double* out) {
  __shared__ double s_p[kMaxSketch], s_v[kMaxSketch];
  __shared__ int s_last;
  const int i = blockIdx.x, k = threadIdx.x;
  const double* G = gram + kMaxSketch * kMaxSketch;
  // v_j = (L^{-1})_ji / D_j
  if (k < M) s_v[k] = k < i ? 0.0 : (k == i ? 1.0 : gram[k * kMaxSketch + i]) * gram[k * kMaxSketch + k];
  __syncthreads();
  double p = 0.0;
  if (k < M) {
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    const int j0 = max(k + 1, i);
    int j = j0;
    for (; j + 3 < M; j += 4)
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = fma(gram[(j + u) * kMaxSketch + k], s_v[j + u], a[u]);
    for (; j < M; ++j) a[0] = fma(gram[j * kMaxSketch + k], s_v[j], a[0]);
    p = (a[0] + a[1]) + (a[2] + a[3]) + s_v[k];
    s_p[k] = p;
  }
  __syncthreads();
  double g = 0.0;
  if (k < M) {
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    int j = 0;
    for (; j + 3 < M; j += 4)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        a[u] = fma(0.5 * (G[(j + u) * kMaxSketch + k] + G[k * kMaxSketch + j + u]), s_p[j + u], a[u]);
    for (; j < M; ++j) a[0] = fma(0.5 * (G[j * kMaxSketch + k] + G[k * kMaxSketch + j]), s_p[j], a[0]);
    g = (a[0] + a[1]) + (a[2] + a[3]);
    s_v[k] = p * g;
    if (k == i) {
      out[kCoreAux + 3 * i] = g;
      out[kCoreAux + 3 * i + 2] = p;
    }
  }
  __syncthreads();
  if (k == 0) {
    double q = 0.0;
    for (int j = 0; j < M; ++j) q += s_v[j];
    out[kCoreAux + 3 * i + 1] = q;
  }
  __threadfence();
  __syncthreads();
  if (k == 0)
    s_last = atomicAdd(reinterpret_cast<unsigned long long*>(out + kCoreAux + 3 * kMaxSketch), 1ull) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (k < M) s_p[k] = __ldcg(out + kCoreAux + 3 * k);
  __syncthreads();
  double t = 0.0;
  if (k < M) {
    double S = 0.0;
    for (int j = 0; j < M; ++j) S += s_p[j];
    t = S + (1.0 - __ldcg(out + kCoreAux + 3 * k + 1)) / __ldcg(out + kCoreAux + 3 * k + 2);
    s_v[k] = t;
    out[8 + k] = t;
  }
  __syncthreads();
  if (k == 0) {
    double mean = 0.0;
    for (int j = 0; j < M; ++j) mean += s_v[j];
    mean /= M;
    double var = 0.0;
    for (int j = 0; j < M; ++j) var += (s_v[j] - mean) * (s_v[j] - mean);
    var /= (M - 1);
    out[0] = mean;
    out[1] = sqrt(var / M);
  }
}

#endif  // WL_TRACE_KERNELS

}  // namespace wl
