// Spectral-scale Lanczos kernels (k = 1, double-float basis): launchers.
#define WL_SPEC_KERNELS
#include <algorithm>

#include "wl_host.h"
#include "wl_spec.cuh"

namespace wl {

int sp_blocks() {
  int nb = 0, dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (const void*)sp_s_multi, kPhaseBlock, 0);
  return (nb < 1 ? 1 : nb) * sms;
}

cudaError_t launch_sp_start(const SpArgs& a, int mode, int grid_u, cudaStream_t s) {
  if (mode == 0)
    sp_init<<<grid_u, kPhaseBlock, 0, s>>>(a);
  else
    sp_restart<<<1, 32, 0, s>>>(a.st, mode == 2 ? 1 : 0);
  return cudaGetLastError();
}

// Graphs of more rows take the steps that stream the vectors (eight of them:
// Chung-Lu, 400003 nodes 250 -> 202 us, R-MAT scale 17 about a tenth less; the
// others were 10% to 40% slower by it); up to it the vectors always fit.
constexpr int64_t kSpStreamRows = 250000;

// grid, threads and shared memory of the cooperative steps
static void sp_coop_shape(const SpArgs& a, int64_t nnz, int sms, int* grid, int* threads, size_t* smem, int* nhead) {
  const int64_t units = a.g.n * kSpCoopLpr;
  *grid = (int)std::max<int64_t>(1, std::min<int64_t>(sms, (units + 255) / 256));
  const int64_t rows = coop_rows_local(a.g.n, *grid, kSpCoopCh);
  const int64_t passes = (rows * kSpCoopLpr + kSpCoopThreads - 1) / kSpCoopThreads;
  *threads = (int)std::max<int64_t>(256, (rows * kSpCoopLpr / passes + 31) / 32 * 32);
  const int64_t nslot = rows + (a.nmid + *grid - 1) / *grid + (a.g.nhub + *grid - 1) / *grid;
  const size_t vec = (size_t)nslot * 3 * sizeof(float2);
  *nhead = (int)std::min<int64_t>({a.g.n, nnz / (4 * *grid), (int64_t)((kSpCoopSmem - vec) / sizeof(float2))});
  *smem = vec + (size_t)*nhead * sizeof(float2);
}
// rows and listed rows of a CTA at that limit, three vectors each
static_assert(2 * (kSpStreamRows / 128 + 2 * kSpCoopCh) * 3 * sizeof(float2) <= kSpCoopSmem, "a run's vectors fit");

cudaError_t launch_sp_steps_coop(const SpArgs& a, int64_t nnz, int sms, CoopBar* bar, int j0, int j1, int cap,
                                 int check, double rtol, cudaStream_t s) {
  const bool stream = a.g.n > kSpStreamRows;
  static PerDevice attr;
  if (cudaError_t e = attr.once([] {
        return cudaFuncSetAttribute(sp_coop, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSpCoopSmem);
      });
      e != cudaSuccess)
    return e;
  static PerDevice attr1;
  if (cudaError_t e = attr1.once([] {
        return cudaFuncSetAttribute(sp_k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kK1Smem);
      });
      e != cudaSuccess)
    return e;
  SpCoopArgs ca{a, bar, 0, 0, cap, 0};
  int grid = k1_grid(a.g.n, sms), threads = k1_threads<float2>();
  ca.nhead = k1_head<float2>(a.g.n, nnz, grid);
  size_t smem = k1_smem<float2>(ca.nhead);
  if (!stream) sp_coop_shape(a, nnz, sms, &grid, &threads, &smem, &ca.nhead);
  for (int j = j0; j < j1; j = ca.j1) {
    ca.j0 = j;
    ca.j1 = std::min(j1, (j / check + 1) * check);
    cudaError_t e = cudaMemsetAsync(&bar->count, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    void* args[] = {&ca};
    e = cudaLaunchCooperativeKernel(stream ? (const void*)sp_k1 : (const void*)sp_coop, dim3(grid), dim3(threads), args, smem, s);
    if (e != cudaSuccess) return e;
    sp_eig<<<1, 2 * kSpEigT, 0, s>>>(a.st, rtol);
  }
  return cudaGetLastError();
}

cudaError_t launch_sp_ritz(const SpArgs& a, int grid_u, cudaStream_t s) {
  sp_ritz<<<grid_u, kPhaseBlock, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_sp_round(const SpJob* jobs, const int* off_s, const int* off_u, int np, int grid_s, int grid_u,
                            int steps, int check, unsigned eig_mask, bool any_ritz, bool any_init, SpOut* out,
                            cudaStream_t s) {
  if (np <= 0) return cudaSuccess;
  if (any_ritz) sp_ritz_multi<<<grid_u, kPhaseBlock, 0, s>>>(jobs, off_u, np);
  sp_prep_multi<<<np, 128, 0, s>>>(jobs, np);
  if (any_init) sp_init_multi<<<grid_u, kPhaseBlock, 0, s>>>(jobs, off_u, np);
  for (int st = 0; st < steps; ++st) {
    sp_s_multi<<<grid_s, kPhaseBlock, 0, s>>>(jobs, off_s, np, st);
    sp_u_multi<<<grid_u, kPhaseBlock, 0, s>>>(jobs, off_u, np, st);
    if (eig_mask >> st & 1u) sp_eig_multi<<<np, 2 * kSpEigT, 0, s>>>(jobs, np, st, check);
  }
  sp_pack_multi<<<(np + 127) / 128, 128, 0, s>>>(jobs, np, out);
  return cudaGetLastError();
}

}  // namespace wl
