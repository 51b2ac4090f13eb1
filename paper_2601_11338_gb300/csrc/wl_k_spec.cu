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
// others were 10% to 40% slower by it), and any graph whose vectors don't fit
// in the SMs there are (fewer than some 130).
constexpr int64_t kSpStreamRows = 250000;

// grid, threads and shared memory of the cooperative steps on `sms` SMs
SpShape sp_coop_shape(int64_t n, int64_t nnz, int nmid, int nhub, int sms) {
  SpShape sh;
  const int64_t units = n * kSpCoopLpr;
  sh.grid = (int)std::max<int64_t>(1, std::min<int64_t>(sms, (units + 255) / 256));
  const int64_t rows = coop_rows_local(n, sh.grid, kSpCoopCh);
  const int64_t nslot = rows + (nmid + sh.grid - 1) / sh.grid + (nhub + sh.grid - 1) / sh.grid;
  const size_t vec = (size_t)nslot * 3 * sizeof(float2);
  sh.stream = n > kSpStreamRows || vec > kSpCoopSmem;
  if (sh.stream) {
    sh.grid = k1_grid(n, sms);
    sh.threads = k1_threads<float2>();
    sh.nhead = k1_head<float2>(n, nnz, sh.grid);
    sh.smem = k1_smem<float2>(sh.nhead);
    return sh;
  }
  const int64_t passes = (rows * kSpCoopLpr + kSpCoopThreads - 1) / kSpCoopThreads;
  sh.threads = (int)std::max<int64_t>(256, (rows * kSpCoopLpr / passes + 31) / 32 * 32);
  sh.nhead = (int)std::min<int64_t>({n, nnz / (4 * sh.grid), (int64_t)((kSpCoopSmem - vec) / sizeof(float2))});
  sh.smem = vec + (size_t)sh.nhead * sizeof(float2);
  return sh;
}

cudaError_t launch_sp_steps_coop(const SpArgs& a, int64_t nnz, int sms, CoopBar* bar, int j0, int j1, int cap,
                                 int check, double rtol, cudaStream_t s) {
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
  const SpShape sh = sp_coop_shape(a.g.n, nnz, a.nmid, a.g.nhub, sms);
  SpCoopArgs ca{a, bar, 0, 0, cap, sh.nhead};
  for (int j = j0; j < j1; j = ca.j1) {
    ca.j0 = j;
    ca.j1 = std::min(j1, (j / check + 1) * check);
    cudaError_t e = cudaMemsetAsync(&bar->count, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    void* args[] = {&ca};
    e = cudaLaunchCooperativeKernel(sh.stream ? (const void*)sp_k1 : (const void*)sp_coop, dim3(sh.grid),
                                    dim3(sh.threads), args, sh.smem, s);
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
