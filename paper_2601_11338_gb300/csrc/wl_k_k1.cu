// One-column kernels: cooperative CG and the double-float residual.
#include <algorithm>

#include "wl_host.h"
#include "wl_k1.cuh"

namespace wl {

template <typename T, bool SH>
static cudaError_t run_cg(CoopArgs<T> a, int64_t nnz, int sms, cudaStream_t s) {
  static PerDevice attr;
  if (cudaError_t e = attr.once([] {
        return cudaFuncSetAttribute(cg_k1<T, SH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kK1Smem);
      });
      e != cudaSuccess)
    return e;
  const int grid = k1_grid(a.a.g.n, sms);
  a.nhead = k1_head<T>(a.a.g.n, nnz, grid);
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel((const void*)cg_k1<T, SH>, dim3(grid), dim3(k1_threads<T>()), args,
                                     k1_smem<T>(a.nhead), s);
}

template <typename T>
cudaError_t launch_cg_k1(const CoopArgs<T>& a, int64_t nnz, int sms, cudaStream_t s) {
  return a.a.dshift ? run_cg<T, true>(a, nnz, sms, s) : run_cg<T, false>(a, nnz, sms, s);
}
template cudaError_t launch_cg_k1<float>(const CoopArgs<float>&, int64_t, int, cudaStream_t);
template cudaError_t launch_cg_k1<double>(const CoopArgs<double>&, int64_t, int, cudaStream_t);

template <bool SH>
static cudaError_t run_res(const DfResArgs& a, int64_t nnz, int sms, cudaStream_t s) {
  static PerDevice attr;
  if (cudaError_t e = attr.once([] {
        return cudaFuncSetAttribute(df_res_k1<SH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kK1Smem);
      });
      e != cudaSuccess)
    return e;
  const int grid = k1_grid(a.g.n, sms), nhead = k1_head<float>(a.g.n, nnz, grid);
  df_res_k1<SH><<<grid, k1_threads<float>(), k1_smem<float>(nhead), s>>>(a, nhead);
  return cudaGetLastError();
}

cudaError_t launch_df_res_k1(const DfResArgs& a, int64_t nnz, int sms, cudaStream_t s) {
  return a.dsh_h ? run_res<true>(a, nnz, sms, s) : run_res<false>(a, nnz, sms, s);
}

}  // namespace wl
