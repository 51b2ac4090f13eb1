// FP64 instances of the cooperative CG kernel, K = 1, 2, 4, ..., 64 columns.
#include <algorithm>

#include "wl_coop.cuh"
#include "wl_host.h"

namespace wl {

template <int K>
static bool run(const CoopArgs<double>& a, int64_t nnz, int sms, bool clusters, cudaStream_t s, cudaError_t* e) {
  CoopShape sh;
  if (!cgc_device_shape<double, K>(a.a.g, nnz, sms, a.a.dshift != nullptr, clusters, &sh)) return false;
  *e = a.a.dshift ? cgc_launch<double, K, true>(a, sh, s) : cgc_launch<double, K, false>(a, sh, s);
  return true;
}

bool launch_cg_coop_f64(int K, const CoopArgs<double>& a, int64_t nnz, int sms, bool clusters, cudaStream_t s,
                        cudaError_t* e) {
  switch (K) {
    case 1: return run<1>(a, nnz, sms, clusters, s, e);
    case 2: return run<2>(a, nnz, sms, clusters, s, e);
    case 4: return run<4>(a, nnz, sms, clusters, s, e);
    case 8: return run<8>(a, nnz, sms, clusters, s, e);
    case 16: return run<16>(a, nnz, sms, clusters, s, e);
    case 32: return run<32>(a, nnz, sms, clusters, s, e);
    case 64: return run<64>(a, nnz, sms, clusters, s, e);
  }
  return false;
}

bool cg_coop_fits_f64(int K, const PhaseGraph& g, int64_t nnz, int sms, bool shifted, bool clusters) {
  CoopShape sh;
  switch (K) {
    case 1: return cgc_device_shape<double, 1>(g, nnz, sms, shifted, clusters, &sh);
    case 2: return cgc_device_shape<double, 2>(g, nnz, sms, shifted, clusters, &sh);
    case 4: return cgc_device_shape<double, 4>(g, nnz, sms, shifted, clusters, &sh);
    case 8: return cgc_device_shape<double, 8>(g, nnz, sms, shifted, clusters, &sh);
    case 16: return cgc_device_shape<double, 16>(g, nnz, sms, shifted, clusters, &sh);
    case 32: return cgc_device_shape<double, 32>(g, nnz, sms, shifted, clusters, &sh);
    case 64: return cgc_device_shape<double, 64>(g, nnz, sms, shifted, clusters, &sh);
  }
  return false;
}

// the shape alone, for a device of `sms` SMs (no GPU needed)
bool cg_coop_shape_f64(int K, const PhaseGraph& g, int64_t nnz, int sms, bool clusters, CoopShape* sh) {
  switch (K) {
    case 1: return cgc_shape<double, 1>(g, nnz, sms, clusters, sh);
    case 2: return cgc_shape<double, 2>(g, nnz, sms, clusters, sh);
    case 4: return cgc_shape<double, 4>(g, nnz, sms, clusters, sh);
    case 8: return cgc_shape<double, 8>(g, nnz, sms, clusters, sh);
    case 16: return cgc_shape<double, 16>(g, nnz, sms, clusters, sh);
    case 32: return cgc_shape<double, 32>(g, nnz, sms, clusters, sh);
    case 64: return cgc_shape<double, 64>(g, nnz, sms, clusters, sh);
  }
  return false;
}

}  // namespace wl
