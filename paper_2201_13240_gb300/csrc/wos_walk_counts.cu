// wos_walk_counts.cu -- small FP32 solves with per-point counts, and small batches: the generic walk kernels
// that run one walk per lane and leave the sums to walk_sum_kernel.
#include "wos_walk_impl.cuh"

namespace wos {

cudaError_t launch_walks_counts_f32(const WalkLaunch& L, int num_sms, cudaStream_t stream) {
  return (L.dim == 2) ? launch_walks_t<2, float, SPREAD_ALWAYS>(L, num_sms, stream)
                      : launch_walks_t<3, float, SPREAD_ALWAYS>(L, num_sms, stream);
}

}  // namespace wos
