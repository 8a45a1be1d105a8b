// pa_eval_lanes_fin1.cu -- the lane-per-chromosome FP32 evaluation
// (pa_eval_lanes.cuh), finite-M SINR, scalar table rows: a translation unit of its
// own so that the variants compile in parallel.
#include "pa_eval_lanes.cuh"

namespace pa {

cudaError_t lanes_dispatch_fin1(int NC, const LanesArgs& a, size_t smem, int num_sms,
                                int64_t tiles, cudaStream_t st) {
  return pick_lanes<1, true>(NC, a, smem, num_sms, tiles, st);
}

}  // namespace pa
