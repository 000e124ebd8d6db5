// d2_lane_b8.cu -- the lane kernels (d2_lane.cuh) for one shape: 8 lanes a pair, up to 32 x 32 supports.
#include "d2_lane.cuh"

namespace d2k {

using Shape = LaneShape<8, 8, 2, 8>;

cudaError_t lane_run_b8(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                        const SolveCfg& cfg, const LaneArgs& A, long long total_obj,
                        long long work, const ExactOut& X, cudaStream_t st) {
  return lane_launch<Shape>(ob, cv, seg_size, K, cfg, A, total_obj, work, X, st);
}

cudaError_t stats_lane_b8(long long out[6]) { return read_unit_stats(out); }

}  // namespace d2k
