// d2_lane_a8_pairs.cu -- pair lists and FP64-throughout solves by lanes
// (d2_lane.cuh) for one shape: 4 lanes a pair, up to 16 x 16 supports.
#include "d2_lane.cuh"

namespace d2k {

using Shape = LaneShape<4, 4, 1, 8>;
using Shape64 = LaneShape<4, 4, 1, 8, double>;

cudaError_t lane_all64_a8(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                          const SolveCfg& cfg, const LaneArgs& A, long long total_obj,
                          long long work, const ExactOut& X, cudaStream_t st) {
  return lane_all64_launch<Shape64>(ob, cv, seg_size, K, cfg, A, total_obj, work, X, st);
}

cudaError_t lane_pairs_a8(const ObjView& ob, const CentView& cv, const PairJob& J,
                          const SolveCfg& cfg, cudaStream_t st) {
  return lane_pairs_launch<Shape, Shape64>(ob, cv, J, cfg, st);
}

cudaError_t stats_lane_a8_pairs(long long out[6]) { return read_unit_stats(out); }

}  // namespace d2k
