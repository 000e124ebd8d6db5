// d2_lane_e6_pairs.cu -- pair lists and FP64-throughout solves by lanes
// (d2_lane.cuh) for one shape: 16 lanes a pair, up to 64 x 32 supports.
#include "d2_lane.cuh"

namespace d2k {

using Shape = LaneShape<16, 8, 4, 6>;
// FP64: a warp a pair, whose candidates then last as long as they
// can (64,000 uneven pairs, 64 x 32: 12.2 -> 7.8 ms).
using Shape64 = LaneShape<32, 8, 4, 3, double>;

cudaError_t lane_all64_e6(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                          const SolveCfg& cfg, const LaneArgs& A, long long total_obj,
                          long long work, const ExactOut& X, cudaStream_t st) {
  return lane_all64_launch<Shape64>(ob, cv, seg_size, K, cfg, A, total_obj, work, X, st);
}

cudaError_t lane_pairs_e6(const ObjView& ob, const CentView& cv, const PairJob& J,
                          const SolveCfg& cfg, cudaStream_t st) {
  return lane_pairs_launch<Shape, Shape64>(ob, cv, J, cfg, st);
}

cudaError_t stats_lane_e6_pairs(long long out[6]) { return read_unit_stats(out); }

}  // namespace d2k
