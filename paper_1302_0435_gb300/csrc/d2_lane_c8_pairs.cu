// d2_lane_c8_pairs.cu -- pair lists and FP64-throughout solves by lanes
// (d2_lane.cuh) for one shape: 8 lanes a pair, up to 48 x 16 supports.
#include "d2_lane.cuh"

namespace d2k {

using Shape = LaneShape<8, 4, 2, 8>;
// FP64: 16 lanes a pair, so that two pairs share a scan and not four
// (64,000 pairs of 48 x 16: 13.4 -> 10.3 ms; of 24 x 16 5.0 -> 5.7).
using Shape64 = LaneShape<16, 4, 2, 4, double>;

cudaError_t lane_all64_c8(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                          const SolveCfg& cfg, const LaneArgs& A, long long total_obj,
                          long long work, const ExactOut& X, cudaStream_t st) {
  return lane_all64_launch<Shape64>(ob, cv, seg_size, K, cfg, A, total_obj, work, X, st);
}

cudaError_t lane_pairs_c8(const ObjView& ob, const CentView& cv, const PairJob& J,
                          const SolveCfg& cfg, cudaStream_t st) {
  return lane_pairs_launch<Shape, Shape64>(ob, cv, J, cfg, st);
}

cudaError_t stats_lane_c8_pairs(long long out[6]) { return read_unit_stats(out); }

}  // namespace d2k
