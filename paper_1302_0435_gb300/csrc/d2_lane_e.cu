// d2_lane_e.cu -- the lane screen (d2_lane.cuh): 32 centroid supports and 33 to 64 of the bag.
#include "d2_lane.cuh"

namespace d2k {

cudaError_t lane_screen_e(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                          const SolveCfg& cfg, const LaneArgs& A, long long total_obj,
                          long long work, const ExactOut& X, cudaStream_t st) {
#define RUN(...) \
  lane_launch<LaneShape<__VA_ARGS__>>(ob, cv, seg_size, K, cfg, A, total_obj, work, X, st)
  if (cfg.mmax <= 48) return RUN(16, 8, 4, 5);
  return RUN(16, 8, 4, 6);
#undef RUN
}

cudaError_t stats_lane_e(long long out[6]) { return read_unit_stats(out); }

}  // namespace d2k
