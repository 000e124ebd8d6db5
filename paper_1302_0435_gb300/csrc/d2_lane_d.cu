// d2_lane_d.cu -- the lane screen (d2_lane.cuh): 16 centroid supports and 17 to 64 of the bag.
#include "d2_lane.cuh"

namespace d2k {

cudaError_t lane_screen_d(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                          const SolveCfg& cfg, const LaneArgs& A, long long total_obj,
                          long long work, const ExactOut& X, cudaStream_t st) {
#define RUN(...) \
  lane_launch<LaneShape<__VA_ARGS__>>(ob, cv, seg_size, K, cfg, A, total_obj, work, X, st)
  if (cfg.mmax <= 32) return RUN(8, 4, 2, 6);
  if (cfg.mmax <= 48) return RUN(8, 4, 2, 8);
  return RUN(16, 4, 4, 5);
#undef RUN
}

cudaError_t stats_lane_d(long long out[6]) { return read_unit_stats(out); }

}  // namespace d2k
