// d2_lane_c.cu -- the lane screen (d2_lane.cuh): 32 centroid supports, masks of 64 bits, larger bags.
#include "d2_lane.cuh"

namespace d2k {

cudaError_t lane_screen_c(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                          const SolveCfg& cfg, const LaneArgs& A, long long total_obj,
                          long long work, const ExactOut& X, cudaStream_t st) {
#define RUN(...) \
  lane_launch<LaneShape<__VA_ARGS__>>(ob, cv, seg_size, K, cfg, A, total_obj, work, X, st)
  if (cfg.mmax <= 24) return RUN(8, 8, 2, 7);
  return RUN(8, 8, 2, 8);
#undef RUN
}

cudaError_t stats_lane_c(long long out[6]) { return read_unit_stats(out); }

}  // namespace d2k
