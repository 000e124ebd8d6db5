// d2_lane_a.cu -- the lane screen (d2_lane.cuh): 16 centroid supports, masks of 32 bits.
#include "d2_lane.cuh"

namespace d2k {

cudaError_t lane_screen_a(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                          const SolveCfg& cfg, const LaneArgs& A, long long total_obj,
                          long long work, const ExactOut& X, cudaStream_t st) {
#define RUN(...) \
  lane_launch<LaneShape<__VA_ARGS__>>(ob, cv, seg_size, K, cfg, A, total_obj, work, X, st)
  if (cfg.mmax <= 8) return RUN(4, 4, 1, 6);
  if (cfg.mmax <= 12) return RUN(4, 4, 1, 7);
  return RUN(4, 4, 1, 8);
#undef RUN
}

cudaError_t stats_lane_a(long long out[6]) { return read_unit_stats(out); }

}  // namespace d2k
