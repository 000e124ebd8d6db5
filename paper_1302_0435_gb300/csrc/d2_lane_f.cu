// d2_lane_f.cu -- the lane screen (d2_lane.cuh): 64 centroid supports.
#include "d2_lane.cuh"

namespace d2k {

cudaError_t lane_screen_f(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                          const SolveCfg& cfg, const LaneArgs& A, long long total_obj,
                          long long work, const ExactOut& X, cudaStream_t st) {
#define RUN(...) \
  lane_launch<LaneShape<__VA_ARGS__>>(ob, cv, seg_size, K, cfg, A, total_obj, work, X, st)
  if (cfg.mmax <= 32) return RUN(32, 16, 4, 3);
  return RUN(32, 16, 4, 4);
#undef RUN
}

cudaError_t stats_lane_f(long long out[6]) { return read_unit_stats(out); }

}  // namespace d2k
