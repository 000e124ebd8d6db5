// d2_lane.cu -- the FP32 screen of an assignment with several pairs per warp
// (d2_lane.cuh): object masses, lists of the pairs to solve, the chunks and
// shapes of the launches, and the merge of a pair's intervals into each
// object's candidates.
#include "d2_lane.cuh"

namespace d2k {
namespace {

// Ranks of the rows along each object's principal direction, one warp per
// object: the orders of the ranked staircase (order_rows in d2_solve.cuh).
__global__ void __launch_bounds__(128) k_lane_axes(ObjView ob, int mmax, const long long* mass,
                                                   const unsigned char* bad, int mstride,
                                                   unsigned char* rows, float* axes) {
  __shared__ long long P[4][64], Pr[4][64];
  __shared__ int rank[4][64], id[4][64];
  __shared__ float mu[4][256], dir[4][256], proj[4][64];
  Grp<32> g;
  const int w = threadIdx.x >> 5;
  const int d = ob.d;
  for (long long i = (long long)blockIdx.x * 4 + w; i < ob.count; i += (long long)gridDim.x * 4) {
    if (bad[i]) continue;
    const long long o0 = ob.off[i];
    const int m = (int)(ob.off[i + 1] - o0);
    long long carry = 0;
    for (int b = 0; b < m; b += 32) {  // inclusive prefix of the masses
      const int a = b + g.lane;
      long long v = a < m ? mass[i * mstride + a] : 0LL;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, v, o);
        if (g.lane >= o) v += u;
      }
      v += carry;
      if (a < m) P[w][a] = v;
      carry = __shfl_sync(0xffffffffu, v, 31);
    }
    __syncwarp();
    PairMem<float> s{};
    s.P = P[w]; s.Pr = Pr[w]; s.rrank = rank[w]; s.rid = id[w];
    s.mu = mu[w]; s.dir = dir[w]; s.proj = proj[w];
    order_rows<32>(g, s, ob, o0, m, d);
    for (int a = g.lane; a < m; a += 32) rows[i * mstride + a] = (unsigned char)id[w][a];
    for (int k = g.lane; k < d; k += 32) {
      axes[i * 2 * d + k] = mu[w][k];
      axes[i * 2 * d + d + k] = dir[w][k];
    }
    __syncwarp();
  }
}

// The kept pairs of the chunk (bits of cfg.keep): a thread counts its
// object's, a block takes its run of the list with one addition, so the list
// is nearly in object order and an object's pairs are together, centroids
// increasing (ostart: its first entry).
__global__ void __launch_bounds__(256) k_lane_list(LaneArgs A, long long total_obj,
                                                   const unsigned* keep, int kw, uint2* list,
                                                   unsigned long long* ostart) {
  __shared__ unsigned wsum[8];
  __shared__ unsigned long long base;
  long long first, cnt;
  lane_chunk(A, total_obj, &first, &cnt);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (long long t0 = (long long)blockIdx.x * 256; t0 < cnt; t0 += (long long)gridDim.x * 256) {
    const long long t = t0 + threadIdx.x;
    const unsigned* kb = nullptr;
    unsigned c = 0;
    if (t < cnt) {
      const long long i = A.oidx ? (long long)A.oidx[first + t] : A.obase + first + t;
      kb = keep + i * kw;
      for (int k = 0; k < kw; ++k) c += __popc(kb[k]);
    }
    unsigned x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned u = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += u;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned s = 0;
      for (int k = 0; k < 8; ++k) { const unsigned v = wsum[k]; wsum[k] = s; s += v; }
      base = atomicAdd(A.ctr + 1, (unsigned long long)s);
    }
    __syncthreads();
    if (t < cnt) {
      unsigned long long p = base + wsum[w] + x - c;
      ostart[t] = p;
      for (int k = 0; k < kw; ++k)
        for (unsigned b = kb[k]; b; b &= b - 1)
          list[p++] = make_uint2((unsigned)t, (unsigned)(32 * k + __ffs((int)b) - 1));
    }
    __syncthreads();
  }
}

// Per object: the candidates among its pairs (every lower end that reaches
// the smallest upper end), as k_merge writes them.  One warp per object.
__global__ void __launch_bounds__(128) k_lane_merge(ObjView ob, LaneArgs A, long long total_obj,
                                                    int K, int mmax, const unsigned* keep, int kw,
                                                    const unsigned long long* ostart, int* cand,
                                                    bool fp64) {
  long long first, cnt;
  lane_chunk(A, total_obj, &first, &cnt);
  const int lane = threadIdx.x & 31;
  for (long long t = (long long)blockIdx.x * 4 + (threadIdx.x >> 5); t < cnt;
       t += (long long)gridDim.x * 4) {
    const long long i = A.oidx ? (long long)A.oidx[first + t] : A.obase + first + t;
    int* out = cand + i * kMergedInts;
    const long long mm = ob.off[i + 1] - ob.off[i];
    if (mm < 1 || mm > mmax || A.obad[i]) {
      if (lane == 0) out[0] = -2;
      continue;
    }
    unsigned long long s = (unsigned long long)t * (unsigned)K;
    int c = K;
    if (A.list) {
      s = ostart[t];
      unsigned x = 0;
      for (int k = lane; k < kw; k += 32) x += __popc(keep[i * kw + k]);
      c = (int)__reduce_add_sync(0xffffffffu, x);
    }
    if (fp64) {  // exact values: the smallest, ties to the smallest centroid
      double best = NAN;
      int bj = INT_MAX;
      for (int p = lane; p < c; p += 32) {
        const double v = A.rec[s + p].d64;
        if (v < best || bj == INT_MAX || (isnan(best) && !isnan(v))) { best = v; bj = p; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
        const bool take = isnan(best) ? (!isnan(ov) || oj < bj)
                                      : (ov < best || (ov == best && oj < bj));
        if (take) { best = ov; bj = oj; }
      }
      if (lane == 0) {
        out[0] = 1;
        out[1] = bj;
        const long long bits = __double_as_longlong(best);
        out[1 + kCandCap] = (int)(unsigned)(bits & 0xffffffffLL);
        out[2 + kCandCap] = (int)(bits >> 32);
      }
      continue;
    }
    float hi = FLT_MAX;
    int at = INT_MAX;
    for (int p = lane; p < c; p += 32) {
      const float h = A.rec[s + p].hi;
      if (h < hi || at == INT_MAX) { hi = h; at = p; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, hi, o);
      const int oa = __shfl_xor_sync(0xffffffffu, at, o);
      if (oh < hi || (oh == hi && oa < at)) { hi = oh; at = oa; }
    }
    int num = 0;
    for (int p0 = 0; p0 < c; p0 += 32) {
      const int p = p0 + lane;
      const bool in = p < c && A.rec[s + p].lo <= hi;
      const unsigned b = __ballot_sync(0xffffffffu, in);
      const int pos = num + __popc(b & ((1u << lane) - 1u));
      if (in && pos < kCandCap) out[1 + pos] = A.list ? (int)A.list[s + p].y : p;
      num += __popc(b);
    }
    if (lane == 0) {
      out[0] = num > kCandCap ? -1 : num;
      const long long bits = __double_as_longlong(at == INT_MAX ? (double)NAN : A.rec[s + at].d64);
      out[1 + kCandCap] = (int)(unsigned)(bits & 0xffffffffLL);
      out[2 + kCandCap] = (int)(bits >> 32);
    }
  }
}

unsigned grid_for(long long n, int per, int most) {
  const long long b = (n + per - 1) / per;
  return (unsigned)(b < 1 ? 1 : (b < most ? b : most));
}

}  // namespace

size_t lane_scratch_offset(long long count) {
  const size_t b = (4 + (((size_t)count * kMergedInts + 3) & ~(size_t)3)) * 4;
  return (b + 255) / 256 * 256;
}

// The lanes per pair follow the launch's bounds: enough column lanes for the
// centroid's blocks of 4 supports, enough lanes that a pair's nodes are 3 to
// 8 per lane, and few enough that the pairs the shared memory holds (about
// 1.6 KB at 16 x 16, 3.4 KB at 16 x 32, 21 KB at 64 x 64) still give each
// scheduler several warps.  The narrower shapes (a6, a7, b5, b7, c6, e5, f3)
// are the wide ones of their lanes with fewer row slots, and so less shared
// memory a pair.
static cudaError_t lane_dispatch(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                                 const SolveCfg& cfg, const LaneArgs& A, long long total_obj,
                                 long long work, const ExactOut& X, cudaStream_t st) {
  auto run = [&](auto unit) { return unit(ob, cv, seg_size, K, cfg, A, total_obj, work, X, st); };
  const int m = cfg.mmax, n = cfg.nmax;
  if (m > 64 || n > 64) return cudaErrorInvalidValue;
  if (cfg.mode == 0 && !X.labels) {  // FP64 throughout: the widest shapes only
    if (n <= 16) return run(m <= 16 ? lane_all64_a8 : m <= 48 ? lane_all64_c8 : lane_all64_d5);
    if (n <= 32) return run(m <= 16 ? lane_all64_b6 : m <= 32 ? lane_all64_b8 : lane_all64_e6);
    return run(lane_all64_f4);
  }
  if (n <= 16) {
    if (m <= 16) return run(m <= 8 ? lane_run_a6 : m <= 12 ? lane_run_a7 : lane_run_a8);
    return run(m <= 32 ? lane_run_c6 : m <= 48 ? lane_run_c8 : lane_run_d5);
  }
  if (n <= 32) {
    if (m <= 16) return run(m <= 8 ? lane_run_b5 : lane_run_b6);
    if (m <= 32) return run(m <= 24 ? lane_run_b7 : lane_run_b8);
    return run(m <= 48 ? lane_run_e5 : lane_run_e6);
  }
  return run(m <= 32 ? lane_run_f3 : lane_run_f4);
}

cudaError_t lane_pairs(const ObjView& ob, const CentView& cv, const PairJob& J,
                       const SolveCfg& cfg, cudaStream_t st) {
  auto run = [&](auto unit) { return unit(ob, cv, J, cfg, st); };
  const int m = cfg.mmax, n = cfg.nmax;
  if (m > 64 || n > 64) return cudaErrorInvalidValue;
  if (n <= 16) return run(m <= 16 ? lane_pairs_a8 : m <= 48 ? lane_pairs_c8 : lane_pairs_d5);
  if (n <= 32) return run(m <= 16 ? lane_pairs_b6 : m <= 32 ? lane_pairs_b8 : lane_pairs_e6);
  return run(lane_pairs_f4);
}

// Screen of the launch's objects: merged candidate lists (k_merge's records)
// at cand + 4, and with X.labels their exact pass.
cudaError_t lane_screen(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                        const SolveCfg& cfg, int* cand, int* d_err, cudaStream_t st,
                        const TcWork* tw, const WarmStore* ws, ExactOut X) {
  const long long total_obj = cfg.dev_lo ? ob.count : (cfg.nobj >= 0 ? cfg.nobj : ob.count);
  if (total_obj <= 0) return cudaSuccess;
  const LaneScratch ls = lane_scratch(ob.count, K, cfg.mmax, cfg.nmax, cfg.max_pairs, !cfg.mass);
  int* merged = cand + 4;
  unsigned char* mem = reinterpret_cast<unsigned char*>(cand) + lane_scratch_offset(ob.count);
  LaneArgs A{};
  A.ctr = reinterpret_cast<unsigned long long*>(mem);
  A.mstride = cfg.mmax;
  long long* omass = reinterpret_cast<long long*>(mem + ls.mass);
  unsigned char* obad = mem + ls.bad;
  unsigned long long* ostart = reinterpret_cast<unsigned long long*>(mem + ls.start);
  uint2* list = reinterpret_cast<uint2*>(mem + ls.list);
  A.omass = omass;
  A.obad = obad;
  A.rec = reinterpret_cast<PairRec*>(mem + ls.rec);
  A.tree = X.labels ? mem + ls.tree : nullptr;
  A.tstride = ls.tstride;
  if (ws) {
    A.by_pair = true;
    A.tree = ws->par8;
    A.tstride = ws->ns;
    A.warm = ws->warm != 0;
    A.keep_was = cfg.keep ? cfg.keep_was : nullptr;
    A.rows = cfg.rows;
    A.axes = cfg.axes;
  }
  A.list = cfg.keep ? list : nullptr;
  A.oidx = cfg.oidx;
  A.obase = cfg.obase;
  A.lo = cfg.dev_lo;
  A.hi = cfg.dev_hi;
  A.t0 = 0;
  A.cap = total_obj;
  X.cand = merged;
  X.ostart = ostart;
  X.fb = reinterpret_cast<int*>(mem + ls.fb);
  X.err = d_err;
  cudaError_t e = cudaMemsetAsync(A.ctr, 0, cfg.first ? 32 : 16, st);
  if (e != cudaSuccess) return e;
  if (cfg.mass) {
    A.omass = cfg.mass;
    A.obad = cfg.bad;
    A.mstride = cfg.mstride;
  } else {
    e = bag_prep(ob, &cfg, cfg.mmax, omass, obad, A.mstride, nullptr, nullptr, st);
    if (e != cudaSuccess) return e;
  }
  const bool tc = tw && tw->C && cfg.mmax <= 64;
  if (tc && cfg.dev_lo) return cudaErrorInvalidValue;  // its chunks are cut on the host
  long long per = ls.objects;
  if (tc) per = std::max<long long>(1, std::min(per, tw->rows_cap / cfg.mmax));
  for (long long t0 = 0; t0 < total_obj; t0 += per) {
    const long long most = std::min(per, total_obj - t0);
    A.t0 = t0;
    A.cap = most;
    if (t0 > 0 && (e = cudaMemsetAsync(A.ctr, 0, 16, st)) != cudaSuccess) return e;
    SolveCfg sc = cfg;
    if (tc) {
      e = tc_chunk(ob, *tw, cfg.oidx ? cfg.oidx + t0 : nullptr, cfg.oidx ? 0 : cfg.obase + t0, most,
                   cfg.mmax, 0, -1, d_err, st);
      if (e != cudaSuccess) return e;
      sc.tile.C = tw->C;
      sc.tile.trow = tw->trow;
      sc.tile.nx = tw->nx;
      sc.tile.cn = tw->cents.cn;
      sc.tile.cd = tw->cents.cd;
      sc.tile.ldc = tw->cents.ncols;
      sc.tile.col0 = 0;
    }
    if (A.list) {
      k_lane_list<<<grid_for(most, 256, 8 * cfg.sms), 256, 0, st>>>(A, total_obj, cfg.keep,
                                                                    cfg.keep_words, list, ostart);
      note_launches(1);
    }
    ExactOut none;
    none.err = d_err;
    e = lane_dispatch(ob, cv, seg_size, K, sc, A, total_obj, most * (long long)K, none, st);
    if (e != cudaSuccess) return e;
    if (cfg.screen_only) continue;
    k_lane_merge<<<grid_for(most, 4, 16 * cfg.sms), 128, 0, st>>>(
        ob, A, total_obj, K, cfg.mmax, cfg.keep, cfg.keep_words, ostart, merged, cfg.mode == 0);
    note_launches(1);
    if (X.labels) {
      e = lane_dispatch(ob, cv, seg_size, K, cfg, A, total_obj, most, X, st);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaGetLastError();
}

cudaError_t lane_axes(const ObjView& ob, const SolveCfg& cfg, cudaStream_t st) {
  if (ob.count <= 0) return cudaSuccess;
  k_lane_axes<<<grid_for(ob.count, 4, 16 * cfg.sms), 128, 0, st>>>(
      ob, cfg.mmax, cfg.mass, cfg.bad, cfg.mstride, cfg.rows, cfg.axes);
  note_launches(1);
  return cudaGetLastError();
}

void lane_fallback(const ObjView& ob, int K, int* cand, SolveCfg* cfg) {
  const LaneScratch ls = lane_scratch(ob.count, K, cfg->mmax, cfg->nmax, cfg->max_pairs, !cfg->mass);
  unsigned char* mem = reinterpret_cast<unsigned char*>(cand) + lane_scratch_offset(ob.count);
  const long long* ctr = reinterpret_cast<const long long*>(mem);
  cfg->oidx = reinterpret_cast<const int*>(mem + ls.fb);
  cfg->obase = 0;
  cfg->nobj = -1;
  cfg->dev_lo = ctr + 3;
  cfg->dev_hi = ctr + 2;
}

}  // namespace d2k
