// d2_kernels.cu -- the small kernels of the assignment step for sm_103a
// (bag validation, centroid preparation, node bins, single-pair cost
// matrices, fixed-order sums) and the dispatch of the solver launches
// (per-pair Mallows distance, Eq. (D2opt) with z fixed; nearest-centroid
// assignment, Alg. 2 Step 2) to the units d2_npl1..4.cu that instantiate
// them for 1..4 tree nodes per lane.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>

#include "d2_internal.h"
#include "d2_solver.cuh"

#include "d2_solve.cuh"

namespace d2k {

__global__ void k_scan_bags(const long long* off, long long count, int* info) {
  for (long long b = blockIdx.x * (long long)blockDim.x + threadIdx.x; b < count;
       b += (long long)gridDim.x * blockDim.x) {
    const long long m = off[b + 1] - off[b];
    if (m < 1 || (b == 0 && off[0] != 0)) atomicOr(&info[1], 1);
    atomicMax(&info[0], (int)(m > INT_MAX ? INT_MAX : (m < 0 ? 0 : m)));
  }
}

__global__ void k_check_bags(const long long* off, long long count, int maxm, int* err) {
  for (long long b = blockIdx.x * (long long)blockDim.x + threadIdx.x; b < count;
       b += (long long)gridDim.x * blockDim.x) {
    const long long m = off[b + 1] - off[b];
    if (m < 1 || m > maxm || (b == 0 && off[0] != 0)) atomicOr(err, kErrInvalid);
  }
}

template <int G>
__global__ void k_prep_centroids(const void* loc, int ldt, const void* w, int wdt,
                                 const long long* off, long long K, int d, float* loc32,
                                 double* loc64, long long* Qpre, double* w64, int* err) {
  Grp<G> g;
  const int gpb = blockDim.x / G;
  for (long long j = (long long)blockIdx.x * gpb + threadIdx.x / G; j < K;
       j += (long long)gridDim.x * gpb) {
    const long long c0 = off[j];
    const long long n = off[j + 1] - c0;
    if (n < 1 || n > 64) {
      if (g.lane == 0) atomicOr(err, kErrInvalid);
      continue;
    }
    bool ok = wdt == 0 ? load_prefix<G>(g, static_cast<const double*>(w) + c0, (int)n, Qpre + c0)
                       : load_prefix<G>(g, static_cast<const float*>(w) + c0, (int)n, Qpre + c0);
    if (!ok && g.lane == 0) atomicOr(err, kErrInvalid);
    // normalised FP64 weights as seen by the solver
    for (int r = g.lane; r < n; r += G) {
      const long long prev = r > 0 ? Qpre[c0 + r - 1] : 0LL;
      w64[c0 + r] = ok ? (double)(Qpre[c0 + r] - prev) * kInvMass : 0.0;
    }
    for (long long e = g.lane; e < n * d; e += G) {
      const double v = ldx<double>(loc, ldt, c0 * d + e);
      loc64[c0 * d + e] = v;
      loc32[c0 * d + e] = (float)v;
    }
  }
}

__global__ void k_bin_of(const long long* off, long long count, int* bins) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    const long long m = off[i + 1] - off[i];
    bins[i] = (m < 1 || m > kSizeBins) ? -1 : (int)(m - 1);
  }
}

__global__ void k_cost_matrix(ObjView ob, CentView cv, long long i, long long j, int mode,
                              double* C) {
  const long long o0 = ob.off[i];
  const int m = (int)(ob.off[i + 1] - o0);
  const long long c0 = cv.off[j];
  const int n = (int)(cv.off[j + 1] - c0);
  for (int t = threadIdx.x; t < m * n; t += blockDim.x) {
    const int a = t / n, r = t % n;
    if (cv.A) {  // symbol table (ids checked before the launch; clamped reads)
      int xs = (int)ldx<double>(ob.loc, ob.ldt, o0 + a), ys = (int)cv.loc64[c0 + r];
      xs = xs < 0 ? 0 : (xs >= cv.A ? cv.A - 1 : xs);
      ys = ys < 0 ? 0 : (ys >= cv.A ? cv.A - 1 : ys);
      C[t] = mode == 0 ? cv.tab64[xs * cv.A + ys] : (double)cv.tab32[xs * cv.A + ys];
    } else if (mode == 0) {
      double acc = 0.0;
      for (int k = 0; k < cv.d; ++k) {
        const double df = ldx<double>(ob.loc, ob.ldt, (o0 + a) * cv.d + k) - cv.loc64[(c0 + r) * cv.d + k];
        acc = fma(df, df, acc);
      }
      C[t] = acc;
    } else {
      float acc = 0.f;
      for (int k = 0; k < cv.d; ++k) {
        const float df = ldx<float>(ob.loc, ob.ldt, (o0 + a) * cv.d + k) - cv.loc32[(c0 + r) * cv.d + k];
        acc = fmaf(df, df, acc);
      }
      C[t] = (double)acc;
    }
  }
}

__global__ void k_check_symbols(const void* loc, int ldt, long long T, int A, int* err) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < T;
       t += (long long)gridDim.x * blockDim.x) {
    const double v = ldx<double>(loc, ldt, t);
    if (!(v >= 0.0 && v < (double)A && v == floor(v))) atomicOr(err, kErrInvalid);
  }
}

__global__ void k_check_bag_symbols(const void* loc, int ldt, const long long* off, long long count,
                                    int A, int* err) {
  const long long T = off[count];
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < T;
       t += (long long)gridDim.x * blockDim.x) {
    const double v = ldx<double>(loc, ldt, t);
    if (!(v >= 0.0 && v < (double)A && v == floor(v))) atomicOr(err, kErrInvalid);
  }
}

// Mean and spread of one bag from its masses (inclusive int64 prefix, units
// of 2^-62) in FP64: lanes over coordinates for the mean, over supports for
// the spread.
template <typename GetX>
__device__ __forceinline__ void bag_mean_var(const Grp<32>& g, const long long* pre, int m, int d,
                                             GetX x, double* mu, double* var) {
  for (int k = g.lane; k < d; k += 32) {
    double acc = 0.0;
    for (int a = 0; a < m; ++a) {
      const double w = (double)(pre[a] - (a > 0 ? pre[a - 1] : 0LL)) * kInvMass;
      acc = fma(w, x(a, k), acc);
    }
    mu[k] = acc;
  }
  __syncwarp();
  double v = 0.0;
  for (int a = g.lane; a < m; a += 32) {
    const double w = (double)(pre[a] - (a > 0 ? pre[a - 1] : 0LL)) * kInvMass;
    double s2 = 0.0;
    for (int k = 0; k < d; ++k) {
      const double df = x(a, k) - mu[k];
      s2 = fma(df, df, s2);
    }
    v = fma(w, s2, v);
  }
  v = gsum<32>(g, v);
  if (g.lane == 0) *var = v;
}

// Masses, means and spreads of the bags, 8 lanes per object (4 objects a warp:
// the FP64 pipe charges a warp instruction the same for 6 active lanes as for
// 32, and a warp per object kept it at 6 to 16; 200,000 image bags 1.14 ms).
// The arithmetic is load_prefix's and bag_mean_var's on 32 lanes, sum by sum:
// slot l of a sum holds supports l and l + 32, and the slots are added in
// halves (16, 8 within a lane, 4, 2, 1 across lanes), so the values are the
// same to the last bit.  Masses [count][mstride] and flags (1: a bag the
// solver rejects), moments optional.
__device__ __forceinline__ double slots8(const double (&v)[4]) {
  double x = (v[0] + v[2]) + (v[1] + v[3]);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

__global__ void __launch_bounds__(128) k_bag_prep(ObjView ob, const int* oidx, const long long* lo,
                                                  const long long* hi, long long obase,
                                                  long long total, int mmax, long long* mass,
                                                  unsigned char* bad, int mstride, double* mu,
                                                  double* var) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31, l8 = lane & 7;
  const long long first = lo ? *lo : 0;
  const long long cnt = lo ? *hi - first : total;
  const int d = ob.d;
  const long long step = (long long)gridDim.x * 16;
  for (long long t0 = (long long)blockIdx.x * 16 + (threadIdx.x >> 5) * 4; t0 < cnt; t0 += step) {
    const long long t = t0 + (lane >> 3);
    const bool have = t < cnt;
    const long long i = have ? (oidx ? (long long)oidx[first + t] : obase + first + t) : 0;
    long long o0 = 0;
    int m = 0;
    if (have) {
      o0 = ob.off[i];
      const long long mm = ob.off[i + 1] - o0;
      m = mm >= 1 && mm <= mmax ? (int)mm : 0;
    }
    double w[8];
    bool wrong = m == 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int a = l8 + 8 * q;
      w[q] = 0.0;
      if (a < m) {
        w[q] = ob.wdt == 0 ? static_cast<const double*>(ob.w)[o0 + a]
                           : (double)static_cast<const float*>(ob.w)[o0 + a];
        wrong |= !(w[q] >= 0.0) || isinf(w[q]);
      }
    }
    double v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = w[q] + w[q + 4];
    const double s = slots8(v);
    wrong |= !(s > 0.0) || isinf(s);
    const unsigned wb = __ballot_sync(kAll, wrong) >> (lane & 24);
    const bool ok = have && (wb & 0xffu) == 0u;
    const double inv = 1.0 / s;
    long long qv[8], part = 0, bigv = -1;
    int bigi = INT_MAX;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int a = l8 + 8 * q;
      qv[q] = 0;
      if (ok && a < m) {
        qv[q] = __double2ll_rn(w[q] * inv * 4611686018427387904.0);
        if (qv[q] < 0) qv[q] = 0;
        part += qv[q];
        if (qv[q] > bigv) { bigv = qv[q]; bigi = a; }
      }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      part += __shfl_xor_sync(kAll, part, o);
      const long long ov = __shfl_xor_sync(kAll, bigv, o);
      const int oi = __shfl_xor_sync(kAll, bigi, o);
      if (ov > bigv || (ov == bigv && oi < bigi)) { bigv = ov; bigi = oi; }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {  // the rounding residual goes to the largest
      if (l8 + 8 * q == bigi) qv[q] += kMass - part;
      if (mass && ok && l8 + 8 * q < m) mass[i * mstride + l8 + 8 * q] = qv[q];
    }
    if (bad && have && l8 == 0) bad[i] = ok ? 0 : 1;
    if (!mu) continue;
    // mean: a lane per coordinate, supports in order; spread: a lane per
    // support, coordinates in order
    double wm[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) wm[q] = (double)qv[q] * kInvMass;
    const int top = __reduce_max_sync(kAll, ok ? (unsigned)m : 0u);
    for (int kb = 0; kb < d; kb += 8) {
      const int k = kb + l8;
      double acc = 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (8 * q < top) {
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const double wa = __shfl_sync(kAll, wm[q], (lane & 24) + u);
            const int a = 8 * q + u;
            if (ok && a < m && k < d) acc = fma(wa, ldx<double>(ob.loc, ob.ldt, (o0 + a) * d + k), acc);
          }
        }
      }
      if (ok && k < d) mu[i * d + k] = acc;
    }
    __syncwarp();
    double vs[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int a = l8 + 8 * q;
      if (ok && a < m) {
        double s2 = 0.0;
        for (int k = 0; k < d; ++k) {
          const double df = ldx<double>(ob.loc, ob.ldt, (o0 + a) * d + k) - mu[i * d + k];
          s2 = fma(df, df, s2);
        }
        vs[q & 3] = fma(wm[q], s2, vs[q & 3]);
      }
    }
    const double vv = slots8(vs);
    if (have && l8 == 0) var[i] = ok ? vv : (double)NAN;
    __syncwarp();
  }
}

// Centroid moments; muT32 [d][K]: the means rounded to FP32, coordinate by
// coordinate (k_prune_keep reads 32 centroids' worth at once), cn [K]: the
// FP32 norm of each mean, rounded up, vb [K]: the spread rounded down and up.
__global__ void k_cent_moments(CentView cv, double* mu, double* var, float* muT32, float* cn, float2* vb) {
  Grp<32> g;
  const int wb = threadIdx.x >> 5;
  for (long long j = (long long)blockIdx.x * 4 + wb; j < cv.K; j += (long long)gridDim.x * 4) {
    const long long c0 = cv.off[j];
    const int n = (int)(cv.off[j + 1] - c0);
    const int d = cv.d;
    const double* y = cv.loc64 + c0 * d;
    bag_mean_var(g, cv.Qpre + c0, n, d, [&](int r, int k) { return y[r * d + k]; }, mu + j * d,
                 var + j);
    __syncwarp();
    float s = 0.f;
    for (int k = g.lane; k < d; k += 32) {
      const float x = __double2float_rn(mu[j * d + k]);
      muT32[(long long)k * cv.K + j] = x;
      s = __fmaf_ru(x, x, s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = __fadd_ru(s, __shfl_xor_sync(0xffffffffu, s, o));
    if (g.lane == 0) {
      cn[j] = __fsqrt_ru(s);
      vb[j] = make_float2(__double2float_rd(var[j]), __double2float_ru(var[j]));
    }
    __syncwarp();
  }
}

// One warp per 4 objects of a segment: UB over the segment's K centroids, then
// the keep bits.  The FP64 rule of the bounds (in d2_internal.h) decides, but
// only where FP32 cannot: with the means rounded to FP32 (each by at most
// 2^-24 of its coordinate), s32 = sum (x32 - y32)^2 by FMA is within
//   e = (d + 4) 2^-24 s32 + 2 sqrt(s32) h + h^2,  h = 2^-23 (|x| + |y|),
// of the FP64 s; UB is the FP64 minimum over the centroids whose FP32 value
// plus spread reaches the smallest upper end, and a keep bit is the FP64
// comparison only where the two intervals meet (about one centroid an object).
// GB300 runs FP64 at 1/64 of FP32: all in FP64 this took 3.7 ms for 120,000 x
// 256 in 16 dimensions (twice the K distances of d FP64 terms per object).
template <int B>
__global__ void __launch_bounds__(128) k_prune_keep(ObjView ob, long long seg_size, int K,
                                                    long long KT, int d, const double* mu_o,
                                                    const double* var_o, const double* mu_c,
                                                    const double* var_c, const float* muT32,
                                                    const float* cn, const float2* vb,
                                                    unsigned* keep, int kw, unsigned* keep_was) {
  constexpr unsigned kAll = 0xffffffffu;
  // the objects' means in FP32 (a conversion costs an FP64 issue)
  __shared__ float xs_[4][B][256];
  const int lane = threadIdx.x & 31;
  float(*xs)[256] = xs_[threadIdx.x >> 5];
  const long long step = (long long)gridDim.x * 4 * B;
  for (long long i0 = ((long long)blockIdx.x * 4 + (threadIdx.x >> 5)) * B; i0 < ob.count;
       i0 += step) {
    long long cb[B];
    double vi[B], best[B];
    float hx[B], up[B];
    bool valid[B];
    bool same = true;
    __syncwarp();
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const long long i = min(i0 + b, ob.count - 1);
      cb[b] = seg_of(ob, i, seg_size) * (long long)K;
      vi[b] = var_o[i];
      valid[b] = !isnan(vi[b]) && cb[b] + K <= KT;
      same &= cb[b] == cb[0];
      float s = 0.f;
      for (int k = lane; k < d; k += 32) {
        const float x = valid[b] ? __double2float_rn(mu_o[i * d + k]) : 0.f;
        xs[b][k] = x;
        s = __fmaf_ru(x, x, s);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s = __fadd_ru(s, __shfl_xor_sync(kAll, s, o));
      hx[b] = __fsqrt_ru(s);
      up[b] = INFINITY;
      best[b] = INFINITY;
    }
    __syncwarp();
    auto dist32 = [&](int j, float (&s)[B]) {
#pragma unroll
      for (int b = 0; b < B; ++b) s[b] = 0.f;
      for (int k = 0; k < d; ++k) {
        float y = same ? __ldg(muT32 + k * KT + min(cb[0] + j, KT - 1)) : 0.f;
#pragma unroll
        for (int b = 0; b < B; ++b) {
          if (!same) y = __ldg(muT32 + k * KT + min(cb[b] + j, KT - 1));
          const float df = xs[b][k] - y;
          s[b] = fmaf(df, df, s[b]);
        }
      }
    };
    auto err32 = [&](int b, int j, float s) {
      const float h = __fmul_ru(__fadd_ru(hx[b], __ldg(cn + min(cb[b] + j, KT - 1))), 0x1p-23f);
      const float e = __fmaf_ru(__fmul_ru(2.f, __fsqrt_ru(s)), h, __fmul_ru(h, h));
      return __fadd_ru(__fmul_ru(__fmaf_ru((float)(d + 4) * 0x1p-24f, s, e), 1.f + 0x1p-10f),
                       FLT_MIN);  // underflow of the squares
    };
    auto lb = [&](int b, int j) {  // the FP64 value that decides
      const double* xi = mu_o + min(i0 + b, ob.count - 1) * d;
      const double* yj = mu_c + (cb[b] + j) * d;
      double s2 = 0.0;
      for (int k = 0; k < d; ++k) {
        const double df = xi[k] - yj[k];
        s2 = fma(df, df, s2);
      }
      return s2;
    };
    // smallest upper end of s + spread
    for (int j = lane; j < K; j += 32) {
      float s[B];
      dist32(j, s);
#pragma unroll
      for (int b = 0; b < B; ++b)
        if (valid[b])
          up[b] = fminf(up[b], __fadd_ru(__fadd_ru(s[b], err32(b, j, s[b])), __ldg(vb + cb[b] + j).y));
    }
#pragma unroll
    for (int b = 0; b < B; ++b)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) up[b] = fminf(up[b], __shfl_xor_sync(kAll, up[b], o));
    for (int j = lane; j < K; j += 32) {
      float s[B];
      dist32(j, s);
#pragma unroll
      for (int b = 0; b < B; ++b)
        if (valid[b]) {
          const float low = __fadd_rd(__fsub_rd(s[b], err32(b, j, s[b])), __ldg(vb + cb[b] + j).x);
          if (!(low > up[b])) best[b] = fmin(best[b], lb(b, j) + var_c[cb[b] + j]);
        }
    }
    double ub[B];
    float ubl[B], ubh[B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) best[b] = fmin(best[b], __shfl_xor_sync(kAll, best[b], o));
      ub[b] = (vi[b] + best[b]) * (1.0 + 0x1p-40);
      ubl[b] = __fmul_rd(__double2float_rd(ub[b]), 1.f - 0x1p-20f);
      ubh[b] = __fmul_ru(__double2float_ru(ub[b]), 1.f + 0x1p-20f);
    }
    for (int w = 0; w < kw; ++w) {
      const int j = w * 32 + lane;
      float s[B];
      dist32(min(j, K - 1), s);
#pragma unroll
      for (int b = 0; b < B; ++b) {
        // keep unless the lower bound is above the upper bound (NaN keeps)
        bool k = j < K;
        if (k && valid[b]) {
          const float e = err32(b, j, s[b]);
          if (__fsub_rd(s[b], e) > ubh[b]) k = false;
          else if (!(__fadd_ru(s[b], e) < ubl[b])) k = !(lb(b, j) * (1.0 - 0x1p-40) > ub[b]);
        }
        const unsigned bits = __ballot_sync(kAll, k);
        if (lane == 0 && i0 + b < ob.count) {
          unsigned* at = keep + (i0 + b) * kw + w;
          if (keep_was) keep_was[(i0 + b) * kw + w] = *at;
          *at = bits;
        }
      }
    }
  }
}

// Fixed-order sum (one block, strided partials then a tree): deterministic.
__global__ void k_sum_fixed(const double* v, long long n, double* out) {
  __shared__ double sh[256];
  double acc = 0.0;
  for (long long t = threadIdx.x; t < n; t += blockDim.x) acc += v[t];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

// ------------------------------------------------------------ launchers --

static unsigned long long g_launches = 0;
void note_launches(long long k) { __atomic_fetch_add(&g_launches, (unsigned long long)k, __ATOMIC_RELAXED); }
long long launches() { return (long long)__atomic_load_n(&g_launches, __ATOMIC_RELAXED); }

// Sum of the solver counters of the units that hold the solver kernels.
cudaError_t solver_stats(long long out[6]) {
#define X(u) stats_lane_##u,
#define XP(u) stats_lane_##u##_pairs,
  cudaError_t (*const units[])(long long*) = {stats_npl1, stats_npl2, stats_npl3, stats_npl4,
                                              D2_LANE_SHAPES(X) D2_LANE_WIDE(XP)};
#undef X
#undef XP
  for (int i = 0; i < 6; ++i) out[i] = 0;
  for (auto f : units) {
    long long v[6];
    const cudaError_t e = f(v);
    if (e != cudaSuccess) return e;
    for (int i = 0; i < 6; ++i) out[i] += v[i];
  }
  return cudaSuccess;
}

int device_sms(int dev) {
  int v = 0;
  cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
  return v > 0 ? v : 1;
}

cudaError_t scan_bags(const long long* off, long long count, int* d_info, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(d_info, 0, 2 * sizeof(int), st);
  if (e != cudaSuccess) return e;
  if (count <= 0) return cudaSuccess;
  const long long blocks = (count + 255) / 256;
  k_scan_bags<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(off, count, d_info);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t check_bags(const long long* off, long long count, int maxm, int* d_err,
                       cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  const long long blocks = (count + 255) / 256;
  k_check_bags<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(off, count, maxm, d_err);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t prep_centroids(const void* loc, int ldt, const void* w, int wdt, const long long* off,
                           long long K, int d, float* loc32, double* loc64, long long* Qpre,
                           double* w64, int* d_err, cudaStream_t st) {
  const long long blocks = (K + 3) / 4;
  k_prep_centroids<32><<<(unsigned)(blocks < 65535 ? blocks : 65535), 128, 0, st>>>(
      loc, ldt, w, wdt, off, K, d, loc32, loc64, Qpre, w64, d_err);
  note_launches(1);
  return cudaGetLastError();
}

// Tree shape for supports up to (mmax, nmax): one warp (G = 32 lanes) per
// pair, each lane owning NPL tree nodes (m+n <= 32*NPL).
#define D2_BINS(X) \
  X(32, 1)         \
  X(32, 2)         \
  X(32, 3)         \
  X(32, 4)

static bool pick_shape(int mmax, int nmax, int* G, int* npl) {
  const int N = mmax + nmax;
  if (N > 128) return false;
  *G = 32;
  *npl = (N + 31) / 32;
  return true;
}

cudaError_t mallows_pairs(const ObjView& ob, const CentView& cv, const long long* pobj,
                          const long long* pcen, long long npairs, const SolveCfg& cfg,
                          double* dist2, FlowOut fo, int* status, int* d_err, cudaStream_t st) {
  if (npairs <= 0) return cudaSuccess;
  int G, NP;
  if (!pick_shape(cfg.mmax, cfg.nmax, &G, &NP)) return cudaErrorInvalidValue;
  if (cfg.done) {  // by lanes; below, the few pairs it left
    const PairJob J{pobj, pcen, npairs, dist2, status, fo, cfg.done, d_err};
    const cudaError_t e = lane_pairs(ob, cv, J, cfg, st);
    if (e != cudaSuccess) return e;
  }
#define X(g_, n_)                                                                          \
  if (G == g_ && NP == n_)                                                                \
    return mallows_pairs_npl##n_(ob, cv, pobj, pcen, npairs, cfg, dist2, fo, status, d_err, st);
  D2_BINS(X)
#undef X
  return cudaErrorInvalidValue;
}

cudaError_t assign(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                   const SolveCfg& cfg0, const double* omega, int* labels, double* dist2,
                   double* eps_terms, FlowOut fo, int* cand, int* d_err, cudaStream_t st,
                   const WarmStore* ws, const TcWork* tw) {
  if (ob.count <= 0) return cudaSuccess;
  SolveCfg cfg = cfg0;
  if (cfg.lanes && cand && (cfg.mode == 1 ? !ws || !ws->pos8 : true)) {
    ExactOut X;
    if ((cfg.lane_exact || cfg.mode == 0) && !cfg.screen_only) {
      X.omega = omega;
      X.labels = labels;
      X.dist2 = dist2;
      X.eps_terms = eps_terms;
      X.fo = fo;
    }
    const cudaError_t e = lane_screen(ob, cv, seg_size, K, cfg, cand, d_err, st, tw, ws, X);
    if (e != cudaSuccess || cfg.screen_only) return e;
    cfg.screened = true;
    if (cfg.mode == 0) return cudaSuccess;
    if (X.labels) {  // the few objects k_exact still solves
      if (!cfg.last) return cudaSuccess;
      if (cfg.mall > cfg.mmax) cfg.mmax = cfg.mall;
      lane_fallback(ob, K, cand, &cfg);
    }
  }
  int G, NP;
  if (!pick_shape(cfg.mmax, cfg.nmax, &G, &NP)) return cudaErrorInvalidValue;
#define X(g_, n_)                                                                            \
  if (G == g_ && NP == n_)                                                                  \
    return assign_npl##n_(ob, cv, seg_size, K, cfg, omega, labels, dist2, eps_terms, fo, cand, d_err, st, ws, tw);
  D2_BINS(X)
#undef X
  return cudaErrorInvalidValue;
}

cudaError_t bin_objects(const ObjView& ob, int* bins_out, cudaStream_t st) {
  if (ob.count <= 0) return cudaSuccess;
  const unsigned b = (unsigned)std::min<long long>((ob.count + 255) / 256, 4096);
  k_bin_of<<<b, 256, 0, st>>>(ob.off, ob.count, bins_out);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t cost_matrix(const ObjView& ob, const CentView& cv, long long i, long long j, int mode,
                        double* C, cudaStream_t st) {
  k_cost_matrix<<<1, 256, 0, st>>>(ob, cv, i, j, mode, C);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t check_symbols(const void* loc, int ldt, long long T, int A, int* d_err,
                          cudaStream_t st) {
  if (T <= 0) return cudaSuccess;
  const unsigned b = (unsigned)std::min<long long>((T + 255) / 256, 4096);
  k_check_symbols<<<b, 256, 0, st>>>(loc, ldt, T, A, d_err);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t check_bag_symbols(const void* loc, int ldt, const long long* off, long long count,
                              int A, int* d_err, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  k_check_bag_symbols<<<(unsigned)(152 * 4), 256, 0, st>>>(loc, ldt, off, count, A, d_err);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t bag_prep(const ObjView& ob, const SolveCfg* range, int mmax, long long* mass,
                     unsigned char* bad, int mstride, double* mu, double* var, cudaStream_t st) {
  long long total = ob.count;
  const int* oidx = nullptr;
  const long long *lo = nullptr, *hi = nullptr;
  long long obase = 0;
  if (range) {
    oidx = range->oidx;
    lo = range->dev_lo;
    hi = range->dev_hi;
    obase = range->obase;
    if (!lo && range->nobj >= 0) total = range->nobj;
  }
  if (total <= 0) return cudaSuccess;
  const long long blocks = (total + 15) / 16;
  k_bag_prep<<<(unsigned)(blocks < 4096 ? blocks : 4096), 128, 0, st>>>(
      ob, oidx, lo, hi, obase, total, mmax, mass, bad, mstride, mu, var);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t cent_moments(const CentView& cv, const CentMoments& cm, cudaStream_t st) {
  if (cv.K <= 0) return cudaSuccess;
  const long long blocks = (cv.K + 3) / 4;
  k_cent_moments<<<(unsigned)(blocks < 8192 ? blocks : 8192), 128, 0, st>>>(cv, cm.mu, cm.var,
                                                                            cm.muT32, cm.cn, cm.vb);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t prune_keep(const ObjView& ob, long long seg_size, int K, long long KT, int d,
                       const double* mu_o, const double* var_o, const CentMoments& cm,
                       unsigned* keep, int kw, unsigned* keep_was, cudaStream_t st) {
  if (ob.count <= 0) return cudaSuccess;
  if (kw < (K + 31) / 32) return cudaErrorInvalidValue;
  // 4 objects a warp share the centroid loads once that still fills the GPU
  auto go = [&](auto kern, int b) {
    const long long blocks = (ob.count + 4 * b - 1) / (4 * b);
    kern<<<(unsigned)(blocks < 8192 ? blocks : 8192), 128, 0, st>>>(
        ob, seg_size, K, KT, d, mu_o, var_o, cm.mu, cm.var, cm.muT32, cm.cn, cm.vb, keep, kw,
        keep_was);
  };
  if (ob.count >= 16384) go(k_prune_keep<4>, 4);
  else go(k_prune_keep<1>, 1);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t sum_fixed_order(const double* v, long long n, double* out, cudaStream_t st) {
  k_sum_fixed<<<1, 256, 0, st>>>(v, n, out);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace d2k
