// d2_lane.cuh -- the FP32 screen with several pairs per warp.
//
// A transportation LP of the sizes the framework meets (a few to 64 supports
// a side) gives one warp too little parallel work: with a warp per pair most
// of a pivot's warp instructions (reductions, path searches, preorder
// bookkeeping) serve one pair, and a cold 16 x 16 pair took about 11,000 of
// them.  Here a pair is solved by G lanes, 32/G pairs share a warp in lock
// step, and the basis tree is kept in a form whose pivot touches only the
// cycle:
//   par[y]  parent, flow[y] int64 flow of the edge (y, par[y]), pot[y],
//   D[y]    the set of nodes in the subtree of y, as a bit mask (32*MW bits).
// The entering cell's cycle is the two walks up from its ends to the first
// node whose mask holds the other end; the leaving node's mask is the cut-off
// side S, whose potentials shift; and only the cycle's masks change: a node
// of the re-hung path gets S less its old path child's set, the nodes above
// it lose S, those of the other side gain it.  One lane walks each side.
// The walks' loops are a few dozen instructions; the first form of this
// kernel, which tested every node's mask against both ends in unrolled
// per-lane loops, ran 13,000 instructions of code and stalled on instruction
// fetch 4.2 of 9.5 cycles per issue (7,500 cycles per pivot with 12 warps on
// an SM).
//
// Shared memory of a warp is laid out in 16-byte units, unit u of its pair p
// at (u * PW + p) * 16 with PW = 32/G pairs, and lane g of pair p is warp lane
// g * PW + p: the lanes of a quarter warp that touch a unit each (128-bit
// accesses) then cover 128 consecutive bytes, as do a half warp's 64-bit and
// a warp's 32-bit ones, and two pairs on different units never meet in a
// bank.  (With the pairs' lanes side by side instead, half of all shared
// wavefronts were bank conflicts.)  Nodes: row a is node a, column r is node
// MP + r; both bounds and with them every own-node address are compile-time
// constants.  Unused rows and columns hold +inf costs and empty masks.
//
// The pivot rule is the one of Simplex (d2_solver.cuh): the most negative
// reduced cost enters (ties to the smallest cell), the smallest flow leaves
// (ties to the smallest cell), Bland's rule after 2N degenerate pivots,
// potentials shifted incrementally and refreshed every 64 pivots.
#pragma once
#include "d2_solve.cuh"

namespace d2k {
namespace {

// G lanes per pair, L of them across the blocks of 4 columns (the other
// factor G / L splits the rows), MW 32-bit words per node mask, NPL node
// slots per lane: 4 L columns and G NPL - 4 L rows.
template <int G_, int L_, int MW_, int NPL_, typename T_ = float>
struct LaneShape {
  using T = T_;  // costs and potentials: FP32 screens, or FP64 throughout
  static constexpr int G = G_, L = L_, MW = MW_, NPL = NPL_;
  static constexpr int TS = (int)sizeof(T);
  static constexpr int PW = 32 / G;           // pairs per warp
  static constexpr int RS = G / L;            // row groups
  static constexpr int PS = PW * 16;          // bytes between a pair's units
  static constexpr int NS = G * NPL;          // node slots
  static constexpr int MP = NS - 4 * L;       // row slots; columns are nodes MP ..
  static constexpr int KR = MP / G;           // own slots that are rows
  // blocks of two warps per SM the registers leave room for
  static constexpr int kMinBlocks = G == 32 ? 5 : (G == 16 ? 8 : 10);
  static_assert(MP > 0 && MP % G == 0 && NS <= 32 * MW, "lane shape");
  // A node's record: its flow and mask in a 16-byte unit, with the parent in
  // the fourth word where the mask is one word (one 128-bit access per step
  // of a walk); masks of 4 words have a unit of their own.
  static constexpr int kPot = 0;
  static constexpr int kNode = kPot + NPL * 32 * TS;
  static constexpr int kD4 = kNode + NPL * 512;               // MW = 4
  static constexpr int kPar = kD4 + (MW == 4 ? NPL * 512 : 0);  // MW > 1
  static constexpr int kCode = kPar + (MW > 1 ? (NS + 15) / 16 * PS : 0);
  static constexpr int kTile = kCode + (NS + 15) / 16 * PS;
};

// Bytes of a warp with room for mmax rows of nb column blocks.
template <class Sh>
inline size_t lane_warp_bytes(int mmax, int nb) {
  return (size_t)Sh::kTile + (size_t)((mmax + 3) & ~3) * nb * Sh::PS * (Sh::TS / 4);
}

template <int MW>
struct Mask {
  unsigned w[MW];
  __device__ __forceinline__ bool meets(const Mask& o) const {
    unsigned x = w[0] & o.w[0];
#pragma unroll
    for (int i = 1; i < MW; ++i) x |= w[i] & o.w[i];
    return x != 0u;
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < MW; ++i) w[i] = 0u;
  }
  __device__ __forceinline__ void set(int e) {
#pragma unroll
    for (int i = 0; i < MW; ++i)
      if ((e >> 5) == i) w[i] |= 1u << (e & 31);
  }
  __device__ __forceinline__ void drop(int e) {
#pragma unroll
    for (int i = 0; i < MW; ++i)
      if ((e >> 5) == i) w[i] &= ~(1u << (e & 31));
  }
  __device__ __forceinline__ Mask minus(const Mask& o) const {
    Mask r;
#pragma unroll
    for (int i = 0; i < MW; ++i) r.w[i] = w[i] & ~o.w[i];
    return r;
  }
  __device__ __forceinline__ Mask plus(const Mask& o) const {
    Mask r;
#pragma unroll
    for (int i = 0; i < MW; ++i) r.w[i] = w[i] | o.w[i];
    return r;
  }
};

// One pair's view of its warp's shared memory and its solver state; every
// lane of the warp runs the same code (a pair without work has live = false
// and only joins the shuffles).
template <typename T>
struct V4 {
  T x, y, z, w;
};

template <class Sh>
struct Lane {
  using T = typename Sh::T;
  static constexpr int G = Sh::G, L = Sh::L, MW = Sh::MW, NPL = Sh::NPL, RS = Sh::RS;
  static constexpr int PW = Sh::PW, PS = Sh::PS, MP = Sh::MP, NS = Sh::NS, KR = Sh::KR;
  static constexpr unsigned kAll = 0xffffffffu;
  char* sp;         // the pair's first unit
  int nb;           // column blocks of the tile
  int g, gl, rg;    // lane in the pair, its column lane, its row group
  int m, n, N, root;
  bool live;
  int cand;         // kList: the lane's best cell of the last full scan (INT_MAX: none)
  // FP64 pricing by candidates: the scan of a tile costs the FP64 pipe (a 64th
  // of the FP32 rate) 12 operations per 4 cells, so a pivot first takes the
  // best of the lanes' cells of the last scan at the current potentials, and
  // the tile is scanned when a pair of the warp has none left.
  // (64,000 pairs in FP64: 64 x 64 182 -> 80 ms, 32 x 32 35 -> 27)
  static constexpr bool kList = Sh::TS == 8 && Sh::G >= 8;

  __device__ __forceinline__ Lane(char* warp_base, int nb_) : nb(nb_) {
    const int lane = threadIdx.x & 31;
    g = lane / PW;
    gl = g & (L - 1);
    rg = g / L;
    sp = warp_base + (lane & (PW - 1)) * 16;
    m = n = 1;
    N = 2;
    root = 0;
    live = false;
  }

  // ---- shared memory: any node, and the own node of slot k (y = g + G k) ----
  // a block of 4 columns of row a (one unit of floats, two of doubles)
  __device__ __forceinline__ char* tp(int a, int cb) const {
    return sp + Sh::kTile + (a * nb + cb) * (PS * (Sh::TS / 4));
  }
  __device__ __forceinline__ float4& tile4(int a, int cb) const {
    return *reinterpret_cast<float4*>(tp(a, cb));
  }
  __device__ __forceinline__ static V4<T> ld4(const char* p) {
    if constexpr (Sh::TS == 4) {
      const float4 v = *reinterpret_cast<const float4*>(p);
      return V4<T>{v.x, v.y, v.z, v.w};
    } else {
      const double2 a = *reinterpret_cast<const double2*>(p);
      const double2 b = *reinterpret_cast<const double2*>(p + PS);
      return V4<T>{a.x, a.y, b.x, b.y};
    }
  }
  __device__ __forceinline__ static void st4(char* p, const V4<T>& v) {
    if constexpr (Sh::TS == 4) {
      *reinterpret_cast<float4*>(p) = make_float4(v.x, v.y, v.z, v.w);
    } else {
      *reinterpret_cast<double2*>(p) = make_double2(v.x, v.y);
      *reinterpret_cast<double2*>(p + PS) = make_double2(v.z, v.w);
    }
  }
  __device__ __forceinline__ T& cell(int a, int r) const {
    constexpr int per = 16 / Sh::TS;  // values a unit
    return *reinterpret_cast<T*>(tp(a, r >> 2) + ((r & 3) / per) * PS + (r % per) * Sh::TS);
  }
  __device__ __forceinline__ float4& pot4(int q) const {
    return *reinterpret_cast<float4*>(sp + Sh::kPot + q * PS);
  }
  // potentials of nodes 4 q .. 4 q + 3
  __device__ __forceinline__ V4<T> potq(int q) const {
    return ld4(sp + Sh::kPot + q * (PS * (Sh::TS / 4)));
  }
  __device__ __forceinline__ T& pot(int y) const {
    constexpr int per = 16 / Sh::TS;
    return *reinterpret_cast<T*>(sp + Sh::kPot + (y / per) * PS + (y % per) * Sh::TS);
  }
  __device__ __forceinline__ T& potk(int k) const {
    constexpr int per = 16 / Sh::TS;
    return *reinterpret_cast<T*>(sp + Sh::kPot + (g / per) * PS + (g % per) * Sh::TS +
                                 k * (32 * Sh::TS));
  }
  __device__ __forceinline__ char* rec(int y) const { return sp + Sh::kNode + y * PS; }
  __device__ __forceinline__ long long& flow(int y) const {
    return *reinterpret_cast<long long*>(rec(y));
  }
  __device__ __forceinline__ long long& flowk(int k) const { return flow(g + G * k); }
  // a second float per node, in the mask's place (once the masks are done with)
  __device__ __forceinline__ float& aux(int y) const {
    return *reinterpret_cast<float*>(rec(y) + 8);
  }
  template <int SEC>
  __device__ __forceinline__ unsigned char& u8at(int y) const {
    return *reinterpret_cast<unsigned char*>(sp + SEC + (y >> 4) * PS + (y & 15));
  }
  template <int SEC>
  __device__ __forceinline__ unsigned char& u8own(int k) const {
    // y >> 4 and y & 15 of y = g + G k, split into a lane part and a slot part
    if constexpr (G >= 16)
      return *reinterpret_cast<unsigned char*>(sp + SEC + (g >> 4) * PS + (g & 15) +
                                               k * (G / 16) * PS);
    else
      return *reinterpret_cast<unsigned char*>(sp + SEC + g + ((G * k) >> 4) * PS + ((G * k) & 15));
  }
  __device__ __forceinline__ unsigned par(int y) const {
    if constexpr (MW == 1) return *reinterpret_cast<unsigned*>(rec(y) + 12);
    else return u8at<Sh::kPar>(y);
  }
  __device__ __forceinline__ void put_par(int y, unsigned v) const {
    if constexpr (MW == 1) *reinterpret_cast<unsigned*>(rec(y) + 12) = v;
    else u8at<Sh::kPar>(y) = (unsigned char)v;
  }
  __device__ __forceinline__ Mask<MW> getD(int y) const {
    Mask<MW> d;
    if constexpr (MW == 1) {
      d.w[0] = *reinterpret_cast<const unsigned*>(rec(y) + 8);
    } else if constexpr (MW == 2) {
      const uint2 v = *reinterpret_cast<const uint2*>(rec(y) + 8);
      d.w[0] = v.x; d.w[1] = v.y;
    } else {
      const uint4 v = *reinterpret_cast<const uint4*>(sp + Sh::kD4 + y * PS);
      d.w[0] = v.x; d.w[1] = v.y; d.w[2] = v.z; d.w[3] = v.w;
    }
    return d;
  }
  __device__ __forceinline__ void putD(int y, const Mask<MW>& d) const {
    if constexpr (MW == 1) *reinterpret_cast<unsigned*>(rec(y) + 8) = d.w[0];
    else if constexpr (MW == 2) *reinterpret_cast<uint2*>(rec(y) + 8) = make_uint2(d.w[0], d.w[1]);
    else *reinterpret_cast<uint4*>(sp + Sh::kD4 + y * PS) =
        make_uint4(d.w[0], d.w[1], d.w[2], d.w[3]);
  }
  // the whole record
  __device__ __forceinline__ void load(int y, long long& f, Mask<MW>& d, unsigned& p) const {
    const uint4 v = *reinterpret_cast<const uint4*>(rec(y));
    f = (long long)(((unsigned long long)v.y << 32) | v.x);
    if constexpr (MW == 1) {
      d.w[0] = v.z;
      p = v.w;
    } else if constexpr (MW == 2) {
      d.w[0] = v.z; d.w[1] = v.w;
      p = u8at<Sh::kPar>(y);
    } else {
      d = getD(y);
      p = u8at<Sh::kPar>(y);
    }
  }
  __device__ __forceinline__ void store(int y, long long f, const Mask<MW>& d, unsigned p) const {
    const unsigned lo = (unsigned)(unsigned long long)f, hi = (unsigned)((unsigned long long)f >> 32);
    if constexpr (MW == 1) {
      *reinterpret_cast<uint4*>(rec(y)) = make_uint4(lo, hi, d.w[0], p);
    } else {
      if constexpr (MW == 2) {
        *reinterpret_cast<uint4*>(rec(y)) = make_uint4(lo, hi, d.w[0], d.w[1]);
      } else {
        *reinterpret_cast<uint2*>(rec(y)) = make_uint2(lo, hi);
        *reinterpret_cast<uint4*>(sp + Sh::kD4 + y * PS) =
            make_uint4(d.w[0], d.w[1], d.w[2], d.w[3]);
      }
      u8at<Sh::kPar>(y) = (unsigned char)p;
    }
  }
  __device__ __forceinline__ int node(int k) const { return g + G * k; }
  // own slot k holds a node of the pair (rows first: a compile-time split)
  __device__ __forceinline__ bool nodek(int k) const {
    return k < KR ? g + G * k < m : g + G * k - MP < n;
  }
  __device__ __forceinline__ static bool is_row(int y) { return y < MP; }
  __device__ __forceinline__ bool has_node(int y) const { return y < MP ? y < m : y - MP < n; }
  // tile cell of the edge (y, p)
  __device__ __forceinline__ float edge_cost(int y, int p) const {
    return is_row(y) ? cell(y, p - MP) : cell(p, y - MP);
  }
  // own slot k's node in a set whose words were shifted right by g
  // (G k + g: word (G k) >> 5 since G divides 32)
  __device__ __forceinline__ static bool ink(const Mask<MW>& shifted, int k) {
    return (shifted.w[(G * k) >> 5] >> ((G * k) & 31)) & 1u;
  }

  // ---- reductions over the pair's lanes (warp lanes g * PW + p) ----
  template <typename V>
  __device__ __forceinline__ static V sum(V v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kAll, v, o * PW);
    return v;
  }
  __device__ __forceinline__ static float maxf(float v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kAll, v, o * PW));
    return v;
  }
  __device__ __forceinline__ static unsigned maxu(unsigned v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kAll, v, o * PW));
    return v;
  }
  __device__ __forceinline__ static unsigned oru(unsigned v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v |= __shfl_xor_sync(kAll, v, o * PW);
    return v;
  }
  // smallest (value, key) over W neighbouring lanes of the pair
  template <int W, typename V>
  __device__ __forceinline__ static void min_key(V& v, int& key) {
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) {
      const V ov = __shfl_xor_sync(kAll, v, o * PW);
      const int ok = __shfl_xor_sync(kAll, key, o * PW);
      if (ov < v || (ov == v && ok < key)) { v = ov; key = ok; }
    }
  }

  // Sum over the pair's nodes of the double in each node's flow slot, in an
  // order that does not depend on the shape: slot y mod 32 (compact node
  // index, rows then columns) over its nodes in order, then halves of the
  // slots.
  __device__ __forceinline__ double sum_nodes() {
    __syncwarp();
    double v[32 / G];
#pragma unroll
    for (int s = 0; s < 32 / G; ++s) {
      v[s] = 0.0;
#pragma unroll
      for (int k = 0; k < MW; ++k) {
        const int c = g + G * s + 32 * k;
        if (live && c < N) {
          const double x = *reinterpret_cast<double*>(&flow(c < m ? c : c - m + MP));
          v[s] = k == 0 ? x : v[s] + x;
        }
      }
    }
#pragma unroll
    for (int h = 16 / G; h > 0; h >>= 1)
#pragma unroll
      for (int s = 0; s < h; ++s) v[s] += v[s + h];
    __syncwarp();
    return sum(v[0]);
  }

  // ---- start: rows in turn on centred costs ----
  // Every remaining row in cyclic order sends as much mass as both ends hold
  // to its cheapest remaining column, the cost of a column taken against its
  // mean over the object (vm: sum_a p_a c_ar, the lane's 4 columns): two bags
  // far apart cost nearly f(a) + g(r), and what tells the columns apart is
  // the rest.  The end that runs out (the row on a tie) leaves and hangs from
  // the other; the last line of either kind is the root and takes the rest.
  // Flows are the int64 masses, so the basis is exactly feasible.  Pivots a
  // pair from there, and a warp per pair's from the ranked staircase and from
  // Vogel's rule (all pairs of some thousand bags of each workload law, by the
  // library's counters with start_rule 0, 1 and 2): image 8.8 (22.3), uneven
  // 5.6 (19.8, 12.7), serving 35.7 (126, 69.6), high_dim 56.2 (247, 67.2),
  // sequences 15.4 (52.9, 14.1).  A step reads one row of the tile, where
  // Vogel's rule keeps the two best of every line.  flow holds the masses, D
  // the singletons.
  __device__ __forceinline__ void start_rows(const V4<T>& vm) {
    unsigned long long ra = m >= 64 ? ~0ull : ((1ull << m) - 1ull);
    unsigned long long ca = n >= 64 ? ~0ull : ((1ull << n) - 1ull);
    int nr = m, nc = n, cur = -1;
    for (;;) {
      const bool act = live && nr > 1 && nc > 1;
      if (!__any_sync(kAll, act)) break;
      T best = T(INFINITY);
      int key = INT_MAX;
      int a = 0;
      if (act) {
        const unsigned long long later = ra & ~((2ull << (cur & 63)) - 1ull);
        a = __ffsll((long long)((cur >= 0 && later) ? later : ra)) - 1;
        if (gl < nb) {
          const V4<T> c = ld4(tp(a, gl));
          const unsigned al = (unsigned)(ca >> (4 * gl)) & 15u;
          const T d[4] = {c.x - vm.x, c.y - vm.y, c.z - vm.z, c.w - vm.w};
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (((al >> i) & 1u) && d[i] < best) { best = d[i]; key = 4 * gl + i; }
        }
      }
      min_key<L>(best, key);
      long long ma = 0, mr = 0;
      int r = 0;
      if (act) {
        r = key == INT_MAX ? __ffsll((long long)ca) - 1 : key;
        ma = flow(a);
        mr = flow(MP + r);
      }
      __syncwarp();
      if (act) {
        const bool row_leaves = ma <= mr;
        if (g == 0) {
          const int y = row_leaves ? a : MP + r, z = row_leaves ? MP + r : a;
          put_par(y, (unsigned)z);
          store(z, row_leaves ? mr - ma : ma - mr, getD(z).plus(getD(y)), 0xffu);
        }
        if (row_leaves) { ra &= ~(1ull << a); --nr; }
        else { ca &= ~(1ull << r); --nc; }
        cur = a;
      }
      __syncwarp();
    }
    // the last line takes the rest
    const bool row_root = nr == 1;
    if (live)
      root = row_root ? __ffsll((long long)ra) - 1 : MP + __ffsll((long long)ca) - 1;
    Mask<MW> d;
    d.clear();
#pragma unroll 1
    for (int k = 0; k < NPL; ++k) {
      const int y = node(k);
      if (live && nodek(k)) {
        const bool row = k < KR;
        const bool left = row ? (ra >> y) & 1ull : (ca >> (y - MP)) & 1ull;
        if (left && row != row_root) {
          put_par(y, (unsigned)root);
          d = d.plus(getD(y));
        }
      }
    }
#pragma unroll
    for (int i = 0; i < MW; ++i) d.w[i] = oru(d.w[i]);
    if (live && g == 0) store(root, 0, getD(root).plus(d), 0xffu);
    __syncwarp();
  }

  // The object's masses into its rows' flow slots, as load_prefix makes them
  // (the same sums in the same order: slot l holds supports l and l + 32, the
  // slots are added in halves).  Returns false for a bag the solver rejects.
  template <typename W>
  __device__ __forceinline__ bool row_masses(bool act, const W* w, bool put = true) {
    constexpr int SL = 32 / G;  // own slots of the sum
    double x[KR];
    bool wrong = false;
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      x[k] = 0.0;
      if (act && node(k) < m) {
        x[k] = (double)w[node(k)];
        wrong |= !(x[k] >= 0.0) || isinf(x[k]);
      }
    }
    double v[SL];
#pragma unroll
    for (int s = 0; s < SL; ++s) {
      v[s] = s < KR ? x[s] : 0.0;
      if (s + SL < KR) v[s] += x[s + SL];
    }
#pragma unroll
    for (int h = SL / 2; h > 0; h >>= 1)
#pragma unroll
      for (int s = 0; s < h; ++s) v[s] += v[s + h];
    const double s = sum(v[0]);
    wrong |= act && (!(s > 0.0) || isinf(s));
    if (oru(wrong ? 1u : 0u)) act = false;
    const double inv = 1.0 / s;
    long long q[KR], part = 0, bigv = -1;
    int bigi = INT_MAX;
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      q[k] = 0;
      if (act && node(k) < m) {
        q[k] = __double2ll_rn(x[k] * inv * 4611686018427387904.0);
        if (q[k] < 0) q[k] = 0;
        part += q[k];
        if (q[k] > bigv) { bigv = q[k]; bigi = node(k); }
      }
    }
    part = sum(part);
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      const long long ov = __shfl_xor_sync(kAll, bigv, o * PW);
      const int oi = __shfl_xor_sync(kAll, bigi, o * PW);
      if (ov > bigv || (ov == bigv && oi < bigi)) { bigv = ov; bigi = oi; }
    }
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      if (act && node(k) == bigi) q[k] += kMass - part;
      if (put) flowk(k) = q[k];
    }
    return act;
  }

  // Flows (and with MASKS the subtree sets) of the tree in par: the edge above
  // a node carries the net mass of its subtree, rows positive and columns
  // negative, summed by walking every node's mass up to the root.  On entry
  // flow holds the masses and D the singletons; exact integers, so the flows
  // are those the tree was saved with.  Returns whether the tree is
  // inconsistent or a flow negative.
  template <bool MASKS>
  __device__ __forceinline__ bool from_parents() {
    bool bad = false;
    long long b[NPL];
#pragma unroll
    for (int k = 0; k < NPL; ++k) b[k] = k < KR ? flowk(k) : -flowk(k);
    __syncwarp();
#pragma unroll
    for (int k = 0; k < NPL; ++k)
      if (live) flowk(k) = 0;
    __syncwarp();
    // the own nodes walk together, a step of all of them at a time
    int x[NPL];
    unsigned going = 0u;
#pragma unroll
    for (int k = 0; k < NPL; ++k) {
      x[k] = node(k);
      if (live && nodek(k)) going |= 1u << k;
    }
#pragma unroll 1
    for (int it = 0; it < NS && going; ++it) {
#pragma unroll
      for (int k = 0; k < NPL; ++k) {
        if ((going >> k) & 1u) {
          if (x[k] == root) {
            if (MASKS && it > 0) or_mask(root, node(k));
            going &= ~(1u << k);
          } else {
            atomicAdd(reinterpret_cast<unsigned long long*>(&flow(x[k])), (unsigned long long)b[k]);
            if (MASKS && it > 0) or_mask(x[k], node(k));
            const unsigned p = par(x[k]);
            if (p >= (unsigned)NS || is_row(x[k]) == is_row((int)p)) {
              bad = true;
              going &= ~(1u << k);
            } else {
              x[k] = (int)p;
            }
          }
        }
      }
    }
    bad |= going != 0u;  // no way to the root
    __syncwarp();
#pragma unroll
    for (int k = 0; k < NPL; ++k) {
      if (live) {
        if (k >= KR) flowk(k) = -flowk(k);
        bad |= nodek(k) && flowk(k) < 0;
      }
    }
    return oru(bad ? 1u : 0u) != 0u;
  }
  __device__ __forceinline__ void or_mask(int x, int y) const {
    char* at = MW == 4 ? sp + Sh::kD4 + x * PS : rec(x) + 8;
    atomicOr(reinterpret_cast<unsigned*>(at) + (y >> 5), 1u << (y & 31));
  }

  // ---- start: northwest staircase ----
  // Rows and columns in the orders of the code section (row of rank q at q,
  // column of rank q at MP + q): down when the row is used up first (ties
  // down), the new line hangs from the other kind's current one.  A node
  // carries everything after it once a node hangs from it, else itself.
  // flow holds the masses, D the singletons.
  __device__ __forceinline__ void start_staircase() {
    int iq = 0, jq = 0;
    int a = u8at<Sh::kCode>(0), r = MP + u8at<Sh::kCode>(MP);
    Mask<MW> rest;  // nodes not touched before `last`
#pragma unroll
    for (int w = 0; w < MW; ++w) rest.w[w] = 0u;
    if (live) {
#pragma unroll 1
      for (int y = 0; y < m; ++y) rest.set(y);
#pragma unroll 1
      for (int y = 0; y < n; ++y) rest.set(MP + y);
    }
    long long p = 0, q = 0;
    if (live) {
      p = flow(a);
      q = flow(r);
      root = a;
    }
    __syncwarp();
    // the root, then column r hanging from it
    const Mask<MW> all = rest;
    int last = r;
    if (live) {
      rest.drop(a);
      const long long f = p < q ? p : q;
      if (g == 0) {
        store(a, 0, all, 0xffu);
        Mask<MW> one;
        one.clear();
        one.set(r);
        store(r, f, one, (unsigned)a);
      }
      p -= f;
      q -= f;
    }
#pragma unroll 1
    for (int s = 2;; ++s) {
      const bool act = live && s < N;
      if (!__any_sync(kAll, act)) break;
      int y = 0, z = 0;
      long long f = 0;
      if (act) {
        const bool down = iq < m - 1 && (p <= q || jq == n - 1);
        z = down ? r : a;  // the new node hangs from z
        y = down ? (int)u8at<Sh::kCode>(++iq) : MP + (int)u8at<Sh::kCode>(MP + ++jq);
        const long long w = flow(y);
        if (down) {
          f = w < q ? w : q;
          p = w - f;
          q -= f;
          a = y;
        } else {
          f = p < w ? p : w;
          q = w - f;
          p -= f;
          r = y;
        }
      }
      __syncwarp();
      if (act) {
        if (g == 0) {
          if (z == last) putD(last, rest);  // `last` and what follows it
          Mask<MW> one;
          one.clear();
          one.set(y);
          store(y, f, one, (unsigned)z);
        }
        rest.drop(last);
        last = y;
      }
    }
    __syncwarp();
  }

  // Accumulate the own nodes' edge terms acc over the path to the root by
  // pointer jumping with alternating signs, acc(y) = acc(y) -+ acc(ancestor);
  // at(y) is where node y's value lives meanwhile (and at the end).  Returns
  // whether the tree is inconsistent.
  template <typename T, typename At>
  __device__ __forceinline__ bool jump(T (&acc)[NPL], At at) {
    bool bad = false;
    unsigned cd[NPL];  // ancestor | 128 * parity
#pragma unroll
    for (int k = 0; k < NPL; ++k) {
      cd[k] = (unsigned)root;
      if (live && nodek(k) && node(k) != root) {
        const unsigned p = par(node(k));
        if (p >= (unsigned)NS || (k < KR) == is_row((int)p)) bad = true;
        else cd[k] = p | 128u;
      }
    }
#pragma unroll 1
    for (int round = 0; round < 9; ++round) {  // depth < 128: at most 8
      __syncwarp();
#pragma unroll
      for (int k = 0; k < NPL; ++k) {
        if (live) {
          u8own<Sh::kCode>(k) = (unsigned char)cd[k];
          at(node(k)) = acc[k];
        }
      }
      __syncwarp();
      bool moved = false;
#pragma unroll
      for (int k = 0; k < NPL; ++k) {
        const int an = (int)(cd[k] & 127u);
        const unsigned c2 = u8at<Sh::kCode>(an);
        const T v = at(an);
        const bool mv = live && an != root;
        const T nx = (cd[k] & 128u) ? acc[k] - v : acc[k] + v;
        acc[k] = mv ? nx : acc[k];
        cd[k] = mv ? ((c2 & 127u) | ((cd[k] ^ c2) & 128u)) : cd[k];
        moved |= mv;
      }
      if (!__any_sync(kAll, moved)) break;
    }
    __syncwarp();
    return bad;
  }

  // Potentials from the tree: pot(root) = 0, pot(y) = c(y, par y) - pot(par y).
  __device__ __forceinline__ bool refresh() {
    T acc[NPL];
#pragma unroll
    for (int k = 0; k < NPL; ++k) {
      acc[k] = T(0);
      if (live && nodek(k) && node(k) != root) {
        const int p = (int)par(node(k));
        if (p < NS && (k < KR) != is_row(p))
          acc[k] = k < KR ? cell(node(k), p - MP) : cell(p, node(k) - MP);
      }
    }
    return jump(acc, [&](int y) -> T& { return pot(y); });
  }

  // Most negative reduced cost of the tile (ties to the smallest cell
  // key (a << 8) | r); key INT_MAX if none is negative.
  __device__ __forceinline__ void price(bool act, T& best, int& key) {
    best = T(0);
    key = INT_MAX;
    if (act && gl < nb) {
      int brow = -1;
      const V4<T> v = potq((MP >> 2) + gl);
      const char* at = tp(4 * rg, gl);
      const int step = nb * (PS * (Sh::TS / 4));
#pragma unroll 1
      for (int a = 4 * rg; a < m; a += 4 * RS) {
        const V4<T> u = potq(a >> 2);
        const T uu[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const V4<T> c = ld4(at + i * step);
          T lo;
          if constexpr (Sh::TS == 4) {  // two columns an instruction
            const float2 nu = make_float2(-uu[i], -uu[i]);
            const float2 d0 = __fadd2_rn(__fadd2_rn(make_float2(c.x, c.y), nu),
                                         make_float2(-v.x, -v.y));
            const float2 d1 = __fadd2_rn(__fadd2_rn(make_float2(c.z, c.w), nu),
                                         make_float2(-v.z, -v.w));
            lo = fminf(fminf(d0.x, d0.y), fminf(d1.x, d1.y));
          } else {
            lo = fmin(fmin(c.x - uu[i] - v.x, c.y - uu[i] - v.y),
                      fmin(c.z - uu[i] - v.z, c.w - uu[i] - v.w));
          }
          if (lo < best) { best = lo; brow = a + i; }
        }
        at += 4 * RS * step;
      }
      if (brow >= 0) {
        const V4<T> c = ld4(tp(brow, gl));
        const T u = pot(brow);
        int r = 3;
        if (c.z - u - v.z == best) r = 2;
        if (c.y - u - v.y == best) r = 1;
        if (c.x - u - v.x == best) r = 0;
        key = (brow << 8) | (4 * gl + r);
      }
    }
    if constexpr (kList) {
      if (act) cand = key;
    }
    min_key<G>(best, key);
  }

  // The most negative of the lanes' candidates below -tol, key INT_MAX if none.
  __device__ __forceinline__ void price_list(bool act, T tol, T& best, int& key) {
    best = T(0);
    key = INT_MAX;
    if (act && cand != INT_MAX) {
      const int a = cand >> 8, r = cand & 0xff;
      const T d = cell(a, r) - pot(a) - pot(MP + r);
      if (d < -tol) { best = d; key = cand; }
    }
    min_key<G>(best, key);
  }

  // Bland's rule: the smallest cell with reduced cost below -tol.
  __device__ void price_bland(bool act, T tol, T& best, int& key) {
    best = T(0);
    key = INT_MAX;
    if (act && gl < nb) {
#pragma unroll 1
      for (int a = 0; a < m && key == INT_MAX; ++a) {
        if ((a >> 2) % RS != rg) continue;
#pragma unroll 1
        for (int i = 0; i < 4 && key == INT_MAX; ++i) {
          const int r = 4 * gl + i;
          const T d = cell(a, r) - pot(a) - pot(MP + r);
          if (d < -tol) { best = d; key = (a << 8) | r; }
        }
      }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      const T ov = __shfl_xor_sync(kAll, best, o * PW);
      const int ok = __shfl_xor_sync(kAll, key, o * PW);
      if (ok < key) { best = ov; key = ok; }
    }
  }

  // Group minimum of a 64-bit value that is never negative.
  __device__ __forceinline__ static long long min64(long long v) {
    if constexpr (G == 32) {
      const unsigned hi = (unsigned)((unsigned long long)v >> 32), lo = (unsigned)v;
      const unsigned mh = __reduce_min_sync(kAll, hi);
      const unsigned ml = __reduce_min_sync(kAll, hi == mh ? lo : 0xffffffffu);
      return (long long)(((unsigned long long)mh << 32) | ml);
    } else {
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) {
        const long long w = __shfl_xor_sync(kAll, v, o * PW);
        v = w < v ? w : v;
      }
      return v;
    }
  }

  // The pivot of the wide shapes (16 or 32 lanes a pair): no walk, every lane
  // tests its own nodes' masks against both ends (a node is on the cycle iff
  // its subtree holds exactly one), and a node of the cut path hands its old
  // parent the edge between them.  At 64 x 64 a side's walk is about 11 steps
  // of dependent loads: 6.0 k cycles a pivot against 3.6 k for this form.
  __device__ __forceinline__ int pivot_scan(bool act, int key, T dE) {
    const int ea = act ? key >> 8 : 0;
    const int eB = act ? MP + (key & 0xff) : MP;
    Mask<MW> mA, mB;
    mA.clear();
    mB.clear();
    if (act) {
      mA.set(ea);
      mB.set(eB);
    }
    unsigned aS = 0u, bS = 0u;  // own nodes on the row / column side
    long long th = LLONG_MAX;
    unsigned tk = 0u;  // own slots holding the smallest flow
#pragma unroll
    for (int k = 0; k < NPL; ++k) {
      const Mask<MW> D = getD(node(k));
      const long long f = flowk(k);
      const bool a = D.meets(mA), b = D.meets(mB);
      aS |= (a && !b) ? 1u << k : 0u;
      bS |= (b && !a) ? 1u << k : 0u;
      if (k < KR ? (a && !b) : (b && !a)) {
        tk = f < th ? 1u << k : (f == th ? tk | (1u << k) : tk);
        th = f < th ? f : th;
      }
    }
    const long long own = th;
    if (th < 0) th = LLONG_MAX;  // inconsistent: no leaving edge
    th = min64(th);
    int tkey = INT_MAX;
    if (own == th && th != LLONG_MAX) {
#pragma unroll 1
      for (unsigned t = tk; t; t &= t - 1) {
        const int y = node(__ffs((int)t) - 1), p = (int)par(y);
        const int kk = ((is_row(y) ? (y << 8) | (p - MP) : (p << 8) | (y - MP)) << 7) | y;
        tkey = min(tkey, kk);
      }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) tkey = min(tkey, __shfl_xor_sync(kAll, tkey, o * PW));
    const bool good = act && tkey != INT_MAX;
    const int zL = good ? tkey & 0x7f : 0;
    Mask<MW> S;
    S.clear();
    if (good) S = getD(zL);
    const bool aside = S.meets(mA);  // the leaving side holds the row end
    const int enode = aside ? ea : eB, onode = aside ? eB : ea;
    Mask<MW> Sg;  // S seen from the own slots
#pragma unroll
    for (int i = 0; i < MW; ++i) Sg.w[i] = S.w[i] >> g;
    const unsigned on = good ? (aS | bS) : 0u;
    const unsigned minus = (aS & ((1u << KR) - 1u)) | (bS & ~((1u << KR) - 1u));
    const unsigned lbits = aside ? aS : bS;
    // read everything, then write
    Mask<MW> Dn[NPL];
    long long nf[NPL];
    unsigned op[NPL];
#pragma unroll
    for (int k = 0; k < NPL; ++k) {
      op[k] = 0u;
      if ((on >> k) & 1u) {
        const bool inS = ink(Sg, k);
        Mask<MW> D;
        load(node(k), nf[k], D, op[k]);
        nf[k] += ((minus >> k) & 1u) ? -th : th;
        Dn[k] = inS ? S.minus(D) : (((lbits >> k) & 1u) ? D.minus(S) : D.plus(S));
      }
    }
    __syncwarp();
    const T se = is_row(enode) ? dE : -dE;  // shift of a row's potential
#pragma unroll
    for (int k = 0; k < NPL; ++k) {
      const bool inS = ink(Sg, k);
      if ((on >> k) & 1u) {
        const int y = node(k);
        if (!inS) store(y, nf[k], Dn[k], op[k]);
        else if (y != zL) store((int)op[k], nf[k], Dn[k], (unsigned)y);
        if (inS && y == enode) store(y, th, S, (unsigned)onode);
      }
      if (inS) potk(k) += k < KR ? se : -se;
    }
    __syncwarp();
    return good ? (th > 0 ? 1 : 0) : -1;
  }

  // One pivot on entering cell `key` with reduced cost dE < 0.  Returns 1 if
  // flow moved, 0 if none did, -1 if the tree is inconsistent.  Lane 0 of the pair walks
  // the row side of the cycle, lane 1 the column side.
  __device__ __forceinline__ int pivot(bool act, int key, T dE) {
    const int ea = key >> 8, eB = MP + (key & 0xff);
    const bool walker = act && g < 2;
    const bool colside = (g & 1) != 0;
    const int x0 = colside ? eB : ea, x1 = colside ? ea : eB;
    Mask<MW> far;  // the other end
    far.clear();
    if (act) far.set(x1);
    // 1. up to the first node above both ends; the edges that lose flow hang
    // from rows on the row side and from columns on the column side
    long long th = LLONG_MAX;
    int tkey = INT_MAX;  // (row, column, node) of the smallest flow
    bool lost = false;
    if (walker) {
      int x = x0;
      lost = true;
#pragma unroll 1
      for (int it = 0; it < NS; ++it) {
        long long f;
        Mask<MW> D;
        unsigned p;
        load(x, f, D, p);
        if (D.meets(far)) { lost = false; break; }
        if (p >= (unsigned)NS) break;
        const bool row = is_row(x);
        if (row != colside && f <= th) {
          const int kk = ((row ? (x << 8) | ((int)p - MP) : ((int)p << 8) | (x - MP)) << 7) | x;
          if (f < th || kk < tkey) { th = f; tkey = kk; }
        }
        x = (int)p;
      }
    }
    // the smaller of the two sides (ties to the smaller cell)
    const long long oth = __shfl_xor_sync(kAll, th, PW);
    const int okey = __shfl_xor_sync(kAll, tkey, PW);
    const bool mine = th < oth || (th == oth && tkey < okey);  // this side leaves
    th = mine ? th : oth;
    tkey = mine ? tkey : okey;
    const int src = threadIdx.x & (PW - 1);  // lane 0 of the pair
    const int olost = __shfl_xor_sync(kAll, (int)lost, PW);
    int z = (tkey == INT_MAX || th < 0 || lost || olost) ? -1 : tkey & 0x7f;
    // to the pair's other lanes: node, whether flow moves, which side leaves
    z = __shfl_sync(kAll, z * 4 + (th > 0 ? 2 : 0) + (mine ? 0 : 1), src);
    const int zL = z >> 2;
    const bool good = act && zL >= 0;
    const int enode = (z & 1) ? eB : ea;
    Mask<MW> S;
    S.clear();
    if (good) S = getD(zL);
    __syncwarp();
    // 2. potentials of the cut-off side
    const T se = is_row(enode) ? dE : -dE;
    Mask<MW> Sg;  // S seen from the own slots
#pragma unroll
    for (int i = 0; i < MW; ++i) Sg.w[i] = S.w[i] >> g;
#pragma unroll
    for (int k = 0; k < NPL; ++k)
      if (ink(Sg, k)) potk(k) += k < KR ? se : -se;
    // 3. the walks again: flows, masses of the subtrees, the re-hung path
    if (walker && good) {
      int x = x0;
      bool path = mine;  // still below the leaving edge: the edge turns round
      unsigned prev = (unsigned)x1;
      long long carry = th;
      Mask<MW> dprev;
      dprev.clear();
#pragma unroll 1
      for (int it = 0; it < NS; ++it) {
        long long f;
        Mask<MW> D;
        unsigned p;
        load(x, f, D, p);
        if (D.meets(far)) break;
        const long long nf = is_row(x) != colside ? f - th : f + th;
        const Mask<MW> nd = path ? S.minus(dprev) : (mine ? D.minus(S) : D.plus(S));
        store(x, path ? carry : nf, nd, path ? prev : p);
        carry = nf;
        dprev = D;
        prev = (unsigned)x;
        path = path && x != zL;
        x = (int)p;
      }
    }
    __syncwarp();
    return good ? (z >> 1) & 1 : -1;
  }

  // Pivot until no reduced cost is below -tol.  Optimality is accepted on the
  // incrementally shifted potentials (the screen's error bound covers their
  // drift).  Returns kStOk, kStNotConverged or kStInvalid.
  // With fresh_stop it is accepted on potentials just recomputed only.
  __device__ __forceinline__ int run(int max_pivots, T tol, int* pivots, bool fresh_stop = false) {
    int st = kStOk;
    int done = 0, degen = 0, since = 64;
    bool bland = false, open = live;
    if constexpr (kList) cand = INT_MAX;
    for (;;) {
      const bool due = open && since >= 64;
      if (__any_sync(kAll, due)) {  // the first round, then every 64 pivots
        const bool was = live;
        live = due;
        const bool b = refresh();
        live = was;
        if (due) since = 0;
        if (maxu(due && b ? 1u : 0u)) { st = kStInvalid; open = false; }
      }
      T dE;
      int key;
      if constexpr (kList) {
        price_list(open && !bland, tol, dE, key);
        if (__any_sync(kAll, open && !bland && key == INT_MAX)) price(open && !bland, dE, key);
      } else {
        price(open && !bland, dE, key);
      }
      if (__any_sync(kAll, open && bland)) {
        T d2;
        int k2;
        price_bland(open && bland, tol, d2, k2);
        if (bland) { dE = d2; key = k2; }
      }
      bool none = open && !(dE < -tol && key != INT_MAX);
      if (fresh_stop && none && since > 0) {  // once more on fresh potentials
        none = false;
        since = 64;
        key = INT_MAX;
      }
      if (none) open = false;
      if (open && done >= max_pivots) { st = kStNotConverged; open = false; }
      if (!__any_sync(kAll, open)) break;
      const bool go = open && key != INT_MAX;
      int moved;
      if constexpr (G >= 16) moved = pivot_scan(go, go ? key : 0, dE);
      else moved = pivot(go, go ? key : 0, dE);
      if (go) {
        if (moved < 0) {
          st = kStInvalid;
          open = false;
        } else {
          ++done;
          ++since;
          if (moved) { degen = 0; bland = false; }
          else if (++degen >= 2 * N) bland = true;
        }
      }
    }
    *pivots += done;
    return st;
  }
};

// ---- ground-cost tiles -------------------------------------------------

// Tile of FP32 bags with a small compile-time dimension: the lane keeps its 4
// centroid supports in registers (each read once per pair) and takes the
// object's rows one by one.  Same operations in the same order as cost_cells.
template <class Sh, int D>
__device__ __forceinline__ float lane_cost_small(const Lane<Sh>& P, const float* __restrict__ x,
                                                 const float* __restrict__ y) {
  float cmax = 0.f;
  if (!P.live || P.gl >= P.nb) return cmax;
  float2 y0[D], y1[D];  // columns 0, 1 and 2, 3, negated
  const int r0 = 4 * P.gl, last = P.n - 1;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    y0[k] = make_float2(-__ldg(y + min(r0, last) * D + k), -__ldg(y + min(r0 + 1, last) * D + k));
    y1[k] = make_float2(-__ldg(y + min(r0 + 2, last) * D + k),
                        -__ldg(y + min(r0 + 3, last) * D + k));
  }
  const int mq = (P.m + 3) >> 2;
#pragma unroll 1
  for (int a = 4 * P.rg; a < 4 * mq; a += (a & 3) == 3 ? 4 * Sh::RS - 3 : 1) {
    float4 c = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
    if (a < P.m) {
      float2 c0 = make_float2(0.f, 0.f), c1 = make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const float xv = __ldg(x + a * D + k);
        const float2 xx = make_float2(xv, xv);
        const float2 d0 = __fadd2_rn(xx, y0[k]), d1 = __fadd2_rn(xx, y1[k]);
        c0 = __ffma2_rn(d0, d0, c0);
        c1 = __ffma2_rn(d1, d1, c1);
      }
      c.x = r0 <= last ? c0.x : INFINITY;
      c.y = r0 + 1 <= last ? c0.y : INFINITY;
      c.z = r0 + 2 <= last ? c1.x : INFINITY;
      c.w = r0 + 3 <= last ? c1.y : INFINITY;
      cmax = r0 <= last && c0.x > cmax ? c0.x : cmax;
      cmax = r0 + 1 <= last && c0.y > cmax ? c0.y : cmax;
      cmax = r0 + 2 <= last && c1.x > cmax ? c1.x : cmax;
      cmax = r0 + 3 <= last && c1.y > cmax ? c1.y : cmax;
    }
    P.tile4(a, P.gl) = c;
  }
  return cmax;
}

// Any dimension: 4 x 4 cells at a time, the coordinates in steps of V
// (V = 4: vector loads, d a multiple of 4 and 16-byte aligned rows).
template <class Sh, typename X, int V>
__device__ __forceinline__ float lane_cost_any(const Lane<Sh>& P, const X* __restrict__ x,
                                               const float* __restrict__ y, int d) {
  float cmax = 0.f;
  if (!P.live || P.gl >= P.nb) return cmax;
  const int mq = (P.m + 3) >> 2;
  const float* yp[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) yp[j] = y + (long long)min(4 * P.gl + j, P.n - 1) * d;
#pragma unroll 1
  for (int q = P.rg; q < mq; q += Sh::RS) {
    const X* xp[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) xp[i] = x + (long long)min(4 * q + i, P.m - 1) * d;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll 1
    for (int k = 0; k < d; k += V) {
      float xv[4][V], yv[4][V];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if constexpr (V == 4) {
          const float4 t = __ldg(reinterpret_cast<const float4*>(xp[i] + k));
          xv[i][0] = t.x; xv[i][1] = t.y; xv[i][2] = t.z; xv[i][3] = t.w;
          const float4 s = __ldg(reinterpret_cast<const float4*>(yp[i] + k));
          yv[i][0] = s.x; yv[i][1] = s.y; yv[i][2] = s.z; yv[i][3] = s.w;
        } else {
          xv[i][0] = cvt<float>(xp[i][k]);
          yv[i][0] = __ldg(yp[i] + k);
        }
      }
#pragma unroll
      for (int t = 0; t < V; ++t)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float df = xv[i][t] - yv[j][t];
            acc[i][j] = fmaf(df, df, acc[i][j]);
          }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float c[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool in = 4 * q + i < P.m && 4 * P.gl + j < P.n;
        c[j] = in ? acc[i][j] : INFINITY;
        if (in && acc[i][j] > cmax) cmax = acc[i][j];
      }
      P.tile4(4 * q + i, P.gl) = make_float4(c[0], c[1], c[2], c[3]);
    }
  }
  return cmax;
}

// One value per cell from `f(a, r)`: symbol tables and ready-made tiles.
template <class Sh, typename F>
__device__ __forceinline__ float lane_cost_from(const Lane<Sh>& P, F f) {
  float cmax = 0.f;
  if (!P.live || P.gl >= P.nb) return cmax;
  const int mq = (P.m + 3) >> 2;
#pragma unroll 1
  for (int q = P.rg; q < mq; q += Sh::RS) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int a = 4 * q + i;
      float c[4] = {INFINITY, INFINITY, INFINITY, INFINITY};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = 4 * P.gl + j;
        if (a < P.m && r < P.n) {
          c[j] = f(a, r);
          cmax = c[j] > cmax ? c[j] : cmax;
        }
      }
      P.tile4(a, P.gl) = make_float4(c[0], c[1], c[2], c[3]);
    }
  }
  return cmax;
}

// Mean of each column over the object, sum_a p_a c_ar (the lane's 4 columns).
template <class Sh>
__device__ __forceinline__ float4 lane_col_means(const Lane<Sh>& P) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (P.live && P.gl < P.nb) {
#pragma unroll 1
    for (int a = 4 * P.rg; a < P.m; a += (a & 3) == 3 ? 4 * Sh::RS - 3 : 1) {
      const float p = (float)P.flow(a) * (float)kInvMass;
      const float4 c = P.tile4(a, P.gl);
      v.x = fmaf(p, c.x, v.x);
      v.y = fmaf(p, c.y, v.y);
      v.z = fmaf(p, c.z, v.z);
      v.w = fmaf(p, c.w, v.w);
    }
  }
#pragma unroll
  for (int o = Sh::G / 2; o >= Sh::L; o >>= 1) {  // the row groups
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o * Sh::PW);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o * Sh::PW);
    v.z += __shfl_xor_sync(0xffffffffu, v.z, o * Sh::PW);
    v.w += __shfl_xor_sync(0xffffffffu, v.w, o * Sh::PW);
  }
  return v;
}

// The pair's FP32 tile, its largest cost and its column means.
template <class Sh>
__device__ __forceinline__ float lane_tile(const Lane<Sh>& P, const ObjView& ob, long long o0,
                                           const CentView& cv, long long c0, const float* tile_g,
                                           long long ldc, V4<float>& vm) {
  float cmax;
  if (tile_g) {  // made ahead by the tensor cores: rows of 16 B where aligned
    if (((reinterpret_cast<uintptr_t>(tile_g) | (uintptr_t)(ldc * 4)) & 15) == 0 &&
        (P.n & 3) == 0) {
      cmax = 0.f;
      if (P.live && P.gl < P.nb && 4 * P.gl < P.n) {
        const int mq = (P.m + 3) >> 2;
#pragma unroll 1
        for (int q = P.rg; q < mq; q += Sh::RS) {
          float4 c[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            c[i] = 4 * q + i < P.m
                       ? __ldg(reinterpret_cast<const float4*>(tile_g + (4 * q + i) * ldc + 4 * P.gl))
                       : make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            P.tile4(4 * q + i, P.gl) = c[i];
            if (4 * q + i < P.m)
              cmax = fmaxf(cmax, fmaxf(fmaxf(c[i].x, c[i].y), fmaxf(c[i].z, c[i].w)));
          }
        }
      } else if (P.live && P.gl < P.nb) {
        const int mq = (P.m + 3) >> 2;
#pragma unroll 1
        for (int q = P.rg; q < mq; q += Sh::RS)
#pragma unroll 1
          for (int i = 0; i < 4; ++i)
            P.tile4(4 * q + i, P.gl) = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
      }
    } else {
      cmax = lane_cost_from(P, [&](int a, int r) { return __ldg(tile_g + a * ldc + r); });
    }
  } else if (cv.A) {
    const float* ys = cv.loc32 + c0;
    cmax = lane_cost_from(P, [&](int a, int r) {
      int xs = (int)ldx<float>(ob.loc, ob.ldt, o0 + a);
      int yy = (int)ys[r];
      xs = xs < 0 ? 0 : (xs >= cv.A ? cv.A - 1 : xs);
      yy = yy < 0 ? 0 : (yy >= cv.A ? cv.A - 1 : yy);
      return __ldg(cv.tab32 + xs * cv.A + yy);
    });
  } else {
    const int d = cv.d;
    const float* y = cv.loc32 + c0 * d;
    const long long o = o0 * d;
    if (ob.ldt == 1) {
      const float* x = static_cast<const float*>(ob.loc) + o;
      if (d == 6) cmax = lane_cost_small<Sh, 6>(P, x, y);
      else if (d == 3) cmax = lane_cost_small<Sh, 3>(P, x, y);
      else if ((d & 3) == 0 && ((reinterpret_cast<uintptr_t>(ob.loc) |
                                 reinterpret_cast<uintptr_t>(cv.loc32)) & 15) == 0)
        cmax = lane_cost_any<Sh, float, 4>(P, x, y, d);
      else cmax = lane_cost_any<Sh, float, 1>(P, x, y, d);
    } else if (ob.ldt == 2) {
      cmax = lane_cost_any<Sh, __nv_bfloat16, 1>(
          P, static_cast<const __nv_bfloat16*>(ob.loc) + o, y, d);
    } else {
      cmax = lane_cost_any<Sh, double, 1>(P, static_cast<const double*>(ob.loc) + o, y, d);
    }
  }
  cmax = Lane<Sh>::maxf(cmax);
  const float4 mean = lane_col_means(P);  // the lane's own cells
  vm = V4<float>{mean.x, mean.y, mean.z, mean.w};
  __syncwarp();
  return cmax;
}

// ---- certificate ---------------------------------------------------------

// certify_fp64 (d2_solve.cuh) on a lane pair: the same arithmetic, bounds and
// tests; only the order of the objective's FP64 sum differs.  Overwrites the
// tile's basic cells, the flows and the masks (kept: par).
template <class Sh>
__device__ __forceinline__ bool lane_certify(Lane<Sh>& P, bool go, const ObjView& ob, long long o0,
                             const CentView& cv, long long c0, float cmax, float ecost,
                             double* D64, float* tau_out, int* nchk) {
  constexpr int NPL = Sh::NPL;
  constexpr unsigned kAll = 0xffffffffu;
  const bool keep_live = P.live;
  P.live = go;
  constexpr int MP = Sh::MP, NS = Sh::NS;
  const int xt = (cv.A == 0 && ob.ldt != 0) ? ob.ldt : 0;
  // basic cells in double-float: objective terms into the flow slots (the
  // flows are done with), residuals of the FP32 potentials into aux
  bool bad = false;
#pragma unroll 1
  for (int k = 0; k < NPL; ++k) {
    const int y = P.node(k);
    if (!go || !(k < Sh::KR ? y < P.m : y - MP < P.n)) continue;
    double term = 0.0;
    float res = 0.f;
    if (y != P.root) {
      const int p = (int)P.par(y);
      const bool row = y < MP;
      if (p >= NS || row == (p < MP)) {
        bad = true;
      } else {
        const int a = row ? y : p;
        const int r = (row ? p : y) - MP;
        float ch, cl;
        cost_dd(xt, ob, o0, cv, c0, a, r, ch, cl);
        const double w = (double)P.flow(y) * kInvMass;
        term = fma(w, (double)cl, w * (double)ch);
        float s1, e1;
        two_sum(ch, -P.pot(y), s1, e1);
        e1 = __fadd_rn(e1, cl);
        float s2, e2;
        two_sum(s1, -P.pot(p), s2, e2);
        res = __fadd_rn(s2, __fadd_rn(e2, e1));
      }
    }
    *reinterpret_cast<double*>(&P.flow(y)) = term;
    P.aux(y) = res;
  }
  const double D = P.sum_nodes();
  *D64 = D;
  float delta[NPL];
#pragma unroll
  for (int k = 0; k < NPL; ++k) delta[k] = go && P.nodek(k) ? P.aux(P.node(k)) : 0.f;
  bad |= P.jump(delta, [&](int y) -> float& { return P.aux(y); });  // corrections
  unsigned pm = 0u, dm = 0u;
#pragma unroll 1
  for (int k = 0; k < NPL; ++k) {
    const int y = P.node(k);
    if (go && P.has_node(y)) {
      const float b = P.pot(y), dl = P.aux(y);  // (aux holds the sums jump ended with)
      *reinterpret_cast<float2*>(&P.flow(y)) = make_float2(b, dl);
      const float u = b + dl;
      P.pot(y) = u;
      pm = max(pm, __float_as_uint(fabsf(u)));
      dm = max(dm, __float_as_uint(fabsf(dl)));
      if (y != P.root && !bad) {
        const int p = (int)P.par(y);
        if (y < MP) P.cell(y, p - MP) = INFINITY;
        else P.cell(p, y - MP) = INFINITY;
      }
    }
  }
  const float pmax = __uint_as_float(Lane<Sh>::maxu(pm));
  const float dmax = __uint_as_float(Lane<Sh>::maxu(dm));
  __syncwarp();
  if (Lane<Sh>::oru(bad ? 1u : 0u)) { *D64 = NAN; go = false; }
  if (!isfinite(D) || !isfinite(pmax) || !isfinite(dmax) || !(cmax < FLT_MAX)) go = false;
  const float tau = fmaxf(__fmul_rd(__double2float_rd(D), 0x1p-24f), __fmul_rd(cmax, 0x1p-43f));
  if (go) *tau_out = tau;
  const float err = __fmul_ru((float)(P.N + 1),
                              __fmaf_ru((float)(6 * cv.d + 32) * 0x1p-48f, cmax,
                                        __fmul_ru(dmax, 0x1p-24f)));
  const float E = __fmul_ru(__fadd_ru(ecost, __fmul_ru(__fmaf_ru(5.f, pmax, 2.f * cmax), 0x1p-24f)),
                            1.f + 0x1p-10f);
  const float thr = __fsub_ru(__fadd_ru(E, err), tau);
  const float thr_dd = __fsub_ru(err, tau);
  // pass 1: the FP32 test of every cell (a NaN reduced cost is flagged)
  bool flagged = false;
  const bool col = go && P.gl < P.nb;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  const int mq = (P.m + 3) >> 2;
  if (col) {
    v = P.pot4((MP >> 2) + P.gl);
#pragma unroll 1
    for (int q = P.rg; q < mq; q += Sh::RS) {
      const float4 u4 = P.pot4(q);
      const float uu[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float u = uu[i];
        const float4 c = P.tile4(4 * q + i, P.gl);
        flagged |= !(c.x - u - v.x >= thr) | !(c.y - u - v.y >= thr) | !(c.z - u - v.z >= thr) |
                   !(c.w - u - v.w >= thr);
      }
    }
  }
  bool fail = false;
  if (__any_sync(kAll, flagged)) {
    // pass 2 (few pairs): the flagged cells re-priced in double-float
    int cnt = 0;
    if (flagged) {
#pragma unroll 1
      for (int q = P.rg; q < mq; q += Sh::RS) {
#pragma unroll 1
        for (int t = 0; t < 16; ++t) {
          const int a = 4 * q + (t >> 2), r = 4 * P.gl + (t & 3);
          if (a >= P.m || r >= P.n) continue;
          if (!(P.cell(a, r) - P.pot(a) - P.pot(MP + r) >= thr)) {
            ++cnt;
            float ch, cl;
            cost_dd(xt, ob, o0, cv, c0, a, r, ch, cl);
            const float2 pu = *reinterpret_cast<float2*>(&P.flow(a));
            const float2 pv = *reinterpret_cast<float2*>(&P.flow(MP + r));
            dd_add(ch, cl, -pu.x, -pu.y);
            dd_add(ch, cl, -pv.x, -pv.y);
            fail |= !((double)ch + (double)cl >= (double)thr_dd);
          }
        }
      }
    }
    *nchk += cnt;
  }
  fail = Lane<Sh>::oru(fail ? 1u : 0u) != 0u;
  P.live = keep_live;
  __syncwarp();
  return go && !fail;
}

// ---- the screen ------------------------------------------------------------

// Objects of the chunk: first list entry and count.
__device__ __forceinline__ void lane_chunk(const LaneArgs& A, long long total, long long* first,
                                           long long* cnt) {
  long long b = A.t0, e = total;
  if (A.lo) {
    b += *A.lo;
    e = *A.hi;
  }
  *first = b;
  const long long c = e - b;
  *cnt = c < 0 ? 0 : (c < A.cap ? c : A.cap);
}

// The staircase's orders into the code section: the rows' and columns' ranks
// along the object's principal direction (order_rows wrote the rows, the mean
// and the direction; the columns as order_cols), or their own order.
template <class Sh>
__device__ __forceinline__ void lane_order(Lane<Sh>& P, const LaneArgs& A, bool ranked, long long i,
                                           const float* y32, int d) {
  constexpr int NPL = Sh::NPL, KR = Sh::KR, MP = Sh::MP;
  if (ranked) {
    const float* mu = A.axes + i * 2 * d;
    const float* dir = mu + d;
#pragma unroll
    for (int k = KR; k < NPL; ++k) {
      if (P.live && P.nodek(k)) {
        const float* y = y32 + (P.node(k) - MP) * d;
        float dot = 0.f;
#pragma unroll 1
        for (int t = 0; t < d; ++t) dot = fmaf(__ldg(y + t) - __ldg(mu + t), __ldg(dir + t), dot);
        P.potk(k) = order_value(dot);
      }
    }
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k < NPL; ++k) {
    if (P.live && P.nodek(k)) {
      const int y = P.node(k);
      if (!ranked) {
        P.template u8own<Sh::kCode>(k) = (unsigned char)(k < KR ? y : y - MP);
      } else if (k < KR) {
        P.template u8own<Sh::kCode>(k) = A.rows[i * A.mstride + y];
      } else {
        const int r = y - MP;
        const float v = P.potk(k);
        int rank = 0;
#pragma unroll 1
        for (int b = 0; b < P.n; ++b) {
          const float u = P.pot(MP + b);
          rank += (u < v || (u == v && b < r)) ? 1 : 0;
        }
        P.template u8at<Sh::kCode>(MP + rank) = (unsigned char)r;
      }
    }
  }
  __syncwarp();
}

// WARM: a level's rounds.  Every pair's basis (its parents) is kept in A.tree
// by pair (i K + j), and a round starts from the one its last round saved, if
// the pair was solved then (A.warm, A.keep_was); trees of at most 32 nodes
// start cold from the ranked staircase, and in a later round from the plain
// one, as the warp-per-pair screen does, so that a level's trajectory, which
// depends on the basis where a centroid's supports coincide, stays the same.
template <class Sh, bool CERT, bool WARM>
__global__ void __launch_bounds__(64, Sh::kMinBlocks)
    k_lane_screen(ObjView ob, CentView cv, long long seg_size, int K, SolveCfg cfg, LaneArgs A,
                  long long total_obj) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int NPL = Sh::NPL, PW = Sh::PW;
  Lane<Sh> P(reinterpret_cast<char*>(smem) + (threadIdx.x >> 5) * A.warp_bytes, A.nb);
  const int lane = threadIdx.x & 31;
  long long first, cnt;
  lane_chunk(A, total_obj, &first, &cnt);
  const unsigned long long total = A.list ? A.ctr[1] : (unsigned long long)cnt * (unsigned)K;
  const float rel = (float)(cv.d + 3) * 0x1p-24f + 0x1p-17f;
  int n_scr = 0, p_scr = 0, n_cert = 0, n_chk = 0;
  for (;;) {
    unsigned long long q0 = 0;
    if (lane == 0) q0 = atomicAdd(A.ctr, (unsigned long long)PW);
    q0 = __shfl_sync(kAll, q0, 0);
    if (q0 >= total) break;
    const unsigned long long q = q0 + (lane & (PW - 1));
    P.live = q < total;
    long long tt = 0, i = 0, o0 = 0, c0 = 0, cb = 0;
    int j = 0;
    if (P.live) {
      if (A.list) {
        const uint2 e = A.list[q];
        tt = e.x;
        j = (int)e.y;
      } else {
        tt = (long long)(q / (unsigned)K);
        j = (int)(q - (unsigned long long)tt * (unsigned)K);
      }
      i = A.oidx ? (long long)A.oidx[first + tt] : A.obase + first + tt;
      o0 = ob.off[i];
      const long long mm = ob.off[i + 1] - o0;
      cb = seg_of(ob, i, seg_size) * (long long)K;
      P.live = mm >= 1 && mm <= cfg.mmax && cb + K <= cv.K && !A.obad[i];
      if (P.live) {
        c0 = cv.off[cb + j];
        const long long nn = cv.off[cb + j + 1] - c0;
        P.live = nn >= 1 && nn <= cfg.nmax;
        P.m = (int)mm;
        P.n = (int)nn;
      }
    }
    if (!P.live) P.m = P.n = 1;
    P.N = P.m + P.n;
    // masses, singleton masks, potentials of the unused slots
#pragma unroll 1
    for (int k = 0; k < NPL; ++k) {
      const int y = P.node(k);
      long long w = 0;
      Mask<Sh::MW> d;
      d.clear();
      if (P.live && P.has_node(y)) {
        d.set(y);
        if (y < Sh::MP) {
          w = A.omass[i * A.mstride + y];
        } else {
          const int r = y - Sh::MP;
          w = cv.Qpre[c0 + r] - (r > 0 ? cv.Qpre[c0 + r - 1] : 0LL);
        }
      }
      P.store(y, w, d, 0xffu);
      P.potk(k) = 0.f;
    }
    __syncwarp();
    const float* tile_g = nullptr;
    float nxm = 0.f;
    if (cfg.tile.C) {
      if (P.live) {
        const long long trow0 = cfg.tile.trow[tt];
        tile_g = cfg.tile.C + trow0 * cfg.tile.ldc + (c0 - cfg.tile.col0);
#pragma unroll 1
        for (int a = P.g; a < P.m; a += Sh::G) nxm = fmaxf(nxm, cfg.tile.nx[trow0 + a]);
      } else {
        tile_g = cfg.tile.C;
      }
      nxm = Lane<Sh>::maxf(nxm);
    }
    V4<float> vm;
    const float cmax = lane_tile<Sh>(P, ob, o0, cv, c0, tile_g, cfg.tile.ldc, vm);
    bool wbad = false;  // a saved basis that is not a feasible tree
    if constexpr (WARM) {
      const bool lv = P.live;
      const bool fresh = !A.warm || (A.keep_was &&
                                     !((A.keep_was[i * cfg.keep_words + (j >> 5)] >> (j & 31)) & 1u));
      const unsigned char* tr = A.tree + (unsigned long long)(i * (long long)K + j) * A.tstride;
      P.live = lv && !fresh;
      int root = INT_MAX;
#pragma unroll
      for (int k = 0; k < NPL; ++k) {
        if (P.live && P.nodek(k)) {
          const int y = P.node(k);
          unsigned p = tr[k < Sh::KR ? y : y - Sh::MP + P.m];
          if (p == 0xffu) root = min(root, y);
          else if (p >= (unsigned)P.m) p = p - P.m + Sh::MP;
          P.put_par(y, p);
        }
      }
#pragma unroll
      for (int o = Sh::G / 2; o > 0; o >>= 1)
        root = min(root, __shfl_xor_sync(kAll, root, o * PW));
      if (P.live) P.root = root == INT_MAX ? 0 : root;
      __syncwarp();
      if (__any_sync(kAll, P.live)) wbad = P.template from_parents<true>();
      P.live = lv && fresh;
      if (__any_sync(kAll, P.live)) {
        if constexpr (Sh::MW == 1) {
          lane_order<Sh>(P, A, !A.warm, i, cv.loc32 + c0 * cv.d, cv.d);
          P.start_staircase();
        } else {
          P.start_rows(vm);
        }
      }
      P.live = lv;
      __syncwarp();
    } else {
      P.start_rows(vm);
    }
    int piv = 0;
    int st = P.run(cfg.budget * P.N, tol32(cmax), &piv);
    if (WARM && wbad) st = kStInvalid;
    if (P.live && P.g == 0) {
      ++n_scr;
      p_scr += piv;
    }
    if (A.tree && P.live) {  // the basis, for the exact pass (parents, compact node numbers)
      unsigned char* tr = A.tree + (WARM ? (unsigned long long)(i * (long long)K + j) : q) *
                                       (unsigned long long)A.tstride;
#pragma unroll 1
      for (int k = 0; k < NPL; ++k) {
        const int y = P.node(k);
        if (P.has_node(y)) {
          const unsigned p = P.par(y);
          tr[y < Sh::MP ? y : y - Sh::MP + P.m] =
              (unsigned char)(y == P.root || st == kStInvalid
                                  ? 0xffu
                                  : (p < (unsigned)Sh::MP ? p : p - Sh::MP + P.m));
        }
      }
    }
    float tc_e = 0.f;
    if (cfg.tile.C && P.live) tc_e = tc_bound(cv.d, nxm, cfg.tile.cn[cb + j], cfg.tile.cd[cb + j]);
    PairRec rec;
    rec.d64 = NAN;
    if constexpr (CERT) {
      double D64 = NAN;
      float tau = 0.f;
      const float ecost = cfg.tile.C ? tc_e : (cv.A ? 0x1p-23f : (float)(cv.d + 3) * 0x1p-24f) * cmax;
      const bool cert = lane_certify<Sh>(P, P.live && st == kStOk, ob, o0, cv, c0, cmax, ecost, &D64,
                                         &tau, &n_chk);
      const float dhi = __double2float_ru(D64);
      if (cert) {
        if (P.g == 0) ++n_cert;
        rec.lo = __fsub_rd(__fmul_rd(__double2float_rd(D64), 1.f - 0x1p-22f), tau);
        rec.hi = __fmul_ru(dhi, 1.f + 0x1p-22f);
        rec.d64 = D64;
      } else {
        rec.lo = -FLT_MAX;
        rec.hi = st == kStOk && isfinite(D64) ? __fmul_ru(dhi, 1.f + 0x1p-22f) : FLT_MAX;
      }
      if (P.live && P.g == 0 && cfg.pair64) cfg.pair64[i * (long long)K + j] = rec.d64;
    } else {
      // FP32 objective and its error bound
      float acc = 0.f;
#pragma unroll 1
      for (int k = 0; k < NPL; ++k) {
        const int y = P.node(k);
        if (P.live && P.has_node(y) && y != P.root) {
          const int p = (int)P.par(y);
          if (p < Sh::NS) acc += ((float)P.flow(y) * (float)kInvMass) * P.edge_cost(y, p);
        }
      }
      const float D = Lane<Sh>::sum(acc);
      const float e = D * rel + cmax * 0x1p-14f + tc_e;
      const bool good = st == kStOk && isfinite(D) && isfinite(e);
      if (P.live && P.g == 0 && cfg.pair_out) {
        float* po = cfg.pair_out + 2 * (i * (long long)K + j);
        po[0] = D;
        po[1] = st != kStOk ? INFINITY : e;
      }
      // a solve that failed has no bound; one whose costs are not finite is
      // no candidate
      rec.lo = good ? D - e : (st == kStOk ? INFINITY : -FLT_MAX);
      rec.hi = good ? D + e : FLT_MAX;
    }
    if (q < total && P.g == 0) {
      if (!P.live) {
        rec.lo = -FLT_MAX;
        rec.hi = FLT_MAX;
        rec.d64 = NAN;
        if (cfg.pair_out) cfg.pair_out[2 * (i * (long long)K + j)] = NAN;
        if (cfg.pair64) cfg.pair64[i * (long long)K + j] = NAN;
      }
      A.rec[q] = rec;
    }
    __syncwarp();
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    n_scr += __shfl_xor_sync(kAll, n_scr, o);
    p_scr += __shfl_xor_sync(kAll, p_scr, o);
    n_cert += __shfl_xor_sync(kAll, n_cert, o);
    n_chk += __shfl_xor_sync(kAll, n_chk, o);
  }
  if (lane == 0) add_stats(n_scr, p_scr, 0, 0, n_cert, n_chk);
}

// Basis flows of the tree in shared memory as records (one entry
// per node but the root, in node order).
template <class Sh>
__device__ __forceinline__ void lane_flows(const Lane<Sh>& P, int* fc, double* fw,
                                           long long stride) {
  constexpr int MP = Sh::MP;
  const int rc = P.root < MP ? P.root : P.root - MP + P.m;
#pragma unroll
  for (int k = 0; k < Sh::NPL; ++k) {
    const int y = P.node(k);
    if (P.nodek(k) && y != P.root) {
      const int p = (int)P.par(y);
      const int e = k < Sh::KR ? y : y - MP + P.m;
      fc[e < rc ? e : e - 1] = k < Sh::KR ? (y << 16) | (p - MP) : (p << 16) | (y - MP);
      fw[e < rc ? e : e - 1] = (double)P.flowk(k) * kInvMass;
    }
  }
#pragma unroll 1
  for (long long e = P.N - 1 + P.g; e < stride; e += Sh::G) {
    fc[e] = -1;
    fw[e] = 0.0;
  }
}

// ---- the exact pass --------------------------------------------------------

// Exact value of one pair from the basis the screen saved: the basic cells'
// costs, the objective and the potentials in FP64, and the optimality test of
// k_exact (no FP64 reduced cost below -2^-43 c_max) with the FP32 tile as its
// filter: a cell whose FP32 reduced cost clears the rounding bound E of
// lane_certify has a non-negative FP64 one, the few others are priced in FP64.
// Returns 0 if the basis is optimal, 1 with the most negative cell (key, dE)
// if not, 2 for an inconsistent tree or a value that is not finite.  `value`
// false: only the flows are wanted (certified pairs).
template <class Sh>
__device__ __forceinline__ int lane_verify(Lane<Sh>& P, bool go, bool value, char* pot64,
                                           const ObjView& ob, long long o0, const CentView& cv,
                                           long long c0, double* D64, int* ekey, float* edE) {
  constexpr int NPL = Sh::NPL, MP = Sh::MP, PS = Sh::PS;
  constexpr unsigned kAll = 0xffffffffu;
  P.live = go;
  auto u64 = [&](int y) -> double& {
    return *reinterpret_cast<double*>(pot64 + (y >> 1) * PS + (y & 1) * 8);
  };
  const bool bad = P.template from_parents<false>();
  const bool full = go && value && !bad;
  if (!__any_sync(kAll, full)) return go && bad ? 2 : 0;
  double worst = 0.0;  // most negative reduced cost below -tol
  int wkey = INT_MAX;
  P.live = full;
  V4<float> vm;
  const float cmax = lane_tile<Sh>(P, ob, o0, cv, c0, nullptr, 0, vm);
  // basic cells in FP64
  double edge[NPL];
#pragma unroll 1
  for (int k = 0; k < NPL; ++k) {
    const int y = P.node(k);
    double c = 0.0;
    if (full && (k < Sh::KR ? y < P.m : y - MP < P.n) && y != P.root) {
      const int p = (int)P.par(y);
      c = y < MP ? cost64_cell(ob, o0, cv, c0, y, p - MP) : cost64_cell(ob, o0, cv, c0, p, y - MP);
    }
    u64(y) = c;
  }
#pragma unroll
  for (int k = 0; k < NPL; ++k) edge[k] = u64(P.node(k));
  __syncwarp();
  double pot[NPL];
#pragma unroll
  for (int k = 0; k < NPL; ++k) pot[k] = edge[k];
  bool fail = P.jump(pot, u64);
  float pm = 0.f;
#pragma unroll
  for (int k = 0; k < NPL; ++k) {
    const int y = P.node(k);
    if (full && P.nodek(k)) {
      const float u = __double2float_rn(pot[k]);
      P.pot(y) = u;
      pm = fmaxf(pm, fabsf(u));
      fail |= !isfinite(u);
      if (y != P.root) {  // a basic cell's reduced cost is zero
        const int p = (int)P.par(y);
        if (k < Sh::KR) P.cell(y, p - MP) = INFINITY;
        else P.cell(p, y - MP) = INFINITY;
      }
    }
  }
  const float pmax = Lane<Sh>::maxf(pm);
  __syncwarp();
  const float ecost = (cv.A ? 0x1p-23f : (float)(cv.d + 3) * 0x1p-24f) * cmax;
  const float E = __fmul_ru(__fadd_ru(ecost, __fmul_ru(__fmaf_ru(5.f, pmax, 2.f * cmax), 0x1p-24f)),
                            1.f + 0x1p-10f);
  if (!(cmax < FLT_MAX) || !isfinite(E)) fail = true;
  const double tol = (double)cmax * (0x1p-43 * (1.0 - 0x1p-12));
  const int mq = (P.m + 3) >> 2;
  if (full && P.gl < P.nb) {
    const float4 v = P.pot4((MP >> 2) + P.gl);
    const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll 1
    for (int a = 4 * P.rg; a < 4 * mq; a += (a & 3) == 3 ? 4 * Sh::RS - 3 : 1) {
      const float u = P.pot(a);
      const float4 c = P.tile4(a, P.gl);
      const float cc[4] = {c.x, c.y, c.z, c.w};
      unsigned flag = 0u;
#pragma unroll
      for (int t = 0; t < 4; ++t) flag |= !(cc[t] - u - vv[t] >= E) ? 1u << t : 0u;
#pragma unroll 1
      for (; flag; flag &= flag - 1) {
        const int r = 4 * P.gl + __ffs((int)flag) - 1;
        if (a < P.m && r < P.n) {
          const double dd = cost64_cell(ob, o0, cv, c0, a, r) - u64(a) - u64(MP + r);
          if (!(dd >= -tol)) {
            fail |= isnan(dd);
            if (dd < worst) { worst = dd; wkey = (a << 8) | r; }
          }
        }
      }
    }
  }
  // objective (the flow slots become its terms; kept for the flow records)
  long long fl[NPL];
#pragma unroll
  for (int k = 0; k < NPL; ++k) {
    fl[k] = P.flowk(k);
    if (full && P.nodek(k))
      *reinterpret_cast<double*>(&P.flowk(k)) = ((double)fl[k] * kInvMass) * edge[k];
  }
  const double D = P.sum_nodes();
#pragma unroll
  for (int k = 0; k < NPL; ++k) P.flowk(k) = fl[k];
  __syncwarp();
  if (full) *D64 = D;
  fail |= full && !isfinite(D);
  fail = Lane<Sh>::oru(fail ? 1u : 0u) != 0u;
#pragma unroll
  for (int o = Sh::G / 2; o > 0; o >>= 1) {
    const double od = __shfl_xor_sync(kAll, worst, o * Sh::PW);
    const int ok = __shfl_xor_sync(kAll, wkey, o * Sh::PW);
    if (od < worst || (od == worst && ok < wkey)) { worst = od; wkey = ok; }
  }
  *ekey = wkey;
  *edE = __double2float_rn(worst);
  if (go && (bad || (full && fail))) return 2;
  return full && wkey != INT_MAX ? 1 : 0;
}

// Tests of a basis before its pair is left to the warp-per-pair kernel.  A test
// builds the tile and the FP64 potentials anew (130 us on one warp at 32 x 32 in
// 16 dimensions), where that kernel pivots on.  Ordinary bags need no pivot at
// all; one whose supports nearly coincide took up to 20, and its launch waited
// (4,000 pairs of merged centroids 7.4 -> 2.1 ms, ten rounds of 256 such bags
// 39.6 -> 15.0; 2 tests 13.5, 6 tests 19.6).
constexpr int kRepairs = 3;

// The candidates of the chunk's objects (k_lane_merge's records) to their
// labels and exact distances, as k_exact: a basis that is not optimal in FP64
// takes its pivot here (the same entering cell) and is tested again; an object
// with a candidate that still does not verify is listed for k_exact (fb,
// counted in ctr[2]).
template <class Sh>
__global__ void __launch_bounds__(64, Sh::kMinBlocks)
    k_lane_exact(ObjView ob, CentView cv, long long seg_size, int K, SolveCfg cfg, LaneArgs A,
                 long long total_obj, ExactOut X) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int NPL = Sh::NPL, PW = Sh::PW, MP = Sh::MP;
  char* warp_base = reinterpret_cast<char*>(smem) + (threadIdx.x >> 5) * A.warp_bytes;
  Lane<Sh> P(warp_base, A.nb);
  char* pot64 = warp_base + A.warp_bytes - (Sh::NS / 2) * Sh::PS + (P.sp - warp_base);
  const int lane = threadIdx.x & 31;
  long long first, cnt;
  lane_chunk(A, total_obj, &first, &cnt);
  int n_ex = 0, p_ex = 0;
  const long long step = (long long)gridDim.x * (blockDim.x >> 5) * PW;
#pragma unroll 1
  for (long long t0 = ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * PW; t0 < cnt;
       t0 += step) {
    const long long t = t0 + (lane & (PW - 1));
    const bool have = t < cnt;
    long long i = 0, o0 = 0, cb = 0;
    const int* mr = X.cand;
    int nc = 0;
    if (have) {
      i = A.oidx ? (long long)A.oidx[first + t] : A.obase + first + t;
      mr = X.cand + i * kMergedInts;
      nc = mr[0];
      o0 = ob.off[i];
      P.m = (int)(ob.off[i + 1] - o0);
      cb = seg_of(ob, i, seg_size) * (long long)K;
    }
    const bool invalid = have && nc == -2;
    bool fallback = have && (nc == -1 || nc == 0);
    if (!have || nc < 1) { nc = 0; P.m = 1; }
    double d64c = NAN;
    if ((cfg.certify || cfg.mode == 0) && nc == 1)
      d64c = __longlong_as_double(((long long)mr[2 + kCandCap] << 32) |
                                  (long long)(unsigned)mr[1 + kCandCap]);
    const bool known = cfg.mode == 0 || !isnan(d64c);  // (FP64 throughout: always)
    double best = NAN;
    int best_j = -1;
#pragma unroll 1
    for (int c = 0; __any_sync(kAll, c < nc); ++c) {
      const bool go = c < nc && !fallback && (!known || X.fo.cell);
      int j = 0;
      long long c0 = 0;
      P.n = 1;
      unsigned long long q = 0;
      if (go) {
        j = mr[1 + c];
        c0 = cv.off[cb + j];
        P.n = (int)(cv.off[cb + j + 1] - c0);
        if (A.by_pair) {
          q = (unsigned long long)(i * (long long)K + j);
        } else if (A.list) {  // the pair's place in the list: kept centroids before j
          const unsigned* kb = cfg.keep + i * cfg.keep_words;
          q = X.ostart[t] + __popc(kb[j >> 5] & ((1u << (j & 31)) - 1u));
#pragma unroll 1
          for (int w = 0; w < (j >> 5); ++w) q += __popc(kb[w]);
        } else {
          q = (unsigned long long)t * (unsigned)K + (unsigned)j;
        }
      }
      P.N = P.m + P.n;
      P.live = go;
      // the saved tree, then (again after each pivot) the masses
      const unsigned char* tr = A.tree + q * (unsigned long long)A.tstride;
      int root = INT_MAX;
      __syncwarp();
#pragma unroll
      for (int k = 0; k < NPL; ++k) {
        const int y = P.node(k);
        unsigned p = 0xffu;
        if (go && P.nodek(k)) {
          p = tr[k < Sh::KR ? y : y - MP + P.m];
          if (p == 0xffu) root = min(root, y);
          else if (p >= (unsigned)P.m) p = p - P.m + MP;
        }
        P.put_par(y, p);
        P.potk(k) = 0.f;
      }
#pragma unroll
      for (int o = Sh::G / 2; o > 0; o >>= 1)
        root = min(root, __shfl_xor_sync(kAll, root, o * PW));
      P.root = root == INT_MAX ? 0 : root;
      auto masses = [&](bool on) {
        __syncwarp();
#pragma unroll 1
        for (int k = 0; k < NPL; ++k) {
          const int y = P.node(k);
          if (!on) continue;
          long long w = 0;
          Mask<Sh::MW> one;
          one.clear();
          if (y < MP ? y < P.m : y - MP < P.n) {
            one.set(y);
            if (y < MP) {
              w = A.omass[i * A.mstride + y];
            } else {
              const int r = y - MP;
              w = cv.Qpre[c0 + r] - (r > 0 ? cv.Qpre[c0 + r - 1] : 0LL);
            }
          }
          P.store(y, w, one, P.par(y));
        }
        __syncwarp();
      };
      double D = d64c;
      bool todo = go;
      int verdict = go ? 2 : 0;
#pragma unroll 1
      for (int att = 0; att < kRepairs; ++att) {
        masses(todo);
        int key;
        float dE;
        const int v = lane_verify<Sh>(P, todo, !known, pot64, ob, o0, cv, c0, &D, &key, &dE);
        if (todo) verdict = v;
        todo = todo && v == 1;
        if (!__any_sync(kAll, todo)) break;
        masses(todo);
        P.live = todo;
        P.template from_parents<true>();
        int moved;
        if constexpr (Sh::G >= 16) moved = P.pivot_scan(todo, todo ? key : 0, dE);
        else moved = P.pivot(todo, todo ? key : 0, dE);
        if (todo && moved < 0) {
          verdict = 2;
          todo = false;
        }
        if (todo && P.g == 0) ++p_ex;
      }
      P.live = go;
      if (go && verdict != 0) fallback = true;
      if (go && verdict == 0 && !known && P.g == 0) {
        ++n_ex;
        if (cfg.pair64) cfg.pair64[i * (long long)K + j] = D;
      }
      const bool better = c < nc && !fallback && (best_j < 0 || D < best);
      if (better) {
        best = D;
        best_j = mr[1 + c];
        if (X.fo.cell) {  // basis flows: one entry per node but the root
          lane_flows<Sh>(P, X.fo.cell + i * X.fo.stride, X.fo.w + i * X.fo.stride, X.fo.stride);
        }
      }
      __syncwarp();
    }
    if (have && P.g == 0) {
      if (fallback) {
        X.fb[atomicAdd(A.ctr + 2, 1ull)] = (int)i;
      } else {
        X.labels[i] = invalid ? -1 : best_j;
        const double dd = invalid ? NAN : best;
        X.dist2[i] = dd;
        if (X.eps_terms) X.eps_terms[i] = (X.omega ? X.omega[i] : 1.0) * dd;
        if (invalid) atomicOr(X.err, kErrInvalid);
      }
    }
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    n_ex += __shfl_xor_sync(kAll, n_ex, o);
    p_ex += __shfl_xor_sync(kAll, p_ex, o);
  }
  if (lane == 0) add_stats(0, 0, n_ex, p_ex);
}

// ---- pair lists, and FP64 throughout ---------------------------------------

// FP64 tile, its largest cost and its column means (the arithmetic of
// cost64_cell).
template <class Sh>
__device__ __forceinline__ double lane_tile64(const Lane<Sh>& P, const ObjView& ob, long long o0,
                                              const CentView& cv, long long c0, V4<double>& vm) {
  double cmax = 0.0;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  if (P.live && P.gl < P.nb) {
    const int mq = (P.m + 3) >> 2;
#pragma unroll 1
    for (int q = P.rg; q < mq; q += Sh::RS) {
#pragma unroll 1
      for (int a = 4 * q; a < 4 * q + 4; ++a) {
        double c[4];
        const double p = a < P.m ? (double)P.flow(a) * kInvMass : 0.0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int r = 4 * P.gl + j;
          c[j] = INFINITY;
          if (a < P.m && r < P.n) {
            c[j] = cost64_cell(ob, o0, cv, c0, a, r);
            cmax = c[j] > cmax ? c[j] : cmax;
            v[j] = fma(p, c[j], v[j]);
          }
        }
        P.st4(P.tp(a, P.gl), V4<double>{c[0], c[1], c[2], c[3]});
      }
    }
  }
#pragma unroll
  for (int o = Sh::G / 2; o >= Sh::L; o >>= 1)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o * Sh::PW);
#pragma unroll
  for (int o = Sh::G / 2; o > 0; o >>= 1) {
    const double w = __shfl_xor_sync(0xffffffffu, cmax, o * Sh::PW);
    cmax = w > cmax ? w : cmax;
  }
  vm = V4<double>{v[0], v[1], v[2], v[3]};
  __syncwarp();
  return cmax;
}

// Masses, singleton sets and zero potentials of a pair (m, n, live set); the
// object's weights are quantised here.  Returns false for a rejected bag.
template <class Sh>
__device__ __forceinline__ bool lane_load(Lane<Sh>& P, bool act, const ObjView& ob, long long o0,
                                          const CentView& cv, long long c0) {
#pragma unroll
  for (int k = 0; k < Sh::NPL; ++k) {
    const int y = P.node(k);
    long long w = 0;
    Mask<Sh::MW> d;
    d.clear();
    if (act && P.nodek(k)) {
      d.set(y);
      if (k >= Sh::KR) {
        const int r = y - Sh::MP;
        w = cv.Qpre[c0 + r] - (r > 0 ? cv.Qpre[c0 + r - 1] : 0LL);
      }
    }
    P.store(y, w, d, 0xffu);
    P.potk(k) = 0;
  }
  __syncwarp();
  const bool ok = ob.wdt == 0 ? P.row_masses(act, static_cast<const double*>(ob.w) + o0)
                              : P.row_masses(act, static_cast<const float*>(ob.w) + o0);
  __syncwarp();
  return ok;
}

// The masses and singleton sets again, the tree kept.
template <class Sh>
__device__ __forceinline__ void lane_reset(Lane<Sh>& P, bool on, const ObjView& ob, long long o0,
                                           const CentView& cv, long long c0) {
  __syncwarp();
#pragma unroll 1
  for (int k = 0; k < Sh::NPL; ++k) {
    const int y = P.node(k);
    if (!on) continue;
    long long w = 0;
    Mask<Sh::MW> one;
    one.clear();
    if (y < Sh::MP ? y < P.m : y - Sh::MP < P.n) {
      one.set(y);
      if (y >= Sh::MP) {
        const int r = y - Sh::MP;
        w = cv.Qpre[c0 + r] - (r > 0 ? cv.Qpre[c0 + r - 1] : 0LL);
      }
    }
    P.store(y, w, one, P.par(y));
  }
  __syncwarp();
  if (ob.wdt == 0) P.row_masses(on, static_cast<const double*>(ob.w) + o0, on);
  else P.row_masses(on, static_cast<const float*>(ob.w) + o0, on);
  __syncwarp();
}

// FP64 throughout: start, pivots and objective on the FP64 tile.
template <class Sh>
__device__ __forceinline__ int lane_solve64(Lane<Sh>& P, const ObjView& ob, long long o0,
                                            const CentView& cv, long long c0, int budget,
                                            double* D, int* piv) {
  V4<double> vm;
  const double cmax = lane_tile64<Sh>(P, ob, o0, cv, c0, vm);
  P.start_rows(vm);
  const int st = P.run(budget * P.N, tol64(cmax), piv, true);
  long long fl[Sh::NPL];
#pragma unroll
  for (int k = 0; k < Sh::NPL; ++k) {
    fl[k] = P.flowk(k);
    const int y = P.node(k);
    double t = 0.0;
    if (P.live && P.nodek(k) && y != P.root) {
      const int p = (int)P.par(y);
      if (p < Sh::NS && (k < Sh::KR) != (p < Sh::MP))
        t = ((double)fl[k] * kInvMass) *
            (k < Sh::KR ? P.cell(y, p - Sh::MP) : P.cell(p, y - Sh::MP));
    }
    if (P.live && P.nodek(k)) *reinterpret_cast<double*>(&P.flowk(k)) = t;
  }
  *D = P.sum_nodes();
#pragma unroll
  for (int k = 0; k < Sh::NPL; ++k) P.flowk(k) = fl[k];
  __syncwarp();
  return st;
}

// Listed pairs, one pass: FP32 shapes solve in FP32, then verify and repair in
// FP64 as the exact pass does; FP64 shapes solve in FP64 throughout.  done[t]:
// the pair's results are written (0: left to the warp-per-pair kernel).
template <class Sh>
__global__ void __launch_bounds__(64, Sh::kMinBlocks)
    k_lane_pairs(ObjView ob, CentView cv, PairJob J, SolveCfg cfg, int nb, int warp_bytes) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int PW = Sh::PW;
  char* warp_base = reinterpret_cast<char*>(smem) + (threadIdx.x >> 5) * warp_bytes;
  Lane<Sh> P(warp_base, nb);
  char* pot64 = warp_base + warp_bytes - (Sh::NS / 2) * Sh::PS + (P.sp - warp_base);
  const int lane = threadIdx.x & 31;
  int n_ex = 0, p_ex = 0;
  const long long step = (long long)gridDim.x * (blockDim.x >> 5) * PW;
#pragma unroll 1
  for (long long t0 = ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * PW;
       t0 < J.npairs; t0 += step) {
    const long long t = t0 + (lane & (PW - 1));
    bool act = false;
    long long o0 = 0, c0 = 0;
    P.m = P.n = 1;
    if (t < J.npairs) {
      const long long i = J.pobj[t], j = J.pcen[t];
      if (i >= 0 && i < ob.count && j >= 0 && j < cv.K) {
        o0 = ob.off[i];
        c0 = cv.off[j];
        const long long mm = ob.off[i + 1] - o0, nn = cv.off[j + 1] - c0;
        act = mm >= 1 && mm <= cfg.mmax && nn >= 1 && nn <= cfg.nmax;
        if (act) {
          P.m = (int)mm;
          P.n = (int)nn;
        }
      }
    }
    P.N = P.m + P.n;
    P.live = act;
    P.root = 0;
    __syncwarp();
    act = lane_load<Sh>(P, act, ob, o0, cv, c0);
    P.live = act;
    double D = NAN;
    int st = kStInvalid, piv = 0;
    if constexpr (Sh::TS == 8) {
      st = lane_solve64<Sh>(P, ob, o0, cv, c0, cfg.budget, &D, &piv);
    } else {
      V4<float> vm;
      const float cmax = lane_tile<Sh>(P, ob, o0, cv, c0, nullptr, 0, vm);
      P.start_rows(vm);
      const int s32 = P.run(cfg.budget * P.N, tol32(cmax), &piv);
      // the basis in FP64, pivots while it is not optimal there
      bool todo = act && s32 == kStOk;
      bool good = false;
#pragma unroll 1
      for (int att = 0; att < kRepairs; ++att) {
        lane_reset<Sh>(P, todo, ob, o0, cv, c0);
        int key;
        float dE;
        const int v = lane_verify<Sh>(P, todo, true, pot64, ob, o0, cv, c0, &D, &key, &dE);
        if (todo && v == 0) good = true;
        todo = todo && v == 1;
        if (!__any_sync(kAll, todo)) break;
        lane_reset<Sh>(P, todo, ob, o0, cv, c0);
        P.live = todo;
        P.template from_parents<true>();
        int moved;
        if constexpr (Sh::G >= 16) moved = P.pivot_scan(todo, todo ? key : 0, dE);
        else moved = P.pivot(todo, todo ? key : 0, dE);
        if (todo && moved < 0) todo = false;
        if (todo) ++piv;
      }
      P.live = act;
      st = good ? kStOk : kStInvalid;
    }
    if (act && P.g == 0) {
      ++n_ex;
      p_ex += piv;
    }
    const bool write = act && (Sh::TS == 8 ? st != kStInvalid : st == kStOk);
    if (t < J.npairs && P.g == 0) {
      J.done[t] = write ? 1 : 0;
      if (write) {
        J.dist2[t] = D;
        if (J.status) J.status[t] = st == kStOk ? 0 : -3;
        if (st == kStNotConverged) atomicOr(J.err, kErrNotConverged);
      }
    }
    if (write && J.fo.cell) lane_flows<Sh>(P, J.fo.cell + t * J.fo.stride, J.fo.w + t * J.fo.stride, J.fo.stride);
    __syncwarp();
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    n_ex += __shfl_xor_sync(kAll, n_ex, o);
    p_ex += __shfl_xor_sync(kAll, p_ex, o);
  }
  if (lane == 0) add_stats(0, 0, n_ex, p_ex);
}

// Every pair of the chunk in FP64 throughout: its value (rec) and basis (tree).
template <class Sh>
__global__ void __launch_bounds__(64, Sh::kMinBlocks)
    k_lane_all64(ObjView ob, CentView cv, long long seg_size, int K, SolveCfg cfg, LaneArgs A,
                 long long total_obj, int* err) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int PW = Sh::PW;
  Lane<Sh> P(reinterpret_cast<char*>(smem) + (threadIdx.x >> 5) * A.warp_bytes, A.nb);
  const int lane = threadIdx.x & 31;
  long long first, cnt;
  lane_chunk(A, total_obj, &first, &cnt);
  const long long total = cnt * (long long)K;
  int n_ex = 0, p_ex = 0;
  const long long step = (long long)gridDim.x * (blockDim.x >> 5) * PW;
#pragma unroll 1
  for (long long q0 = ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * PW;
       q0 < total; q0 += step) {
    const long long q = q0 + (lane & (PW - 1));
    bool act = q < total;
    long long i = 0, o0 = 0, c0 = 0;
    int j = 0;
    P.m = P.n = 1;
    if (act) {
      const long long tt = q / K;
      j = (int)(q - tt * K);
      i = A.oidx ? (long long)A.oidx[first + tt] : A.obase + first + tt;
      o0 = ob.off[i];
      const long long mm = ob.off[i + 1] - o0;
      const long long cb = seg_of(ob, i, seg_size) * (long long)K;
      act = mm >= 1 && mm <= cfg.mmax && cb + K <= cv.K && !A.obad[i];
      if (act) {
        c0 = cv.off[cb + j];
        const long long nn = cv.off[cb + j + 1] - c0;
        act = nn >= 1 && nn <= cfg.nmax;
        if (act) {
          P.m = (int)mm;
          P.n = (int)nn;
        }
      }
    }
    P.N = P.m + P.n;
    P.live = act;
    P.root = 0;
    __syncwarp();
    act = lane_load<Sh>(P, act, ob, o0, cv, c0);
    P.live = act;
    double D = NAN;
    int piv = 0;
    const int st = lane_solve64<Sh>(P, ob, o0, cv, c0, cfg.budget, &D, &piv);
    if (act && P.g == 0) {
      ++n_ex;
      p_ex += piv;
      if (st == kStInvalid) atomicOr(err, kErrInvalid);
      if (st == kStNotConverged) atomicOr(err, kErrNotConverged);
    }
    if (act && A.tree) {
      unsigned char* tr = A.tree + (unsigned long long)q * A.tstride;
#pragma unroll
      for (int k = 0; k < Sh::NPL; ++k) {
        if (P.nodek(k)) {
          const int y = P.node(k);
          const unsigned p = P.par(y);
          tr[k < Sh::KR ? y : y - Sh::MP + P.m] = (unsigned char)(
              y == P.root ? 0xffu : (p < (unsigned)Sh::MP ? p : p - Sh::MP + P.m));
        }
      }
    }
    if (q < total && P.g == 0) {
      PairRec r;
      r.lo = r.hi = 0.f;
      r.d64 = act && st != kStInvalid ? D : NAN;
      A.rec[q] = r;
      if (cfg.pair64) cfg.pair64[i * (long long)K + j] = r.d64;
    }
    __syncwarp();
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    n_ex += __shfl_xor_sync(kAll, n_ex, o);
    p_ex += __shfl_xor_sync(kAll, p_ex, o);
  }
  if (lane == 0) add_stats(0, 0, n_ex, p_ex);
}

// Blocks of two warps where they fit, one otherwise.
template <typename Kern, typename... Args>
cudaError_t lane_blocks(Kern kern, int warp_bytes, int sms, long long warps_of_work,
                        cudaStream_t st, const Args&... args) {
  const int warps = 2 * warp_bytes <= 113 * 1024 ? 2 : 1;
  const size_t smem = (size_t)warp_bytes * warps;
  unsigned grid = 1;
  const cudaError_t e = launch_cfg(kern, smem, 32 * warps, sms, warps_of_work, warps, &grid);
  if (e != cudaSuccess) return e;
  kern<<<grid, 32 * warps, smem, st>>>(args...);
  note_launches(1);
  return cudaGetLastError();
}

// One launch of the shape: the screen (X.labels null) or the exact pass.
template <class Sh>
cudaError_t lane_launch(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                        const SolveCfg& cfg, LaneArgs A, long long total_obj, long long work,
                        const ExactOut& X, cudaStream_t st) {
  if (cfg.mode == 0 && !X.labels) return cudaErrorInvalidValue;  // lane_all64_launch
  A.nb = (cfg.nmax + 3) / 4;
  if (cfg.mmax > Sh::MP || A.nb > Sh::L) return cudaErrorInvalidConfiguration;
  A.warp_bytes = (int)lane_warp_bytes<Sh>(cfg.mmax, A.nb);
  const long long warps = (work + Sh::PW - 1) / Sh::PW;
  if (X.labels) {
    A.warp_bytes += Sh::NS / 2 * Sh::PS;  // FP64 potentials
    return lane_blocks(k_lane_exact<Sh>, A.warp_bytes, cfg.sms, warps, st, ob, cv, seg_size, K, cfg,
                       A, total_obj, X);
  }
  auto screen = [&](auto kern) {
    return lane_blocks(kern, A.warp_bytes, cfg.sms, warps, st, ob, cv, seg_size, K, cfg, A,
                       total_obj);
  };
  if (A.by_pair)
    return cfg.certify ? screen(k_lane_screen<Sh, true, true>) : screen(k_lane_screen<Sh, false, true>);
  return cfg.certify ? screen(k_lane_screen<Sh, true, false>) : screen(k_lane_screen<Sh, false, false>);
}

// Every pair of the chunk in FP64 throughout, on an FP64 shape.
template <class S8>
cudaError_t lane_all64_launch(const ObjView& ob, const CentView& cv, long long seg_size, int K,
                              const SolveCfg& cfg, LaneArgs A, long long total_obj, long long work,
                              const ExactOut& X, cudaStream_t st) {
  static_assert(S8::TS == 8, "an FP64 shape");
  A.nb = (cfg.nmax + 3) / 4;
  if (cfg.mmax > S8::MP || A.nb > S8::L) return cudaErrorInvalidConfiguration;
  A.warp_bytes = (int)lane_warp_bytes<S8>(cfg.mmax, A.nb);
  return lane_blocks(k_lane_all64<S8>, A.warp_bytes, cfg.sms, (work + S8::PW - 1) / S8::PW, st, ob,
                     cv, seg_size, K, cfg, A, total_obj, X.err);
}

// Pair lists: FP32 with the exact test (shape Sh) or FP64 throughout (S8).
template <class Sh, class S8>
cudaError_t lane_pairs_launch(const ObjView& ob, const CentView& cv, const PairJob& J,
                              const SolveCfg& cfg, cudaStream_t st) {
  static_assert(Sh::TS == 4 && S8::TS == 8 && S8::MP >= Sh::MP && S8::L == Sh::L, "pair shapes");
  const int nb = (cfg.nmax + 3) / 4;
  if (cfg.mmax > Sh::MP || nb > Sh::L) return cudaErrorInvalidConfiguration;
  if (cfg.mode == 0) {
    const int wb = (int)lane_warp_bytes<S8>(cfg.mmax, nb);
    return lane_blocks(k_lane_pairs<S8>, wb, cfg.sms, (J.npairs + S8::PW - 1) / S8::PW, st, ob, cv,
                       J, cfg, nb, wb);
  }
  const long long warps = (J.npairs + Sh::PW - 1) / Sh::PW;
  const int wb = (int)lane_warp_bytes<Sh>(cfg.mmax, nb) + Sh::NS / 2 * Sh::PS;
  return lane_blocks(k_lane_pairs<Sh>, wb, cfg.sms, warps, st, ob, cv, J, cfg, nb, wb);
}

}  // namespace
}  // namespace d2k
