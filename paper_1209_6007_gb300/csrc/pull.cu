// pull.cu - Bc-Reach (Algorithm 2 with the identical-vertex terms of
// Section 3.3.3) on pieces of small BFS depth that do not fit shared memory,
// with every SM of the GPU working on the same BFS level of many source
// batches at a time.
//
// A slab is 256 sources of one piece (consecutive vertices of a BFS order of
// it, so they sit close together and reach most vertices on the same level)
// and one row of state per vertex of the piece.  A wave is as many slabs, of
// any pieces, as give the GPU a million rows or more, and the grid-wide wait
// after every BFS level is paid once per wave.
//
// Per row v of a slab:
//   M[l][v]    256-bit mask per BFS level l: the sources that reach v on l;
//   seen[v]    the sources that have reached v so far;
//   S4[v][256], S8[v][256]  4 or 8 bytes per source: the path count times
//              ident, exact in 32 bits while the level's bound allows (S4),
//              then in 64, then FP64, scaled by a power of two per (level,
//              source) near the end of the double range (S8); replaced in
//              phase 2 by the coefficient of Eq. 3: FP64 in S8, with FP32
//              dependencies a float in S4 while counts are integers, else a
//              float and a binary exponent in S8.  The values of a level are
//              gathered for every shortest-path edge, from more memory than
//              L2 holds: four bytes in place of eight halve that traffic.
//
// Phase 1, level L to L+1: every row v that some source has not reached yet
// reads its neighbours' masks of level L.  The bits of M[L][u] that are not in
// seen[v] are exactly the shortest-path edges u -> v, so one walk of the row
// finds the level and the neighbours whose counts S[u][s] add up to v's.
// Phase 2, levels deepest first: a row v with sources on level l sums the
// coefficients of its neighbours u over M[l+1][u] & M[l][v] and turns its own
// slots into coefficients
//   delta = reach - 1 + sigma * sum,   c = ident (1 + delta) / sigma,
// adding reach[s] ident[s] delta to bc'.
// A row belongs to one warp: nothing is pushed, no atomics but bc's, nothing
// to clear between batches.
//
// How a warp works: the entries of PULL_UNIT rows are walked 32 at a time, one
// per lane whatever row they belong to (rows are short, so a lane per entry
// of one row would idle), and those whose mask meets the row's go into a list
// in shared memory.  Then, row by row, the lanes turn from entries to
// sources: the row's sources are laid side by side by rank, 32 at a time, and
// each lane adds up its own source's values over the row's list.
//
// Rows longer than PULL_LIST entries are cut into at most PULL_LIST items,
// handed out first; each leaves its partial sums with their mask, and the
// last to finish adds them up like a list of neighbours and completes the row.
//
// What bounds it: the latency of the gathers and the instructions around them
// (a third of the issue slots with FP64 dependencies, half with FP32; a fifth of
// HBM bandwidth, a third at 424,000 vertices), with FP64 dependencies also the FP64
// pipe (half busy).  256 sources to a slab: a neighbour is on a
// shortest path for 40 of 256 sources where it is for 14 of 64, so walking,
// listing and ranking cost a third per source; waves of 2^20 rows: waves of
// 2^18 measured 10-15 % slower (the tail of every pass).  Four CTAs per SM: at
// 48 registers (five) it spills and the FP64 cases lose what FP32 gains.
// On one GB300, whole calls: 87,000 vertices, 1.15 M entries, FP32 dependencies,
// every vertex a source 302 ms (1,340 ms with one 64-source batch on the whole
// GPU and pushed counts); 13,690 vertices FP64 14.6 ms (80 ms with 32 sources
// per CTA); 7,009 vertices plain 3.9 ms (21.5 ms with one source per CTA).
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "bc_math.cuh"
#include "common.h"
#include "coop.cuh"

namespace bcs {

constexpr int PULL_THREADS = 256;
constexpr int PULL_WARPS = PULL_THREADS / 32;
constexpr int PULL_CTAS = 4;     // per SM (register budget: 64)
constexpr int PULL_W = 256;      // sources of a slab
constexpr int PULL_WORDS = PULL_W / 32;
constexpr int PULL_LGU = 4;
constexpr int PULL_UNIT = 1 << PULL_LGU;  // rows handed out together
// or fewer (a power of two) while a wave has no more than PULL_SPREAD of these
// per warp: a warp takes its rows one after the other, and few units leave the
// other warps idle (a ring of 1,600 vertices joined to 21 neighbours on either
// side: 9.8 ms in sixteens, 3.0 with 2 per warp, 2.6 with 4 and with 8).  Not
// where most rows are long: those are items, and the units would be empty.
constexpr int PULL_SPREAD = 4;
constexpr int PULL_LIST = 64;    // neighbours a warp keeps; longer rows are cut into items
constexpr int PULL_SHARDS = 8;   // work counters, on separate cache lines
// Rows of a wave: PULL_SLABS slabs of the largest piece, from PULL_ROWS to
// PULL_ROWS_TOP.  Few slabs of a large piece leave a pass uneven (424,000 vertices,
// two slabs a wave 7.65 s, nine 7.26; 87,000 vertices, 12 slabs 298 ms, 24 289),
// many of small ones leave L2 (pieces up to 4,096 vertices, 2^20 rows 51.4 ms,
// 2^21 52.9).
constexpr int64_t PULL_ROWS = 1 << 20, PULL_ROWS_TOP = 1 << 22;
constexpr int PULL_SLABS = 24;
constexpr size_t PULL_BYTES = (size_t)12 << 30;  // the state they may take (one slab at least)
constexpr int64_t PULL_ROWS_MAX = 1 << 30; // rows of a wave are indexed in 32 bits
constexpr int PULL_W_MIN = 32;   // fewest values of a row where memory is short
constexpr int PULL_REC = 600;    // log2 of a level's largest count from which the next level keeps one per source

struct PullSlab {
  int32_t job, base, cnt;  // the job's sources [base, base + cnt)
  int32_t n, row0;         // rows, the first one's index in the wave (a multiple of PULL_UNIT)
  int32_t h0, nh;          // items of long rows, the first one's index in the wave
  int32_t pad;
};

struct PullJobDev {
  int64_t row_off, vtx_off, ord_off, item_off;
};

struct PullItem {
  int32_t v, part, count;  // row, which part of it, parts (item index - part: the row's first item)
  int32_t size;            // row entries per part
};

struct PullChunk {  // part of a piece's rows, for the kernel that lists long rows
  int32_t job, v0, v1;
};

struct PullArgs {
  const PullSlab *slabs;
  const int32_t *wave;  // [nwaves + 1] first slab of each wave
  int32_t nwaves;
  const PullJobDev *jobs;
  const PullItem *items;
  const int64_t *g_row;
  const int32_t *g_col, *g_reach, *g_ident, *order;
  const double *g_init;
  double *bcp;
  double *S8;
  uint32_t *S4;
  uint32_t *M, *seen;       // PULL_WORDS words per row
  int32_t *umap;            // [items + units of a wave] slab of each
  double *ws;               // [slabs][PULL_W] source weights
  unsigned long long *lmax; // nullable: [lcap][slabs][PULL_W] largest count of (level, source)
  unsigned long long *gmax; // [lcap + 1] largest count of a level, 0 when it is empty
  int32_t *ctr;             // [2 lcap][PULL_SHARDS][32]
  double *hpart;            // [items][PULL_W] partial sums
  uint32_t *hmask;          // [items][PULL_WORDS] the sources that have one
  int32_t *hctr;            // [items]
  const int32_t *idmax;     // largest ident
  const double *recip;      // reciprocals of the integers below RECIP_TABLE
  int64_t rows;             // row capacity of a wave
  uint32_t w;               // NARROW: values of a row in S4 and S8, the most sources of a slab
  int64_t slabs_cap;
  int32_t lcap, flg;        // flg: log2 of the most neighbours of a row
  GridBarrier bar;
  int *err;
  unsigned long long *dag_total;
  int sig_cap;
  unsigned long long *trace;  // nullable: (tag, time) pairs of the first waves' passes (BCS_TRACE)
};
constexpr int PULL_TRACE_WAVES = 2, PULL_TRACE_CAP = 1024;

// A listed neighbour: the sources its edge is on a shortest path for, its row
// (of S, or of the partial sums) and the row of the unit it is listed for.
struct __align__(16) PullEnt {
  uint32_t mask[PULL_WORDS];
  uint32_t from;
  int32_t row, pad[2];
};

struct __align__(16) PullWarp {  // a warp's scratch
  PullEnt ent[PULL_LIST];
  uint32_t want[PULL_UNIT][PULL_WORDS], got[PULL_UNIT][PULL_WORDS];
  uint8_t rank[PULL_W];
};

__device__ __forceinline__ void two_sum_add(float &hi, float &lo, float t) {  // Knuth's TwoSum
  const float s = __fadd_rn(hi, t), b = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(t, b)));
  hi = s;
}

// Sums over a row's list of values of type Val.  Path counts: in 32 or 64
// bits from either, FP64 from any (a zero is an entry the source is not in).
template <class T, class V>
struct SumCount {
  using Val = V;
  T x = 0;
  __device__ __forceinline__ void add(V c) { x += (T)c; }
  __device__ __forceinline__ double bits() const { return __longlong_as_double((long long)x); }
};
template <class V>
struct SumCount<double, V> {
  using Val = V;
  double x = 0.0;
  __device__ __forceinline__ void add(V c) { x += c ? i64_to_f64_pos((long long)c) : 0.0; }
  __device__ __forceinline__ double bits() const { return x; }
};
struct SumF64 {
  using Val = double;
  double x = 0.0;
  __device__ __forceinline__ void add(double c) { x += c; }
  __device__ __forceinline__ double bits() const { return x; }
};
using SumI64 = SumCount<long long, long long>;
// FP32 coefficients as hi + lo.
struct SumFloat {
  using Val = float;
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float c) { two_sum_add(hi, lo, c); }
  __device__ __forceinline__ double bits() const { return __hiloint2double(__float_as_int(lo), __float_as_int(hi)); }
};
// FP32 coefficients with a binary exponent, taken relative to the exponent ex
// of the row's own count.
struct SumScaled {
  using Val = double;
  float hi = 0.0f, lo = 0.0f;
  int ex = 0;
  __device__ __forceinline__ void add(double c) {
    const int d = max(ex - __double2hiint(c), -127);  // 2^-127 and below: 0
    two_sum_add(hi, lo, __int_as_float(__double2loint(c)) * __int_as_float((127 + d) << 23));
  }
  __device__ __forceinline__ double bits() const { return __hiloint2double(__float_as_int(lo), __float_as_int(hi)); }
};
struct SumPairs {  // partial sums of either
  using Val = double;
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(double c) {
    two_sum_add(hi, lo, __int_as_float(__double2loint(c)));
    lo += __int_as_float(__double2hiint(c));
  }
  __device__ __forceinline__ double bits() const { return __hiloint2double(__float_as_int(lo), __float_as_int(hi)); }
};

// Add up the values of source src (< 0: none) of the list entries [i, i + c), w
// values to a row of V.
// Every sum takes zeros for the entries the source is not in, so that the
// loads of four entries are in flight together and no lane branches.
template <class Sum>
__device__ __forceinline__ void pull_sum(Sum &a, const PullWarp &W, int i, int c, const void *V, int src, uint32_t w) {
  using T = typename Sum::Val;
  const uint32_t bit = src < 0 ? 0u : 1u << (src & 31);
  const uint32_t *m = &W.ent[i].mask[src < 0 ? 0 : src >> 5];
  const PullEnt *e = W.ent + i;
  const T *const v = (const T *)V + max(src, 0);
  constexpr int STEP = sizeof(PullEnt) / 4;
  for (; c >= 4; c -= 4, e += 4, m += 4 * STEP) {
    T x[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      x[q] = 0;
      if (m[q * STEP] & bit) x[q] = v[(size_t)e[q].from * w];
    }
#pragma unroll
    for (int q = 0; q < 4; q++) a.add(x[q]);
  }
  if (c & 2) {
    T x0 = 0, x1 = 0;
    if (m[0] & bit) x0 = v[(size_t)e[0].from * w];
    if (m[STEP] & bit) x1 = v[(size_t)e[1].from * w];
    a.add(x0);
    a.add(x1);
    e += 2;
    m += 2 * STEP;
  }
  if (c & 1) {
    T x0 = 0;
    if (m[0] & bit) x0 = v[(size_t)e[0].from * w];
    a.add(x0);
  }
}

// Units [returned, + take) of a pass, or -1 when none are left
// (warp-collective).  Shard h owns the grabs h, h + PULL_SHARDS, ...; a warp
// stays on its shard until it is used up, then moves to the next one with
// work left (every failed claim follows another warp's successful one).
__device__ __forceinline__ int pull_grab(int32_t *ctr, int total, int take, int &shard, int lane) {
  const int grabs = (total + take - 1) / take;
  for (;;) {
    int g = 0;
    if (lane == 0) {
      int32_t *c = ctr + shard * 32;
      const int lim = (grabs - shard + PULL_SHARDS - 1) / PULL_SHARDS;
      g = *(volatile int32_t *)c < lim ? atomicAdd(c, 1) : lim;
    }
    g = __shfl_sync(0xffffffffu, g, 0) * PULL_SHARDS + shard;
    if (g < grabs) return g * take;
    bool left = false;
    if (lane < PULL_SHARDS)
      left = *(volatile int32_t *)(ctr + lane * 32) < (grabs - lane + PULL_SHARDS - 1) / PULL_SHARDS;
    const unsigned bm = __ballot_sync(0xffffffffu, left);
    if (!bm) return -1;
    const unsigned rot = (bm | (bm << PULL_SHARDS)) >> (shard + 1);
    shard = (shard + __ffs(rot)) % PULL_SHARDS;
  }
}

// What a warp works on: the rows of a unit (lane k < PULL_UNIT holds row k)
// or one item of a long row (as a unit of that row alone).
struct PullUnit {
  int32_t v0;           // the first row's vertex
  uint32_t r0;          // and its index in the wave
  uint32_t row0;        // the slab's first row
  int64_t vtx_off;      // the piece's first vertex
  const int32_t *col;   // the first row's entries
  // per lane: entries of the rows up to and with row k that are walked, and
  // what to add to a walked entry's number to find it in col
  uint32_t incl, shift;
  unsigned rows;        // rows with sources to walk for, as bits
  unsigned own;         // rows of the unit, as bits (long rows are not)
  int j;                // slab of the wave
};

// Walk the unit's entries and list those whose masks meet the rows' (in
// W.want), up to PULL_LIST at a time, then take(row, first, count) for each
// row that has any (all of a row's entries in one list).
template <class Take>
__device__ __forceinline__ void pull_walk(PullWarp &W, const PullUnit &U, const uint32_t *M, int lane, Take take) {
  const uint32_t T = __shfl_sync(0xffffffffu, U.incl, PULL_UNIT - 1);
  const unsigned below = (1u << lane) - 1u;
  for (uint32_t fa = 0; fa < T;) {
    // whole rows of at most PULL_LIST entries together
    const unsigned fits = __ballot_sync(0xffffffffu, lane < PULL_UNIT && U.incl <= fa + PULL_LIST);
    const uint32_t fb = __shfl_sync(0xffffffffu, U.incl, 31 - __clz(fits));
    int cnt = 0;
    __syncwarp();  // the list's last readers are done
    for (uint32_t f0 = fa; f0 < fb; f0 += 32) {
      const uint32_t f = f0 + lane;
      int k = 0;  // rows that end at or before entry f
#pragma unroll
      for (int s = PULL_UNIT / 2; s > 0; s >>= 1)
        if (__shfl_sync(0xffffffffu, U.incl, k + s - 1) <= f) k += s;
      const uint32_t sh = __shfl_sync(0xffffffffu, U.shift, k);
      uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
      uint32_t r = 0u;
      if (f < fb) {
        r = U.row0 + (uint32_t)__ldg(U.col + (uint32_t)(f + sh));
        const uint4 *const m = (const uint4 *)(M + (size_t)r * PULL_WORDS), *const w = (const uint4 *)W.want[k];
        a = m[0], b = m[1];
        const uint4 wa = w[0], wb = w[1];
        a.x &= wa.x, a.y &= wa.y, a.z &= wa.z, a.w &= wa.w;
        b.x &= wb.x, b.y &= wb.y, b.z &= wb.z, b.w &= wb.w;
      }
      const bool hit = (a.x | a.y | a.z | a.w | b.x | b.y | b.z | b.w) != 0u;
      const unsigned nz = __ballot_sync(0xffffffffu, hit);
      if (hit) {
        PullEnt &e = W.ent[cnt + __popc(nz & below)];
        *(uint4 *)&e.mask[0] = a;
        *(uint4 *)&e.mask[4] = b;
        e.from = r;
        e.row = k;
      }
      cnt += __popc(nz);
    }
    __syncwarp();
    for (int i = 0; i < cnt;) {
      const int row = W.ent[i].row;
      int c = 0;
      for (;;) {  // the entries of the same row
        const int at = i + c + lane;
        const unsigned same = __ballot_sync(0xffffffffu, at < cnt && W.ent[min(at, PULL_LIST - 1)].row == row);
        c += same == 0xffffffffu ? 32 : __ffs(~same) - 1;
        if (same != 0xffffffffu) break;
      }
      take(row, i, c);
      i += c;
    }
    fa = fb;
  }
}

// The union of the masks of list entries [i, i + c): word (lane & 7).
__device__ __forceinline__ uint32_t pull_union(const PullWarp &W, int i, int c, int lane) {
  uint32_t g = 0u;
  for (int h = lane >> 3; h < c; h += 4) g |= W.ent[i + h].mask[lane & 7];
  g |= __shfl_xor_sync(0xffffffffu, g, 8);
  return g | __shfl_xor_sync(0xffffffffu, g, 16);
}

// Lay the sources of a mask (word (lane & 7) in each lane) side by side in
// W.rank; returns how many there are.
__device__ __forceinline__ int pull_rank(PullWarp &W, uint32_t g, int lane) {
  const unsigned below = (1u << lane) - 1u;
  int n = 0;
  __syncwarp();  // the last mask's readers are done
#pragma unroll
  for (int w = 0; w < PULL_WORDS; w++) {
    const uint32_t m = __shfl_sync(0xffffffffu, g, w);
    if ((m >> lane) & 1u) W.rank[n + __popc(m & below)] = (uint8_t)(32 * w + lane);
    n += __popc(m);
  }
  __syncwarp();
  return n;
}

// log2 (floor) of a level's largest count
__device__ __forceinline__ int pull_lg(unsigned long long g, bool is_int) {
  return is_int ? 63 - __clzll((long long)g) : (int)((g >> 52) & 0x7ff) - 1023;
}

// NARROW: rows of A.w values, for pieces whose state does not fit with PULL_W (as
// a number known to the compiler only there: it costs the other 1 to 3 %).
template <bool REACH, bool IDENT, bool FP32, bool NARROW>
__global__ void __launch_bounds__(PULL_THREADS, PULL_CTAS) k_bcreach_pull(const __grid_constant__ PullArgs A) {
  using Real = typename std::conditional<FP32, float, double>::type;
  __shared__ PullWarp s_warp[PULL_WARPS];
  __shared__ int s_lgu;  // log2 of a unit's rows (in a register it costs the FP32 case 2.7 %)
  const int lane = threadIdx.x & 31;
  PullWarp &W = s_warp[threadIdx.x >> 5];
  const int64_t gtid = (int64_t)blockIdx.x * PULL_THREADS + threadIdx.x;
  const int64_t nthreads = (int64_t)gridDim.x * PULL_THREADS;
  const int nwarps = (int)(nthreads >> 5);
  const uint32_t SW = NARROW ? A.w : (uint32_t)PULL_W;
  double *const S8 = A.S8;
  uint32_t *const S4 = A.S4;
  const int idl = IDENT ? 32 - __clz(max(*A.idmax, 1) - 1) : 0;  // ceil(log2)
  const int grow = A.flg + idl;  // a level's counts are below 2^grow times the largest of the level before
  const int t_hi = 1000 - grow, t_lo = t_hi - 400;
  unsigned long long dag = 0;
  int tpos = 0;
  auto mark = [&](int w, unsigned tag) {  // the end of a pass
    if (A.trace && w < PULL_TRACE_WAVES && gtid == 0 && tpos < PULL_TRACE_CAP) {
      unsigned long long t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      A.trace[2 * tpos] = ((unsigned long long)w << 32) | tag;
      A.trace[2 * tpos + 1] = t;
      tpos++;
    }
  };
  // whether the largest count of (level, source) is on record: the level
  // before it is FP64 and past 2^PULL_REC
  auto recorded = [&](int l, int lint) {
    return A.lmax && l >= 1 && l - 1 >= lint && pull_lg(__ldcg(A.gmax + l - 1), false) > PULL_REC;
  };
  // the power of two to drop from the counts of (level, source) when they are summed
  auto drop = [&](int l, int j, int src) {
    const int k = pull_lg(__ldcg(A.lmax + ((size_t)l * A.slabs_cap + j) * PULL_W + src), false) + 1 + grow;
    return k > t_hi ? k - t_lo : 0;
  };
  for (int w = 0; w < A.nwaves; w++) {
    const int s0 = A.wave[w], J = A.wave[w + 1] - s0;
    const PullSlab *const slabs = A.slabs + s0;
    const int nu = (slabs[J - 1].row0 + slabs[J - 1].n + PULL_UNIT - 1) / PULL_UNIT;
    const int nh = slabs[J - 1].h0 + slabs[J - 1].nh;
    int total;  // items first
    {
      int lgu = PULL_LGU;
      while (lgu > 0 && nh < nu * (PULL_UNIT / 2) && nh + (nu << (PULL_LGU + 1 - lgu)) <= PULL_SPREAD * nwarps) lgu--;
      if (threadIdx.x == 0) s_lgu = lgu;  // read after the waits below
      total = nh + (nu << (PULL_LGU - lgu));
    }
    const int take = max(1, min(8, nu / (nwarps * 8)));
    // ---------------------------------------------- the wave's tables
    for (int64_t i = gtid; i < nh + nu; i += nthreads) {
      const bool item = i < nh;
      const int key = item ? (int)i : (int)(i - nh) * PULL_UNIT;
      int lo = 0, hi = J;  // the last slab that starts at or before the key
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if ((item ? slabs[mid].h0 : slabs[mid].row0) <= key) lo = mid;
        else hi = mid;
      }
      A.umap[i] = lo;
      if (item) A.hctr[i] = 0;
    }
    for (int64_t i = gtid; i < 2 * A.lcap * PULL_SHARDS; i += nthreads) A.ctr[i * 32] = 0;
    for (int64_t i = gtid; i <= A.lcap; i += nthreads) A.gmax[i] = i == 0 ? 1ull : 0ull;
    if (A.lmax)
      for (int64_t i = gtid; i < (int64_t)A.lcap * A.slabs_cap * PULL_W; i += nthreads) A.lmax[i] = 0ull;
    mark(w, 0xE000u);
    if (!grid_wait(A.bar)) return;
    // ---------------------------------------------- level 0: the sources
    for (int64_t i = gtid; i < (int64_t)nu * PULL_UNIT * PULL_WORDS; i += nthreads) {
      const int cnt = slabs[A.umap[nh + i / (PULL_UNIT * PULL_WORDS)]].cnt - 32 * (int)(i % PULL_WORDS);
      A.M[i] = 0u;
      A.seen[i] = cnt >= 32 ? 0u : cnt <= 0 ? 0xffffffffu : 0xffffffffu << cnt;
    }
    if (!grid_wait(A.bar)) return;
    for (int64_t i = gtid; i < (int64_t)J * PULL_W; i += nthreads) {
      const PullSlab sl = slabs[i / PULL_W];
      const int k = (int)(i % PULL_W);
      double wsv = 0.0;
      if (k < sl.cnt) {
        const PullJobDev jb = A.jobs[sl.job];
        const int32_t s = __ldg(A.order + jb.ord_off + sl.base + k);
        const size_t r = (size_t)sl.row0 + s;
        atomicOr(A.M + r * PULL_WORDS + (k >> 5), 1u << (k & 31));  // a repeated source is two bits of one row
        atomicOr(A.seen + r * PULL_WORDS + (k >> 5), 1u << (k & 31));
        S4[r * SW + k] = 1u;
        if (REACH || IDENT)
          wsv = (REACH ? (A.g_init ? __ldg(A.g_init + jb.vtx_off + s) + 1.0 : (double)__ldg(A.g_reach + jb.vtx_off + s))
                       : 1.0) *
                (IDENT ? (double)__ldg(A.g_ident + jb.vtx_off + s) : 1.0);
      }
      if (REACH || IDENT) A.ws[i] = wsv;
    }
    if (!grid_wait(A.bar)) return;
    mark(w, 0xF000u);
    // Unit u of a pass; its rows' masks (of `masks`, complemented with flip)
    // in W.want.  Rows without a source, and long rows, are not walked.
    auto load_unit = [&](int u, PullUnit &U, PullItem &it, bool walk, const uint32_t *masks, uint32_t flip) {
      const int lgu = *(volatile int *)&s_lgu;
      const uint32_t r0 = (uint32_t)(u - nh) << lgu;
      U.j = A.umap[u < nh ? (uint32_t)u : nh + r0 / PULL_UNIT];
      const PullSlab sl = slabs[U.j];
      const PullJobDev jb = A.jobs[sl.job];
      U.row0 = (uint32_t)sl.row0;
      U.vtx_off = jb.vtx_off;
      const int64_t *const row = A.g_row + jb.row_off;
      int64_t b = 0, e = 0;
      int rows = 1;
      if (u >= nh) {
        U.r0 = r0;
        U.v0 = (int32_t)(U.r0 - U.row0);
        rows = min(1 << lgu, sl.n - U.v0);  // none past the slab's last row
        if (lane <= rows) b = __ldg(row + U.v0 + lane);
        e = __shfl_down_sync(0xffffffffu, b, 1);
        U.own = __ballot_sync(0xffffffffu, lane < rows && e - b <= PULL_LIST);
        it.count = 0;
      } else {
        it = A.items[jb.item_off + (u - sl.h0)];
        U.v0 = it.v;
        U.r0 = U.row0 + (uint32_t)it.v;
        U.own = 1u;
        b = __ldg(row + it.v) + (int64_t)it.part * it.size;
        e = min(__ldg(row + it.v + 1), b + it.size);
      }
      // 16 bytes of the rows' masks per lane: row lane / 2
      static_assert(PULL_UNIT * PULL_WORDS == 128, "a unit's masks are 16 bytes per lane");
      uint4 m = make_uint4(0u, 0u, 0u, 0u);
      if ((lane >> 1) < rows) {
        m = ((const uint4 *)(masks + (size_t)U.r0 * PULL_WORDS))[lane];
        m.x ^= flip, m.y ^= flip, m.z ^= flip, m.w ^= flip;
      }
      __syncwarp();  // the last unit's readers are done
      ((uint4 *)W.want)[lane] = m;
      unsigned any = __ballot_sync(0xffffffffu, (m.x | m.y | m.z | m.w) != 0u);
      any |= any >> 1;  // even bits: rows
      unsigned act = any & 0x55555555u;
      act = (act | (act >> 1)) & 0x33333333u;
      act = (act | (act >> 2)) & 0x0f0f0f0fu;
      act = (act | (act >> 4)) & 0x00ff00ffu;
      act = (act | (act >> 8)) & 0x0000ffffu;
      U.rows = act & U.own;
      const int64_t b0 = __shfl_sync(0xffffffffu, b, 0);
      U.col = A.g_col + b0;
      const uint32_t deg = (walk && ((U.rows >> lane) & 1u)) ? (uint32_t)(e - b) : 0u;
      uint32_t incl = deg;
#pragma unroll
      for (int o = 1; o < PULL_UNIT; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      U.incl = incl;
      U.shift = (uint32_t)(b - b0) - (incl - deg);
      __syncwarp();
    };
    // A long row's partial sums.  An item of more than PULL_LIST entries adds
    // several lists into its own; `have` (word lane & 7) the sources it holds.
    auto leave = [&](int u, int src, uint32_t have, auto sum, auto merge) {
      double *const p = A.hpart + (size_t)u * PULL_W + src;
      const bool old = (__shfl_sync(0xffffffffu, have, src < 0 ? 0 : src >> 5) >> (src & 31)) & 1u;
      if (src >= 0) {
        if (old) {
          merge.add(*(const typename decltype(merge)::Val *)p);
          const double more = sum.bits();
          merge.add(*(const typename decltype(merge)::Val *)&more);
          *p = merge.bits();
        } else {
          *p = sum.bits();
        }
      }
    };
    // whether this item is the row's last to finish (its sums are in scratch)
    auto last_of = [&](int u, const PullItem &it, uint32_t have) {
      if (lane < PULL_WORDS) A.hmask[(size_t)u * PULL_WORDS + lane] = have;
      __threadfence();
      __syncwarp();
      int last = 0;
      if (lane == 0) last = atomicAdd(A.hctr + (u - it.part), 1) == it.count - 1;
      last = __shfl_sync(0xffffffffu, last, 0);
      if (last) {
        __threadfence();
        if (lane == 0) A.hctr[u - it.part] = 0;
      }
      return last != 0;
    };
    // the row's items as a list: their masks and scratch rows
    auto list_items = [&](int u, const PullItem &it) {
      __syncwarp();
      for (int c = lane; c < it.count; c += 32) {
        const int f = u - it.part + c;
        const uint4 *const m = (const uint4 *)(A.hmask + (size_t)f * PULL_WORDS);
        PullEnt &e = W.ent[c];
        *(uint4 *)&e.mask[0] = __ldcg(m);
        *(uint4 *)&e.mask[4] = __ldcg(m + 1);
        e.from = (uint32_t)f;
        e.row = 0;
      }
      __syncwarp();
    };
    // ---------------------------------------------- phase 1
    int L = 0, l64 = A.lcap + 1, lint = A.lcap + 1;  // the first level not in 32 bits, the first FP64 one
    for (;;) {
      const unsigned long long gm = __ldcg(A.gmax + L);
      if (gm == 0ull) break;
      if (L + 2 >= A.lcap) {
        if (gtid == 0) atomicOr(A.err, ERR_DEPTH);
        return;
      }
      const bool kind = L < lint;
      const int lgm = pull_lg(gm, kind);
      if (lgm >= A.sig_cap && gtid == 0) atomicOr(A.err, ERR_OVERFLOW);
      // level L+1's counts stay integers, in 32 or 64 bits, while the largest
      // of them, times ident, is sure to fit
      const bool kind_next = kind && lgm + 1 + grow < 62, short_cur = L < l64;
      const bool short_next = short_cur && lgm + 1 + grow <= 32;
      if (kind && !kind_next) lint = L + 1;
      if (short_cur && !short_next) l64 = L + 1;
      const bool scaled = recorded(L, lint), rec_next = !kind_next && recorded(L + 1, lint);
      const uint32_t *const Mc = A.M + (size_t)L * A.rows * PULL_WORDS;
      uint32_t *const Mn = A.M + (size_t)(L + 1) * A.rows * PULL_WORDS;
      unsigned long long wmax = 0ull;
      int shard = (int)((gtid >> 5) % PULL_SHARDS);
      for (;;) {
        const int u0 = pull_grab(A.ctr + (size_t)(2 * L) * PULL_SHARDS * 32, total, take, shard, lane);
        if (u0 < 0) break;
        for (int u = u0; u < min(u0 + take, total); u++) {
          PullUnit U;
          PullItem it;
          load_unit(u, U, it, true, A.seen, 0xffffffffu);
          const bool item = it.count > 0;
          // the count of (row k, src) is complete: store it (id: the row's ident)
          auto ident = [&](int k) { return IDENT ? __ldg(A.g_ident + U.vtx_off + U.v0 + k) : 1; };
          auto store = [&](size_t at, int src, double bits, int id) {
            if (src < 0) return;
            unsigned long long x = (unsigned long long)__double_as_longlong(bits);
            if (short_next) {
              const uint32_t y = IDENT ? (uint32_t)x * (uint32_t)id : (uint32_t)x;
              S4[at + src] = y;
              wmax = max(wmax, (unsigned long long)y);
              return;
            }
            if (kind_next) {
              if (IDENT && id != 1) x *= (unsigned long long)id;
            } else if (scaled || (IDENT && id != 1)) {
              double d = bits;
              if (scaled) d *= pow2_int(-drop(L, U.j, src));
              if (IDENT) d *= (double)id;
              x = (unsigned long long)__double_as_longlong(d);
            }
            ((unsigned long long *)S8)[at + src] = x;
            wmax = max(wmax, x);  // positive doubles order like their bits
            if (rec_next) atomicMax(A.lmax + ((size_t)(L + 1) * A.slabs_cap + U.j) * PULL_W + src, x);
          };
          // the sums of the row's list for src, in the types of the two levels
          auto counts = [&](int i, int c, int src, auto done) {
            auto sum = [&](auto a, const void *V) {
              pull_sum(a, W, i, c, V, src, SW);
              done(a);
            };
            if (short_next) sum(SumCount<uint32_t, uint32_t>(), S4);
            else if (kind_next && short_cur) sum(SumCount<unsigned long long, uint32_t>(), S4);
            else if (kind_next) sum(SumI64(), S8);
            else if (short_cur) sum(SumCount<double, uint32_t>(), S4);
            else if (kind) sum(SumCount<double, long long>(), S8);
            else sum(SumF64(), S8);
          };
          if (!item) {
            ((uint4 *)W.got)[lane] = make_uint4(0u, 0u, 0u, 0u);
            pull_walk(W, U, Mc, lane, [&](int k, int i, int c) {
              const uint32_t g = pull_union(W, i, c, lane);
              if (lane < PULL_WORDS) W.got[k][lane] = g;
              const int n = pull_rank(W, g, lane), id = ident(k);
              const size_t at = (size_t)(U.r0 + k) * SW;
              for (int t = 0; t < n; t += 32) {
                const int src = t + lane < n ? (int)W.rank[t + lane] : -1;
                counts(i, c, src, [&](const auto &a) { store(at, src, a.bits(), id); });
              }
            });
            __syncwarp();
            if ((U.own >> (lane >> 1)) & 1u) {
              const uint4 g = ((const uint4 *)W.got)[lane];
              const size_t at = (size_t)U.r0 * (PULL_WORDS / 4) + lane;
              ((uint4 *)Mn)[at] = g;
              if (g.x | g.y | g.z | g.w) {
                const uint4 q = ((const uint4 *)W.want)[lane];
                ((uint4 *)A.seen)[at] = make_uint4(~q.x | g.x, ~q.y | g.y, ~q.z | g.z, ~q.w | g.w);
              }
            }
            continue;
          }
          if (!U.rows) {  // every source has reached the row
            if (it.part == 0 && lane < PULL_WORDS) Mn[(size_t)U.r0 * PULL_WORDS + lane] = 0u;
            continue;
          }
          uint32_t have = 0u;
          const uint32_t f0 = __shfl_sync(0xffffffffu, U.incl, 0);
          PullUnit part = U;
          for (uint32_t f = 0; f < f0; f += PULL_LIST) {  // a list at a time
            part.col = U.col + f;
            part.incl = min(f0 - f, (uint32_t)PULL_LIST);
            part.shift = 0u;
            pull_walk(W, part, Mc, lane, [&](int, int i, int c) {
              const uint32_t g = pull_union(W, i, c, lane);
              const int n = pull_rank(W, g, lane);
              for (int t = 0; t < n; t += 32) {
                const int src = t + lane < n ? (int)W.rank[t + lane] : -1;
                counts(i, c, src, [&](const auto &a) {
                  if (kind_next) leave(u, src, have, a, SumI64());
                  else leave(u, src, have, a, SumF64());
                });
              }
              have |= g;
            });
          }
          if (!last_of(u, it, have)) continue;
          list_items(u, it);
          const uint32_t g = pull_union(W, 0, it.count, lane);
          const int n = pull_rank(W, g, lane), id = ident(0);
          const size_t at = (size_t)U.r0 * SW;
          for (int t = 0; t < n; t += 32) {
            const int src = t + lane < n ? (int)W.rank[t + lane] : -1;
            if (kind_next) {
              SumI64 a;
              pull_sum(a, W, 0, it.count, A.hpart, src, PULL_W);
              store(at, src, a.bits(), id);
            } else {
              SumF64 a;
              pull_sum(a, W, 0, it.count, A.hpart, src, PULL_W);
              store(at, src, a.bits(), id);
            }
          }
          if (lane < PULL_WORDS) {
            Mn[(size_t)U.r0 * PULL_WORDS + lane] = g;
            if (g) A.seen[(size_t)U.r0 * PULL_WORDS + lane] = ~W.want[0][lane] | g;
          }
        }
      }
      // the level's largest count, once per warp
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) wmax = max(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
      if (lane == 0 && wmax > __ldcg(A.gmax + L + 1)) atomicMax(A.gmax + L + 1, wmax);
      if (!grid_wait(A.bar)) return;
      mark(w, 0x1000u | (unsigned)L);
      L++;
    }
    const int Lmax = L - 1;
    // ---------------------------------------------- phase 2
    for (int l = Lmax; l >= 1; l--) {
      const bool kind = l < lint, kind_next = l + 1 < lint, is_short = l < l64, scaled = recorded(l, lint);
      const uint32_t *const Ml = A.M + (size_t)l * A.rows * PULL_WORDS, *const Ms = Ml + (size_t)A.rows * PULL_WORDS;
      int shard = (int)((gtid >> 5) % PULL_SHARDS);
      for (;;) {
        const int u0 = pull_grab(A.ctr + (size_t)(2 * l + 1) * PULL_SHARDS * 32, total, take, shard, lane);
        if (u0 < 0) break;
        for (int u = u0; u < min(u0 + take, total); u++) {
          PullUnit U;
          PullItem it;
          load_unit(u, U, it, l < Lmax, Ml, 0u);
          if (!U.rows) continue;
          const bool item = it.count > 0;
          // what a row's sources share
          struct Row {
            size_t at;    // first slot
            int id;
            Real init;    // reach - 1
          };
          auto row_of = [&](int k) {
            const int64_t v = U.vtx_off + U.v0 + k;
            return Row{(size_t)(U.r0 + k) * SW, IDENT ? __ldg(A.g_ident + v) : 1,
                       REACH ? (A.g_init ? (Real)__ldg(A.g_init + v) : (Real)(__ldg(A.g_reach + v) - 1)) : (Real)0};
          };
          // an integer count (exact: the stored value is a multiple of ident)
          auto count = [&](const Row &r, int src) -> long long {
            if (is_short) {
              uint32_t g = S4[r.at + src];
              if (IDENT && r.id != 1) g /= (uint32_t)r.id;
              return g;
            }
            long long g = ((const long long *)S8)[r.at + src];
            if (IDENT && r.id != 1) g /= r.id;
            return g;
          };
          // a count as binary exponent and mantissa (FP32)
          auto split = [&](const Row &r, int src, int &e, float &m) {
            if (kind) {
              split_pow2_i64(count(r, src), e, m);
            } else {
              const double st = S8[r.at + src];
              split_pow2(IDENT && r.id != 1 ? st / (double)r.id : st, e, m);
            }
          };
          auto exponent = [&](const Row &r, int src) {
            int e = 0;
            float m;
            if (src >= 0) {
              split(r, src, e, m);
              if (scaled) e -= drop(l, U.j, src);
            }
            return e;
          };
          // delta and coefficient of one source of a row; returns its bc' term
          auto settle64 = [&](const Row &r, int src, double x) -> double {
            if (src < 0) return 0.0;
            double sg;
            int idx = 0;  // the count, if it is an integer in the table of reciprocals
            if (kind) {
              const long long g = count(r, src);
              idx = g < RECIP_TABLE ? (int)g : 0;
              sg = i64_to_f64_pos(g);
            } else {
              sg = S8[r.at + src];
              if (IDENT && r.id != 1) sg /= (double)r.id;
              if (scaled) x *= pow2_int(-drop(l, U.j, src));
            }
            const double d = REACH ? fma(sg, x, (double)r.init) : sg * x;
            if (l > 1) {  // the sources' own dependencies are not needed
              const double rc = idx ? __ldg(A.recip + idx) : recip_pos(sg);
              const double kr = IDENT && r.id != 1 ? (double)r.id * rc : rc;
              S8[r.at + src] = fma(d, kr, kr);
            }
            return REACH || IDENT ? A.ws[(size_t)U.j * PULL_W + src] * d : d;
          };
          // (the term and its sum are FP64 whatever the dependencies: 1.3 % of the
          // FP32 case's time, and exact where 24 bits are not)
          auto settle32 = [&](const Row &r, int src, float hi, float lo, double sum) -> double {
            if (src < 0) return sum;
            const float init = r.init, kv = (float)r.id;
            float m, d;
            int e = 0;
            if (kind && kind_next) {
              m = is_short ? __uint2float_rn((uint32_t)count(r, src)) : __ll2float_rn(count(r, src));
            } else {
              split(r, src, e, m);  // the sum is relative to the count's exponent
            }
            d = fmaf(m, hi, fmaf(m, lo, init));
            if (l > 1) {
              if (kind) {
                if (!kind_next) m = __ll2float_rn(count(r, src));
                ((float *)S4)[r.at + src] = fmaf(kv, d, kv) / m;
              } else {
                S8[r.at + src] = __hiloint2double(e, __float_as_int(fmaf(kv, d, kv) / m));
              }
            }
            return REACH || IDENT ? fma(A.ws[(size_t)U.j * PULL_W + src], (double)d, sum) : sum + (double)d;
          };
          auto add_bc = [&](int k, double c) {  // bc' of row k's vertex
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
            if (lane == 0) atomicAdd(A.bcp + U.vtx_off + U.v0 + k, c);
          };
          // row k with list entries [i, i + c): neighbours, or the items of a long row
          auto row_done = [&](int k, int i, int c, bool items) {
            const int n = pull_rank(W, W.want[k][lane & 7], lane);
            const Row r = row_of(k);
            if constexpr (FP32) {
              double sum = 0.0;
              for (int t = 0; t < n; t += 32) {
                const int src = t + lane < n ? (int)W.rank[t + lane] : -1;
                float hi, lo;
                if (items) {
                  SumPairs a;
                  pull_sum(a, W, i, c, A.hpart, src, PULL_W);
                  hi = a.hi, lo = a.lo;
                } else if (kind_next) {
                  SumFloat a;
                  pull_sum(a, W, i, c, S4, src, SW);
                  hi = a.hi, lo = a.lo;
                } else {
                  SumScaled a;
                  a.ex = exponent(r, src);
                  pull_sum(a, W, i, c, S8, src, SW);
                  hi = a.hi, lo = a.lo;
                }
                sum = settle32(r, src, hi, lo, sum);
              }
              add_bc(k, sum);
            } else {
              double sum = 0.0;
              for (int t = 0; t < n; t += 32) {
                const int src = t + lane < n ? (int)W.rank[t + lane] : -1;
                SumF64 a;
                pull_sum(a, W, i, c, items ? A.hpart : S8, src, items ? PULL_W : SW);
                sum += settle64(r, src, a.x);
              }
              add_bc(k, sum);
            }
          };
          auto count_dag = [&](int i, int c) {
            unsigned n = 0;
            for (int h = lane >> 3; h < c; h += 4) n += __popc(W.ent[i + h].mask[lane & 7]);
            dag += n;
          };
          if (!item) {
            unsigned left = U.rows;
            pull_walk(W, U, Ms, lane, [&](int k, int i, int c) {
              count_dag(i, c);
              row_done(k, i, c, false);
              left &= ~(1u << k);
            });
            for (; left; left &= left - 1u) row_done(__ffs(left) - 1, 0, 0, false);  // no successors
            continue;
          }
          uint32_t have = 0u;
          const uint32_t f0 = __shfl_sync(0xffffffffu, U.incl, 0);
          PullUnit part = U;
          const Row r = row_of(0);
          for (uint32_t f = 0; f < f0; f += PULL_LIST) {
            part.col = U.col + f;
            part.incl = min(f0 - f, (uint32_t)PULL_LIST);
            part.shift = 0u;
            pull_walk(W, part, Ms, lane, [&](int, int i, int c) {
              count_dag(i, c);
              const uint32_t g = pull_union(W, i, c, lane);
              const int n = pull_rank(W, g, lane);
              for (int t = 0; t < n; t += 32) {
                const int src = t + lane < n ? (int)W.rank[t + lane] : -1;
                if constexpr (FP32) {
                  if (kind_next) {
                    SumFloat a;
                    pull_sum(a, W, i, c, S4, src, SW);
                    leave(u, src, have, a, SumPairs());
                  } else {
                    SumScaled a;
                    a.ex = exponent(r, src);
                    pull_sum(a, W, i, c, S8, src, SW);
                    leave(u, src, have, a, SumPairs());
                  }
                } else {
                  SumF64 a;
                  pull_sum(a, W, i, c, S8, src, SW);
                  leave(u, src, have, a, SumF64());
                }
              }
              have |= g;
            });
          }
          if (!last_of(u, it, have)) continue;
          list_items(u, it);
          row_done(0, 0, it.count, true);
        }
      }
      if (!grid_wait(A.bar)) return;
      mark(w, 0x2000u | (unsigned)l);
    }
    if (Lmax < 1 && !grid_wait(A.bar)) return;  // the next wave's tables overwrite what the last pass reads
  }
  for (int o = 16; o > 0; o >>= 1) dag += __shfl_xor_sync(0xffffffffu, dag, o);
  if (lane == 0 && dag) atomicAdd(A.dag_total, dag);
}

// ------------------------------------------------------------ preparation
// Items of the rows longer than PULL_LIST: counted per job, then (fill)
// listed in the job's range of the table.
__global__ void k_pull_items(const PullChunk *__restrict__ chunks, const CompDesc *__restrict__ comps,
                             const int32_t *__restrict__ job_comp, const int64_t *__restrict__ g_row, int32_t *cnt,
                             const int64_t *__restrict__ item_off, PullItem *items, bool fill) {
  const PullChunk c = chunks[blockIdx.x];
  const int64_t *row = g_row + comps[job_comp[c.job]].row_off;
  for (int32_t v = c.v0 + threadIdx.x; v < c.v1; v += blockDim.x) {
    const int64_t d = row[v + 1] - row[v];
    if (d <= PULL_LIST) continue;
    // parts of a multiple of PULL_LIST entries, at most PULL_LIST of them
    const int64_t size = PULL_LIST * ((d + (int64_t)PULL_LIST * PULL_LIST - 1) / ((int64_t)PULL_LIST * PULL_LIST));
    const int parts = (int)((d + size - 1) / size);
    const int at = atomicAdd(cnt + c.job, parts);
    if (fill)
      for (int k = 0; k < parts; k++) items[item_off[c.job] + at + k] = PullItem{v, k, parts, (int32_t)size};
  }
}

__global__ void k_pull_idmax(int64_t n, const int32_t *__restrict__ ident, int32_t *out) {
  int m = 1;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    m = max(m, ident[i]);
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

// BFS of each listed piece from its first vertex, one piece per CTA at a
// time: its vertices in the order the search reaches them, their tree parents,
// the deepest level and how many it reached.  Levels are narrow or the piece is
// small (a large piece is given up at a level wider than PIECE_BFS_WIDE: the
// whole GPU searches it): the wait after a level is CTA-wide, and the level's
// vertices are kept in shared memory.
constexpr int PIECE_BFS_THREADS = 1024;
constexpr int PIECE_BFS_RING = 2048;
// Rows of more than PIECE_BFS_LONG entries wait for the end of their level and
// are taken by a warp each, those of more than PIECE_BFS_HUGE by the whole CTA:
// one thread on a hub's row holds up everybody (a power-law piece of 13,700
// vertices: 0.72 to 0.29 ms).
constexpr int PIECE_BFS_LONG = 64;
constexpr int PIECE_BFS_HUGE = 2048;
constexpr int PIECE_BFS_LONGS = 1024;  // kept of a level; more are walked by their thread
constexpr int PIECE_BFS_HUGES = 64;
constexpr int PIECE_BFS_WIDE = 8192;
__global__ void __launch_bounds__(PIECE_BFS_THREADS) k_piece_bfs(const CompDesc *__restrict__ comps,
                                                                 const int32_t *__restrict__ list, int nlist,
                                                                 int *next, const int64_t *__restrict__ g_row,
                                                                 const int32_t *__restrict__ g_col,
                                                                 const int64_t *__restrict__ ord_off, int32_t *order,
                                                                 int32_t *parent, int32_t *level, int32_t *depth,
                                                                 int32_t *reached, PieceBfsEnd end) {
  __shared__ int s_i, s_tail, s_nlong, s_nhuge;
  __shared__ int32_t s_ring[2][PIECE_BFS_RING];
  __shared__ int32_t s_long[PIECE_BFS_LONGS], s_huge[PIECE_BFS_HUGES];
  const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  constexpr int WARPS = PIECE_BFS_THREADS / 32;
  for (;;) {
    if (threadIdx.x == 0) s_i = atomicAdd(next, 1);
    __syncthreads();
    const int i = s_i;
    if (i >= nlist) return;
    const CompDesc c = comps[list[i]];
    const int64_t *row = g_row + c.row_off;
    int32_t *const q = order + ord_off[i], *const lv = level + ord_off[i], *const par = parent + ord_off[i];
    for (int32_t v = threadIdx.x; v < c.n; v += PIECE_BFS_THREADS) lv[v] = v == 0 ? 0 : -1;
    if (threadIdx.x == 0) {
      q[0] = s_ring[0][0] = 0;
      par[0] = -1;
      s_tail = 1;
      s_nlong = s_nhuge = 0;
    }
    __syncthreads();
    // v's entries e, e + step, ... below e1
    auto walk = [&](int32_t v, int64_t e, int64_t e1, int step, int32_t *ring_next, int hi, int L) {
      for (; e < e1; e += 4 * step) {
        int32_t u[4], l[4];
#pragma unroll
        for (int j = 0; j < 4; j++) u[j] = e + j * step < e1 ? g_col[e + j * step] : -1;
#pragma unroll
        for (int j = 0; j < 4; j++) l[j] = u[j] >= 0 ? *(volatile int32_t *)(lv + u[j]) : 0;
#pragma unroll
        for (int j = 0; j < 4; j++)
          if (l[j] < 0) l[j] = atomicCAS(lv + u[j], -1, L + 1);
#pragma unroll
        for (int j = 0; j < 4; j++)
          if (l[j] < 0) {
            const int t = atomicAdd(&s_tail, 1);
            q[t] = u[j];
            par[u[j]] = v;
            if (t - hi < PIECE_BFS_RING) ring_next[t - hi] = u[j];
          }
      }
    };
    int lo = 0, hi = 1, L = 0;
    while (lo < hi) {
      const int32_t *const ring = s_ring[L & 1];
      int32_t *const ring_next = s_ring[(L + 1) & 1];
      // a next level found too wide ends the search at once
      auto too_wide = [&]() { return c.n > PIECE_BFS_MAX_N && *(volatile int *)&s_tail - hi > PIECE_BFS_WIDE; };
      for (int k = lo + (int)threadIdx.x; k < hi && !too_wide(); k += PIECE_BFS_THREADS) {
        const int32_t v = k - lo < PIECE_BFS_RING ? ring[k - lo] : q[k];
        const int64_t e0 = row[v], e1 = row[v + 1];
        if (e1 - e0 > PIECE_BFS_HUGE) {
          const int t = atomicAdd(&s_nhuge, 1);
          if (t < PIECE_BFS_HUGES) {
            s_huge[t] = v;
            continue;
          }
        }
        if (e1 - e0 > PIECE_BFS_LONG) {
          const int t = atomicAdd(&s_nlong, 1);
          if (t < PIECE_BFS_LONGS) {
            s_long[t] = v;
            continue;
          }
        }
        walk(v, e0, e1, 1, ring_next, hi, L);
      }
      __syncthreads();
      const int nlong = min(s_nlong, PIECE_BFS_LONGS), nhuge = min(s_nhuge, PIECE_BFS_HUGES);
      for (int j = 0; j < nhuge && !too_wide(); j++)
        walk(s_huge[j], row[s_huge[j]] + threadIdx.x, row[s_huge[j] + 1], PIECE_BFS_THREADS, ring_next, hi, L);
      for (int j = warp; j < nlong && !too_wide(); j += WARPS)
        walk(s_long[j], row[s_long[j]] + lane, row[s_long[j] + 1], 32, ring_next, hi, L);
      __syncthreads();
      lo = hi;
      hi = *(volatile int *)&s_tail;
      if (threadIdx.x == 0) s_nlong = s_nhuge = 0;
      __syncthreads();
      L++;
      if (c.n > PIECE_BFS_MAX_N && hi - lo > PIECE_BFS_WIDE) break;
      if (lo < hi && L >= end.levels && hi <= (int64_t)end.width * L) break;
    }
    if (threadIdx.x == 0) {
      depth[i] = L - 1;
      reached[i] = lo == hi ? hi : L >= end.levels && hi <= (int64_t)end.width * L ? -2 : -1;
    }
  }
}

int piece_bfs(Ctx &ctx, const std::vector<CompDesc> &comps, const CompDesc *d_comps, const std::vector<int32_t> &list,
              const BcInput &in, const std::vector<int64_t> &ord_off, int32_t *order, int32_t *parent, PieceBfsEnd end,
              std::vector<int32_t> *depth, std::vector<int32_t> *reached) {
  const int P = (int)list.size();
  depth->assign(P, 0);
  reached->assign(P, 0);
  if (P == 0) return BCS_OK;
  int64_t tot = 0;
  for (int i = 0; i < P; i++) tot = std::max(tot, ord_off[i] + comps[list[i]].n);
  DBuf<int32_t> d_list, d_level, d_out;
  DBuf<int64_t> d_off;
  BCS_TRY(d_list.alloc(P, ctx.stream));
  BCS_TRY(d_off.alloc(P, ctx.stream));
  BCS_TRY(d_level.alloc(tot, ctx.stream));
  BCS_TRY(d_out.alloc(2 * P + 1, ctx.stream));  // depth, reached, the queue's counter
  BCS_CUDA(cudaMemcpyAsync(d_list.p, list.data(), P * sizeof(int32_t), cudaMemcpyHostToDevice, ctx.stream));
  BCS_CUDA(cudaMemcpyAsync(d_off.p, ord_off.data(), P * sizeof(int64_t), cudaMemcpyHostToDevice, ctx.stream));
  BCS_CUDA(cudaMemsetAsync(d_out.p + 2 * P, 0, sizeof(int32_t), ctx.stream));
  k_piece_bfs<<<std::min(P, ctx.num_sms * 2), PIECE_BFS_THREADS, 0, ctx.stream>>>(
      d_comps, d_list.p, P, d_out.p + 2 * P, in.row, in.col, d_off.p, order, parent, d_level.p, d_out.p, d_out.p + P,
      end);
  ctx.launches++;
  BCS_CUDA(cudaGetLastError());
  BCS_CUDA(cudaMemcpyAsync(depth->data(), d_out.p, P * sizeof(int32_t), cudaMemcpyDeviceToHost, ctx.stream));
  BCS_CUDA(cudaMemcpyAsync(reached->data(), d_out.p + P, P * sizeof(int32_t), cudaMemcpyDeviceToHost, ctx.stream));
  BCS_CUDA(cudaStreamSynchronize(ctx.stream));
  return BCS_OK;
}

// ------------------------------------------------------------ host side
int pull_depth_limit() { return 250; }

// bytes of state per row for levels up to depth_bound, and per item of a long row
static size_t pull_row_bytes(int depth_bound, int w) { return 12 * (size_t)w + 4 * PULL_WORDS * (size_t)(depth_bound + 4) + 1; }
constexpr size_t PULL_ITEM_BYTES = 8 * PULL_W + 4 * PULL_WORDS + 8;

static size_t pull_state_bytes(int64_t n, int64_t nnz, int depth_bound, int w) {
  if (n > PULL_ROWS_MAX - PULL_UNIT) return SIZE_MAX;
  return (size_t)(n + PULL_UNIT) * pull_row_bytes(depth_bound, w) + (size_t)(nnz / PULL_LIST) * 2 * PULL_ITEM_BYTES;
}
size_t pull_piece_bytes(int64_t n, int64_t nnz, int depth_bound) { return pull_state_bytes(n, nnz, depth_bound, PULL_W); }

// The most values to a row with which a piece's state fits three quarters of
// the memory there is (or PULL_ONE_LAUNCH, with all of them), 0 when not even
// PULL_W_MIN do: of 200 GB, 58 million vertices of ten levels get 256, 180
// million 32.
int pull_width(int64_t n, int64_t nnz, int depth_bound, size_t free_bytes) {
  if (test_memory() == 0 && pull_piece_bytes(n, nnz, depth_bound) <= PULL_ONE_LAUNCH) return PULL_W;
  for (int w = PULL_W; w >= PULL_W_MIN; w /= 2)
    if (pull_state_bytes(n, nnz, depth_bound, w) <= free_bytes / 4 * 3) return w;
  return 0;
}

template <bool R, bool I, bool F>
static int pull_launch_t(Ctx &ctx, PullArgs &A) {
  const auto kernel = A.w < PULL_W ? k_bcreach_pull<R, I, F, true> : k_bcreach_pull<R, I, F, false>;
  int per_sm = 0;
  BCS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, PULL_THREADS, 0));
  if (per_sm < 1) {
    set_error("the pull Bc-Reach kernel cannot be resident");
    return BCS_ECUDA;
  }
  per_sm = std::min(per_sm, PULL_CTAS);
  void *args[] = {(void *)&A};
  BCS_CUDA(cudaLaunchCooperativeKernel((const void *)kernel, dim3(ctx.num_sms * per_sm),
                                       dim3(PULL_THREADS), args, 0, ctx.stream));
  ctx.launches++;
  return BCS_OK;
}

static int run_pull_jobs(Ctx &ctx, const std::vector<CompDesc> &comps, const std::vector<PullJob> &jobs,
                         const BcInput &in, bool fp32, const int32_t *d_order, const CompDesc *d_comps, int per_batch,
                         int *d_err, unsigned long long *d_dag) {
  const cudaStream_t s = ctx.stream;
  const int NJ = (int)jobs.size();
  // items of long rows
  std::vector<int32_t> nitems(NJ, 0), job_comp(NJ);
  std::vector<int64_t> item_off(NJ, 0);
  DBuf<int32_t> d_jobcomp, d_cnt;
  DBuf<int64_t> d_itemoff;
  DBuf<PullChunk> d_chunks;
  DBuf<PullItem> d_items;
  int64_t items_total = 0, fan = 1, nmax = 1, rows_total = 0, nbatches = 0;
  int depth = 1;
  {
    std::vector<PullChunk> chunks;
    constexpr int32_t CH = 8192;
    for (int k = 0; k < NJ; k++) {
      const CompDesc &c = comps[jobs[k].ci];
      job_comp[k] = jobs[k].ci;
      fan = std::max<int64_t>(fan, c.maxdeg);
      nmax = std::max<int64_t>(nmax, c.n);
      depth = std::max(depth, jobs[k].depth_bound);
      if (c.maxdeg > PULL_LIST)
        for (int32_t v = 0; v < c.n; v += CH) chunks.push_back(PullChunk{k, v, std::min(c.n, v + CH)});
    }
    if (!chunks.empty()) {
      BCS_TRY(d_jobcomp.alloc(NJ, s));
      BCS_TRY(d_cnt.alloc(NJ, s));
      BCS_TRY(d_itemoff.alloc(NJ, s));
      BCS_TRY(d_chunks.alloc(chunks.size(), s));
      BCS_CUDA(cudaMemcpyAsync(d_jobcomp.p, job_comp.data(), NJ * sizeof(int32_t), cudaMemcpyHostToDevice, s));
      BCS_CUDA(cudaMemcpyAsync(d_chunks.p, chunks.data(), chunks.size() * sizeof(PullChunk), cudaMemcpyHostToDevice, s));
      BCS_CUDA(cudaMemsetAsync(d_cnt.p, 0, NJ * sizeof(int32_t), s));
      k_pull_items<<<(unsigned)chunks.size(), 256, 0, s>>>(d_chunks.p, d_comps, d_jobcomp.p, in.row, d_cnt.p, nullptr,
                                                           nullptr, false);
      BCS_CUDA(cudaGetLastError());
      BCS_CUDA(cudaMemcpyAsync(nitems.data(), d_cnt.p, NJ * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
      BCS_CUDA(cudaStreamSynchronize(s));
      for (int k = 0; k < NJ; k++) {
        item_off[k] = items_total;
        items_total += nitems[k];
      }
      BCS_TRY(d_items.alloc(std::max<int64_t>(items_total, 1), s));
      BCS_CUDA(cudaMemcpyAsync(d_itemoff.p, item_off.data(), NJ * sizeof(int64_t), cudaMemcpyHostToDevice, s));
      BCS_CUDA(cudaMemsetAsync(d_cnt.p, 0, NJ * sizeof(int32_t), s));
      k_pull_items<<<(unsigned)chunks.size(), 256, 0, s>>>(d_chunks.p, d_comps, d_jobcomp.p, in.row, d_cnt.p,
                                                           d_itemoff.p, d_items.p, true);
      ctx.launches += 2;
      BCS_CUDA(cudaGetLastError());
    }
  }
  size_t free_b = 0;
  BCS_TRY(device_free_bytes(&free_b));
  int w = PULL_W;  // the pieces were let in by pull_width
  for (const PullJob &j : jobs)
    w = std::min(w, std::max(PULL_W_MIN, pull_width(comps[j.ci].n, comps[j.ci].nnz, j.depth_bound, free_b)));
  const int per_slab = std::min(per_batch * (PULL_W / 64), w);  // sources of a slab
  // slabs, cut into waves of about the same number of rows
  auto up = [](int64_t x) { return (x + PULL_UNIT - 1) / PULL_UNIT * PULL_UNIT; };
  for (const PullJob &j : jobs) {
    rows_total += (j.nsrc + per_slab - 1) / per_slab * up(comps[j.ci].n);
    nbatches += (j.nsrc + per_batch - 1) / per_batch;
  }
  const size_t per_row = pull_row_bytes(depth, w), budget = std::min<size_t>(free_b / 2, PULL_BYTES);
  const int64_t wave_rows = std::max(PULL_ROWS, std::min(PULL_ROWS_TOP, PULL_SLABS * nmax));
  const int64_t nw = (rows_total + wave_rows - 1) / wave_rows;
  const int64_t target = std::max(up(nmax), up((rows_total + nw - 1) / std::max<int64_t>(nw, 1)) + up(nmax) / 2);
  std::vector<PullSlab> slabs;
  std::vector<int32_t> wave(1, 0);
  int64_t r = 0, h = 0, rmax = 0, hmax = 0, jmax = 0;
  auto close = [&]() {
    if ((int64_t)slabs.size() == wave.back()) return;
    rmax = std::max(rmax, r);
    hmax = std::max(hmax, h);
    jmax = std::max<int64_t>(jmax, (int64_t)slabs.size() - wave.back());
    wave.push_back((int32_t)slabs.size());
    r = h = 0;
  };
  for (int k = 0; k < NJ; k++) {
    const CompDesc &c = comps[jobs[k].ci];
    for (int64_t b = 0; b < jobs[k].nsrc; b += per_slab) {
      const int64_t rows_after = r + up(c.n);
      if (rows_after > target ||
          (size_t)rows_after * per_row + (size_t)(h + nitems[k]) * PULL_ITEM_BYTES > budget)
        close();
      slabs.push_back(PullSlab{k, (int32_t)b, (int32_t)std::min<int64_t>(per_slab, jobs[k].nsrc - b), c.n, (int32_t)r,
                               (int32_t)h, nitems[k], 0});
      r += up(c.n);
      h += nitems[k];
    }
  }
  close();
  if (slabs.empty()) return BCS_OK;
  std::vector<PullJobDev> hj(NJ);
  for (int k = 0; k < NJ; k++) {
    const CompDesc &c = comps[jobs[k].ci];
    hj[k] = PullJobDev{c.row_off, c.vtx_off, jobs[k].ord_off, item_off[k]};
  }
  const int lcap = depth + 3;
  PullArgs A;
  std::memset(&A, 0, sizeof(A));
  A.flg = 0;
  while (((int64_t)1 << A.flg) < fan) A.flg++;
  // counts can only come near the end of the double range when the levels
  // allow it (ident is at most fan: pieces merged more than once have few
  // neighbours of large ident, so the degree alone is no bound)
  int fan_lg = 0;
  for (const PullJob &j : jobs)
    while ((double)((int64_t)1 << fan_lg) < comps[j.ci].fan) fan_lg++;
  const bool may_scale = (int64_t)lcap * std::max(A.flg + (in.ident ? fan_lg : 0), 1) > PULL_REC;
  DBuf<PullSlab> d_slabs;
  DBuf<int32_t> d_wave, umap, ctr, hctr, idmax;
  DBuf<PullJobDev> d_jobs;
  DBuf<double> S8, ws, hpart;
  DBuf<uint32_t> S4, M, seen, hmask;
  DBuf<unsigned long long> lmax, gmax, barw, trace;
  const bool tracing = std::getenv("BCS_TRACE") != nullptr;
  if (tracing) {
    BCS_TRY(trace.alloc(2 * PULL_TRACE_CAP, s));
    BCS_CUDA(cudaMemsetAsync(trace.p, 0, 2 * PULL_TRACE_CAP * 8, s));
    A.trace = trace.p;
  }
  const int64_t rows = up(rmax);
  BCS_TRY(d_slabs.alloc(slabs.size(), s));
  BCS_TRY(d_wave.alloc(wave.size(), s));
  BCS_TRY(d_jobs.alloc(NJ, s));
  BCS_TRY(S8.alloc((size_t)rows * w, s));
  BCS_TRY(S4.alloc((size_t)rows * w, s));
  BCS_TRY(M.alloc((size_t)lcap * rows * PULL_WORDS, s));
  BCS_TRY(seen.alloc((size_t)rows * PULL_WORDS, s));
  BCS_TRY(umap.alloc(rows / PULL_UNIT + hmax, s));
  BCS_TRY(ws.alloc((size_t)jmax * PULL_W, s));
  if (may_scale) BCS_TRY(lmax.alloc((size_t)lcap * jmax * PULL_W, s));
  BCS_TRY(gmax.alloc(lcap + 1, s));
  BCS_TRY(ctr.alloc((size_t)2 * lcap * PULL_SHARDS * 32, s));
  BCS_TRY(hpart.alloc((size_t)hmax * PULL_W, s));
  BCS_TRY(hmask.alloc((size_t)hmax * PULL_WORDS, s));
  BCS_TRY(hctr.alloc(hmax, s));
  BCS_TRY(idmax.alloc(1, s));
  BCS_TRY(barw.alloc(1, s));
  BCS_CUDA(cudaMemcpyAsync(d_slabs.p, slabs.data(), slabs.size() * sizeof(PullSlab), cudaMemcpyHostToDevice, s));
  BCS_CUDA(cudaMemcpyAsync(d_wave.p, wave.data(), wave.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
  BCS_CUDA(cudaMemcpyAsync(d_jobs.p, hj.data(), NJ * sizeof(PullJobDev), cudaMemcpyHostToDevice, s));
  BCS_CUDA(cudaMemsetAsync(barw.p, 0, sizeof(unsigned long long), s));
  BCS_CUDA(cudaMemsetAsync(idmax.p, 0, sizeof(int32_t), s));
  if (in.ident) {
    int64_t ntot = 0;
    for (const CompDesc &c : comps) ntot = std::max<int64_t>(ntot, c.vtx_off + c.n);
    k_pull_idmax<<<(int)std::min<int64_t>((ntot + 255) / 256, (int64_t)ctx.num_sms * 8), 256, 0, s>>>(ntot, in.ident,
                                                                                                  idmax.p);
    ctx.launches++;
    BCS_CUDA(cudaGetLastError());
  }
  A.slabs = d_slabs.p;
  A.wave = d_wave.p;
  A.nwaves = (int32_t)wave.size() - 1;
  A.jobs = d_jobs.p;
  A.items = d_items.p;
  A.g_row = in.row;
  A.g_col = in.col;
  A.g_reach = in.init ? nullptr : in.reach;
  A.g_ident = in.ident;
  A.order = d_order;
  A.g_init = in.init;
  A.bcp = in.bcp;
  A.S8 = S8.p;
  A.S4 = S4.p;
  A.M = M.p;
  A.seen = seen.p;
  A.umap = umap.p;
  A.ws = ws.p;
  A.lmax = lmax.p;
  A.gmax = gmax.p;
  A.ctr = ctr.p;
  A.hpart = hpart.p;
  A.hmask = hmask.p;
  A.hctr = hctr.p;
  A.idmax = idmax.p;
  BCS_TRY(recip_table(ctx, &A.recip));
  A.rows = rows;
  A.w = (uint32_t)w;
  A.slabs_cap = jmax;
  A.lcap = lcap;
  A.bar = GridBarrier{(unsigned int *)barw.p, (unsigned int *)barw.p + 1, d_err, (long long)ctx.max_wait};
  A.err = d_err;
  A.dag_total = d_dag;
  A.sig_cap = std::min(ctx.sigma_cap_lg2, 1024);  // 1024: infinities
  const bool R = in.reach != nullptr || in.init != nullptr, I = in.ident != nullptr;
  BCS_TRY(BCS_DISPATCH3(pull_launch_t, R, I, fp32, ctx, A));
  ctx.stats.n_wide_batches += nbatches;
  if (tracing) {  // the first waves' pass times (us)
    std::fprintf(stderr, "[bcs trace] pull: %d pieces, %zu slabs in %d waves of up to %lld rows, %lld items, %d levels at most, %d values to a row\n",
                 NJ, slabs.size(), A.nwaves, (long long)rows, (long long)hmax, lcap, w);
    std::vector<unsigned long long> tr(2 * PULL_TRACE_CAP);
    BCS_CUDA(cudaMemcpyAsync(tr.data(), trace.p, tr.size() * 8, cudaMemcpyDeviceToHost, s));
    BCS_CUDA(cudaStreamSynchronize(s));
    std::string line;
    for (int i = 1; i < PULL_TRACE_CAP && tr[2 * i + 1]; i++) {
      const unsigned tag = (unsigned)(tr[2 * i] & 0xffffffffu);
      char buf[64];
      const char *kind = (tag >> 12) == 1 ? "p1L" : (tag >> 12) == 2 ? "p2L" : (tag >> 12) == 0xE ? "tables" : "sources";
      std::snprintf(buf, sizeof(buf), " %s%u:%.1f", kind, tag & 0xfffu, (tr[2 * i + 1] - tr[2 * i - 1]) * 1e-3);
      line += buf;
    }
    std::fprintf(stderr, "[bcs trace] pull passes us:%s\n", line.c_str());
  }
  return BCS_OK;
}

int run_pull(Ctx &ctx, const std::vector<CompDesc> &comps, const std::vector<PullJob> &jobs_in, const BcInput &in,
             bool fp32, const int32_t *d_order, const CompDesc *d_comps, int per_batch, int *d_err,
             unsigned long long *d_dag) {
  // deep pieces apart from shallow ones (a wave runs as many levels as its
  // deepest slab), large ones first
  std::vector<PullJob> jobs(jobs_in);
  std::stable_sort(jobs.begin(), jobs.end(), [&](const PullJob &a, const PullJob &b) {
    const int da = a.depth_bound / 8, db = b.depth_bound / 8;
    return da != db ? da > db : comps[a.ci].n > comps[b.ci].n;
  });
  // A launch's rows have masks for the levels of its deepest piece.  Where a
  // shallow piece would outgrow a launch's memory by that (it was let in by its
  // own levels), a launch for every depth.
  int depth = 0;
  for (const PullJob &j : jobs) depth = std::max(depth, j.depth_bound);
  bool apart = false;
  for (const PullJob &j : jobs)
    apart = apart || (j.depth_bound / 8 != depth / 8 &&
                      pull_piece_bytes(comps[j.ci].n, comps[j.ci].nnz, depth) > PULL_ONE_LAUNCH);
  for (size_t a = 0; a < jobs.size();) {
    size_t b = jobs.size();
    if (apart) {
      b = a;
      while (b < jobs.size() && jobs[b].depth_bound / 8 == jobs[a].depth_bound / 8) b++;
    }
    BCS_TRY(run_pull_jobs(ctx, comps, std::vector<PullJob>(jobs.begin() + a, jobs.begin() + b), in, fp32, d_order,
                          d_comps, per_batch, d_err, d_dag));
    a = b;
  }
  return BCS_OK;
}

}  // namespace bcs
