// bcreach.cu - Bc-Reach (Algorithm 2 with the identical-vertex terms of
// Section 3.3.3) over many components: the plan that sends each to a kernel,
// the autotuner, and the one-source-per-CTA kernel in global memory.
//
// Per source s of a component (local ids, reach r[], ident k[]):
//   phase 1 (BFS, Algorithm 1):  d[s] = 0, sigma[s] = 1,
//     sigma[w] += sigma[v] * (v == s ? 1 : k[v])  for every DAG edge v -> w
//   phase 2 (Eq. 3 with reach and ident):
//     delta[v] = r[v] - 1 + sum_{w: d[w] = d[v]+1} sigma[v]/sigma[w] * k[w] * (1 + delta[w])
//     bc'[v]  += r[s] * k[s] * delta[v]   for v != s
// Phase 2 is evaluated in the equivalent "coefficient" form
//     c[w] = k[w] (1 + delta[w]) / sigma[w],   delta[v] = r[v] - 1 + sigma[v] * sum_w c[w]
// so that each shortest-path-DAG edge costs one addition and each vertex one
// reciprocal (in small.cu, pull.cu and deep.cu from a table for small integer
// counts).
//
// The one-source-per-CTA kernel is level-synchronous: the BFS queue doubles as
// the stack of Algorithm 1 and its level boundaries are kept, so phase 2 walks
// the levels deepest first and pulls from the successors (no atomics in phase
// 2).
//
// Path counts are exact 64-bit integers while a level's growth bound stays
// below 2^62; past it they are FP64 and each level carries a power-of-two
// exponent: when a level's largest count passes 2^960 the whole level is
// scaled by an exact power of two, and phase 2 multiplies by 2^(e[L] - e[L+1]).
//
// FP32 mode keeps delta and the per-edge sums in FP32: c is stored as an FP32
// value relative to the binary exponent of sigma[w] (held next to it), so
// sigma's full range is kept without FP64 arithmetic in phase 2.
#include <algorithm>
#include <cfloat>
#include <cstdlib>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <numeric>
#include <set>

#include "bc_math.cuh"
#include "common.h"

namespace bcs {

constexpr int LARGE_THREADS = 512;
// BFS depth above which large pieces run one source per CTA rather than 32
constexpr int MS_DEPTH_LIMIT = 64;
// Large pieces whose BFS eccentricity (from their first vertex) is at most
// PULL_MAX_ECC run on the pull kernel (pull.cu)
constexpr int PULL_MAX_ECC = 40;
// (a whole graph of several components, of n vertices of which `pairs` ordered
// pairs share one: unless they are many small ones.  The pull kernel looks at
// every vertex for every slab of sources, some 0.65 ps a level and (source,
// vertex), and at the pairs for 60; the kernels below at the pairs alone, for
// 200 to 400, and 20 ns a source.  1,000 paths of 30 vertices: 18 ms on it, 2.0
// on them, 10,000 paths 1,071 and 13; 30 power-law graphs of 1,000 8.3 and 6.6;
// one of 5,000 and 3,000 rings of 9 5.2 and 12)
static bool pull_reaches(int64_t n, int64_t pairs, int depth) {
  return (depth + 1.0) * (double)n * (double)n < 370.0 * (double)pairs + 3e4 * (double)n;
}
// and deeper ones than this, of small degree, on the deep kernel (deep.cu)
constexpr int DEEP_MIN_ECC = 40;
// Pieces that cannot run MID_SOURCES sources at once in that budget (some 800
// vertices and more) go to the pull kernel instead, if they are shallow and
// come in numbers: its cost is per level and slab (256 sources of a piece), so
// it wants few levels and slabs of at least MID_MIN_ROWS rows together.
// Batch of 16- to 4,096-vertex graphs: small and pull kernel 96 ms without
// the rule, 56 with it (59 from 1 source on, 56 from 3); a lone piece
// of 1,400 vertices 0.29 ms here, 1.08 there.
constexpr int MID_SOURCES = 2;
constexpr int MID_PIECE_ECC = 8;
constexpr int64_t MID_MIN_ROWS = 1 << 15;
// Source lists of at most FEW_ROUNDS rounds of CTAs (three per SM).  All kernels
// then wait for the latency of their levels, one source per CTA for the fewest,
// and the search by one CTA that orders the sources for the others takes about as
// long as one source.
// Graphs of up to FEW_MAX_N vertices whose entries and longest row take these
// rounds less than FEW_US: no search (15,200 vertices in 38
// layers, 32 sources, 0.93 ms, 2.4 on the pull kernel; a ring of 6,000, 1 source,
// 9.7 ms, 18 on the deep one).  Above it the pull kernel is sooner (20,000
// vertices of a power law, 300 sources, 1.4 ms and 2.4), if the graph is not
// deep.  Of mean degree FEW_MEAN_DEG or less it may be a road, where more than
// FEW_ROAD_SOURCES, or a graph above FEW_ROAD_MAX_N, are worth the order (24,600
// vertices of a road, 1 source 2.3 ms, 2.8 without; a square grid of 10,000: 400 sources
// 1.8 ms on the deep kernel, 2.8; 1 source 1.5 and 1.1; a power-law graph of 3,400
// with pendants, 100 sources, 0.99 on the pull kernel, 0.64).  Above FEW_DENSE_DEG the
// pull kernel cuts the rows, and is sooner (800 vertices of degree 100 in a few
// levels, 1 source 0.48 ms and 0.58; 1,600 in 16 levels 0.86 and 1.02).
constexpr int32_t FEW_MAX_N = 32768, FEW_ROAD_MAX_N = 16384;
constexpr double FEW_US = 470.0;
constexpr int64_t FEW_ROUNDS = 2, FEW_MEAN_DEG = 6, FEW_ROAD_SOURCES = 128, FEW_DENSE_DEG = 64;
static double one_source_us(const CompDesc &c) { return 1.8e-3 * (double)c.nnz + 1.2 * c.maxdeg; }
// With one round the search is given up after these levels: of any width where a graph is small
// and no road, else when they hold few vertices (20,000 in a path, 30 sources: 54
// ms so, 105 with the order).  Where it ends in a small component of such a graph
// (and of at most FEW_APART_MAX_N vertices: a CTA's state is cleared for it) the
// others are not searched: 5,000 rings of 9, 200 sources 0.36 ms, 0.66 with them.
constexpr int32_t FEW_APART_MAX_N = 1 << 17;
constexpr PieceBfsEnd FEW_END = {12, INT32_MAX}, FEW_NARROW_END = {256, 16};
// BCS_LARGE_PATH=mid: the pull kernel on connected pieces of at most this
// many vertices and MID_MAX_ECC levels
constexpr int MID_MAX_N = 65536;
constexpr int MID_MAX_ECC = 30;

__device__ __forceinline__ double cta_max(double x, volatile double *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  double r = red[0];
  for (int i = 1; i < ((int)blockDim.x >> 5); i++) r = fmax(r, red[i]);
  __syncthreads();
  return r;
}

__device__ __forceinline__ int vld(const int32_t *p) { return *(volatile const int32_t *)p; }

template <bool FP32>
struct CoefT;
template <>
struct CoefT<false> {
  using type = double;
};
template <>
struct CoefT<true> {
  using type = Coef32;
};

// Reciprocals 1/k of the integers k < RECIP_TABLE (entry 0 unused), filled
// once per device by IEEE division (correctly rounded).
static __device__ double g_recip_table[RECIP_TABLE];

__global__ void k_fill_recip_table() {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < RECIP_TABLE; k += gridDim.x * blockDim.x)
    g_recip_table[k] = k == 0 ? 0.0 : 1.0 / (double)k;
}

// State of one source in global memory.
template <bool FP32>
struct SrcState {
  int32_t *d;
  double *sig;
  typename CoefT<FP32>::type *coef;  // sigma * ident in phase 1
  int32_t *queue;
  int32_t *lvl_start;  // levels + 2
  int32_t *lvl_exp;    // levels + 1
  int *qtail;          // shared counter
  double *red;         // shared, 17 doubles: maxima, and the source weight
};
constexpr int RED_WS = 16;  // slot of the source weight in SrcState::red

struct Weights {
  const int32_t *reach;   // local, nullable
  const int32_t *ident;   // local, nullable
  const double *init_d;   // reach - 1 as FP64, nullable, possibly fractional (it then replaces reach)
};

struct Debug {
  int32_t *d;
  double *sig;
  int32_t *exp;
  double *delta;
};

// One source of Bc-Reach over a component held as (row, col) with local ids,
// by one CTA.  The distances start at -1 and are put back that way through the
// queue at the end.  acc is private to the CTA (plain adds).  dag counts the
// shortest-path DAG edges seen in phase 2.
//
// Path counts are integers.  While the growth bound fan^L of a level stays
// below 2^62 they are summed as exact 64-bit integers (the FP64 pipe is the
// scarce one on GB300, and below 2^53 the values are the same bits as an
// FP64 sum); the first level whose bound could pass 2^62 converts the level
// before it to FP64 once, and from there on counts are FP64 with a
// power-of-two exponent per level.  sig holds int64 on the integer levels.
// Counts are pulled in a second pass over a level and successors found by
// their level (pushing through L2 atomics measured slower on deep graphs).
template <bool REACH, bool IDENT, bool FP32>
__device__ void bcreach_source(const int32_t s, const int64_t *__restrict__ row, const int32_t *__restrict__ col,
                               const Weights wt, const SrcState<FP32> st, double *acc, const double fan, int *err,
                               const Debug *dbg, unsigned long long &dag, int *lmax_out) {
  const int rank = (int)threadIdx.x, size = (int)blockDim.x;
  int32_t *const d = st.d;
  double *const sig = st.sig;
  long long *const sigi = (long long *)st.sig;
  double *const sk = (double *)st.coef;  // sigma[v] * (v == s ? 1 : ident[v]) in phase 1
  long long *const ski = (long long *)st.coef;
  long long *const pull_src = IDENT ? ski : sigi;  // sigma * ident (the source counts once)
  if (rank == 0) {
    d[s] = 0;
    sigi[s] = 1;
    ski[s] = 1;
    st.queue[0] = s;
    *st.qtail = 1;
    st.lvl_start[0] = 0;
    st.lvl_start[1] = 1;
    st.lvl_exp[0] = 0;
  }
  __syncthreads();
  // ---------------------------------------------------------- phase 1
  int lo = 0, hi = 1, L = 0, ecur = 0;
  int lint = 1 << 30;  // first FP64 level
  // growth bound of the current level's counts as a power of two, kept in
  // integers: level-uniform FP64 tests would be evaluated by every lane
  const int flg = ceil_log2_pos(fan);
  int blg = 0;
  for (;;) {
    // discover level L+1 (integer work only)
    for (int i = lo + rank; i < hi; i += size) {
      const int32_t v = st.queue[i];
      const int64_t eb = row[v], ee = row[v + 1];
      for (int64_t e = eb; e < ee; e++) {
        const int32_t w = col[e];
        if (vld(d + w) < 0 && atomicCAS(d + w, -1, L + 1) == -1) st.queue[atomicAdd(st.qtail, 1)] = w;
      }
    }
    __syncthreads();
    const int nhi = vld(st.qtail);
    __syncthreads();
    if (nhi == hi) break;
    blg += flg;
    if (lint > L + 1 && blg >= 62) {
      // level L+1 may not fit 63 bits: it is pulled in FP64 from level L
      lint = L + 1;
      for (int i = lo + rank; i < hi; i += size) {
        const int32_t v = st.queue[i];
        sk[v] = (double)pull_src[v];
      }
      __syncthreads();
    }
    if (L + 1 < lint) {  // path counts of level L+1, pulled from level L (one add per DAG edge)
      for (int i = hi + rank; i < nhi; i += size) {
        const int32_t w = st.queue[i];
        long long a = 0;
        const int64_t eb = row[w], ee = row[w + 1];
        for (int64_t e = eb; e < ee; e++) {
          const int32_t u = col[e];
          if (d[u] == L) a += pull_src[u];
        }
        sigi[w] = a;
        if (IDENT) ski[w] = a * (long long)wt.ident[w];
      }
    } else {
      for (int i = hi + rank; i < nhi; i += size) {
        const int32_t w = st.queue[i];
        double a = 0.0;
        const int64_t eb = row[w], ee = row[w + 1];
        for (int64_t e = eb; e < ee; e++) {
          const int32_t u = col[e];
          if (d[u] == L) a += sk[u];
        }
        sig[w] = a;
        sk[w] = IDENT ? a * (double)wt.ident[w] : a;
      }
      if (blg > 900) {
        __syncthreads();
        double m = 0.0;
        for (int i = hi + rank; i < nhi; i += size) m = fmax(m, sig[st.queue[i]]);
        m = cta_max(m, st.red);
        if (!(m <= DBL_MAX)) {
          if (rank == 0) atomicOr(err, ERR_OVERFLOW);
        } else if (m > 0x1p960) {
          const int k = ilogb(m) - 959;
          for (int i = hi + rank; i < nhi; i += size) {
            const int32_t w = st.queue[i];
            sig[w] = scalbn(sig[w], -k);
            sk[w] = scalbn(sk[w], -k);
          }
          m = scalbn(m, -k);
          ecur += k;
        }
        blg = m >= 1.0 ? ceil_log2_pos(m) : 0;
        __syncthreads();
      }
    }
    lo = hi;
    hi = nhi;
    L++;
    if (rank == 0) {
      st.lvl_start[L + 1] = hi;
      st.lvl_exp[L] = ecur;
    }
  }
  const int Lmax = L;
  if (lmax_out && rank == 0) atomicMax(lmax_out, Lmax);
  // the source's weight reach[s] * ident[s] waits in shared memory: read
  // per vertex, it is never recomputed (FP64) inside the divergent loop
  if (rank == 0) {
    const long long is = IDENT ? (long long)wt.ident[s] : 1ll;
    st.red[RED_WS] = (REACH && wt.init_d) ? (wt.init_d[s] + 1.0) * (double)is
                                          : (double)((REACH ? (long long)wt.reach[s] : 1ll) * is);
  }
  __syncthreads();
  // ---------------------------------------------------------- phase 2
  unsigned long long ndag = 0;
  for (int l = Lmax; l >= 0; l--) {
    const int a = st.lvl_start[l], b = st.lvl_start[l + 1];
    const int de = (l < Lmax) ? st.lvl_exp[l] - st.lvl_exp[l + 1] : 0;
    const double scl = pow2_int(de);
    const bool is_int = l < lint;
    for (int i = a + rank; i < b; i += size) {
      const int32_t v = st.queue[i];
      double dv;
      // successors first as a bit mask (integer work), then one addition for
      // each: an FP64 warp instruction costs the pipe the same whatever its
      // active lanes, so the FP64 loop should run as few iterations as
      // possible (the DAG out-degree, not the degree)
      auto successors = [&](auto add) {
        if (l == Lmax) return;
        const int64_t eb = row[v], ee = row[v + 1];
        for (int64_t e0 = eb; e0 < ee; e0 += 32) {
          uint32_t mask = 0u;
          const int cnt = (int)((ee - e0) < 32 ? (ee - e0) : 32);
          for (int j = 0; j < cnt; j++) mask |= (uint32_t)(d[col[e0 + j]] == l + 1) << j;
          ndag += __popc(mask);
          for (; mask; mask &= mask - 1u) add(col[e0 + __ffs(mask) - 1]);
        }
      };
      if (!FP32) {
        const double sv = is_int ? i64_to_f64_pos(sigi[v]) : sig[v];
        double sum = 0.0;
        successors([&](int32_t w) { sum += ((const double *)st.coef)[w]; });
        if (de != 0) sum *= scl;
        const double init = REACH ? (wt.init_d ? wt.init_d[v] : (double)(wt.reach[v] - 1)) : 0.0;
        dv = fma(sv, sum, init);
        if (l > 0) {  // the source's coefficient is never read
          const double kv = IDENT ? (double)wt.ident[v] : 1.0;
          ((double *)st.coef)[v] = fma(kv, dv, kv) * recip_pos(sv);
        }
      } else {
        int ev;
        float mv;
        if (is_int) split_pow2_i64(sigi[v], ev, mv);
        else split_pow2(sig[v], ev, mv);
        ev += st.lvl_exp[l];
        float sum = 0.0f;
        successors([&](int32_t w) {
          const Coef32 c = ((const Coef32 *)st.coef)[w];
          const int x = ev - c.e;  // <= 0: sigma[v] <= sigma[w]
          if (x >= -126) sum = fmaf(c.c, __int_as_float((127 + x) << 23), sum);
        });
        const float df = fmaf(mv, sum, REACH ? (wt.init_d ? (float)wt.init_d[v] : (float)(wt.reach[v] - 1)) : 0.0f);
        dv = (double)df;
        if (l > 0) {
          const float kv = IDENT ? (float)wt.ident[v] : 1.0f;
          Coef32 cv;
          cv.c = fmaf(kv, df, kv) / mv;
          cv.e = ev;
          ((Coef32 *)st.coef)[v] = cv;
        }
      }
      if (v != s) acc[v] = fma(st.red[RED_WS], dv, acc[v]);
      if (dbg) dbg->delta[v] = dv;
    }
    __syncthreads();
  }
  dag += ndag;
  if (dbg) {
    for (int i = rank; i < hi; i += size) {
      const int32_t v = st.queue[i];
      const int lv = d[v];
      dbg->d[v] = lv;
      dbg->sig[v] = lv < lint ? (double)sigi[v] : sig[v];
      dbg->exp[v] = st.lvl_exp[lv];
    }
    __syncthreads();
  }
  for (int i = rank; i < hi; i += size) d[st.queue[i]] = -1;
  __syncthreads();
}

// ---------------------------------------------------------- large path
struct LargeSrc {
  int32_t comp;
  int32_t s;
};

// Per-CTA global scratch of the large path: each array holds grid * nmax
// entries, CTA b owning [b * nmax, (b+1) * nmax) (lvl arrays: nmax + 2).
struct LargeScratch {
  int32_t *d;      // -1 between sources
  int32_t *queue;
  double *sig;     // 0 between sources
  double *coef;    // 8 bytes per vertex in both precisions
  double *acc;     // 0 between components
  int32_t *lvl_start;
  int32_t *lvl_exp;
  int64_t nmax;
};

template <bool REACH, bool IDENT, bool FP32>
__global__ void __launch_bounds__(LARGE_THREADS) k_bcreach_large(
    const LargeSrc *__restrict__ work, int64_t nwork, unsigned long long *counter, const CompDesc *__restrict__ comps,
    const int64_t *__restrict__ g_row, const int32_t *__restrict__ g_col, const int32_t *__restrict__ g_reach,
    const int32_t *__restrict__ g_ident, const double *__restrict__ g_init, double *bcp, LargeScratch sc, int *err,
    Debug dbg_in, int use_dbg, unsigned long long *dag_total, int *lmax) {
  __shared__ unsigned long long s_idx;
  __shared__ int s_qtail;
  __shared__ double s_red[RED_WS + 1];
  const size_t b = blockIdx.x;
  SrcState<FP32> st;
  st.d = sc.d + b * sc.nmax;
  st.queue = sc.queue + b * sc.nmax;
  st.sig = sc.sig + b * sc.nmax;
  st.coef = (typename CoefT<FP32>::type *)(sc.coef + b * sc.nmax);
  double *acc = sc.acc + b * sc.nmax;
  st.lvl_start = sc.lvl_start + b * (sc.nmax + 2);
  st.lvl_exp = sc.lvl_exp + b * (sc.nmax + 2);
  st.qtail = &s_qtail;
  st.red = s_red;
  unsigned long long dag = 0;
  int cur = -1;
  for (;;) {
    if (threadIdx.x == 0) s_idx = atomicAdd(counter, 1ull);
    __syncthreads();
    const unsigned long long idx = s_idx;
    __syncthreads();
    const int next = idx < (unsigned long long)nwork ? work[idx].comp : -1;
    if (next != cur && cur >= 0) {  // flush the accumulator of the previous component
      const CompDesc c = comps[cur];
      for (int v = threadIdx.x; v < c.n; v += blockDim.x) {
        if (acc[v] != 0.0) atomicAdd(bcp + c.vtx_off + v, acc[v]);
        acc[v] = 0.0;
      }
      __syncthreads();
    }
    cur = next;
    if (next < 0) break;
    const CompDesc c = comps[cur];
    Weights wt{REACH && !g_init ? g_reach + c.vtx_off : nullptr, IDENT ? g_ident + c.vtx_off : nullptr,
               REACH && g_init ? g_init + c.vtx_off : nullptr};
    bcreach_source<REACH, IDENT, FP32>(work[idx].s, g_row + c.row_off, g_col, wt, st, acc, c.fan, err,
                                       use_dbg ? &dbg_in : nullptr, dag, lmax);
  }
  if (dag_total && dag) atomicAdd(dag_total, dag);
}

// bytes of global scratch per large-path CTA
static size_t large_scratch_bytes(int64_t nmax) { return (size_t)nmax * (4 + 4 + 8 + 8 + 8) + (size_t)(nmax + 2) * 8; }

// ---------------------------------------------------------- host side
// The reciprocal table, filled once per device (on the legacy stream, which
// orders it before any later work of every blocking stream).
static int recip_table_ready(int device) {
  static std::mutex mu;
  static std::set<int> done;
  std::lock_guard<std::mutex> lk(mu);
  if (!done.count(device)) {
    k_fill_recip_table<<<4, 256>>>();
    BCS_CUDA(cudaGetLastError());
    BCS_CUDA(cudaDeviceSynchronize());
    done.insert(device);
  }
  return BCS_OK;
}

int recip_table(Ctx &ctx, const double **out) {
  BCS_TRY(recip_table_ready(ctx.device));
  void *p = nullptr;
  BCS_CUDA(cudaGetSymbolAddress(&p, g_recip_table));
  *out = (const double *)p;
  return BCS_OK;
}

template <bool R, bool I, bool F>
static int launch_large_t(Ctx &ctx, int grid, const LargeSrc *work, int64_t nwork, unsigned long long *counter,
                          const CompDesc *comps, const BcInput &in, const LargeScratch &sc, int *err,
                          const Debug &dbg, int use_dbg, unsigned long long *dag, int *lmax = nullptr) {
  k_bcreach_large<R, I, F><<<grid, LARGE_THREADS, 0, ctx.stream>>>(work, nwork, counter, comps, in.row, in.col,
                                                                  in.reach, in.ident, in.init, in.bcp, sc, err, dbg,
                                                                  use_dbg, dag, lmax);
  ctx.launches++;
  BCS_CUDA(cudaGetLastError());
  return BCS_OK;
}

// The small-path work splits the autotuner tries: most sources a CTA runs
// at once, and the shared-memory budget per CTA (100 KB: 2 CTAs per SM,
// 72 KB: 3, 54 KB: 4).  Without it a CTA runs up to 16 with 54 KB (SMALL_BUDGET),
// which is not among them and the fastest on all that was measured: 5.04 ms on
// the articulation-vertex workload (these 7.2, 5.7, 5.2, 7.2), 0.52 on 500 graphs of
// up to 300 vertices (0.71, 0.71, 0.60, 0.78).
struct Split {
  int ng_cap;
  size_t budget;
};
static const Split TUNE_SPLITS[] = {{8, SMALL_SMEM}, {8, 72 * 1024}, {8, 54 * 1024}, {4, SMALL_SMEM}};

// Process-wide cache of the autotuner's choice (index + 1 into TUNE_SPLITS)
// per shape bucket.
static std::mutex g_tune_mu;
static std::map<long long, int> g_tune;

static int tuned_split(long long key) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  auto it = g_tune.find(key);
  return it == g_tune.end() ? 0 : it->second;
}

static void remember_split(long long key, int choice) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tune[key] = choice;
}

// Besides the small-path work split, the autotuner picks, by timing each
// candidate once per shape bucket and caching the fastest:
//  * the small/large threshold: the fixed rule (SMALL_SMEM, and numerous
//    shallow pieces of many vertices to the pull kernel: MID_SOURCES), or the
//    shared memory a piece may need for one source to take the small path
//    (SMALL_LIMITS); pieces above it take the large-piece path.  Timed over the
//    pieces that fit the largest limit.
//  * the kernel of each large piece: the pull kernel (where the
//    piece's depth allows it), 32-source batches (where its depth is below
//    4 x MS_DEPTH_LIMIT: their cost grows with the levels of a batch), or
//    one source per CTA, each timed on a sample of the piece's sources that
//    fills the GPU for that kernel.
// Every candidate runs into a scratch accumulator; the call then runs with
// the choice.  Without the autotuner the fixed limits above decide.
static const size_t SMALL_LIMITS[] = {0, SMALL_SMEM, 64 * 1024, 40 * 1024};  // 0: the fixed rule
static std::map<long long, int> g_tune_limit, g_tune_large;

static int tuned_in(std::map<long long, int> &m, long long key) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  auto it = m.find(key);
  return it == m.end() ? 0 : it->second;
}

static void remember_in(std::map<long long, int> &m, long long key, int v) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  m[key] = v;
}

static long long bits_of(double x) { return x < 1.0 ? 0 : (long long)std::log2(x) + 1; }

// One Bc-Reach run over `comps` into a scratch accumulator, timed; the
// call's statistics are left as they were.
static int time_candidate(Ctx &ctx, const std::vector<CompDesc> &comps, const BcInput &in, const BcPlanOpts &po,
                          double *ms) {
  int64_t ntot = 1;
  for (const CompDesc &c : comps) ntot = std::max<int64_t>(ntot, c.vtx_off + c.n);
  DBuf<double> scratch;
  BCS_TRY(scratch.alloc(ntot, ctx.stream));
  BCS_CUDA(cudaMemsetAsync(scratch.p, 0, ntot * sizeof(double), ctx.stream));
  BcInput in2 = in;
  in2.bcp = scratch.p;
  const bool at = ctx.autotune;
  const bcs_stats saved = ctx.stats;
  const size_t npend = ctx.pending.size();
  ctx.autotune = false;
  StageTimer t(ctx.stream);
  t.start();
  const int rc = run_bcreach(ctx, comps, in2, po);
  *ms = t.stop_ms();
  ctx.autotune = at;
  ctx.stats = saved;
  for (size_t i = npend; i < ctx.pending.size(); i++) {  // the candidate's stage times are not the call's
    cudaEventSynchronize(ctx.pending[i].b);
    cudaEventDestroy(ctx.pending[i].a);
    cudaEventDestroy(ctx.pending[i].b);
  }
  ctx.pending.resize(npend);
  return rc;
}

// Times the large-piece kernels on samples of one piece's sources (every
// vertex a source) and sets *choice to the fastest per source.  The samples
// are what each kernel sees in a full run: consecutive vertices of the BFS
// order from the piece's first vertex (d_ord) for the pull kernel,
// consecutive ids for the others.
static int tune_large_piece(Ctx &ctx, const CompDesc &c, const BcInput &in, const BcPlanOpts &po, bool wide_ok,
                            bool deep_ok, int depth, const int32_t *d_ord, int *choice) {
  struct Cand {
    int path;
    int64_t m;
  };
  const int64_t ns = nsrc_of(c), sms = ctx.num_sms;
  std::vector<Cand> cands;
  // the pull kernel on about a wave of rows
  if (wide_ok) cands.push_back({LARGE_PATH_WIDE, std::max<int64_t>(512, 64 * (((int64_t)1 << 21) / c.n))});
  if (depth <= 4 * MS_DEPTH_LIMIT) cands.push_back({LARGE_PATH_BATCHED, 32 * sms});
  if (deep_ok) cands.push_back({LARGE_PATH_DEEP, 24 * sms});
  cands.push_back({LARGE_PATH_PER_SOURCE, 6 * sms});
  *choice = cands[0].path;
  if (cands.size() == 1) return BCS_OK;
  double best = 0.0;
  for (const Cand &cd : cands) {
    const int64_t m = std::min(cd.m, std::max<int64_t>(1, ns / 4));
    const int64_t at = (ns - m) / 2;
    std::vector<int64_t> src(m);
    if (cd.path == LARGE_PATH_WIDE) {
      std::vector<int32_t> h(m);
      BCS_CUDA(cudaMemcpyAsync(h.data(), d_ord + at, m * sizeof(int32_t), cudaMemcpyDeviceToHost, ctx.stream));
      BCS_CUDA(cudaStreamSynchronize(ctx.stream));
      for (int64_t i = 0; i < m; i++) src[i] = h[i];
    } else {
      for (int64_t i = 0; i < m; i++) src[i] = at + i;
    }
    BcPlanOpts p2 = po;
    p2.sources = src.data();
    p2.nsources = m;
    p2.large_path = cd.path;
    p2.force_large = true;
    double ms = 0.0;
    BCS_TRY(time_candidate(ctx, std::vector<CompDesc>{c}, in, p2, &ms));
    const double rate = (double)m / std::max(ms, 1e-3);
    if (std::getenv("BCS_TRACE"))
      std::fprintf(stderr, "[bcs] tune large piece n=%d kernel %d: %lld sources in %.3f ms\n", c.n, cd.path,
                   (long long)m, ms);
    if (rate > best) {
      best = rate;
      *choice = cd.path;
    }
  }
  return BCS_OK;
}

__global__ void k_positions(int32_t n, const int32_t *__restrict__ order, uint32_t *pos) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) pos[order[i]] = i;
}
__global__ void k_gather_u32(int64_t k, const int32_t *__restrict__ at, const uint32_t *__restrict__ from, uint32_t *to) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += (int64_t)gridDim.x * blockDim.x)
    to[i] = from[at[i]];
}

// The caller's sources in the order of the piece's BFS: sources that are
// searched together then share more of their levels (1,000 random sources of a
// power-law graph of 291,000 vertices: 17.2 to 15.2 ms).
static int sort_by_position(Ctx &ctx, int32_t n, const int32_t *order, int32_t *src, int64_t k) {
  DBuf<uint32_t> pos, keys, tk;
  DBuf<int32_t> tv;
  BCS_TRY(pos.alloc(n, ctx.stream));
  BCS_TRY(keys.alloc(k, ctx.stream));
  BCS_TRY(tk.alloc(k, ctx.stream));
  BCS_TRY(tv.alloc(k, ctx.stream));
  k_positions<<<std::min((n + 255) / 256, ctx.num_sms * 8), 256, 0, ctx.stream>>>(n, order, pos.p);
  k_gather_u32<<<(int)std::min<int64_t>((k + 255) / 256, ctx.num_sms * 8), 256, 0, ctx.stream>>>(k, src, pos.p, keys.p);
  ctx.launches += 2;
  BCS_CUDA(cudaGetLastError());
  int bits = 1;
  while (bits < 32 && ((int64_t)1 << bits) < n) bits++;
  return radix_sort_pairs(ctx, keys.p, src, tk.p, tv.p, k, bits);
}


int run_bcreach(Ctx &ctx, const std::vector<CompDesc> &comps_in, const BcInput &in, const BcPlanOpts &po) {
  Tracer tr("bcreach", ctx.stream);
  const bool R = in.reach != nullptr || in.init != nullptr, I = in.ident != nullptr, F = po.fp32_delta;
  const bool dbg = po.dbg_d || po.dbg_sig || po.dbg_exp || po.dbg_delta;
  const int64_t C = (int64_t)comps_in.size();
  if (po.sources && (C != 1 || po.srcmap)) {
    set_error("a source list needs exactly one component and no source map");
    return BCS_EINVAL;
  }
  // a host source list is the one component's source map (uploaded below)
  std::vector<CompDesc> comps_src;
  if (po.sources) {
    comps_src = comps_in;
    comps_src[0].src_off = 0;
    comps_src[0].nsrc = (int32_t)po.nsources;
  }
  const std::vector<CompDesc> &comps = po.sources ? comps_src : comps_in;
  // the large-piece kernel, if fixed: by the caller, or by BCS_LARGE_PATH
  // (wide|batched|per_source; wide_all, for tests: every piece runs on the
  // large-piece path, and on the pull kernel wherever that can take it)
  int lp_mode = po.large_path;
  bool all_large = false;
  if (const char *e = std::getenv("BCS_LARGE_PATH")) {
    if (!std::strcmp(e, "wide_all") || !std::strcmp(e, "mid_all") || !std::strcmp(e, "deep_all")) all_large = true;
    if (!std::strcmp(e, "deep") || !std::strcmp(e, "deep_all")) lp_mode = LARGE_PATH_DEEP;
    if (!std::strcmp(e, "mid_all")) lp_mode = LARGE_PATH_MID;
    if (!std::strcmp(e, "wide") || !std::strcmp(e, "wide_all")) lp_mode = LARGE_PATH_WIDE;
    if (!std::strcmp(e, "batched")) lp_mode = LARGE_PATH_BATCHED;
    if (!std::strcmp(e, "per_source")) lp_mode = LARGE_PATH_PER_SOURCE;
    if (!std::strcmp(e, "mid")) lp_mode = LARGE_PATH_MID;
  }
  const bool tune = ctx.autotune && lp_mode == LARGE_PATH_AUTO && !dbg && !po.sources && !po.srcmap &&
                    !po.force_large && !po.per_source_large;
  // the small/large threshold
  size_t small_limit = po.small_limit ? po.small_limit : SMALL_SMEM;
  bool mid_rule = !po.small_limit && lp_mode == LARGE_PATH_AUTO && !dbg && !po.per_source_large;
  if (tune && !po.small_limit) {
    double cost = 0.0, band = 0.0;  // of the pieces that fit the largest limit, and of those above the lowest
    const size_t lowest = SMALL_LIMITS[sizeof(SMALL_LIMITS) / sizeof(SMALL_LIMITS[0]) - 1];
    auto fits_any = [&](const CompDesc &c, size_t *s1) {
      if (c.n < 2 || nsrc_of(c) == 0 || !small_takes(c.n, c.nnz, 1)) return false;
      *s1 = small_smem_bytes(c.n, c.nnz, 1, R, I);
      return *s1 <= SMALL_SMEM;
    };
    for (const CompDesc &c : comps) {
      size_t s1 = 0;
      if (!fits_any(c, &s1)) continue;
      const double work = (double)nsrc_of(c) * (double)(c.nnz + c.n);
      cost += work;
      if (s1 > lowest) band += work;
    }
    if (band > 0.0) {
      const long long key = ((long long)(R * 2 + I) << 40) | (bits_of(cost) << 20) | bits_of(band);
      int ch = tuned_in(g_tune_limit, key);
      if (!ch) {
        std::vector<CompDesc> elig;
        for (const CompDesc &c : comps) {
          size_t s1 = 0;
          if (fits_any(c, &s1)) elig.push_back(c);
        }
        double best = 1e300;
        for (int k = 0; k < (int)(sizeof(SMALL_LIMITS) / sizeof(SMALL_LIMITS[0])); k++) {
          BcPlanOpts p2 = po;
          p2.small_limit = SMALL_LIMITS[k];
          double ms = 0.0;
          BCS_TRY(time_candidate(ctx, elig, in, p2, &ms));
          if (k == 0) BCS_TRY(time_candidate(ctx, elig, in, p2, &ms));  // the first got the memory pool going
          if (std::getenv("BCS_TRACE"))
            std::fprintf(stderr, "[bcs] tune small/large threshold %zu B: %.3f ms\n", SMALL_LIMITS[k], ms);
          if (ms < best) {
            best = ms;
            ch = k + 1;
          }
        }
        remember_in(g_tune_limit, key, ch);
      }
      mid_rule = SMALL_LIMITS[ch - 1] == 0;
      small_limit = mid_rule ? SMALL_SMEM : SMALL_LIMITS[ch - 1];
      ctx.stats.tuned |= 1;
    }
  }
  ctx.stats.small_limit = (int64_t)small_limit;
  std::vector<SmallItem> items;
  std::vector<LargeSrc> work;
  std::vector<int32_t> large, small;
  small.reserve(C);
  int64_t nmax_large = 0, nmax_small = 0;
  double work_se = 0.0, work_sv = 0.0, total_small_cost = 0.0;
  std::vector<int32_t> mids;  // pieces of the small path that the pull kernel may take instead
  auto small_takes_sources = [&](const CompDesc &c, int g) {
    return small_takes(c.n, c.nnz, g) && small_smem_bytes(c.n, c.nnz, g, R, I) <= SMALL_BUDGET;
  };
  auto pull_rows = [&](const CompDesc &c) { return (nsrc_of(c) + 255) / 256 * (int64_t)c.n; };
  auto to_small = [&](int32_t ci) {
    const CompDesc &c = comps[ci];
    small.push_back(ci);
    total_small_cost += (double)nsrc_of(c) * (double)(c.nnz + c.n);
    nmax_small = std::max<int64_t>(nmax_small, c.n);
  };
  for (int64_t ci = 0; ci < C; ci++) {
    const CompDesc &c = comps[ci];
    if (c.n < 2) continue;
    const int64_t ns = nsrc_of(c);
    if (ns == 0) continue;
    work_se += (double)ns * (double)c.nnz;
    work_sv += (double)ns * (double)c.n;
    const bool fits = !po.force_large && !all_large && !dbg && c.n <= 65535 &&
                      small_takes(c.n, c.nnz, 1) && small_smem_bytes(c.n, c.nnz, 1, R, I) <= small_limit;
    if (fits && mid_rule && !small_takes_sources(c, MID_SOURCES)) {
      mids.push_back((int32_t)ci);
    } else if (fits) {
      to_small((int32_t)ci);
    } else {
      large.push_back((int32_t)ci);
      nmax_large = std::max<int64_t>(nmax_large, c.n);
    }
  }
  {
    int64_t rows = 0;
    for (int32_t ci : mids) rows += pull_rows(comps[ci]);
    if (rows < MID_MIN_ROWS) {
      for (int32_t ci : mids) to_small(ci);
      mids.clear();
    }
  }
  // Large pieces of small BFS depth: the pull kernel, the sources of a piece
  // taken in the order of its BFS from its first vertex (neighbouring sources
  // share most of their levels).  That search also bounds the depth: no source
  // reaches deeper than twice its eccentricity.  BCS_LARGE_PATH=wide takes
  // every large piece whose depth allows it, mid the connected ones of at most
  // MID_MAX_N vertices; batched|per_source take none.
  DBuf<CompDesc> d_comps;
  if (!small.empty() || !large.empty() || !mids.empty()) {
    BCS_TRY(d_comps.alloc(C, ctx.stream));
    BCS_CUDA(cudaMemcpyAsync(d_comps.p, comps.data(), C * sizeof(CompDesc), cudaMemcpyHostToDevice, ctx.stream));
  }
  std::vector<PullJob> pull;
  // deep pieces of small degree: deep.cu (src_off: the caller's sources in pull_order, < 0: every vertex)
  struct DeepJob {
    int32_t ci, nsrc;
    int depth_bound;
    int64_t ord_off, src_off;
  };
  std::vector<DeepJob> deep;
  DBuf<int32_t> pull_order, pull_parent;  // BFS orders and tree parents, a piece after the other
  // large pieces the autotuner gave to 32-source batches, or to one source per CTA
  std::vector<int32_t> ms_tuned, ps_tuned;
  {
    const bool force_wide = lp_mode == LARGE_PATH_WIDE, force_mid = lp_mode == LARGE_PATH_MID;
    const bool none = lp_mode == LARGE_PATH_BATCHED || lp_mode == LARGE_PATH_PER_SOURCE || dbg || po.per_source_large;
    std::vector<int32_t> rest, cand;
    std::vector<int64_t> off;
    int64_t total = 0;
    PieceBfsEnd end;
    bool no_search = false;
    bool cheap = false;  // one source per CTA is
    if (po.sources && lp_mode == LARGE_PATH_AUTO) {
      const CompDesc &c = comps[0];
      const int64_t wave = 3 * (int64_t)ctx.num_sms, rounds = (po.nsources + wave - 1) / wave;
      const bool road = c.nnz <= FEW_MEAN_DEG * c.n;
      const bool small_n = c.n < (road ? FEW_ROAD_MAX_N : FEW_MAX_N) && c.nnz <= FEW_DENSE_DEG * c.n;
      cheap = rounds <= FEW_ROUNDS && rounds * one_source_us(c) < FEW_US;
      no_search = small_n && cheap && (po.nsources <= FEW_ROAD_SOURCES || !road);
      if (rounds <= 1) end = small_n && !road ? FEW_END : FEW_NARROW_END;
      // deeper than the pull kernel takes, and a row too long for the deep one
      if (c.maxdeg > DEEP_MAX_DEG && end.levels > PULL_MAX_ECC + 2) end = PieceBfsEnd{PULL_MAX_ECC + 2, INT32_MAX};
    }
    for (int32_t ci : large) {
      const CompDesc &c = comps[ci];
      if (none || no_search || (c.src_off >= 0 && !po.sources) || (force_mid && c.n > MID_MAX_N)) {
        rest.push_back(ci);
        continue;
      }
      cand.push_back(ci);
      off.push_back(total);
      total += c.n + (po.sources ? po.nsources : 0);
    }
    const size_t nlarge = cand.size();
    for (int32_t ci : mids) {
      if (comps[ci].src_off >= 0) {
        to_small(ci);
        continue;
      }
      cand.push_back(ci);
      off.push_back(total);
      total += comps[ci].n;
    }
    if (!cand.empty()) {
      BCS_TRY(pull_order.alloc(total, ctx.stream));
      BCS_TRY(pull_parent.alloc(total, ctx.stream));
    }
    std::vector<int32_t> cta_depth, cta_reached;
    BCS_TRY(piece_bfs(ctx, comps, d_comps.p, cand, in, off, pull_order.p, pull_parent.p, end, &cta_depth, &cta_reached));
    for (size_t k = 0; k < nlarge; k++) {
      const int32_t ci = cand[k];
      const CompDesc &c = comps[ci];
      int32_t *const ord = pull_order.p + off[k];
      int depth = cta_depth[k];
      int64_t reached = cta_reached[k];
      bool apart = false;  // a graph of many small components
      if (reached == -2 || (cheap && reached >= 0 && reached < c.n / 4 && c.n <= FEW_APART_MAX_N)) {
        rest.push_back(ci);
        continue;
      }
      if (reached < 0)  // large and wide: the whole GPU
        BCS_TRY(bfs_queue(ctx, in.row + c.row_off, in.col, c.n, 0, ord, pull_parent.p + off[k], &depth, &reached));
      if (reached != c.n && c.row_off == 0 && !force_mid) {
        // a whole graph of several components (the plain calls; pieces are
        // connected): every component searched from its smallest vertex
        DevGraph g{c.n, c.nnz, in.row, in.col};
        int64_t pairs = 0;
        BCS_TRY(bfs_queue_components(ctx, g, ord, pull_parent.p + off[k], &depth, &pairs));
        reached = c.n;
        apart = !pull_reaches(c.n, pairs, depth);
      }
      // every source's BFS depth is at most twice its component's root's
      const int bound = 2 * depth + 2;
      const bool ok = bound <= pull_depth_limit() && reached == c.n && (!force_mid || depth <= MID_MAX_ECC);
      bool deep_ok = false;
      if (reached == c.n && (lp_mode == LARGE_PATH_DEEP || (depth > DEEP_MIN_ECC && !force_wide && !force_mid))) {
        size_t free_b = 0;
        BCS_TRY(device_free_bytes(&free_b));
        deep_ok = deep_takes(c, bound, free_b);
      }
      // tuning pays only over many sources
      const bool tune_this = tune && c.src_off < 0 && nsrc_of(c) >= 24LL * ctx.num_sms;
      int choice = LARGE_PATH_AUTO;
      if (tune_this) {
        // what the piece may run on and the precision are part of its shape: a
        // choice made without them may not be open here, or not the fastest
        const long long key = ((long long)(((F * 2 + ok) * 2 + deep_ok) * 4 + R * 2 + I) << 40) | (bits_of(c.n) << 24) |
                              (bits_of((double)c.nnz / c.n) << 16) | bits_of(depth);
        choice = tuned_in(g_tune_large, key);
        if (!choice) {
          BCS_TRY(tune_large_piece(ctx, c, in, po, ok, deep_ok, depth, ord, &choice));
          remember_in(g_tune_large, key, choice);
        }
        if (choice == LARGE_PATH_BATCHED) ms_tuned.push_back(ci);
        if (choice == LARGE_PATH_PER_SOURCE) ps_tuned.push_back(ci);
        if (choice != LARGE_PATH_WIDE && choice != LARGE_PATH_DEEP) {
          ctx.stats.tuned |= 1ll << choice;
          continue;
        }
      }
      bool take = ok && lp_mode != LARGE_PATH_DEEP && choice != LARGE_PATH_DEEP && (!apart || force_wide || choice == LARGE_PATH_WIDE);
      if (choice == LARGE_PATH_AUTO && !force_wide && !force_mid) take = take && depth <= PULL_MAX_ECC;
      if (take && (test_memory() > 0 || pull_piece_bytes(c.n, c.nnz, bound) > PULL_ONE_LAUNCH)) {  // its state has to fit
        size_t free_b = 0;
        BCS_TRY(device_free_bytes(&free_b));
        take = pull_width(c.n, c.nnz, bound, free_b) > 0;
      }
      if (!take && !deep_ok) {  // (a chosen kernel's memory may be gone)
        rest.push_back(ci);
        continue;
      }
      if (tune_this) ctx.stats.tuned |= 1ll << (take ? LARGE_PATH_WIDE : LARGE_PATH_DEEP);
      if (po.sources) {  // the caller's sources
        std::vector<int32_t> h(po.nsources);
        for (int64_t i = 0; i < po.nsources; i++) h[i] = (int32_t)po.sources[i];
        BCS_CUDA(cudaMemcpyAsync(ord + c.n, h.data(), h.size() * sizeof(int32_t), cudaMemcpyHostToDevice, ctx.stream));
        BCS_CUDA(cudaStreamSynchronize(ctx.stream));
      }
      if (po.sources && take && po.nsources > 256)  // one slab's order is no matter
        BCS_TRY(sort_by_position(ctx, c.n, ord, ord + c.n, po.nsources));
      const int64_t src_off = po.sources ? off[k] + c.n : -1;
      if (take) pull.push_back(PullJob{ci, (int32_t)nsrc_of(c), bound, po.sources ? src_off : off[k]});
      else deep.push_back(DeepJob{ci, (int32_t)nsrc_of(c), bound, off[k], src_off});
    }
    large.swap(rest);
    int64_t rows = 0;
    auto shallow = [&](size_t k) { return cta_reached[k] == comps[cand[k]].n && cta_depth[k] <= MID_PIECE_ECC; };
    for (size_t k = nlarge; k < cand.size(); k++)
      if (shallow(k)) rows += pull_rows(comps[cand[k]]);
    for (size_t k = nlarge; k < cand.size(); k++) {
      const int32_t ci = cand[k];
      if (rows < MID_MIN_ROWS || !shallow(k)) to_small(ci);
      else pull.push_back(PullJob{ci, (int32_t)nsrc_of(comps[ci]), 2 * cta_depth[k] + 2, off[k]});
    }
  }
  // The small-path work split: a piece runs up to `ng_cap` sources at once
  // per CTA (the most that fit in SMALL_SMEM); the launch takes exactly the
  // shared memory its largest item needs, so occupancy follows the plan.
  // Items of similar cost go first-largest into a persistent queue.
  // pieces by cost class (the power of two of n + nnz), largest first, in
  // piece order within a class: the persistent queue hands out the longest
  // items first.  A counting sort: one pass, no comparisons.
  {
    int64_t cnt[65] = {0};
    std::vector<int32_t> cls(small.size());
    for (size_t k = 0; k < small.size(); k++) {
      const CompDesc &c = comps[small[k]];
      cls[k] = 63 - __builtin_clzll((unsigned long long)(c.nnz + c.n) | 1ull);
      cnt[cls[k]]++;
    }
    int64_t off[65], o = 0;
    for (int b = 64; b >= 0; b--) {
      off[b] = o;
      o += cnt[b];
    }
    std::vector<int32_t> sorted(small.size());
    for (size_t k = 0; k < small.size(); k++) sorted[off[cls[k]]++] = small[k];
    small.swap(sorted);
  }
  double coop_cost = 0.0;
  int64_t small_sources = 0;
  for (int32_t ci : small) {
    const CompDesc &c = comps[ci];
    if (c.maxdeg > SMALL_COOP_DEG && c.n > SMALL_COOP_N) coop_cost += (double)nsrc_of(c) * (double)(c.nnz + c.n);
    small_sources += nsrc_of(c);
  }
  const bool small_coop = coop_cost > 0.875 * total_small_cost;
  auto plan_small = [&](int ng_cap, size_t budget, std::vector<SmallItem> &out, size_t &smem, int &grid) -> int {
    out.clear();
    smem = 0;
    std::vector<int> ngs(small.size());
    // no more sources at once than leave every SM two items (a graph of 312
    // vertices: 83 us with seven at once on 45 SMs, 47 with one)
    ng_cap = (int)std::max<int64_t>(1, std::min<int64_t>(ng_cap, small_sources / (2 * (int64_t)ctx.num_sms)));
    for (size_t k = 0; k < small.size(); k++) {
      const CompDesc &c = comps[small[k]];
      int ng = 1;  // a piece that does not fit the budget even alone still runs (up to SMALL_SMEM)
      for (int cand = ng_cap; cand >= 1; cand--)
        if (small_takes(c.n, c.nnz, cand) && small_smem_bytes(c.n, c.nnz, cand, R, I) <= budget) {
          ng = cand;
          break;
        }
      ngs[k] = ng;
      smem = std::max(smem, small_smem_bytes(c.n, c.nnz, ng, R, I));
    }
    int per_sm = 1;
    BCS_TRY(small_ctas_per_sm(ctx, R, I, F, small_variant(ctx, F, small_coop, small_sources, smem), smem, &per_sm));
    grid = ctx.num_sms * per_sm;
    const double target = total_small_cost / (double)((int64_t)grid * 8) + 1.0;
    for (size_t k = 0; k < small.size(); k++) {
      const CompDesc &c = comps[small[k]];
      const int ng = ngs[k];
      const int64_t ns = nsrc_of(c);
      int64_t chunk = (int64_t)std::max(1.0, target / (double)(c.nnz + c.n));
      chunk = ((chunk + ng - 1) / ng) * ng;
      for (int64_t b = 0; b < ns; b += chunk)
        out.push_back(SmallItem{small[k], (int32_t)b, (int32_t)std::min<int64_t>(ns, b + chunk), ng});
    }
    grid = (int)std::min<int64_t>(grid, (int64_t)out.size());
    return BCS_OK;
  };
  nmax_large = 0;  // of what is left for the kernels below
  for (int32_t ci : large) nmax_large = std::max<int64_t>(nmax_large, comps[ci].n);
  for (int32_t ci : ms_tuned) nmax_large = std::max<int64_t>(nmax_large, comps[ci].n);
  for (int32_t ci : ps_tuned) nmax_large = std::max<int64_t>(nmax_large, comps[ci].n);
  // Large pieces: 32 sources per CTA when there are enough batches to give
  // every SM two of them and their scratch fits at least one CTA per SM,
  // else one source per CTA (more CTAs in flight).
  // BCS_LARGE_PATH=batched|per_source overrides the choice.
  int64_t nbatches = 0;
  for (int32_t ci : large) nbatches += (nsrc_of(comps[ci]) + 31) / 32;
  bool use_ms = !large.empty() && !dbg && !po.per_source_large && !po.srcmap && nbatches >= 2 * (int64_t)ctx.num_sms;
  if (use_ms) {
    // its per-CTA scratch grows with the piece: with fewer CTAs than SMs the
    // batches serialise (high-diameter graphs of millions of vertices)
    int64_t fit = 0;
    BCS_TRY(ms_ctas_that_fit(nmax_large, &fit));
    if (fit < ctx.num_sms) use_ms = false;
  }
  bool forced = false;  // a fixed large path (BCS_LARGE_PATH, or the caller's) overrides the choice
  if (!large.empty() && !dbg && !po.per_source_large && !po.srcmap) {
    if (lp_mode == LARGE_PATH_BATCHED) use_ms = forced = true;
    if (lp_mode == LARGE_PATH_PER_SOURCE) {
      use_ms = false;
      forced = true;
    }
  }
  // the one-source-per-CTA list for large pieces, from the `skip`-th source
  // of each piece on (debug output, the depth probe's remainder, or the
  // fallback when a graph is too deep for the 32-source kernel)
  // the sources of large pieces with a device source map, on the host
  std::vector<std::vector<int64_t>> large_map(po.srcmap ? large.size() : 0);
  if (po.srcmap) {
    for (size_t k = 0; k < large.size(); k++) {
      const CompDesc &c = comps[large[k]];
      if (c.src_off < 0) continue;
      large_map[k].resize(nsrc_of(c));
      if (!large_map[k].empty())
        BCS_CUDA(cudaMemcpyAsync(large_map[k].data(), po.srcmap + c.src_off, large_map[k].size() * sizeof(int64_t),
                                 cudaMemcpyDeviceToHost, ctx.stream));
    }
    BCS_CUDA(cudaStreamSynchronize(ctx.stream));
  }
  auto large_src = [&](size_t k, int64_t i) -> int32_t {
    if (po.sources) return (int32_t)po.sources[i];
    if (po.srcmap && comps[large[k]].src_off >= 0) return (int32_t)large_map[k][i];
    return (int32_t)i;
  };
  auto build_work = [&](int64_t skip) {
    work.clear();
    for (size_t k = 0; k < large.size(); k++) {
      const int64_t ns = nsrc_of(comps[large[k]]);
      for (int64_t i = skip; i < ns; i++) work.push_back(LargeSrc{large[k], large_src(k, i)});
    }
  };
  if (!use_ms) build_work(0);
  tr.mark("classify");
  int ng_cap = small_max_sources();
  size_t budget = SMALL_BUDGET;
  size_t smem_small = 0;
  int grid_small = 0;
  // the autotuner's choice for this shape bucket, if it has one already
  long long tune_key = 0;
  int tuned = 0;
  if (ctx.autotune && !small.empty()) {
    const int kb = 64 - __builtin_clzll((unsigned long long)std::max<int64_t>(nmax_small, 1));
    const int wb = (int)std::log2(std::max(total_small_cost, 1.0));
    tune_key = ((long long)(R * 4 + I * 2 + F) << 40) | ((long long)kb << 20) | (long long)wb;
    tuned = tuned_split(tune_key);
    if (tuned) {
      ng_cap = TUNE_SPLITS[tuned - 1].ng_cap;
      budget = TUNE_SPLITS[tuned - 1].budget;
    }
  }
  if (!small.empty()) BCS_TRY(plan_small(ng_cap, budget, items, smem_small, grid_small));
  tr.mark("plan0");
  ctx.stats.n_small_items = (int64_t)items.size();
  ctx.stats.n_large_sources = 0;
  for (int32_t ci : large) ctx.stats.n_large_sources += nsrc_of(comps[ci]);
  for (int32_t ci : ms_tuned) ctx.stats.n_large_sources += nsrc_of(comps[ci]);
  for (int32_t ci : ps_tuned) ctx.stats.n_large_sources += nsrc_of(comps[ci]);
  for (const PullJob &j : pull) ctx.stats.n_large_sources += j.nsrc;
  for (const DeepJob &j : deep) ctx.stats.n_large_sources += j.nsrc;
  for (const DeepJob &j : deep) ctx.stats.n_deep_sources += j.nsrc;
  ctx.stats.work_sources_entries = work_se;
  ctx.stats.work_sources_vertices = work_sv;
  if (small.empty() && large.empty() && pull.empty() && deep.empty() && ms_tuned.empty() && ps_tuned.empty()) return BCS_OK;

  DBuf<int> d_err;
  DBuf<unsigned long long> d_dag;
  BCS_TRY(d_err.alloc(4, ctx.stream));
  BCS_TRY(d_dag.alloc(1, ctx.stream));
  BCS_CUDA(cudaMemsetAsync(d_dag.p, 0, sizeof(unsigned long long), ctx.stream));
  BCS_CUDA(cudaMemsetAsync(d_err.p, 0, 4 * sizeof(int), ctx.stream));
  DBuf<int64_t> d_srcs;
  if (po.sources && !items.empty()) {
    BCS_TRY(d_srcs.alloc(po.nsources, ctx.stream));
    BCS_CUDA(cudaMemcpyAsync(d_srcs.p, po.sources, po.nsources * sizeof(int64_t), cudaMemcpyHostToDevice, ctx.stream));
  }
  tr.mark("upload");
  if (!items.empty()) {
    StageTimer tm(ctx.stream);
    tm.start();
    const size_t grid_cap = (size_t)ctx.num_sms * 8;  // resident CTAs per SM at most
    DBuf<int32_t> lvl;
    BCS_TRY(lvl.alloc(small_scratch_words(grid_cap, nmax_small), ctx.stream));
    DBuf<SmallItem> d_items;
    BCS_TRY(d_items.alloc(std::max<size_t>(items.size() * 2, 1), ctx.stream));
    auto run_small = [&](const std::vector<SmallItem> &its, size_t smem, int grid, double *target) -> int {
      if (its.size() > d_items.n) BCS_TRY(d_items.alloc(its.size(), ctx.stream));
      BCS_CUDA(cudaMemcpyAsync(d_items.p, its.data(), its.size() * sizeof(SmallItem), cudaMemcpyHostToDevice,
                               ctx.stream));
      BCS_CUDA(cudaMemsetAsync(d_err.p + 1, 0, sizeof(int), ctx.stream));
      BcInput tin = in;
      tin.bcp = target;
      return launch_small(ctx, F, small_variant(ctx, F, small_coop, small_sources, smem), grid, smem, d_items.p, (int)its.size(), d_err.p + 1, d_comps.p, tin,
                          po.sources ? d_srcs.p : po.srcmap, lvl.p, nmax_small, d_err.p, d_dag.p);
    };
    tr.mark("alloc");
    if (ctx.autotune && tuned == 0) {
      // tune once per shape bucket: time each split into a scratch
      // accumulator and keep the fastest
      int best = 0;
      {
        int64_t ntot = 0;
        for (const CompDesc &c : comps) ntot = std::max<int64_t>(ntot, c.vtx_off + c.n);
        DBuf<double> scratch;
        BCS_TRY(scratch.alloc(ntot, ctx.stream));
        double best_ms = 1e30;
        for (int cand = 0; cand < (int)(sizeof(TUNE_SPLITS) / sizeof(TUNE_SPLITS[0])); cand++) {
          std::vector<SmallItem> its;
          size_t sm = 0;
          int gr = 0;
          BCS_TRY(plan_small(TUNE_SPLITS[cand].ng_cap, TUNE_SPLITS[cand].budget, its, sm, gr));
          BCS_CUDA(cudaMemsetAsync(scratch.p, 0, ntot * 8, ctx.stream));
          StageTimer tt(ctx.stream);
          tt.start();
          BCS_TRY(run_small(its, sm, gr, scratch.p));
          const double ms = tt.stop_ms();
          if (std::getenv("BCS_TRACE"))
            std::fprintf(stderr, "[bcs] tune small split ng_cap=%d budget=%zu: %zu items, %d CTAs, %zu B smem, %.3f ms\n",
                         TUNE_SPLITS[cand].ng_cap, TUNE_SPLITS[cand].budget, its.size(), gr, sm, ms);
          if (ms < best_ms) {
            best_ms = ms;
            best = cand + 1;
          }
        }
        BCS_CUDA(cudaMemsetAsync(d_dag.p, 0, sizeof(unsigned long long), ctx.stream));
        remember_split(tune_key, best);
      }
      ng_cap = TUNE_SPLITS[best - 1].ng_cap;
      budget = TUNE_SPLITS[best - 1].budget;
      BCS_TRY(plan_small(ng_cap, budget, items, smem_small, grid_small));
      ctx.stats.n_small_items = (int64_t)items.size();
      tm.start();
    }
    tr.mark("plan");
    ctx.stats.small_ng_cap = ng_cap;
    ctx.stats.small_smem_budget = (int64_t)budget;
    BCS_TRY(run_small(items, smem_small, grid_small, in.bcp));
    tm.stop_into(ctx, &ctx.stats.ms_bcreach_small);
    tr.mark("small");
  }
  if (!pull.empty()) {
    StageTimer tm(ctx.stream);
    tm.start();
    int per_batch = 64;  // a quarter of a slab (for tests: an eighth)
    if (const char *e = std::getenv("BCS_WIDE_SOURCES"))
      if (lp_mode != LARGE_PATH_MID) per_batch = std::atoi(e) <= 32 ? 32 : 64;
    BCS_TRY(run_pull(ctx, comps, pull, in, F, pull_order.p, d_comps.p, per_batch, d_err.p, d_dag.p));
    tm.stop_into(ctx, &ctx.stats.ms_bcreach_large);
    tr.mark("pull");
  }
  for (const DeepJob &j : deep) {
    StageTimer tm(ctx.stream);
    tm.start();
    BCS_TRY(run_deep(ctx, comps[j.ci], in, F, pull_order.p + j.ord_off, pull_parent.p + j.ord_off, j.src_off < 0 ? nullptr : pull_order.p + j.src_off,
                     j.nsrc, j.depth_bound, d_err.p, d_dag.p));
    tm.stop_into(ctx, &ctx.stats.ms_bcreach_large);
    tr.mark("deep");
  }
  // one source per CTA over the given list; *d_lmax (optional) receives the
  // deepest BFS level any of them reached
  auto run_per_source = [&](const std::vector<LargeSrc> &w, int *d_lmax) -> int {
    StageTimer tm(ctx.stream);
    tm.start();
    DBuf<LargeSrc> d_work;
    DBuf<unsigned long long> counter;
    BCS_TRY(d_work.alloc(w.size(), ctx.stream));
    BCS_CUDA(cudaMemcpyAsync(d_work.p, w.data(), w.size() * sizeof(LargeSrc), cudaMemcpyHostToDevice, ctx.stream));
    BCS_TRY(counter.alloc(1, ctx.stream));
    BCS_CUDA(cudaMemsetAsync(counter.p, 0, sizeof(unsigned long long), ctx.stream));
    // CTAs: up to 3 per SM, fewer when the scratch would take more than half
    // of the free device memory
    size_t free_b = 0;
    BCS_TRY(device_free_bytes(&free_b));
    int64_t grid = (int64_t)ctx.num_sms * 3;
    grid = std::min<int64_t>(grid, (int64_t)w.size());
    const size_t per = large_scratch_bytes(nmax_large);
    if ((size_t)grid * per > free_b / 2) grid = std::max<int64_t>(1, (int64_t)(free_b / 2 / per));
    const size_t G = (size_t)grid, NM = (size_t)nmax_large;
    DBuf<int32_t> sd, sq, sls, sle;
    DBuf<double> ssig, scoef, sacc;
    BCS_TRY(sd.alloc(G * NM, ctx.stream));
    BCS_TRY(sq.alloc(G * NM, ctx.stream));
    BCS_TRY(ssig.alloc(G * NM, ctx.stream));
    BCS_TRY(scoef.alloc(G * NM, ctx.stream));
    BCS_TRY(sacc.alloc(G * NM, ctx.stream));
    BCS_TRY(sls.alloc(G * (NM + 2), ctx.stream));
    BCS_TRY(sle.alloc(G * (NM + 2), ctx.stream));
    BCS_CUDA(cudaMemsetAsync(sd.p, 0xFF, G * NM * sizeof(int32_t), ctx.stream));
    BCS_CUDA(cudaMemsetAsync(ssig.p, 0, G * NM * sizeof(double), ctx.stream));
    BCS_CUDA(cudaMemsetAsync(sacc.p, 0, G * NM * sizeof(double), ctx.stream));
    LargeScratch sc{sd.p, sq.p, ssig.p, scoef.p, sacc.p, sls.p, sle.p, (int64_t)NM};
    Debug dbgs{po.dbg_d, po.dbg_sig, po.dbg_exp, po.dbg_delta};
    BCS_TRY(BCS_DISPATCH3(launch_large_t, R, I, F, ctx, (int)grid, d_work.p, (int64_t)w.size(), counter.p, d_comps.p,
                          in, sc, d_err.p, dbgs, dbg ? 1 : 0, d_dag.p, d_lmax));
    tm.stop_into(ctx, &ctx.stats.ms_bcreach_large);
    return BCS_OK;
  };
  int64_t skip = 0;  // leading sources of each large piece already done
  if (use_ms && !forced) {
    // Depth probe: the first wave runs one source per CTA (useful work
    // either way) and reports how deep its BFS went.  The 32-source kernel
    // pays per BFS level and queues a vertex once per distinct level its
    // sources reach it at, so on deep graphs (roads, grids) the remaining
    // sources also run one per CTA.
    const int64_t wave = (int64_t)ctx.num_sms * 3;
    skip = std::max<int64_t>(1, wave / (int64_t)large.size());
    std::vector<LargeSrc> probe;
    for (size_t k = 0; k < large.size(); k++) {
      const int64_t ns = nsrc_of(comps[large[k]]);
      for (int64_t i = 0; i < std::min(ns, skip); i++) probe.push_back(LargeSrc{large[k], large_src(k, i)});
    }
    DBuf<int> d_lmax;
    BCS_TRY(d_lmax.alloc(1, ctx.stream));
    BCS_CUDA(cudaMemsetAsync(d_lmax.p, 0, sizeof(int), ctx.stream));
    BCS_TRY(run_per_source(probe, d_lmax.p));
    int lmax = 0;
    BCS_CUDA(cudaMemcpyAsync(&lmax, d_lmax.p, sizeof(int), cudaMemcpyDeviceToHost, ctx.stream));
    BCS_CUDA(cudaStreamSynchronize(ctx.stream));
    if (lmax > MS_DEPTH_LIMIT) {
      use_ms = false;
      build_work(skip);
    }
  }
  if (use_ms) {
    StageTimer tm(ctx.stream);
    tm.start();
    bool depth_failed = false;
    BCS_TRY(run_ms(ctx, comps, large, in, F, po.sources, po.nsources, skip, d_comps.p, d_err.p, d_dag.p,
                   &depth_failed));
    if (depth_failed) build_work(skip);
    tm.stop_into(ctx, &ctx.stats.ms_bcreach_large);
  }
  // the pieces the autotuner placed (every vertex a source)
  if (!ms_tuned.empty()) {
    StageTimer tm(ctx.stream);
    tm.start();
    bool depth_failed = false;
    BCS_TRY(run_ms(ctx, comps, ms_tuned, in, F, nullptr, 0, 0, d_comps.p, d_err.p, d_dag.p, &depth_failed));
    if (depth_failed) ps_tuned.insert(ps_tuned.end(), ms_tuned.begin(), ms_tuned.end());
    tm.stop_into(ctx, &ctx.stats.ms_bcreach_large);
  }
  for (int32_t ci : ps_tuned) {
    if (po.sources)
      for (int64_t i = 0; i < po.nsources; i++) work.push_back(LargeSrc{ci, (int32_t)po.sources[i]});
    else
      for (int32_t i = 0; i < comps[ci].n; i++) work.push_back(LargeSrc{ci, i});
  }
  if (!work.empty()) BCS_TRY(run_per_source(work, nullptr));
  int h_err = 0;
  unsigned long long h_dag = 0;
  BCS_CUDA(cudaMemcpyAsync(&h_err, d_err.p, sizeof(int), cudaMemcpyDeviceToHost, ctx.stream));
  BCS_CUDA(cudaMemcpyAsync(&h_dag, d_dag.p, sizeof(h_dag), cudaMemcpyDeviceToHost, ctx.stream));
  BCS_CUDA(cudaStreamSynchronize(ctx.stream));
  ctx.stats.dag_edges += (int64_t)h_dag;
  if (h_err & ERR_OVERFLOW) {
    set_error("shortest-path counts overflowed the FP64 range within one BFS level");
    return BCS_EOVERFLOW;
  }
  if (h_err & ERR_DEPTH) {
    set_error("a Bc-Reach batch needed more BFS levels than its bound");
    return BCS_ECUDA;
  }
  if (h_err & ERR_TIMEOUT) {
    set_error("a grid-wide wait of the Bc-Reach kernel ran out (opts->max_wait)");
    return BCS_ETIMEOUT;
  }
  return BCS_OK;
}

}  // namespace bcs
