// deep.cu - Bc-Reach (Algorithm 2 with the identical-vertex terms of
// Section 3.3.3) on deep pieces of small degree (roads, grids): many BFS
// levels, each of a few vertices per source.
//
// On such a piece no two sources reach a vertex on the same level, so a lane
// works on one (source, vertex) pair.  A CTA searches G sources at once, level
// by level, with one queue for the pairs of all of them: a level has enough
// pairs for every thread, and the wait after it is CTA-wide.
//
// The vertices are renumbered in preorder of a BFS tree of the piece: runs of
// numbers are runs of tree paths, compact in the graph (16 consecutive vertices
// of a road graph are at most 13 apart; 84 in the order of the BFS queue).  So
// the G sources of a CTA, consecutive numbers, reach a vertex within a few
// levels of each other, and with the sources of a vertex side by side its
// values are fetched once for all of them.  Per CTA, at vertex * G + source:
//   code  two bits: 0 not reached, else 1 + (BFS level mod 3); neighbours are
//         at most one level apart, so a neighbour's code tells the level above
//         from the same one and the one below.  In shared memory while
//         DEEP_MAX_G sources fit there, else in global memory;
//   S     path count times ident (exact int64 while the level's bound allows,
//         else FP64 with a power of two per (level, source)), replaced in
//         phase 2 by the coefficient of Eq. 3;
// and Q, the pairs in the order reached, a level after the other (the current
// level's first DEEP_RING in shared memory too).
//
// Phase 1, level L, one walk of each pair's row: the counts of its neighbours
// on level L-1 are summed; the others that are not on L are on L+1, and the
// ones not reached yet are claimed (an atomic OR: whoever claims writes the
// same code) and queued.  Phase 2, levels deepest first: a pair sums its
// successors' coefficients (Eq. 3 in the coefficient form of bcreach.cu).
//
// What bounds it: with many sources the FP64 pipe (half busy) and the latency of
// a level's chain of loads; with one source per CTA that chain alone (ring,
// row, codes, counts: about 5 us a level and phase).  On one GB300, whole calls:
// 20,929 vertices, every vertex a source, FP64 26 ms (one source per CTA 244 ms;
// queue places in place of codes, which cost a compare-and-swap and a scattered
// store per pair in L2, 33 ms); 456 sources on 682,544 vertices, FP32, 28 ms
// (146 ms).  Three CTAs of 512 threads: 62 KB of codes per CTA leave no L1 and
// measured 35 ms, 52 KB 22 ms, 42 KB 22.6 ms, two CTAs of 768 threads 27 ms
// (all for the kernel alone).

#include <cuda/atomic>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "bc_math.cuh"
#include "common.h"

namespace bcs {

constexpr int DEEP_THREADS = 512;
constexpr int DEEP_CTAS = 3;    // per SM
constexpr int DEEP_MAX_G = 16;  // sources per CTA
constexpr int DEEP_RING = 1024; // queue places of a level kept in shared memory
constexpr size_t DEEP_BYTES = (size_t)32 << 30;  // state of all CTAs
constexpr size_t DEEP_SMEM = 54 * 1024;  // codes in shared memory, per CTA (three to an SM, with L1 left)
constexpr int DEEP_PER_COPY = 48;  // sources to a copy of bc'
constexpr int DEEP_MORE = 1 << 31;  // flag on a row's first entry: more than four entries

struct DeepArgs {
  // the piece, renumbered: a row's first four entries (-1: none), and the rest
  // of the longer rows (xcol[xrow[v] .. xrow[v + 1]))
  const int4 *adj;
  const int64_t *xrow;
  const int32_t *xcol;
  const int32_t *ident;  // nullable
  const double *init;    // nullable: reach - 1
  const int32_t *src;    // the sources
  int32_t n, nsrc, G;
  int gs;               // a pair is queued as vertex << gs | source
  uint32_t words;       // code words of a CTA
  size_t cap;           // G * n
  uint32_t *code;       // codes in global memory (nullable: shared memory)
  uint32_t *Q;
  double *S;
  int32_t *lvl;         // [lcap + 2] first queue place of each level
  int32_t *exps;        // [lcap + 2][G] power of two taken off the counts of (level, source)
  int lcap, flg;
  double *acc;          // [copies][n] bc', by new id: a CTA adds to copy blockIdx.x mod copies
  int copies;
  const double *recip;  // reciprocals of the integers below RECIP_TABLE
  int *work;            // next source
  int *err;
  unsigned long long *dag_total;
};

// The sum of up to four FP64 values (has: which are present), the present ones
// moved to the front by integer selects: an FP64 instruction holds the pipe
// whatever its active lanes, and most pairs have one or two of the four, so a
// warp issues one or two additions in place of four.
__device__ __forceinline__ double deep_sum(const double *x, const bool *has, unsigned mask) {
  double p = has[0] ? x[0] : 0.0, q = 0.0, r = 0.0;
  int n = has[0];
#pragma unroll
  for (int j = 1; j < 3; j++)
    if (has[j]) {
      if (n == 0) p = x[j];
      else if (n == 1) q = x[j];
      else r = x[j];
      n++;
    }
  double t = 0.0;  // the fourth value, or the only ones left
  if (has[3]) {
    if (n == 0) p = x[3];
    else if (n == 1) q = x[3];
    else if (n == 2) r = x[3];
    else t = x[3];
    n++;
  }
  if (__any_sync(mask, n > 1)) p += q;
  if (__any_sync(mask, n > 2)) p += r;
  if (__any_sync(mask, n > 3)) p += t;
  return p;
}

template <bool REACH, bool IDENT, bool FP32, bool SHARED>
__global__ void __launch_bounds__(DEEP_THREADS, DEEP_CTAS) k_bcreach_deep(const __grid_constant__ DeepArgs A) {
  extern __shared__ uint32_t s_code[];
  __shared__ uint32_t s_ring[2][DEEP_RING];  // the level's pairs, and the next one's
  __shared__ unsigned long long s_max[DEEP_MAX_G];  // largest count of each source on the level, as bits
  __shared__ double s_ws[DEEP_MAX_G];
  __shared__ int s_drop[DEEP_MAX_G];  // power of two to take off when the level is summed
  __shared__ int s_exp[DEEP_MAX_G];   // what was taken off so far
  __shared__ int s_dexp[DEEP_MAX_G];  // phase 2: exponent of the level less that of the next
  __shared__ int s_first, s_tail, s_top;
  const int tid = threadIdx.x, lane = tid & 31;
  const size_t cta = blockIdx.x;
  uint32_t *const code = SHARED ? s_code : A.code + cta * (size_t)A.words;
  uint32_t *const Q = A.Q + cta * A.cap;
  double *const S = A.S + cta * A.cap;
  double *const acc = A.acc + (cta % A.copies) * (size_t)A.n;
  int32_t *const lvl = A.lvl + cta * (A.lcap + 2);
  int32_t *const exps = A.exps + cta * (size_t)(A.lcap + 2) * A.G;
  const uint32_t G = (uint32_t)A.G, gmask = (1u << A.gs) - 1u;
  unsigned long long dag = 0;
  unsigned edges = 0;  // shortest-path edges of the group at hand
  auto look = [&](uint32_t x) {  // the code at place x
    return (*(volatile uint32_t *)(code + (x >> 4)) >> (2 * (x & 15u))) & 3u;
  };
  auto claim = [&](uint32_t x, uint32_t c) {  // whether this thread is the first to reach place x
    const uint32_t sft = 2 * (x & 15u);
    return ((atomicOr(code + (x >> 4), c << sft) >> sft) & 3u) == 0u;
  };
  auto rest = [&](int64_t e, int64_t ee) {  // up to four entries of a long row
    return make_int4(e < ee ? __ldg(A.xcol + e) : -1, e + 1 < ee ? __ldg(A.xcol + e + 1) : -1,
                     e + 2 < ee ? __ldg(A.xcol + e + 2) : -1, e + 3 < ee ? __ldg(A.xcol + e + 3) : -1);
  };
  for (;;) {
    if (tid == 0) s_first = atomicAdd(A.work, A.G);
    for (uint32_t i = tid; i < A.words; i += DEEP_THREADS) code[i] = 0u;
    __syncthreads();
    const int first = s_first, cnt = min(A.G, A.nsrc - first);
    if (cnt <= 0) break;
    if (tid < cnt) {
      const int32_t v = __ldg(A.src + first + tid);
      const uint32_t x = (uint32_t)v * G + (uint32_t)tid;
      s_ring[0][tid] = Q[tid] = ((uint32_t)v << A.gs) | (uint32_t)tid;
      atomicOr(code + (x >> 4), 1u << (2 * (x & 15u)));
      ((long long *)S)[x] = 1;
      s_ws[tid] = (REACH ? __ldg(A.init + v) + 1.0 : 1.0) * (IDENT ? (double)__ldg(A.ident + v) : 1.0);
      s_drop[tid] = s_exp[tid] = 0;
      s_max[tid] = 0ull;
    }
    if (tid == 0) {
      s_tail = cnt;
      lvl[0] = 0;
      lvl[1] = cnt;
    }
    __syncthreads();
    // ---------------------------------------------------------- phase 1
    uint32_t lo = 0, hi = (uint32_t)cnt;
    int L = 0, lint = 1 << 30, blg = 0;  // lint: the first FP64 level; blg: log2 bound on the level's counts
    int lscale = 1 << 30;                // levels past this one have exponents
    uint32_t cc = 1u;                    // the level's code
    for (;;) {
      const bool kind = L < lint, kind_prev = L - 1 < lint, measure = !kind && blg > 900;
      const bool drop = L > lscale;
      const uint32_t cp = cc == 1u ? 3u : cc - 1u, cn = cc == 3u ? 1u : cc + 1u;  // the levels' beside it
      const uint32_t *const ring = s_ring[L & 1];
      uint32_t *const ring_next = s_ring[(L + 1) & 1];
      for (uint32_t i0 = lo + (tid & ~31); i0 < hi; i0 += DEEP_THREADS) {  // whole warps
        const uint32_t i = i0 + lane;
        const bool on = i < hi;
        uint32_t v = 0, g = 0;
        int4 a = make_int4(-1, -1, -1, -1);
        bool more = false;
        if (on) {
          const uint32_t it = i - lo < DEEP_RING ? ring[i - lo] : Q[i];
          v = it >> A.gs;
          g = it & gmask;
          a = __ldg(A.adj + v);
          more = a.x < -1;  // the flag on a vertex id
          a.x = a.x == -1 ? -1 : a.x & ~DEEP_MORE;
        }
        long long ai = 0;
        double ad = 0.0;
        // four neighbours (-1: none): sum, claim and queue (warp-collective)
        auto step = [&](const int4 &n4, bool first4) {
          const int32_t u[4] = {n4.x, n4.y, n4.z, n4.w};
          uint32_t q[4];
#pragma unroll
          for (int j = 0; j < 4; j++) q[j] = u[j] >= 0 ? look((uint32_t)u[j] * G + g) : cc;
          double x[4];
          bool pred[4];
#pragma unroll
          for (int j = 0; j < 4; j++) {
            x[j] = 0.0;
            pred[j] = q[j] == cp && L > 0;
            if (pred[j]) x[j] = S[(uint32_t)u[j] * G + g];
          }
          unsigned bm[4];
          bool won[4];
          int mine = 0, all = 0;
#pragma unroll
          for (int j = 0; j < 4; j++) {
            won[j] = q[j] == 0u && claim((uint32_t)u[j] * G + g, cn);
            edges += q[j] == 0u || q[j] == cn;
          }
#pragma unroll
          for (int j = 0; j < 4; j++) {  // queue what was claimed, one counter update per warp
            bm[j] = __ballot_sync(0xffffffffu, won[j]);
            mine += __popc(bm[j] & ((1u << lane) - 1u));
            all += __popc(bm[j]);
          }
          if (all) {
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_tail, all);
            at = __shfl_sync(0xffffffffu, at, 0) + mine;
#pragma unroll
            for (int j = 0; j < 4; j++)
              if (won[j]) {
                const uint32_t w = ((uint32_t)u[j] << A.gs) | g;
                Q[at] = w;
                if ((uint32_t)at - hi < DEEP_RING) ring_next[(uint32_t)at - hi] = w;
                at++;
              }
          }
          if (kind) {
#pragma unroll
            for (int j = 0; j < 4; j++) ai += __double_as_longlong(x[j]);
          } else {
            if (kind_prev) {
#pragma unroll
              for (int j = 0; j < 4; j++)
                if (pred[j]) x[j] = i64_to_f64_pos(__double_as_longlong(x[j]));
            }
            const double t = deep_sum(x, pred, 0xffffffffu);
            ad = first4 ? t : ad + t;
          }
        };
        step(a, true);
        if (__any_sync(0xffffffffu, more)) {
          int64_t e = 0, ee = 0;
          if (more) {
            e = __ldg(A.xrow + v);
            ee = __ldg(A.xrow + v + 1);
          }
          while (__any_sync(0xffffffffu, e < ee)) {
            step(rest(e, ee), false);
            e += 4;
          }
        }
        if (on && L > 0) {
          const uint32_t x = v * G + g;
          const int id = IDENT ? __ldg(A.ident + v) : 1;
          if (kind) {
            ((long long *)S)[x] = IDENT ? ai * id : ai;
          } else {
            if (drop) ad *= pow2_int(-s_drop[g]);
            if (IDENT && id != 1) ad *= (double)id;
            S[x] = ad;
            if (measure) atomicMax(s_max + g, (unsigned long long)__double_as_longlong(ad));
          }
        }
      }
      __syncthreads();
      const uint32_t tail = (uint32_t)s_tail;
      // the counts of level L+1: integers while the bound allows; the largest
      // counts are looked at when the bound nears the end of the double range
      if (L + 1 < lint && blg + A.flg >= 62) lint = L + 1;
      if (measure) {
        if (tid == 0) s_top = 0;
        __syncthreads();
        if (tid < cnt) {
          const unsigned long long m = s_max[tid];
          int lg = m ? (int)((m >> 52) & 0x7ff) - 1022 : 0;  // the count is below 2^lg
          if (lg > 1023) atomicOr(A.err, ERR_OVERFLOW);
          const int k = lg > 960 ? lg - 959 : 0;
          s_drop[tid] = k;
          s_max[tid] = 0ull;
          atomicMax(&s_top, lg - k);
        }
        __syncthreads();
        blg = s_top;
        if (lscale > L) lscale = L;
      } else if (drop || L == lscale) {
        if (tid < cnt) s_drop[tid] = 0;
      }
      if (L >= lscale && tid < cnt) s_exp[tid] += s_drop[tid];  // of level L+1
      if (tail == hi) break;
      if (L + 2 > A.lcap) {
        if (tid == 0) atomicOr(A.err, ERR_DEPTH);
        return;
      }
      blg += A.flg;
      if (L >= lscale && tid < cnt) exps[(size_t)(L + 1) * A.G + tid] = s_exp[tid];
      lo = hi;
      hi = tail;
      L++;
      cc = cn;
      if (tid == 0) lvl[L + 1] = (int32_t)hi;
      __syncthreads();
    }
    const int Lmax = L;
    dag += edges;
    edges = 0;
    __syncthreads();
    // ---------------------------------------------------------- phase 2
    uint32_t b = hi;  // end of the level
    for (int l = Lmax; l >= 1; l--) {
      const bool kind = l < lint;
      const uint32_t cn = cc == 3u ? 1u : cc + 1u;  // the next level's code
      const uint32_t s0 = (uint32_t)lvl[l];
      const bool sc = l >= lscale && l < Lmax;  // the level and the next may have other exponents
      const bool absolute = l > lscale;
      if (absolute || sc) {
        __syncthreads();
        if (tid < cnt) {
          s_exp[tid] = absolute ? exps[(size_t)l * A.G + tid] : 0;
          s_dexp[tid] = sc ? s_exp[tid] - exps[(size_t)(l + 1) * A.G + tid] : 0;
        }
        __syncthreads();
      }
      for (uint32_t i = s0 + tid; i < b; i += DEEP_THREADS) {
        const unsigned here = __activemask();  // the warp's lanes of the level (the last warp may be partial)
        const uint32_t it = Q[i];
        const uint32_t v = it >> A.gs, g = it & gmask;
        int4 a = __ldg(A.adj + v);
        const double own = S[v * G + g];
        const bool more = a.x < -1;
        a.x = a.x == -1 ? -1 : a.x & ~DEEP_MORE;
        const int32_t u[4] = {a.x, a.y, a.z, a.w};
        double x[4];
        bool su[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
          su[j] = l < Lmax && u[j] >= 0 && look((uint32_t)u[j] * G + g) == cn;
          x[j] = 0.0;
          if (su[j]) x[j] = S[(uint32_t)u[j] * G + g];
        }
        const int id = IDENT ? __ldg(A.ident + v) : 1;
        int ev = 0;
        float mv = 1.0f;
        double sv = 1.0;
        int idx = 0;  // the count, if it is an integer in the table of reciprocals
        if (kind) {
          long long c = __double_as_longlong(own);
          if (IDENT && id != 1) c /= id;  // exact: the stored count is a multiple of ident
          if (FP32) {
            split_pow2_i64(c, ev, mv);
          } else {
            idx = c < RECIP_TABLE ? (int)c : 0;
            sv = i64_to_f64_pos(c);
          }
        } else {
          sv = IDENT && id != 1 ? own / (double)id : own;
          if (FP32) split_pow2(sv, ev, mv);
        }
        if (FP32 && absolute) ev += s_exp[g];
        double sum = 0.0;
        float sumf = 0.0f;
        auto add = [&](double c) {
          if (!FP32) {
            sum += c;
          } else {
            const int d = ev - __double2hiint(c);  // <= 0: sigma[v] <= sigma[w]
            if (d >= -126) sumf = fmaf(__int_as_float(__double2loint(c)), __int_as_float((127 + d) << 23), sumf);
          }
        };
        if (!FP32) {
          sum = deep_sum(x, su, here);
        } else {
#pragma unroll
          for (int j = 0; j < 4; j++)
            if (su[j]) add(x[j]);
        }
        if (more && l < Lmax) {
          const int64_t ee = __ldg(A.xrow + v + 1);
          for (int64_t e = __ldg(A.xrow + v); e < ee; e += 4) {
            const int4 r = rest(e, ee);
            const int32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
            for (int j = 0; j < 4; j++)
              if (w[j] >= 0 && look((uint32_t)w[j] * G + g) == cn) add(S[(uint32_t)w[j] * G + g]);
          }
        }
        if (!FP32) {
          if (sc) sum *= pow2_int(s_dexp[g]);
          const double d = REACH ? fma(sv, sum, __ldg(A.init + v)) : sv * sum;
          if (l > 1) {  // the sources' own dependencies are not needed
            const double r = idx ? __ldg(A.recip + idx) : recip_pos(sv);
            const double kr = IDENT && id != 1 ? (double)id * r : r;
            S[v * G + g] = fma(d, kr, kr);
          }
          atomicAdd(acc + v, s_ws[g] * d);
        } else {
          const float d = fmaf(mv, sumf, REACH ? (float)__ldg(A.init + v) : 0.0f), kv = (float)id;
          if (l > 1) S[v * G + g] = __hiloint2double(ev, __float_as_int(fmaf(kv, d, kv) / mv));
          atomicAdd(acc + v, s_ws[g] * (double)d);
        }
      }
      __syncthreads();
      b = s0;
      cc = cc == 1u ? 3u : cc - 1u;
    }
  }
  for (int o = 16; o > 0; o >>= 1) dag += __shfl_xor_sync(0xffffffffu, dag, o);
  if (lane == 0 && dag) atomicAdd(A.dag_total, dag);
}

// Preorder of the BFS tree (parent[v], -1 at the roots; order: the vertices in
// BFS order, a component after the other, its root first): subtree sizes and
// each child's offset among its siblings, bottom-up (a vertex is passed on by
// whichever child completes it last), then every vertex walks up until it
// meets an ancestor that has its number.
__global__ void k_deep_children(int32_t n, const int32_t *__restrict__ parent, int32_t *nchild) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    if (parent[v] >= 0) atomicAdd(nchild + parent[v], 1);
}

__global__ void k_deep_sizes(int32_t n, const int32_t *__restrict__ parent, const int32_t *__restrict__ nchild,
                             int32_t *done, int32_t *cursor, int32_t *off) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (nchild[i] != 0) continue;
    int32_t v = i, size = 1;
    for (int32_t p = parent[v]; p >= 0; p = parent[v]) {
      off[v] = atomicAdd(cursor + p, size);
      // the last child to arrive sees every sibling's size
      cuda::atomic_ref<int32_t, cuda::thread_scope_device> d(done[p]);
      if (d.fetch_add(1, cuda::memory_order_acq_rel) + 1 != nchild[p]) break;
      size = 1 + *(volatile int32_t *)(cursor + p);
      v = p;
    }
  }
}

__global__ void k_deep_preorder(int32_t n, const int32_t *__restrict__ order, const int32_t *__restrict__ parent,
                                const int32_t *__restrict__ off, int32_t *pre) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int32_t v = order[i];
    int32_t acc = 0, a = v;
    for (;;) {
      const int32_t p = parent[a];
      if (p < 0) {  // a root: its place in the order
        acc += a == v ? i : *(volatile int32_t *)(pre + a);
        break;
      }
      acc += 1 + off[a];
      const int32_t pp = *(volatile int32_t *)(pre + p);
      if (pp >= 0) {
        acc += pp;
        break;
      }
      a = p;
    }
    *(volatile int32_t *)(pre + v) = acc;
  }
}

// the roots' numbers first: the walks end there
__global__ void k_deep_roots(int32_t n, const int32_t *__restrict__ order, const int32_t *__restrict__ parent,
                             int32_t *pre) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int32_t v = order[i];
    pre[v] = parent[v] < 0 ? i : -1;
  }
}

__global__ void k_deep_order(int32_t n, const int32_t *__restrict__ inv, const int64_t *__restrict__ row, int32_t *order,
                             int64_t *extra) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    order[inv[v]] = v;
    const int64_t d = row[v + 1] - row[v];
    extra[inv[v]] = d > 4 ? d - 4 : 0;
    if (v == 0) extra[n] = 0;
  }
}

// the renumbered piece: rows, weights, and every vertex as a source
__global__ void k_deep_rows(int32_t n, const int32_t *__restrict__ order, const int32_t *__restrict__ inv,
                            const int64_t *__restrict__ row, const int32_t *__restrict__ col,
                            const int64_t *__restrict__ xrow, int32_t *xcol, const int32_t *__restrict__ reach,
                            const double *__restrict__ init_f, const int32_t *__restrict__ ident, int4 *adj,
                            double *init, int32_t *id, int32_t *src) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int32_t v = order[i];
    const int64_t b = row[v], d = row[v + 1] - b;
    int32_t u[4];
#pragma unroll
    for (int j = 0; j < 4; j++) u[j] = j < d ? inv[col[b + j]] : -1;
    if (d > 4) u[0] |= DEEP_MORE;
    adj[i] = make_int4(u[0], u[1], u[2], u[3]);
    for (int64_t e = 4; e < d; e++) xcol[xrow[i] + e - 4] = inv[col[b + e]];
    if (init) init[i] = init_f ? init_f[v] : (double)(reach[v] - 1);
    if (id) id[i] = ident[v];
    if (src) src[i] = i;
  }
}

__global__ void k_deep_sources(int32_t k, const int32_t *__restrict__ given, const int32_t *__restrict__ inv,
                               int32_t *src) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < k; i += gridDim.x * blockDim.x) src[i] = inv[given[i]];
}

__global__ void k_deep_add(int32_t n, const int32_t *__restrict__ order, const double *__restrict__ acc, int copies,
                           double *bcp) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double t = 0.0, lost = 0.0;  // what the additions round off is kept (hundreds of copies)
    for (int c = 0; c < copies; c++) {
      const double a = acc[(size_t)c * n + i], sum = t + a, of_a = sum - t;
      lost += (t - (sum - of_a)) + (a - of_a);
      t = sum;
    }
    t += lost;
    if (t != 0.0) bcp[order[i]] += t;
  }
}

template <bool R, bool I, bool F>
static int deep_launch_t(Ctx &ctx, int grid, size_t smem, const DeepArgs &A) {
  if (smem) {
    BCS_CUDA(cudaFuncSetAttribute(k_bcreach_deep<R, I, F, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DEEP_SMEM));
    k_bcreach_deep<R, I, F, true><<<grid, DEEP_THREADS, smem, ctx.stream>>>(A);
  } else {
    k_bcreach_deep<R, I, F, false><<<grid, DEEP_THREADS, 0, ctx.stream>>>(A);
  }
  ctx.launches++;
  BCS_CUDA(cudaGetLastError());
  return BCS_OK;
}

// bytes of one CTA's state with G sources (codes in global memory)
static size_t deep_cta_bytes(int64_t n, int depth_bound, int64_t G) {
  return (size_t)(G * 12 + 8) * (size_t)n + ((size_t)n * G + 15) / 16 * 4 + ((size_t)depth_bound + 6) * 4 * (size_t)(G + 1);
}

bool deep_takes(const CompDesc &c, int depth_bound, size_t free_bytes) {
  return c.maxdeg <= DEEP_MAX_DEG && c.n < (1 << 30) && depth_bound < (1 << 30) &&
         16 * deep_cta_bytes(c.n, depth_bound, 1) <= free_bytes / 2;
}

int run_deep(Ctx &ctx, const CompDesc &c, const BcInput &in, bool fp32, const int32_t *d_bfs, const int32_t *d_parent,
             const int32_t *d_sources, int32_t nsrc, int depth_bound, int *d_err, unsigned long long *d_dag) {
  if (nsrc <= 0) return BCS_OK;
  const cudaStream_t s = ctx.stream;
  const int64_t n = c.n;
  const bool R = in.reach != nullptr || in.init != nullptr, I = in.ident != nullptr;
  // enough sources per CTA that one round of CTAs takes them all, as far as
  // memory and the 32-bit pair ids allow
  size_t free_b = 0;
  BCS_TRY(device_free_bytes(&free_b));
  const size_t budget = std::min<size_t>(free_b / 2, DEEP_BYTES);
  int64_t grid = std::min<int64_t>((int64_t)ctx.num_sms * DEEP_CTAS, nsrc);
  grid = std::max<int64_t>(1, std::min<int64_t>(grid, (int64_t)(budget / deep_cta_bytes(n, depth_bound, 1))));
  // a level of a CTA should have a pair for every thread (a source's levels are
  // about n over three quarters of the bound wide)
  const int64_t width = std::max<int64_t>(1, n / std::max<int64_t>(1, (int64_t)depth_bound * 3 / 4));
  const int64_t want = std::max<int64_t>(1, (DEEP_THREADS + DEEP_THREADS / 2) / width);
  int64_t G = std::min<int64_t>(std::min<int64_t>(DEEP_MAX_G, want), (nsrc + grid - 1) / grid);
  G = std::max<int64_t>(1, std::min<int64_t>(G, ((int64_t)1 << 31) / n));
  const int64_t fit = (int64_t)DEEP_SMEM * 4 / n;  // sources whose codes fit shared memory
  if (fit < G && fit >= (G + 1) / 2) G = fit;
  while (G > 1 && (size_t)grid * deep_cta_bytes(n, depth_bound, G) > budget) G--;
  const int64_t rounds = (nsrc + grid * G - 1) / (grid * G);
  G = (nsrc + grid * rounds - 1) / (grid * rounds);  // rounds of equal size
  int gs = 0;
  while ((1 << gs) < G) gs++;
  const size_t words = ((size_t)n * G + 15) / 16;
  const bool shared = words * 4 <= DEEP_SMEM;
  DeepArgs A;
  std::memset(&A, 0, sizeof(A));
  DBuf<int4> adj;
  DBuf<int32_t> inv, order, id, src, lvl, exps, work, nchild, done, cursor, off, xcol;
  DBuf<int64_t> extra, xrow, tot;
  DBuf<double> init, acc, S;
  DBuf<uint32_t> code, Q;
  BCS_TRY(inv.alloc(n, s));
  BCS_TRY(order.alloc(n, s));
  BCS_TRY(nchild.alloc(n, s));
  BCS_TRY(done.alloc(n, s));
  BCS_TRY(cursor.alloc(n, s));
  BCS_TRY(off.alloc(n, s));
  BCS_TRY(extra.alloc(n + 1, s));
  BCS_TRY(xrow.alloc(n + 1, s));
  BCS_TRY(tot.alloc(1, s));
  BCS_TRY(xcol.alloc(c.nnz, s));
  BCS_TRY(adj.alloc(n, s));
  // A sum over all sources in one accumulator would round tens of thousands of
  // times: one copy per DEEP_PER_COPY sources, added up at the end (20,000
  // sources: error 1e-14 in one, 5e-16 in copies)
  A.copies = (int)std::max<int64_t>(1, std::min<int64_t>(grid, (nsrc + DEEP_PER_COPY - 1) / DEEP_PER_COPY));
  BCS_TRY(acc.alloc((size_t)A.copies * n, s));
  if (R) BCS_TRY(init.alloc(n, s));
  if (I) BCS_TRY(id.alloc(n, s));
  BCS_TRY(src.alloc(d_sources ? nsrc : n, s));
  A.lcap = depth_bound + 2;
  A.G = (int32_t)G;
  A.words = (uint32_t)words;
  A.cap = (size_t)G * n;
  if (!shared) BCS_TRY(code.alloc((size_t)grid * words, s));
  BCS_TRY(Q.alloc((size_t)grid * A.cap, s));
  BCS_TRY(S.alloc((size_t)grid * A.cap, s));
  BCS_TRY(lvl.alloc((size_t)grid * (A.lcap + 2), s));
  BCS_TRY(exps.alloc((size_t)grid * (A.lcap + 2) * G, s));
  BCS_TRY(work.alloc(1, s));
  BCS_CUDA(cudaMemsetAsync(acc.p, 0, (size_t)A.copies * n * sizeof(double), s));
  BCS_CUDA(cudaMemsetAsync(work.p, 0, sizeof(int32_t), s));
  const int64_t *row = in.row + c.row_off;
  const int blocks = (int)std::min<int64_t>((n + 255) / 256, (int64_t)ctx.num_sms * 8);
  const int32_t ni = (int32_t)n;
  BCS_CUDA(cudaMemsetAsync(nchild.p, 0, n * sizeof(int32_t), s));
  BCS_CUDA(cudaMemsetAsync(done.p, 0, n * sizeof(int32_t), s));
  BCS_CUDA(cudaMemsetAsync(cursor.p, 0, n * sizeof(int32_t), s));
  k_deep_children<<<blocks, 256, 0, s>>>(ni, d_parent, nchild.p);
  k_deep_roots<<<blocks, 256, 0, s>>>(ni, d_bfs, d_parent, inv.p);
  k_deep_sizes<<<blocks, 256, 0, s>>>(ni, d_parent, nchild.p, done.p, cursor.p, off.p);
  k_deep_preorder<<<blocks, 256, 0, s>>>(ni, d_bfs, d_parent, off.p, inv.p);
  k_deep_order<<<blocks, 256, 0, s>>>(ni, inv.p, row, order.p, extra.p);
  ctx.launches += 5;
  BCS_CUDA(cudaGetLastError());
  BCS_TRY(launch_exclusive_scan(ctx, extra.p, xrow.p, n + 1, tot.p));
  k_deep_rows<<<blocks, 256, 0, s>>>(ni, order.p, inv.p, row, in.col, xrow.p, xcol.p,
                                     in.reach && !in.init ? in.reach + c.vtx_off : nullptr,
                                     in.init ? in.init + c.vtx_off : nullptr, I ? in.ident + c.vtx_off : nullptr, adj.p,
                                     init.p, id.p, d_sources ? nullptr : src.p);
  ctx.launches++;
  if (d_sources) {
    k_deep_sources<<<(nsrc + 255) / 256, 256, 0, s>>>(nsrc, d_sources, inv.p, src.p);
    ctx.launches++;
  }
  BCS_CUDA(cudaGetLastError());
  A.adj = adj.p;
  A.ident = id.p;
  A.init = init.p;
  A.src = src.p;
  A.xrow = xrow.p;
  A.xcol = xcol.p;
  A.n = (int32_t)n;
  A.nsrc = nsrc;
  A.gs = gs;
  A.code = code.p;
  A.Q = Q.p;
  A.S = S.p;
  A.lvl = lvl.p;
  A.exps = exps.p;
  // a level's stored counts grow by the degree and by ident (at most a degree) per level
  int f = 0;
  while ((double)((int64_t)1 << f) < c.fan) f++;
  A.flg = std::max(1, I ? 2 * f : f);
  A.acc = acc.p;
  BCS_TRY(recip_table(ctx, &A.recip));
  A.work = work.p;
  A.err = d_err;
  A.dag_total = d_dag;
  BCS_TRY(BCS_DISPATCH3(deep_launch_t, R, I, fp32, ctx, (int)grid, shared ? words * 4 : 0, A));
  k_deep_add<<<blocks, 256, 0, s>>>(ni, order.p, acc.p, A.copies, in.bcp + c.vtx_off);
  ctx.launches++;
  BCS_CUDA(cudaGetLastError());
  if (std::getenv("BCS_TRACE"))
    std::fprintf(stderr, "[bcs trace] deep: n=%lld, %d sources on %lld CTAs, %lld at a time each (codes in %s memory), depth at most %d\n",
                 (long long)n, nsrc, (long long)grid, (long long)G, shared ? "shared" : "global", depth_bound);
  return BCS_OK;
}

}  // namespace bcs
