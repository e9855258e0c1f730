// small.cu - Bc-Reach (Algorithm 2 with the identical-vertex terms of
// Section 3.3.3) over many pieces that fit shared memory, one persistent
// launch.
//
// A CTA takes an item (a piece and a range of its sources), loads the piece
// and searches G of its sources at a time, level by level with CTA-wide waits.
// A lane works on one (vertex, source) pair of the level, whichever source it
// belongs to, from one queue for all G: BFS levels of small pieces are short,
// and a warp per source left half of its lanes idle.
//
// In shared memory, per vertex code, one word: two bits per source, 0 not
// reached, else 1 + (BFS level mod 3).  Neighbours are at most one level apart,
// so a neighbour's code tells the level above from the same one and the one
// below.  At place vertex * G + source:
//   S     path count times ident (exact int64 while the level's bound allows,
//         else FP64 with a power of two per (level, source)), replaced in
//         phase 2 by the coefficient of Eq. 3;
//   succ  the pair's successors among its row's first 32 entries, as bits;
//   acc   the pair's bc' terms over some rounds of sources (then added up over
//         the G places of a vertex: one FP64 atomic for all of them);
// and the queue of pairs, a level after the other.
//
// Phase 1, level L, one walk of each pair's row: the counts of its neighbours
// on level L-1 are summed (integer adds), the others that are not on L are on
// L+1, and the ones not reached yet are claimed (an atomic OR: whoever claims
// writes the same code) and queued.  Phase 2, levels deepest first: a pair sums
// its successors' coefficients over the set bits (an FP64 instruction holds
// the pipe whatever its active lanes, so the loop runs over successors, not
// entries), delta = reach - 1 + sigma * sum, c = ident (1 + delta) / sigma.
//
// Bound by issue (54 %) and the waits between short levels: 22 bytes of state
// per pair leave some 300 pairs of a level in flight per CTA.  On the
// articulation-vertex workload (130 M pairs, 788 M row entries) 5.0 ms against
// 7.1 with a group of warps per source, four groups at most and 100 KB; 10
// warps per CTA take 5.02, 8 take 5.14, 12 or 16 with more memory 5.11 and
// 5.76; rows padded to four entries took 5.7 (the padding costs sources).
#include <algorithm>
#include <map>
#include <mutex>
#include <set>
#include <type_traits>

#include "bc_math.cuh"
#include "common.h"

namespace bcs {

constexpr int SMALL_THREADS = 320;
constexpr int SMALL_GLOBAL_THREADS = 512;
constexpr int SMALL_LONGS = 8;    // long rows of a warp's pairs taken by the whole warp, at most
constexpr int SMALL_MAX_G = 16;   // sources per CTA at once, at most (two bits each in a word)
// rounds of G sources between additions to bc': both chains of additions stay short
__host__ __device__ constexpr int small_flush(bool global) { return global ? 64 : 16; }
constexpr int FIXED_COPIES = 32;  // of bc', in the fixed-scratch launch
constexpr int SMALL_LEVELS = 64;  // level offsets kept in shared memory, the rest in global scratch

int small_max_sources() { return SMALL_MAX_G; }

// SMALL_COOP: where a warp's pairs have at most SMALL_LONGS rows of more than 32
// entries, the warp takes those together: a hub's row taken by one lane holds
// up the level.  Where no row is long the ballots and the registers cost more
// than they give (articulation-vertex workload: 5.0 ms without, 6.2 with).
// SMALL_FOUR: four CTAs per SM.  With FP32 dependencies it takes 56 registers by
// itself, three CTAs, which is the faster where there is work for many rounds
// (articulation-vertex workload 5.42 ms, 5.48 with four), but not for one or two
// (a ring of 500, one source per CTA: 0.62 and 0.39).
// GLOBAL (a piece above shared memory, G = 1): codes and queue in shared
// memory, the counts and sums in global memory (`state`), the rows the caller's.
template <bool REACH, bool IDENT, bool FP32, int VARIANT, bool GLOBAL>
__global__ void __launch_bounds__(GLOBAL ? SMALL_GLOBAL_THREADS : SMALL_THREADS, GLOBAL ? 2 : VARIANT != SMALL_PLAIN ? 4 : 0) k_bcreach_small(
    const SmallItem *__restrict__ items, int nitems, int *item_counter, const CompDesc *__restrict__ comps,
    const int64_t *__restrict__ g_row, const int32_t *__restrict__ g_col, const int32_t *__restrict__ g_reach,
    const int32_t *__restrict__ g_ident, const double *__restrict__ g_init, const int64_t *__restrict__ srcs,
    const double *__restrict__ recip, double *bcp, size_t bcp_stride, int32_t *lvl_scratch, int lvl_stride, int lvl_G,
    unsigned char *state, size_t state_stride, int *err, unsigned long long *dag_total) {
  constexpr bool COOP = VARIANT == SMALL_COOP;
  constexpr int NT = GLOBAL ? SMALL_GLOBAL_THREADS : SMALL_THREADS;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long s_max[SMALL_MAX_G];  // largest count of each source on the level, as bits
  __shared__ double s_ws[SMALL_MAX_G];
  __shared__ int s_drop[SMALL_MAX_G];  // power of two to take off when the level is summed
  __shared__ int s_exp[SMALL_MAX_G];   // what was taken off so far
  __shared__ int s_dexp[SMALL_MAX_G];  // phase 2: exponent of the level less that of the next
  __shared__ int s_lvl[SMALL_LEVELS];
  __shared__ int s_item, s_tail, s_top;
  const int tid = threadIdx.x, lane = tid & 31;
  const int tid0 = COOP ? tid & ~31 : tid;  // COOP: whole warps run through a level together
  int32_t *const lvl_far = lvl_scratch + (size_t)blockIdx.x * lvl_stride * (lvl_G + 1);
  int32_t *const exps = lvl_far + lvl_stride;  // [level][G]
  double *const bcp_cta = bcp + bcp_stride * (blockIdx.x % FIXED_COPIES);  // stride 0: one bc' for all
  unsigned long long dag = 0;
  for (;;) {
    if (tid == 0) s_item = atomicAdd(item_counter, 1);
    __syncthreads();
    const int it_no = s_item;
    if (it_no >= nitems) break;
    const SmallItem item = items[it_no];
    const CompDesc c = comps[item.comp];
    const int n = c.n, nnz = (int)c.nnz;
    const uint32_t G = (uint32_t)item.ngroups;
    const int gs = 32 - __clz((int)G - 1);  // ceil(log2 G) (G = 1: 0)
    const uint32_t gmask = (1u << gs) - 1u;
    unsigned char *p = GLOBAL ? state + state_stride * blockIdx.x : smem;
    uint16_t *row = nullptr, *col = nullptr;
    if (!GLOBAL) {
      row = (uint16_t *)p;
      p += align16((size_t)(n + 1) * 2);
      col = (uint16_t *)p;
      p += align16((size_t)(nnz + 3) * 2);
    }
    auto row_of = [&](uint32_t v) -> int { return GLOBAL ? (int)__ldg(g_row + v) : (int)row[v]; };
    auto col_at = [&](int e) -> uint32_t { return GLOBAL ? (uint32_t)__ldg(g_col + e) : (uint32_t)col[e]; };
    double *init = nullptr;
    int32_t *ident = nullptr;
    if (REACH) {
      init = (double *)p;
      p += align16((size_t)n * 8);
    }
    if (IDENT) {
      ident = (int32_t *)p;
      p += align16((size_t)n * 4);
    }
    uint32_t *const code = (uint32_t *)(GLOBAL ? smem : p);
    if (!GLOBAL) p += align16((size_t)n * 4);
    const size_t pairs = (size_t)n * G;
    double *const S = (double *)p;
    long long *const Si = (long long *)p;
    p += align16(pairs * 8);
    double *const acc = (double *)p;
    p += align16(pairs * 8);
    uint32_t *const succ_of = (uint32_t *)p;
    p += align16(pairs * 4);
    uint16_t *const Q = (uint16_t *)(GLOBAL ? smem + align16((size_t)n * 4) : p);
    if (!GLOBAL) {
      const int64_t *const grow = g_row + c.row_off;
      const int64_t r0 = grow[0];
      for (int v = tid; v <= n; v += NT) row[v] = (uint16_t)(grow[v] - r0);
      for (int e = tid; e < nnz + 3; e += NT) col[e] = e < nnz ? (uint16_t)__ldg(g_col + r0 + e) : (uint16_t)0;
    }
    for (int v = tid; v < n; v += NT) {
      if (REACH) init[v] = g_init ? g_init[c.vtx_off + v] : (double)(g_reach[c.vtx_off + v] - 1);
      if (IDENT) ident[v] = g_ident[c.vtx_off + v];
    }
    for (uint32_t x = tid; x < (uint32_t)pairs; x += NT) acc[x] = 0.0;
    // bound on the growth of a level's stored counts: the degree, and ident (at most a degree)
    const int flg = max(1, ceil_log2_pos(c.fan) * (IDENT ? 2 : 1));
    int rounds = 0;
    for (int first = item.s_begin; first < item.s_end; first += (int)G) {
      const int cnt = min((int)G, item.s_end - first);
      for (int i = tid; i < n; i += NT) code[i] = 0u;
      __syncthreads();  // the piece is loaded; the codes are clear
      if (tid < cnt) {
        const int i = first + tid;
        const uint32_t v = (uint32_t)((srcs && c.src_off >= 0) ? (int32_t)srcs[c.src_off + i] : i);
        const uint32_t x = v * G + (uint32_t)tid;
        Q[tid] = (uint16_t)((v << gs) | (uint32_t)tid);
        atomicOr(code + v, 1u << (2 * tid));
        Si[x] = 1;
        s_ws[tid] = (REACH ? init[v] + 1.0 : 1.0) * (IDENT ? (double)ident[v] : 1.0);
        s_drop[tid] = s_exp[tid] = 0;
        s_max[tid] = 0ull;
      }
      if (tid == 0) {
        s_tail = cnt;
        s_lvl[0] = 0;
        s_lvl[1] = cnt;
      }
      __syncthreads();
      // -------------------------------------------------------- phase 1
      int lo = 0, hi = cnt, L = 0;
      int lint = 1 << 30, blg = 0;  // the first FP64 level; log2 bound on the level's counts
      int lscale = 1 << 30;         // levels past this one have exponents
      uint32_t cc = 1u;             // the level's code
      unsigned edges = 0;
      for (;;) {
        const bool kind = L < lint, kind_prev = L - 1 < lint, measure = !kind && blg > 900;
        const bool drop = L > lscale;
        const uint32_t cp = cc == 1u ? 3u : cc - 1u, cn = cc == 3u ? 1u : cc + 1u;  // the levels' beside it
        // mode 0: integer counts, 1: FP64 from the integers of the level above, 2: FP64
        auto pass = [&](auto mode) {
          constexpr int MODE = decltype(mode)::value;
          for (int i0 = lo + tid0; i0 < hi; i0 += NT) {
            const int i = COOP ? i0 + lane : i0;
            const bool valid = !COOP || i < hi;
            const uint32_t it = valid ? Q[i] : 0u, v = it >> gs, g = it & gmask, x = v * G + g;
            const uint32_t sh = 2 * g, field = 3u << sh, above = cp << sh, same = cc << sh;
            const int rb = valid ? row_of(v) : 0, re = valid ? row_of(v + 1) : 0;
            unsigned longs = COOP ? __ballot_sync(0xffffffffu, re - rb > 32) : 0u;
            if (COOP && __popc(longs) > SMALL_LONGS) longs = 0u;
            long long ai = 0;
            double ad = 0.0;
            uint32_t succ0 = 0u;
            auto claim = [&](uint32_t u, uint32_t g, uint32_t field) {  // the first to set the bits has claimed the vertex
              if ((atomicOr(code + u, cn << (2 * g)) & field) == 0u)
                Q[atomicAdd(&s_tail, 1)] = (uint16_t)((u << gs) | g);
            };
            if (!(longs >> lane & 1u)) {
              const double *const Sg = S + g;
              for (int e0 = rb; e0 < re; e0 += 32) {
                uint32_t succ = 0u, open = 0u;  // on the level below, and of these not reached yet
                const int e1 = min(re, e0 + 32);
                for (int e = e0; e < e1; e += 4) {
                  uint32_t u[4], f[4];  // past the row's end: taken as on the level at hand
#pragma unroll
                  for (int j = 0; j < 4; j++) u[j] = col_at(GLOBAL ? min(e + j, e1 - 1) : e + j);
#pragma unroll
                  for (int j = 0; j < 4; j++) f[j] = *(volatile uint32_t *)(code + u[j]) & field;
#pragma unroll
                  for (int j = 1; j < 4; j++) f[j] = e + j < e1 ? f[j] : same;
                  uint32_t s4 = 0u, o4 = 0u;
#pragma unroll
                  for (int j = 0; j < 4; j++) {
                    double y = 0.0;
                    if (f[j] == above) y = Sg[u[j] * G];
                    s4 |= (f[j] != same && f[j] != above) ? 1u << j : 0u;
                    o4 |= f[j] == 0u ? 1u << j : 0u;
                    if (MODE == 0) ai += __double_as_longlong(y);
                    else if (MODE == 1) ad += f[j] == above ? i64_to_f64_pos(__double_as_longlong(y)) : 0.0;
                    else ad += y;
                  }
                  succ |= s4 << (e - e0);
                  open |= o4 << (e - e0);
                }
                for (uint32_t m = open; m; m &= m - 1u) claim(col_at(e0 + __ffs(m) - 1), g, field);
                edges += __popc(succ);
                if (e0 == rb) succ0 = succ;
              }
            }
            for (unsigned m = longs; COOP && m; m &= m - 1u) {  // long rows: the warp
              const int l = __ffs(m) - 1;
              const uint32_t gl = __shfl_sync(0xffffffffu, it, l) & gmask, fl = 3u << (2 * gl);
              const int b = __shfl_sync(0xffffffffu, rb, l), e = __shfl_sync(0xffffffffu, re, l);
              long long si = 0;
              double sd = 0.0;
              for (int k = b + lane; k < e; k += 32) {
                const uint32_t u = col_at(k), f = *(volatile uint32_t *)(code + u) & fl;
                if (f == cp << (2 * gl)) {
                  const double y = S[u * G + gl];
                  if (MODE == 0) si += __double_as_longlong(y);
                  else if (MODE == 1) sd += i64_to_f64_pos(__double_as_longlong(y));
                  else sd += y;
                } else if (f != cc << (2 * gl)) {
                  edges++;
                  if (f == 0u) claim(u, gl, fl);
                }
              }
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) {
                if (MODE == 0) si += __shfl_xor_sync(0xffffffffu, si, o);
                else sd += __shfl_xor_sync(0xffffffffu, sd, o);
              }
              if (lane == l) {
                ai = si;
                ad = sd;
              }
            }
            if (!valid) continue;
            succ_of[x] = succ0;
            if (L > 0) {
              const int id = IDENT ? ident[v] : 1;
              if (MODE == 0) {
                Si[x] = IDENT ? ai * id : ai;
              } else {
                if (drop) ad *= pow2_int(-s_drop[g]);
                if (IDENT && id != 1) ad *= (double)id;
                S[x] = ad;
                if (measure) atomicMax(s_max + g, (unsigned long long)__double_as_longlong(ad));
              }
            }
          }
        };
        if (kind) pass(std::integral_constant<int, 0>());
        else if (kind_prev) pass(std::integral_constant<int, 1>());
        else pass(std::integral_constant<int, 2>());
        __syncthreads();
        const int tail = s_tail;
        // the counts of level L+1: integers while the bound allows; the largest
        // counts are looked at when the bound nears the end of the double range
        if (L + 1 < lint && blg + flg >= 62) lint = L + 1;
        if (measure) {
          if (tid == 0) s_top = 0;
          __syncthreads();
          if (tid < cnt) {
            const unsigned long long m = s_max[tid];
            const int lg = m ? (int)((m >> 52) & 0x7ff) - 1022 : 0;  // the count is below 2^lg
            if (lg > 1023) atomicOr(err, ERR_OVERFLOW);
            const int k = lg > 960 ? lg - 959 : 0;
            s_drop[tid] = k;
            s_max[tid] = 0ull;
            atomicMax(&s_top, lg - k);
          }
          __syncthreads();
          blg = s_top;
          if (lscale > L) lscale = L;
        } else if (drop) {
          if (tid < cnt) s_drop[tid] = 0;
        }
        if (L >= lscale && tid < cnt) s_exp[tid] += s_drop[tid];  // of level L+1
        if (tail == hi) break;
        blg += flg;
        if (L >= lscale && tid < cnt) exps[(size_t)(L + 1) * G + tid] = s_exp[tid];
        lo = hi;
        hi = tail;
        L++;
        cc = cn;
        if (tid == 0) {
          if (L + 1 < SMALL_LEVELS) s_lvl[L + 1] = hi;
          else lvl_far[L + 1] = hi;
        }
        __syncthreads();
      }
      const int Lmax = L;
      dag += edges;
      // -------------------------------------------------------- phase 2
      // (level 0 holds the sources: their own dependencies are not needed)
      int b = hi;
      for (int l = Lmax; l >= 1; l--) {
        const bool kind = l < lint;
        const uint32_t cn = cc == 3u ? 1u : cc + 1u;
        const int a = l < SMALL_LEVELS ? s_lvl[l] : lvl_far[l];
        const bool sc = l >= lscale && l < Lmax;  // the level and the next may have other exponents
        const bool absolute = l > lscale;
        if (absolute || sc) {
          __syncthreads();
          if (tid < cnt) {
            s_exp[tid] = absolute ? exps[(size_t)l * G + tid] : 0;
            s_dexp[tid] = sc ? s_exp[tid] - exps[(size_t)(l + 1) * G + tid] : 0;
          }
          __syncthreads();
        }
        for (int i0 = a + tid0; i0 < b; i0 += NT) {
          const int i = COOP ? i0 + lane : i0;
          const bool valid = !COOP || i < b;
          const uint32_t it = valid ? Q[i] : 0u, v = it >> gs, g = it & gmask, x = v * G + g;
          const int rb = valid ? row_of(v) : 0;
          uint32_t m = valid ? succ_of[x] : 0u;
          int re = 0;
          unsigned longs = 0u;
          if (COOP) {
            re = valid ? row_of(v + 1) : 0;
            longs = __ballot_sync(0xffffffffu, re - rb > 32);
            if (__popc(longs) > SMALL_LONGS) longs = 0u;
          }
          const int id = IDENT ? ident[v] : 1;
          int ev = 0;
          float mv = 1.0f;
          double sv = 1.0;
          int idx = 0;  // the count, if it is an integer in the table of reciprocals
          if (valid) {
            if (kind) {
              long long s = Si[x];
              if (IDENT && id != 1) s /= id;  // exact: the stored count is a multiple of ident
              if (FP32) {
                split_pow2_i64(s, ev, mv);
              } else {
                idx = s < RECIP_TABLE ? (int)s : 0;
                sv = i64_to_f64_pos(s);
              }
            } else {
              sv = IDENT && id != 1 ? S[x] / (double)id : S[x];
              if (FP32) split_pow2(sv, ev, mv);
            }
            if (FP32 && absolute) ev += s_exp[g];
          }
          double sum = 0.0;
          float sumf = 0.0f;
          auto add = [&](double cw, int ev) {
            if (!FP32) {
              sum += cw;
            } else {
              const int d = ev - __double2hiint(cw);  // <= 0: sigma[v] <= sigma[w]
              if (d >= -126) sumf = fmaf(__int_as_float(__double2loint(cw)), __int_as_float((127 + d) << 23), sumf);
            }
          };
          if (COOP && l < Lmax)
            for (unsigned ml = longs; ml; ml &= ml - 1u) {  // long rows: the warp, by the codes
              const int from = __ffs(ml) - 1;
              const uint32_t gl = __shfl_sync(0xffffffffu, it, from) & gmask;
              const int rl = __shfl_sync(0xffffffffu, rb, from), el = __shfl_sync(0xffffffffu, re, from);
              const int evl = FP32 ? __shfl_sync(0xffffffffu, ev, from) : 0;
              const double sum0 = sum;
              const float sumf0 = sumf;
              sum = 0.0;
              sumf = 0.0f;
              for (int e = rl + lane; e < el; e += 32) {
                const uint32_t w = col_at(e);
                if (((code[w] >> (2 * gl)) & 3u) == cn) add(S[w * G + gl], evl);
              }
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) {
                if (!FP32) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                else sumf += __shfl_xor_sync(0xffffffffu, sumf, o);
              }
              if (lane != from) {
                sum = sum0;
                sumf = sumf0;
              }
            }
          if (!valid) continue;
          if (m) {  // the first one is taken as it is
            if (!FP32) {
              sum = S[col_at(rb + __ffs(m) - 1) * G + g];
              m &= m - 1u;
            }
            for (; m; m &= m - 1u) add(S[col_at(rb + __ffs(m) - 1) * G + g], ev);
          }
          if (l < Lmax && !(longs >> lane & 1u))
            for (int e = rb + 32; e < (COOP ? re : row_of(v + 1)); e++) {  // entries past the 32nd: by their codes
              const uint32_t w = col_at(e);
              if (((code[w] >> (2 * g)) & 3u) == cn) add(S[w * G + g], ev);
            }
          double dv;
          if (!FP32) {
            if (sc) sum *= pow2_int(s_dexp[g]);
            dv = REACH ? fma(sv, sum, init[v]) : sv * sum;
            if (l > 1) {
              const double r = idx ? __ldg(recip + idx) : recip_pos(sv);
              const double kr = IDENT && id != 1 ? (double)id * r : r;
              S[x] = fma(dv, kr, kr);
            }
          } else {
            const float df = fmaf(mv, sumf, REACH ? (float)init[v] : 0.0f), kv = (float)id;
            if (l > 1) S[x] = __hiloint2double(ev, __float_as_int(fmaf(kv, df, kv) / mv));
            dv = (double)df;
          }
          acc[x] = fma(s_ws[g], dv, acc[x]);
        }
        __syncthreads();
        b = a;
        cc = cc == 1u ? 3u : cc - 1u;
      }
      // the places' bc' terms, added up in order; every small_flush rounds, so
      // that no sum is a long chain of additions
      if (first + (int)G < item.s_end && ++rounds % small_flush(GLOBAL)) continue;
      for (int v = tid; v < n; v += NT) {
        double t = 0.0;
        for (uint32_t g = 0; g < G; g++) {
          t += acc[(uint32_t)v * G + g];
          acc[(uint32_t)v * G + g] = 0.0;
        }
        if (t != 0.0) atomicAdd(bcp_cta + c.vtx_off + v, t);
      }
    }
    __syncthreads();
  }
  for (int o = 16; o > 0; o >>= 1) dag += __shfl_xor_sync(0xffffffffu, dag, o);
  if (dag_total && lane == 0 && dag) atomicAdd(dag_total, dag);
}

// ------------------------------------------------------------ host side
// The kernel's attribute (opt-in shared memory) and its occupancy per
// shared-memory size are queried once per device and cached: each query is a
// driver call on the host's critical path.
static std::mutex g_small_mu;
static std::map<long long, int> g_small_occ;  // (variant, device, smem) -> CTAs per SM

template <bool R, bool I, bool F, int V, bool GLOBAL>
static int small_prepare(int device) {
  static std::mutex mu;
  static std::set<int> done;
  std::lock_guard<std::mutex> lk(mu);
  if (!done.count(device)) {
    BCS_CUDA(cudaFuncSetAttribute(k_bcreach_small<R, I, F, V, GLOBAL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)SMALL_SMEM));
    done.insert(device);
  }
  return BCS_OK;
}

template <bool R, bool I, bool F, int V, bool GLOBAL>
static int small_ctas_c(int device, size_t smem, int *out) {
  const long long key = ((long long)(R * 32 + I * 16 + F * 8 + V * 2 + GLOBAL) << 48) | ((long long)device << 32) |
                        (long long)smem;
  {
    std::lock_guard<std::mutex> lk(g_small_mu);
    auto it = g_small_occ.find(key);
    if (it != g_small_occ.end()) {
      *out = it->second;
      return BCS_OK;
    }
  }
  BCS_TRY((small_prepare<R, I, F, V, GLOBAL>(device)));
  BCS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_bcreach_small<R, I, F, V, GLOBAL>,
                                                         GLOBAL ? SMALL_GLOBAL_THREADS : SMALL_THREADS, smem));
  if (*out < 1) *out = 1;
  std::lock_guard<std::mutex> lk(g_small_mu);
  g_small_occ[key] = *out;
  return BCS_OK;
}

template <bool R, bool I, bool F>
static int small_ctas_t(int device, int variant, size_t smem, int *out) {
  if (variant == SMALL_COOP) return small_ctas_c<R, I, F, SMALL_COOP, false>(device, smem, out);
  if constexpr (F)
    if (variant == SMALL_FOUR) return small_ctas_c<R, I, F, SMALL_FOUR, false>(device, smem, out);
  return small_ctas_c<R, I, F, SMALL_PLAIN, false>(device, smem, out);
}

int small_ctas_per_sm(Ctx &ctx, bool R, bool I, bool F, int variant, size_t smem, int *out) {
  return BCS_DISPATCH3(small_ctas_t, R, I, F, ctx.device, variant, smem, out);
}

int small_variant(const Ctx &ctx, bool fp32, bool coop, int64_t sources, size_t smem) {
  if (coop) return SMALL_COOP;
  const bool rounds = sources > 3 * (int64_t)ctx.num_sms && sources <= 16 * (int64_t)ctx.num_sms;
  return fp32 && rounds && smem <= SMALL_BUDGET ? SMALL_FOUR : SMALL_PLAIN;
}

size_t small_scratch_words(int64_t ctas, int64_t nmax) { return (size_t)ctas * (SMALL_MAX_G + 1) * (nmax + 2); }

struct SmallLaunch {
  const SmallItem *items;
  int nitems;
  int *counter;
  const CompDesc *comps;
  const int64_t *srcs;
  size_t bcp_stride;
  int32_t *lvl;
  int lvl_stride, lvl_G;
  unsigned char *state;
  size_t state_stride;
  int *err;
  unsigned long long *dag;
};

template <bool R, bool I, bool F, int V, bool GLOBAL>
static int small_launch_c(Ctx &ctx, int grid, size_t smem, const BcInput &in, const SmallLaunch &a) {
  BCS_TRY((small_prepare<R, I, F, V, GLOBAL>(ctx.device)));
  const double *recip = nullptr;
  BCS_TRY(recip_table(ctx, &recip));
  k_bcreach_small<R, I, F, V, GLOBAL><<<grid, GLOBAL ? SMALL_GLOBAL_THREADS : SMALL_THREADS, smem, ctx.stream>>>(
      a.items, a.nitems, a.counter, a.comps, in.row, in.col, in.reach, in.ident, in.init, a.srcs, recip,
      in.bcp, a.bcp_stride, a.lvl, a.lvl_stride, a.lvl_G, a.state, a.state_stride, a.err, a.dag);
  ctx.launches++;
  BCS_CUDA(cudaGetLastError());
  return BCS_OK;
}

template <bool R, bool I, bool F>
static int small_launch_t(Ctx &ctx, int variant, int grid, size_t smem, const BcInput &in, const SmallLaunch &a) {
  if (variant == SMALL_COOP) return small_launch_c<R, I, F, SMALL_COOP, false>(ctx, grid, smem, in, a);
  if constexpr (F)
    if (variant == SMALL_FOUR) return small_launch_c<R, I, F, SMALL_FOUR, false>(ctx, grid, smem, in, a);
  return small_launch_c<R, I, F, SMALL_PLAIN, false>(ctx, grid, smem, in, a);
}

int launch_small(Ctx &ctx, bool fp32, int variant, int grid, size_t smem, const SmallItem *items, int nitems, int *counter,
                 const CompDesc *comps, const BcInput &in, const int64_t *srcs, int32_t *scratch, int64_t nmax,
                 int *err, unsigned long long *dag) {
  const bool R = in.reach != nullptr || in.init != nullptr, I = in.ident != nullptr;
  const SmallLaunch a{items, nitems, counter, comps, srcs, 0, scratch, (int)nmax + 2, SMALL_MAX_G, nullptr, 0, err, dag};
  return BCS_DISPATCH3(small_launch_t, R, I, fp32, ctx, variant, grid, smem, in, a);
}

// ------------------------------------- plain Brandes in a fixed scratch
// The scratch: the descriptor, the item counter and the error word (256 bytes
// each), the items, copies of bc', then per CTA the level offsets and exponents
// and, for a piece above shared memory, its counts and sums.

__global__ void k_fixed_setup(CompDesc *comp, CompDesc desc, int *counter, int *err, SmallItem *items, int nitems, int per,
                              int G) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nitems) items[i] = SmallItem{0, i * per, min(desc.n, (i + 1) * per), G};
  if (i == 0) {
    *comp = desc;
    *counter = 0;
    *err = 0;
  }
}

// One bc' of thousands of sources' terms would round as often: there are
// FIXED_COPIES, and adding those up keeps what the additions round off (2,600
// vertices: error 5.9e-16 in one, 1.2e-16 so).
__global__ void k_fixed_add(int n, const double *__restrict__ part, double *bc) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    double t = 0.0, lost = 0.0;
    for (int c = 0; c < FIXED_COPIES; c++) {
      const double a = part[(size_t)c * n + v], sum = t + a, of_a = sum - t;
      lost += (t - (sum - of_a)) + (a - of_a);
      t = sum;
    }
    bc[v] = t + lost;
  }
}

template <bool F, bool GLOBAL>
static int fixed_launch(Ctx &ctx, const CompDesc &desc, size_t smem, int G, size_t lvl_bytes, size_t state_bytes,
                        BcInput in, unsigned char *scratch, size_t bytes) {
  const int64_t n = desc.n;
  const size_t head = FIXED_HEAD + fixed_up256((size_t)n * sizeof(SmallItem));
  int per_sm = 1;
  BCS_TRY((small_ctas_c<false, false, F, SMALL_COOP, GLOBAL>(ctx.device, smem, &per_sm)));
  const size_t part_bytes = fixed_up256((size_t)FIXED_COPIES * n * 8);
  const int64_t fit = (int64_t)((bytes - head - part_bytes) / (lvl_bytes + state_bytes));
  const int64_t ctas = std::max<int64_t>(1, std::min<int64_t>((int64_t)ctx.num_sms * per_sm, fit));
  // two items per CTA, or more of as many rounds as are added up at once
  const int per = G * (int)std::max<int64_t>(1, std::min<int64_t>(n / (ctas * 2 * G), small_flush(GLOBAL)));
  SmallLaunch a{};
  a.nitems = (int)((n + per - 1) / per);
  const int grid = (int)std::min<int64_t>(ctas, a.nitems);
  double *const part = (double *)(scratch + head), *const bc = in.bcp;
  a.comps = (const CompDesc *)scratch;
  a.counter = (int *)(scratch + 256);
  a.err = (int *)(scratch + FIXED_ERR);
  a.items = (const SmallItem *)(scratch + FIXED_HEAD);
  a.lvl = (int32_t *)(scratch + head + part_bytes);
  a.lvl_stride = (int)n + 2;
  a.lvl_G = G;
  a.bcp_stride = (size_t)n;
  a.state = scratch + head + part_bytes + (size_t)grid * lvl_bytes;
  a.state_stride = state_bytes;
  in.bcp = part;
  BCS_CUDA(cudaMemsetAsync(part, 0, part_bytes, ctx.stream));
  k_fixed_setup<<<(a.nitems + 255) / 256, 256, 0, ctx.stream>>>((CompDesc *)scratch, desc, a.counter, a.err,
                                                                (SmallItem *)(scratch + FIXED_HEAD), a.nitems, per, G);
  ctx.launches++;
  BCS_CUDA(cudaGetLastError());
  BCS_TRY((small_launch_c<false, false, F, SMALL_COOP, GLOBAL>(ctx, grid, smem, in, a)));
  k_fixed_add<<<(int)((n + 63) / 64), 64, 0, ctx.stream>>>((int)n, part, bc);
  ctx.launches++;
  BCS_CUDA(cudaGetLastError());
  return BCS_OK;
}

int launch_plain_fixed_scratch(Ctx &ctx, const int64_t *row, const int32_t *col, int32_t n, int64_t nnz, double *bc,
                               unsigned char *scratch, size_t bytes, bool fp32) {
  int *const err = (int *)(scratch + FIXED_ERR);
  // n bounds the degree, hence the growth of path counts per level
  CompDesc desc{};
  desc.n = n;
  desc.nnz = nnz;
  desc.src_off = -1;
  desc.fan = (double)std::max(n, 1);
  BcInput in;
  in.row = row;
  in.col = col;
  in.bcp = bc;
  if (small_takes(n, nnz, 1) && small_smem_bytes(n, nnz, 1, false, false) <= SMALL_SMEM) {
    // no more sources at once than leave every SM two items
    int G = (int)std::max<int64_t>(1, std::min<int64_t>(SMALL_MAX_G, n / (2 * (int64_t)ctx.num_sms)));
    while (G > 1 && small_smem_bytes(n, nnz, G, false, false) > SMALL_BUDGET) G--;
    const size_t smem = small_smem_bytes(n, nnz, G, false, false), lvl = fixed_up256((size_t)(G + 1) * (n + 2) * 4);
    if (fp32) BCS_TRY((fixed_launch<true, false>(ctx, desc, smem, G, lvl, 0, in, scratch, bytes)));
    else BCS_TRY((fixed_launch<false, false>(ctx, desc, smem, G, lvl, 0, in, scratch, bytes)));
  } else {
    const size_t smem = align16((size_t)n * 4) + align16((size_t)n * 2), lvl = fixed_up256((size_t)2 * (n + 2) * 4);
    const size_t state = fixed_up256(align16((size_t)n * 8) * 2 + align16((size_t)n * 4));
    if (fp32) BCS_TRY((fixed_launch<true, true>(ctx, desc, smem, 1, lvl, state, in, scratch, bytes)));
    else BCS_TRY((fixed_launch<false, true>(ctx, desc, smem, 1, lvl, state, in, scratch, bytes)));
  }
  int h_err = 0;
  BCS_CUDA(cudaMemcpyAsync(&h_err, err, sizeof(int), cudaMemcpyDeviceToHost, ctx.stream));
  BCS_CUDA(cudaStreamSynchronize(ctx.stream));
  if (h_err & ERR_OVERFLOW) {
    set_error("shortest-path counts overflowed the FP64 range within one BFS level");
    return BCS_EOVERFLOW;
  }
  return BCS_OK;
}

}  // namespace bcs
