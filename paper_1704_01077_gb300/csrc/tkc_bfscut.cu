// Batched BFSCut: Algorithm 1 with updateBoundsBFSCut (Algorithm 4) for up to
// 512 sources at once, as one persistent cooperative kernel per call.
//
// Sources of one batch occupy bit "slots" of a per-vertex row of W 64-bit
// words: seen (visited by slot b), F (frontier of slot b) and N (next level of
// slot b, top-down only).  One loop iteration advances every active slot by one
// BFS level:
//   phase A  expand: top-down over the frontier list (atomic OR into N) or
//            bottom-up over the vertices with an in-arc (OR of in-neighbours' F
//            rows, stopping once every missing bit is found), direction chosen
//            per level;
//   phase B  finalize: new = N, seen |= new, F' = new, per-slot level sizes and
//            out-degree sums by warp bit-transpose + popcount; old F rows cleared
//            (after a bottom-up level, which appends to no list, by the bits of
//            the old frontier's bitmap);
//   epilogue (last block to reach the team's barrier): per-slot S, n_d, gamma,
//            merge of finished searches into the top-k, x = k-th farness, the
//            BFSCut test of the Section 6 lemma at r in [alpha', omega] (Section 8.2), and
//            the next step's direction.
// When every slot of a batch is done, a clear step zeroes the rows the batch
// touched and the epilogue seeds the next batch from the source order,
// abandoning sources already at level 0 when their bound exceeds x.
//
// A call is an opening launch over a batch of promising sources (k_open_keys,
// k_open_pick), a filter that drops the sources which the threshold it leaves
// abandons after levels 0, 1 and 2 (k_filter_test, k_filter_compact), and the
// main launch over the rest by teams of SMs; one-source searches and the
// deterministic schedule are a single launch over the order as it stands.
//
// What bounds it: on small graphs the chain of dependent memory accesses of a
// level (two barriers, an epilogue, an L2 load 150 ns, a returning atomic 440
// ns); on large ones the gathers of bottom-up levels, by latency and
// instructions issued rather than by bandwidth (DRAM at a tenth to a quarter).
//
// Every grid-wide wait is bounded by a clock64 budget; on expiry the kernel
// records TKC_ETIMEOUT and every block returns.
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "tkc_internal.cuh"

namespace tkc {

typedef unsigned long long u64;
typedef uint32_t u32;
typedef unsigned __int128 u128;

static constexpr unsigned FULL = 0xffffffffu;
static constexpr int kPackShift = 38;
static constexpr u64 kArcMask = (1ull << kPackShift) - 1;
static constexpr int kTopMax = TKC_MAX_K;

// ------------------------------------------------------------------ memory ordering

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned *p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_volatile_i32(const int *p) { return *(volatile const int *)p; }
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// One 128-bit word, read and written whole.
__device__ __forceinline__ ulonglong2 ld_relaxed_128(const ulonglong2 *p) {
  ulonglong2 v;
  asm volatile("{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }"
               : "=l"(v.x), "=l"(v.y)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_128(ulonglong2 *p, unsigned long long lo, unsigned long long hi) {
  asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p), "l"(lo), "l"(hi)
               : "memory");
}

// Barrier over the `nblocks` blocks of one team (all co-resident: the launch
// is cooperative).  The last block to arrive runs `epi` (whole block) before
// releasing the others.  Returns false when a wait ran out or met an error
// recorded by this team or any other: a block that leaves never arrives again,
// so the blocks of its team meet the error at their next wait.
//
// A level of a small graph is two of these and little else, so the wait polls
// the generation alone, at full rate at first (an L2 round trip each), and
// looks at the error words only every 16th time: with both words read on every
// poll and a sleep between, a release took 2.7 us to be seen.
template <typename Epi>
__device__ __forceinline__ bool team_sync(Ctl *ctl, Shared *sh, unsigned nblocks, uint64_t timeout, Epi epi) {
  __shared__ int s_last, s_ok;
  __shared__ unsigned s_gen;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned gen = ld_acquire_u32(&ctl->bar_gen);
    s_gen = gen;
    s_ok = 1;
    __threadfence();
    unsigned arrived = atomicAdd(&ctl->bar_count, 1u) + 1u;
    s_last = (arrived == nblocks);
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    epi();
    __syncthreads();
    if (threadIdx.x == 0) {
      ctl->bar_count = 0;
      __threadfence();
      st_release_u32(&ctl->bar_gen, s_gen + 1u);
    }
  } else if (threadIdx.x == 0) {
    const long long t0 = clock64();
    for (unsigned poll = 1; ld_acquire_u32(&ctl->bar_gen) == s_gen; ++poll) {
      const bool late = (uint64_t)(clock64() - t0) > timeout;
      if ((poll & 15u) == 0 || late) {
        if (late) {
          atomicCAS(&ctl->err, 0, TKC_ETIMEOUT);
          atomicCAS(&sh->err, 0, TKC_ETIMEOUT);
          atomicCAS(&ctl->err_where, 0, 1);
        }
        if (ld_volatile_i32(&ctl->err) != 0 || ld_volatile_i32(&sh->err) != 0) {
          s_ok = 0;
          break;
        }
      }
      if (poll > 64) __nanosleep(128);
    }
    __threadfence();
  }
  __syncthreads();
  return s_ok != 0;
}

// ------------------------------------------------------------------ exact arithmetic

// The Section 6 lemma at radius d, evaluated at reach r >= nd:
//   L = S_d + (d+1)(r - n_d) + max(0, r - n_d - g)
__device__ __forceinline__ u64 cut_sum(u64 Sd, u64 d, u64 nd, u64 g, u64 r) {
  u64 rem = r - nd;
  return Sd + (d + 1) * rem + (rem > g ? rem - g : 0);
}

// a/(ra-1)^2 < b/(rb-1)^2 for ra, rb >= 2
__device__ __forceinline__ bool ratio_less(u64 a, u64 ra, u64 b, u64 rb) {
  return (u128)a * (u128)((rb - 1) * (rb - 1)) < (u128)b * (u128)((ra - 1) * (ra - 1));
}

// True when the farness lower bound exceeds x = (Sx, rx) strictly for every
// r in [max(lo, nd), hi].  The bound divided by (r-1)^2 is linear-over-square
// on [lo', kink] and on [kink, hi] (kink = nd + g), so by the Section 8 lemma
// on such bounds its minimum over the interval is at lo', hi or the kink.
__device__ bool cut_exceeds(u64 Sd, u64 d, u64 nd, u64 g, u64 lo, u64 hi, u64 Sx, u64 rx) {
  if (lo < nd) lo = nd;
  if (hi < lo) hi = lo;
  u64 kink = nd + g;
  u64 cand[3] = {lo, hi, kink};
  int nc = (kink > lo && kink < hi) ? 3 : 2;
  for (int i = 0; i < nc; ++i) {
    u64 r = cand[i];
    if (r <= 1) continue;  // r = 1 is farness +inf, above any finite x
    u64 L = cut_sum(Sd, d, nd, g, r);
    // not (L/(r-1)^2 > Sx/(rx-1)^2)  ->  keep searching
    if (!ratio_less(Sx, rx, L, r)) return false;
  }
  return true;
}

// NBCut's stop (Algorithm 1 with computeBoundsNB): the source's order key
// floor(2^46 L') with L' <= S/(r-1)^2 exceeds x = Sx/(rx-1)^2 strictly.  The
// order is sorted by key, so every later source of the graph exceeds x too.
__device__ __forceinline__ bool nb_exceeds(u64 key, u64 Sx, u64 rx) {
  return (u128)key * (u128)((rx - 1) * (rx - 1)) > ((u128)Sx << 46);
}

// List order.  Closeness: (S, r, id) by farness ascending, then id ascending
// (r >= 2 here).  Harmonic: the key is the FP64 bit pattern of h >= 0, which
// orders like the value; larger h first, then smaller id.
__device__ __forceinline__ bool entry_less(bool harmonic, u64 Sa, u32 ra, u32 ia, u64 Sb, u32 rb, u32 ib) {
  if (harmonic) return Sa != Sb ? Sa > Sb : ia < ib;
  u128 lhs = (u128)Sa * (u128)((u64)(rb - 1) * (u64)(rb - 1));
  u128 rhs = (u128)Sb * (u128)((u64)(ra - 1) * (u64)(ra - 1));
  if (lhs != rhs) return lhs < rhs;
  return ia < ib;
}

// Harmonic centrality (the paper's closing generalisation to sums of f(d) with
// f = 1/d): after level d, the vertices not yet found lie at distance >= d+1,
// at most g of them at d+1, and there are at most omega - n_d of them, so
//   h <= U = H_d + min(g, w)/(d+1) + max(0, w - g)/(d+2),  w = omega - n_d.
// The search is abandoned when fl(U * (1 + 2^-20)) < x: the margin covers the
// rounding of H_d and U and of the FP64 h it is compared with (depths < 2^32).
constexpr double kHMargin = 1.0 + 1.0 / 1048576.0;


// Bottom-up walks, batches of at most 256 bits: in-arcs a lane takes per step
// when it walks a short in-row alone (U), and per lane per step when the warp
// walks a long one (HU).  Search kernel, distance sums of 4 096 sources of
// R-MAT 20 and NBCut on a directed Erdos-Renyi graph of 1.2 million vertices and
// 9.6 million arcs (both on the labelled copy): 4 and 4 10.7 and 14.4 ms; U 2
// 10.6 and 14.3, U 8 11.1 and 14.8; HU 2 11.0 and 14.2, HU 8 11.1 and 14.4.
#ifndef TKC_BU_U
#define TKC_BU_U 4
#endif
#ifndef TKC_BU_HU
#define TKC_BU_HU 4
#endif

// Threads per block of the search kernel (one block per SM).  The level loops
// wait on dependent row gathers, so more resident warps hide more latency:
// the 64- and 128-bit kernels run 32 warps per SM, at the price of a few
// spilled registers (the two searches above, 64- and 128-bit: 1024 threads 10.7
// and 14.4 ms, 512 threads 15.3 and 17.0; 768 threads for 128-bit batches 15.1).
#ifndef TKC_THREADS_W2
#define TKC_THREADS_W2 1024
#endif
template <int W>
constexpr int kThreads = W == 1 ? 1024 : W == 2 ? TKC_THREADS_W2 : 512;
// Small graphs and one-source searches: short levels, where the block-wide
// barriers and scans of the larger blocks cost more than they hide.
constexpr int kMinThreads = 512;
constexpr int kMaxThreads = 1024;

__device__ __forceinline__ bool harmonic_below(double Hd, u64 d, u64 nd, u64 g, u64 omega, u64 xbits) {
  const u64 w = omega > nd ? omega - nd : 0;
  const u64 near_ = g < w ? g : w, far_ = w > g ? w - g : 0;
  const double t1 = __ddiv_rn((double)near_, (double)(d + 1));
  const double t2 = __ddiv_rn((double)far_, (double)(d + 2));
  const double U = __dadd_rn(__dadd_rn(Hd, t1), t2);
  return __dmul_rn(U, kHMargin) < __longlong_as_double((long long)xbits);
}

// ------------------------------------------------------------------ warp helpers

// 32x32 bit-matrix transpose across a warp: afterwards bit l of lane i equals
// bit i of lane l's input.
__device__ __forceinline__ uint32_t warp_transpose32(uint32_t x, int lane) {
  uint32_t m = 0x0000FFFFu;
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) {
    uint32_t y = __shfl_xor_sync(FULL, x, j);
    x = (lane & j) ? ((x & ~m) | ((y >> j) & m)) : ((x & m) | ((y & m) << j));
    m ^= m << (j >> 1);
  }
  return x;
}

// OR of a 64-bit word over the warp: one warp reduction per 32-bit half
// (measured 5% off the search kernel against five rounds of shuffles).
__device__ __forceinline__ u64 warp_or(u64 x) {
  const uint32_t lo = __reduce_or_sync(FULL, (uint32_t)x), hi = __reduce_or_sync(FULL, (uint32_t)(x >> 32));
  return ((u64)hi << 32) | lo;
}

// Adds, for every slot bit of the 32 lanes' rows, the number of lanes with
// the bit set and the sum of those lanes' `od` into the block counters.  (A
// search finds a vertex once, so its sums stay below the graph's arcs and so
// below 2^32; 64-bit shared-memory additions would be compare-and-swap loops.)
template <int W>
__device__ __forceinline__ void warp_count_slots(const u64 (&nw)[W], uint32_t od, unsigned *s_cnt,
                                                 unsigned *s_wsum, int lane) {
  uint32_t anyw = 0;
#pragma unroll
  for (int j = 0; j < W; ++j) anyw |= (nw[j] != 0);
  if (__ballot_sync(FULL, anyw) == 0) return;
  uint32_t odm = anyw ? od : 0u;
  uint32_t maxod = __reduce_max_sync(FULL, odm);
  int planes = 32 - __clz(maxod);
  // all 2W halves transposed first, so that the out-degree bit planes (one
  // ballot each) serve every half
  uint32_t colv[2 * W], cv[2 * W];
  uint32_t cmax = 0;
#pragma unroll
  for (int jh = 0; jh < 2 * W; ++jh) {
    const uint32_t x = (uint32_t)(nw[jh >> 1] >> (32 * (jh & 1)));
    colv[jh] = __ballot_sync(FULL, x != 0) ? warp_transpose32(x, lane) : 0u;
    cv[jh] = __popc(colv[jh]);
    cmax = cv[jh] > cmax ? cv[jh] : cmax;
  }
  const uint32_t maxc = __reduce_max_sync(FULL, cmax);
  uint32_t ws[2 * W];
#pragma unroll
  for (int jh = 0; jh < 2 * W; ++jh) ws[jh] = 0;
  // about 6 instructions per half for a walk step or a plane, 1 more per plane
  if ((int)maxc * 12 * W <= planes * (1 + 12 * W)) {
    // walk the set bits: fetch each contributing lane's out-degree
    for (uint32_t it = 0; it < maxc; ++it) {
#pragma unroll
      for (int jh = 0; jh < 2 * W; ++jh) {
        const int src = colv[jh] ? (__ffs(colv[jh]) - 1) : 0;
        const uint32_t v = __shfl_sync(FULL, odm, src);
        if (colv[jh]) {
          ws[jh] += v;
          colv[jh] &= colv[jh] - 1;
        }
      }
    }
  } else {
    // bit planes of the out-degrees: sum = sum_p 2^p popc(col & plane_p)
    for (int p = 0; p < planes; ++p) {
      const uint32_t plane = __ballot_sync(FULL, (odm >> p) & 1u);
#pragma unroll
      for (int jh = 0; jh < 2 * W; ++jh) ws[jh] += (uint32_t)__popc(colv[jh] & plane) << p;
    }
  }
#pragma unroll
  for (int jh = 0; jh < 2 * W; ++jh) {
    if (cv[jh]) {
      const int slot = 32 * jh + lane;
      atomicAdd(&s_cnt[slot], cv[jh]);
      atomicAdd(&s_wsum[slot], ws[jh]);
    }
  }
}

// Warp-aggregated append of the lanes with `pred` to a list whose counter
// packs count << 38 | arcs.  Writes list[pos] = v and loff[pos] = arc prefix.
__device__ __forceinline__ void warp_append(bool pred, uint32_t v, uint32_t od, u64 *packed, uint32_t *list,
                                            uint32_t *loff, int lane) {
  uint32_t mask = __ballot_sync(FULL, pred);
  if (mask == 0) return;
  uint32_t a = pred ? od : 0u;
  // inclusive scan of arcs over lanes
  uint32_t incl = a;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += t;
  }
  uint32_t total = __shfl_sync(FULL, incl, 31);
  int leader = __ffs(mask) - 1;
  u64 base = 0;
  if (lane == leader) base = atomicAdd(packed, ((u64)__popc(mask) << kPackShift) | (u64)total);
  base = __shfl_sync(FULL, base, leader);
  if (pred) {
    uint32_t pos = (uint32_t)(base >> kPackShift) + __popc(mask & ((1u << lane) - 1u));
    list[pos] = v;
    loff[pos] = (uint32_t)((base & kArcMask) + (incl - a));
  }
}

// warp_append for T entries per lane, one atomic for all of them (in lane order).
template <int T>
__device__ __forceinline__ void warp_append_steps(const bool (&pred)[T], const uint32_t (&v)[T],
                                                  const uint32_t (&od)[T], u64 *packed, uint32_t *list,
                                                  uint32_t *loff, int lane) {
  uint32_t cnt = 0, arcs = 0;
#pragma unroll
  for (int t = 0; t < T; ++t) {
    cnt += pred[t];
    arcs += pred[t] ? od[t] : 0u;
  }
  if (__ballot_sync(FULL, cnt != 0) == 0) return;
  uint32_t ci = cnt, ai = arcs;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t tc = __shfl_up_sync(FULL, ci, o), ta = __shfl_up_sync(FULL, ai, o);
    if (lane >= o) {
      ci += tc;
      ai += ta;
    }
  }
  u64 base = 0;
  if (lane == 31) base = atomicAdd(packed, ((u64)ci << kPackShift) | (u64)ai);
  base = __shfl_sync(FULL, base, 31);
  uint32_t pos = (uint32_t)(base >> kPackShift) + ci - cnt;
  uint32_t at = (uint32_t)(base & kArcMask) + ai - arcs;
#pragma unroll
  for (int t = 0; t < T; ++t) {
    if (!pred[t]) continue;
    list[pos] = v[t];
    loff[pos] = at;
    ++pos;
    at += od[t];
  }
}

__device__ __forceinline__ void warp_append_plain(bool pred, uint32_t v, unsigned *counter, uint32_t *list,
                                                  int lane) {
  uint32_t mask = __ballot_sync(FULL, pred);
  if (mask == 0) return;
  int leader = __ffs(mask) - 1;
  uint32_t base = 0;
  if (lane == leader) base = atomicAdd(counter, (unsigned)__popc(mask));
  base = __shfl_sync(FULL, base, leader);
  if (pred) list[base + __popc(mask & ((1u << lane) - 1u))] = v;
}

template <int W>
__device__ __forceinline__ void load_row(const u64 *base, uint32_t v, u64 (&r)[W]) {
  const u64 *p = base + (size_t)v * W;
  if constexpr (W == 1) {
    r[0] = p[0];
  } else {
#pragma unroll
    for (int j = 0; j < W; j += 2) {
      ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(p + j);
      r[j] = t.x;
      r[j + 1] = t.y;
    }
  }
}

template <int W>
__device__ __forceinline__ void store_row(u64 *base, uint32_t v, const u64 (&r)[W]) {
  u64 *p = base + (size_t)v * W;
  if constexpr (W == 1) {
    p[0] = r[0];
  } else {
#pragma unroll
    for (int j = 0; j < W; j += 2) *reinterpret_cast<ulonglong2 *>(p + j) = make_ulonglong2(r[j], r[j + 1]);
  }
}

template <int W>
__device__ __forceinline__ bool row_nonzero(const u64 (&r)[W]) {
  u64 a = 0;
#pragma unroll
  for (int j = 0; j < W; ++j) a |= r[j];
  return a != 0;
}

// Zeroes the frontier rows of the listed vertices and their frontier bits.
// A long list clears the whole bitmap (of vertices [v0, v1), where all listed
// ones lie) instead of one bit per vertex.
template <int W>
__device__ __forceinline__ void clear_frontier(u64 *F, uint32_t *FB, const uint32_t *list, uint32_t count, uint32_t v0,
                                               uint32_t v1, uint64_t gthread, uint64_t nthreads) {
  for (uint64_t i = gthread; i < (uint64_t)count * W; i += nthreads) {
    uint32_t v = list[i / W];
    F[(size_t)v * W + (i % W)] = 0;
  }
  if (count > (v1 - v0) / 32) {
    for (uint64_t i = v0 / 32 + gthread; i < v1 / 32 + 1; i += nthreads) FB[i] = 0;
  } else {
    for (uint64_t i = gthread; i < count; i += nthreads) {
      uint32_t v = list[i];
      atomicAnd(&FB[v >> 5], ~(1u << (v & 31)));
    }
  }
}

// Zeroes the rows of vertices [v0, v1).
template <int W>
__device__ __forceinline__ void clear_rows(u64 *F, uint32_t v0, uint32_t v1, uint64_t gthread, uint64_t nthreads) {
  if constexpr (W == 1) {
    for (uint64_t i = v0 + gthread; i < v1; i += nthreads) F[i] = 0;
  } else {
    ulonglong2 *q = reinterpret_cast<ulonglong2 *>(F);
    for (uint64_t i = (uint64_t)v0 * (W / 2) + gthread; i < (uint64_t)v1 * (W / 2); i += nthreads)
      q[i] = make_ulonglong2(0, 0);
  }
}

// Zeroes the frontier's rows and bits: by its list, or, when a bottom-up level
// left it without one, all of [v0, v1).
template <int W>
__device__ __forceinline__ void clear_old_frontier(bool has_list, u64 *F, uint32_t *FB, const uint32_t *list,
                                                   uint32_t count, uint32_t v0, uint32_t v1, uint64_t gthread,
                                                   uint64_t nthreads) {
  if (count == 0) return;
  if (has_list) {
    clear_frontier<W>(F, FB, list, count, v0, v1, gthread, nthreads);
  } else {
    clear_rows<W>(F, v0, v1, gthread, nthreads);
    for (uint64_t i = v0 / 32 + gthread; i < v1 / 32 + 1; i += nthreads) FB[i] = 0;
  }
}

// updateBoundsLB: the slots whose bits are new in this vertex's row found it at
// this depth.
template <int W>
__device__ __forceinline__ void record_levels(const RunParams &p, uint32_t w, const u64 (&nw)[W], uint32_t depth) {
  const uint32_t v = p.unlab ? p.unlab[w] : w;  // the vertex whose search label is w
  uint16_t *row = p.lvl + (size_t)v * p.lvl_stride + (size_t)p.team * p.B;
#pragma unroll
  for (int q = 0; q < W; ++q) {
    u64 b = nw[q];
    while (b) {
      const int j = __ffsll((long long)b) - 1;
      b &= b - 1;
      row[64 * q + j] = (uint16_t)depth;
    }
  }
}

// ------------------------------------------------------------------ shared state

template <int W>
struct Smem {
  unsigned cnt[64 * W];
  unsigned wsum[64 * W];
  u64 active[W];
  // epilogue scratch
  u64 tS[kTopMax];
  uint32_t tr[kTopMax], tid[kTopMax];
  u64 cS[64 * W];
  uint32_t cr[64 * W], cid[64 * W], cg[64 * W];
  unsigned ncand;
  unsigned nactive;
  unsigned scan[kMaxThreads / 32 + 1];
  u64 scan64[kMaxThreads / 32 + 1];
  u64 acc[4];
  unsigned bu_next;  // bottom-up level: next of this block's vertex chunks
  u64 bu_new;        // and its new vertices, packed like nl_packed
  alignas(8) uint32_t cmd[kCmdWords];  // the step's control words (Ctl from `step` on)
};
static_assert(offsetof(Ctl, step) % 8 == 0 && kCmdWords <= 64, "the control words are copied as they lie");

// Block-wide exclusive scan of one uint32 per thread; returns the prefix and
// writes the total to *total.
template <int W>
__device__ uint32_t block_exscan(Smem<W> &sm, uint32_t x, uint32_t *total) {
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();
  if (lane == 31) sm.scan[wid] = incl;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t run = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
      uint32_t t = sm.scan[i];
      sm.scan[i] = run;
      run += t;
    }
    sm.scan[blockDim.x >> 5] = run;
  }
  __syncthreads();
  uint32_t res = sm.scan[wid] + incl - x;
  *total = sm.scan[blockDim.x >> 5];
  __syncthreads();
  return res;
}

template <int W>
__device__ u64 block_exscan64(Smem<W> &sm, u64 x, u64 *total) {
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  u64 incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    u64 t = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();
  if (lane == 31) sm.scan64[wid] = incl;
  __syncthreads();
  if (threadIdx.x == 0) {
    u64 run = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
      u64 t = sm.scan64[i];
      sm.scan64[i] = run;
      run += t;
    }
    sm.scan64[blockDim.x >> 5] = run;
  }
  __syncthreads();
  u64 res = sm.scan64[wid] + incl - x;
  *total = sm.scan64[blockDim.x >> 5];
  __syncthreads();
  return res;
}

// ------------------------------------------------------------------ epilogues

// The k-th entry of graph g's list as last published.
struct Thresh {
  bool have;
  u64 S;
  uint32_t r, id;
};

__device__ __forceinline__ Thresh thresh_of(const RunParams &p, uint32_t g) {
  const ulonglong2 v = ld_relaxed_128(p.x + g);
  Thresh t;
  t.S = v.x;
  t.r = (uint32_t)(v.y >> 32);
  t.id = (uint32_t)v.y;
  t.have = t.r != 0;
  return t;
}

// Publishes graph g's current k-th entry (caller holds the list's lock).
__device__ __forceinline__ void publish_thresh(const RunParams &p, uint32_t g) {
  if (*(volatile unsigned *)&p.g_ntop[g] != p.kk) return;
  const size_t i = (size_t)g * p.kk + p.kk - 1;
  const u64 S = *(volatile u64 *)&p.top_S[i];
  const u64 r = *(volatile uint32_t *)&p.top_r[i], id = *(volatile uint32_t *)&p.top_id[i];
  st_relaxed_128(p.x + g, S, r << 32 | id);
}

// Lock of graph g's list, taken by one thread; a wait beyond the budget is an
// error.
__device__ __forceinline__ bool lock_list(const RunParams &p, uint32_t g) {
  long long t0 = clock64();
  unsigned ns = 32;
  while (atomicCAS(&p.g_lock[g], 0, 1) != 0) {
    if (ld_volatile_i32(&p.sh->err) != 0 || (uint64_t)(clock64() - t0) > p.timeout) {
      atomicCAS(&p.sh->err, 0, TKC_ETIMEOUT);
      atomicCAS(&p.ctl->err, 0, TKC_ETIMEOUT);
      return false;
    }
    __nanosleep(ns);
    if (ns < 256) ns <<= 1;
  }
  __threadfence();
  return true;
}

__device__ __forceinline__ void unlock_list(const RunParams &p, uint32_t g) {
  __threadfence();
  atomicExch(&p.g_lock[g], 0);
}

// Merges the block's candidate list (sm.cS/cr/cid, sm.ncand entries) into the
// list of graph g (all candidates are g's).  Every entry's new position is its
// rank among the old list and the candidates (keys are unique: farness then
// id), so each position below k gets exactly one writer and the old list is
// read from a shared copy.
template <int W>
__device__ void merge_topk_one(const RunParams &p, Smem<W> &sm, uint32_t g) {
  const uint32_t kk = p.kk;
  const size_t at = (size_t)g * kk;
  uint32_t ntop = *(volatile unsigned *)&p.g_ntop[g];
  uint32_t nc = sm.ncand;
  if (nc == 0) return;
  for (uint32_t i = threadIdx.x; i < ntop; i += blockDim.x) {
    sm.tS[i] = *(volatile u64 *)&p.top_S[at + i];
    sm.tr[i] = *(volatile uint32_t *)&p.top_r[at + i];
    sm.tid[i] = *(volatile uint32_t *)&p.top_id[at + i];
  }
  __syncthreads();
  // rank of each candidate among existing entries and other candidates
  for (uint32_t i = threadIdx.x; i < nc; i += blockDim.x) {
    u64 S = sm.cS[i];
    uint32_t r = sm.cr[i], id = sm.cid[i];
    uint32_t lo = 0, hi = ntop;  // first existing entry not less than the candidate
    while (lo < hi) {
      uint32_t mid = (lo + hi) >> 1;
      if (entry_less(p.harmonic, sm.tS[mid], sm.tr[mid], sm.tid[mid], S, r, id)) lo = mid + 1;
      else hi = mid;
    }
    uint32_t rank = lo;
    for (uint32_t j = 0; j < nc; ++j)
      if (j != i && entry_less(p.harmonic, sm.cS[j], sm.cr[j], sm.cid[j], S, r, id)) ++rank;
    if (rank < kk) {
      p.top_S[at + rank] = S;
      p.top_r[at + rank] = r;
      p.top_id[at + rank] = id;
    }
  }
  for (uint32_t i = threadIdx.x; i < ntop; i += blockDim.x) {
    uint32_t rank = i;
    for (uint32_t j = 0; j < nc; ++j)
      if (entry_less(p.harmonic, sm.cS[j], sm.cr[j], sm.cid[j], sm.tS[i], sm.tr[i], sm.tid[i])) ++rank;
    if (rank < kk) {
      p.top_S[at + rank] = sm.tS[i];
      p.top_r[at + rank] = sm.tr[i];
      p.top_id[at + rank] = sm.tid[i];
    }
  }
  __syncthreads();
  uint32_t nnew = ntop + nc < kk ? ntop + nc : kk;
  if (threadIdx.x == 0) p.g_ntop[g] = nnew;
  __syncthreads();
}

// A batch of several graphs: the thread holding a graph's first candidate
// inserts that graph's candidates into its list one by one, under its lock.
template <int W>
__device__ void merge_topk_many(const RunParams &p, Smem<W> &sm) {
  const uint32_t kk = p.kk;
  const uint32_t nc = sm.ncand;
  for (uint32_t i = threadIdx.x; i < nc; i += blockDim.x) {
    const uint32_t g = sm.cg[i];
    bool first = true;
    for (uint32_t j = 0; j < i && first; ++j) first = sm.cg[j] != g;
    if (!first || !lock_list(p, g)) continue;
    volatile u64 *tS = p.top_S + (size_t)g * kk;
    volatile uint32_t *tr = p.top_r + (size_t)g * kk, *ti = p.top_id + (size_t)g * kk;
    uint32_t cnt = *(volatile unsigned *)&p.g_ntop[g];
    for (uint32_t j = i; j < nc; ++j) {
      if (sm.cg[j] != g) continue;
      u64 S = sm.cS[j];
      uint32_t r = sm.cr[j], id = sm.cid[j];
      if (cnt == kk && !entry_less(p.harmonic, S, r, id, tS[kk - 1], tr[kk - 1], ti[kk - 1])) continue;
      uint32_t pos = cnt < kk ? cnt++ : kk - 1;
      while (pos > 0 && entry_less(p.harmonic, S, r, id, tS[pos - 1], tr[pos - 1], ti[pos - 1])) {
        tS[pos] = tS[pos - 1];
        tr[pos] = tr[pos - 1];
        ti[pos] = ti[pos - 1];
        --pos;
      }
      tS[pos] = S;
      tr[pos] = r;
      ti[pos] = id;
    }
    *(volatile unsigned *)&p.g_ntop[g] = cnt;
    publish_thresh(p, g);
    unlock_list(p, g);
  }
  __syncthreads();
}

template <int W>
__device__ __forceinline__ void merge_topk(const RunParams &p, Smem<W> &sm) {
  __shared__ int s_ok;
  if (sm.ncand == 0) return;
  const int g = p.ng == 1 ? 0 : p.g_bu ? p.ctl->bgraph : -1;
  if (g < 0) {
    merge_topk_many(p, sm);
    return;
  }
  if (threadIdx.x == 0) s_ok = lock_list(p, g);
  __syncthreads();
  if (!s_ok) return;
  __threadfence();
  merge_topk_one(p, sm, g);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    publish_thresh(p, g);
    unlock_list(p, g);
  }
  __syncthreads();
}

__device__ __forceinline__ void graph_count(const RunParams &p, uint32_t g, int which, u64 v) {
  if (p.g_ctr && v) atomicAdd(&p.g_ctr[(size_t)g * 4 + which], v);
}

// Adds a finished search to the candidate list if it can enter the top list.
template <int W>
__device__ __forceinline__ void offer_candidate(const RunParams &p, Smem<W> &sm, u64 S, uint32_t r, uint32_t v,
                                                uint32_t g, const Thresh &x) {
  if (x.have && !entry_less(p.harmonic, S, r, v, x.S, x.r, x.id)) return;
  unsigned pos = atomicAdd(&sm.ncand, 1u);
  sm.cS[pos] = S;
  sm.cr[pos] = r;
  sm.cid[pos] = v;
  sm.cg[pos] = g;
}

// Epilogue after a level: update every active slot, merge finished searches,
// apply the cut test, choose the next step.
__device__ __forceinline__ void trace_stamp(const RunParams &p, int slot) {
  if (p.trace && threadIdx.x == 0) {
    u64 idx = ((volatile Ctl *)p.ctl)->trace_n;
    if (idx < p.trace_cap) {
      const u64 t = now_ns();
      p.trace[idx * 16 + slot] = t;
    }
  }
}

// Direction of the next level: bottom-up when the frontier's arcs are a large
// share of all arcs; several graphs, and the batch's searches all in one:
// of that graph's arcs (a batch of several graphs stays top-down).
__device__ __forceinline__ int choose_dir(const RunParams &p, u64 fl_arcs) {
  u64 arcs = p.arcs;
  if (p.g_bu) {
    const int g = p.ctl->bgraph;
    if (g < 0) return 0;
    arcs = p.off[p.g_base[g + 1]] - p.off[p.g_base[g]];
  }
  return ((u128)fl_arcs * p.bu_num > (u128)arcs * p.bu_den) ? 1 : 0;
}

// Frontier lists at most this long are never compacted (the pass and its
// barrier would cost more than the dead entries).
constexpr uint32_t kCompactMin = 4096;

// Runs in one block while the team waits, so it is written for few dependent
// round trips to L2: slots, counters, the threshold and the control words are
// loaded together, a thread keeps its slot in registers, statistics are added
// without waiting, and the threshold is read again only after a merge.
template <int W>
__device__ __noinline__ void epilogue_level(const RunParams &p, Smem<W> &sm) {
  static_assert(64 * W <= kMinThreads, "a thread per slot");
  Ctl *c = p.ctl;
  trace_stamp(p, 13);
  const uint32_t s = threadIdx.x;
  Slot sl;
  unsigned cn = 0;
  u64 ws = 0;
  bool act = false;
  if (s < p.B) {
    sl = p.slots[s];
    cn = p.cnt[s];
    ws = p.wsum[s];
    act = sl.state == 1;
  }
  Thresh x = thresh_of(p, p.ng == 1 || !act ? 0u : sl.graph);
  // the level just run (thread 0)
  u64 packed = 0, fa = 0, lsv = 0, lsa = 0, lsr = 0;
  uint32_t fl = 0;
  int dir = 0;
  if (threadIdx.x == 0) {
    volatile Ctl *vc = c;
    packed = vc->nl_packed;
    fa = vc->fl_arcs;
    lsv = vc->lvl_scan_v;
    lsa = vc->lvl_scan_a;
    lsr = vc->lvl_scan_r;
    fl = vc->fl_count;
    dir = vc->dir;
    sm.ncand = 0;
    sm.nactive = 0;
  }
  if (threadIdx.x < 4) sm.acc[threadIdx.x] = 0;
  __syncthreads();
  // 1. per-slot level update
  bool cont = false;
  if (act) {
    p.cnt[s] = 0;
    p.wsum[s] = 0;
    if (cn == 0) {
      // the BFS from sl.v is complete: S and r = n_d are exact
      sl.state = 2;
      const u64 key = p.harmonic ? (u64)__double_as_longlong(sl.H) : sl.S;
      p.res_S[sl.v] = key;
      p.res_r[sl.v] = (uint32_t)sl.nd;
      p.slots[s].state = 2;
      graph_count(p, sl.graph, 3, 1);
      offer_candidate(p, sm, key, (uint32_t)sl.nd, sl.v, sl.graph, x);
    } else {
      const int directed = p.g_directed ? p.g_directed[sl.graph] : p.directed;
      sl.d += 1;
      if (p.hist) {
        if (sl.d < p.hist_cap)
          p.hist[((size_t)p.team * p.B + s) * p.hist_cap + sl.d] = cn;
        else
          atomicCAS(&c->err, 0, TKC_EOVERFLOW);
      }
      sl.S += (u64)sl.d * cn;
      if (p.harmonic) sl.H = __dadd_rn(sl.H, __ddiv_rn((double)cn, (double)sl.d));
      sl.nd += cn;
      sl.g = ws - (directed ? 0ull : (u64)cn);
      sl.arcs = ws;
      cont = true;
    }
  }
  __syncthreads();
  // 2. top-k merge and the new threshold
  if (sm.ncand) {
    merge_topk(p, sm);
    if (cont) x = thresh_of(p, p.ng == 1 ? 0u : sl.graph);
  }
  // 3. BFSCut test for the slots that continue
  bool below = false;
  if (cont) {
    below = !p.nocut && !sl.nocut && x.have &&
                       (p.harmonic ? harmonic_below(sl.H, sl.d, sl.nd, sl.g, sl.omega, x.S)
                                   : cut_exceeds(sl.S, sl.d, sl.nd, sl.g, sl.alpha, sl.omega, x.S, x.r));
    if (below) {
      p.slots[s].state = 2;
      graph_count(p, sl.graph, 2, 1);
    } else {
      p.slots[s] = sl;
      graph_count(p, sl.graph, 0, sl.arcs);
    }
  }
  // the warp's slots together: a thread per slot, so a warp's continuing slots
  // are half a word of the active mask (arcs are below 2^32: two 16-bit sums)
  if (threadIdx.x < 64 * W) {
    const bool stay = cont && !below;
    const unsigned m = __ballot_sync(FULL, stay), mf = __ballot_sync(FULL, act && !cont), mc = __ballot_sync(FULL, below);
    const uint32_t arcs = stay ? (uint32_t)sl.arcs : 0u;
    const uint32_t lo = __reduce_add_sync(FULL, arcs & 0xffffu), hi = __reduce_add_sync(FULL, arcs >> 16);
    if ((threadIdx.x & 31) == 0) {
      reinterpret_cast<uint32_t *>(sm.active)[threadIdx.x >> 5] = m;
      if (m) {
        atomicAdd(&sm.nactive, (unsigned)__popc(m));
        atomicAdd(&sm.acc[2], lo + ((u64)hi << 16));
      }
      if (mf) atomicAdd(&sm.acc[0], (u64)__popc(mf));
      if (mc) atomicAdd(&sm.acc[1], (u64)__popc(mc));
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const u64 nl = packed >> kPackShift, nla = packed & kArcMask;
    // next step first, then the statistics
    c->nl_packed = 0;
    c->cur ^= 1;
    c->lcur ^= 1;
    c->bdepth += 1;
    c->fl_count = (uint32_t)nl;
    c->fl_arcs = nla;
    c->fl_list = dir == 0;
    if (dir != 0) c->clear_all = 1;
    c->level_id += 1;
#pragma unroll
    for (int j = 0; j < W; ++j) c->active[j] = sm.active[j];
    if (sm.nactive == 0) {
      c->step = 1;  // clear the batch's rows, then seed the next batch
    } else if (nl > kCompactMin && sm.acc[2] * 2 < nla) {
      // the new frontier list was built before this level's cuts: when the
      // surviving searches' own frontier arcs (sm.acc[2], an upper bound on
      // the arcs of the list entries they still use) are less than half of
      // the list's, compact it first, so that the level neither expands nor
      // (bottom-up) matches against rows of abandoned searches
      c->step = 2;
    } else {
      const int next = choose_dir(p, nla);
      if (next == 0 && dir != 0) {
        c->step = 2;  // the bottom-up level left no list: build it from the bitmap
      } else {
        c->step = 0;
        c->dir = next;
      }
    }
    // cost model of the level just run (bytes that must move):
    //  top-down : per frontier vertex list+offsets (16) + F row read and clear;
    //             per frontier arc column (4) + seen row read + N row update;
    //             per new vertex list (8) + N read/clear, seen read/write, F write
    //  bottom-up: per swept list entry (vertices with an in-arc) the entry (4)
    //             and its seen row; per scanned vertex in-offsets (8); per
    //             scanned in-arc its column (4) and frontier-bitmap word (4);
    //             per F row loaded the row; per new vertex seen/F writes; per
    //             old frontier vertex F row clear
    const u64 rb = 8ull * W;
    u64 bytes;
    if (dir == 0) {
      bytes = fl * (16 + 2 * rb) + fa * (4 + 2 * rb) + nl * (8 + 5 * rb);
      atomicAdd(&c->st_td_levels, 1ull);
      atomicAdd(&c->st_td_frontier, (u64)fl);
      atomicAdd(&c->st_td_arcs, fa);
      atomicAdd(&c->st_td_new, nl);
    } else {
      const u64 swept = p.g_bu ? p.g_bu[2 * (size_t)c->bgraph] : p.bu_list ? p.n_bu : p.n;
      bytes = swept * (4 + rb) + lsv * 8 + lsa * 8 + lsr * rb + nl * 2 * rb + fl * rb;
      atomicAdd(&c->st_bu_levels, 1ull);
      atomicAdd(&c->st_bu_swept, swept);
      atomicAdd(&c->st_bu_rows, lsr);
      atomicAdd(&c->st_bu_scan_v, lsv);
      atomicAdd(&c->st_bu_scan_a, lsa);
      atomicAdd(&c->st_bu_new, nl);
      atomicAdd(&c->st_bu_frontier, (u64)fl);
      c->lvl_scan_v = 0;
      c->lvl_scan_a = 0;
      c->lvl_scan_r = 0;
    }
    atomicAdd(&c->alg_bytes, bytes);
    if (sm.acc[0]) atomicAdd(&c->bfs_finished, sm.acc[0]);
    if (sm.acc[1]) atomicAdd(&c->bfs_cut, sm.acc[1]);
    if (sm.acc[2]) atomicAdd(&c->edges_visited, sm.acc[2]);
    atomicAdd(&c->levels, 1ull);
    if (p.trace) {
      u64 idx = c->trace_n++;
      if (idx < p.trace_cap) {
        const u64 t = now_ns();
        u64 *rec = p.trace + idx * 16;
        rec[0] = t;
        rec[1] = (u64)dir;
        rec[2] = fl;
        rec[3] = fa;
        rec[4] = nl;
        rec[5] = lsv;
        rec[6] = lsa;
        rec[7] = sm.nactive;
      }
    }
  }
  __syncthreads();
}

// Epilogue after a compaction step: the compacted list (built in the next-list
// buffer, from the old list or from the frontier's bitmap) becomes the frontier list, and the level's direction is chosen from
// its arcs.
template <int W>
__device__ __noinline__ void epilogue_compact(const RunParams &p, Smem<W> &sm) {
  Ctl *c = p.ctl;
  if (threadIdx.x == 0) {
    const u64 packed = c->nl_packed;
    const u64 before = c->fl_count, after = packed >> kPackShift;
    c->nl_packed = 0;
    c->lcur ^= 1;
    c->fl_count = (uint32_t)after;
    c->fl_arcs = packed & kArcMask;
    c->fl_list = 1;
    c->st_compactions += 1;
    c->st_compact_dropped += before - after;
    // list entry and row read per old entry, row cleared per dropped one, list written per kept one
    c->alg_bytes += before * (4 + 8ull * W) + (before - after) * 8ull * W + after * 8;
    c->step = 0;
    c->dir = choose_dir(p, c->fl_arcs);
  }
  __syncthreads();
}

// The bound after level 1 of source v (S_1 = its out-degree, n_1 = 1 more, at
// most g2 vertices at distance 2) exceeds the threshold.
__device__ __forceinline__ bool level1_exceeds(const RunParams &p, uint32_t od, uint32_t alpha, uint32_t omega,
                                               u64 g2, u64 xS, uint32_t xr) {
  if (p.harmonic) return harmonic_below((double)od, 1, 1ull + od, g2, omega, xS);
  return cut_exceeds(od, 1, 1ull + od, g2, alpha, omega, xS, xr);
}

// omega of v, capped by what its graph can reach at all.
__device__ __forceinline__ uint32_t omega_of(const RunParams &p, uint32_t v, uint32_t g) {
  const uint32_t o = p.omega[v];
  if (!p.n_cls) return o;
  const uint32_t *nc = p.n_cls + 4 * (size_t)g;
  const uint32_t cap = nc[0] + nc[1] + nc[2] + nc[3] + 1;
  return o < cap ? o : cap;
}

// Several graphs after their openings, the order graph by graph: takes up to
// `room` positions of one graph -- of graph `same` (0xffffffff: any) -- so that
// a batch's searches share one graph's arcs and may run bottom-up over it.
// Returns the first position (p.norder: none) and their number in *take.  (A
// failed exchange means another team took positions.)
__device__ __forceinline__ uint32_t take_of_graph(const RunParams &p, uint32_t room, uint32_t same, uint32_t *take) {
  uint32_t cur = *(volatile unsigned *)&p.sh->cursor;
  while (cur < p.norder) {
    const uint32_t g = p.gid[p.order[cur]];
    if (same != 0xffffffffu && g != same) break;
    const uint32_t end = p.g_end[g];
    const bool stopped = p.lb_key && *(volatile unsigned *)&p.g_stop[g];
    const uint32_t next = stopped || end - cur < room ? end : cur + room;
    const uint32_t old = atomicCAS(&p.sh->cursor, cur, next);
    if (old != cur) {
      cur = old;
    } else if (stopped) {
      cur = next;
    } else {
      *take = next - cur;
      return cur;
    }
  }
  *take = 0;
  return p.norder;
}

// Epilogue after a clear step: seed the next batch of up to B sources.
template <int W>
__device__ __noinline__ void epilogue_seed(const RunParams &p, Smem<W> &sm) {
  Ctl *c = p.ctl;
  trace_stamp(p, 13);
  const uint32_t B = p.B;
  u64 *Fcur = c->cur ? p.F1 : p.F0;
  uint32_t *FBcur = c->cur ? p.FB1 : p.FB0;
  uint32_t *FL = c->lcur ? p.L1 : p.L0;
  uint32_t *FLoff = c->lcur ? p.Loff1 : p.Loff0;
  uint32_t assigned = 0, last_base = 0;
  u64 arcs_total = 0, started = 0, cut0 = 0;
  __shared__ uint32_t s_base, s_take, s_gmin, s_gmax;
  __shared__ int s_gate;
  if (threadIdx.x == 0) {
    s_gmin = 0xffffffffu;
    s_gmax = 0;
  }
  if (threadIdx.x < W) sm.active[threadIdx.x] = 0;
  // One graph and several teams, no threshold yet: the other teams start only
  // after team 0's first batch.  Until then every source they took would be
  // searched to the end; afterwards most are abandoned at once.
  if (threadIdx.x == 0) {
    volatile Shared *vsh = p.sh;
    if (p.team == 0 && c->batches >= 1) vsh->first_done = 1u;
    s_gate = p.teams > 1 && p.team != 0 && p.ng == 1 && !p.nocut && vsh->first_done == 0u &&
             vsh->cursor < p.norder && vsh->err == 0 && !thresh_of(p, 0).have;
  }
  __syncthreads();
  if (s_gate) {
    if (threadIdx.x == 0) {
      __nanosleep(2000);
      c->fl_count = 0;
      c->fl_arcs = 0;
      c->vl_count = 0;
      c->clear_all = 0;
      c->nl_packed = 0;
      c->level_id += 1;
      for (int j = 0; j < W; ++j) c->active[j] = 0;
      c->step = 1;  // another empty clear step, then this check again
    }
    for (uint32_t s = threadIdx.x; s < B; s += blockDim.x) p.slots[s].state = 0;
    __syncthreads();
    return;
  }
  // take sources from the shared cursor, `room` positions at a time, so that
  // every position taken is either abandoned at level 0 or gets a slot
  // (updateBoundsLB runs: one batch per team, its levels are read afterwards)
  const bool lb_done = p.lvl && c->batches >= 1;
  while (!lb_done && assigned < B) {
    const uint32_t room = B - assigned;
    if (threadIdx.x == 0) {
      if (p.g_bu && p.g_end && p.g_rest == 0)
        s_base = take_of_graph(p, room, assigned ? s_gmin : 0xffffffffu, &s_take);
      else {
        s_base = atomicAdd(&p.sh->cursor, room);
        s_take = room;
      }
    }
    __syncthreads();
    const uint32_t base = s_base, most = s_take;
    __syncthreads();
    if (base >= p.norder) break;
    last_base = base;
    const uint32_t cnt = most < p.norder - base ? most : p.norder - base;
    const uint32_t idx = base + threadIdx.x;
    const bool valid = threadIdx.x < cnt;
    uint32_t v = valid ? p.order[idx] : 0;
    const uint32_t sv = valid && p.lab ? p.lab[v] : v;  // its row's label
    uint32_t od = valid ? p.off[sv + 1] - p.off[sv] : 0;
    uint32_t gv = (valid && p.gid) ? p.gid[v] : 0;
    uint32_t a = valid ? p.alpha[v] : 0, o = valid ? omega_of(p, v, gv) : 0;
    // level 0: S_0 = 0, n_0 = 1, gamma_1 = out-degree
    // (cut1: abandoned after level 1, whose arcs count as visited)
    bool cut = false, cut1 = false, stop = false;
    // several graphs: a graph whose search stopped skips its later sources
    const bool stopped = valid && p.lb_key && p.gid && *(volatile unsigned *)&p.g_stop[gv];
    if (valid && !stopped && !p.nocut && idx >= p.nocut_prefix) {
      Thresh x = thresh_of(p, gv);
      if (p.harmonic) {
        stop = x.have && p.lb_key &&
               __dmul_rn(__longlong_as_double((long long)~p.lb_key[v]), kHMargin) <
                   __longlong_as_double((long long)x.S);
        cut = !stop && x.have && harmonic_below(0.0, 0, 1, od, o, x.S);
        cut1 = !stop && x.have && !cut && p.lvl2 && level1_exceeds(p, od, a, o, p.lvl2[v], x.S, x.r);
      } else {
        stop = x.have && p.lb_key && nb_exceeds(p.lb_key[v], x.S, x.r);
        cut = !stop && x.have && cut_exceeds(0, 0, 1, od, a, o, x.S, x.r);
        cut1 = !stop && x.have && !cut && p.lvl2 && level1_exceeds(p, od, a, o, p.lvl2[v], x.S, x.r);
      }
      cut |= cut1;
    }
    // nothing after a stopped position of its graph is searched, by any team
    if (stop) {
      if (!p.gid) {
        atomicMax(&p.sh->cursor, p.norder);
      } else {
        *(volatile unsigned *)&p.g_stop[gv] = 1u;
        // sources graph by graph: the rest of this graph's run is skipped at
        // once (only after the openings, where the run is contiguous)
        if (p.g_end && idx >= p.g_rest) atomicMax(&p.sh->cursor, p.g_end[gv]);
      }
    }
    if (stopped && p.g_end && idx >= p.g_rest) atomicMax(&p.sh->cursor, p.g_end[gv]);
    const bool take = valid && !cut && !stop && !stopped;
    uint32_t total;
    uint32_t pre = block_exscan(sm, take ? 1u : 0u, &total);
    if (cut) {
      graph_count(p, gv, 1, 1);
      graph_count(p, gv, 2, 1);
      if (cut1) {
        graph_count(p, gv, 0, od);
        atomicAdd(&c->edges_visited, (u64)od);
      }
    }
    uint32_t s = assigned + pre;
    u64 myarcs = take ? od : 0;
    u64 arcs_pre_total;
    u64 arcs_pre = block_exscan64(sm, myarcs, &arcs_pre_total);
    if (take) {
      Slot sl;
      sl.S = 0;
      sl.nd = 1;
      sl.g = od;
      sl.arcs = od;
      sl.v = v;
      sl.d = 0;
      sl.alpha = a;
      sl.omega = o;
      sl.state = 1;
      sl.graph = gv;
      sl.nocut = idx < p.nocut_prefix;
      sl.pad = 0;
      sl.H = 0.0;
      if (p.g_bu) {
        atomicMin(&s_gmin, gv);
        atomicMax(&s_gmax, gv);
      }
      if (p.lvl_src) p.lvl_src[p.team * B + s] = v;
      p.slots[s] = sl;
      graph_count(p, gv, 1, 1);
      graph_count(p, gv, 0, od);
      u64 bit = 1ull << (s & 63);
      p.seen[(size_t)sv * W + (s >> 6)] = bit;
      Fcur[(size_t)sv * W + (s >> 6)] = bit;
      atomicOr(&FBcur[sv >> 5], 1u << (sv & 31));
      FL[s] = sv;
      FLoff[s] = (uint32_t)(arcs_total + arcs_pre);
      p.VL[s] = sv;
      atomicOr(reinterpret_cast<uint32_t *>(sm.active) + (s >> 5), 1u << (s & 31));
    }
    uint32_t ncut;
    block_exscan(sm, cut ? 1u : 0u, &ncut);
    assigned += total;
    arcs_total += arcs_pre_total;
    started += total + ncut;
    cut0 += ncut;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // the clear step just zeroed these rows
    const u64 seen_rows = !c->clear_all ? c->vl_count : c->bgraph >= 0 && p.g_bu ? p.g_base[c->bgraph + 1] - p.g_base[c->bgraph] : p.n;
    c->alg_bytes += (seen_rows + c->fl_count) * 8ull * W + (c->clear_all ? 0ull : 4ull * c->vl_count);
    c->st_cleared += seen_rows + c->fl_count;
    c->st_seeded += assigned;
    c->cursor = last_base;
    c->bfs_started += started;
    c->bfs_cut += cut0;
    c->edges_visited += arcs_total;
    c->fl_count = assigned;
    c->fl_arcs = arcs_total;
    c->fl_list = 1;
    c->clear_all = 0;
    c->vl_count = assigned;
    c->bdepth = 0;
    c->nl_packed = 0;
    c->level_id += 1;
    if (p.trace) {
      u64 idx = c->trace_n++;
      if (idx < p.trace_cap) {
        const u64 t = now_ns();
        u64 *rec = p.trace + idx * 16;
        rec[0] = t;
        rec[1] = 2;  // seed step
        rec[2] = assigned;
        rec[3] = arcs_total;
        rec[4] = last_base;
        rec[5] = cut0;
        rec[6] = c->vl_count;
        rec[7] = p.g_ntop[0];
      }
    }
    c->batches += 1;
    for (int j = 0; j < W; ++j) c->active[j] = sm.active[j];
    if (assigned == 0) {
      c->done = 1;
      if (p.team == 0) ((volatile Shared *)p.sh)->first_done = 1u;
    } else {
      c->step = 0;
      c->bgraph = s_gmin == s_gmax ? (int)s_gmin : -1;
      c->dir = choose_dir(p, arcs_total);
    }
  }
  // slots beyond `assigned` are free
  for (uint32_t s = assigned + threadIdx.x; s < B; s += blockDim.x) p.slots[s].state = 0;
  __syncthreads();
}

// ------------------------------------------------------------------ the kernel

template <int W, int TPB>
__global__ void __launch_bounds__(TPB, 1) bfscut_kernel(RunParams p0) {
  __shared__ Smem<W> sm;
  // this block's team: its own control block, slots, rows, lists and stamps
  __shared__ RunParams p;
  // teams: no more than batches left by the filter, each then of more blocks (at
  // most p0.team_blocks, a warp per 32 vertices); spare blocks leave at once
  uint32_t teams = p0.teams;
  if (p0.norder_dev && p0.ng == 1) {
    const uint32_t batches = (p0.sh->norder + p0.B - 1) / p0.B;
    teams = batches < teams ? (batches ? batches : 1u) : teams;
  }
  uint32_t bpt = gridDim.x / teams;  // blocks per team
  if (teams != p0.teams && bpt > p0.team_blocks) bpt = p0.team_blocks;
  const uint32_t team = blockIdx.x / bpt;
  const uint32_t tb = blockIdx.x % bpt;
  if (team >= teams) return;
  if (threadIdx.x == 0) {
    p = p0;
    p.teams = teams;
    p.team = team;
    p.ctl = p0.ctl + team;
    p.slots = p0.slots + (size_t)team * 64 * kMaxWords;
    p.cnt = p0.cnt + (size_t)team * 64 * kMaxWords;
    p.wsum = p0.wsum + (size_t)team * 64 * kMaxWords;
    p.seen = p0.seen + team * p0.row_stride;
    p.F0 = p0.F0 + team * p0.row_stride;
    p.F1 = p0.F1 + team * p0.row_stride;
    p.N = p0.N + team * p0.row_stride;
    p.FB0 = p0.FB0 + team * p0.fb_stride;
    p.FB1 = p0.FB1 + team * p0.fb_stride;
    p.L0 = p0.L0 + team * p0.vtx_stride;
    p.L1 = p0.L1 + team * p0.vtx_stride;
    p.Loff0 = p0.Loff0 + team * p0.vtx_stride;
    p.Loff1 = p0.Loff1 + team * p0.vtx_stride;
    p.VL = p0.VL + team * p0.vtx_stride;
    p.stamp = p0.stamp + team * p0.vtx_stride;
    if (p0.norder_dev) p.norder = p0.sh->norder;
    if (p0.bu_cnt) {
      p.n_bu = p0.bu_cnt[0];
      p.n_bu_heavy = p0.bu_cnt[1];
    }
    if (p0.trace) {
      p.trace_cap = p0.trace_cap / p0.teams;
      p.trace = p0.trace + (size_t)team * p.trace_cap * 16;
    }
    if (tb == 0) p.ctl->t_start = now_ns();
  }
  __syncthreads();
  Ctl *c = p.ctl;
  const int lane = threadIdx.x & 31;
  const uint32_t gwarp = (tb * TPB + threadIdx.x) >> 5;
  const uint32_t nwarps = (bpt * TPB) >> 5;
  const uint32_t gthread = tb * TPB + threadIdx.x;
  const uint32_t nthreads = bpt * TPB;

  while (true) {
    // the control words of this step, one round trip for all of them
    if (threadIdx.x < kCmdWords) sm.cmd[threadIdx.x] = ((volatile uint32_t *)&c->step)[threadIdx.x];
    __syncthreads();
    const Ctl *vc = reinterpret_cast<const Ctl *>(reinterpret_cast<const char *>(sm.cmd) - offsetof(Ctl, step));
    const int step = vc->step;
    if (vc->done) break;
    const int cur = vc->cur;
    u64 *Fcur = cur ? p.F1 : p.F0;
    u64 *Fnext = cur ? p.F0 : p.F1;
    uint32_t *FBcur = cur ? p.FB1 : p.FB0;
    uint32_t *FBnext = cur ? p.FB0 : p.FB1;
    const int lcur = vc->lcur;
    uint32_t *FL = lcur ? p.L1 : p.L0;
    uint32_t *FLoff = lcur ? p.Loff1 : p.Loff0;
    uint32_t *NL = lcur ? p.L0 : p.L1;
    uint32_t *NLoff = lcur ? p.Loff0 : p.Loff1;
    const uint32_t fl_count = vc->fl_count;
    // the vertices this batch's searches can touch
    const int bg = p.g_bu ? vc->bgraph : -1;
    const uint32_t v0 = bg >= 0 ? p.g_base[bg] : 0u, v1 = bg >= 0 ? p.g_base[bg + 1] : p.n;
    if (step == 1) {
      if (tb == 0) trace_stamp(p, 8);
      // ---- clear step: zero the rows touched by the finished batch
      if (vc->clear_all) {
        clear_rows<W>(p.seen, v0, v1, gthread, nthreads);
      } else {
        const uint32_t vl = vc->vl_count;
        for (uint64_t i = gthread; i < (uint64_t)vl * W; i += nthreads) {
          uint32_t v = p.VL[i / W];
          p.seen[(size_t)v * W + (i % W)] = 0;
        }
      }
      clear_old_frontier<W>(vc->fl_list, Fcur, FBcur, FL, fl_count, v0, v1, gthread, nthreads);
      if (tb == 0) trace_stamp(p, 12);
      if (!team_sync(c, p.sh, bpt, p.timeout, [&] { epilogue_seed<W>(p, sm); })) break;
      continue;
    }
    if (step == 2) {
      // ---- compaction: list the frontier vertices with a bit of a search
      // still active (rows masked to those bits); zero the rows and frontier
      // bits of the others, which only abandoned or finished searches used
      u64 act[W];
#pragma unroll
      for (int q = 0; q < W; ++q) act[q] = vc->active[q];
      auto keep_active = [&](uint32_t u, bool valid) {
        uint32_t od = 0;
        bool keep = false;
        if (valid) {
          u64 row[W], f[W];
          load_row<W>(Fcur, u, row);
          bool same = true;
#pragma unroll
          for (int q = 0; q < W; ++q) {
            f[q] = row[q] & act[q];
            same &= f[q] == row[q];
          }
          keep = row_nonzero<W>(f);
          if (!keep) atomicAnd(&FBcur[u >> 5], ~(1u << (u & 31)));
          if (!same) store_row<W>(Fcur, u, f);
          if (keep) od = p.off[u + 1] - p.off[u];
        }
        warp_append(keep, u, od, &c->nl_packed, NL, NLoff, lane);
      };
      if (vc->fl_list) {
        for (uint32_t base = gwarp * 32; base < fl_count; base += nwarps * 32) {
          const bool valid = base + lane < fl_count;
          keep_active(valid ? FL[base + lane] : 0u, valid);
        }
      } else {
        // no list: the frontier's bitmap, 32 words a warp, a word's vertices at a time
        const uint32_t w1 = v1 / 32 + 1;
        for (uint32_t base = v0 / 32 + gwarp * 32; base < w1; base += nwarps * 32) {
          const uint32_t word = base + lane < w1 ? FBcur[base + lane] : 0u;
          for (unsigned m = __ballot_sync(FULL, word != 0); m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            const uint32_t bits = __shfl_sync(FULL, word, src);
            keep_active((base + src) * 32 + lane, (bits >> lane) & 1u);
          }
        }
      }
      if (!team_sync(c, p.sh, bpt, p.timeout, [&] { epilogue_compact<W>(p, sm); })) break;
      continue;
    }
    if (tb == 0) trace_stamp(p, 8);
    const int dir = vc->dir;
    const uint32_t level_id = vc->level_id;
    const uint32_t depth = vc->bdepth + 1;  // depth of the level being discovered
    const u64 fl_arcs = vc->fl_arcs;
    if (threadIdx.x < W) sm.active[threadIdx.x] = vc->active[threadIdx.x];
    for (int i = threadIdx.x; i < 64 * W; i += TPB) {
      sm.cnt[i] = 0;
      sm.wsum[i] = 0;
    }
    if (threadIdx.x == 0) {
      sm.acc[2] = 0;
      sm.acc[3] = 0;
      sm.bu_next = 0;
      sm.bu_new = 0;
    }
    __syncthreads();
    u64 scanned = 0;
    uint32_t scanned_v = 0, rows_read = 0;
    if (dir == 0) {
      // ---- phase A, top-down: OR each frontier row into its out-neighbours' N rows
      constexpr uint32_t APS = 32 / W;  // arcs per warp step
      // arcs per warp task: about two tasks per warp, at least one step, so a
      // small level still spreads over every warp (each step is a chain of
      // dependent loads)
      constexpr int TU = W <= 2 ? 4 : 2;  // warp steps unrolled per iteration
      u64 CH = (fl_arcs + 2ull * nwarps - 1) / (2ull * nwarps);
      // (a frontier too small for TU steps on every warp: one task per warp, of
      // as few steps as that takes, since the level then lasts one task's chain)
      if (fl_arcs <= (u64)nwarps * (TU * APS)) {
        CH = (fl_arcs + nwarps - 1) / nwarps;
        CH = (CH + APS - 1) / APS * APS;
      } else {
        CH = (CH + TU * APS - 1) / (TU * APS) * (TU * APS);
      }
      const int grp = lane / W, j = lane % W;
      const u64 actj = sm.active[j];
      for (u64 base = (u64)gwarp * CH; base < fl_arcs; base += (u64)nwarps * CH) {
        u64 end = base + CH < fl_arcs ? base + CH : fl_arcs;
        // entry holding arc `base`: last i with FLoff[i] <= base, by a 32-way
        // search (one round trip per factor of 32)
        uint32_t lo = 0, hi = fl_count;
        while (hi - lo > 1) {
          const uint32_t stepw = (hi - lo + 31) / 32, at = lo + stepw * (uint32_t)lane;
          const unsigned m = __ballot_sync(FULL, lane == 0 || (at < hi && FLoff[at] <= base));
          lo += stepw * (31u - (uint32_t)__clz(m));
          hi = lo + stepw < hi ? lo + stepw : hi;
        }
        uint32_t ent = lo;
        // TU warp steps per iteration: every arc's loads are issued before
        // any arc's atomic
        for (u64 e0 = base; e0 < end; e0 += TU * APS) {
          u64 ew[TU];
          uint32_t iw[TU], uw[TU], ww[TU];
          u64 fw[TU], bw[TU], cw[TU];
          uint32_t ii = ent;
#pragma unroll
          for (int t = 0; t < TU; ++t) {
            ew[t] = e0 + (u64)t * APS + grp;
            if (ew[t] < end)
              while (ii + 1 < fl_count && FLoff[ii + 1] <= ew[t]) ++ii;
            iw[t] = ii;
          }
#pragma unroll
          for (int t = 0; t < TU; ++t) uw[t] = ew[t] < end ? FL[iw[t]] : 0;
#pragma unroll
          for (int t = 0; t < TU; ++t) fw[t] = ew[t] < end ? Fcur[(size_t)uw[t] * W + j] & actj : 0;
#pragma unroll
          for (int t = 0; t < TU; ++t) ww[t] = fw[t] ? p.col[p.off[uw[t]] + (uint32_t)(ew[t] - FLoff[iw[t]])] : 0;
#pragma unroll
          for (int t = 0; t < TU; ++t) {
            bw[t] = fw[t] ? fw[t] & ~p.seen[(size_t)ww[t] * W + j] : 0;
            cw[t] = fw[t] ? *(volatile u64 *)(p.N + (size_t)ww[t] * W + j) : 0;
          }
          // The word's first contributor saw it zero, so only those may be the
          // vertex's first: of one word the one whose OR met zero, of several
          // the one whose stamp is new.  Their degrees are loaded beside the
          // atomics, and the TU steps append together (one returning atomic).
          bool app[TU];
          uint32_t od[TU];
#pragma unroll
          for (int t = 0; t < TU; ++t) {
            const bool go = (bw[t] & ~cw[t]) != 0, first = go && cw[t] == 0;
            od[t] = first ? p.off[ww[t] + 1] - p.off[ww[t]] : 0;
            if constexpr (W == 1) {
              app[t] = go && atomicOr(p.N + ww[t], bw[t]) == 0;
            } else {
              if (go) atomicOr(p.N + (size_t)ww[t] * W + j, bw[t]);
              app[t] = first && atomicExch(&p.stamp[ww[t]], level_id) != level_id;
            }
          }
          warp_append_steps<TU>(app, ww, od, &c->nl_packed, NL, NLoff, lane);
          ent = __reduce_max_sync(FULL, ii);
        }
      }
      scanned = 0;
      if (gthread == 0) atomicAdd(&c->edges_scanned, fl_arcs);
      if (tb == 0) trace_stamp(p, 9);
      if (!team_sync(c, p.sh, bpt, p.timeout, [] {})) break;
      if (tb == 0) trace_stamp(p, 10);
      // ---- phase B: finalize the next level, clear the old frontier rows
      const uint32_t nl_count = (uint32_t)(((volatile Ctl *)c)->nl_packed >> kPackShift);
      for (uint32_t base = gwarp * 32; base < nl_count; base += nwarps * 32) {
        uint32_t i = base + lane;
        bool valid = i < nl_count;
        u64 nw[W], sr[W];
        uint32_t w = 0, od = 0;
        bool was_empty = false;
#pragma unroll
        for (int q = 0; q < W; ++q) nw[q] = 0;
        if (valid) {
          w = NL[i];
          od = p.off[w + 1] - p.off[w];
          load_row<W>(p.N, w, nw);
          load_row<W>(p.seen, w, sr);
          was_empty = !row_nonzero<W>(sr);
          u64 z[W];
#pragma unroll
          for (int q = 0; q < W; ++q) {
            sr[q] |= nw[q];
            z[q] = 0;
          }
          store_row<W>(p.seen, w, sr);
          store_row<W>(Fnext, w, nw);
          store_row<W>(p.N, w, z);
          atomicOr(&FBnext[w >> 5], 1u << (w & 31));
          if (p.lvl) record_levels<W>(p, w, nw, depth);
        }
        warp_count_slots<W>(nw, od, sm.cnt, sm.wsum, lane);
        if (!vc->clear_all) warp_append_plain(valid && was_empty, w, &c->vl_count, p.VL, lane);
      }
      clear_old_frontier<W>(vc->fl_list, Fcur, FBcur, FL, fl_count, v0, v1, gthread, nthreads);
    } else {
      // ---- phase A, bottom-up: each vertex ORs its in-neighbours' frontier rows
      u64 act[W];
#pragma unroll
      for (int q = 0; q < W; ++q) act[q] = sm.active[q];
      // Work items of the sweep list (vertices with an in-arc), dealt
      // round-robin to the team's blocks, whose warps take them from a shared
      // counter as they finish: first groups of 32 long in-rows, group j
      // holding list entries j, j + hg, j + 2 hg, ... so that the longest rows
      // land in different warps; then chunks of kBuChunkVerts consecutive
      // entries of the shorter rows (labels ascending), or of 32.
      const uint32_t *list = bg >= 0 ? p.bu_list + v0 : p.bu_list;
      const uint32_t nheavy = bg >= 0 ? p.g_bu[2 * bg + 1] : list ? p.n_bu_heavy : 0u;
      const uint32_t nlight = bg >= 0 ? p.g_bu[2 * bg] - nheavy : list ? p.n_bu - nheavy : p.n;
      const uint32_t hg = (nheavy + 31) / 32;
      // a frontier of more than half the swept vertices: its bits are not worth
      // testing (a row that is not on it is zero)
      const bool dense = (u64)fl_count * 2 > (u64)nheavy + nlight;
      u64 new_arcs = 0;
      uint32_t new_count = 0;
      // chunks of kBuChunkVerts entries, of 32 when that leaves warps with fewer
      // than four chunks: a level then waits for a warp's 32 entries, not 128
      const uint32_t bch = nlight >= 4 * kBuChunkVerts * nwarps ? kBuChunkVerts : 32u;
      const uint32_t nitems = hg + (nlight + bch - 1) / bch;
      for (;;) {
        uint32_t j = 0;
        if (lane == 0) j = atomicAdd(&sm.bu_next, 1u);
        j = __shfl_sync(FULL, j, 0);
        const u64 gi64 = (u64)tb + (u64)bpt * j;
        if (gi64 >= nitems) break;
        const uint32_t gi = (uint32_t)gi64;
        const bool hitem = gi < hg;
        const uint32_t g0 = hitem ? 0u : (gi - hg) * bch;
        const uint32_t g1 = hitem ? 32u : (g0 + bch < nlight ? g0 + bch : nlight);
        for (uint32_t base = g0; base < g1; base += 32) {
          bool valid;
          uint32_t w;
          if (hitem) {
            const uint32_t e = gi + hg * (uint32_t)lane;
            valid = e < nheavy;
            w = valid ? list[e] : 0;
          } else {
            valid = base + lane < g1;
            w = valid ? (list ? list[nheavy + base + lane] : base + lane) : 0;
          }
          u64 nw[W], sr[W], miss[W];
          uint32_t od = 0, e0 = 0, ee = 0;
          bool any = false, heavy = false;
#pragma unroll
          for (int q = 0; q < W; ++q) {
            nw[q] = 0;
            miss[q] = 0;
          }
          if (valid) {
            load_row<W>(p.seen, w, sr);
#pragma unroll
            for (int q = 0; q < W; ++q) {
              miss[q] = act[q] & ~sr[q];
              any |= miss[q] != 0;
            }
            e0 = p.ioff[w];
            ee = p.ioff[w + 1];
            heavy = any && ee - e0 > p.heavy_in;
            if (any && !heavy) {
              // U in-arcs per step, software-pipelined: step i's rows (of the
              // in-neighbours on a frontier) are loaded together with step
              // i+1's frontier bits and step i+2's columns, so a step waits on
              // one round trip instead of three (1.5% off the kernel on R-MAT
              // 22); the early exit is tested once per step (extra rows only
              // repeat found bits)
              constexpr int U = W >= 8 ? 2 : TKC_BU_U;
              uint32_t e = e0;
              uint32_t c0[U], c1[U], f0[U];
#pragma unroll
              for (int j = 0; j < U; ++j) {
                c0[j] = e + j < ee ? p.icol[e + j] : 0xffffffffu;
                c1[j] = e + U + j < ee ? p.icol[e + U + j] : 0xffffffffu;
              }
#pragma unroll
              for (int j = 0; j < U; ++j)
                f0[j] = c0[j] != 0xffffffffu && (dense || ((FBcur[c0[j] >> 5] >> (c0[j] & 31)) & 1u));
              for (; e < ee; e += U) {
                uint32_t c2[U], f1[U];
#pragma unroll
                for (int j = 0; j < U; ++j) c2[j] = e + 2 * U + j < ee ? p.icol[e + 2 * U + j] : 0xffffffffu;
#pragma unroll
                for (int j = 0; j < U; ++j)
                  f1[j] = c1[j] != 0xffffffffu && (dense || ((FBcur[c1[j] >> 5] >> (c1[j] & 31)) & 1u));
#pragma unroll
                for (int j = 0; j < U; ++j) {
                  if (f0[j]) {
                    u64 fr[W];
                    load_row<W>(Fcur, c0[j], fr);
                    ++rows_read;
#pragma unroll
                    for (int q = 0; q < W; ++q) nw[q] |= fr[q] & miss[q];
                  }
                }
                bool full = true;
#pragma unroll
                for (int q = 0; q < W; ++q) full &= nw[q] == miss[q];
                if (full) {
                  e += U;
                  break;
                }
#pragma unroll
                for (int j = 0; j < U; ++j) {
                  c0[j] = c1[j];
                  c1[j] = c2[j];
                  f0[j] = f1[j];
                }
              }
              scanned += (e < ee ? e : ee) - e0;
              scanned_v += 1;
            }
          }
          // vertices of high in-degree: the whole warp walks their in-arcs
          // (coalesced column reads, HU per lane per step) so that one lane does
          // not hold the level up; same result as the lane loop (the OR of the
          // frontier rows of in-neighbours, or every missing bit found)
          for (unsigned hv = __ballot_sync(FULL, heavy); hv; hv &= hv - 1) {
            const int src = __ffs(hv) - 1;
            const uint32_t hb = __shfl_sync(FULL, e0, src), he = __shfl_sync(FULL, ee, src);
            u64 hm[W], acc[W];
#pragma unroll
            for (int q = 0; q < W; ++q) {
              hm[q] = __shfl_sync(FULL, miss[q], src);
              acc[q] = 0;
            }
            constexpr int HU = W >= 8 ? 1 : W >= 4 ? 2 : TKC_BU_HU;
            uint32_t e = hb;
            // the next step's columns are loaded before this step's frontier
            // bits and rows are waited on, so their latency overlaps
            uint32_t nx[HU];
#pragma unroll
            for (int j = 0; j < HU; ++j) {
              const uint32_t i = hb + 32 * j + lane;
              nx[j] = i < he ? p.icol[i] : 0xffffffffu;
            }
            for (; e < he; e += 32 * HU) {
              uint32_t uu[HU], fb[HU];
#pragma unroll
              for (int j = 0; j < HU; ++j) {
                uu[j] = nx[j];
                const uint32_t i = e + 32 * HU + 32 * j + lane;
                nx[j] = i < he ? p.icol[i] : 0xffffffffu;
              }
#pragma unroll
              for (int j = 0; j < HU; ++j)
                fb[j] = uu[j] != 0xffffffffu && (dense || ((FBcur[uu[j] >> 5] >> (uu[j] & 31)) & 1u));
#pragma unroll
              for (int j = 0; j < HU; ++j) {
                if (fb[j]) {
                  u64 fr[W];
                  load_row<W>(Fcur, uu[j], fr);
                  ++rows_read;
#pragma unroll
                  for (int q = 0; q < W; ++q) acc[q] |= fr[q] & hm[q];
                }
              }
              // early exit once every missing bit is found
              bool full = true;
#pragma unroll
              for (int q = 0; q < W; ++q) full &= warp_or(acc[q]) == hm[q];
              if (full) {
                e += 32 * HU;
                break;
              }
            }
#pragma unroll
            for (int q = 0; q < W; ++q) acc[q] = warp_or(acc[q]);
            if (lane == src) {
#pragma unroll
              for (int q = 0; q < W; ++q) nw[q] = acc[q];
              scanned += (e < he ? e : he) - hb;
              scanned_v += 1;
            }
          }
          bool isnew = valid && row_nonzero<W>(nw);
          if (isnew) {
            od = p.off[w + 1] - p.off[w];
#pragma unroll
            for (int q = 0; q < W; ++q) sr[q] |= nw[q];
            store_row<W>(p.seen, w, sr);
            store_row<W>(Fnext, w, nw);
            if (p.lvl) record_levels<W>(p, w, nw, depth);
          }
          // the next frontier's bitmap starts all zero (each level clears the
          // bits of its own frontier), so setting the new vertices' bits
          // suffices: one atomic per bitmap word the group's new vertices share
          // (shorter rows: labels ascending, a few words), one per vertex for the
          // long rows (labels scattered)
          if (hitem) {
            if (isnew) atomicOr(&FBnext[w >> 5], 1u << (w & 31));
          } else {
            for (unsigned pend = __ballot_sync(FULL, isnew); pend;) {
              const int l = __ffs(pend) - 1;
              const uint32_t word = __shfl_sync(FULL, w >> 5, l);
              const bool mine = isnew && (w >> 5) == word;
              const unsigned bits = __reduce_or_sync(FULL, mine ? 1u << (w & 31) : 0u);
              if (lane == l) atomicOr(&FBnext[word], bits);
              pend &= ~__ballot_sync(FULL, mine);
            }
          }
          warp_count_slots<W>(nw, od, sm.cnt, sm.wsum, lane);
          // counted, not listed: a list costs two more round trips of atomics
          // per 32 vertices, and the next bottom-up level needs none
          new_arcs += od;
          new_count += isnew;
        }
      }
      for (int o = 16; o > 0; o >>= 1) new_arcs += __shfl_down_sync(FULL, new_arcs, o);
      new_count = __reduce_add_sync(FULL, new_count);
      if (lane == 0 && new_count) atomicAdd(&sm.bu_new, ((u64)new_count << kPackShift) | new_arcs);
      if (tb == 0) trace_stamp(p, 9);
      if (!team_sync(c, p.sh, bpt, p.timeout, [] {})) break;
      if (tb == 0) trace_stamp(p, 10);
      // ---- phase B: only the old frontier rows need clearing
      clear_old_frontier<W>(vc->fl_list, Fcur, FBcur, FL, fl_count, v0, v1, gthread, nthreads);
    }
    if (tb == 0) trace_stamp(p, 11);
    // flush the block's per-slot counters
    // (a lane's counts are below 2^32: half-words add up in one reduction each)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) scanned += __shfl_down_sync(FULL, scanned, o);
    scanned_v = __reduce_add_sync(FULL, scanned_v);
    const u64 rows64 = (u64)__reduce_add_sync(FULL, rows_read & 0xffffu) +
                       ((u64)__reduce_add_sync(FULL, rows_read >> 16) << 16);
    if (lane == 0 && scanned) atomicAdd(&sm.acc[3], scanned);
    if (lane == 0 && scanned_v) atomicAdd(&sm.acc[2], (u64)scanned_v);
    if (lane == 0 && rows64) atomicAdd(&c->lvl_scan_r, rows64);
    __syncthreads();
    for (int i = threadIdx.x; i < 64 * W; i += TPB) {
      if (sm.cnt[i]) {
        atomicAdd(&p.cnt[i], sm.cnt[i]);
        atomicAdd(&p.wsum[i], (u64)sm.wsum[i]);
      }
    }
    if (threadIdx.x == 0 && sm.acc[3]) {
      atomicAdd(&c->edges_scanned, sm.acc[3]);
      atomicAdd(&c->lvl_scan_a, sm.acc[3]);
    }
    if (threadIdx.x == 0 && sm.acc[2]) atomicAdd(&c->lvl_scan_v, sm.acc[2]);
    if (threadIdx.x == 0 && sm.bu_new) atomicAdd(&c->nl_packed, sm.bu_new);
    if (tb == 0) trace_stamp(p, 12);
    if (!team_sync(c, p.sh, bpt, p.timeout, [&] { epilogue_level<W>(p, sm); })) break;
  }
  if (tb == 0 && threadIdx.x == 0) c->t_end = now_ns();
}

// ------------------------------------------------------------------ before the launches

// Zeroes the control blocks (each starts with an empty clear step, whose
// epilogue seeds the first batch), the shared block and, with nlist > 0, the
// per-graph list state and res_r of n vertices.
__global__ void k_run_init(Ctl *ctl, uint32_t nctl, unsigned level_base, Shared *sh, uint32_t nlist, unsigned *g_ntop,
                           unsigned *g_stop, int *g_lock, u64 *g_ctr, ulonglong2 *x, uint32_t *res_r,
                           uint32_t n) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
  static_assert(sizeof(Ctl) % 8 == 0, "control blocks are zeroed by 64-bit words");
  for (uint32_t i = t; i < nctl * (uint32_t)(sizeof(Ctl) / 8); i += nt) {
    const uint32_t w = i % (uint32_t)(sizeof(Ctl) / 8);
    if (w == offsetof(Ctl, step) / 8 || w == offsetof(Ctl, level_id) / 8) continue;
    reinterpret_cast<u64 *>(ctl)[i] = 0;
  }
  for (uint32_t i = t; i < nctl; i += nt) {
    // the two words skipped above
    u64 *w = reinterpret_cast<u64 *>(ctl + i);
    w[offsetof(Ctl, step) / 8] = 0;
    w[offsetof(Ctl, level_id) / 8] = 0;
    ctl[i].step = 1;
    ctl[i].level_id = level_base;
  }
  if (t == 0) *sh = Shared{};
  for (uint32_t i = t; i < nlist; i += nt) {
    g_ntop[i] = g_stop[i] = 0;
    g_lock[i] = 0;
    x[i] = make_ulonglong2(0, 0);
    for (int j = 0; j < 4; ++j) g_ctr[4 * (size_t)i + j] = 0;
  }
  if (nlist)
    for (uint32_t i = t; i < n; i += nt) res_r[i] = 0;
}

// Between the opening and the main launch: the sources of order[0, count)
// that the thresholds so far abandon before they start -- by NBCut's stop
// (not counted, as at seeding), by the level-0 bound, or by the bound after
// level 1 with a level-2 size from in-degree classes -- are dropped in one
// grid-wide pass, so that the teams' batches hold only sources that search.
//
// Level 2 of a source holds, of the n_c vertices of class c, at most
// min(n_c, walks of length 2 ending in class c): vertices of small in-degree
// are counted almost exactly, and the many walks that end in the few vertices
// of large in-degree count each of those once.  (The plain sum of walks, which
// gamma and the NB bounds use, exceeds the graph for any hub.)  A source left
// over is searched with that bound in lvl2, tested again when it is seeded.
//
// Positions are dealt to the blocks with a stride, since sources of long rows
// are neighbours in the order; a lane sums a row of at most kRowLane arcs, a
// warp one of at most kRowWarp, the block longer ones, four loads in flight
// per thread.  keep: a flag per position; tile_cnt: kept positions per tile of
// `tile`; taken: positions already searched by the opening (nullable, the
// first ntaken).
constexpr int kFilterTPB = 256;
constexpr uint32_t kRowLane = 16, kRowWarp = 512;

__device__ __forceinline__ void add4(uint4 &a, const uint4 &b) {
  a.x += b.x;
  a.y += b.y;
  a.z += b.z;
  a.w += b.w;
}

// Sums of the class counts over the out-neighbours row[0, len), every
// `step`-th from the first.  (Each sum is at most the graph's arcs, below 2^32.)
__device__ __forceinline__ uint4 sum_classes(const uint32_t *__restrict__ row, const uint4 *__restrict__ cls,
                                             uint32_t len, uint32_t step) {
  uint4 s = make_uint4(0, 0, 0, 0);
  uint32_t i = 0;  // len is below 2^26
  for (; i + 3 * step < len; i += 4 * step) {
    uint4 c[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) c[j] = cls[row[i + j * step]];
#pragma unroll
    for (int j = 0; j < 4; ++j) add4(s, c[j]);
  }
  for (; i < len; i += step) add4(s, cls[row[i]]);
  return s;
}

__device__ __forceinline__ uint4 warp_sum4(uint4 t) {
  t.x = __reduce_add_sync(FULL, t.x);
  t.y = __reduce_add_sync(FULL, t.y);
  t.z = __reduce_add_sync(FULL, t.z);
  t.w = __reduce_add_sync(FULL, t.w);
  return t;
}

struct RowScratch {
  unsigned n;
  uint32_t b[kFilterTPB], len[kFilterTPB];
  uint4 sum[kFilterTPB];
};

// Every thread's sum over its own row col[b, b + len) (len 0: none); called by
// the whole block.
__device__ __forceinline__ uint4 block_sum_rows(RowScratch &rs, const uint32_t *__restrict__ col,
                                                const uint4 *__restrict__ cls, uint32_t b, uint32_t len) {
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) rs.n = 0;
  __syncthreads();
  uint4 s = make_uint4(0, 0, 0, 0);
  unsigned slot = 0;
  if (len > kRowWarp) {
    slot = atomicAdd(&rs.n, 1u);
    rs.b[slot] = b;
    rs.len[slot] = len;
    rs.sum[slot] = s;
  }
  if (len <= kRowLane) s = sum_classes(col + b, cls, len, 1);
  for (unsigned m = __ballot_sync(FULL, len > kRowLane && len <= kRowWarp); m; m &= m - 1) {
    const int src = __ffs(m) - 1;
    const uint32_t rb = __shfl_sync(FULL, b, src), rl = __shfl_sync(FULL, len, src);  // rl >= 17
    uint4 t = make_uint4(0, 0, 0, 0);
    if ((uint32_t)lane < rl) t = sum_classes(col + rb + lane, cls, rl - lane, 32);
    t = warp_sum4(t);
    if (lane == src) s = t;
  }
  __syncthreads();
  for (unsigned i = 0; i < rs.n; ++i) {
    // rows longer than kRowWarp hold at least one arc per thread of the block
    const uint4 t = warp_sum4(sum_classes(col + rs.b[i] + threadIdx.x, cls, rs.len[i] - threadIdx.x, kFilterTPB));
    if (lane == 0) {
      atomicAdd(&rs.sum[i].x, t.x);
      atomicAdd(&rs.sum[i].y, t.y);
      atomicAdd(&rs.sum[i].z, t.z);
      atomicAdd(&rs.sum[i].w, t.w);
    }
  }
  __syncthreads();
  if (len > kRowWarp) s = rs.sum[slot];
  return s;
}
static_assert(kRowWarp >= (uint32_t)kFilterTPB, "a block's row has an arc for every thread");

// Bound on the size of level 2 from the class sums s of a source's out-neighbours.
__device__ __forceinline__ uint32_t level2_bound(const RunParams &p, const uint4 &s, uint32_t od, uint32_t g) {
  const int directed = p.g_directed ? p.g_directed[g] : p.directed;
  const u64 gamma = (u64)s.x + s.y + s.z + s.w - (directed ? 0u : od);
  const uint32_t *nc = p.n_cls + 4 * (size_t)g;
  const u64 by_class = (u64)min(s.x, nc[0]) + min(s.y, nc[1]) + min(s.z, nc[2]) + min(s.w, nc[3]);
  return (uint32_t)(gamma < by_class ? gamma : by_class);  // by_class <= n
}

__global__ void __launch_bounds__(kFilterTPB) k_filter_test(RunParams p, uint32_t count, uint32_t tile,
                                                            const uint32_t *__restrict__ off,
                                                            const uint32_t *__restrict__ col,
                                                            const uint4 *__restrict__ cls, const uint8_t *taken,
                                                            uint32_t ntaken, Ctl *c, uint8_t *keep,
                                                            uint32_t *tile_cnt, uint32_t *lvl2) {
  __shared__ RowScratch rs;
  const int lane = threadIdx.x & 31;
  u64 started = 0, visited = 0;
  for (u64 first = blockIdx.x; first < count; first += (u64)kFilterTPB * gridDim.x) {
    const u64 idx = first + (u64)threadIdx.x * gridDim.x;
    const bool valid = idx < count;
    bool kept = valid && !(taken && idx < ntaken && taken[idx]);
    bool test1 = false;
    uint32_t v = 0, g = 0, od = 0, a = 0, om = 0, b = 0, xr = 0;
    u64 xS = 0;
    if (kept) {
      v = p.order[idx];
      if (p.gid) g = p.gid[v];
      b = off[v];
      od = off[v + 1] - b;
      if (idx >= p.nocut_prefix) {
        const ulonglong2 x = p.x[g];
        xS = x.x;
        xr = (uint32_t)(x.y >> 32);
      }
    }
    if (xr != 0) {
      const bool stop = p.lb_key && (p.harmonic ? __dmul_rn(__longlong_as_double((long long)~p.lb_key[v]), kHMargin) <
                                                      __longlong_as_double((long long)xS)
                                                : nb_exceeds(p.lb_key[v], xS, xr));
      if (stop) {
        kept = false;
      } else {
        a = p.alpha[v];
        om = omega_of(p, v, g);
        test1 = !(p.harmonic ? harmonic_below(0.0, 0, 1, od, om, xS) : cut_exceeds(0, 0, 1, od, a, om, xS, xr));
        if (!test1) {
          kept = false;
          ++started;
          graph_count(p, g, 1, 1);
          graph_count(p, g, 2, 1);
        }
      }
    }
    // level 1 (uncut sources and those without a threshold keep the bound)
    const uint4 s = block_sum_rows(rs, col, cls, b, kept ? od : 0u);
    if (kept) {
      const uint32_t g2 = level2_bound(p, s, od, g);
      lvl2[v] = g2;
      if (test1 && level1_exceeds(p, od, a, om, g2, xS, xr)) {
        kept = false;
        ++started;
        visited += od;
        graph_count(p, g, 1, 1);
        graph_count(p, g, 2, 1);
        graph_count(p, g, 0, od);
      }
    }
    if (valid) {
      keep[idx] = kept;
      if (kept) atomicAdd(&tile_cnt[idx / tile], 1u);
    }
    __syncthreads();
  }
  for (int o = 16; o > 0; o >>= 1) {
    started += __shfl_down_sync(FULL, started, o);
    visited += __shfl_down_sync(FULL, visited, o);
  }
  if (lane == 0 && started) {
    atomicAdd(&c->bfs_started, started);
    atomicAdd(&c->bfs_cut, started);
  }
  if (lane == 0 && visited) atomicAdd(&c->edges_visited, visited);
}

// The opening's sources, one graph.  Which sources open is free (every one is
// searched or abandoned once), and the threshold they leave decides how many
// the filter keeps.  The order's head is not the best choice: in NBCut's order
// the sources whose omega is far above their reach come first (R-MAT 22: the
// first 128 sources left 3 000 and more for the main launch).  So the pool --
// the first kOpenPool positions -- is ranked by the bound after level 1 with
// level 2 by class and omega capped, which the threshold test itself uses.
// key: high word of the bound's FP64 bits (only an order: exactness is not
// needed), smallest first; sources never cut come first of all.
__global__ void __launch_bounds__(kFilterTPB) k_open_keys(RunParams p, uint32_t pool,
                                                          const uint32_t *__restrict__ off,
                                                          const uint32_t *__restrict__ col,
                                                          const uint4 *__restrict__ cls, uint32_t *key) {
  __shared__ RowScratch rs;
  for (u64 first = blockIdx.x; first < pool; first += (u64)kFilterTPB * gridDim.x) {
    const u64 idx = first + (u64)threadIdx.x * gridDim.x;
    const bool valid = idx < pool;
    uint32_t v = 0, b = 0, od = 0;
    if (valid) {
      v = p.order[idx];
      b = off[v];
      od = off[v + 1] - b;
    }
    const uint4 s = block_sum_rows(rs, col, cls, b, od);
    if (valid) {
      const u64 g2 = level2_bound(p, s, od, 0), n1 = 1ull + od;
      const uint32_t om = omega_of(p, v, 0);
      uint32_t k = 0;
      if (idx >= p.nocut_prefix) {
        if (p.harmonic) {
          const u64 w = om > n1 ? om - n1 : 0, near_ = g2 < w ? g2 : w;
          const double U = (double)od + 0.5 * (double)near_ + (double)(w - near_) / 3.0;
          k = ~(uint32_t)((u64)__double_as_longlong(U) >> 32);
        } else {
          u64 lo = p.alpha[v];
          lo = lo < n1 ? n1 : lo;
          const u64 hi = om < lo ? lo : om, kink = n1 + g2;
          double best = __longlong_as_double(0x7ff0000000000000ll);
          const u64 cand[3] = {lo, hi, kink > lo && kink < hi ? kink : hi};
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            const double r1 = (double)(cand[i] - 1);
            const double f = (double)cut_sum(od, 1, n1, g2, cand[i]) / (r1 * r1);  // r >= 2: od >= 1
            best = f < best ? f : best;
          }
          k = (uint32_t)((u64)__double_as_longlong(best) >> 32);
        }
      }
      key[idx] = k;
    }
    __syncthreads();
  }
}

// The nopen <= pool positions of smallest key (the first of equal ones), in
// the order's order: one block, the keys in registers, four passes of 8 bits
// for the nopen-th key and one scan.
constexpr int kPickTPB = 1024, kPickPer = kOpenPool / kPickTPB;
__global__ void __launch_bounds__(kPickTPB) k_open_pick(const uint32_t *order, const uint32_t *key, uint32_t pool,
                                                        uint32_t nopen, uint32_t *out, uint8_t *taken) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t s_prefix, s_need, s_warp[2][kPickTPB / 32 + 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t base = threadIdx.x * kPickPer;
  uint32_t k[kPickPer];
#pragma unroll
  for (int i = 0; i < kPickPer; ++i) k[i] = base + i < pool ? key[base + i] : 0xffffffffu;
  if (threadIdx.x == 0) {
    s_prefix = 0;
    s_need = nopen;
  }
  for (int shift = 24; shift >= 0; shift -= 8) {
    if (threadIdx.x < 256) hist[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t prefix = s_prefix, need = s_need, mask = shift == 24 ? 0u : 0xffffffffu << (shift + 8);
#pragma unroll
    for (int i = 0; i < kPickPer; ++i)
      if (base + i < pool && (k[i] & mask) == prefix) atomicAdd(&hist[(k[i] >> shift) & 255u], 1u);
    __syncthreads();
    if (wid == 0) {
      // lane l: bins 8l .. 8l + 7; the bin holding the need-th key
      uint32_t sum = 0;
      for (int j = 0; j < 8; ++j) sum += hist[8 * lane + j];
      uint32_t incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += t;
      }
      uint32_t before = incl - sum;
      if (before < need && incl >= need) {
        int j = 0;
        while (before + hist[8 * lane + j] < need) before += hist[8 * lane + j++];
        s_prefix = prefix | (uint32_t)(8 * lane + j) << shift;
        s_need = need - before;
      }
    }
    __syncthreads();
  }
  // all keys below the nopen-th, and the first s_need equal to it
  const uint32_t T = s_prefix, need = s_need;
  uint32_t below = 0, equal = 0;
#pragma unroll
  for (int i = 0; i < kPickPer; ++i) {
    below += base + i < pool && k[i] < T;
    equal += base + i < pool && k[i] == T;
  }
  uint32_t bi = below, ei = equal;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t tb = __shfl_up_sync(FULL, bi, o), te = __shfl_up_sync(FULL, ei, o);
    if (lane >= o) {
      bi += tb;
      ei += te;
    }
  }
  if (lane == 31) {
    s_warp[0][wid] = bi;
    s_warp[1][wid] = ei;
  }
  __syncthreads();
  uint32_t nb = bi - below, ne = ei - equal;  // below / equal ones before this thread's
  for (int w = 0; w < wid; ++w) {
    nb += s_warp[0][w];
    ne += s_warp[1][w];
  }
#pragma unroll
  for (int i = 0; i < kPickPer; ++i) {
    if (base + i >= pool) break;
    const bool eq = k[i] == T, take = k[i] < T || (eq && ne < need);
    taken[base + i] = take;
    if (take) out[nb + (ne < need ? ne : need)] = order[base + i];
    nb += k[i] < T;
    ne += eq;
  }
}

// The kept sources in order (a block per tile); per graph one past its last
// kept position; the main launch's control blocks continue the level stamps
// of the opening's and the shared cursor starts over.
__global__ void __launch_bounds__(kFilterTPB) k_filter_compact(RunParams p, uint32_t count, uint32_t tile,
                                                               const Ctl *open, uint32_t nopen, Ctl *ctl,
                                                               uint32_t nctl, const uint8_t *keep,
                                                               const uint32_t *tile_cnt, uint32_t *out,
                                                               uint32_t *g_end) {
  __shared__ uint32_t s_base;
  __shared__ uint32_t s_warp[kFilterTPB / 32];
  if (threadIdx.x == 0) s_base = 0;
  __syncthreads();
  uint32_t before = 0;
  for (uint32_t i = threadIdx.x; i < blockIdx.x; i += kFilterTPB) before += tile_cnt[i];
  before = __reduce_add_sync(FULL, before);
  if ((threadIdx.x & 31) == 0 && before) atomicAdd(&s_base, before);
  __syncthreads();
  uint32_t at = s_base;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const u64 base = (u64)blockIdx.x * tile;
  if (tile_cnt[blockIdx.x] != 0) {
    for (uint32_t o = 0; o < tile; o += kFilterTPB) {
      const u64 idx = base + o + threadIdx.x;
      const bool k = idx < count && keep[idx];
      const unsigned m = __ballot_sync(FULL, k);
      if (lane == 0) s_warp[wid] = __popc(m);
      __syncthreads();
      uint32_t pos = at;
      for (int w = 0; w < kFilterTPB / 32; ++w) {
        if (w < wid) pos += s_warp[w];
        at += s_warp[w];
      }
      if (k) {
        pos += __popc(m & ((1u << lane) - 1u));
        const uint32_t v = p.order[idx];
        out[pos] = v;
        if (g_end) atomicMax(&g_end[p.gid[v]], pos + 1);
      }
      __syncthreads();
    }
  }
  if (threadIdx.x == 0 && blockIdx.x == gridDim.x - 1) {
    p.sh->norder = at;
    p.sh->cursor = 0;
    p.sh->first_done = 0;
  }
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    unsigned lvl = 0;
    for (uint32_t i = 0; i < nopen; ++i) lvl = open[i].level_id > lvl ? open[i].level_id : lvl;
    for (uint32_t i = 0; i < nctl; ++i) ctl[i].level_id = lvl + 1;
  }
}

// ------------------------------------------------------------------ host side

int run_init(tkc_ctx *ctx, uint32_t nctl, uint32_t n, uint32_t ng, bool reset_lists) {
  Workspace &w = ctx->ws;
  const uint32_t work = reset_lists ? (n > ng ? n : ng) : 1024;
  const uint32_t blocks = work / 1024 + 1 < (uint32_t)ctx->num_sms * 8 ? work / 1024 + 1 : (uint32_t)ctx->num_sms * 8;
  TKC_LAUNCH(k_run_init<<<blocks, 256, 0, ctx->stream>>>(w.ctl, nctl, w.level_base, w.sh, reset_lists ? ng : 0u,
                                                         w.g_ntop, w.g_stop, w.g_lock, w.g_ctr, w.x, w.res_r, n));
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

// Blocks for `count` positions: several per SM before a block takes more than
// one position per thread, since a few positions may be long rows.
static uint32_t filter_blocks(tkc_ctx *ctx, uint32_t count) {
  const uint32_t nb = (count + 7) / 8, most = (uint32_t)ctx->num_sms * 8;
  return nb < 1 ? 1 : nb < most ? nb : most;
}

int run_pick_opening(tkc_ctx *ctx, const RunParams &p, const tkc_graph *g, uint32_t count, uint32_t nopen) {
  Workspace &w = ctx->ws;
  cudaStream_t st = ctx->stream;
  const uint32_t pool = count < kOpenPool ? count : kOpenPool;
  TKC_LAUNCH(k_open_keys<<<filter_blocks(ctx, pool), kFilterTPB, 0, st>>>(p, pool, g->off, g->col, g->cls, w.o_key));
  TKC_LAUNCH(k_open_pick<<<1, kPickTPB, 0, st>>>(p.order, w.o_key, pool, nopen, w.o_order, w.o_taken));
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

int run_filter(tkc_ctx *ctx, const RunParams &p, const tkc_graph *g, uint32_t open_teams, uint32_t main_teams,
               uint32_t count, bool picked) {
  Workspace &w = ctx->ws;
  cudaStream_t st = ctx->stream;
  // at most kFilterTiles tiles, so that a compacting block sums the counts before it itself
  uint32_t tile = (count + kFilterTiles - 1) / kFilterTiles;
  tile = (tile + kFilterTPB - 1) / kFilterTPB * kFilterTPB;
  if (tile == 0) tile = kFilterTPB;
  const uint32_t ntiles = count ? (count + tile - 1) / tile : 1;
  Ctl *main_ctl = w.ctl + open_teams;
  TKC_TRY(cudaMemsetAsync(w.f_count, 0, ntiles * sizeof(uint32_t), st));
  if (p.gid) TKC_TRY(cudaMemsetAsync(w.f_end, 0, (size_t)p.ng * sizeof(uint32_t), st));
  TKC_LAUNCH(k_filter_test<<<filter_blocks(ctx, count), kFilterTPB, 0, st>>>(
      p, count, tile, g->off, g->col, g->cls, picked ? w.o_taken : nullptr, kOpenPool < count ? kOpenPool : count,
      main_ctl, w.f_keep, w.f_count, w.lvl2));
  TKC_LAUNCH(k_filter_compact<<<ntiles, kFilterTPB, 0, st>>>(p, count, tile, w.ctl, open_teams, main_ctl, main_teams,
                                                             w.f_keep, w.f_count, w.f_order,
                                                             p.gid ? w.f_end : nullptr));
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

// The larger blocks pay off on batched searches of large graphs (NBCut on
// R-MAT 22 1.36 -> 1.07 ms of kernel time); one-source searches and graphs below
// 2^20 vertices run 512 threads per block.  Near the line it depends on the graph
// (NBCut, 512 and 1024 threads: R-MAT 16 0.25 and 0.28 ms, R-MAT 18 0.28 and 0.31,
// R-MAT 19 0.37 and 0.39, Barabasi-Albert 131 072 0.27 and 0.31, 10^6 1.23 and 1.02).
static bool wide_blocks(const RunParams &p) {
  if (p.large_blocks) return p.large_blocks == 1;
  return p.B > 1 && p.n >= (1u << 20);
}

template <int W, int TPB>
static int occupancy_of(int *blocks_per_sm) {
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, bfscut_kernel<W, TPB>, TPB, 0);
  return e == cudaSuccess ? TKC_OK : TKC_ECUDA;
}

// Co-resident blocks of the W-word kernel, the smaller of its two block sizes'
// (either may be launched with this count).
template <int W>
static int occupancy_both(int *blocks_per_sm) {
  int a = 0, b = 0;
  int rc = occupancy_of<W, kThreads<W>>(&a);
  if (rc == TKC_OK) rc = occupancy_of<W, kMinThreads>(&b);
  if (rc != TKC_OK) return rc;
  *blocks_per_sm = a < b ? a : b;
  return TKC_OK;
}

int max_coresident_blocks(tkc_ctx *ctx, int words) {
  int per_sm = 0;
  int rc = TKC_OK;
  switch (words) {
    case 1: rc = occupancy_both<1>(&per_sm); break;
    case 2: rc = occupancy_both<2>(&per_sm); break;
    case 4: rc = occupancy_both<4>(&per_sm); break;
    case 8: rc = occupancy_both<8>(&per_sm); break;
    default: return 0;
  }
  if (rc != TKC_OK) return 0;
  return per_sm * ctx->num_sms;
}

template <int W, int TPB>
static cudaError_t launch_tpb(const RunParams &p, int blocks, cudaStream_t st) {
  void *args[] = {(void *)&p};
  note_launches(1);
  return cudaLaunchCooperativeKernel((const void *)bfscut_kernel<W, TPB>, dim3(blocks), dim3(TPB), args, 0, st);
}

template <int W>
static cudaError_t launch(const RunParams &p, int blocks, cudaStream_t st) {
  if (kThreads<W> != kMinThreads && wide_blocks(p)) return launch_tpb<W, kThreads<W>>(p, blocks, st);
  return launch_tpb<W, kMinThreads>(p, blocks, st);
}

int run_bfscut(tkc_ctx *ctx, const RunParams &p, int words, int blocks) {
  cudaError_t e;
  switch (words) {
    case 1: e = launch<1>(p, blocks, ctx->stream); break;
    case 2: e = launch<2>(p, blocks, ctx->stream); break;
    case 4: e = launch<4>(p, blocks, ctx->stream); break;
    case 8: e = launch<8>(p, blocks, ctx->stream); break;
    default: return TKC_EINVAL;
  }
  TKC_TRY(e);
  return TKC_OK;
}

}  // namespace tkc
