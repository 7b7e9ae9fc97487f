// Reach bounds alpha(v) <= r(v) <= omega(v) for directed graphs on the GPU
// (Section 8.4, Algorithm 6).
//
//  1. Strongly connected components:
//     trim   vertices with no active in-arc or no active out-arc are their own
//            SCC (repeated until nothing changes);
//     FW-BW  the SCC of a pivot (largest in-degree x out-degree among the rest)
//            is the intersection of its forward and backward reach;
//     colour the rest: every vertex takes the largest id that reaches it
//            (max propagation along arcs); a vertex whose colour is its own id
//            is a root, and its SCC is the set of same-colour vertices that
//            reach it (backward propagation); repeat on what is left.
//     Each SCC is named by one of its vertices.
//  2. The biggest SCC (ties: the one holding the smallest vertex id) gets its
//     exact reach from one BFS; a backward BFS marks the SCCs that reach it (the
//     pivot's, when that SCC is its own).
//  3. Condensation arcs (SCC pairs) are sorted and deduplicated, so the DAG's
//     arc set has no repeats, and Algorithm 6's recurrences are evaluated
//     sinks-first by peeling: an SCC is ready once all its successors are.
//       alpha(X) = w(X) + max alpha(Y), omega(X) = w(X) + sum omega(Y), or
//       omega(X) = w(X) + omega(C~) + sum of omega(Y) over successors Y not
//       reachable from C~ when X reaches C~;  omega clamped to n.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "tkc_arcs.cuh"
#include "tkc_grid.cuh"
#include "tkc_internal.cuh"

namespace tkc {

typedef uint32_t u32;
typedef unsigned long long u64;
static constexpr unsigned FULL = 0xffffffffu;
static constexpr u32 INF = 0xffffffffu;

// scan / sort helpers of tkc_prep.cu
int scan_exclusive_u32(const u32 *in, u32 *out, u64 len, u32 *tmp, cudaStream_t st);
int radix_sort_u32_pairs(u32 *key, u32 *val, u32 n, int bits, cudaStream_t st);

namespace {

unsigned grid_of(u64 work, unsigned tpb = 256, unsigned cap = 152 * 16) {
  u64 b = (work + tpb - 1) / tpb;
  return (unsigned)std::max<u64>(1, std::min<u64>(b, cap));
}

// ---------------------------------------------------------------- trimming

// (comp: every vertex its own until its SCC is found, so that later passes may
// run before the host knows that all are)
__global__ void k_trim_init(const u32 *off, const u32 *ioff, u32 n, u32 *outd, u32 *ind, uint8_t *active, u32 *comp) {
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    outd[v] = off[v + 1] - off[v];
    ind[v] = ioff[v + 1] - ioff[v];
    active[v] = 1;
    comp[v] = v;
  }
}

// Removes vertices without an active in-arc or out-arc (each is its own SCC)
// and lowers the counters of their neighbours, round after round until none is
// left (one cooperative launch).  One warp per removed vertex walks its arcs.
// changed: two zero words, used in turn.
constexpr int kLoopTPB = 256;  // threads per block of the launches that loop over rounds

__global__ void __launch_bounds__(kLoopTPB) k_trim(const u32 *off, const u32 *col, const u32 *ioff, const u32 *icol,
                                                   u32 n, u32 *outd, u32 *ind, uint8_t *active, u32 *comp,
                                                   u32 *changed, GridBar *bar, u64 timeout) {
  const int lane = threadIdx.x & 31;
  for (u32 round = 0;; ++round) {
    u32 *ch = changed + (round & 1);
    for (u32 base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; base < n; base += gridDim.x * blockDim.x) {
      u32 v = base + lane;
      bool rm = v < n && active[v] && (outd[v] == 0 || ind[v] == 0);
      if (rm) {
        active[v] = 0;
        comp[v] = v;
      }
      u32 mask = __ballot_sync(FULL, rm);
      if (mask && lane == 0) *ch = 1;
      while (mask) {
        int src = __ffs(mask) - 1;
        mask &= mask - 1;
        u32 x = base + src;
        for (u32 i = off[x] + lane; i < off[x + 1]; i += 32) atomicSub(&ind[col[i]], 1u);
        for (u32 i = ioff[x] + lane; i < ioff[x + 1]; i += 32) atomicSub(&outd[icol[i]], 1u);
      }
    }
    // the other word was read by every block before it arrived here
    if (!grid_sync(bar, timeout, [&] { changed[(round & 1) ^ 1] = 0; })) return;
    if (*(volatile u32 *)ch == 0) return;
  }
}

// ---------------------------------------------------------------- reach BFS, one cooperative launch

// Control block of the reach BFS: grid barrier, then the frontier queues'
// packed counters (count << 38 | out-arcs).
struct BfsCtl {
  GridBar bar;
  unsigned level;
  unsigned long long q[2];
};

constexpr int kBfsThreads = 512;
constexpr int kQShift = 38;
constexpr u64 kQArcs = (1ull << kQShift) - 1;

// Appends the lanes with `pred` to a queue whose counter packs count << 38 |
// out-arcs (one atomic per warp); qo[pos] = the arcs of the entries before.
__device__ __forceinline__ void q_append(bool pred, u32 v, u32 od, unsigned long long *packed, u32 *q, u64 *qo,
                                         int lane) {
  const unsigned m = __ballot_sync(FULL, pred);
  if (!m) return;
  u32 a = pred ? od : 0u;
  u32 incl = a;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u32 t = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += t;
  }
  const u32 tot = __shfl_sync(FULL, incl, 31);
  const int leader = __ffs(m) - 1;
  unsigned long long base = 0;
  if (lane == leader) base = atomicAdd(packed, ((unsigned long long)__popc(m) << kQShift) | tot);
  base = __shfl_sync(FULL, base, leader);
  if (pred) {
    const u32 pos = (u32)(base >> kQShift) + __popc(m & ((1u << lane) - 1u));
    q[pos] = v;
    qo[pos] = (base & kQArcs) + (incl - a);
  }
}

// Reachability from src along the arcs (off, col); (roff, rcol) are the same
// arcs reversed.  mark[v] = the step at which v was reached, INF if never
// (src: 0).  A step expands the frontier queue top-down (its arcs split evenly
// over the warps, so a hub's row is shared by many; a vertex is claimed by
// compare-and-swap) or, when the frontier's arcs exceed 1/8 of all arcs,
// bottom-up: every unreached vertex looks for any reached in-neighbour and
// stops at the first (only reachability is asked for).
__global__ void __launch_bounds__(kBfsThreads) k_bfs_reach(const u32 *off, const u32 *col, const u32 *roff,
                                                          const u32 *rcol, u32 n, u64 arcs, u32 *mark, u32 *q0,
                                                          u32 *q1, u64 *qo0, u64 *qo1, BfsCtl *c, u64 timeout) {
  const int lane = threadIdx.x & 31;
  const u32 gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int cur = 0;; cur ^= 1) {
    const unsigned long long qp = ((volatile BfsCtl *)c)->q[cur];
    const u32 qn = (u32)(qp >> kQShift);
    const u64 qa = qp & kQArcs;
    if (qn == 0) break;
    const u32 step = ((volatile BfsCtl *)c)->level + 1;
    const u32 *Q = cur ? q1 : q0;
    const u64 *QO = cur ? qo1 : qo0;
    u32 *NQ = cur ? q0 : q1;
    u64 *NQO = cur ? qo0 : qo1;
    unsigned long long *npk = &c->q[cur ^ 1];
    if (qa * 8 <= arcs) {
      // about two arc ranges per warp, whole warp steps of 32 arcs
      u64 ch = (qa + 2ull * nwarps - 1) / (2ull * nwarps);
      ch = (ch + 31) / 32 * 32;
      for (u64 a0 = (u64)gwarp * ch; a0 < qa; a0 += (u64)nwarps * ch) {
        const u64 a1 = a0 + ch < qa ? a0 + ch : qa;
        u32 lo = 0, hi = qn;  // last entry with QO <= a0
        while (hi - lo > 1) {
          const u32 mid = (lo + hi) >> 1;
          if (QO[mid] <= a0) lo = mid;
          else hi = mid;
        }
        u32 ent = lo;
        for (u64 s0 = a0; s0 < a1; s0 += 32) {
          const u64 a = s0 + lane;
          u32 w = 0;
          bool got = false;
          u32 e = ent;
          if (a < a1) {
            while (e + 1 < qn && QO[e + 1] <= a) ++e;
            w = col[off[Q[e]] + (u32)(a - QO[e])];
            got = mark[w] == INF && atomicCAS(&mark[w], INF, step) == INF;
          }
          q_append(got, w, got ? off[w + 1] - off[w] : 0u, npk, NQ, NQO, lane);
          ent = __reduce_max_sync(FULL, e);
        }
      }
    } else {
      for (u32 base = gwarp * 32; base < n; base += nwarps * 32) {
        const u32 v = base + lane;
        bool got = false;
        u32 b = 0, e = 0;
        if (v < n && mark[v] == INF) {
          b = roff[v];
          e = roff[v + 1];
        }
        const bool light = e - b <= 32;
        // short in-rows: the lane alone, four in-neighbours per step
        if (light)
          for (u32 k = b; k < e && !got; k += 4) {
            u32 mu[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) mu[j] = k + j < e ? mark[rcol[k + j]] : INF;
#pragma unroll
            for (int j = 0; j < 4; ++j) got |= mu[j] < step;
          }
        // long in-rows: the whole warp, 32 in-neighbours per step, until one is reached
        for (unsigned hv = __ballot_sync(FULL, !light); hv; hv &= hv - 1) {
          const int src = __ffs(hv) - 1;
          const u32 hb = __shfl_sync(FULL, b, src), he = __shfl_sync(FULL, e, src);
          bool hit = false;
          for (u32 k0 = hb; k0 < he && !hit; k0 += 32) {
            const u32 k = k0 + lane;
            hit = __any_sync(FULL, k < he && mark[rcol[k]] < step);
          }
          if (lane == src) got = hit;
        }
        if (got) mark[v] = step;
        q_append(got, v, got ? off[v + 1] - off[v] : 0u, npk, NQ, NQO, lane);
      }
    }
    const bool ok = grid_sync(&c->bar, timeout, [&] {
      c->q[cur] = 0;
      c->level = step;
    });
    if (!ok) return;
  }
}

// The vertex a packed maximum names (k_pivot, k_biggest), INF for none.
__device__ __forceinline__ u32 named_vertex(u64 best) { return best ? 0xffffffffu - (u32)(best & 0xffffffffu) : INF; }

// From vertex src, or with src = INF from the pivot named by *best (none: the
// search ends at once).
__global__ void k_bfs_start(const u32 *off, u32 *mark, u32 *q0, u64 *qo0, BfsCtl *c, u32 src, const u64 *best) {
  if (src == INF) src = named_vertex(*best);
  if (src == INF) return;
  mark[src] = 0;
  q0[0] = src;
  qo0[0] = 0;
  c->q[0] = (1ull << kQShift) | (unsigned long long)(off[src + 1] - off[src]);
}

// Several sources at once (*nsrc distinct vertices): all at step 0.  One block.
__global__ void k_bfs_start_many(const u32 *off, const u32 *src, const u32 *nsrc, u32 *mark, u32 *q0, u64 *qo0,
                                 BfsCtl *c) {
  __shared__ u64 s_warp[32], s_run;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const u32 n = *nsrc;
  if (threadIdx.x == 0) s_run = 0;
  __syncthreads();
  for (u32 base = 0; base < n; base += blockDim.x) {
    const u32 i = base + threadIdx.x;
    u32 v = 0;
    u64 d = 0;
    if (i < n) {
      v = src[i];
      d = off[v + 1] - off[v];
    }
    u64 incl = d;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 t = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    u64 before = s_run;
    for (int w = 0; w < wid; ++w) before += s_warp[w];
    if (i < n) {
      mark[v] = 0;
      q0[i] = v;
      qo0[i] = before + incl - d;
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int w = 0; w < nw; ++w) s_run += s_warp[w];
    __syncthreads();
  }
  if (threadIdx.x == 0) c->q[0] = ((unsigned long long)n << kQShift) | s_run;
}

// Reachability along (off, col) into mark (see k_bfs_reach) from vertex src;
// from the pivot that *best names (src = INF); or from the *nsrc vertices of
// srcs.  One cooperative launch, no host wait: *c (zero) holds its error word
// for the caller.
int bfs_reach(tkc_ctx *ctx, const u32 *off, const u32 *col, const u32 *roff, const u32 *rcol, u32 n, u64 arcs,
              u32 *mark, u32 src, const u64 *best, const u32 *srcs, const u32 *nsrc, BfsCtl *c, cudaStream_t st) {
  u32 *q = nullptr;
  u64 *qo = nullptr;
  TKC_TRY(dev_malloc(&q, (size_t)2 * n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&qo, (size_t)2 * n * sizeof(u64), st));
  TKC_TRY(cudaMemsetAsync(mark, 0xff, (size_t)n * sizeof(u32), st));
  u32 *q0 = q, *q1 = q + n;
  u64 *qo0 = qo, *qo1 = qo + n;
  if (srcs) {
    TKC_LAUNCH(k_bfs_start_many<<<1, 1024, 0, st>>>(off, srcs, nsrc, mark, q0, qo0, c));
  } else {
    TKC_LAUNCH(k_bfs_start<<<1, 1, 0, st>>>(off, mark, q0, qo0, c, src, best));
  }
  u64 timeout = grid_timeout(ctx);
  void *args[] = {(void *)&off,  (void *)&col, (void *)&roff, (void *)&rcol, (void *)&n,
                  (void *)&arcs, (void *)&mark, (void *)&q0,  (void *)&q1,   (void *)&qo0,
                  (void *)&qo1,  (void *)&c,    (void *)&timeout};
  const int blocks = grid_blocks(ctx, k_bfs_reach, kBfsThreads, n);
  if (blocks <= 0) return TKC_ECUDA;
  note_launches(1);
  TKC_TRY(cudaLaunchCooperativeKernel((const void *)k_bfs_reach, dim3(blocks), dim3(kBfsThreads), args, 0, st));
  TKC_TRY(cudaFreeAsync(q, st));
  TKC_TRY(cudaFreeAsync(qo, st));
  return TKC_OK;
}

// ---------------------------------------------------------------- pivot and FW-BW

__global__ void k_pivot(const u32 *outd, const u32 *ind, const uint8_t *active, u32 n, u64 *best) {
  u64 b = 0;
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    if (active[v]) {
      u64 score = (u64)outd[v] * (u64)ind[v];
      score = score > 0xffffffffull ? 0xffffffffull : score;
      u64 key = (score << 32) | (u64)(0xffffffffu - v);  // larger score, then smaller id
      b = key > b ? key : b;
    }
  for (int o = 16; o; o >>= 1) {
    u64 t = __shfl_down_sync(FULL, b, o);
    b = t > b ? t : b;
  }
  if ((threadIdx.x & 31) == 0 && b) atomicMax(best, b);
}

__global__ void k_fwbw_mark(const u32 *fw, const u32 *bw, u32 n, uint8_t *active, u32 *comp, const u64 *best) {
  const u32 pivot = named_vertex(*best);  // none: nothing is reached both ways
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    if (active[v] && fw[v] != INF && bw[v] != INF) {
      comp[v] = pivot;
      active[v] = 0;
    }
}

// Several graphs as one union (gid: graph of each vertex, graphs in
// contiguous vertex ranges): the pivot of every graph, best[g] packed like
// k_pivot's.  Lanes of one graph first take their warp's maximum, so each
// graph sees about one atomic per warp.
__global__ void k_pivot_many(const u32 *outd, const u32 *ind, const uint8_t *active, const u32 *gid, u32 n,
                             u64 *best) {
  for (u32 base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; base < n; base += gridDim.x * blockDim.x) {
    const u32 v = base + (threadIdx.x & 31);
    u32 score = 0, g = 0xffffffffu;
    if (v < n) {
      g = gid[v];
      if (active[v]) {
        const u64 s = (u64)outd[v] * (u64)ind[v];
        score = s > 0xffffffffull ? 0xffffffffu : (u32)s;
      }
    }
    const unsigned peers = __match_any_sync(FULL, g);
    const u32 hi = __reduce_max_sync(peers, score);
    const u32 lo = __reduce_max_sync(peers, score == hi && v < n ? 0xffffffffu - v : 0u);
    if (v < n && hi > 0 && (int)(threadIdx.x & 31) == __ffs(peers) - 1)
      atomicMax(&best[g], ((u64)hi << 32) | (u64)lo);
  }
}

// The graphs' pivots as a list (graphs without one are skipped); count in *cnt.
__global__ void k_pivot_list(const u64 *best, u32 ng, u32 *piv, u32 *list, u32 *cnt) {
  for (u32 g = blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += gridDim.x * blockDim.x) {
    const u64 b = best[g];
    piv[g] = b ? 0xffffffffu - (u32)(b & 0xffffffffu) : INF;
    if (b) list[atomicAdd(cnt, 1u)] = piv[g];
  }
}

// fw, bw: reach from / to all pivots at once.  The graphs are disjoint, so a
// vertex reached either way is reached by its own graph's pivot only, and it
// lies in that pivot's SCC when reached both ways.
__global__ void k_fwbw_mark_many(const u32 *fw, const u32 *bw, const u32 *gid, const u32 *piv, u32 n,
                                 uint8_t *active, u32 *comp) {
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    if (active[v] && fw[v] != INF && bw[v] != INF) {
      comp[v] = piv[gid[v]];
      active[v] = 0;
    }
}

// ---------------------------------------------------------------- colouring

// One colouring round over the active vertices, one cooperative launch: the
// colours (the largest id that reaches a vertex) propagate along arcs until
// nothing changes, then `found` spreads backwards from the roots among
// vertices of one colour, and what was found is assigned.
// changed: two zero words, used in turn.
__global__ void __launch_bounds__(kLoopTPB) k_color_round(const u32 *off, const u32 *col, const u32 *ioff,
                                                          const u32 *icol, u32 n, uint8_t *active, u32 *color,
                                                          u32 *found, u32 *comp, u32 *changed, GridBar *bar,
                                                          u64 timeout) {
  const int lane = threadIdx.x & 31;
  const u32 first = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  for (u32 v = first; v < n; v += step) {
    color[v] = active[v] ? v : INF;
    found[v] = 0;
  }
  if (!grid_sync(bar, timeout, [] {})) return;
  u32 round = 0;
  // colour[w] = max(colour[w], colour[v]) over active arcs v -> w
  for (;; ++round) {
    u32 *chg = changed + (round & 1);
    for (u32 base = first & ~31u; base < n; base += step) {
      const u32 v = base + lane;
      u32 mask = __ballot_sync(FULL, v < n && active[v]);
      u32 ch = 0;
      while (mask) {
        const int src = __ffs(mask) - 1;
        mask &= mask - 1;
        const u32 x = base + src;
        const u32 cx = color[x];
        for (u32 i = off[x] + lane; i < off[x + 1]; i += 32) {
          const u32 w = col[i];
          if (active[w] && color[w] < cx) {
            atomicMax(&color[w], cx);
            ch = 1;
          }
        }
      }
      if (__any_sync(FULL, ch) && lane == 0) *chg = 1;
    }
    if (!grid_sync(bar, timeout, [&] { changed[(round & 1) ^ 1] = 0; })) return;
    if (*(volatile u32 *)chg == 0) break;
  }
  ++round;
  // the roots
  for (u32 v = first; v < n; v += step)
    if (active[v] && color[v] == v) found[v] = 1;
  if (!grid_sync(bar, timeout, [] {})) return;
  // found spreads along in-arcs among vertices of the same colour
  for (;; ++round) {
    u32 *chg = changed + (round & 1);
    for (u32 base = first & ~31u; base < n; base += step) {
      const u32 v = base + lane;
      u32 mask = __ballot_sync(FULL, v < n && active[v] && found[v]);
      u32 ch = 0;
      while (mask) {
        const int src = __ffs(mask) - 1;
        mask &= mask - 1;
        const u32 x = base + src;
        const u32 cx = color[x];
        for (u32 i = ioff[x] + lane; i < ioff[x + 1]; i += 32) {
          const u32 u = icol[i];
          if (active[u] && color[u] == cx && !found[u]) {
            found[u] = 1;
            ch = 1;
          }
        }
      }
      if (__any_sync(FULL, ch) && lane == 0) *chg = 1;
    }
    if (!grid_sync(bar, timeout, [&] { changed[(round & 1) ^ 1] = 0; })) return;
    if (*(volatile u32 *)chg == 0) break;
  }
  for (u32 v = first; v < n; v += step)
    if (active[v] && found[v]) {
      comp[v] = color[v];
      active[v] = 0;
    }
}

// ---------------------------------------------------------------- component statistics

// Size and smallest vertex of every SCC.  Lanes holding the same SCC add up
// in the warp first: one big SCC would otherwise take one atomic per vertex on
// a single address.
__global__ void k_comp_stats(const u32 *comp, u32 n, u32 *wgt, u32 *minid) {
  const int lane = threadIdx.x & 31;
  for (u32 base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; base < n; base += gridDim.x * blockDim.x) {
    const u32 v = base + lane;
    const bool valid = v < n;
    const u32 c = valid ? comp[v] : INF;
    const unsigned grp = __match_any_sync(FULL, c);
    if (valid && lane == __ffs(grp) - 1) {
      atomicAdd(&wgt[c], (u32)__popc(grp));
      atomicMin(&minid[c], v);  // the group's first lane holds its smallest id
    }
  }
}

__global__ void k_biggest(const u32 *wgt, const u32 *minid, u32 n, u64 *best) {
  u64 b = 0;
  for (u32 c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x)
    if (wgt[c]) {
      u64 key = ((u64)wgt[c] << 32) | (u64)(0xffffffffu - minid[c]);
      b = key > b ? key : b;
    }
  for (int o = 16; o; o >>= 1) {
    u64 t = __shfl_down_sync(FULL, b, o);
    b = t > b ? t : b;
  }
  if ((threadIdx.x & 31) == 0 && b) atomicMax(best, b);
}

// The biggest SCC: that of the vertex *best names; the graph it lies in (gid
// may be null: 0) and that graph's pivot.
__global__ void k_big(const u32 *comp, const u64 *best, const u32 *gid, const u32 *piv, const u64 *best0, u32 *big,
                      u32 *big_graph, u32 *big_pivot) {
  const u32 v = named_vertex(*best);
  *big = comp[v];
  *big_graph = gid ? gid[v] : 0;
  *big_pivot = gid ? piv[gid[v]] : named_vertex(*best0);
}

// Vertices reached, of graph *only (gid may be null: all).
__global__ void k_count_reached(const u32 *dist, u32 n, const u32 *gid, const u32 *only, u32 *cnt) {
  u32 c = 0;
  const u32 g = gid ? *only : 0;
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    c += dist[v] != INF && (!gid || gid[v] == g);
  c = __reduce_add_sync(FULL, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(cnt, c);
}

// Forgets what the searches reached in the other graphs.
__global__ void k_keep_graph(const u32 *gid, u32 g, u32 n, u32 *fw, u32 *bw) {
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    if (gid[v] != g) fw[v] = bw[v] = INF;
}

// ---------------------------------------------------------------- condensation

// Arcs between different SCCs.  Arcs are dealt to warps in fixed chunks with
// their sources found by search (tkc_arcs.cuh), so a hub's out-row is spread
// over many warps.  The count pass writes each block's count; after an
// exclusive scan of those, the emit pass (same grid, so the same arcs per
// block) writes each block's arcs from its offset on, placed by a
// shared-memory cursor: no global atomics.  (The pairs are sorted afterwards,
// so their order within a block does not matter.)
template <bool emit>
__global__ void k_cross(const u32 *off, const u32 *col, const u32 *comp, u32 n, u64 arcs, u32 *blk, u32 *cu,
                        u32 *cv) {
  __shared__ u32 s_cnt;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) s_cnt = 0;
  __syncthreads();
  const u32 base = emit ? blk[blockIdx.x] : 0u;
  u32 c = 0;
  grid_walk_arcs(off, n, arcs, [&](u32 u, u64 i, bool valid, u32) {
    const u32 a = valid ? comp[u] : 0u;
    const u32 t = valid ? comp[col[i]] : 0u;
    const bool cross = valid && t != a;
    if (!emit) {
      c += cross;
      return;
    }
    const unsigned m = __ballot_sync(FULL, cross);
    if (!m) return;
    u32 pos = 0;
    if (lane == 0) pos = atomicAdd(&s_cnt, (u32)__popc(m));
    pos = __shfl_sync(FULL, pos, 0);
    if (cross) {
      const u32 k = base + pos + __popc(m & ((1u << lane) - 1u));
      cu[k] = a;
      cv[k] = t;
    }
  });
  if (!emit) {
    c = __reduce_add_sync(FULL, c);
    if (lane == 0 && c) atomicAdd(&s_cnt, c);
    __syncthreads();
    if (threadIdx.x == 0) blk[blockIdx.x] = s_cnt;
  }
}

// flag[i] = 1 for the first of each run of equal (cu, cv) pairs (sorted input)
__global__ void k_unique_flags(const u32 *cu, const u32 *cv, u32 m, u32 *flag) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x)
    flag[i] = (i == 0 || cu[i] != cu[i - 1] || cv[i] != cv[i - 1]) ? 1u : 0u;
  if (blockIdx.x == 0 && threadIdx.x == 0) flag[m] = 0;
}

// Keeps the first of each run of equal pairs and counts successors and
// predecessors per SCC; lanes holding the same SCC add up in the warp first
// (one SCC may be the target of a large share of all pairs).
__global__ void k_unique_compact(const u32 *cu, const u32 *cv, const u32 *pos, u32 m, u32 *ou, u32 *ov,
                                 u32 *succ_cnt, u32 *pred_cnt) {
  const int lane = threadIdx.x & 31;
  for (u32 base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; base < m; base += gridDim.x * blockDim.x) {
    const u32 i = base + lane;
    const bool keep = i < m && pos[i + 1] != pos[i];
    const u32 a = keep ? cu[i] : INF, t = keep ? cv[i] : INF;
    if (keep) {
      ou[pos[i]] = a;
      ov[pos[i]] = t;
    }
    const unsigned ga = __match_any_sync(FULL, a), gt = __match_any_sync(FULL, t);
    if (keep && lane == __ffs(ga) - 1) atomicAdd(&succ_cnt[a], (u32)__popc(ga));
    if (keep && lane == __ffs(gt) - 1) atomicAdd(&pred_cnt[t], (u32)__popc(gt));
  }
}

// Predecessor lists: each pair's source into its target's list (positions
// claimed once per warp and target SCC).
__global__ void k_pred_scatter(const u32 *ou, const u32 *ov, const u32 *pairs, const u32 *poff, u32 *pcur, u32 *pred) {
  const u32 m = *pairs;
  const int lane = threadIdx.x & 31;
  for (u32 base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; base < m; base += gridDim.x * blockDim.x) {
    const u32 i = base + lane;
    const u32 c = i < m ? ov[i] : INF;
    const unsigned grp = __match_any_sync(FULL, c);
    const int leader = __ffs(grp) - 1;
    u32 at = 0;
    if (c != INF && lane == leader) at = atomicAdd(&pcur[c], (u32)__popc(grp));
    at = __shfl_sync(FULL, at, leader);
    if (c != INF) pred[poff[c] + at + __popc(grp & ((1u << lane) - 1u))] = ou[i];
  }
}

// ---------------------------------------------------------------- Algorithm 6, sinks first

__global__ void k_sinks(const u32 *wgt, const u32 *soff, u32 n, u32 *rem, u32 *list, u32 *count) {
  for (u32 c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
    if (!wgt[c]) continue;
    u32 d = soff[c + 1] - soff[c];
    rem[c] = d;
    if (d == 0) list[atomicAdd(count, 1u)] = c;
  }
}

// Evaluates alpha/omega of the ready SCCs (all successors done).  A lane
// reduces over the successors of its own SCC when there are at most 32; the
// whole warp over longer successor lists.
__device__ __forceinline__ void dp_eval(const u32 *list, u32 cnt, const u32 *soff, const u32 *succ, const u32 *wgt,
                          const u32 *dist_from_big, const u32 *dist_to_big, u32 big, u64 reach_big, u32 n, u64 *A,
                          u64 *O) {
  const int lane = threadIdx.x & 31;
  for (u32 base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; base < cnt; base += gridDim.x * blockDim.x) {
    const u32 i = base + lane;
    const u32 c = i < cnt ? list[i] : INF;
    u32 b = 0, e = 0;
    if (c != INF && c != big) {
      b = soff[c];
      e = soff[c + 1];
    }
    const bool light = e - b <= 32;
    u64 amax = 0, osum = 0, onot = 0;
    if (light)
      for (u32 k = b; k < e; ++k) {
        const u32 y = succ[k];
        amax = A[y] > amax ? A[y] : amax;
        osum += O[y];
        if (dist_from_big[y] == INF) onot += O[y];
      }
    for (unsigned hv = __ballot_sync(FULL, !light); hv; hv &= hv - 1) {
      const int src = __ffs(hv) - 1;
      const u32 hb = __shfl_sync(FULL, b, src), he = __shfl_sync(FULL, e, src);
      u64 wa = 0, wo = 0, wn = 0;
      for (u32 k = hb + lane; k < he; k += 32) {
        const u32 y = succ[k];
        wa = A[y] > wa ? A[y] : wa;
        wo += O[y];
        if (dist_from_big[y] == INF) wn += O[y];
      }
      for (int o = 16; o; o >>= 1) {
        const u64 t = __shfl_xor_sync(FULL, wa, o);
        wa = t > wa ? t : wa;
        wo += __shfl_xor_sync(FULL, wo, o);
        wn += __shfl_xor_sync(FULL, wn, o);
      }
      if (lane == src) {
        amax = wa;
        osum = wo;
        onot = wn;
      }
    }
    if (c == INF) continue;
    u64 a, o;
    if (c == big) {
      a = o = reach_big;
    } else {
      if (dist_to_big[c] != INF) osum = onot + O[big];
      a = amax + wgt[c];
      o = osum + wgt[c];
      if (o > n) o = n;
    }
    A[c] = a;
    O[c] = o;
  }
}

// Predecessor lists longer than this are released by the whole grid.
constexpr u32 kDpHuge = 4096;

// Appends the lanes with `rel` to the ready list (one atomic per warp).
__device__ __forceinline__ void ready_append(bool rel, u32 p, u32 *next, u32 *next_cnt, int lane) {
  const unsigned m = __ballot_sync(FULL, rel);
  if (!m) return;
  u32 pos = 0;
  if (lane == 0) pos = atomicAdd(next_cnt, (u32)__popc(m));
  pos = __shfl_sync(FULL, pos, 0);
  if (rel) next[pos + __popc(m & ((1u << lane) - 1u))] = p;
}

// Releases the predecessors of the SCCs just evaluated: an SCC whose last
// unevaluated successor this was joins the next ready list.  A lane walks
// lists of at most 32, the warp longer ones; lists above kDpHuge are left to
// dp_release_huge (listed in huge[]).
__device__ __forceinline__ void dp_release(const u32 *list, u32 cnt, const u32 *poff, const u32 *pred, u32 *rem, u32 *next,
                             u32 *next_cnt, u32 *huge, u32 *nhuge) {
  const int lane = threadIdx.x & 31;
  for (u32 base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; base < cnt; base += gridDim.x * blockDim.x) {
    const u32 i = base + lane;
    u32 b = 0, e = 0;
    if (i < cnt) {
      const u32 c = list[i];
      b = poff[c];
      e = poff[c + 1];
      if (e - b > kDpHuge) {
        huge[atomicAdd(nhuge, 1u)] = c;
        e = b;
      }
    }
    const bool light = e - b <= 32;
    const u32 np = light ? e - b : 0;
    const u32 maxn = __reduce_max_sync(FULL, np);
    for (u32 j = 0; j < maxn; ++j) {
      u32 p = 0;
      bool rel = false;
      if (j < np) {
        p = pred[b + j];
        rel = atomicSub(&rem[p], 1u) == 1u;
      }
      ready_append(rel, p, next, next_cnt, lane);
    }
    for (unsigned hv = __ballot_sync(FULL, !light); hv; hv &= hv - 1) {
      const int src = __ffs(hv) - 1;
      const u32 hb = __shfl_sync(FULL, b, src), he = __shfl_sync(FULL, e, src);
      for (u32 k0 = hb; k0 < he; k0 += 32) {
        const u32 k = k0 + lane;
        u32 p = 0;
        bool rel = false;
        if (k < he) {
          p = pred[k];
          rel = atomicSub(&rem[p], 1u) == 1u;
        }
        ready_append(rel, p, next, next_cnt, lane);
      }
    }
  }
}

// The listed SCCs with more than kDpHuge predecessors, each by the whole grid.
__device__ __forceinline__ void dp_release_huge(const u32 *huge, u32 nh, const u32 *poff, const u32 *pred, u32 *rem,
                                  u32 *next, u32 *next_cnt) {
  const int lane = threadIdx.x & 31;
  for (u32 h = 0; h < nh; ++h) {
    const u32 c = huge[h];
    const u32 b = poff[c], e = poff[c + 1];
    for (u32 k0 = b + ((blockIdx.x * blockDim.x + threadIdx.x) & ~31u); k0 < e; k0 += gridDim.x * blockDim.x) {
      const u32 k = k0 + lane;
      u32 p = 0;
      bool rel = false;
      if (k < e) {
        p = pred[k];
        rel = atomicSub(&rem[p], 1u) == 1u;
      }
      ready_append(rel, p, next, next_cnt, lane);
    }
  }
}

// Sinks first until every SCC is evaluated, one cooperative launch: a round
// evaluates the ready list and releases the predecessors into the next one
// (and, when there are any, the long predecessor lists by the whole grid).
// cnt[3]: list lengths, round r's in cnt[r % 2], and unused; nhuge[3]: in turn.
__global__ void __launch_bounds__(kLoopTPB) k_dp(u32 *listA, u32 *listB, u32 *cnt, const u32 *soff, const u32 *succ,
                                                 const u32 *poff, const u32 *pred, const u32 *wgt,
                                                 const u32 *dist_from_big, const u32 *dist_to_big, u32 big,
                                                 u64 reach_big, u32 n, u64 *A, u64 *O, u32 *rem, u32 *huge, u32 *nhuge,
                                                 GridBar *bar, u64 timeout) {
  for (u32 r = 0;; ++r) {
    const u32 c = *(volatile u32 *)&cnt[r & 1];
    if (c == 0) return;
    const u32 *cur = r & 1 ? listB : listA;
    u32 *next = r & 1 ? listA : listB, *next_cnt = &cnt[(r & 1) ^ 1], *nh = &nhuge[r % 3];
    dp_eval(cur, c, soff, succ, wgt, dist_from_big, dist_to_big, big, reach_big, n, A, O);
    dp_release(cur, c, poff, pred, rem, next, next_cnt, huge, nh);
    // every block has read cnt[r % 2] and, a round ago, nhuge[(r + 2) % 3]
    if (!grid_sync(bar, timeout, [&] {
          cnt[r & 1] = 0;
          nhuge[(r + 2) % 3] = 0;
        }))
      return;
    const u32 m = *(volatile u32 *)nh;
    if (m) {
      dp_release_huge(huge, m, poff, pred, rem, next, next_cnt);
      if (!grid_sync(bar, timeout, [] {})) return;
    }
  }
}

__global__ void k_write_bounds(const u32 *comp, u32 n, const u64 *A, const u64 *O, const u32 *wgt, u32 *alpha,
                               u32 *omega, u32 *scc_size) {
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    u32 c = comp[v];
    alpha[v] = (u32)A[c];
    omega[v] = (u32)(O[c] < n ? O[c] : n);
    scc_size[v] = wgt[c];
  }
}

struct DevBufs {
  std::vector<void *> ptrs;
  cudaStream_t st;
  ~DevBufs() {
    for (void *p : ptrs) cudaFreeAsync(p, st);
  }
  template <typename T>
  cudaError_t get(T **p, size_t count) {
    cudaError_t e = dev_malloc(p, std::max<size_t>(count, 1) * sizeof(T), st);
    if (e == cudaSuccess) ptrs.push_back(*p);
    return e;
  }
};

}  // namespace

// Device words of one call, read together.
struct SccWords {
  GridBar bar;       // of the launches that loop over rounds
  BfsCtl bfs[4];     // of the reach searches
  u64 best0, best;   // the first pivot; the biggest SCC's vertex
  u64 left;          // the pivot of what neither trimming nor the first pivot took (0: nothing)
  u32 flag[2];       // round flags
  u32 big, big_graph, big_pivot;  // the biggest SCC, its graph and that graph's pivot
  u32 reach;                      // vertices reached from that pivot (or from big)
};

int reach_directed_gpu(tkc_graph *g, const u32 *gid, u32 ng) {
  tkc_ctx *ctx = g->ctx;
  cudaStream_t st = ctx->stream;
  const u32 n = g->n;
  const bool many = gid && ng > 1;
  DevBufs b;
  b.st = st;
  u32 *outd, *ind, *comp, *fw, *bw, *color, *found, *wgt, *minid;
  uint8_t *active;
  SccWords *wd;
  TKC_TRY(b.get(&outd, n));
  TKC_TRY(b.get(&ind, n));
  TKC_TRY(b.get(&comp, n));
  TKC_TRY(b.get(&fw, n));
  TKC_TRY(b.get(&bw, n));
  TKC_TRY(b.get(&wgt, n));
  TKC_TRY(b.get(&minid, n));
  TKC_TRY(b.get(&active, n));
  TKC_TRY(b.get(&wd, 1));
  TKC_TRY(cudaMemsetAsync(wd, 0, sizeof(SccWords), st));
  u64 timeout = grid_timeout(ctx);
  GridBar *bar = &wd->bar;
  u32 *flag = wd->flag;
  auto loop_launch = [&](const void *kernel, int blocks, void **args) {
    if (blocks <= 0) return cudaErrorCooperativeLaunchTooLarge;
    note_launches(1);
    return cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(kLoopTPB), args, 0, st);
  };
  SccWords h = {};
  auto error_of = [&]() {
    int e = h.bar.err;
    for (const BfsCtl &c : h.bfs)
      if (!e) e = c.bar.err;
    return e;
  };
  // trims until stable, then finds the pivot of what is left
  auto trim_and_pivot = [&](u64 *best) -> int {
    TKC_TRY(cudaMemsetAsync(flag, 0, 2 * sizeof(u32), st));
    TKC_TRY(cudaMemsetAsync(best, 0, sizeof(u64), st));
    void *args[] = {(void *)&g->off, (void *)&g->col, (void *)&g->ioff, (void *)&g->icol, (void *)&n, (void *)&outd,
                    (void *)&ind, (void *)&active, (void *)&comp, (void *)&flag, (void *)&bar, (void *)&timeout};
    TKC_TRY(loop_launch((const void *)k_trim, grid_blocks(ctx, k_trim, kLoopTPB, n), args));
    TKC_LAUNCH(k_pivot<<<grid_of(n), 256, 0, st>>>(outd, ind, active, n, best));
    TKC_TRY(cudaGetLastError());
    return TKC_OK;
  };
  // sizes of the SCCs, the biggest one, what the first pivot reaches, and the
  // arcs between SCCs (counted per block; their number is blk[cross_grid])
  const unsigned cross_grid = grid_of(arc_threads(g->arcs));
  u32 *blk = nullptr, *blk_tmp = nullptr, *piv = nullptr;
  TKC_TRY(b.get(&blk, (size_t)cross_grid + 1));
  TKC_TRY(b.get(&blk_tmp, ((size_t)cross_grid + 1) / 4096 + 2));
  auto statistics = [&]() -> int {
    TKC_TRY(cudaMemsetAsync(wgt, 0, (size_t)n * sizeof(u32), st));
    TKC_TRY(cudaMemsetAsync(minid, 0xff, (size_t)n * sizeof(u32), st));
    TKC_TRY(cudaMemsetAsync(&wd->best, 0, sizeof(u64), st));
    TKC_TRY(cudaMemsetAsync(&wd->reach, 0, sizeof(u32), st));
    TKC_LAUNCH(k_comp_stats<<<grid_of(n), 256, 0, st>>>(comp, n, wgt, minid));
    TKC_LAUNCH(k_biggest<<<grid_of(n), 256, 0, st>>>(wgt, minid, n, &wd->best));
    TKC_LAUNCH(k_big<<<1, 1, 0, st>>>(comp, &wd->best, many ? gid : nullptr, piv, &wd->best0, &wd->big, &wd->big_graph,
                                 &wd->big_pivot));
    TKC_LAUNCH(k_count_reached<<<grid_of(n), 256, 0, st>>>(fw, n, many ? gid : nullptr, &wd->big_graph, &wd->reach));
    TKC_TRY(cudaMemsetAsync(blk + cross_grid, 0, sizeof(u32), st));
    TKC_LAUNCH(k_cross<false><<<cross_grid, 256, 0, st>>>(g->off, g->col, comp, n, g->arcs, blk, nullptr, nullptr));
    return scan_exclusive_u32(blk, blk, (u64)cross_grid + 1, blk_tmp, st);
  };
  TKC_LAUNCH(k_trim_init<<<grid_of(n), 256, 0, st>>>(g->off, g->ioff, n, outd, ind, active, comp));
  TKC_RC(trim_and_pivot(&wd->best0));
  // Forward and backward reach of the pivot.  The searches run over the whole
  // graph, not only the untrimmed vertices: a trimmed vertex is its own SCC, so
  // the intersection is the same, and the full reach sets serve again below
  // when this SCC is the biggest.
  if (many) {
    // Several graphs: one pivot per graph and one forward and one backward
    // search from all of them, so that every graph's largest SCC is found in
    // this round (with a single pivot, only one graph's would be, and the
    // colouring rounds would take the rest).
    u64 *gbest;
    u32 *plist, *pcnt;
    TKC_TRY(b.get(&gbest, ng));
    TKC_TRY(b.get(&piv, ng));
    TKC_TRY(b.get(&plist, ng));
    TKC_TRY(b.get(&pcnt, 1));
    TKC_TRY(cudaMemsetAsync(gbest, 0, (size_t)ng * sizeof(u64), st));
    TKC_TRY(cudaMemsetAsync(pcnt, 0, sizeof(u32), st));
    TKC_LAUNCH(k_pivot_many<<<grid_of(n), 256, 0, st>>>(outd, ind, active, gid, n, gbest));
    TKC_LAUNCH(k_pivot_list<<<grid_of(ng), 256, 0, st>>>(gbest, ng, piv, plist, pcnt));
    TKC_RC(bfs_reach(ctx, g->off, g->col, g->ioff, g->icol, n, g->arcs, fw, 0, nullptr, plist, pcnt, &wd->bfs[0], st));
    TKC_RC(bfs_reach(ctx, g->ioff, g->icol, g->off, g->col, n, g->arcs, bw, 0, nullptr, plist, pcnt, &wd->bfs[1], st));
    TKC_LAUNCH(k_fwbw_mark_many<<<grid_of(n), 256, 0, st>>>(fw, bw, gid, piv, n, active, comp));
  } else {
    TKC_RC(bfs_reach(ctx, g->off, g->col, g->ioff, g->icol, n, g->arcs, fw, INF, &wd->best0, nullptr, nullptr,
                     &wd->bfs[0], st));
    TKC_RC(bfs_reach(ctx, g->ioff, g->icol, g->off, g->col, n, g->arcs, bw, INF, &wd->best0, nullptr, nullptr,
                     &wd->bfs[1], st));
    TKC_LAUNCH(k_fwbw_mark<<<grid_of(n), 256, 0, st>>>(fw, bw, n, active, comp, &wd->best0));
  }
  TKC_RC(trim_and_pivot(&wd->left));
  // Usually nothing is left, so what follows is enqueued before the host knows
  // (one wait for all of it; every vertex has a valid SCC name throughout).
  TKC_RC(statistics());
  u32 m = 0;
  TKC_TRY(read_back2(&h, wd, sizeof(SccWords), &m, blk + cross_grid, sizeof(u32), st));
  TKC_RC(error_of());
  if (h.left) {
    TKC_TRY(b.get(&color, n));
    TKC_TRY(b.get(&found, n));
    while (h.left) {
      // colouring round over the remaining vertices
      TKC_TRY(cudaMemsetAsync(flag, 0, 2 * sizeof(u32), st));
      void *args[] = {(void *)&g->off, (void *)&g->col, (void *)&g->ioff, (void *)&g->icol, (void *)&n,
                      (void *)&active, (void *)&color, (void *)&found, (void *)&comp, (void *)&flag, (void *)&bar,
                      (void *)&timeout};
      TKC_TRY(loop_launch((const void *)k_color_round, grid_blocks(ctx, k_color_round, kLoopTPB, n), args));
      TKC_RC(trim_and_pivot(&wd->left));
      TKC_TRY(read_back(&h, wd, sizeof(SccWords), st));
      TKC_RC(error_of());  // (a round that ran out of its budget would repeat for ever)
    }
    TKC_RC(statistics());
    TKC_TRY(read_back2(&h, wd, sizeof(SccWords), &m, blk + cross_grid, sizeof(u32), st));
  }
  TKC_TRY(cudaMemcpyAsync(g->comp, comp, (size_t)n * sizeof(u32), cudaMemcpyDeviceToDevice, st));
  // exact reach of the biggest SCC (forward), and the SCCs that reach it
  // (backward); only reachability is used, the same from every vertex of the
  // SCC, so the sweeps from its graph's pivot serve when that names the biggest
  // SCC (several graphs: without what the other graphs' pivots reached)
  u32 big = h.big;
  if (big == h.big_pivot) {
    if (many) TKC_LAUNCH(k_keep_graph<<<grid_of(n), 256, 0, st>>>(gid, h.big_graph, n, fw, bw));
  } else {
    TKC_RC(bfs_reach(ctx, g->off, g->col, g->ioff, g->icol, n, g->arcs, fw, big, nullptr, nullptr, nullptr, &wd->bfs[2],
                     st));
    TKC_RC(bfs_reach(ctx, g->ioff, g->icol, g->off, g->col, n, g->arcs, bw, big, nullptr, nullptr, nullptr, &wd->bfs[3],
                     st));
    TKC_TRY(cudaMemsetAsync(&wd->reach, 0, sizeof(u32), st));
    TKC_LAUNCH(k_count_reached<<<grid_of(n), 256, 0, st>>>(fw, n, nullptr, nullptr, &wd->reach));
    TKC_TRY(read_back(&h, wd, sizeof(SccWords), st));
    TKC_RC(error_of());
  }
  u64 reach_big = h.reach;
  // condensation arcs, sorted by (cu, cv) and deduplicated
  u32 *cu, *cv, *pos, *tmp, *su, *sv, *soff, *poff, *pcur, *pred, *rem, *listA, *listB;
  u64 *A, *O;
  TKC_TRY(b.get(&cu, m));
  TKC_TRY(b.get(&cv, m));
  TKC_TRY(b.get(&pos, (size_t)m + 1));
  TKC_TRY(b.get(&su, m));
  TKC_TRY(b.get(&sv, m));
  TKC_TRY(b.get(&soff, (size_t)n + 1));
  TKC_TRY(b.get(&poff, (size_t)n + 1));
  TKC_TRY(b.get(&pcur, n));
  TKC_TRY(b.get(&tmp, (std::max<size_t>(m, n) + 1) / 4096 + 2));
  TKC_LAUNCH(k_cross<true><<<cross_grid, 256, 0, st>>>(g->off, g->col, comp, n, g->arcs, blk, cu, cv));
  int bits = 0;
  while (bits < 32 && ((n - 1) >> bits) != 0) ++bits;
  TKC_RC(radix_sort_u32_pairs(cv, cu, m, bits, st));  // by target
  TKC_RC(radix_sort_u32_pairs(cu, cv, m, bits, st));  // then by source, stable
  TKC_LAUNCH(k_unique_flags<<<grid_of(m), 256, 0, st>>>(cu, cv, m, pos));
  TKC_RC(scan_exclusive_u32(pos, pos, (u64)m + 1, tmp, st));
  TKC_TRY(cudaMemsetAsync(soff, 0, ((size_t)n + 1) * sizeof(u32), st));
  TKC_TRY(cudaMemsetAsync(poff, 0, ((size_t)n + 1) * sizeof(u32), st));
  TKC_LAUNCH(k_unique_compact<<<grid_of(m), 256, 0, st>>>(cu, cv, pos, m, su, sv, soff, poff));
  TKC_RC(scan_exclusive_u32(soff, soff, (u64)n + 1, tmp, st));
  TKC_RC(scan_exclusive_u32(poff, poff, (u64)n + 1, tmp, st));
  TKC_TRY(b.get(&pred, m));
  TKC_TRY(cudaMemsetAsync(pcur, 0, (size_t)n * sizeof(u32), st));
  TKC_LAUNCH(k_pred_scatter<<<grid_of(m), 256, 0, st>>>(su, sv, pos + m, poff, pcur, pred));
  // su is sorted by source with unique pairs, so sv is the successor list
  // indexed by soff; Algorithm 6 sinks first
  TKC_TRY(b.get(&rem, n));
  TKC_TRY(b.get(&listA, n));
  TKC_TRY(b.get(&listB, n));
  TKC_TRY(b.get(&A, n));
  TKC_TRY(b.get(&O, n));
  u32 *huge = nullptr, *cnt = nullptr;
  TKC_TRY(b.get(&huge, (size_t)m / kDpHuge + 1));
  TKC_TRY(b.get(&cnt, 6));
  TKC_TRY(cudaMemsetAsync(cnt, 0, 6 * sizeof(u32), st));
  TKC_LAUNCH(k_sinks<<<grid_of(n), 256, 0, st>>>(wgt, soff, n, rem, listA, cnt));
  {
    u32 *nhuge = cnt + 3;
    void *args[] = {(void *)&listA, (void *)&listB, (void *)&cnt, (void *)&soff, (void *)&sv, (void *)&poff,
                    (void *)&pred, (void *)&wgt, (void *)&fw, (void *)&bw, (void *)&big, (void *)&reach_big,
                    (void *)&n, (void *)&A, (void *)&O, (void *)&rem, (void *)&huge, (void *)&nhuge, (void *)&bar,
                    (void *)&timeout};
    TKC_TRY(loop_launch((const void *)k_dp, grid_blocks(ctx, k_dp, kLoopTPB, n), args));
  }
  TKC_LAUNCH(k_write_bounds<<<grid_of(n), 256, 0, st>>>(comp, n, A, O, wgt, g->alpha, g->omega, g->scc_size));
  TKC_TRY(cudaGetLastError());
  TKC_TRY(read_back(&h, wd, sizeof(SccWords), st));
  return error_of();
}

}  // namespace tkc
