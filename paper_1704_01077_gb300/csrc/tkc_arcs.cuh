// Warp-cooperative walks over the arcs of a CSR graph, balanced by arcs.
//
// Kernels that visit every arc u -> v with its source u (in-arc CSR build,
// SCC condensation) give each warp a fixed range of arc indices instead of a
// set of vertices: a vertex with a long out-row (an R-MAT hub holds about
// 10^5 arcs) is then spread over many warps rather than walked by one, and
// short rows are taken 32 at a time.  The source of each arc comes from a
// 32-way search of the offsets and a window of 32 consecutive row ends held
// one per lane.
#pragma once

#include <cstdint>

namespace tkc {

// Largest u in [0, n) with off[u] <= a, for a < off[n] (so that u's row holds
// arc a).  32-way search: each round every lane probes one of 32 evenly
// spaced offsets and the range shrinks to one gap.  Called by all 32 lanes
// with the same arguments; every lane returns the same u.  Lane 0's probe holds
// by the invariant and is not asked: the check of a CSR walks offsets that may
// not start at 0, and a round in which no lane answered would have no gap to
// shrink to.  So u < n and the search ends whatever the offsets hold.
__device__ __forceinline__ uint32_t warp_arc_source(const uint32_t *off, uint32_t n, uint64_t a, int lane) {
  uint32_t lo = 0, hi = n;  // off[lo] <= a; the answer lies in [lo, hi)
  while (hi - lo > 1) {
    const uint32_t step = (hi - lo + 31) / 32;
    const uint32_t p = lo + step * (uint32_t)lane;
    const bool ok = lane == 0 || (p < hi && off[p] <= a);  // true on a prefix of the lanes
    const unsigned m = __ballot_sync(0xffffffffu, ok);
    const uint32_t l = 31u - (uint32_t)__clz(m);
    lo += step * l;
    hi = lo + step < hi ? lo + step : hi;
  }
  return lo;
}

// Calls f(u, i, valid, rs) for the arcs i of [a0, a1), 32 at a time (lane j
// takes arc t0 + j of each group; `valid` is false past a1, and then u and i
// are not arcs of the graph), u the source of arc i and rs the first arc of
// u's row (only with kRowStart; 0 otherwise).  a0 < a1 <= off[n].  All 32
// lanes run the same number of groups, so f may use warp collectives.  With
// offsets that are not nondecreasing the sources are meaningless, but every
// offset read stays within off[0 .. n] and the walk ends.
template <bool kRowStart = false, typename F>
__device__ __forceinline__ void warp_walk_arcs(const uint32_t *off, uint32_t n, uint64_t a0, uint64_t a1, int lane,
                                               F &&f) {
  uint32_t u = warp_arc_source(off, n, a0, lane);
  uint32_t wstart = kRowStart ? off[u] : 0u;  // first arc of the window's first row
  while (a0 < a1) {
    // row ends of the window u .. u + 31 (past the last vertex: no end)
    const uint64_t w = (uint64_t)u + 1 + (uint32_t)lane;
    const uint32_t vend = w <= n ? off[w] : 0xffffffffu;
    const uint32_t wlast = __shfl_sync(0xffffffffu, vend, 31);
    const uint64_t stop = a1 < (uint64_t)wlast ? a1 : (uint64_t)wlast;
    for (uint64_t t0 = a0; t0 < stop; t0 += 32) {
      const uint64_t i = t0 + (uint32_t)lane;
      // rows of the window ending at or before i (vend is nondecreasing)
      uint32_t cnt = 0;
#pragma unroll
      for (uint32_t s = 16; s > 0; s >>= 1) {
        const uint32_t x = __shfl_sync(0xffffffffu, vend, (int)(cnt + s - 1));
        if ((uint64_t)x <= i) cnt += s;
      }
      uint32_t rs = 0;
      if (kRowStart) {
        const uint32_t prev = __shfl_sync(0xffffffffu, vend, (int)((cnt + 31) & 31));
        rs = cnt ? prev : wstart;
      }
      f(u + cnt, i, i < stop, rs);
    }
    if (stop > a0) a0 = stop;
    wstart = wlast;
    u += 32;
  }
}

// Arcs per warp task of the walks above.  A task is a chain of dependent loads
// (the search, a window of row ends per 32 rows, 32 arcs a step), so a small
// graph is cut into shorter tasks that fill the chip -- about 8 192 warps, the
// least a task's search is worth being 128 arcs -- and a large one into tasks
// of 2 048 arcs.  (With 2 048 at every size, the graphs of 1 000 to 200 000
// vertices that a multi-graph call loads took 50 us of validation and 114 us
// of symmetry check each on average, nearly all of it one warp's chain.)
__host__ __device__ inline uint32_t arc_chunk(uint64_t arcs) {
  const uint64_t c = (arcs / 8192 + 31) / 32 * 32;
  return c < 128 ? 128u : c > 2048 ? 2048u : (uint32_t)c;
}

// Threads that give every task its own warp.
inline uint64_t arc_threads(uint64_t arcs) { return (arcs + arc_chunk(arcs) - 1) / arc_chunk(arcs) * 32; }

// Calls f(u, i, valid, rs) for every arc of the graph, the arcs dealt to the
// grid's warps in tasks of arc_chunk(arcs) consecutive indices (task c to warp
// c mod warps: a kernel launched twice with the same grid gives each block
// the same arcs).
// Block `block` of `nblocks`: of the grid, or of the part of it that a launch
// over several graphs gives this one.
template <bool kRowStart = false, typename F>
__device__ __forceinline__ void blocks_walk_arcs(const uint32_t *off, uint32_t n, uint64_t arcs, uint32_t block,
                                                 uint32_t nblocks, F &&f) {
  const int lane = threadIdx.x & 31;
  const uint64_t warp = ((uint64_t)block * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)nblocks * blockDim.x) >> 5;
  const uint32_t chunk = arc_chunk(arcs);
  for (uint64_t a0 = warp * chunk; a0 < arcs; a0 += nwarps * chunk) {
    const uint64_t a1 = a0 + chunk < arcs ? a0 + chunk : arcs;
    warp_walk_arcs<kRowStart>(off, n, a0, a1, lane, f);
  }
}

template <bool kRowStart = false, typename F>
__device__ __forceinline__ void grid_walk_arcs(const uint32_t *off, uint32_t n, uint64_t arcs, F &&f) {
  blocks_walk_arcs<kRowStart>(off, n, arcs, blockIdx.x, gridDim.x, f);
}

}  // namespace tkc
