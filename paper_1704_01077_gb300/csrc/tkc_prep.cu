// Preprocessing for Algorithm 1: CSR validation and in-arc CSR, the
// computeBoundsDeg source order (Section 4), and the reach bounds alpha/omega
// (exact component sizes for undirected graphs here; Algorithm 6 of Section
// 8.4 for directed graphs in tkc_scc.cu).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "tkc_arcs.cuh"
#include "tkc_grid.cuh"
#include "tkc_internal.cuh"

namespace tkc {

typedef uint32_t u32;
typedef unsigned long long u64;
static constexpr unsigned FULL = 0xffffffffu;

// ------------------------------------------------------------------ device-wide exclusive scan

static constexpr int kScanTPB = 1024;
static constexpr int kScanItems = 4;
static constexpr int kScanTile = kScanTPB * kScanItems;

__device__ __forceinline__ u32 block_exscan_1024(u32 x, u32 *s_warp, u32 *total) {
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  u32 incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    u32 t = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    u32 v = lane < (int)(blockDim.x >> 5) ? s_warp[lane] : 0;
    u32 vi = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      u32 t = __shfl_up_sync(FULL, vi, o);
      if (lane >= o) vi += t;
    }
    s_warp[lane] = vi - v;
    if (lane == 31) s_warp[32] = vi;
  }
  __syncthreads();
  u32 res = s_warp[wid] + incl - x;
  *total = s_warp[32];
  __syncthreads();
  return res;
}

__global__ void k_scan_bsum(const u32 *in, u64 len, u32 *bsum) {
  __shared__ u32 s_warp[33];
  u64 base = (u64)blockIdx.x * kScanTile + (u64)threadIdx.x * kScanItems;
  u32 s = 0;
  for (int i = 0; i < kScanItems; ++i)
    if (base + i < len) s += in[base + i];
  u32 total;
  block_exscan_1024(s, s_warp, &total);
  if (threadIdx.x == 0) bsum[blockIdx.x] = total;
}

__global__ void k_scan_small(u32 *a, u32 len) {
  __shared__ u32 s_warp[33];
  u32 per = (len + kScanTPB - 1) / kScanTPB;
  u32 lo = threadIdx.x * per, hi = min(len, lo + per);
  u32 s = 0;
  for (u32 i = lo; i < hi; ++i) s += a[i];
  u32 total;
  u32 pre = block_exscan_1024(s, s_warp, &total);
  for (u32 i = lo; i < hi; ++i) {
    u32 t = a[i];
    a[i] = pre;
    pre += t;
  }
}

// Second pass: every block scans its tile from the sum of the tiles before it,
// which bsum[block] holds (kSummed, after k_scan_small) or which the block adds
// up itself.
template <bool kSummed>
__global__ void k_scan_apply(const u32 *in, u32 *out, u64 len, const u32 *bsum) {
  __shared__ u32 s_warp[33];
  __shared__ u32 s_base;
  u32 before = 0;
  if (kSummed) {
    before = bsum[blockIdx.x];
  } else {
    u32 mine = 0;
    for (u32 i = threadIdx.x; i < blockIdx.x; i += kScanTPB) mine += bsum[i];
    mine = __reduce_add_sync(FULL, mine);
    if (threadIdx.x == 0) s_base = 0;
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&s_base, mine);
    __syncthreads();
    before = s_base;
  }
  u64 base = (u64)blockIdx.x * kScanTile + (u64)threadIdx.x * kScanItems;
  u32 v[kScanItems];
  u32 s = 0;
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = base + i < len ? in[base + i] : 0;
    s += v[i];
  }
  u32 total;
  u32 pre = block_exscan_1024(s, s_warp, &total) + before;
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i < len) out[base + i] = pre;
    pre += v[i];
  }
}

// The whole scan by one block, tile after tile.
__global__ void k_scan_one(const u32 *in, u32 *out, u32 len) {
  __shared__ u32 s_warp[33];
  u32 before = 0;
  for (u32 t = 0; t < len; t += kScanTile) {
    const u32 base = t + threadIdx.x * kScanItems;
    u32 v[kScanItems];
    u32 s = 0;
    for (int i = 0; i < kScanItems; ++i) {
      v[i] = base + i < len ? in[base + i] : 0;
      s += v[i];
    }
    u32 total;
    u32 pre = block_exscan_1024(s, s_warp, &total) + before;
    for (int i = 0; i < kScanItems; ++i) {
      if (base + i < len) out[base + i] = pre;
      pre += v[i];
    }
    before += total;
  }
}

// out[i] = sum of in[0..i); in and out may alias.  tmp holds ceil(len/4096) words.
// A launch costs more than a short scan's work, so up to 4 tiles are one
// block's (2 us a tile), and up to 1 024 tiles take two launches, each block
// adding up at most 1 024 tile sums; only longer ones scan the sums between.
static int scan_exclusive(const u32 *in, u32 *out, u64 len, u32 *tmp, cudaStream_t st) {
  if (len == 0) return TKC_OK;
  u64 nb = (len + kScanTile - 1) / kScanTile;
  if (nb > (u64)kScanTPB * 4096) return TKC_EOVERFLOW;
  if (nb <= 4) {
    TKC_LAUNCH(k_scan_one<<<1, kScanTPB, 0, st>>>(in, out, (u32)len));
  } else if (nb <= 1024) {
    TKC_LAUNCH(k_scan_bsum<<<(unsigned)nb, kScanTPB, 0, st>>>(in, len, tmp));
    TKC_LAUNCH(k_scan_apply<false><<<(unsigned)nb, kScanTPB, 0, st>>>(in, out, len, tmp));
  } else {
    TKC_LAUNCH(k_scan_bsum<<<(unsigned)nb, kScanTPB, 0, st>>>(in, len, tmp));
    TKC_LAUNCH(k_scan_small<<<1, kScanTPB, 0, st>>>(tmp, (u32)nb));
    TKC_LAUNCH(k_scan_apply<true><<<(unsigned)nb, kScanTPB, 0, st>>>(in, out, len, tmp));
  }
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

// ------------------------------------------------------------------ CSR validation and transpose

enum : u32 { kBadOffsets = 1, kBadRange = 2, kSelfLoop = 4, kUnsorted = 8, kAsymmetric = 16 };

// Offsets from 0 to arcs, monotone and within arcs (a thread per vertex); ids
// in range, no self-loop, each row strictly increasing (sorted, no
// duplicates), checked arc by arc.
__device__ __forceinline__ void validate_csr(const u32 *off, const u32 *col, u32 n, u64 arcs, u32 block, u32 nblocks,
                                             u32 *flags) {
  const int lane = threadIdx.x & 31;
  u32 f = 0;
  if (block == 0 && threadIdx.x == 0 && (off[0] != 0 || off[n] != arcs)) f |= kBadOffsets;
  for (u64 v = (u64)block * blockDim.x + threadIdx.x; v < n; v += (u64)nblocks * blockDim.x) {
    const u32 b = off[v], e = off[v + 1];
    if (e < b || e > arcs) f |= kBadOffsets;
  }
  // the arcs in chunks with their sources (tkc_arcs.cuh: a hub's row is
  // spread over many warps; reads stay in bounds even when the offsets are
  // bad, which the loop above reports)
  blocks_walk_arcs<true>(off, n, arcs, block, nblocks, [&](u32 u, u64 i, bool valid, u32 rs) {
    if (!valid) return;
    const u32 c = col[i];
    if (c >= n) f |= kBadRange;
    if (c == u) f |= kSelfLoop;
    if (i > rs && col[i - 1] >= c) f |= kUnsorted;
  });
  f = __reduce_or_sync(FULL, f);
  if (lane == 0 && f) atomicOr(flags, f);
}

// Undirected input: every arc u->v needs the arc v->u (binary search in v's
// row; the graph already passed k_validate, so rows are sorted).  Arcs in
// chunks with their sources (tkc_arcs.cuh), so a hub's row is spread over
// many warps.
__device__ __forceinline__ void symmetric_csr(const u32 *off, const u32 *col, u32 n, u64 arcs, u32 block, u32 nblocks,
                                              u32 *flags) {
  const int lane = threadIdx.x & 31;
  u32 f = 0;
  blocks_walk_arcs(off, n, arcs, block, nblocks, [&](u32 u, u64 i, bool valid, u32) {
    if (!valid) return;
    const u32 v = col[i];
    u32 lo = off[v], hi = off[v + 1];
    const u32 end = hi;
    while (lo < hi) {
      const u32 mid = (lo + hi) >> 1;
      if (col[mid] < u) lo = mid + 1;
      else hi = mid;
    }
    if (lo >= end || col[lo] != u) f |= kAsymmetric;
  });
  f = __reduce_or_sync(FULL, f);
  if (lane == 0 && f) atomicOr(flags, f);
}

__global__ void k_validate(const u32 *off, const u32 *col, u32 n, u64 arcs, u32 *flags) {
  validate_csr(off, col, n, arcs, blockIdx.x, gridDim.x, flags);
}

__global__ void k_symmetric(const u32 *off, const u32 *col, u32 n, u64 arcs, u32 *flags) {
  symmetric_csr(off, col, n, arcs, blockIdx.x, gridDim.x, flags);
}

// The checks of many graphs in one launch: graph i of the table has blocks
// blk0[kSym] .. of the grid.  A graph of 1 000 to 200 000 vertices fills the
// chip for 6 (validation) or 13 us, mostly one chain of loads; 512 of them,
// half undirected, took 3.2 and 3.4 ms one launch after the other.
template <bool kSym>
__global__ void k_check_many(const CsrCheck *__restrict__ t, u32 ng, u32 *flags) {
  const int lane = threadIdx.x & 31;
  u32 lo = 0, hi = ng;  // blk0[lo] <= this block: the last such graph has it (others of that blk0 have no block)
  while (hi - lo > 1) {
    const u32 step = (hi - lo + 31) / 32, p = lo + step * (u32)lane;
    const unsigned m = __ballot_sync(FULL, p < hi && t[p].blk0[kSym] <= blockIdx.x);
    lo += step * (31u - (u32)__clz(m));
    hi = lo + step < hi ? lo + step : hi;
  }
  const CsrCheck c = t[lo];
  const u32 block = blockIdx.x - c.blk0[kSym];
  if (kSym) symmetric_csr(c.off, c.col, c.n, c.arcs, block, c.nblk[kSym], flags + lo);
  else validate_csr(c.off, c.col, c.n, c.arcs, block, c.nblk[kSym], flags + lo);
}

// In-degrees: cnt[v] += 1 per arc u -> v, 32 consecutive arcs per warp step
// (coalesced column reads).  Lanes adding to the same vertex (the hubs of
// skewed in-degree distributions) add their count in one atomic.
__global__ void k_in_count(const u32 *__restrict__ col, u64 arcs, u32 *__restrict__ cnt) {
  const int lane = threadIdx.x & 31;
  for (u64 base = ((u64)blockIdx.x * blockDim.x + threadIdx.x) & ~31ull; base < arcs;
       base += (u64)gridDim.x * blockDim.x) {
    const u64 i = base + lane;
    const bool valid = i < arcs;
    const u32 v = valid ? col[i] : 0xffffffffu;
    const unsigned peers = __match_any_sync(FULL, v);
    if (valid && __ffs(peers) - 1 == lane) atomicAdd(&cnt[v], (u32)__popc(peers));
  }
}

// The in-arc columns: arc u -> v takes slot cursor[v]++ of v's in-row (cursor
// starts at ioff).  Arcs are dealt to warps in fixed chunks with their
// sources found by search (tkc_arcs.cuh), so a hub's out-row is spread over
// many warps.  Lanes writing the same in-row take consecutive slots from one
// atomic.  In-rows come out roughly in ascending source order (chunks are
// taken in arc order).
__global__ void k_in_fill(const u32 *__restrict__ off, const u32 *__restrict__ col, u32 n, u64 arcs,
                          u32 *__restrict__ cursor, u32 *__restrict__ icol) {
  const int lane = threadIdx.x & 31;
  grid_walk_arcs(off, n, arcs, [&](u32 u, u64 i, bool valid, u32) {
    const u32 v = valid ? col[i] : 0xffffffffu;
    const unsigned peers = __match_any_sync(FULL, v);
    const int leader = __ffs(peers) - 1;
    u32 pos = 0;
    if (valid && leader == lane) pos = atomicAdd(&cursor[v], (u32)__popc(peers));
    pos = __shfl_sync(FULL, pos, leader) + (u32)__popc(peers & ((1u << lane) - 1u));
    if (valid) icol[pos] = u;
  });
}

static unsigned grid_for(u64 work, unsigned tpb, unsigned cap = 152 * 16) {
  u64 b = (work + tpb - 1) / tpb;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (unsigned)b;
}

// Enqueues the structural checks of g's CSR (offsets, ids, self-loops, row
// order); violations are ORed into the device word *flag.  No host wait.
static int enqueue_validate(const tkc_graph *g, u32 *flag) {
  if (g->n == 0) return TKC_OK;
  cudaStream_t st = g->ctx->stream;
  TKC_LAUNCH(k_validate<<<grid_for(std::max<u64>(g->n, arc_threads(g->arcs)), 256), 256, 0,
                          st>>>(g->off, g->col, g->n, g->arcs, flag));
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

// Enqueues the symmetry check of an undirected graph into *flag; only for a
// CSR that passed enqueue_validate (it searches rows for ids).
static int enqueue_symmetric(const tkc_graph *g, u32 *flag) {
  if (g->n == 0 || g->directed) return TKC_OK;
  cudaStream_t st = g->ctx->stream;
  TKC_LAUNCH(k_symmetric<<<grid_for(arc_threads(g->arcs), 256), 256, 0, st>>>(
      g->off, g->col, g->n, g->arcs, flag));
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

// The blocks of each check of graph g in a launch over many graphs.
void check_entry(const tkc_graph *g, u32 blk0[2], CsrCheck *c) {
  c->off = g->off;
  c->col = g->col;
  c->n = g->n;
  c->arcs = g->arcs;
  c->nblk[0] = g->n ? grid_for(std::max<u64>(g->n, arc_threads(g->arcs)), 256) : 0;
  c->nblk[1] = g->n && !g->directed ? grid_for(arc_threads(g->arcs), 256) : 0;
  for (int s = 0; s < 2; ++s) {
    c->blk0[s] = blk0[s];
    blk0[s] += c->nblk[s];
  }
}

// Enqueues the structural (sym = 0) or the symmetry checks (1: only after the
// structural ones passed) of the ng graphs of the device table t, `blocks` in
// all; violations are ORed into flags[i].  No host wait.
int enqueue_check_many(tkc_ctx *ctx, const CsrCheck *t, u32 ng, int sym, u32 blocks, u32 *flags) {
  if (blocks == 0) return TKC_OK;
  if (sym) {
    TKC_LAUNCH(k_check_many<true><<<blocks, 256, 0, ctx->stream>>>(t, ng, flags));
  } else {
    TKC_LAUNCH(k_check_many<false><<<blocks, 256, 0, ctx->stream>>>(t, ng, flags));
  }
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

int validate_graph(tkc_graph *g) {
  cudaStream_t st = g->ctx->stream;
  if (g->n == 0) return TKC_OK;
  u32 *flags = nullptr;
  TKC_TRY(dev_malloc(&flags, sizeof(u32), st));
  TKC_TRY(cudaMemsetAsync(flags, 0, sizeof(u32), st));
  TKC_RC(enqueue_validate(g, flags));
  u32 hf = 0;
  TKC_TRY(read_back(&hf, flags, sizeof(u32), st));
  if (hf == 0 && !g->directed) {
    TKC_RC(enqueue_symmetric(g, flags));
    TKC_TRY(read_back(&hf, flags, sizeof(u32), st));
  }
  TKC_TRY(cudaFreeAsync(flags, st));
  if (hf) return TKC_EGRAPH;
  if (!g->directed) {
    g->ioff = g->off;
    g->icol = g->col;
  }
  return TKC_OK;  // a directed graph's in-arc CSR is built on first use (ensure_in_csr)
}

// Fills the in-arc columns of the CSR (off, col) with n vertices into icol,
// given its in-row offsets ioff (rows not sorted: an in-row holds its arcs in
// the order the fill reached them, roughly ascending source id).
static int fill_in_arcs(const u32 *off, const u32 *col, u32 n, u64 arcs, const u32 *ioff, u32 *icol,
                        cudaStream_t st) {
  if (!arcs) return TKC_OK;
  u32 *cursor = nullptr;
  TKC_TRY(dev_malloc(&cursor, (size_t)n * sizeof(u32), st));
  TKC_TRY(cudaMemcpyAsync(cursor, ioff, (size_t)n * sizeof(u32), cudaMemcpyDeviceToDevice, st));
  TKC_LAUNCH(k_in_fill<<<grid_for(arc_threads(arcs), 256), 256, 0, st>>>(
      off, col, n, arcs, cursor, icol));
  TKC_TRY(cudaGetLastError());
  TKC_TRY(cudaFreeAsync(cursor, st));
  return TKC_OK;
}

// Transpose of the CSR (off, col) with n vertices: the in-arc CSR.  *ioff and
// *icol are allocated here (on failure: null or an allocation, without content).
static int transpose_csr(const u32 *off, const u32 *col, u32 n, u64 arcs, u32 **ioff, u32 **icol,
                         cudaStream_t st) {
  u32 *tmp = nullptr;
  *ioff = *icol = nullptr;
  TKC_TRY(dev_malloc(ioff, ((size_t)n + 1) * sizeof(u32), st));
  TKC_TRY(dev_malloc(icol, std::max<size_t>(arcs, 1) * sizeof(u32), st));
  TKC_TRY(dev_malloc(&tmp, (((size_t)n + 1) / kScanTile + 2) * sizeof(u32), st));
  TKC_TRY(cudaMemsetAsync(*ioff, 0, ((size_t)n + 1) * sizeof(u32), st));
  if (arcs) {
    TKC_LAUNCH(k_in_count<<<grid_for(arcs, 256), 256, 0, st>>>(col, arcs, *ioff));
    TKC_TRY(cudaGetLastError());
  }
  TKC_RC(scan_exclusive(*ioff, *ioff, (u64)n + 1, tmp, st));
  TKC_RC(fill_in_arcs(off, col, n, arcs, *ioff, *icol, st));
  TKC_TRY(cudaFreeAsync(tmp, st));
  return TKC_OK;
}

// In-arc CSR of g.
int build_in_csr(const tkc_graph *g) {
  if (g->n == 0) return TKC_OK;
  cudaStream_t st = g->ctx->stream;
  u32 *ioff, *icol;
  const int rc = transpose_csr(g->off, g->col, g->n, g->arcs, &ioff, &icol, st);
  if (rc != TKC_OK) {  // the handle stays without one: its pointer says that it is complete
    if (ioff) cudaFreeAsync(ioff, st);
    if (icol) cudaFreeAsync(icol, st);
    return rc;
  }
  g->ioff = ioff;
  g->icol = icol;
  return TKC_OK;
}

// The in-arc CSR, built the first time a step needs it (a graph loaded only
// to join a multi-graph launch never does: the union builds its own).
int ensure_in_csr(const tkc_graph *g) {
  if (g->ioff || g->n == 0) return TKC_OK;
  return build_in_csr(g);
}

// ------------------------------------------------------------------ stable LSD radix sort (8-bit digits)

static constexpr int kRsTPB = 256;
static constexpr int kRsWarps = kRsTPB / 32;
// Elements per lane.  A pass is a chain of as many digit ranks per warp, so up
// to kRsFew tiles of 4 the tiles are that short (65 536 pairs with tiles of 16
// kept 16 blocks busy: 18 us a pass with its scan, 9 us now).  Up to kRsFew tiles of either length
// every block adds up the tiles' digit counts itself (k_rs_scatter, kOwnScan)
// and the scan between the two launches of a pass is left out.
static constexpr int kRsShort = 4, kRsLong = 16;
static constexpr u32 kRsFew = 128;

// Digit counts of the tiles: hist[digit * ntiles + tile], with kOwnScan
// hist[tile * 256 + digit].
template <int kRounds, bool kOwnScan>
__global__ void k_rs_count(const u32 *__restrict__ key, u32 n, int shift, u32 *__restrict__ hist, u32 ntiles) {
  __shared__ u32 cnt[256];
  cnt[threadIdx.x] = 0;
  __syncthreads();
#pragma unroll 4
  for (int r = 0; r < kRounds; ++r) {
    const u64 i = (u64)blockIdx.x * (kRsTPB * kRounds) + r * kRsTPB + threadIdx.x;
    if (i < n) atomicAdd(&cnt[(key[i] >> shift) & 255u], 1u);
  }
  __syncthreads();
  hist[kOwnScan ? blockIdx.x * 256 + threadIdx.x : threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];
}

// Rank of this lane's element among its warp's so far with the same digit d
// (256: no element); counts: the warp's running counts per digit.
__device__ __forceinline__ u32 warp_rank(u32 d, u32 *counts, int lane) {
  const unsigned peers = __match_any_sync(FULL, d);
  u32 r = 0;
  if (d < 256u) r = counts[d] + __popc(peers & ((1u << lane) - 1u));
  __syncwarp();
  if (d < 256u && __ffs(peers) - 1 == lane) counts[d] += __popc(peers);
  __syncwarp();
  return r;
}

// Stable scatter: a warp ranks its 512 consecutive elements in order, the
// warps' counts per digit are summed in warp order, and hist (scanned) holds
// where each tile's elements of a digit start.  Eight bits a pass: half the
// passes, and so half the traffic and launches, of four bits.
template <int kRounds, bool kOwnScan>
__global__ void __launch_bounds__(kRsTPB) k_rs_scatter(const u32 *__restrict__ key, const u32 *__restrict__ val,
                                                       u32 *__restrict__ key_out, u32 *__restrict__ val_out, u32 n,
                                                       int shift, const u32 *__restrict__ hist, u32 ntiles) {
  __shared__ u32 cnt[kRsWarps][256];
  __shared__ u32 s_digits[kRsWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kRsWarps * 256; i += kRsTPB) (&cnt[0][0])[i] = 0;
  __syncthreads();
  const u64 base = (u64)blockIdx.x * (kRsTPB * kRounds) + wid * (32 * kRounds) + lane;
  u32 k[kRounds], rank[kRounds];
#pragma unroll
  for (int r = 0; r < kRounds; ++r) k[r] = base + 32 * r < n ? key[base + 32 * r] : 0u;
#pragma unroll
  for (int r = 0; r < kRounds; ++r)
    rank[r] = warp_rank(base + 32 * r < n ? (k[r] >> shift) & 255u : 256u, cnt[wid], lane);
  __syncthreads();
  u32 at;  // where this tile's elements of digit threadIdx.x start
  if (kOwnScan) {
    static_assert(kRsTPB == 256, "a thread per digit");
    u32 before = 0, total = 0;
#pragma unroll 8
    for (u32 t = 0; t < ntiles; ++t) {
      const u32 c = hist[t * 256 + threadIdx.x];
      if (t < blockIdx.x) before += c;
      total += c;
    }
    u32 incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u32 t = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) s_digits[wid] = incl;
    __syncthreads();
    at = incl - total + before;
    for (int w = 0; w < wid; ++w) at += s_digits[w];
  } else {
    at = hist[threadIdx.x * ntiles + blockIdx.x];
  }
#pragma unroll
  for (int w = 0; w < kRsWarps; ++w) {
    const u32 t = cnt[w][threadIdx.x];
    cnt[w][threadIdx.x] = at;
    at += t;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    if (base + 32 * r >= n) break;
    const u32 pos = cnt[wid][(k[r] >> shift) & 255u] + rank[r];
    key_out[pos] = k[r];
    val_out[pos] = val[base + 32 * r];
  }
}

// All passes of a short sort in one block: keys and values stay in shared
// memory (a launch and two more for its scan, per pass, cost more than the work).
static constexpr int kRsOneTPB = 1024;
static constexpr int kRsOneRounds = 8;
static constexpr u32 kRsOneMax = kRsOneTPB * kRsOneRounds;
static constexpr size_t kRsOneSmem = (2 * (size_t)kRsOneMax + 32 * 256 + 33) * sizeof(u32);
__global__ void __launch_bounds__(kRsOneTPB) k_rs_one(u32 *key, u32 *val, u32 n, int passes) {
  extern __shared__ u32 sm[];
  u32 *sk = sm, *sv = sk + kRsOneMax, *cnt = sv + kRsOneMax, *s_warp = cnt + 32 * 256;  // cnt[warp][digit]
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (u32 i = threadIdx.x; i < n; i += kRsOneTPB) {
    sk[i] = key[i];
    sv[i] = val[i];
  }
  const u32 base = wid * (32 * kRsOneRounds) + lane;
  for (int ps = 0; ps < passes; ++ps) {
    const int shift = 8 * ps;
    for (int i = threadIdx.x; i < 32 * 256; i += kRsOneTPB) cnt[i] = 0;
    __syncthreads();
    u32 k[kRsOneRounds], v[kRsOneRounds], rank[kRsOneRounds];
#pragma unroll
    for (int r = 0; r < kRsOneRounds; ++r) {
      const bool valid = base + 32 * r < n;
      k[r] = valid ? sk[base + 32 * r] : 0u;
      v[r] = valid ? sv[base + 32 * r] : 0u;
    }
#pragma unroll
    for (int r = 0; r < kRsOneRounds; ++r)
      rank[r] = warp_rank(base + 32 * r < n ? (k[r] >> shift) & 255u : 256u, cnt + 256 * wid, lane);
    __syncthreads();
    // starts: digits in order, each digit's warps in order; a thread takes 8
    // warps of one digit
    const u32 d = threadIdx.x >> 2, w0 = (threadIdx.x & 3) * 8;
    u32 sum = 0;
    for (int w = 0; w < 8; ++w) sum += cnt[256 * (w0 + w) + d];
    u32 total;
    u32 at = block_exscan_1024(sum, s_warp, &total);
    for (int w = 0; w < 8; ++w) {
      const u32 t = cnt[256 * (w0 + w) + d];
      cnt[256 * (w0 + w) + d] = at;
      at += t;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRsOneRounds; ++r) {
      if (base + 32 * r >= n) break;
      const u32 pos = cnt[256 * wid + ((k[r] >> shift) & 255u)] + rank[r];
      sk[pos] = k[r];
      sv[pos] = v[r];
    }
    __syncthreads();
  }
  for (u32 i = threadIdx.x; i < n; i += kRsOneTPB) {
    key[i] = sk[i];
    val[i] = sv[i];
  }
}

// Sorts (key, val) by key ascending, keeping the input order of equal keys.
// Only the low `bits` bits of the keys are looked at (rounded up to whole
// digits: keys have no bits above).  Result lands in key/val.
static int radix_sort_pairs(u32 *key, u32 *val, u32 n, int bits, cudaStream_t st) {
  if (n <= 1 || bits <= 0) return TKC_OK;
  const int passes = (bits + 7) / 8;
  if (n <= kRsOneMax) {
    TKC_TRY(cudaFuncSetAttribute(k_rs_one, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRsOneSmem));
    TKC_LAUNCH(k_rs_one<<<1, kRsOneTPB, kRsOneSmem, st>>>(key, val, n, passes));
    TKC_TRY(cudaGetLastError());
    return TKC_OK;
  }
  const int rounds = n <= kRsFew * kRsTPB * kRsShort ? kRsShort : kRsLong;
  const u32 ntiles = (n + kRsTPB * rounds - 1) / (kRsTPB * rounds);
  const bool own = ntiles <= kRsFew;
  u32 *k2 = nullptr, *v2 = nullptr, *hist = nullptr, *tmp = nullptr;
  size_t hlen = (size_t)256 * ntiles;
  TKC_TRY(dev_malloc(&k2, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&v2, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&hist, hlen * sizeof(u32), st));
  TKC_TRY(dev_malloc(&tmp, (hlen / kScanTile + 2) * sizeof(u32), st));
  u32 *ka = key, *va = val, *kb = k2, *vb = v2;
  for (int ps = 0; ps < passes; ++ps) {
    if (rounds == kRsShort) {
      TKC_LAUNCH(k_rs_count<kRsShort, true><<<ntiles, kRsTPB, 0, st>>>(ka, n, 8 * ps, hist, ntiles));
      TKC_LAUNCH(k_rs_scatter<kRsShort, true><<<ntiles, kRsTPB, 0, st>>>(ka, va, kb, vb, n, 8 * ps, hist, ntiles));
    } else if (own) {
      TKC_LAUNCH(k_rs_count<kRsLong, true><<<ntiles, kRsTPB, 0, st>>>(ka, n, 8 * ps, hist, ntiles));
      TKC_LAUNCH(k_rs_scatter<kRsLong, true><<<ntiles, kRsTPB, 0, st>>>(ka, va, kb, vb, n, 8 * ps, hist, ntiles));
    } else {
      TKC_LAUNCH(k_rs_count<kRsLong, false><<<ntiles, kRsTPB, 0, st>>>(ka, n, 8 * ps, hist, ntiles));
      TKC_RC(scan_exclusive(hist, hist, hlen, tmp, st));
      TKC_LAUNCH(k_rs_scatter<kRsLong, false><<<ntiles, kRsTPB, 0, st>>>(ka, va, kb, vb, n, 8 * ps, hist, ntiles));
    }
    TKC_TRY(cudaGetLastError());
    std::swap(ka, kb);
    std::swap(va, vb);
  }
  if (ka != key) {
    TKC_TRY(cudaMemcpyAsync(key, ka, (size_t)n * sizeof(u32), cudaMemcpyDeviceToDevice, st));
    TKC_TRY(cudaMemcpyAsync(val, va, (size_t)n * sizeof(u32), cudaMemcpyDeviceToDevice, st));
  }
  TKC_TRY(cudaFreeAsync(k2, st));
  TKC_TRY(cudaFreeAsync(v2, st));
  TKC_TRY(cudaFreeAsync(hist, st));
  TKC_TRY(cudaFreeAsync(tmp, st));
  return TKC_OK;
}

int scan_exclusive_u32(const u32 *in, u32 *out, u64 len, u32 *tmp, cudaStream_t st) {
  return scan_exclusive(in, out, len, tmp, st);
}

int radix_sort_u32_pairs(u32 *key, u32 *val, u32 n, int bits, cudaStream_t st) {
  return radix_sort_pairs(key, val, n, bits, st);
}

// ------------------------------------------------------------------ computeBoundsDeg

__global__ void k_maxdeg(const u32 *off, u32 n, u32 *maxd, u32 *nzero) {
  u32 m = 0, z = 0;
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    u32 d = off[v + 1] - off[v];
    m = max(m, d);
    z += d == 0;
  }
  m = __reduce_max_sync(FULL, m);
  z = __reduce_add_sync(FULL, z);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(maxd, m);
    atomicAdd(nzero, z);
  }
}

__global__ void k_deg_keys(const u32 *off, u32 n, u32 maxd, u32 *key, u32 *val) {
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    key[v] = maxd - (off[v + 1] - off[v]);  // larger degree -> smaller key
    val[v] = v;                              // ids ascending: the sort is stable
  }
}

int ensure_degree_order(tkc_graph *g) {
  if (g->have_order) return TKC_OK;
  cudaStream_t st = g->ctx->stream;
  const u32 n = g->n;
  if (n == 0) {
    g->have_order = true;
    return TKC_OK;
  }
  u32 *keys = nullptr, *stats = nullptr;
  if (!g->deg_order) TKC_TRY(dev_malloc(&g->deg_order, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&keys, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&stats, 2 * sizeof(u32), st));
  TKC_TRY(cudaMemsetAsync(stats, 0, 2 * sizeof(u32), st));
  TKC_LAUNCH(k_maxdeg<<<grid_for(n, 256), 256, 0, st>>>(g->off, n, stats, stats + 1));
  TKC_TRY(cudaGetLastError());
  u32 hs[2];
  TKC_TRY(read_back(hs, stats, sizeof(hs), st));
  TKC_LAUNCH(k_deg_keys<<<grid_for(n, 256), 256, 0, st>>>(g->off, n, hs[0], keys, g->deg_order));
  TKC_TRY(cudaGetLastError());
  int bits = 0;
  while (bits < 32 && (hs[0] >> bits) != 0) ++bits;
  TKC_RC(radix_sort_pairs(keys, g->deg_order, n, bits, st));
  TKC_TRY(cudaFreeAsync(keys, st));
  TKC_TRY(cudaFreeAsync(stats, st));
  g->n_src_deg = n - hs[1];
  g->have_order = true;
  return TKC_OK;
}

// ------------------------------------------------------------------ vertices of out-degree 0

__global__ void k_zero_flag(const u32 *off, u32 n, u32 *flag) {
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v <= n; v += gridDim.x * blockDim.x)
    flag[v] = v < n && off[v + 1] == off[v];
}

__global__ void k_zero_out(const u32 *off, const u32 *pos, u32 n, u32 *out, u32 *cnt) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *cnt = pos[n];
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    if (off[v + 1] == off[v]) out[pos[v]] = v;
}

// The vertices of out-degree 0 in id order (closeness 0: they end a list
// that fewer than k vertices with reach above 1 fill), by one compaction;
// the degree order's tail holds the same, but needs a sort.
int ensure_zero_list(const tkc_graph *g) {
  if (g->have_zero) return TKC_OK;
  cudaStream_t st = g->ctx->stream;
  const u32 n = g->n;
  if (n == 0) {
    g->have_zero = true;
    return TKC_OK;
  }
  u32 *flag = nullptr, *tmp = nullptr;
  TKC_TRY(dev_malloc(&flag, ((size_t)n + 1) * sizeof(u32), st));
  TKC_TRY(dev_malloc(&tmp, (((size_t)n + 1) / kScanTile + 2) * sizeof(u32), st));
  if (!g->zero_ids) TKC_TRY(dev_malloc(&g->zero_ids, (size_t)n * sizeof(u32), st));
  TKC_LAUNCH(k_zero_flag<<<grid_for((u64)n + 1, 256), 256, 0, st>>>(g->off, n, flag));
  TKC_RC(scan_exclusive(flag, flag, (u64)n + 1, tmp, st));
  if (!g->n_zero) TKC_TRY(dev_malloc(&g->n_zero, sizeof(u32), st));
  TKC_LAUNCH(k_zero_out<<<grid_for(n, 256), 256, 0, st>>>(g->off, flag, n, g->zero_ids, g->n_zero));
  TKC_TRY(cudaGetLastError());
  TKC_TRY(cudaFreeAsync(flag, st));
  TKC_TRY(cudaFreeAsync(tmp, st));
  g->have_zero = true;
  return TKC_OK;
}

// ------------------------------------------------------------------ out-neighbours by in-degree class

// Class of a vertex by its in-degree: 1, 2, 3 to 4, more.  (R-MAT 20: of
// 546 331 sources 6 208 are left by the bound with one class, 211 with the
// in-degrees 1 and more apart, 21 with 1, 2 and more apart, and no fewer with
// up to 33 classes; Barabasi-Albert and Erdos-Renyi graphs: no difference.)
constexpr u32 kClasses = 4;
__device__ __forceinline__ u32 in_class(u32 indeg) { return indeg <= 1 ? 0u : indeg == 2 ? 1u : indeg <= 4 ? 2u : 3u; }

// cls[v] = v's class; n_cls[4 g + c] = vertices of graph g in class c with an in-arc.
__global__ void k_classes(const u32 *__restrict__ ioff, u32 n, const u32 *__restrict__ gid, uint8_t *__restrict__ cls,
                          u32 *__restrict__ n_cls) {
  const int lane = threadIdx.x & 31;
  for (u32 base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; base < n; base += gridDim.x * blockDim.x) {
    const u32 v = base + lane;
    u32 d = 0, c = 0;
    if (v < n) {
      d = ioff[v + 1] - ioff[v];
      c = in_class(d);
      cls[v] = (uint8_t)c;
    }
    const u32 key = d ? kClasses * (gid ? gid[v] : 0u) + c : 0xffffffffu;
    const unsigned peers = __match_any_sync(FULL, key);
    if (d && __ffs(peers) - 1 == lane) atomicAdd(&n_cls[key], (u32)__popc(peers));
  }
}

// cnt[u].{x,y,z,w} += u's out-neighbours of class 0..3: 32 consecutive arcs per
// warp step (a hub's row spread over many warps), the lanes of one source
// added up first, four counts in one word (each at most 32).
__global__ void k_class_counts(const u32 *__restrict__ off, const u32 *__restrict__ col, u32 n, u64 arcs,
                               const uint8_t *__restrict__ cls, uint4 *__restrict__ cnt) {
  const int lane = threadIdx.x & 31;
  grid_walk_arcs(off, n, arcs, [&](u32 u, u64 i, bool valid, u32) {
    const u32 one = valid ? 1u << (8 * cls[col[i]]) : 0u;
    const unsigned peers = __match_any_sync(FULL, valid ? u : 0xffffffffu);
    const u32 s = __reduce_add_sync(peers, one);
    if (valid && __ffs(peers) - 1 == lane) {
      u32 *c = reinterpret_cast<u32 *>(cnt + u);
#pragma unroll
      for (int j = 0; j < (int)kClasses; ++j)
        if ((s >> (8 * j)) & 0xffu) atomicAdd(c + j, (s >> (8 * j)) & 0xffu);
    }
  });
}

// The out-neighbours of every vertex by in-degree class and the class sizes
// (gid/ng: per graph of a union); the in-arc CSR exists.  They bound a
// source's level 2 before it searches: at most min(n_c, sum of the class-c
// counts of its out-neighbours) of the vertices of class c lie there (walks of
// length 2 that end in class c reach each at least once).
int ensure_classes(const tkc_graph *g, const u32 *gid, u32 ng) {
  if (g->cls || g->n == 0) return TKC_OK;
  cudaStream_t st = g->ctx->stream;
  const size_t n = g->n;
  uint8_t *cls = nullptr;
  TKC_TRY(dev_malloc(&cls, n, st));
  if (!g->n_cls) TKC_TRY(dev_malloc(&g->n_cls, (size_t)kClasses * ng * sizeof(u32), st));
  TKC_TRY(dev_malloc(&g->cls, n * sizeof(uint4), st));
  TKC_TRY(cudaMemsetAsync(g->n_cls, 0, (size_t)kClasses * ng * sizeof(u32), st));
  TKC_TRY(cudaMemsetAsync(g->cls, 0, n * sizeof(uint4), st));
  TKC_LAUNCH(k_classes<<<grid_for(n, 256), 256, 0, st>>>(g->ioff, g->n, gid, cls, g->n_cls));
  if (g->arcs)
    TKC_LAUNCH(k_class_counts<<<grid_for(arc_threads(g->arcs), 256), 256, 0, st>>>(
        g->off, g->col, g->n, g->arcs, cls, g->cls));
  TKC_TRY(cudaGetLastError());
  TKC_TRY(cudaFreeAsync(cls, st));
  return TKC_OK;
}

// ------------------------------------------------------------------ bottom-up work order

__global__ void k_bu_keys(const u32 *ioff, u32 n, u32 heavy_in, u32 *key, u32 *val, u32 *count) {
  u32 any = 0, heavy = 0;
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const u32 indeg = ioff[v + 1] - ioff[v];
    // rows walked by a whole warp: by bit length of the in-degree, longest
    // first; then the other vertices with an in-arc; none last
    key[v] = indeg > heavy_in ? (u32)__clz(indeg) : indeg ? 32u : 33u;
    val[v] = v;  // ids ascending: the sort is stable
    any += indeg != 0;
    heavy += indeg > heavy_in;
  }
  for (int o = 16; o > 0; o >>= 1) {
    any += __shfl_down_sync(0xffffffffu, any, o);
    heavy += __shfl_down_sync(0xffffffffu, heavy, o);
  }
  if ((threadIdx.x & 31) == 0 && any) atomicAdd(&count[0], any);
  if ((threadIdx.x & 31) == 0 && heavy) atomicAdd(&count[1], heavy);
}

// The same for a union, graph by graph (keys (graph, class)); g_cnt receives
// each graph's vertices with an in-arc and with a long row.
__global__ void k_bu_keys_many(const u32 *ioff, u32 n, u32 heavy_in, const u32 *gid, u32 *key, u32 *val, u32 *g_cnt) {
  const int lane = threadIdx.x & 31;
  for (u32 base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; base < n; base += gridDim.x * blockDim.x) {
    const u32 v = base + lane;
    u32 indeg = 0, g = 0xffffffffu;
    if (v < n) {
      g = gid[v];
      indeg = ioff[v + 1] - ioff[v];
      key[v] = 64 * g + (indeg > heavy_in ? (u32)__clz(indeg) : indeg ? 32u : 33u);
      val[v] = v;
    }
    // the warp's lanes of one graph add up first
    const unsigned peers = __match_any_sync(FULL, g);
    const unsigned any = __ballot_sync(FULL, indeg != 0) & peers, heavy = __ballot_sync(FULL, indeg > heavy_in) & peers;
    if (v < n && __ffs(peers) - 1 == lane) {
      if (any) atomicAdd(&g_cnt[2 * (size_t)g], (u32)__popc(any));
      if (heavy) atomicAdd(&g_cnt[2 * (size_t)g + 1], (u32)__popc(heavy));
    }
  }
}

// The vertices that bottom-up levels sweep, for the in-arc CSR `ioff`: those
// with an in-arc (no other vertex can be discovered bottom-up; a source is
// seeded directly).  First the n_heavy vertices of more than heavy_in in-arcs,
// whose rows a whole warp walks, longest rows first (bit length of the
// in-degree, then id); then the others by id, so that a warp's 32 entries
// share a few frontier-bitmap words.  Only the order of work depends on it,
// not any result.  *list is allocated here; cnt (device, 2 words) receives
// the number of vertices with an in-arc and of long rows.
// A union (gid, ng graphs): the list graph by graph, every graph's vertices
// from its first id's position on; g_cnt (device, 2 words per graph) receives
// the counts instead.
static int build_bu_list(const u32 *ioff, u32 n, u32 heavy_in, cudaStream_t st, u32 **list, u32 *cnt,
                         const u32 *gid = nullptr, u32 ng = 0, u32 *g_cnt = nullptr) {
  u32 *keys = nullptr, *ids = nullptr;
  TKC_TRY(dev_malloc(&ids, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&keys, (size_t)n * sizeof(u32), st));
  TKC_TRY(cudaMemsetAsync(cnt, 0, 2 * sizeof(u32), st));
  int bits = 6;
  if (gid) {
    TKC_TRY(cudaMemsetAsync(g_cnt, 0, 2 * (size_t)ng * sizeof(u32), st));
    TKC_LAUNCH(k_bu_keys_many<<<grid_for(n, 256), 256, 0, st>>>(ioff, n, heavy_in, gid, keys, ids, g_cnt));
    while ((ng - 1) >> (bits - 6)) ++bits;
  } else {
    TKC_LAUNCH(k_bu_keys<<<grid_for(n, 256), 256, 0, st>>>(ioff, n, heavy_in, keys, ids, cnt));
  }
  TKC_TRY(cudaGetLastError());
  TKC_RC(radix_sort_pairs(keys, ids, n, bits, st));
  TKC_TRY(cudaFreeAsync(keys, st));
  *list = ids;
  return TKC_OK;
}

// ------------------------------------------------------------------ the search kernel's copy of the graph

// Relabelling key: in-degree, larger first (top is at least every in-degree;
// the stable sort keeps ids ascending among equal in-degrees).
__global__ void k_relabel_keys(const u32 *ioff, u32 n, u32 top, u32 *key, u32 *val) {
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    key[v] = top - (ioff[v + 1] - ioff[v]);
    val[v] = v;
  }
}

// lab = the inverse of unlab; out_len[i] and in_len[i] = out- and in-degree
// of vertex unlab[i] (in_len may be null).
__global__ void k_relabel_rows(const u32 *unlab, const u32 *off, const u32 *ioff, u32 n, u32 *lab, u32 *out_len,
                               u32 *in_len) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const u32 v = unlab[i];
    lab[v] = i;
    out_len[i] = off[v + 1] - off[v];
    if (in_len) in_len[i] = ioff[v + 1] - ioff[v];
  }
}

// Row i of the relabelled out-CSR: the out-row of vertex unlab[i], each target
// replaced by its label.  Arcs are dealt to warps in fixed ranges.
__global__ void k_relabel_cols(const u32 *__restrict__ s_off, const u32 *__restrict__ unlab,
                               const u32 *__restrict__ off, const u32 *__restrict__ col,
                               const u32 *__restrict__ lab, u32 n, u64 arcs, u32 *__restrict__ s_col) {
  grid_walk_arcs<true>(s_off, n, arcs, [&](u32 i, u64 a, bool valid, u32 rs) {
    if (valid) s_col[a] = lab[col[off[unlab[i]] + (u32)(a - rs)]];
  });
}

void free_search_csr(const tkc_graph *g) {
  cudaStream_t st = g->ctx->stream;  // stream-ordered: after the work that used them
  if (g->s_ready) {  // a copy still being built on the helper stream
    cudaStreamWaitEvent(st, g->s_ready, 0);
    cudaEventDestroy(g->s_ready);
    g->s_ready = nullptr;
  }
  if (g->s_ioff && g->s_ioff != g->s_off) cudaFreeAsync(g->s_ioff, st);
  if (g->s_icol && g->s_icol != g->s_col) cudaFreeAsync(g->s_icol, st);
  void *ptrs[] = {g->s_off, g->s_col, g->s_lab, g->s_unlab, g->bu_list, g->s_cnt, g->g_bu};
  for (void *q : ptrs)
    if (q) cudaFreeAsync(q, st);
  g->g_bu = nullptr;
  g->s_off = g->s_col = g->s_ioff = g->s_icol = g->s_lab = g->s_unlab = g->s_cnt = nullptr;
  g->bu_list = nullptr;
  g->s_mode = -1;
}

// The graph as the search kernel walks it (ensure_search_csr below).  Plain: the graph itself.
// Relabelled: vertex i of the copy is vertex unlab[i] of the graph, the
// vertices taken by in-degree, largest first.  Bottom-up levels gather the
// frontier rows of in-neighbours, and in-neighbours are mostly vertices of
// large degree; with those first, the rows and frontier bits that levels
// touch most sit together in a few megabytes that stay in L2 (R-MAT 22,
// NBCut: search kernel 51 -> 35 ms).  The copy's in-rows come out in
// ascending label order, largest in-degree first, so that a walk meets the
// likely frontier vertices early.  An undirected graph's copy serves both
// directions (its transpose is itself).  Every result is the same: sources,
// slots, ties and outputs keep the graph's own ids; only the search's rows
// are indexed by labels.
// The labelled copy and its bottom-up list, enqueued on `st` without a host
// wait (the list's counts stay in g->s_cnt, where the search reads them).  The graph's in-arc CSR exists.
static int build_labelled_copy(const tkc_graph *g, cudaStream_t st) {
  const u32 n = g->n;
  u32 *keys = nullptr, *gcol = nullptr, *tmp = nullptr;
  TKC_TRY(dev_malloc(&g->s_cnt, 2 * sizeof(u32), st));
  TKC_TRY(dev_malloc(&g->s_unlab, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&g->s_lab, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&g->s_off, ((size_t)n + 1) * sizeof(u32), st));
  TKC_TRY(dev_malloc(&g->s_ioff, ((size_t)n + 1) * sizeof(u32), st));
  TKC_TRY(dev_malloc(&g->s_icol, std::max<size_t>(g->arcs, 1) * sizeof(u32), st));
  TKC_TRY(dev_malloc(&gcol, std::max<size_t>(g->arcs, 1) * sizeof(u32), st));
  TKC_TRY(dev_malloc(&keys, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&tmp, (((size_t)n + 1) / kScanTile + 2) * sizeof(u32), st));
  // key n - indegree (in [1, n]: no vertex has n in-arcs), ascending
  TKC_LAUNCH(k_relabel_keys<<<grid_for(n, 256), 256, 0, st>>>(g->ioff, n, n, keys, g->s_unlab));
  TKC_TRY(cudaGetLastError());
  int bits = 0;
  while (bits < 32 && (n >> bits) != 0) ++bits;
  TKC_RC(radix_sort_pairs(keys, g->s_unlab, n, bits, st));
  // the copy's row lengths are the graph's degrees in label order: its
  // in-rows need no counting pass
  TKC_TRY(cudaMemsetAsync(g->s_off + n, 0, sizeof(u32), st));
  TKC_TRY(cudaMemsetAsync(g->s_ioff + n, 0, sizeof(u32), st));
  TKC_LAUNCH(k_relabel_rows<<<grid_for(n, 256), 256, 0, st>>>(g->s_unlab, g->off, g->ioff, n, g->s_lab, g->s_off,
                                                              g->s_ioff));
  TKC_TRY(cudaGetLastError());
  TKC_RC(scan_exclusive(g->s_off, g->s_off, (u64)n + 1, tmp, st));
  TKC_RC(scan_exclusive(g->s_ioff, g->s_ioff, (u64)n + 1, tmp, st));
  if (g->arcs) {
    TKC_LAUNCH(k_relabel_cols<<<grid_for(arc_threads(g->arcs), 256), 256, 0, st>>>(
        g->s_off, g->s_unlab, g->off, g->col, g->s_lab, n, g->arcs, gcol));
    TKC_TRY(cudaGetLastError());
  }
  // in-rows by transposition, so that each runs in ascending label order
  TKC_RC(fill_in_arcs(g->s_off, gcol, n, g->arcs, g->s_ioff, g->s_icol, st));
  if (g->directed) {
    g->s_col = gcol;
  } else {
    TKC_TRY(cudaFreeAsync(g->s_off, st));
    TKC_TRY(cudaFreeAsync(gcol, st));
    g->s_off = g->s_ioff;
    g->s_col = g->s_icol;
  }
  TKC_TRY(cudaFreeAsync(keys, st));
  TKC_TRY(cudaFreeAsync(tmp, st));
  g->heavy_in = kHeavyInLabelled;
  return build_bu_list(g->s_ioff, n, g->heavy_in, st, &g->bu_list, g->s_cnt);
}

// A copy started on the helper stream: the context's stream waits for it.
static int finish_started_copy(const tkc_graph *g) {
  if (!g->s_ready) return TKC_OK;
  TKC_TRY(cudaStreamWaitEvent(g->ctx->stream, g->s_ready, 0));
  TKC_TRY(cudaEventDestroy(g->s_ready));
  g->s_ready = nullptr;
  return TKC_OK;
}

int ensure_search_csr(const tkc_graph *g, bool relabel, const u32 *gid, u32 ng) {
  TKC_RC(finish_started_copy(g));
  const int want = relabel ? 1 : 0;
  if (g->s_mode == want || g->n == 0) return TKC_OK;
  TKC_RC(ensure_in_csr(g));
  free_search_csr(g);  // the other labelling's copy, or what a failed build left
  cudaStream_t st = g->ctx->stream;
  if (!relabel) {
    g->heavy_in = kHeavyIn;
    TKC_TRY(dev_malloc(&g->s_cnt, 2 * sizeof(u32), st));
    // (a graph number takes 26 bits of a key beside the class's 6)
    const bool many = gid && ng > 1 && ng <= (1u << 26);
    if (many) TKC_TRY(dev_malloc(&g->g_bu, 2 * (size_t)ng * sizeof(u32), st));
    TKC_RC(build_bu_list(g->ioff, g->n, g->heavy_in, st, &g->bu_list, g->s_cnt, many ? gid : nullptr, ng, g->g_bu));
  } else {
    TKC_RC(build_labelled_copy(g, st));
  }
  g->s_mode = want;
  return TKC_OK;
}

// Starts the labelled copy on the context's helper stream, so that it is
// built while the context's stream runs the preprocessing (degree order,
// reach bounds, NB bounds) with its host waits: it needs only the CSR and
// the in-arc CSR.  ensure_search_csr completes it.
int start_search_csr(const tkc_graph *g) {
  if (g->s_mode == 1 || g->s_ready || g->n == 0) return TKC_OK;
  TKC_RC(ensure_in_csr(g));
  free_search_csr(g);
  tkc_ctx *ctx = g->ctx;
  if (!ctx->aux) {
    TKC_TRY(cudaStreamCreateWithFlags(&ctx->aux, cudaStreamNonBlocking));
    TKC_TRY(cudaEventCreateWithFlags(&ctx->aux_in, cudaEventDisableTiming));
  }
  TKC_TRY(cudaEventRecord(ctx->aux_in, ctx->stream));
  TKC_TRY(cudaStreamWaitEvent(ctx->aux, ctx->aux_in, 0));
  cudaEvent_t ready = nullptr;
  TKC_TRY(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
  const int rc = build_labelled_copy(g, ctx->aux);
  cudaError_t e = rc == TKC_OK ? cudaEventRecord(ready, ctx->aux) : cudaSuccess;
  if (rc != TKC_OK || e != cudaSuccess) {
    cudaEventDestroy(ready);
    cudaStreamSynchronize(ctx->aux);  // what was begun is freed on the other stream
    TKC_TRY(e);
    return rc;
  }
  g->s_ready = ready;
  g->s_mode = 1;
  return TKC_OK;
}

// Keeps the vertices of out-degree >= 1 of a full order, in order.
__global__ void k_flag_src(const u32 *order, const u32 *off, u32 n, u32 *flag) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    u32 v = order[i];
    flag[i] = off[v + 1] > off[v];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) flag[n] = 0;
}

__global__ void k_compact(const u32 *order, const u32 *pos, u32 n, u32 *out) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    if (pos[i + 1] != pos[i]) out[pos[i]] = order[i];
}

int filter_order(tkc_graph *g, const u32 *d_order_all, u32 *d_out, u32 *count) {
  cudaStream_t st = g->ctx->stream;
  const u32 n = g->n;
  u32 *pos = nullptr, *tmp = nullptr;
  TKC_TRY(dev_malloc(&pos, ((size_t)n + 1) * sizeof(u32), st));
  TKC_TRY(dev_malloc(&tmp, (((size_t)n + 1) / kScanTile + 2) * sizeof(u32), st));
  TKC_LAUNCH(k_flag_src<<<grid_for(n, 256), 256, 0, st>>>(d_order_all, g->off, n, pos));
  TKC_RC(scan_exclusive(pos, pos, (u64)n + 1, tmp, st));
  TKC_LAUNCH(k_compact<<<grid_for(n, 256), 256, 0, st>>>(d_order_all, pos, n, d_out));
  TKC_TRY(cudaGetLastError());
  TKC_TRY(read_back(count, pos + n, sizeof(u32), st));
  TKC_TRY(cudaFreeAsync(pos, st));
  TKC_TRY(cudaFreeAsync(tmp, st));
  return TKC_OK;
}

// ------------------------------------------------------------------ reach: undirected components

__device__ __forceinline__ u32 cc_root(const u32 *parent, u32 x) {
  u32 p = parent[x];
  while (p != x) {
    x = p;
    p = parent[x];
  }
  return x;
}

// Components, one cooperative launch: hooks the larger root of every edge's
// endpoints under the smaller one, then points every vertex at its root, until
// no edge joins two roots.  parent[x] <= x always holds, so pointers only
// decrease and no cycle forms.  The arcs are dealt in chunks (tkc_arcs.cuh):
// a warp per vertex left most lanes idle on rows of ten arcs.
// changed: two zero words, used in turn.
constexpr int kCcTPB = 256;
__global__ void __launch_bounds__(kCcTPB) k_cc(const u32 *__restrict__ off, const u32 *__restrict__ col, u32 n,
                                               u64 arcs, u32 *parent, u32 *changed, GridBar *bar, u64 timeout) {
  const int lane = threadIdx.x & 31;
  const u32 first = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  for (u32 v = first; v < n; v += step) parent[v] = v;
  if (!grid_sync(bar, timeout, [] {})) return;
  for (u32 round = 0;; ++round) {
    u32 *chg = changed + (round & 1);
    u32 ch = 0;
    grid_walk_arcs(off, n, arcs, [&](u32 u, u64 i, bool valid, u32) {
      if (!valid) return;
      const u32 v = col[i];
      if (v < u) return;
      const u32 pu = parent[u], pv = parent[v];
      if (pu == pv) return;  // roots already equal
      const u32 ru = cc_root(parent, pu), rv = cc_root(parent, pv);
      if (ru != rv) {
        atomicMin(&parent[max(ru, rv)], min(ru, rv));
        ch = 1;
      }
    });
    ch = __reduce_or_sync(FULL, ch);
    if (lane == 0 && ch) *chg = 1;
    if (!grid_sync(bar, timeout, [&] { changed[(round & 1) ^ 1] = 0; })) return;
    if (*(volatile u32 *)chg == 0) return;  // every vertex points at its root since the last round
    for (u32 v = first; v < n; v += step) parent[v] = cc_root(parent, v);
    if (!grid_sync(bar, timeout, [] {})) return;
  }
}

// Component sizes; the lanes of one component add up first (one component
// usually holds the graph: an atomic per vertex on one address took 0.62 ms on
// a million vertices).
__global__ void k_cc_size(const u32 *parent, u32 n, u32 *size) {
  const int lane = threadIdx.x & 31;
  u32 c = 0xffffffffu, cnt = 0;  // the warp's run of vertices of one component
  for (u32 base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; base < n; base += gridDim.x * blockDim.x) {
    const u32 v = base + lane;
    const u32 r = v < n ? parent[v] : 0xffffffffu;
    const u32 r0 = __shfl_sync(FULL, r, 0);
    if (__all_sync(FULL, r == r0)) {
      if (r0 != c) {
        if (lane == 0 && cnt) atomicAdd(&size[c], cnt);
        c = r0;
        cnt = 0;
      }
      cnt += 32;
    } else {
      const unsigned peers = __match_any_sync(FULL, r);
      if (v < n && __ffs(peers) - 1 == lane) atomicAdd(&size[r], (u32)__popc(peers));
    }
  }
  if (lane == 0 && cnt) atomicAdd(&size[c], cnt);
}

__global__ void k_cc_out(const u32 *parent, const u32 *size, u32 n, u32 *alpha, u32 *omega, u32 *scc_size) {
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    u32 s = size[parent[v]];
    alpha[v] = s;
    omega[v] = s;
    scc_size[v] = s;
  }
}

static int reach_undirected(tkc_graph *g) {
  cudaStream_t st = g->ctx->stream;
  const u32 n = g->n;
  u32 *parent = nullptr, *size = nullptr, *changed = nullptr;
  GridBar *bar = nullptr;
  TKC_TRY(dev_malloc(&parent, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&size, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&bar, sizeof(GridBar) + 2 * sizeof(u32), st));
  TKC_TRY(cudaMemsetAsync(bar, 0, sizeof(GridBar) + 2 * sizeof(u32), st));
  changed = reinterpret_cast<u32 *>(bar + 1);
  {
    u64 arcs = g->arcs, timeout = grid_timeout(g->ctx);
    void *args[] = {(void *)&g->off, (void *)&g->col, (void *)&n, (void *)&arcs, (void *)&parent, (void *)&changed,
                    (void *)&bar, (void *)&timeout};
    const int blocks = grid_blocks(g->ctx, k_cc, kCcTPB, std::max<u64>(n, arc_threads(arcs)));
    if (blocks <= 0) return TKC_ECUDA;
    note_launches(1);
    TKC_TRY(cudaLaunchCooperativeKernel((const void *)k_cc, dim3(blocks), dim3(kCcTPB), args, 0, st));
    int err = 0;
    TKC_TRY(read_back(&err, &bar->err, sizeof(int), st));
    if (err) {
      cudaFreeAsync(parent, st);
      cudaFreeAsync(size, st);
      cudaFreeAsync(bar, st);
      return err;
    }
  }
  TKC_TRY(cudaMemsetAsync(size, 0, (size_t)n * sizeof(u32), st));
  TKC_LAUNCH(k_cc_size<<<grid_for(n, 256), 256, 0, st>>>(parent, n, size));
  TKC_LAUNCH(k_cc_out<<<grid_for(n, 256), 256, 0, st>>>(parent, size, n, g->alpha, g->omega, g->scc_size));
  TKC_TRY(cudaGetLastError());
  TKC_TRY(cudaMemcpyAsync(g->comp, parent, (size_t)n * sizeof(u32), cudaMemcpyDeviceToDevice, st));
  TKC_TRY(cudaFreeAsync(parent, st));
  TKC_TRY(cudaFreeAsync(size, st));
  TKC_TRY(cudaFreeAsync(bar, st));
  return TKC_OK;
}

// ------------------------------------------------------------------ reach: directed

// SCCs and Algorithm 6 run on the device (tkc_scc.cu).
int reach_directed_gpu(tkc_graph *g, const u32 *gid, u32 ng);

int ensure_reach_bounds(tkc_graph *g, const u32 *gid, u32 ng) {
  if (g->have_reach) return TKC_OK;
  cudaStream_t st = g->ctx->stream;
  if (g->n == 0) {
    g->have_reach = true;
    return TKC_OK;
  }
  if (!g->alpha) TKC_TRY(dev_malloc(&g->alpha, (size_t)g->n * sizeof(u32), st));
  if (!g->omega) TKC_TRY(dev_malloc(&g->omega, (size_t)g->n * sizeof(u32), st));
  if (!g->scc_size) TKC_TRY(dev_malloc(&g->scc_size, (size_t)g->n * sizeof(u32), st));
  if (!g->comp) TKC_TRY(dev_malloc(&g->comp, (size_t)g->n * sizeof(u32), st));
  TKC_RC(ensure_in_csr(g));
  TKC_RC(g->directed ? reach_directed_gpu(g, gid, ng) : reach_undirected(g));
  g->have_reach = true;
  return TKC_OK;
}

}  // namespace tkc
