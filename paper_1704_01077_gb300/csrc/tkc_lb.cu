// updateBoundsLB (Section 7, Algorithm 5; Eq. 4 for undirected graphs, Eq. 5
// for directed ones): after a complete BFS from s, every vertex w whose reach
// equals s's (its component; its SCC if directed) has
//   S(w) >= L(l(w)) - outdeg(w),
//   L(i) = 2 sum_{|j-i| <= 1} g_j + sum_{|j-i| > 1} g_j |j-i| - 2     (undirected)
//   L(i) = 2 sum_{j-i <= 1} g_j  + sum_{j-i > 1} g_j (j-i) - 2        (directed)
// with g_j the size of level j of the BFS from s (g_0 = 1: s itself).
//
// Algorithm 1 runs in rounds: the B unsearched vertices of smallest bound key
// (ties by their position in the initial order) are searched completely by the
// persistent kernel, which records for every vertex the level at which each
// slot found it and each slot's level sizes; then a warp per source turns its
// level sizes into L(i) (O(depth), prefix sums), and four lanes per vertex
// raise the vertex's bound with every slot that found it.  The host loop ends
// when the head of the order has a key above the k-th farness.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "tkc_internal.cuh"

namespace tkc {

typedef uint32_t u32;
typedef unsigned long long u64;
typedef unsigned __int128 u128;
static constexpr unsigned FULL = 0xffffffffu;
constexpr int kKeyFrac = 46;  // key = floor(S * 2^46 / (r-1)^2), as the NB order keys

int radix_sort_u32_pairs(u32 *key, u32 *val, u32 n, int bits, cudaStream_t st);
int scan_exclusive_u32(const u32 *in, u32 *out, u64 len, u32 *tmp, cudaStream_t st);

namespace {

unsigned grid_of(u64 work, unsigned tpb = 256, unsigned cap = 152 * 16) {
  u64 b = (work + tpb - 1) / tpb;
  return (unsigned)std::max<u64>(1, std::min<u64>(b, cap));
}

// flag[i] = order0[i] is still a candidate (not searched, out-degree >= 1)
__global__ void k_lb_flags(const u32 *order0, u32 n0, const u32 *off, const uint8_t *done, u32 *flag) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n0; i += gridDim.x * blockDim.x) {
    const u32 v = order0[i];
    flag[i] = !done[v] && off[v + 1] > off[v];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) flag[n0] = 0;
}

__global__ void k_lb_compact(const u32 *order0, const u32 *pos, u32 n0, u32 *out) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n0; i += gridDim.x * blockDim.x)
    if (pos[i + 1] != pos[i]) out[pos[i]] = order0[i];
}

__global__ void k_lb_key_lo(u32 m, const u32 *cand, const u64 *key, u32 *lo, u64 *maxkey) {
  u64 mx = 0;
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const u64 kv = key[cand[i]];
    lo[i] = (u32)kv;
    mx = max(mx, kv);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, (u64)__shfl_xor_sync(FULL, mx, o));
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(maxkey, mx);
}

__global__ void k_lb_key_hi(u32 m, const u32 *cand, const u64 *key, u32 *hi) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) hi[i] = (u32)(key[cand[i]] >> 32);
}

// One warp per source: L(i) for every level i of its BFS, from the level sizes
// g_j (non-zero up to the depth D, zero beyond; g_0 = 1) with prefix sums
// G(j) = sum_{t<=j} g_t, M(j) = sum_{t<=j} t g_t:
//   sum_{j <= i-2} g_j (i-j)  = i G(i-2) - M(i-2)
//   sum_{j >= i+2} g_j (j-i)  = (M_all - M(i+1)) - i (G_all - G(i+1))
// 32 levels a step; the level sizes are zeroed again behind it, so that the
// next round finds them so.  (A thread per source behind a pass over all
// levels a search could have, and a memset of them: 0.27 ms a round on a
// 301 x 299 grid.)
__global__ void k_lb_table(u32 nsrc, u32 *hist, u32 cap, int directed, u64 *Ltab) {
  const int lane = threadIdx.x & 31;
  const u32 s = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (s >= nsrc) return;
  u32 *g = hist + (size_t)s * cap;
  u64 *L = Ltab + (size_t)s * cap;
  // the depth and the totals
  u32 D = 0;
  u64 Gall = 0, Mall = 0;
  for (u32 base = 0;; base += 32) {
    const u32 j = base + lane;
    const u32 c = j == 0 ? 1u : j < cap ? g[j] : 0u;
    const unsigned empty = __ballot_sync(FULL, c == 0);
    const int used = empty ? __ffs(empty) - 1 : 32;
    if (lane < used) {
      Gall += c;
      Mall += (u64)j * c;
    }
    if (used) D = base + used - 1;
    if (empty) break;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Gall += __shfl_xor_sync(FULL, Gall, o);
    Mall += __shfl_xor_sync(FULL, Mall, o);
  }
  auto size_of = [&](u32 j) { return j == 0 ? 1u : j <= D ? g[j] : 0u; };
  u64 Gbase = 0, Mbase = 0;  // up to the levels before this step's
  for (u32 base = 0; base <= D; base += 32) {
    const u32 i = base + lane;
    const u64 c = size_of(i), prev = i ? size_of(i - 1) : 0u, next = size_of(i + 1);
    u64 G = c, M = i * c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 tg = __shfl_up_sync(FULL, G, o), tm = __shfl_up_sync(FULL, M, o);
      if (lane >= o) {
        G += tg;
        M += tm;
      }
    }
    G += Gbase;
    M += Mbase;
    Gbase = __shfl_sync(FULL, G, 31);
    Mbase = __shfl_sync(FULL, M, 31);
    if (i <= D) {
      const u64 Ghi = G + next, Mhi = M + (u64)(i + 1) * next;  // up to i+1
      const u64 above = (Mall - Mhi) - (u64)i * (Gall - Ghi);
      u64 v;
      if (directed) {
        v = 2 * Ghi + above - 2;
      } else {
        const u64 Glo = G - c - prev, Mlo = M - i * c - (i ? (u64)(i - 1) * prev : 0u);  // up to i-2
        v = 2 * (prev + c + next) + ((u64)i * Glo - Mlo) + above - 2;
      }
      L[i] = v;
    }
  }
  __syncwarp();
  for (u32 j = lane; j <= D; j += 32) g[j] = 0;
}

// Raises every vertex's bound with every slot that found it, then resets its
// level row for the next round.  kLanes lanes a vertex, each taking every
// kLanes-th group of 8 slots (a 16-byte load of the row); the sources' graph
// data are staged per block, kStage slots at a time.  Bounds of one reach are
// compared by their sums: (cS / (r-1)^2 > S / (r-1)^2 as cS > S), only others
// by 128-bit products.  (A thread per vertex, a slot at a time: 0.75 ms a round
// of 512 slots on a 301 x 299 grid.)  `vec`: rows of a multiple of 8 slots.
constexpr int kLanes = 4;
constexpr u32 kStage = 512;
__device__ __forceinline__ bool lb_higher(u64 cS, u64 cr, u64 S, u64 r) {
  if (r <= 1) return true;  // no bound yet
  if (cr == r) return cS > S;
  return (u128)cS * (u128)((r - 1) * (r - 1)) > (u128)S * (u128)((cr - 1) * (cr - 1));
}
template <bool kVec>
__global__ void __launch_bounds__(256) k_lb_update(u32 n, u32 B, u32 nsrc, uint16_t *lvl, const u32 *srcs,
                                                   const u32 *comp, const u32 *off, const u64 *Ltab, u32 cap,
                                                   const u32 *res_r, u64 *bS, u32 *bR, u64 *key) {
  constexpr u32 kGroup = kVec ? 8 : 1;
  __shared__ u32 s_src[kStage], s_comp[kStage], s_r[kStage];
  const u32 q = threadIdx.x % kLanes;
  const u32 per_grid = gridDim.x * (blockDim.x / kLanes);
  for (u32 s0 = 0; s0 < nsrc; s0 += kStage) {
    const u32 ns = nsrc - s0 < kStage ? nsrc - s0 : kStage;
    __syncthreads();
    for (u32 i = threadIdx.x; i < ns; i += blockDim.x) {
      const u32 src = srcs[s0 + i];
      s_src[i] = src;
      s_comp[i] = src == 0xffffffffu ? 0u : comp[src];
      s_r[i] = src == 0xffffffffu ? 0u : res_r[src];  // 0: gives no bound
    }
    __syncthreads();
    // (every lane of a warp takes part in every step: the exchange below)
    for (u32 w0 = blockIdx.x * (blockDim.x / kLanes); w0 < n; w0 += per_grid) {
      const u32 w = w0 + threadIdx.x / kLanes;
      const bool valid = w < n;
      u64 S = 0, r = 0;
      bool changed = false;
      if (valid) {
        uint16_t *row = lvl + (size_t)w * B + s0;
        const u64 od = off[w + 1] - off[w];
        const u32 cw = comp[w];
        S = bS[w];
        r = bR[w];
        auto slot = [&](u32 i, u32 l) {
          if (l == 0xffffu) return;
          const u64 cr = s_r[i];
          if (s_src[i] == w || s_comp[i] != cw || od == 0 || cr <= 1) return;
          const u64 cS = Ltab[(size_t)(s0 + i) * cap + l] - od;
          if (lb_higher(cS, cr, S, r)) {
            S = cS;
            r = cr;
            changed = true;
          }
        };
        for (u32 i = q * kGroup; i < ns; i += kLanes * kGroup) {
          if constexpr (kVec) {
            uint4 *p = reinterpret_cast<uint4 *>(row + i);
            const uint4 x = *p;
            if ((x.x & x.y & x.z & x.w) == 0xffffffffu) continue;
            *p = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
            const u32 h[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (u32 j = 0; j < 4; ++j) {
              slot(i + 2 * j, h[j] & 0xffffu);
              slot(i + 2 * j + 1, h[j] >> 16);
            }
          } else {
            const u32 l = row[i];
            if (l == 0xffffu) continue;
            row[i] = 0xffffu;
            slot(i, l);
          }
        }
      }
#pragma unroll
      for (int o = 1; o < kLanes; o <<= 1) {
        const u64 oS = __shfl_xor_sync(FULL, S, o), orr = __shfl_xor_sync(FULL, r, o);
        const bool oc = __shfl_xor_sync(FULL, (int)changed, o) != 0;
        if (oc && (!changed || lb_higher(oS, orr, S, r))) {
          S = oS;
          r = orr;
          changed = true;
        }
      }
      if (valid && changed && q == 0) {
        bS[w] = S;
        bR[w] = (u32)r;
        key[w] = (u64)(((u128)S << kKeyFrac) / (u128)((r - 1) * (r - 1)));
      }
    }
  }
}

__global__ void k_lb_gather(u32 cnt, const u32 *cand, const u64 *key, u64 *out) {
  const u32 i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < cnt) out[i] = key[cand[i]];
}

__global__ void k_lb_done(u32 nsrc, const u32 *srcs, uint8_t *done) {
  const u32 i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nsrc && srcs[i] != 0xffffffffu) done[srcs[i]] = 1;
}

__global__ void k_lb_init(u32 n, const u64 *S0, const u32 *r0, const u64 *key0, u64 *bS, u32 *bR, u64 *key,
                          uint8_t *done) {
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    bS[v] = S0 ? S0[v] : 0;
    bR[v] = S0 ? r0[v] : 2;  // bound 0
    key[v] = S0 ? key0[v] : 0;
    done[v] = 0;
  }
}

}  // namespace

int lb_init(tkc_graph *g, const u64 *S0, const u32 *r0, const u64 *key0, u64 *bS, u32 *bR, u64 *key,
            uint8_t *done) {
  cudaStream_t st = g->ctx->stream;
  TKC_LAUNCH(k_lb_init<<<grid_of(g->n), 256, 0, st>>>(g->n, S0, r0, key0, bS, bR, key, done));
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

// The candidates (initial order, not searched, out-degree >= 1) sorted by
// (key, position in the initial order): a stable compaction, then stable
// radix passes over the low and the high 32 key bits.  Writes *count of them
// to cand (device); synchronises the stream.
int lb_sorted_candidates(tkc_graph *g, const u32 *order0, u32 n0, const uint8_t *done, const u64 *key, u32 *cand,
                         u32 *count, u32 *scratch_pos, u32 *scratch_tmp, u32 *scratch_lo, u64 *scratch_max) {
  cudaStream_t st = g->ctx->stream;
  *count = 0;
  if (n0 == 0) return TKC_OK;
  TKC_LAUNCH(k_lb_flags<<<grid_of(n0), 256, 0, st>>>(order0, n0, g->off, done, scratch_pos));
  TKC_RC(scan_exclusive_u32(scratch_pos, scratch_pos, (u64)n0 + 1, scratch_tmp, st));
  TKC_LAUNCH(k_lb_compact<<<grid_of(n0), 256, 0, st>>>(order0, scratch_pos, n0, cand));
  u32 m = 0;
  TKC_TRY(cudaMemcpyAsync(&m, scratch_pos + n0, sizeof(u32), cudaMemcpyDeviceToHost, st));
  TKC_TRY(cudaMemsetAsync(scratch_max, 0, sizeof(u64), st));
  TKC_TRY(cudaStreamSynchronize(st));
  if (m) {
    TKC_LAUNCH(k_lb_key_lo<<<grid_of(m), 256, 0, st>>>(m, cand, key, scratch_lo, scratch_max));
    u64 mk = 0;
    TKC_TRY(read_back(&mk, scratch_max, sizeof(u64), st));
    int bits = 0;
    while (bits < 64 && (mk >> bits) != 0) ++bits;
    if (bits <= 32) {
      TKC_RC(radix_sort_u32_pairs(scratch_lo, cand, m, bits, st));
    } else {
      TKC_RC(radix_sort_u32_pairs(scratch_lo, cand, m, 32, st));
      TKC_LAUNCH(k_lb_key_hi<<<grid_of(m), 256, 0, st>>>(m, cand, key, scratch_lo));
      TKC_RC(radix_sort_u32_pairs(scratch_lo, cand, m, bits - 32, st));
    }
  }
  TKC_TRY(cudaStreamSynchronize(st));
  *count = m;
  return TKC_OK;
}

int lb_gather_keys(tkc_graph *g, u32 cnt, const u32 *cand, const u64 *key, u64 *out) {
  TKC_LAUNCH(k_lb_gather<<<(cnt + 255) / 256, 256, 0, g->ctx->stream>>>(cnt, cand, key, out));
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

// After a round of complete searches from srcs[0..nsrc) (0xffffffff: slot
// unused): level bounds per source, then every vertex's bound.  lvl rows (B =
// row length) are reset to 0xffff, the level sizes (hist) to 0.
int lb_update(tkc_graph *g, u32 B, u32 nsrc, const u32 *srcs, uint16_t *lvl, u32 *hist, u32 cap,
              u64 *Ltab, const u32 *res_r, u64 *bS, u32 *bR, u64 *key, uint8_t *done) {
  cudaStream_t st = g->ctx->stream;
  TKC_LAUNCH(k_lb_table<<<(nsrc + 7) / 8, 256, 0, st>>>(nsrc, hist, cap, g->directed, Ltab));
  const unsigned blocks = grid_of((u64)g->n * kLanes);
  if (B % 8 == 0) {
    TKC_LAUNCH(k_lb_update<true><<<blocks, 256, 0, st>>>(g->n, B, nsrc, lvl, srcs, g->comp, g->off, Ltab, cap, res_r, bS,
                                                         bR, key));
  } else {
    TKC_LAUNCH(k_lb_update<false><<<blocks, 256, 0, st>>>(g->n, B, nsrc, lvl, srcs, g->comp, g->off, Ltab, cap, res_r,
                                                          bS, bR, key));
  }
  TKC_LAUNCH(k_lb_done<<<(nsrc + 255) / 256, 256, 0, st>>>(nsrc, srcs, done));
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

}  // namespace tkc
