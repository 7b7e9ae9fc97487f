// Grid barrier for cooperative launches whose blocks step through rounds
// together (reach BFS, trimming, colouring, components, NB sweeps, Algorithm
// 6).  A round of one of these on a small graph is a few microseconds of work;
// driven from the host it cost a launch or two, a 4-byte copy and a wait --
// about 15 us -- and there are tens of them in a call.
//
// Every wait is bounded: when it runs out the block records TKC_ETIMEOUT and
// returns false, as the others do at their next wait.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "tkc_internal.cuh"

namespace tkc {

// Device words of one launch's barrier, alone in its cache line; zero at the launch.
struct GridBar {
  unsigned count, gen, pad[30];
  int err;
  unsigned pad1[31];
};

__device__ __forceinline__ unsigned grid_ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// All blocks of the launch; thread 0 of the last one to arrive runs `epi`
// before the others are released.  Returns false after an error.
template <typename Epi>
__device__ __forceinline__ bool grid_sync(GridBar *b, uint64_t timeout, Epi epi) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    s_ok = 1;
    const unsigned gen = grid_ld_acquire(&b->gen);
    __threadfence();
    if (atomicAdd(&b->count, 1u) + 1u == gridDim.x) {
      __threadfence();
      epi();
      b->count = 0;
      __threadfence();
      asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&b->gen), "r"(gen + 1u) : "memory");
    } else {
      const long long t0 = clock64();
      for (unsigned poll = 1; grid_ld_acquire(&b->gen) == gen; ++poll) {
        const bool late = (uint64_t)(clock64() - t0) > timeout;
        if (late) atomicCAS(&b->err, 0, TKC_ETIMEOUT);
        if (((poll & 15u) == 0 || late) && *(volatile int *)&b->err != 0) {
          s_ok = 0;
          break;
        }
        if (poll > 64) __nanosleep(128);
      }
      __threadfence();
    }
  }
  __syncthreads();
  return s_ok != 0;
}

// Blocks of a cooperative launch of `kernel` (tpb threads): enough for `work`
// threads, at most what is resident at once.  0 on error.
template <typename K>
int grid_blocks(const tkc_ctx *ctx, K kernel, int tpb, uint64_t work) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, tpb, 0) != cudaSuccess || per_sm <= 0) return 0;
  const uint64_t want = (work + tpb - 1) / tpb, most = (uint64_t)per_sm * ctx->num_sms;
  return (int)std::max<uint64_t>(1, std::min(want, most));
}

inline uint64_t grid_timeout(const tkc_ctx *ctx) {
  return ctx->opt.timeout_cycles ? ctx->opt.timeout_cycles : (1ull << 34);
}

}  // namespace tkc
