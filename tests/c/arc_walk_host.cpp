// The warp walk of tkc_arcs.cuh on the host: 32 threads stand in for the
// lanes, meeting at every warp collective.  The offsets end at an unmapped
// page and an unmapped range lies before them, so a read out of range ends the
// process; a walk that takes more collectives than any valid one does ends it
// with status 3.  Arguments: n, first arc, one past the last arc, 1 to check
// the sources; the n + 1 offsets follow on standard input.
#include <sys/mman.h>
#include <unistd.h>

#include <atomic>
#include <barrier>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <thread>
#include <vector>

#define __device__
#define __host__
#define __forceinline__ inline
struct Dim {
  unsigned x;
};
static thread_local Dim threadIdx;
static Dim blockIdx{0}, blockDim{32}, gridDim{1};

static std::barrier<> g_meet(32);
static uint32_t g_val[32];
static std::atomic<uint64_t> g_steps{0};
static uint64_t g_most;

static void meet() {
  if (g_steps.fetch_add(1) > g_most) _exit(3);
  g_meet.arrive_and_wait();
}
static unsigned __ballot_sync(unsigned, bool p) {
  g_val[threadIdx.x] = p;
  meet();
  unsigned m = 0;
  for (int l = 0; l < 32; ++l) m |= g_val[l] ? 1u << l : 0u;
  meet();
  return m;
}
static uint32_t __shfl_sync(unsigned, uint32_t v, int src) {
  g_val[threadIdx.x] = v;
  meet();
  const uint32_t r = g_val[src & 31];
  meet();
  return r;
}
static int __clz(unsigned x) { return x ? __builtin_clz(x) : 32; }

#include "tkc_arcs.cuh"

int main(int argc, char **argv) {
  if (argc != 5) return 2;
  const uint32_t n = (uint32_t)strtoul(argv[1], nullptr, 10);
  const uint64_t a0 = strtoull(argv[2], nullptr, 10), a1 = strtoull(argv[3], nullptr, 10);
  const bool check = argv[4][0] == '1';
  const size_t page = (size_t)sysconf(_SC_PAGESIZE), need = ((size_t)n + 1) * 4, body = (need + page - 1) / page * page;
  const size_t guard = (size_t)1 << 34;  // an index of up to 2^32 either way
  char *m = (char *)mmap(nullptr, 2 * guard + body, PROT_NONE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (m == MAP_FAILED || mprotect(m + guard, body, PROT_READ | PROT_WRITE)) return 2;
  uint32_t *off = (uint32_t *)(m + guard + body - need);
  for (uint32_t i = 0; i <= n; ++i)
    if (scanf("%u", &off[i]) != 1) return 2;
  // a search takes 7 rounds at most, a window of 32 rows and a group of 32 arcs 7 collectives each
  g_most = 32 * 2 * 8 * (16 + n / 32 + (a1 - a0) / 32 + (a1 - a0));
  std::vector<uint32_t> src(a1 - a0, 0xffffffffu);
  std::atomic<int> bad{0};
  std::vector<std::thread> lanes;
  for (unsigned l = 0; l < 32; ++l)
    lanes.emplace_back([&, l] {
      threadIdx.x = l;
      tkc::warp_walk_arcs<true>(off, n, a0, a1, (int)l, [&](uint32_t u, uint64_t i, bool valid, uint32_t rs) {
        if (!valid) return;
        if (i < a0 || i >= a1 || src[i - a0] != 0xffffffffu || (check && (u >= n || rs != off[u]))) bad = 1;
        else src[i - a0] = u;
      });
    });
  for (auto &t : lanes) t.join();
  if (check)
    for (uint64_t i = a0; i < a1; ++i) {
      const uint32_t u = src[i - a0];
      if (u >= n || off[u] > i || off[u + 1] <= i) bad = 1;
    }
  return bad;
}
