// Learned source order: per-vertex features, a 5 -> 64 -> 64 -> 1 MLP
// (bf16 weights, fp32 accumulation) with hand-written forward, backward and
// Adam kernels, and the order of sources by predicted farness.
//
// The paper orders sources by a degree bound (computeBoundsDeg, Section 4);
// any order gives the same exact top-k (Algorithm 1 only prunes), so a model
// that predicts farness can only change how soon the k-th threshold x becomes
// tight.  Without a model the degree order is used.
//
// Parameter layout (TKC_MLP_PARAMS floats):
//   W1[64][5] at 0, b1[64] at 320, W2[64][64] at 384, b2[64] at 4480,
//   w3[64] at 4544, b3 at 4608.
// y = w3 . relu(W2 relu(W1 x + b1) + b2) + b3.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "tkc_internal.cuh"

namespace tkc {

typedef uint32_t u32;
typedef unsigned long long u64;
static constexpr unsigned FULL = 0xffffffffu;

constexpr int F = TKC_MLP_FEATURES;
constexpr int H = TKC_MLP_HIDDEN;
constexpr int P = TKC_MLP_PARAMS;
constexpr int oW1 = 0, oB1 = H * F, oW2 = oB1 + H, oB2 = oW2 + H * H, oW3 = oB2 + H, oB3 = oW3 + H;
static_assert(oB3 + 1 == P, "parameter layout");

int radix_sort_u32_pairs(u32 *key, u32 *val, u32 n, int bits, cudaStream_t st);

namespace {

unsigned grid_of(u64 work, unsigned tpb = 256, unsigned cap = 152 * 16) {
  u64 b = (work + tpb - 1) / tpb;
  return (unsigned)std::max<u64>(1, std::min<u64>(b, cap));
}

// ---------------------------------------------------------------- features

// 2-walk count: sum of out-degrees of the out-neighbours (the gamma bound of
// the Section 6 lemma at d = 1, an upper bound on the 2-hop ball), one warp per vertex.
__global__ void k_two_walks(const u32 *off, const u32 *col, u32 n, float *w2) {
  const int lane = threadIdx.x & 31;
  for (u32 v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += (gridDim.x * blockDim.x) >> 5) {
    u64 s = 0;
    for (u32 i = off[v] + lane; i < off[v + 1]; i += 32) {
      u32 u = col[i];
      s += off[u + 1] - off[u];
    }
    for (int o = 16; o; o >>= 1) s += __shfl_down_sync(FULL, s, o);
    if (lane == 0) w2[v] = (float)s;
  }
}

__global__ void k_core_init(const u32 *off, const u32 *ioff, u32 n, int directed, u32 *c) {
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    c[v] = (off[v + 1] - off[v]) + (directed ? ioff[v + 1] - ioff[v] : 0u);
}

// One h-index step of the core-number iteration (Lu, Zhou, Zhang, Stanley,
// Nat. Commun. 2016): c'(v) = the largest h such that at least h neighbours
// have c >= h, neighbours taken over out-arcs (and in-arcs when directed,
// so a vertex linked both ways counts twice: the graph with arc directions
// dropped).  Started from the degree it never rises, and once no value
// changes it is the core number.  Only vertices with a neighbour whose value
// changed in the previous step (dirty_in) are recomputed; a vertex whose value
// changes marks its neighbours in dirty_out and sets *changed.
constexpr int kCoreTPB = 256;      // threads per block of k_core_step
constexpr u32 kCoreBuckets = 256;  // histogram buckets per warp

__global__ void __launch_bounds__(kCoreTPB) k_core_step(const u32 *off, const u32 *col, const u32 *ioff,
                                                        const u32 *icol, u32 n, int directed, const u32 *c, u32 *c2,
                                                        const uint8_t *dirty_in, uint8_t *dirty_out, u32 *changed) {
  __shared__ u32 hist_all[kCoreTPB / 32][kCoreBuckets];
  const int lane = threadIdx.x & 31;
  u32 *hist = hist_all[threadIdx.x >> 5];
  for (u32 base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; base < n; base += gridDim.x * blockDim.x) {
    // lane per vertex: copy the clean ones; the warp then takes the dirty ones
    const u32 mine = base + lane;
    bool dirty = false;
    if (mine < n) {
      dirty = dirty_in[mine] != 0;
      if (!dirty) c2[mine] = c[mine];
    }
    for (unsigned dm = __ballot_sync(FULL, dirty); dm; dm &= dm - 1) {
      const u32 v = base + (__ffs(dm) - 1);
      const u32 cv = c[v];
      // neighbours' values (out-arcs, and in-arcs when directed), visited by the warp
      auto for_each_value = [&](auto &&f) {
        for (u32 i = off[v] + lane; i < off[v + 1]; i += 32) f(c[col[i]]);
        if (directed)
          for (u32 i = ioff[v] + lane; i < ioff[v + 1]; i += 32) f(c[icol[i]]);
      };
      // the value never rises: one pass checks whether it stays (the common
      // case once most values have settled)
      u32 cnt = 0;
      for_each_value([&](u32 x) { cnt += x >= cv; });
      u32 above = __reduce_add_sync(FULL, cnt);  // neighbours with a value above the range searched
      u32 lo = 0, hi = cv;                       // the new value h lies in [lo, hi]
      if (above >= cv) {
        lo = cv;
      } else {
        // h < cv: h = the largest h with (neighbours whose value is >= h) >= h.
        // Each pass spreads [lo, hi] over 256 buckets, counts the neighbours'
        // values per bucket, and keeps the highest bucket whose start still
        // satisfies the condition (the count only falls as h rises, and h = lo
        // always satisfies it): one pass when cv <= 256, at most three below
        // 2^24 -- instead of one pass per halving of [0, cv].
        hi = cv - 1;
        while (lo < hi) {
          const u32 width = (hi - lo) / kCoreBuckets + 1;
          for (u32 j = lane; j < kCoreBuckets; j += 32) hist[j] = 0;
          __syncwarp();
          for_each_value([&](u32 x) {
            if (x >= lo && x <= hi) atomicAdd(&hist[(x - lo) / width], 1u);
          });
          __syncwarp();
          // lane j holds buckets 8j .. 8j+7; suffix sums over the warp from the top
          u32 loc[kCoreBuckets / 32];
          u32 part = 0;
#pragma unroll
          for (int q = kCoreBuckets / 32 - 1; q >= 0; --q) {
            part += hist[lane * (kCoreBuckets / 32) + q];
            loc[q] = part;  // buckets q.. of this lane's group
          }
          u32 incl = part;  // this lane's group total, then the sum of groups j..31
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const u32 t = __shfl_down_sync(FULL, incl, o);
            if (lane + o < 32) incl += t;
          }
          const u32 later = incl - part;  // groups above this lane's
          // highest bucket b with above + (count in buckets >= b) >= lo + b * width
          int best = -1;
#pragma unroll
          for (int q = kCoreBuckets / 32 - 1; q >= 0; --q) {
            const u32 b = lane * (kCoreBuckets / 32) + q;
            const u64 start = (u64)lo + (u64)b * width;
            if (best < 0 && start <= hi && (u64)above + later + loc[q] >= start) best = (int)b;
          }
          const unsigned has = __ballot_sync(FULL, best >= 0);
          const int src = 31 - __clz(has);  // the highest group with such a bucket (group 0 always has one)
          const u32 b = (u32)__shfl_sync(FULL, best, src);
          // neighbours in buckets above b
          const u32 b_above = __shfl_sync(FULL, later + loc[b % (kCoreBuckets / 32)] -
                                                     hist[lane * (kCoreBuckets / 32) + b % (kCoreBuckets / 32)],
                                          src);
          __syncwarp();
          const u32 nlo = lo + b * width;
          const u32 nhi = (u64)nlo + width - 1 < hi ? nlo + width - 1 : hi;
          above += b_above;
          lo = nlo;
          hi = nhi;
        }
      }
      if (lane == 0) c2[v] = lo;
      if (lo != cv) {
        if (lane == 0) *changed = 1;
        for (u32 i = off[v] + lane; i < off[v + 1]; i += 32) dirty_out[col[i]] = 1;
        if (directed)
          for (u32 i = ioff[v] + lane; i < ioff[v + 1]; i += 32) dirty_out[icol[i]] = 1;
      }
    }
  }
}

__global__ void k_features_raw(const u32 *off, const u32 *ioff, const float *w2, const u32 *core, const u32 *scc,
                               u32 n, float *x, double *sums) {
  double s[F] = {0}, q[F] = {0};
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    float f[F];
    f[0] = log1pf((float)(off[v + 1] - off[v]));
    f[1] = log1pf((float)(ioff[v + 1] - ioff[v]));
    f[2] = log1pf(w2[v]);
    f[3] = log1pf((float)core[v]);
    f[4] = log1pf((float)scc[v]);
#pragma unroll
    for (int j = 0; j < F; ++j) {
      x[(size_t)v * F + j] = f[j];
      s[j] += f[j];
      q[j] += (double)f[j] * f[j];
    }
  }
#pragma unroll
  for (int j = 0; j < F; ++j) {
    for (int o = 16; o; o >>= 1) {
      s[j] += __shfl_down_sync(FULL, s[j], o);
      q[j] += __shfl_down_sync(FULL, q[j], o);
    }
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(&sums[j], s[j]);
      atomicAdd(&sums[F + j], q[j]);
    }
  }
}

__global__ void k_features_standardize(float *x, u32 n, const double *sums) {
  __shared__ float mean[F], inv[F];
  if (threadIdx.x < F) {
    double m = sums[threadIdx.x] / n;
    double var = sums[F + threadIdx.x] / n - m * m;
    mean[threadIdx.x] = (float)m;
    inv[threadIdx.x] = (float)(1.0 / sqrt(var > 1e-12 ? var : 1e-12));
  }
  __syncthreads();
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < (u64)n * F; i += (u64)gridDim.x * blockDim.x) {
    int j = (int)(i % F);
    x[i] = (x[i] - mean[j]) * inv[j];
  }
}

// ---------------------------------------------------------------- MLP kernels

__device__ __forceinline__ float weight(const unsigned short *wb, int i) {
  return __bfloat162float(__ushort_as_bfloat16(wb[i]));
}

constexpr int FT = 128;  // samples per forward block

// y[i] for m samples, one thread per sample with its first hidden layer in
// registers: the 64 products of a second-layer unit then read only the unit's
// weights, four to a (broadcast) shared-memory load, so the pass is bound by
// its 4 096 multiply-adds per sample (with the layer in shared memory each of
// them loaded two words).
__global__ void __launch_bounds__(FT) k_mlp_forward(const float *x, u32 m, const unsigned short *wb, float *y) {
  __shared__ __align__(16) float ws[P + 3];
  for (int i = threadIdx.x; i < P; i += FT) ws[i] = weight(wb, i);
  __syncthreads();
  static_assert(oW2 % 4 == 0 && H % 4 == 0, "the second layer's rows are read four words at a time");
  // (by tiles: a position one step past the last of nearly 2^32 samples would start over)
  for (u32 tile = blockIdx.x; tile < (m - 1) / FT + 1; tile += gridDim.x) {
    const u32 i = tile * FT + threadIdx.x;  // tile * FT + FT - 1 is below 2^32
    const bool valid = i < m;
    float xi[F];
#pragma unroll
    for (int f = 0; f < F; ++f) xi[f] = valid ? x[(size_t)i * F + f] : 0.f;
    float h1[H];
#pragma unroll
    for (int o = 0; o < H; ++o) {
      float a = ws[oB1 + o];
#pragma unroll
      for (int f = 0; f < F; ++f) a = fmaf(ws[oW1 + o * F + f], xi[f], a);
      h1[o] = a > 0.f ? a : 0.f;
    }
    float out = ws[oB3];
#pragma unroll 2
    for (int o = 0; o < H; ++o) {
      float a = ws[oB2 + o];
      const float4 *w = reinterpret_cast<const float4 *>(ws + oW2 + o * H);
#pragma unroll
      for (int j = 0; j < H / 4; ++j) {
        const float4 q = w[j];
        a = fmaf(q.x, h1[4 * j], a);
        a = fmaf(q.y, h1[4 * j + 1], a);
        a = fmaf(q.z, h1[4 * j + 2], a);
        a = fmaf(q.w, h1[4 * j + 3], a);
      }
      out = fmaf(ws[oW3 + o], a > 0.f ? a : 0.f, out);
    }
    if (valid) y[i] = out;
  }
}

constexpr int PS = (P + 31) / 32 * 32;  // a block's row of parameter sums
constexpr int TS = 16;        // samples per gradient tile
constexpr int kGradTPB = 256;
constexpr int W2S = H + 1;    // row stride of W2 in shared memory: rows and columns both without conflicts
constexpr int TH = H + 4;     // row stride of the tiles (16-byte aligned rows)

// Gradient of the mean squared error L = (1/m) sum (y_i - t_i)^2 with
// respect to the parameters, the forward pass using the bf16 weights.  A block
// takes tiles of 16 samples, keeps its share of the parameter sums in
// registers over its tiles, and writes them to its row of `part` (and its loss
// to lossp) at the end.  Thread t = 16 y + x computes, of the 16 x 64
// tile products, sample y and units x, x + 16, x + 32, x + 48, and of the 64 x
// 64 sums of the second layer rows 4 y .. 4 y + 3 and those four columns.
// (Bound by latency: 27 million multiply-adds.  With W2's rows 64 words apart
// every read of a column hit one bank 32 times and 2 048 samples took 56 us,
// now 11.)
__global__ void __launch_bounds__(kGradTPB) k_mlp_grad(const float *x, const float *t, u32 m, const unsigned short *wb,
                                                       float *part, double *lossp) {
  __shared__ float w2[H * W2S], w1[H * F], b1[H], b2[H], w3[H];
  __shared__ __align__(16) float X[TS * F], H1[TS * TH], H2[TS * TH], D2[TS * TH];  // H2 holds D1 later
  __shared__ float dy[TS], s_b3;
  __shared__ double s_loss[kGradTPB / 32];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // k_mlp_sum may be launched
  for (int i = threadIdx.x; i < P; i += kGradTPB) {
    const float w = weight(wb, i);
    if (i < oB1) w1[i - oW1] = w;
    else if (i < oW2) b1[i - oB1] = w;
    else if (i < oB2) w2[(i - oW2) / H * W2S + (i - oW2) % H] = w;
    else if (i < oW3) b2[i - oB2] = w;
    else if (i < oB3) w3[i - oW3] = w;
    else s_b3 = w;
  }
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float g2[4][4] = {}, g1[2] = {0.f, 0.f}, gb = 0.f;  // this thread's sums
  double l = 0.0;  // of many small terms from every block: added up in 64 bits
  for (u32 tile = blockIdx.x; tile < (m - 1) / TS + 1; tile += gridDim.x) {  // (by tiles as in the forward pass)
    const u32 base = tile * TS;
    __syncthreads();
    for (int i = threadIdx.x; i < TS * F; i += kGradTPB) {
      const u32 s = base + i / F;
      X[i] = s < m ? x[(size_t)s * F + i % F] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int o = tx + 16 * q;
      float a = b1[o];
#pragma unroll
      for (int f = 0; f < F; ++f) a = fmaf(w1[o * F + f], X[ty * F + f], a);
      H1[ty * TH + o] = a > 0.f ? a : 0.f;
    }
    __syncthreads();
    {
      float a[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) a[q] = b2[tx + 16 * q];
#pragma unroll 4
      for (int j = 0; j < H; j += 4) {
        const float4 h = *reinterpret_cast<const float4 *>(H1 + ty * TH + j);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float *w = w2 + (tx + 16 * q) * W2S + j;
          a[q] = fmaf(w[0], h.x, a[q]);
          a[q] = fmaf(w[1], h.y, a[q]);
          a[q] = fmaf(w[2], h.z, a[q]);
          a[q] = fmaf(w[3], h.w, a[q]);
        }
      }
      float part = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int o = tx + 16 * q;
        a[q] = a[q] > 0.f ? a[q] : 0.f;
        H2[ty * TH + o] = a[q];
        part = fmaf(w3[o], a[q], part);
      }
      // y: the 16 threads of a sample are half a warp
#pragma unroll
      for (int d = 8; d; d >>= 1) part += __shfl_xor_sync(FULL, part, d);
      if (tx == 0) {
        const bool valid = base + ty < m;
        const float e = valid ? part + s_b3 - t[base + ty] : 0.f;
        dy[ty] = 2.f * e / (float)m;
        l += (double)e * (double)e / (double)m;
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int o = tx + 16 * q;
      D2[ty * TH + o] = H2[ty * TH + o] > 0.f ? dy[ty] * w3[o] : 0.f;
    }
    __syncthreads();
    // sums of the second layer, of the biases' and of the output's weights
#pragma unroll 4
    for (int s = 0; s < TS; ++s) {
      const float4 d = *reinterpret_cast<const float4 *>(D2 + s * TH + 4 * ty);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float h = H1[s * TH + tx + 16 * q];
        g2[0][q] = fmaf(d.x, h, g2[0][q]);
        g2[1][q] = fmaf(d.y, h, g2[1][q]);
        g2[2][q] = fmaf(d.z, h, g2[2][q]);
        g2[3][q] = fmaf(d.w, h, g2[3][q]);
      }
    }
    if (threadIdx.x >= 64 && threadIdx.x < 128) {
      const int o = threadIdx.x - 64;
      for (int s = 0; s < TS; ++s) gb += D2[s * TH + o];
    } else if (threadIdx.x >= 128 && threadIdx.x < 192) {
      const int o = threadIdx.x - 128;
      for (int s = 0; s < TS; ++s) gb = fmaf(dy[s], H2[s * TH + o], gb);
    } else if (threadIdx.x == 192) {
      for (int s = 0; s < TS; ++s) gb += dy[s];
    }
    __syncthreads();
    // D1 = dL/d(pre-activation 1), over H2
    {
      float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
      for (int o = 0; o < H; o += 4) {
        const float4 d = *reinterpret_cast<const float4 *>(D2 + ty * TH + o);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float *w = w2 + o * W2S + tx + 16 * q;
          a[q] = fmaf(d.x, w[0], a[q]);
          a[q] = fmaf(d.y, w[W2S], a[q]);
          a[q] = fmaf(d.z, w[2 * W2S], a[q]);
          a[q] = fmaf(d.w, w[3 * W2S], a[q]);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int j = tx + 16 * q;
        H2[ty * TH + j] = H1[ty * TH + j] > 0.f ? a[q] : 0.f;
      }
    }
    __syncthreads();
    const float *D1 = H2;
    for (int r = 0; r < 2; ++r) {
      const int p = threadIdx.x + r * kGradTPB;
      if (p < H * F)
        for (int s = 0; s < TS; ++s) g1[r] = fmaf(D1[s * TH + p / F], X[s * F + p % F], g1[r]);
    }
    if (threadIdx.x < 64)
      for (int s = 0; s < TS; ++s) gb += D1[s * TH + threadIdx.x];
  }
  // the block's sums
  float *row = part + (size_t)blockIdx.x * PS;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) row[oW2 + (4 * ty + r) * H + tx + 16 * q] = g2[r][q];
  for (int r = 0; r < 2; ++r) {
    const int p = threadIdx.x + r * kGradTPB;
    if (p < H * F) row[oW1 + p] = g1[r];
  }
  const int pb = threadIdx.x < 64 ? oB1 + threadIdx.x
                 : threadIdx.x < 128 ? oB2 + threadIdx.x - 64
                 : threadIdx.x < 192 ? oW3 + threadIdx.x - 128
                                     : oB3;
  if (threadIdx.x <= 192) row[pb] = gb;
  // the losses of tx == 0, two samples per warp
  l += __shfl_xor_sync(FULL, l, 16);
  if ((threadIdx.x & 31) == 0) s_loss[threadIdx.x >> 5] = l;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kGradTPB / 32; ++w) t += s_loss[w];
    lossp[blockIdx.x] = t;
  }
}

// The gradient and the loss from the blocks' sums: 32 parameters a block, the
// rows split over its 8 warps, added up four at a time and then by warps, in a
// fixed order.  (Block sums added to grad by atomics, 128 to a word, made the
// error against 64 bits 2.5e-7 for 2 048 samples, this 0.3e-7 to 0.8e-7; a
// 64-bit sum here is no nearer and 4 us slower.)  It is launched early and
// waits for the sums on the device, so that its launch overlaps them.
constexpr int kSumWarps = 8;
__global__ void __launch_bounds__(32 * kSumWarps) k_mlp_sum(const float *part, const double *lossp, u32 rows,
                                                            float *grad, double *loss) {
  __shared__ float s[kSumWarps][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + lane;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  float a = 0.f;
  if (p < P) {
    u32 r = wid;
#pragma unroll 4
    for (; r + 3 * kSumWarps < rows; r += 4 * kSumWarps) {
      const float *q = part + (size_t)r * PS + p;
      a += (q[0] + q[kSumWarps * PS]) + (q[2 * kSumWarps * PS] + q[3 * kSumWarps * PS]);
    }
    for (; r < rows; r += kSumWarps) a += part[(size_t)r * PS + p];
  }
  s[wid][lane] = a;
  __syncthreads();
  if (wid == 0 && p < P) {
    float t[kSumWarps];
#pragma unroll
    for (int w = 0; w < kSumWarps; ++w) t[w] = s[w][lane];
#pragma unroll
    for (int d = 1; d < kSumWarps; d *= 2)
#pragma unroll
      for (int w = 0; w < kSumWarps; w += 2 * d) t[w] += t[w + d];
    grad[p] = t[0];
  } else if (wid == 1 && blockIdx.x == 0) {
    double l = 0.0;
    for (u32 r = lane; r < rows; r += 32) l += lossp[r];
#pragma unroll
    for (int d = 16; d; d >>= 1) l += __shfl_xor_sync(FULL, l, d);
    if (lane == 0) *loss = l;
  }
}

// Adam (Kingma & Ba 2015) on the fp32 master weights; refreshes the bf16 copy.
__global__ void k_adam(float *w, unsigned short *wb, float *mo, float *ve, const float *g, float lr, float b1,
                       float b2, float c1, float c2, float eps) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x) {
    float gi = g[i];
    float m = b1 * mo[i] + (1.f - b1) * gi;
    float v = b2 * ve[i] + (1.f - b2) * gi * gi;
    mo[i] = m;
    ve[i] = v;
    float wi = w[i] - lr * (m / c1) / (sqrtf(v / c2) + eps);
    w[i] = wi;
    wb[i] = __bfloat16_as_ushort(__float2bfloat16_rn(wi));
  }
}

__global__ void k_to_bf16(const float *w, unsigned short *wb) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x)
    wb[i] = __bfloat16_as_ushort(__float2bfloat16_rn(w[i]));
}

// He-uniform weights from splitmix64(seed ^ index); biases zero.
__global__ void k_mlp_init(float *w, u64 seed) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x) {
    u64 z = (seed ^ (u64)i) + 0x9e3779b97f4a7c15ULL;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    z ^= z >> 31;
    float u = (float)(z >> 40) * (1.0f / 16777216.0f) * 2.f - 1.f;  // [-1, 1)
    float fan_in = i < oB1 ? (float)F : (i >= oW2 && i < oB2) || (i >= oW3 && i < oB3) ? (float)H : 0.f;
    w[i] = fan_in > 0.f ? u * sqrtf(6.f / fan_in) : 0.f;
  }
}

// Order keys for predicted farness: smaller prediction first (float bits
// mapped to an order-preserving unsigned integer).
__global__ void k_score_keys(const float *y, u32 n, u32 *key, u32 *val) {
  for (u32 v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    u32 b = __float_as_uint(y[v]);
    key[v] = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
    val[v] = v;
  }
}

}  // namespace

int filter_order(tkc_graph *g, const u32 *d_order_all, u32 *d_out, u32 *count);

// The model's buffers, one allocation (an allocation takes about 40 us).
static int ensure_mlp(tkc_ctx *ctx) {
  MlpState &s = ctx->mlp;
  if (s.w) return TKC_OK;
  unsigned char *base = nullptr;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    unsigned char *p = base + at;
    at += (bytes + 255) / 256 * 256;
    return p;
  };
  for (int pass = 0; pass < 2; ++pass) {
    if (pass) TKC_TRY(cudaMalloc(&base, at));
    at = 0;
    float *w = (float *)take(P * sizeof(float));
    s.wb = (unsigned short *)take(P * sizeof(unsigned short));
    s.m = (float *)take(P * sizeof(float));
    s.v = (float *)take(P * sizeof(float));
    s.grad = (float *)take(P * sizeof(float));
    s.loss = (double *)take(sizeof(double));
    s.lossp = (double *)take((size_t)ctx->num_sms * sizeof(double));
    s.part = (float *)take((size_t)ctx->num_sms * PS * sizeof(float));
    if (pass) s.w = w;  // (set last: it says that the buffers are there)
  }
  return TKC_OK;
}

void free_mlp(tkc_ctx *ctx) {
  MlpState &s = ctx->mlp;
  if (s.w) cudaFree(s.w);
  s = MlpState();
}

static int reset_adam(tkc_ctx *ctx) {
  MlpState &s = ctx->mlp;
  TKC_TRY(cudaMemsetAsync(s.m, 0, P * sizeof(float), ctx->stream));
  TKC_TRY(cudaMemsetAsync(s.v, 0, P * sizeof(float), ctx->stream));
  s.step = 0;
  s.version++;
  s.ready = true;
  return TKC_OK;
}

static int make_features(tkc_graph *g, float *x);

int ensure_features(tkc_graph *g) {
  if (g->features) return TKC_OK;
  TKC_RC(ensure_reach_bounds(g));  // provides the SCC sizes
  TKC_RC(ensure_in_csr(g));
  cudaStream_t st = g->ctx->stream;
  const u32 n = g->n;
  if (n == 0) return TKC_OK;
  float *x = nullptr;
  TKC_TRY(dev_malloc(&x, (size_t)n * F * sizeof(float), st));
  const int rc = make_features(g, x);
  if (rc != TKC_OK) {  // the handle stays without: its pointer says that they are complete
    cudaFreeAsync(x, st);
    return rc;
  }
  g->features = x;
  return TKC_OK;
}

static int make_features(tkc_graph *g, float *x) {
  cudaStream_t st = g->ctx->stream;
  const u32 n = g->n;
  float *w2 = nullptr;
  u32 *c0 = nullptr, *c1 = nullptr;
  double *sums = nullptr;
  TKC_TRY(dev_malloc(&w2, (size_t)n * sizeof(float), st));
  TKC_TRY(dev_malloc(&c0, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&c1, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&sums, 2 * F * sizeof(double), st));
  TKC_LAUNCH(k_two_walks<<<grid_of((u64)n * 32), 256, 0, st>>>(g->off, g->col, n, w2));
  TKC_LAUNCH(k_core_init<<<grid_of(n), 256, 0, st>>>(g->off, g->ioff, n, g->directed, c0));
  u32 *flag = nullptr;
  uint8_t *d0 = nullptr, *d1 = nullptr;
  TKC_TRY(dev_malloc(&flag, sizeof(u32), st));
  TKC_TRY(dev_malloc(&d0, n, st));
  TKC_TRY(dev_malloc(&d1, n, st));
  TKC_TRY(cudaMemsetAsync(d0, 1, n, st));  // every vertex is computed in the first step
  for (u64 it = 0;; ++it) {
    // a step that changes something lowers at least one value, and the values
    // start at the degrees: 2 arcs + 1 steps suffice
    if (it > 2 * g->arcs + 1) return TKC_ETIMEOUT;
    TKC_TRY(cudaMemsetAsync(flag, 0, sizeof(u32), st));
    TKC_TRY(cudaMemsetAsync(d1, 0, n, st));
    TKC_LAUNCH(k_core_step<<<grid_of(n, kCoreTPB), kCoreTPB, 0, st>>>(g->off, g->col, g->ioff, g->icol, n, g->directed, c0, c1, d0,
                                                       d1, flag));
    std::swap(c0, c1);
    std::swap(d0, d1);
    u32 h = 0;
    TKC_TRY(read_back(&h, flag, sizeof(u32), st));
    if (!h) break;
  }
  TKC_TRY(cudaFreeAsync(flag, st));
  TKC_TRY(cudaFreeAsync(d0, st));
  TKC_TRY(cudaFreeAsync(d1, st));
  TKC_TRY(cudaMemsetAsync(sums, 0, 2 * F * sizeof(double), st));
  TKC_LAUNCH(k_features_raw<<<grid_of(n), 256, 0, st>>>(g->off, g->ioff, w2, c0, g->scc_size, n, x, sums));
  TKC_LAUNCH(k_features_standardize<<<grid_of((u64)n * F), 256, 0, st>>>(x, n, sums));
  TKC_TRY(cudaGetLastError());
  TKC_TRY(cudaFreeAsync(w2, st));
  TKC_TRY(cudaFreeAsync(c0, st));
  TKC_TRY(cudaFreeAsync(c1, st));
  TKC_TRY(cudaFreeAsync(sums, st));
  return TKC_OK;
}

static int forward(tkc_ctx *ctx, const float *x, u32 m, float *y) {
  if (m == 0) return TKC_OK;
  TKC_LAUNCH(k_mlp_forward<<<grid_of(m, FT), FT, 0, ctx->stream>>>(x, m, ctx->mlp.wb, y));
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

int ensure_learned_order(tkc_graph *g) {
  tkc_ctx *ctx = g->ctx;
  if (!ctx->mlp.ready) return TKC_EINVAL;
  if (g->learned_order && g->learned_version == ctx->mlp.version) return TKC_OK;
  TKC_RC(ensure_features(g));
  cudaStream_t st = ctx->stream;
  const u32 n = g->n;
  if (!g->learned_order) TKC_TRY(dev_malloc(&g->learned_order, std::max<size_t>(n, 1) * sizeof(u32), st));
  if (n == 0) {
    g->n_src_learned = 0;
    g->learned_version = ctx->mlp.version;
    return TKC_OK;
  }
  float *y = nullptr;
  u32 *key = nullptr, *val = nullptr;
  TKC_TRY(dev_malloc(&y, (size_t)n * sizeof(float), st));
  TKC_TRY(dev_malloc(&key, (size_t)n * sizeof(u32), st));
  TKC_TRY(dev_malloc(&val, (size_t)n * sizeof(u32), st));
  TKC_RC(forward(ctx, g->features, n, y));
  TKC_LAUNCH(k_score_keys<<<grid_of(n), 256, 0, st>>>(y, n, key, val));
  TKC_RC(radix_sort_u32_pairs(key, val, n, 32, st));  // stable: equal predictions keep id order
  TKC_RC(filter_order(g, val, g->learned_order, &g->n_src_learned));
  TKC_TRY(cudaFreeAsync(y, st));
  TKC_TRY(cudaFreeAsync(key, st));
  TKC_TRY(cudaFreeAsync(val, st));
  g->learned_version = ctx->mlp.version;
  return TKC_OK;
}

namespace {
__global__ void k_mark_prefix(const u32 *order, u32 count, uint8_t *mark) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) mark[order[i]] = 1;
}

__global__ void k_unmarked_flags(const u32 *order, u32 n, const uint8_t *mark, u32 *flag) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) flag[i] = !mark[order[i]];
  if (blockIdx.x == 0 && threadIdx.x == 0) flag[n] = 0;
}

__global__ void k_compact_into(const u32 *order, const u32 *pos, u32 n, u32 *out) {
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    if (pos[i + 1] != pos[i]) out[pos[i]] = order[i];
}
}  // namespace

int scan_exclusive_u32(const u32 *in, u32 *out, u64 len, u32 *tmp, cudaStream_t st);

// Seeded order: the `prefix` sources the model predicts closest first (they
// are searched without cutting and set x from exact farness), then every
// other source in the degree order.
int ensure_seeded_order(tkc_graph *g, u32 prefix, bool nb) {
  tkc_ctx *ctx = g->ctx;
  TKC_RC(ensure_learned_order(g));
  TKC_RC(ensure_degree_order(g));
  if (nb && !g->nb_order) return TKC_EINVAL;
  prefix = std::min(prefix, g->n_src_learned);
  const int base_kind = nb ? 1 : 0;
  if (g->seeded_order && g->seeded_version == ctx->mlp.version && g->seeded_prefix == prefix &&
      g->seeded_base == base_kind && (!nb || g->seeded_nb_cap == g->nb_cap))
    return TKC_OK;
  cudaStream_t st = ctx->stream;
  const u32 *base = nb ? g->nb_order : g->deg_order;
  const u32 ns = nb ? g->n_src_nb : g->n_src_deg;
  if (!g->seeded_order) TKC_TRY(dev_malloc(&g->seeded_order, std::max<size_t>(g->n, 1) * sizeof(u32), st));
  uint8_t *mark = nullptr;
  u32 *pos = nullptr, *tmp = nullptr;
  TKC_TRY(dev_malloc(&mark, std::max<size_t>(g->n, 1), st));
  TKC_TRY(dev_malloc(&pos, ((size_t)ns + 1) * sizeof(u32), st));
  TKC_TRY(dev_malloc(&tmp, ((size_t)ns + 1) / 4096 * sizeof(u32) + 16, st));
  TKC_TRY(cudaMemsetAsync(mark, 0, std::max<size_t>(g->n, 1), st));
  if (prefix) {
    TKC_LAUNCH(k_mark_prefix<<<grid_of(prefix), 256, 0, st>>>(g->learned_order, prefix, mark));
    TKC_TRY(cudaMemcpyAsync(g->seeded_order, g->learned_order, prefix * sizeof(u32), cudaMemcpyDeviceToDevice, st));
  }
  TKC_LAUNCH(k_unmarked_flags<<<grid_of(ns + 1), 256, 0, st>>>(base, ns, mark, pos));
  TKC_RC(scan_exclusive_u32(pos, pos, (u64)ns + 1, tmp, st));
  TKC_LAUNCH(k_compact_into<<<grid_of(ns), 256, 0, st>>>(base, pos, ns, g->seeded_order + prefix));
  TKC_TRY(cudaGetLastError());
  TKC_TRY(cudaFreeAsync(mark, st));
  TKC_TRY(cudaFreeAsync(pos, st));
  TKC_TRY(cudaFreeAsync(tmp, st));
  TKC_TRY(cudaStreamSynchronize(st));
  g->seeded_version = ctx->mlp.version;
  g->seeded_prefix = prefix;
  g->seeded_base = base_kind;
  g->seeded_nb_cap = nb ? g->nb_cap : 0;
  return TKC_OK;
}

}  // namespace tkc

using namespace tkc;

extern "C" {

int tkc_mlp_init(tkc_ctx *ctx, uint64_t seed) {
  if (!ctx) return TKC_EINVAL;
  TKC_RC(enter(ctx));
  TKC_RC(ensure_mlp(ctx));
  TKC_LAUNCH(k_mlp_init<<<grid_of(P), 256, 0, ctx->stream>>>(ctx->mlp.w, seed));
  TKC_LAUNCH(k_to_bf16<<<grid_of(P), 256, 0, ctx->stream>>>(ctx->mlp.w, ctx->mlp.wb));
  TKC_RC(reset_adam(ctx));
  TKC_TRY(cudaStreamSynchronize(ctx->stream));
  return TKC_OK;
}

int tkc_set_source_model(tkc_ctx *ctx, const float *params, uint32_t nparams) {
  if (!ctx || !params || nparams != (uint32_t)P) return TKC_EINVAL;
  TKC_RC(enter(ctx));
  TKC_RC(ensure_mlp(ctx));
  TKC_TRY(cudaMemcpyAsync(ctx->mlp.w, params, P * sizeof(float), cudaMemcpyHostToDevice, ctx->stream));
  TKC_LAUNCH(k_to_bf16<<<grid_of(P), 256, 0, ctx->stream>>>(ctx->mlp.w, ctx->mlp.wb));
  TKC_RC(reset_adam(ctx));
  TKC_TRY(cudaStreamSynchronize(ctx->stream));
  return TKC_OK;
}

int tkc_get_source_model(tkc_ctx *ctx, float *params, uint32_t nparams) {
  if (!ctx || !params || nparams != (uint32_t)P || !ctx->mlp.ready) return TKC_EINVAL;
  TKC_RC(enter(ctx));
  TKC_TRY(cudaMemcpyAsync(params, ctx->mlp.w, P * sizeof(float), cudaMemcpyDeviceToHost, ctx->stream));
  TKC_TRY(cudaStreamSynchronize(ctx->stream));
  return TKC_OK;
}

int tkc_vertex_features(tkc_graph *g, float *x) {
  if (!g || (!x && g->n)) return TKC_EINVAL;
  TKC_RC(enter(g->ctx));
  TKC_RC(ensure_features(g));
  if (g->n)
    TKC_TRY(cudaMemcpyAsync(x, g->features, (size_t)g->n * F * sizeof(float), cudaMemcpyDeviceToDevice,
                            g->ctx->stream));
  TKC_TRY(cudaStreamSynchronize(g->ctx->stream));
  return TKC_OK;
}

int tkc_mlp_forward(tkc_ctx *ctx, const float *x, uint32_t m, float *y) {
  if (!ctx || (m && (!x || !y)) || !ctx->mlp.ready) return TKC_EINVAL;
  TKC_RC(enter(ctx));
  TKC_RC(forward(ctx, x, m, y));
  TKC_TRY(cudaStreamSynchronize(ctx->stream));
  return TKC_OK;
}

// The gradient into `grad` (device); the loss stays in the model's loss word.
static int gradient(tkc_ctx *ctx, const float *x, const float *t, u32 m, float *grad) {
  cudaStream_t st = ctx->stream;
  MlpState &s = ctx->mlp;
  // a tile per block, at most a block per SM
  const unsigned blocks = (unsigned)std::min<u64>(((u64)m + TS - 1) / TS, (u64)ctx->num_sms);
  TKC_LAUNCH(k_mlp_grad<<<blocks, kGradTPB, 0, st>>>(x, t, m, s.wb, s.part, s.lossp));
  cudaLaunchAttribute early = {};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((P + 31) / 32);
  cfg.blockDim = dim3(32 * kSumWarps);
  cfg.stream = st;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  note_launches(1);
  TKC_TRY(cudaLaunchKernelEx(&cfg, k_mlp_sum, (const float *)s.part, (const double *)s.lossp, (u32)blocks, grad, s.loss));
  TKC_TRY(cudaGetLastError());
  return TKC_OK;
}

// Waits for the stream; the loss into *loss (may be null).
static int finish_step(tkc_ctx *ctx, float *loss) {
  double l = 0.0;
  if (!loss) {
    TKC_TRY(cudaStreamSynchronize(ctx->stream));
    return TKC_OK;
  }
  TKC_TRY(read_back(&l, ctx->mlp.loss, sizeof(double), ctx->stream));
  *loss = (float)l;
  return TKC_OK;
}

int tkc_mlp_gradient(tkc_ctx *ctx, const float *x, const float *t, uint32_t m, float *grad, float *loss) {
  if (!ctx || !x || !t || !grad || m == 0 || !ctx->mlp.ready) return TKC_EINVAL;
  TKC_RC(enter(ctx));
  TKC_RC(gradient(ctx, x, t, m, grad));
  return finish_step(ctx, loss);
}

int tkc_mlp_train_step(tkc_ctx *ctx, const float *x, const float *t, uint32_t m, float lr, float *loss) {
  if (!ctx || !x || !t || m == 0 || !ctx->mlp.ready || !(lr > 0.f)) return TKC_EINVAL;
  TKC_RC(enter(ctx));
  MlpState &s = ctx->mlp;
  TKC_RC(gradient(ctx, x, t, m, s.grad));
  s.step++;
  const double b1 = 0.9, b2 = 0.999;
  float c1 = (float)(1.0 - pow(b1, (double)s.step)), c2 = (float)(1.0 - pow(b2, (double)s.step));
  TKC_LAUNCH(k_adam<<<grid_of(P), 256, 0, ctx->stream>>>(s.w, s.wb, s.m, s.v, s.grad, lr, (float)b1, (float)b2, c1,
                                                         c2, 1e-8f));
  TKC_TRY(cudaGetLastError());
  s.version++;
  return finish_step(ctx, loss);
}

}  // extern "C"
