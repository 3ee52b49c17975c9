// Learned task-cost model: a small MLP trained on the GPU from per-unit timings.
//
// The paper balances load by over-decomposition and dynamic task scheduling
// (Sec. 3.2) and notes that nonuniform blocking makes block work vary several-fold
// (Sec. 4.4, Table 1). Here the work units are packed statically onto persistent
// CTAs, longest first, so the packing is only as good as the cost estimates. The
// flop count misjudges units made of small or ragged tiles (padding, per-block
// recombination and pipeline overheads do not scale with flops); this MLP learns the
// measured cost of a unit from its features, and bsmm_plan_predict_costs feeds its
// predictions to the packer. Results never depend on it: only the order changes.
//
// Model (F = BSMM_NFEATURES inputs, H = 32): features standardised with stored means
// and deviations, two tanh layers, one linear output = standardised log time.
// Parameters in one float vector: W1[H][F], b1[H], W2[H][H], b2[H], w3[H], b3.
// Training: full-batch mean squared error, Adam; every reduction over samples runs in
// a fixed order (partial sums over tiles of 128 samples, then a sum over the tiles in tile
// order), so training is bit-for-bit reproducible.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "bsmm_internal.h"

using namespace bsmm;

namespace {

constexpr int F = BSMM_NFEATURES;
constexpr int H = 32;
constexpr int NP = H * F + H + H * H + H + H + 1;
constexpr int OW1 = 0, OB1 = H * F, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H, OB3 = OW3 + H;
constexpr int TILE = 128;  // samples per partial sum of the gradient

struct Norm {
  float xmu[F], xsd[F];
  float ymu, ysd;
};

__device__ __forceinline__ void mlp_forward_one(const float* __restrict__ w, const float* x, float* h1, float* h2,
                                                float& y) {
#pragma unroll 4
  for (int j = 0; j < H; j++) {
    float z = w[OB1 + j];
#pragma unroll
    for (int f = 0; f < F; f++) z = fmaf(w[OW1 + j * F + f], x[f], z);
    h1[j] = tanhf(z);
  }
#pragma unroll 4
  for (int j = 0; j < H; j++) {
    float z = w[OB2 + j];
    for (int i = 0; i < H; i++) z = fmaf(w[OW2 + j * H + i], h1[i], z);
    h2[j] = tanhf(z);
  }
  float o = w[OB3];
  for (int i = 0; i < H; i++) o = fmaf(w[OW3 + i], h2[i], o);
  y = o;
}

__global__ void mlp_predict_kernel(const float* __restrict__ params, Norm nm, const float* __restrict__ X, int64_t n,
                                   float* __restrict__ y) {
  __shared__ float w[NP];
  for (int p = threadIdx.x; p < NP; p += blockDim.x) w[p] = params[p];
  __syncthreads();
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  float x[F], h1[H], h2[H], o;
#pragma unroll
  for (int f = 0; f < F; f++) x[f] = (X[s * F + f] - nm.xmu[f]) / nm.xsd[f];
  mlp_forward_one(w, x, h1, h2, o);
  y[s] = o * nm.ysd + nm.ymu;  // log time in the caller's units
}

// Training: one cooperative launch for every step of a fit. Per step, CTAs take tiles of
// TILE samples (forward, backward, the tile's gradient sums in sample order, written to
// part[tile][0..NP], entry NP the sum of squared residuals); after a grid barrier each CTA
// adds a few parameters' partial sums in tile order and applies Adam; after a second barrier
// the next step reads the new parameters.
// A step is a chain of latencies (20000 samples are 12 MFLOP per layer pass), so the layout
// serves those and the shared-memory port, which all 16 warps share: a warp takes 8 samples
// through the whole network, lane = neuron, the neuron's weights in registers and the
// samples' activations read by broadcast, so no barrier is needed before the gradient sums;
// those take 2 x 4 parameters per thread; a parameter's partial sums are fetched by the
// whole CTA at once, and its Adam state stays in its thread. Every sum keeps one order.
// 20000 samples: 22 us per step (the network and its sums 7.5 us per tile, which is what
// their shared-memory reads take; 157 tiles on 152 SMs; a barrier 2 us). As three launches
// per step, with a thread per sample striding through its own rows of shared memory (32-way
// conflicts) and 128 threads for the 1506 gradient sums: 95 us.
constexpr int kTrainThreads = 512;
constexpr int kWarpSamples = TILE / (kTrainThreads / 32);  // 8
constexpr int LD = H + 4;        // row of neurons, padded: 8 rows cover the banks
constexpr int kGather = 4096;    // partial sums fetched at a time
constexpr int kKeep = 2;         // tiles of a CTA whose standardised inputs stay in shared memory
constexpr int64_t kBarrierNs = 4000000000LL;  // bounded wait at a grid barrier
constexpr int kNPpad = (NP + 3) / 4 * 4;      // parameter arrays hold whole 16-byte vectors

struct TrainShared {
  float w1[kNPpad];              // every parameter, as in global memory ...
  float w2[H][LD];               // ... and W2 again in padded rows
  float xs[kKeep][TILE][F];
  float ts[kKeep][TILE];
  float h1[TILE][LD], h2[TILE][LD], d1[TILE][LD], d2[TILE][LD];
  float dy[TILE], r2[TILE];
  float gather[kGather];
};

__device__ __forceinline__ int64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return (int64_t)t;
}

// A grid barrier's words: sync[0] counts arrivals (it only grows, by gridDim.x per barrier),
// sync[1] is the error flag. `missing` is 0, or an arrival that the self-test waits for in
// vain.
struct Barrier {
  unsigned* sync;
  unsigned missing;
  int64_t limit_ns;
};

// Every CTA of the (cooperative) grid arrives; false when the wait ran out, here or in
// another CTA. One thread reads the flag for all: read by each of them, it could change in
// between, and a part of the CTA would leave the kernel while the rest went on to the next
// step's barriers.
__device__ bool grid_barrier(const Barrier& b, unsigned arrivals) {
  unsigned* const sync = b.sync;
  const unsigned target = arrivals + b.missing;
  bool ok = true;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&sync[0], 1u);
    const int64_t t0 = now_ns();
    unsigned spin = 0;
    while ((int)(*(volatile unsigned*)&sync[0] - target) < 0) {  // (the count may wrap)
      if (*(volatile unsigned*)&sync[1]) break;
      if ((++spin & 1023u) == 0 && now_ns() - t0 > b.limit_ns) {
        atomicExch(&sync[1], 1u);
        break;
      }
    }
    __threadfence();
    ok = *(volatile unsigned*)&sync[1] == 0u;
  }
  return __syncthreads_and(ok);
}

// Sums over the tile's samples, in sample order: g[j][i] = sum a[q][j0 + j] b[q][i0 + i]
template <int LDB>
__device__ __forceinline__ void outer_sums(const float (*a)[LD], int j0, const float (*b)[LDB], int i0,
                                           float (&g)[2][4]) {
#pragma unroll
  for (int j = 0; j < 2; j++)
#pragma unroll
    for (int i = 0; i < 4; i++) g[j][i] = 0.0f;
#pragma unroll 4
  for (int q = 0; q < TILE; q++) {
    const float2 av = *reinterpret_cast<const float2*>(&a[q][j0]);
    const float4 bv = *reinterpret_cast<const float4*>(&b[q][i0]);
    g[0][0] = fmaf(av.x, bv.x, g[0][0]);
    g[0][1] = fmaf(av.x, bv.y, g[0][1]);
    g[0][2] = fmaf(av.x, bv.z, g[0][2]);
    g[0][3] = fmaf(av.x, bv.w, g[0][3]);
    g[1][0] = fmaf(av.y, bv.x, g[1][0]);
    g[1][1] = fmaf(av.y, bv.y, g[1][1]);
    g[1][2] = fmaf(av.y, bv.z, g[1][2]);
    g[1][3] = fmaf(av.y, bv.w, g[1][3]);
  }
}
__device__ __forceinline__ float column_sum(const float (*a)[LD], int j) {
  float g = 0.0f;
#pragma unroll 16
  for (int q = 0; q < TILE; q++) g += a[q][j];
  return g;
}
__device__ __forceinline__ float vector_sum(const float* a) {
  float g = 0.0f;
#pragma unroll 4
  for (int q = 0; q < TILE; q += 4) {
    const float4 v = *reinterpret_cast<const float4*>(a + q);
    g += v.x;
    g += v.y;
    g += v.z;
    g += v.w;
  }
  return g;
}

// One tile's partial sums: out[0..NP]; slot: where its inputs are (or go)
__device__ void train_tile(TrainShared& sm, const Norm& nm, const float* __restrict__ X, const float* __restrict__ t,
                           int64_t n, int tile, int slot, bool kept, float* __restrict__ out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int q0 = warp * kWarpSamples;  // this warp's samples
  const int64_t s0 = (int64_t)tile * TILE;
  float(*const xs)[F] = sm.xs[slot];
  float* const ts = sm.ts[slot];
  if (!kept) {  // standardised inputs and targets of the warp's samples
    for (int e = lane; e < kWarpSamples * F; e += 32) {
      const int f = e % F, q = q0 + e / F;
      xs[q][f] = s0 + q < n ? (X[(s0 + q) * F + f] - nm.xmu[f]) / nm.xsd[f] : 0.0f;
    }
    if (lane < kWarpSamples) ts[q0 + lane] = s0 + q0 + lane < n ? (t[s0 + q0 + lane] - nm.ymu) / nm.ysd : 0.0f;
    __syncwarp();
  }
  const float* const w = sm.w1;
  float h1[kWarpSamples], h2[kWarpSamples];
  {
    float wr[F], z[kWarpSamples];
#pragma unroll
    for (int f = 0; f < F; f += 4) *reinterpret_cast<float4*>(wr + f) = *reinterpret_cast<const float4*>(w + OW1 + lane * F + f);
#pragma unroll
    for (int u = 0; u < kWarpSamples; u++) z[u] = w[OB1 + lane];
#pragma unroll
    for (int f = 0; f < F; f += 4)
#pragma unroll
      for (int u = 0; u < kWarpSamples; u++) {
        const float4 x = *reinterpret_cast<const float4*>(&xs[q0 + u][f]);
        z[u] = fmaf(wr[f], x.x, z[u]);
        z[u] = fmaf(wr[f + 1], x.y, z[u]);
        z[u] = fmaf(wr[f + 2], x.z, z[u]);
        z[u] = fmaf(wr[f + 3], x.w, z[u]);
      }
#pragma unroll
    for (int u = 0; u < kWarpSamples; u++) {
      h1[u] = s0 + q0 + u < n ? tanhf(z[u]) : 0.0f;
      sm.h1[q0 + u][lane] = h1[u];
    }
  }
  __syncwarp();
  {
    float z[kWarpSamples];
#pragma unroll
    for (int u = 0; u < kWarpSamples; u++) z[u] = w[OB2 + lane];
#pragma unroll
    for (int i = 0; i < H; i += 4) {
      const float4 wr = *reinterpret_cast<const float4*>(&sm.w2[lane][i]);
#pragma unroll
      for (int u = 0; u < kWarpSamples; u++) {
        const float4 h = *reinterpret_cast<const float4*>(&sm.h1[q0 + u][i]);
        z[u] = fmaf(wr.x, h.x, z[u]);
        z[u] = fmaf(wr.y, h.y, z[u]);
        z[u] = fmaf(wr.z, h.z, z[u]);
        z[u] = fmaf(wr.w, h.w, z[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < kWarpSamples; u++) {
      h2[u] = s0 + q0 + u < n ? tanhf(z[u]) : 0.0f;
      sm.h2[q0 + u][lane] = h2[u];
    }
  }
  __syncwarp();
  float dy = 0.0f;
  if (lane < kWarpSamples) {  // lane = sample: the output and its residual
    const int q = q0 + lane;
    float o = w[OB3];
#pragma unroll
    for (int i = 0; i < H; i += 4) {
      const float4 h = *reinterpret_cast<const float4*>(&sm.h2[q][i]);
      o = fmaf(w[OW3 + i], h.x, o);
      o = fmaf(w[OW3 + i + 1], h.y, o);
      o = fmaf(w[OW3 + i + 2], h.z, o);
      o = fmaf(w[OW3 + i + 3], h.w, o);
    }
    const float r = o - ts[q];
    const bool in = s0 + q < n;
    dy = in ? 2.0f * r / (float)n : 0.0f;
    sm.dy[q] = dy;
    sm.r2[q] = in ? r * r : 0.0f;
  }
  {
    const float w3 = w[OW3 + lane];
#pragma unroll
    for (int u = 0; u < kWarpSamples; u++) {
      const float d = __shfl_sync(0xffffffffu, dy, u);
      sm.d2[q0 + u][lane] = s0 + q0 + u < n ? d * w3 * (1.0f - h2[u] * h2[u]) : 0.0f;
    }
  }
  __syncwarp();
  {
    float g[kWarpSamples];
#pragma unroll
    for (int u = 0; u < kWarpSamples; u++) g[u] = 0.0f;
#pragma unroll
    for (int j = 0; j < H; j += 4) {
      const float wa = sm.w2[j][lane], wb = sm.w2[j + 1][lane], wc = sm.w2[j + 2][lane], wd = sm.w2[j + 3][lane];
#pragma unroll
      for (int u = 0; u < kWarpSamples; u++) {
        const float4 d = *reinterpret_cast<const float4*>(&sm.d2[q0 + u][j]);
        g[u] = fmaf(wa, d.x, g[u]);
        g[u] = fmaf(wb, d.y, g[u]);
        g[u] = fmaf(wc, d.z, g[u]);
        g[u] = fmaf(wd, d.w, g[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < kWarpSamples; u++)
      sm.d1[q0 + u][lane] = s0 + q0 + u < n ? g[u] * (1.0f - h1[u] * h1[u]) : 0.0f;
  }
  __syncthreads();
  // gradient sums over the tile's samples: warps 0-3 W2, 4-5 W1, 6-8 the single rows, 9 the rest
  if (warp < 4) {
    const int j = 2 * (warp * 4 + (lane >> 3)), i = 4 * (lane & 7);
    float g[2][4];
    outer_sums(sm.d2, j, sm.h1, i, g);
#pragma unroll
    for (int u = 0; u < 8; u++) out[OW2 + (j + u / 4) * H + i + u % 4] = g[u / 4][u % 4];
  } else if (warp < 6) {
    const int e = tid - 128;
    if (e < 48) {
      const int j = 2 * (e / 3), f = 4 * (e % 3);
      float g[2][4];
      outer_sums(sm.d1, j, xs, f, g);
#pragma unroll
      for (int u = 0; u < 8; u++) out[OW1 + (j + u / 4) * F + f + u % 4] = g[u / 4][u % 4];
    }
  } else if (warp == 6) {
    out[OB1 + lane] = column_sum(sm.d1, lane);
  } else if (warp == 7) {
    out[OB2 + lane] = column_sum(sm.d2, lane);
  } else if (warp == 8) {
    float g = 0.0f;
#pragma unroll 16
    for (int q = 0; q < TILE; q++) g = fmaf(sm.dy[q], sm.h2[q][lane], g);
    out[OW3 + lane] = g;
  } else if (warp == 9) {
    if (lane < 2) out[OB3 + lane] = vector_sum(lane ? sm.r2 : sm.dy);  // OB3, then NP: the residuals
  }
  __syncthreads();
}
static_assert(OB3 + 1 == NP, "the residual sum follows the last parameter");

// `total` passes over the samples; the first `updates` of them end in an Adam step, the
// others leave the gradient (and grad[NP] = the mean squared residual) in grad.
__global__ void __launch_bounds__(kTrainThreads, 1) mlp_train_kernel(float* params, float* m, float* v, float* grad,
                                                                  float* part, const __grid_constant__ Norm nm,
                                                                  const float* __restrict__ X,
                                                                  const float* __restrict__ t, int64_t n, int tiles,
                                                                  int total, int updates, float lr, Barrier bar) {
  extern __shared__ __align__(16) unsigned char raw[];
  TrainShared& sm = *reinterpret_cast<TrainShared*>(raw);
  const int tid = threadIdx.x, G = gridDim.x;
  const int per = (NP + 1 + G - 1) / G;  // parameters whose sums this CTA adds
  const int p0 = blockIdx.x * per, np = max(0, min(per, NP + 1 - p0));
  double b1k = 1.0, b2k = 1.0;
  float mp = 0.0f, vp = 0.0f, pp = 0.0f;  // the parameter and Adam state of a thread that owns one
  const bool own = np <= kTrainThreads;
  if (own && tid < np && p0 + tid < NP) {
    mp = m[p0 + tid];
    vp = v[p0 + tid];
    pp = params[p0 + tid];
  }
  for (int it = 0; it < total; it++) {
    if (tid < kNPpad / 4) {
      const float4 w4 = __ldcg(reinterpret_cast<const float4*>(params) + tid);
      reinterpret_cast<float4*>(sm.w1)[tid] = w4;
      const int e = 4 * tid - OW2;  // (OW2 and H are multiples of 4)
      if (e >= 0 && e < H * H) *reinterpret_cast<float4*>(&sm.w2[e / H][e % H]) = w4;
    }
    __syncthreads();
    const bool keep = tiles <= kKeep * G;
    for (int tile = blockIdx.x, k = 0; tile < tiles; tile += G, k++)
      train_tile(sm, nm, X, t, n, tile, keep ? k : 0, keep && it > 0, part + (int64_t)tile * (NP + 1));
    if (!grid_barrier(bar, (unsigned)(2 * it + 1) * G)) return;
    // sums over the tiles in tile order: the CTA fetches a batch of its parameters' partial
    // sums at once, then a thread per parameter adds them
    const bool update = it < updates;
    if (update) {
      b1k = __dmul_rn(b1k, 0.9);
      b2k = __dmul_rn(b2k, 0.999);
    }
    for (int pb = 0; pb < np; pb += kTrainThreads) {
      const int cnt = min(kTrainThreads, np - pb);
      int sh = 4;  // cnt <= 2^sh <= kTrainThreads
      while ((1 << sh) < cnt) sh++;
      const int batch = kGather >> sh;  // tiles fetched at a time: kGather / kTrainThreads loads per thread
      const int gp = tid & ((1 << sh) - 1), bt = tid >> sh;
      const float* const src = part + p0 + pb + gp;
      float g = 0.0f;
      for (int b0 = 0; b0 < tiles; b0 += batch) {
        const int nb = min(batch, tiles - b0);
        float x[kGather / kTrainThreads];
#pragma unroll
        for (int u = 0; u < kGather / kTrainThreads; u++) {
          const int b = bt + u * (kTrainThreads >> sh);
          x[u] = gp < cnt && b < nb ? __ldcg(src + (int64_t)(b0 + b) * (NP + 1)) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < kGather / kTrainThreads; u++) sm.gather[((bt + u * (kTrainThreads >> sh)) << sh) + gp] = x[u];
        __syncthreads();
        if (tid < cnt)
#pragma unroll 16
          for (int b = 0; b < nb; b++) g += sm.gather[(b << sh) + tid];
        __syncthreads();
      }
      const int p = p0 + pb + tid;
      if (tid < cnt) {
        if (!update) {
          grad[p] = p == NP ? g / (float)n : g;
        } else if (p < NP) {
          const float c1 = (float)__dsub_rn(1.0, b1k), c2 = (float)__dsub_rn(1.0, b2k);
          const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
          if (!own) {
            mp = m[p];
            vp = v[p];
            pp = params[p];
          }
          const float mm = b1 * mp + (1.0f - b1) * g;
          const float vv = b2 * vp + (1.0f - b2) * g * g;
          pp -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
          m[p] = mp = mm;
          v[p] = vp = vv;
          params[p] = pp;
        }
      }
    }
    if (it + 1 < total && !grid_barrier(bar, (unsigned)(2 * it + 2) * G)) return;
  }
}

uint64_t splitmix64(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

double normal(uint64_t& s) {  // Box-Muller on two 53-bit uniforms
  const double u1 = ((splitmix64(s) >> 11) + 1.0) * 0x1.0p-53;
  const double u2 = (splitmix64(s) >> 11) * 0x1.0p-53;
  return std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2);
}

}  // namespace

struct bsmm_mlp_s {
  Norm norm{};
  int64_t step = 0;
  // params, m, v (kNPpad floats each), grad (NP + 1, padded alike) and the barrier's words in
  // one allocation, owned by params
  DevBuf params, m, v, grad, sync, part;
};

namespace {

bsmm_status mlp_alloc(DevBuf& b, size_t bytes) {
  if (b.p && b.bytes >= bytes) return BSMM_OK;
  if (b.p) cudaFree(b.p);
  b.p = nullptr;
  b.bytes = 0;
  cudaError_t e = cudaMalloc(&b.p, bytes ? bytes : 16);
  if (e != cudaSuccess) {
    b.p = nullptr;
    return set_error(std::string("cudaMalloc: ") + cudaGetErrorString(e)),
           e == cudaErrorMemoryAllocation ? BSMM_ERR_NOMEM : BSMM_ERR_CUDA;
  }
  b.bytes = bytes ? bytes : 16;
  return BSMM_OK;
}

// `total` passes over the samples, the first `updates` of them Adam steps (see
// mlp_train_kernel). The grid's CTAs wait for one another, so the launch is cooperative and
// no larger than what is resident at once.
bsmm_status train(bsmm_mlp_s* mlp, const float* X, const float* t, int64_t n, int total, int updates, float lr,
                  cudaStream_t st, unsigned missing = 0, int64_t limit_ns = kBarrierNs) {
  const int64_t tiles64 = (n + TILE - 1) / TILE;
  if (tiles64 > (1 << 30)) return set_error("too many samples"), BSMM_ERR_INVALID;
  int tiles = (int)tiles64;
  const bsmm_status s = mlp_alloc(mlp->part, sizeof(float) * (size_t)tiles * (NP + 1));
  if (s != BSMM_OK) return s;
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainShared));
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mlp_train_kernel, kTrainThreads, sizeof(TrainShared));
  if (e == cudaSuccess) e = cudaMemsetAsync(mlp->sync.p, 0, 2 * sizeof(unsigned), st);
  if (e == cudaSuccess) {
    const int grid = std::max(1, std::min(tiles, sms * std::max(1, per_sm)));
    float *params = (float*)mlp->params.p, *m = (float*)mlp->m.p, *v = (float*)mlp->v.p, *grad = (float*)mlp->grad.p;
    float* part = (float*)mlp->part.p;
    Barrier bar{(unsigned*)mlp->sync.p, missing, limit_ns};
    void* args[] = {&params, &m, &v, &grad, &part, &mlp->norm, &X, &t, &n, &tiles, &total, &updates, &lr, &bar};
    e = cudaLaunchCooperativeKernel((const void*)mlp_train_kernel, dim3(grid), dim3(kTrainThreads), args,
                                    sizeof(TrainShared), st);
  }
  if (e != cudaSuccess) return set_error(std::string("mlp kernels: ") + cudaGetErrorString(e)), BSMM_ERR_CUDA;
  return BSMM_OK;
}

// After a copy of the launch's outputs has been waited for: did a grid barrier run out?
bsmm_status barrier_status(unsigned flag) {
  if (flag) return set_error("mlp training: a grid barrier timed out"), BSMM_ERR_TIMEOUT;
  return BSMM_OK;
}

// bsmm_mlp_fit (`missing` and `limit_ns`: see Barrier)
bsmm_status fit(bsmm_mlp_s* mlp, const float* X, const float* t, int64_t n, int32_t steps, float lr,
                float* final_loss, void* stream, unsigned missing, int64_t limit_ns) {
  if (!mlp || !X || !t || n <= 0 || steps < 0 || !(lr > 0.0f)) return set_error("bad arguments"), BSMM_ERR_INVALID;
  cudaStream_t st = (cudaStream_t)stream;
  // standardisation from the data (host, FP64 sums in sample order)
  std::vector<float> hx((size_t)n * F), ht(n);
  if (cudaMemcpyAsync(hx.data(), X, sizeof(float) * hx.size(), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaMemcpyAsync(ht.data(), t, sizeof(float) * ht.size(), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return set_error("copy failed"), BSMM_ERR_CUDA;
  {
    // (the features side by side: their sums are independent chains, each in sample order)
    double s1[F] = {}, s2[F] = {}, mu[F];
    for (int64_t i = 0; i < n; i++)
      for (int f = 0; f < F; f++) s1[f] += hx[i * F + f];
    for (int f = 0; f < F; f++) mu[f] = s1[f] / n;
    for (int64_t i = 0; i < n; i++)
      for (int f = 0; f < F; f++) s2[f] += (hx[i * F + f] - mu[f]) * (hx[i * F + f] - mu[f]);
    for (int f = 0; f < F; f++) {
      const double sd = std::sqrt(s2[f] / n);
      mlp->norm.xmu[f] = (float)mu[f];
      mlp->norm.xsd[f] = sd > 0 ? (float)sd : 1.0f;
    }
  }
  {
    double s1 = 0, s2 = 0;
    for (int64_t i = 0; i < n; i++) s1 += ht[i];
    const double mu = s1 / n;
    for (int64_t i = 0; i < n; i++) s2 += (ht[i] - mu) * (ht[i] - mu);
    const double sd = std::sqrt(s2 / n);
    mlp->norm.ymu = (float)mu;
    mlp->norm.ysd = sd > 0 ? (float)sd : 1.0f;
  }
  if (cudaMemsetAsync(mlp->m.p, 0, sizeof(float) * NP, st) != cudaSuccess ||
      cudaMemsetAsync(mlp->v.p, 0, sizeof(float) * NP, st) != cudaSuccess)
    return set_error("memset failed"), BSMM_ERR_CUDA;
  const int total = steps + (final_loss ? 1 : 0);
  if (total == 0) return BSMM_OK;
  const bsmm_status s = train(mlp, X, t, n, total, steps, lr, st, missing, limit_ns);
  if (s != BSMM_OK) return s;
  // (also when no loss is asked for: a training that was cut short is never taken for a whole one)
  unsigned flag = 0;
  if ((final_loss && cudaMemcpyAsync(final_loss, (float*)mlp->grad.p + NP, sizeof(float), cudaMemcpyDeviceToHost, st) !=
                         cudaSuccess) ||
      cudaMemcpyAsync(&flag, (unsigned*)mlp->sync.p + 1, sizeof(flag), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return set_error("copy failed"), BSMM_ERR_CUDA;
  return barrier_status(flag);
}

}  // namespace

extern "C" {

bsmm_status bsmm_mlp_create(bsmm_mlp_t* out, uint64_t seed) {
  if (!out) return set_error("out is NULL"), BSMM_ERR_INVALID;
  *out = nullptr;
  bsmm_mlp_s* mlp = new (std::nothrow) bsmm_mlp_s();
  if (!mlp) return set_error("out of host memory"), BSMM_ERR_NOMEM;
  std::vector<float> p(NP, 0.0f);
  uint64_t s = seed;
  for (int i = 0; i < H * F; i++) p[OW1 + i] = (float)(normal(s) / std::sqrt((double)F));
  for (int i = 0; i < H * H; i++) p[OW2 + i] = (float)(normal(s) / std::sqrt((double)H));
  for (int i = 0; i < H; i++) p[OW3 + i] = (float)(normal(s) / std::sqrt((double)H));
  for (int f = 0; f < F; f++) {
    mlp->norm.xmu[f] = 0.0f;
    mlp->norm.xsd[f] = 1.0f;
  }
  mlp->norm.ymu = 0.0f;
  mlp->norm.ysd = 1.0f;
  constexpr size_t kArray = sizeof(float) * (kNPpad + 4);
  const bsmm_status st = mlp_alloc(mlp->params, 4 * kArray + 16);
  if (st != BSMM_OK) {
    bsmm_mlp_destroy(mlp);
    return st;
  }
  unsigned char* const base = (unsigned char*)mlp->params.p;
  mlp->m.p = base + kArray;
  mlp->v.p = base + 2 * kArray;
  mlp->grad.p = base + 3 * kArray;
  mlp->sync.p = base + 4 * kArray;
  if (cudaMemset(mlp->params.p, 0, 4 * kArray + 16) != cudaSuccess ||
      cudaMemcpy(mlp->params.p, p.data(), sizeof(float) * NP, cudaMemcpyHostToDevice) != cudaSuccess) {
    bsmm_mlp_destroy(mlp);
    return set_error("mlp initialisation copy failed"), BSMM_ERR_CUDA;
  }
  *out = mlp;
  return BSMM_OK;
}

int32_t bsmm_mlp_num_params(void) { return NP; }

bsmm_status bsmm_mlp_set_params(bsmm_mlp_t mlp, const float* params, int64_t n) {
  if (!mlp || !params || n != NP) return set_error("bad arguments (n must be bsmm_mlp_num_params())"), BSMM_ERR_INVALID;
  if (cudaMemcpy(mlp->params.p, params, sizeof(float) * NP, cudaMemcpyHostToDevice) != cudaSuccess)
    return set_error("copy failed"), BSMM_ERR_CUDA;
  return BSMM_OK;
}

bsmm_status bsmm_mlp_get_params(bsmm_mlp_t mlp, float* params, int64_t n) {
  if (!mlp || !params || n != NP) return set_error("bad arguments (n must be bsmm_mlp_num_params())"), BSMM_ERR_INVALID;
  if (cudaMemcpy(params, mlp->params.p, sizeof(float) * NP, cudaMemcpyDeviceToHost) != cudaSuccess)
    return set_error("copy failed"), BSMM_ERR_CUDA;
  return BSMM_OK;
}

bsmm_status bsmm_mlp_set_norm(bsmm_mlp_t mlp, const float* xmu, const float* xsd, float ymu, float ysd) {
  if (!mlp || !xmu || !xsd || !(ysd > 0.0f)) return set_error("bad arguments"), BSMM_ERR_INVALID;
  for (int f = 0; f < F; f++) {
    if (!(xsd[f] > 0.0f)) return set_error("deviations must be > 0"), BSMM_ERR_INVALID;
    mlp->norm.xmu[f] = xmu[f];
    mlp->norm.xsd[f] = xsd[f];
  }
  mlp->norm.ymu = ymu;
  mlp->norm.ysd = ysd;
  return BSMM_OK;
}

bsmm_status bsmm_mlp_get_norm(bsmm_mlp_t mlp, float* xmu, float* xsd, float* ymu, float* ysd) {
  if (!mlp) return set_error("mlp is NULL"), BSMM_ERR_INVALID;
  for (int f = 0; f < F; f++) {
    if (xmu) xmu[f] = mlp->norm.xmu[f];
    if (xsd) xsd[f] = mlp->norm.xsd[f];
  }
  if (ymu) *ymu = mlp->norm.ymu;
  if (ysd) *ysd = mlp->norm.ysd;
  return BSMM_OK;
}

bsmm_status bsmm_mlp_loss_grad(bsmm_mlp_t mlp, const float* X, const float* t, int64_t n, float* loss, float* grad,
                               void* stream) {
  if (!mlp || !X || !t || n <= 0) return set_error("bad arguments"), BSMM_ERR_INVALID;
  cudaStream_t st = (cudaStream_t)stream;
  bsmm_status s = train(mlp, X, t, n, 1, 0, 0.0f, st);
  if (s != BSMM_OK) return s;
  std::vector<float> g(NP + 1);
  unsigned flag = 0;
  if (cudaMemcpyAsync(g.data(), mlp->grad.p, sizeof(float) * (NP + 1), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaMemcpyAsync(&flag, (unsigned*)mlp->sync.p + 1, sizeof(flag), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return set_error("copy failed"), BSMM_ERR_CUDA;
  if ((s = barrier_status(flag)) != BSMM_OK) return s;
  if (loss) *loss = g[NP];
  if (grad) std::memcpy(grad, g.data(), sizeof(float) * NP);
  return BSMM_OK;
}

bsmm_status bsmm_mlp_fit(bsmm_mlp_t mlp, const float* X, const float* t, int64_t n, int32_t steps, float lr,
                         float* final_loss, void* stream) {
  return fit(mlp, X, t, n, steps, lr, final_loss, stream, 0, kBarrierNs);
}

bsmm_status bsmm_selftest_fit(int64_t limit_ns, int32_t with_loss, void* stream) {
  if (limit_ns < 1000000 || limit_ns > 1000000000) return set_error("limit_ns must be in 1e6..1e9"), BSMM_ERR_INVALID;
  constexpr int64_t n = 3 * TILE;  // three CTAs
  bsmm_mlp_t mlp = nullptr;
  DevBuf d;  // X, then t: all zero
  bsmm_status s = bsmm_mlp_create(&mlp, 1);
  if (s == BSMM_OK) s = mlp_alloc(d, sizeof(float) * n * (F + 1));
  if (s == BSMM_OK && cudaMemsetAsync(d.p, 0, sizeof(float) * n * (F + 1), (cudaStream_t)stream) != cudaSuccess)
    s = (set_error("memset failed"), BSMM_ERR_CUDA);
  float loss = 0.0f;
  const float* const X = (const float*)d.p;
  if (s == BSMM_OK) s = fit(mlp, X, X + n * F, n, 2, 1e-3f, with_loss ? &loss : nullptr, stream, 1, limit_ns);
  bsmm_mlp_destroy(mlp);  // (freeing waits for the kernel)
  if (d.p) cudaFree(d.p);
  return s;
}

bsmm_status bsmm_mlp_predict(bsmm_mlp_t mlp, const float* X, int64_t n, float* y, void* stream) {
  if (!mlp || !X || !y || n < 0) return set_error("bad arguments"), BSMM_ERR_INVALID;
  if (n == 0) return BSMM_OK;
  mlp_predict_kernel<<<(int)((n + 127) / 128), 128, 0, (cudaStream_t)stream>>>((const float*)mlp->params.p,
                                                                               mlp->norm, X, n, y);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return set_error(std::string("predict: ") + cudaGetErrorString(e)), BSMM_ERR_CUDA;
  return BSMM_OK;
}

bsmm_status bsmm_plan_predict_costs(bsmm_plan_t plan, bsmm_mlp_t mlp, void* stream) {
  if (!plan || !mlp) return set_error("NULL argument"), BSMM_ERR_INVALID;
  const int64_t n = plan->n_units;
  if (n == 0) return BSMM_OK;
  cudaStream_t st = (cudaStream_t)stream;
  DevBuf dx, dy;
  bsmm_status s = mlp_alloc(dx, sizeof(float) * (size_t)n * F);
  if (s == BSMM_OK) s = mlp_alloc(dy, sizeof(float) * (size_t)n);
  std::vector<float> y(n);
  if (s == BSMM_OK) {
    if (cudaMemcpyAsync(dx.p, plan->features.data(), sizeof(float) * plan->features.size(), cudaMemcpyHostToDevice, st) !=
        cudaSuccess) {
      set_error("copy failed");
      s = BSMM_ERR_CUDA;
    }
  }
  if (s == BSMM_OK) s = bsmm_mlp_predict(mlp, (const float*)dx.p, n, (float*)dy.p, stream);
  if (s == BSMM_OK &&
      (cudaMemcpyAsync(y.data(), dy.p, sizeof(float) * n, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
       cudaStreamSynchronize(st) != cudaSuccess)) {
    set_error("copy failed");
    s = BSMM_ERR_CUDA;
  }
  if (dx.p) cudaFree(dx.p);
  if (dy.p) cudaFree(dy.p);
  if (s != BSMM_OK) return s;
  std::vector<double> cost(n);
  for (int64_t u = 0; u < n; u++) cost[u] = std::exp(std::min(60.0, std::max(-60.0, (double)y[u])));
  return bsmm_plan_set_costs(plan, cost.data());
}

}  // extern "C"

namespace {

constexpr char kMagic[8] = {'B', 'S', 'M', 'M', 'M', 'L', 'P', '\0'};
constexpr uint32_t kFormatVersion = 1;

// FNV-1a, 64 bits, over a byte string
uint64_t fnv1a(const std::vector<unsigned char>& b) {
  uint64_t h = 1469598103934665603ull;
  for (unsigned char c : b) {
    h ^= c;
    h *= 1099511628211ull;
  }
  return h;
}

template <class T>
void put_raw(std::vector<unsigned char>& b, const T* v, size_t n) {
  const unsigned char* p = reinterpret_cast<const unsigned char*>(v);
  b.insert(b.end(), p, p + sizeof(T) * n);
}

template <class T>
bool get_raw(const std::vector<unsigned char>& b, size_t& pos, T* v, size_t n) {
  if (pos + sizeof(T) * n > b.size()) return false;
  std::memcpy(v, b.data() + pos, sizeof(T) * n);
  pos += sizeof(T) * n;
  return true;
}

}  // namespace

extern "C" {

bsmm_status bsmm_mlp_save(bsmm_mlp_t mlp, const char* path) {
  if (!mlp || !path || !*path) return set_error("NULL model or path"), BSMM_ERR_INVALID;
  std::vector<float> prm(NP);
  bsmm_status st = bsmm_mlp_get_params(mlp, prm.data(), NP);
  if (st != BSMM_OK) return st;
  std::vector<unsigned char> b;
  put_raw(b, kMagic, 8);
  const uint32_t hdr[5] = {kFormatVersion, (uint32_t)BSMM_FEATURE_VERSION, (uint32_t)F, (uint32_t)H, (uint32_t)NP};
  put_raw(b, hdr, 5);
  put_raw(b, prm.data(), NP);
  put_raw(b, mlp->norm.xmu, F);
  put_raw(b, mlp->norm.xsd, F);
  put_raw(b, &mlp->norm.ymu, 1);
  put_raw(b, &mlp->norm.ysd, 1);
  const uint64_t sum = fnv1a(b);
  put_raw(b, &sum, 1);
  const std::string tmp = std::string(path) + ".tmp";
  FILE* f = std::fopen(tmp.c_str(), "wb");
  if (!f) return set_error(std::string("cannot write ") + tmp), BSMM_ERR_INVALID;
  const bool ok = std::fwrite(b.data(), 1, b.size(), f) == b.size();
  if (std::fclose(f) != 0 || !ok || std::rename(tmp.c_str(), path) != 0) {
    std::remove(tmp.c_str());
    return set_error(std::string("cannot write ") + path), BSMM_ERR_INVALID;
  }
  return BSMM_OK;
}

bsmm_status bsmm_mlp_load(bsmm_mlp_t* out, const char* path) {
  if (!out || !path || !*path) return set_error("NULL output or path"), BSMM_ERR_INVALID;
  *out = nullptr;
  FILE* f = std::fopen(path, "rb");
  if (!f) return set_error(std::string("cannot open ") + path), BSMM_ERR_INVALID;
  std::vector<unsigned char> b;
  unsigned char buf[4096];
  size_t n;
  while ((n = std::fread(buf, 1, sizeof(buf), f)) > 0) {
    b.insert(b.end(), buf, buf + n);
    if (b.size() > (1u << 20)) break;  // far larger than any model file
  }
  std::fclose(f);
  if (b.size() < 8 + sizeof(uint64_t) || b.size() > (1u << 20))
    return set_error(std::string("not a cost-model file: ") + path), BSMM_ERR_INVALID;
  uint64_t sum = 0;
  std::memcpy(&sum, b.data() + b.size() - sizeof(uint64_t), sizeof(uint64_t));
  b.resize(b.size() - sizeof(uint64_t));
  if (fnv1a(b) != sum) return set_error(std::string("cost-model file checksum mismatch: ") + path), BSMM_ERR_INVALID;
  size_t pos = 0;
  char magic[8];
  uint32_t hdr[5];
  if (!get_raw(b, pos, magic, 8) || std::memcmp(magic, kMagic, 8) != 0 || !get_raw(b, pos, hdr, 5))
    return set_error(std::string("not a cost-model file: ") + path), BSMM_ERR_INVALID;
  if (hdr[0] != kFormatVersion || hdr[1] != (uint32_t)BSMM_FEATURE_VERSION || hdr[2] != (uint32_t)F ||
      hdr[3] != (uint32_t)H || hdr[4] != (uint32_t)NP)
    return set_error(std::string("cost-model file of another format, feature version or shape: ") + path),
           BSMM_ERR_INVALID;
  std::vector<float> prm(NP);
  Norm nm{};
  if (!get_raw(b, pos, prm.data(), NP) || !get_raw(b, pos, nm.xmu, F) || !get_raw(b, pos, nm.xsd, F) ||
      !get_raw(b, pos, &nm.ymu, 1) || !get_raw(b, pos, &nm.ysd, 1) || pos != b.size())
    return set_error(std::string("truncated cost-model file: ") + path), BSMM_ERR_INVALID;
  bsmm_mlp_t m = nullptr;
  bsmm_status st = bsmm_mlp_create(&m, 0);
  if (st == BSMM_OK) st = bsmm_mlp_set_params(m, prm.data(), NP);
  if (st == BSMM_OK) st = bsmm_mlp_set_norm(m, nm.xmu, nm.xsd, nm.ymu, nm.ysd);
  if (st != BSMM_OK) {
    bsmm_mlp_destroy(m);
    return st;
  }
  *out = m;
  return BSMM_OK;
}

void bsmm_mlp_destroy(bsmm_mlp_t mlp) {
  if (!mlp) return;
  for (DevBuf* b : {&mlp->params, &mlp->part})
    if (b->p) cudaFree(b->p);
  delete mlp;
}

}  // extern "C"
