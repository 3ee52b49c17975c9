// Split-precision operands: exponents, scale classes and slices (the error-free slicing of
// split.cu's method; kernels 1 and 2 of its launch order). Everything here works on the
// operands' bit patterns with integer instructions: GB300's FP64 pipe takes 2 lanes per
// clock.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <type_traits>

#include "bsmm_internal.h"
#include "overlap.cuh"

namespace bsmm {

namespace {

// byte offset of element (row, k) inside one 64-byte-swizzled chunk slice (rows of 32 elements)
__device__ __forceinline__ uint32_t swz64(int row, int k) {
  const int ch = k >> 3;
  return (uint32_t)(row * 64 + ((ch ^ ((row >> 1) & 3)) << 4) + ((k & 7) << 1));
}

// ---------------------------------------------------------------- kernel 1: exponents
// The caller's offset of stored tile t of A (isA) or B; transposed storage indexes the
// tables (k,i) / (j,k) (the maximum does not depend on the element order in a tile).
__device__ __forceinline__ void tile_geometry(const SplitArgs& a, bool isA, int t, int& rows, int& cols,
                                              int64_t& off) {
  if (isA) {
    const int i = t / a.K, k = t % a.K;
    rows = a.r[i];
    cols = a.q[k];
    off = a.transa ? a.a_off[(int64_t)k * a.M + i] : a.a_off[t];
  } else {
    const int k = t / a.N, j = t % a.N;
    rows = a.q[k];
    cols = a.c[j];
    off = a.transb ? a.b_off[(int64_t)j * a.K + k] : a.b_off[t];
  }
}

// Magnitude of a double as its bit pattern without the sign: for non-negative doubles the
// bit patterns order like the values, so maxima are taken with integer instructions
// (GB300's FP64 pipe is narrow). A pattern at or above kInfBits is an infinity or a NaN.
constexpr unsigned long long kAbsMask = 0x7FFFFFFFFFFFFFFFull;
constexpr unsigned long long kInfBits = 0x7FF0000000000000ull;
__device__ __forceinline__ unsigned long long mag_bits(double v) {
  return (unsigned long long)__double_as_longlong(v) & kAbsMask;
}

// Smallest e with m < 2^e for the magnitude bits m of a finite nonzero double
// (m = f 2^e with f in [0.5, 1), as frexp gives; subnormals included).
__device__ __forceinline__ int exponent_above(unsigned long long m) {
  const int be = (int)(m >> 52);
  if (be) return be - 1022;
  return -1022 - (__clzll((long long)m) - 12);  // subnormal: leading one at bit 63 - clz
}

// The same for the magnitude bits of a finite nonzero float (subnormals included).
constexpr uint32_t kInfBits32 = 0x7F800000u;
__device__ __forceinline__ int exponent_above32(uint32_t m) {
  const int be = (int)(m >> 23);
  if (be) return be - 126;
  return -126 - (__clz((int)m) - 9);  // subnormal: leading one at bit 31 - clz (22: below 2^-126)
}

__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t n;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
  return n;
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// v into rank 0's copy of a shared variable
__device__ __forceinline__ void store_rank0(unsigned long long* p, unsigned long long v) {
  uint32_t addr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(addr) : "r"((uint32_t)__cvta_generic_to_shared(p)));
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

// Per stored tile, the exponent of its largest magnitude; a CTA per tile, or a cluster of
// CTAs when the tiles alone would leave most SMs idle (a small product's time is this
// kernel's latency: one CTA takes a 160 x 160 tile in 12 rounds of loads). Bound by HBM.
constexpr int kExpThreads = 256;
constexpr int kExpCluster = 8;  // CTAs of a cluster, at most
constexpr int kExpResident = 4 * 152;  // CTAs that fill the machine
__global__ void __launch_bounds__(kExpThreads) split_exp_kernel(const __grid_constant__ SplitArgs a) {
  grid_wait();
  if (a.changes && blockIdx.x == 0 && threadIdx.x < 3) a.changes[threadIdx.x] = 0;
  const int nz = (int)cluster_size(), z = (int)cluster_rank();
  if (nz > 1) cluster_arrive();  // (waited for before rank 0's shared memory is written: it has started)
  const int b = blockIdx.x / nz;
  const bool isA = b < a.n_a_tiles;
  const int t = isA ? a.a_tiles[b] : a.b_tiles[b - a.n_a_tiles];
  int rows, cols;
  int64_t off;
  tile_geometry(a, isA, t, rows, cols, off);
  // complex elements: the tile's doubles (both parts) at twice its complex offset; an A
  // tile holds r x q' doubles (q' = 2q), a B tile q' x c' / 2 (c' = 2c)
  const double* x = (isA ? a.A : a.B) + (off < 0 ? 0 : (a.cplx ? 2 * off : off));
  const int64_t n = (int64_t)rows * cols / (a.cplx && !isA ? 2 : 1);
  const int first = z * kExpThreads + threadIdx.x, step = nz * kExpThreads;
  constexpr int kU = 4;  // loads in flight
  // the largest magnitude as bits: at or above kInfBits when a NaN or infinity is there
  unsigned long long mx = 0;
  if (a.f32 && off >= 0) {
    // float32 tiles start 16-byte aligned (offsets multiples of 4): four floats per load;
    // the float maximum's bits are turned into a double's (both order like the values)
    const float* xf = (isA ? a.Af : a.Bf) + off;
    uint32_t m32 = 0;
    if (off & 3) {
      if (threadIdx.x == 0) atomicOr(a.err, kErrBadOffset);
    } else {
      const uint4* x4 = reinterpret_cast<const uint4*>(xf);
      const int64_t n4 = n >> 2;
      for (int64_t e = first; e < n4; e += kU * step) {
        uint4 v[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) v[u] = e + u * step < n4 ? __ldg(x4 + e + u * step) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < kU; u++)
          m32 = max(m32, max(max(v[u].x & 0x7FFFFFFFu, v[u].y & 0x7FFFFFFFu),
                             max(v[u].z & 0x7FFFFFFFu, v[u].w & 0x7FFFFFFFu)));
      }
      for (int64_t e = (n4 << 2) + first; e < n; e += step) m32 = max(m32, __float_as_uint(__ldg(xf + e)) & 0x7FFFFFFFu);
    }
    // as a double's magnitude bits: equal exponent of the top bit, so exponent_above agrees
    if (m32 >= kInfBits32)
      mx = kInfBits;
    else if (m32)
      mx = (unsigned long long)(exponent_above32(m32) + 1022) << 52;
  } else if (off >= 0) {
    // tiles start 16-byte aligned (even offsets): pairs of doubles
    const longlong2* x2 = reinterpret_cast<const longlong2*>(x);
    const int64_t n2 = n >> 1;
    for (int64_t e = first; e < n2; e += kU * step) {
      longlong2 v[kU];
#pragma unroll
      for (int u = 0; u < kU; u++) v[u] = e + u * step < n2 ? __ldg(x2 + e + u * step) : make_longlong2(0, 0);
#pragma unroll
      for (int u = 0; u < kU; u++) {
        mx = max(mx, (unsigned long long)v[u].x & kAbsMask);
        mx = max(mx, (unsigned long long)v[u].y & kAbsMask);
      }
    }
    if ((n & 1) && first == 0) mx = max(mx, mag_bits(__ldg(x + n - 1)));
  }
  __shared__ unsigned long long red[kExpThreads / 32];
  __shared__ unsigned long long part[kExpCluster];
  for (int o = 16; o; o >>= 1) mx = max(mx, (unsigned long long)__shfl_xor_sync(0xffffffffu, (long long)mx, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  unsigned long long m = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < kExpThreads / 32; w++) m = max(m, red[w]);
  if (nz > 1) {
    cluster_wait();
    if (threadIdx.x == 0) store_rank0(&part[z], m);
    cluster_arrive();
    cluster_wait();
    if (z > 0) return;
    if (threadIdx.x == 0)
      for (int w = 0; w < nz; w++) m = max(m, part[w]);
  }
  if (threadIdx.x == 0) {
    int e = 0;
    if (off < 0 || m >= kInfBits) {
      atomicOr(a.err, off < 0 ? kErrBadOffset : kErrNonFinite);
    } else if (m > 0) {
      e = exponent_above(m);  // smallest e with max|x| < 2^e
    }
    if (isA)
      a.eA[t] = e;
    else
      a.eB[t] = e;
  }
}

// Row/column scaling: one exponent per row of each stored A tile and per column of each
// stored B tile (kZeroLine for an all-zero line). A few CTAs per tile; a line whose elements are
// contiguous is one warp's, lanes along it; otherwise lanes are neighbouring lines and the
// warps share their elements, so loads are coalesced either way (a thread per line read the
// contiguous ones 32 lines apart), 8 of them in flight per thread. Bound by HBM: complex 3072
// (302 MB), A transposed, 92 us; a CTA per tile with one load after the other 160 us. Offsets
// and non-finite values are checked here: the tile exponents are not needed.
constexpr int kLinesY = 4;  // CTAs per tile, sharing its lines
template <typename E>
__global__ void __launch_bounds__(256) split_exp_lines_kernel(const __grid_constant__ SplitArgs a) {
  grid_wait();
  const int b = blockIdx.x;
  if (a.changes && b == 0 && blockIdx.y == 0 && threadIdx.x < 3) a.changes[threadIdx.x] = 0;
  const bool isA = b < a.n_a_tiles;
  const int t = isA ? a.a_tiles[b] : a.b_tiles[b - a.n_a_tiles];
  int rows, cols;
  int64_t off;
  tile_geometry(a, isA, t, rows, cols, off);
  if (off < 0 || (std::is_same<E, float>::value && (off & 3))) {
    if (threadIdx.x == 0) atomicOr(a.err, kErrBadOffset);
    return;
  }
  const int i_or_k = isA ? t / a.K : t / a.N;
  const int k_or_j = isA ? t % a.K : t % a.N;
  const bool tr = isA ? a.transa != 0 : a.transb != 0;
  // Complex elements: the plan's inner and column tilings count both parts, so an A tile is
  // rows x (2 qc) and a B tile (2 qc) x (2 cc) of the real product; a line's exponent is that
  // of the complex row (column) over both parts, and the B column c and its partner c + cc
  // (the same complex column's other part) share it.
  const int parts = a.cplx ? 2 : 1;
  const int nl = isA ? rows : cols / parts;                 // lines
  const int len = (isA ? cols : rows) / parts;              // elements (complex: pairs) per line
  const bool contig = isA ? !tr : tr;
  constexpr bool kF32 = std::is_same<E, float>::value;
  const E* const x = reinterpret_cast<const E*>(kF32 ? (const void*)(isA ? a.Af : a.Bf) : (const void*)(isA ? a.A : a.B)) +
                     parts * off;
  int32_t* const out = isA ? a.eArow + (int64_t)k_or_j * a.Mtot + a.ro[i_or_k]
                           : a.eBcol + (int64_t)i_or_k * a.Ntot + a.co[k_or_j];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the largest magnitude's bits (a float's or a double's)
  auto at = [&](int64_t e) -> unsigned long long {
    if constexpr (kF32)
      return __float_as_uint(__ldg(x + e)) & 0x7FFFFFFFu;
    else
      return mag_bits(__ldg(x + e));
  };
  auto write = [&](int l, unsigned long long m) {
    if (kF32 ? m >= kInfBits32 : m >= kInfBits) atomicOr(a.err, kErrNonFinite);
    int e = kZeroLine;
    if constexpr (kF32) {
      if (m > 0 && m < kInfBits32) e = exponent_above32((uint32_t)m);
    } else if (m > 0 && m < kInfBits) {
      e = exponent_above(m);
    }
    out[l] = e;
    if (!isA && a.cplx) out[nl + l] = e;
  };
  if (contig) {
    const int n = len * parts;
    for (int l = warp + 8 * blockIdx.y; l < nl; l += 8 * kLinesY) {
      unsigned long long m = 0;
      constexpr int kU = 8;  // loads in flight
      for (int u0 = lane; u0 < n; u0 += 32 * kU) {
        unsigned long long v[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) v[u] = u0 + 32 * u < n ? at((int64_t)l * n + u0 + 32 * u) : 0ull;
#pragma unroll
        for (int u = 0; u < kU; u++) m = max(m, v[u]);
      }
      for (int o = 16; o; o >>= 1) m = max(m, (unsigned long long)__shfl_xor_sync(0xffffffffu, (long long)m, o));
      if (lane == 0) write(l, m);
    }
  } else {
    __shared__ unsigned long long red[8][32];
    for (int l0 = 32 * blockIdx.y; l0 < nl; l0 += 32 * kLinesY) {
      const int l = l0 + lane;
      unsigned long long m = 0;
      if (l < nl) {
        constexpr int kU = 8;  // loads in flight
        for (int u0 = warp; u0 < len; u0 += 8 * kU) {
          if (parts == 2) {  // both parts of a complex element at once (16-byte aligned)
            longlong2 v[kU];
#pragma unroll
            for (int u = 0; u < kU; u++) {
              const int64_t e = ((int64_t)(u0 + 8 * u) * nl + l) * 2;
              v[u] = u0 + 8 * u < len ? __ldg(reinterpret_cast<const longlong2*>(x + e)) : make_longlong2(0, 0);
            }
#pragma unroll
            for (int u = 0; u < kU; u++)
              m = max(m, max((unsigned long long)v[u].x & kAbsMask, (unsigned long long)v[u].y & kAbsMask));
          } else {
            unsigned long long v[kU];
#pragma unroll
            for (int u = 0; u < kU; u++) v[u] = u0 + 8 * u < len ? at((int64_t)(u0 + 8 * u) * nl + l) : 0ull;
#pragma unroll
            for (int u = 0; u < kU; u++) m = max(m, v[u]);
          }
        }
      }
      red[warp][lane] = m;
      __syncthreads();
      if (warp == 0 && l < nl) {
        for (int w = 1; w < 8; w++) m = max(m, red[w][lane]);
        write(l, m);
      }
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------- kernel 1b: line scales
// Row/column scaling, per row m of A (per column n of B): Emax = the largest exponent of that
// line over its stored tiles (all-zero lines excluded; 0 when none), and rowexp[k][m] =
// e(m, k) - Emax (colexp likewise), 0 where there is no tile or the line is zero there (its
// slices are zero). A CTA takes 32 lines, its warps the inner blocks in turn.
__global__ void __launch_bounds__(256) split_scale_lines_kernel(const __grid_constant__ SplitArgs a) {
  __shared__ int red[8][32];
  grid_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t t = (int64_t)blockIdx.x * 32 + lane;
  const bool isA = t < a.Mtot;
  const bool in = t < a.Mtot + a.Ntot;
  const int64_t x = isA ? t : t - a.Mtot;
  const int tile = in ? (isA ? a.row_tile[x] : a.col_tile[x]) : 0;
  auto exponent = [&](int k) -> int {  // kZeroLine: no tile, or a zero line
    if (a.q[k] <= 0 || !(isA ? a.am[(int64_t)tile * a.K + k] : a.bm[(int64_t)k * a.N + tile])) return kZeroLine;
    return isA ? a.eArow[(int64_t)k * a.Mtot + x] : a.eBcol[(int64_t)k * a.Ntot + x];
  };
  int em = INT_MIN;
  if (in) {
#pragma unroll 4
    for (int k = warp; k < a.K; k += 8) {
      const int e = exponent(k);
      if (e != kZeroLine) em = max(em, e);
    }
  }
  red[warp][lane] = em;
  __syncthreads();
  for (int w = 0; w < 8; w++) em = max(em, red[w][lane]);
  if (em == INT_MIN) em = 0;
  if (!in) return;
  if (warp == 0) (isA ? a.eAmaxr : a.eBmaxc)[x] = em;
#pragma unroll 4
  for (int k = warp; k < a.K; k += 8) {
    const int e = exponent(k);
    const int16_t d = (int16_t)(e != kZeroLine ? e - em : 0);
    if (isA)
      a.rowexp[(int64_t)k * a.Mtot + x] = d;
    else
      a.colexp[(int64_t)k * a.colexp_ld + x] = d;
  }
}

// ---------------------------------------------------------------- kernel 1c: offsets and scale classes
// For one block of lines (a 128-row block of A or a 32-column block of B) and a range of inner
// blocks, by one CTA of the pack kernel's launch (slicing needs the exponents only, so it runs
// beside this). With one scale per tile, first Emax of each of the block's tiles, the largest
// exponent over all its stored tiles (0 when none), and then the offsets of the block's
// lines, rowexp[k][m] = e_A(i,k) - Emax_A(i) for a stored tile (0 for an absent one), or
// colexp; with one scale per row and column the line kernel wrote them. The contraction adds
// each tile pair's exact integer at the binary position GUARD + rowexp + colexp of a 128-bit
// accumulator whose unit is 2^(Emax_A + Emax_B - 7(s+1) - GUARD).
// Then the scale class. The products of k block k land at element (m, n) at the binary
// position e_A(m,k) + e_B(n,k) - Emax_A(m) - Emax_B(n) (exponents of the row's and the
// column's tile, or line, at k, and their maxima). When the rows of the row block that
// have a tile at k share one exponent e_A(k) (the columns likewise e_B(k)), that position
// is e_A(k) + e_B(k) plus a part that depends only on the row and the column, not on k:
//   urow[k][rb] = e_A(k) - maxE_A(rb),  rowadj[m] = maxE_A(rb) - Emax_A(m) >= 0
// (maxE_A(rb) = the largest Emax_A over the block's rows; the same for columns), so two
// k blocks whose urow + ucol agree may share one TMEM accumulation, drained at
// guard + urow + ucol + rowadj[m] + coladj[n]. kNonUniform marks a k block whose rows (or
// columns) at k have different exponents; rows without a tile (or all-zero lines) there
// take no part.
//
// A CTA takes chains of a few dependent loads, so there are at most kClassMaxRanges of them
// per block of lines, fewer where the blocks are many, and they stand between the slicing
// CTAs of the launch, which use the memory meanwhile (all in front, and 16 per block, they
// held the banded 32768 product's launch for 260 us).
constexpr int kClassMaxRanges = 16;

struct ClassShared {
  int32_t tile[kSplitBM];  // the lines' tiles
  int32_t em[kSplitBM];    // and largest exponents
  uint32_t first[kSplitBM / 32];  // bit: the line is the first of its tile here
  int last;                // this CTA is the last one done
};

__device__ void scale_classes(const SplitArgs& a, ClassShared& sm, int item, int nr, int items) {
  const int blk = item / nr;
  const bool isA = blk < a.RB;
  const int b = isA ? blk : blk - a.RB;
  const int k0 = (int)((int64_t)(item % nr) * a.K / nr), k1 = (int)((int64_t)(item % nr + 1) * a.K / nr);
  const int width = isA ? kSplitBM : 32;
  const int64_t x0 = (int64_t)b * width;
  const int64_t total = isA ? a.Mtot : a.Ntot;
  const int nl = (int)min((int64_t)width, total - x0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < kSplitBM) {
    int t = -1;
    bool first = false;
    if (tid < nl) {
      const int32_t* const of = isA ? a.row_tile : a.col_tile;
      t = of[x0 + tid];
      first = tid == 0 || of[x0 + tid - 1] != t;
      if (a.rowscale) sm.em[tid] = isA ? a.eAmaxr[x0 + tid] : a.eBmaxc[x0 + tid];
    }
    sm.tile[tid] = t;
    const uint32_t bits = __ballot_sync(0xffffffffu, first);
    if (lane == 0) sm.first[warp] = bits;
  }
  __syncthreads();
  if (!a.rowscale) {
    for (int l = warp; l < nl; l += 8) {
      if (!(sm.first[l >> 5] >> (l & 31) & 1)) continue;
      const int t = sm.tile[l];
      int em = INT_MIN;
#pragma unroll 4
      for (int k = lane; k < a.K; k += 32) {
        const int64_t at = isA ? (int64_t)t * a.K + k : (int64_t)k * a.N + t;
        const int e = __ldg((isA ? a.eA : a.eB) + at);
        if (__ldg(a.q + k) > 0 && __ldg((isA ? a.am : a.bm) + at)) em = max(em, e);
      }
      for (int o = 16; o; o >>= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, o));
      if (lane == 0) sm.em[l] = em == INT_MIN ? 0 : em;
    }
    __syncthreads();
    int em = 0;
    if (tid < nl) {  // the line that is first in this line's tile
      int w = tid >> 5;
      uint32_t bits = sm.first[w] & (0xffffffffu >> (31 - (tid & 31)));
      while (!bits) bits = sm.first[--w];
      em = sm.em[w * 32 + 31 - __clz((int)bits)];
    }
    __syncthreads();
    if (tid < nl) sm.em[tid] = em;
    __syncthreads();
  }
  int emx = INT_MIN;
  for (int l = lane; l < nl; l += 32) emx = max(emx, sm.em[l]);
  for (int o = 16; o; o >>= 1) emx = max(emx, __shfl_xor_sync(0xffffffffu, emx, o));
  if (k0 == 0 && tid < nl) {
    (isA ? a.emaxr : a.emaxc)[x0 + tid] = sm.em[tid];
    if (a.urow) (isA ? a.rowadj : a.coladj)[x0 + tid] = (int16_t)(emx - sm.em[tid]);
  }
  const uint8_t* const mask = isA ? a.am : a.bm;
  const int32_t* const exps = isA ? a.eA : a.eB;
#pragma unroll 4
  for (int k = k0 + warp; k < k1; k += 8) {
    const bool some = __ldg(a.q + k) > 0;
    int lo = INT_MAX, hi = INT_MIN;
#pragma unroll
    for (int u = 0; u < kSplitBM / 32; u++) {
      const int l = u * 32 + lane;
      if (l >= nl) continue;
      const int t = sm.tile[l];
      const int64_t at = isA ? (int64_t)t * a.K + k : (int64_t)k * a.N + t;
      bool pres = __ldg(mask + at) != 0 && some;
      int e = 0;
      if (!a.rowscale) {
        const int ev = __ldg(exps + at);  // (whatever is there when no tile is stored)
        e = pres ? ev : 0;
        const int16_t d = (int16_t)(pres ? e - sm.em[l] : 0);
        if (isA)
          a.rowexp[(int64_t)k * a.Mtot + x0 + l] = d;
        else
          a.colexp[(int64_t)k * a.colexp_ld + x0 + l] = d;
      } else if (pres) {
        e = isA ? a.eArow[(int64_t)k * a.Mtot + x0 + l] : a.eBcol[(int64_t)k * a.Ntot + x0 + l];
        pres = e != kZeroLine;
      }
      if (pres) {
        lo = min(lo, e);
        hi = max(hi, e);
      }
    }
    for (int o = 16; o; o >>= 1) {
      lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    int16_t* const cls = isA ? a.urow : a.ucol;
    if (cls && lane == 0)
      cls[isA ? (int64_t)k * a.RB + b : (int64_t)k * a.CB + b] = (int16_t)(lo > hi ? 0 : lo == hi ? lo - emx : kNonUniform);
  }
  if (!a.changes) return;
  // how many of this range's k blocks cannot join the group of the one before (the range's
  // first one is given the benefit of the doubt): what the choice of the contraction goes by
  __syncthreads();
  const int16_t* const cls = isA ? a.urow + b : a.ucol + b;
  const int64_t ld = isA ? a.RB : a.CB;
  const uint64_t* const pres = (isA ? a.presA : a.presB) + (int64_t)b * a.kwords;
  auto present = [&](int k) { return (pres[k >> 6] >> (k & 63) & 1) != 0; };
  int n = 0;
  for (int k = k0 + tid; k < k1; k += blockDim.x) {
    if (!present(k)) continue;
    int kp = k - 1;
    while (kp >= k0 && !present(kp)) kp--;
    const int c = cls[k * ld];
    if (c == kNonUniform || (kp >= k0 && cls[kp * ld] != c)) n++;
  }
  n = __reduce_add_sync(0xffffffffu, n);
  if (lane == 0 && n) atomicAdd(a.changes + (isA ? 0 : 1), n);
  __threadfence();
  __syncthreads();
  if (tid == 0) sm.last = atomicAdd(a.changes + 2, 1) == items - 1;
  __syncthreads();
  if (!sm.last) return;
  // the choice, made once for both kernels
  __threadfence();
  const float fa = (float)__ldcg(a.changes) / (float)a.n_a_blocks, fb = (float)__ldcg(a.changes + 1) / (float)a.n_b_blocks;
  const bool wide = 1.0f - (1.0f - fa) * (1.0f - fb) <= a.max_changes;
  if (tid == 0) a.changes[3] = wide;
  for (int g = tid; g <= a.n_groups; g += blockDim.x) a.sched_sel[g] = wide ? a.sched_ptr[g] : 0;
}

// ---------------------------------------------------------------- kernel 2: slices
// The slicing recurrence N_t = rint(rho_{t-1} 2^(7t)), rho_t = rho_{t-1} - N_t 2^(-7t)
// telescopes: with Z_t = sum_{u<=t} N_u 2^(7(t-u)) one has Z_t = rint(x 2^(7t-e)) (the
// subtracted 128 Z_{t-1} is even, so round-half-even commutes with it), hence
// N_t = Z_t - 128 Z_{t-1}. The signs of Z_t and N_t are x's and -x's alike (half-even is
// symmetric), so magnitudes are sliced and the sign is multiplied in at the end.
//
// Window. V = floor(|x| 2^(7S-e+2)): |x| in units of 2^-2 of the finest slice's unit. Level
// t's unit is then 2^p with p = 2 + 7(S-t), and Z_t = floor((V + 2^(p-1)) / 2^p), except
// that an exact tie has to go to the even quotient. x is at a tie of level t exactly when
// no bit below V is set and V's lowest set bit is bit p-1, so it is at a tie of at most one
// level, and there V +- 1 (up when bit p, the quotient's last bit, is set) rounds as
// half-even asks without changing any other level's rounding. A tie needs V even and
// nothing below it, which a thread tests for its 8 elements at once: seldom true of doubles
// of full mantissa, always of float32 and integer data.
//
// Digits. With r_t = (V + 2^(p-1)) mod 2^p = (V mod 2^p) ^ 2^(p-1), what rounding at level
// t leaves over (biased), N_t 2^p = r_{t-1} - r_t + 2^(p-1) - 2^(p+6). So a digit takes one
// three-input logic instruction (r_t) and one three-input addition, which also adds the
// bits of 2^23: the sum read as a float is 2^23 + (N_t + 64) 2^p, one multiply-add from
// N_t. The multiply-add, the sign and the packing run beside the integer pipe. Three
// levels fit a 32-bit word (p = 2, 9, 16); the next three are those of V >> 21, whose
// dropped bits are the same in both remainders.
//
// What bounds it: HBM (8 bytes read and 2S written per element) and the integer pipe
// together: 16384 dense, six slices, 10.7 GB in 1.96 to 2.02 ms (5.4 TB/s); on 6144 DRAM is
// 64% busy and the integer pipe 79% (per instruction issued 2.2 warps wait for data, 1.4 for
// the pipe). Before, significand windows with variable rounding per level took 2.92 ms
// (integer pipe 80% busy, DRAM 43%, and each block's chunks one after the other with nothing
// in flight between them). float32 8192, four slices: 0.62 to 0.45 ms.
template <typename T>
struct Slice2;  // two slices' values in one word; times the elements' signs
template <>
struct Slice2<__nv_bfloat16> {
  static constexpr uint32_t kOnes = 0x3F803F80u;
  __device__ static uint32_t pack(float lo, float hi) {  // <= 8 significant bits: truncation is exact
    return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
  }
  __device__ static uint32_t mul(uint32_t a, uint32_t b) {
    const __nv_bfloat162 r = __hmul2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
    return *reinterpret_cast<const uint32_t*>(&r);
  }
};
template <>
struct Slice2<__half> {
  static constexpr uint32_t kOnes = 0x3C003C00u;
  __device__ static uint32_t pack(float lo, float hi) {
    const __half2 r = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&r);
  }
  __device__ static uint32_t mul(uint32_t a, uint32_t b) {
    const __half2 r = __hmul2(*reinterpret_cast<__half2*>(&a), *reinterpret_cast<__half2*>(&b));
    return *reinterpret_cast<const uint32_t*>(&r);
  }
};

// |x| = m 2^(be - 1075) with m < 2^53, from the bits of a double or a float (a float's
// significand shifted into a double's place); sgn: a word with x's sign in its top bit.
// ANY: subnormals too; otherwise the leading one is taken for granted (a zero then has a
// be that shifts it out).
template <bool ANY>
__device__ __forceinline__ void decode(double x, uint32_t& lo, uint32_t& hi, int& be, uint32_t& sgn) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  sgn = (uint32_t)(b >> 32);
  lo = (uint32_t)b;
  be = (int)((sgn >> 20) & 0x7FFu);
  hi = (sgn & 0xFFFFFu) | (!ANY || be ? 0x100000u : 0u);
  if constexpr (ANY) be = max(be, 1);
}
template <bool ANY>
__device__ __forceinline__ void decode(float x, uint32_t& lo, uint32_t& hi, int& be, uint32_t& sgn) {
  sgn = __float_as_uint(x);
  be = (int)((sgn >> 23) & 0xFFu);
  const uint32_t m = (sgn & 0x7FFFFFu) | (!ANY || be ? 0x800000u : 0u);
  lo = m << 29;
  hi = m >> 3;
  if constexpr (ANY) be = max(be, 1);
  be += 896;
}

// shifts that give 0 for a count beyond the width (a negative one counts as such)
__device__ __forceinline__ unsigned long long shr64(unsigned long long v, int n) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}
__device__ __forceinline__ unsigned long long shl64(unsigned long long v, int n) {
  unsigned long long r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}
__device__ __forceinline__ uint32_t shr32(uint32_t v, int n) {
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
  return r;
}
__device__ __forceinline__ uint32_t shl32(uint32_t v, int n) {
  uint32_t r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
  return r;
}

// V at an exact tie, moved off it to the side half-even rounds to (see above)
template <int S, typename U>
__device__ __forceinline__ U tie_to_even(U V) {
  constexpr U kTies = (U)(2 * ((1ull << (7 * S)) - 1) / 127);  // bits p-1 of every level
  const U low = V & ((U)0 - V) & kTies;
  return low ? ((V & (low << 1)) ? V + 1 : V - 1) : V;
}

// Largest exponent e of a tile (line) in which an element with exponent field 0, which
// decode<false> takes for a normal one, may leave bits in its window: it is then taken for a
// value below 2^-1022 (a float for one below 2^-126), and its V for one below
// 2^(-1022 + 7S + 2 - e), so above this e it is 0.
template <int S, typename E>
constexpr int kAnyExponent = 7 * S + 3 - (std::is_same<E, float>::value ? 128 : 1024);

// The window of one element, subnormals and tiny tiles included (the shift may be a left
// one). Out of line: only tiles of exponent kAnyExponent and below need it, for doubles
// those of elements below 2^-979 or less, for floats below 2^-83 with six slices, 2^-97 with
// four. (One bound of -900 for both types took a float's zero for 2^-127 there.)
template <int S, typename E>
__device__ __noinline__ unsigned long long slice_window_any(E x, int e) {
  uint32_t lo, hi, sgn;
  int be;
  decode<true>(x, lo, hi, be, sgn);
  const unsigned long long m = ((unsigned long long)hi << 32) | lo;
  const int sh = e + 1073 - 7 * S - be;  // V = m 2^-sh
  if (sh < 1) return tie_to_even<S>(shl64(m, -sh));  // exact
  const unsigned long long V = shr64(m, sh);
  return sh < 64 && shl64(m, 64 - sh) == 0ull ? tie_to_even<S>(V) : V;
}

// The windows of 8 elements: V's low word, V >> 21, and the signs.
template <int S, typename E>
__device__ __forceinline__ void slice_windows(const E (&x)[8], int e, uint32_t (&w0)[8], uint32_t (&w1)[8],
                                              uint32_t (&sgn)[8]) {
  // A normal element of a tile with max|x| < 2^e has be <= e + 1022, so V = m >> sh with
  // sh >= 51 - 7S. The significand's low kPre = 50 - 7S bits are below every V and with 4
  // slices or fewer are dropped first: what is left fits 32 bits. A zero or subnormal
  // element (exponent field 0) shifts everything out: V = 0, as it should be, in tiles above
  // kAnyExponent.
  constexpr int kPre = 50 - 7 * S;
  constexpr bool k32 = S <= 4;
  const int c = e + 1073 - 7 * S;
  uint32_t some = 0xFFFFFFFFu;  // 0: some element may have V even and no bit below it
#pragma unroll
  for (int u = 0; u < 8; u++) {
    uint32_t lo, hi;
    int be;
    decode<false>(x[u], lo, hi, be, sgn[u]);
    const int sh = c - be;
    if constexpr (k32) {
      const uint32_t m = kPre >= 32 ? hi >> (kPre & 31) : __funnelshift_r(lo, hi, kPre & 31);
      const int r = sh - kPre;
      w0[u] = shr32(m, r);
      w1[u] = w0[u] >> 21;
      // the dropped bits (a float's 24-bit significand has none below bit 29)
      uint32_t cut = 0u;
      if constexpr (kPre >= 32)
        cut = lo | (hi & ((1u << (kPre & 31)) - 1u));
      else if constexpr (!std::is_same<E, float>::value)
        cut = lo & ((1u << (kPre & 31)) - 1u);
      some = min(some, shl32(m, 31 - r) | cut);
    } else {
      const unsigned long long V = shr64(((unsigned long long)hi << 32) | lo, sh);
      w0[u] = (uint32_t)V;
      w1[u] = (uint32_t)(V >> 21);
      some = min(some, shl32(lo, 31 - sh));
    }
  }
  if (e <= kAnyExponent<S, E>) {
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const unsigned long long V = slice_window_any<S>(x[u], e);
      w0[u] = (uint32_t)V;
      w1[u] = (uint32_t)(V >> 21);
    }
  } else if (some == 0u) {
#pragma unroll
    for (int u = 0; u < 8; u++) {
      uint32_t lo, hi, sg;
      int be;
      decode<false>(x[u], lo, hi, be, sg);
      const unsigned long long m = ((unsigned long long)hi << 32) | lo;
      const int sh = c - be;
      const bool exact = shl64(m, 64 - sh) == 0ull;  // no bit below V (V = 0 when sh is beyond m's width)
      if constexpr (k32) {
        w0[u] = exact ? tie_to_even<S>(w0[u]) : w0[u];
        w1[u] = w0[u] >> 21;
      } else if (exact) {
        const unsigned long long V = tie_to_even<S>(shr64(m, sh));
        w0[u] = (uint32_t)V;
        w1[u] = (uint32_t)(V >> 21);
      }
    }
  }
}

// Slice i levels above the finest (t = S - i): N_t as an exact float, without its sign.
template <int S, int i>
__device__ __forceinline__ float slice_digit(uint32_t w0, uint32_t w1) {
  static_assert(S <= 6, "two windows of three levels");
  constexpr int p = 2 + 7 * (i % 3);
  constexpr uint32_t kMagic = 0x4B000000u;  // 2^23 as a float
  const uint32_t w = i < 3 ? w0 : w1;
  if constexpr (i == S - 1) {  // the top slice: N_1 = Z_1 <= 128
    const uint32_t f = ((w + (1u << (p - 1))) & ~((1u << p) - 1u)) | kMagic;
    return fmaf(__uint_as_float(f), 1.0f / (1 << p), -(float)(1 << (23 - p)));
  } else {
    const uint32_t r = (w & ((1u << p) - 1u)) ^ (1u << (p - 1));
    const uint32_t ra = (w & ((1u << (p + 7)) - 1u)) ^ (1u << (p + 6));
    const uint32_t f = ra - r + (kMagic + (1u << (p - 1)));
    return fmaf(__uint_as_float(f), 1.0f / (1 << p), -(float)((1 << (23 - p)) + 64));
  }
}

template <typename T, int S, int i>
__device__ __forceinline__ void slice_levels(const uint32_t (&w0)[8], const uint32_t (&w1)[8],
                                             const uint32_t (&sg)[4], uint8_t* dst, int slice_stride) {
  if constexpr (i < S) {
    uint32_t h[4];
#pragma unroll
    for (int u = 0; u < 4; u++)
      h[u] = Slice2<T>::mul(Slice2<T>::pack(slice_digit<S, i>(w0[2 * u], w1[2 * u]),
                                            slice_digit<S, i>(w0[2 * u + 1], w1[2 * u + 1])),
                            sg[u]);
    *reinterpret_cast<uint4*>(dst + (size_t)(S - 1 - i) * slice_stride) = make_uint4(h[0], h[1], h[2], h[3]);
    slice_levels<T, S, i + 1>(w0, w1, sg, dst, slice_stride);
  }
}

// Slice 8 consecutive inner elements (one 16-byte chunk of a swizzled row) of one packed
// row and store the S chunks.
template <typename T, int S, typename E>
__device__ __forceinline__ void slice_store8(const E (&x)[8], int e, uint8_t* dst, int slice_stride) {
  uint32_t w0[8], w1[8], sgn[8], sg[4];
  slice_windows<S>(x, e, w0, w1, sgn);
#pragma unroll
  for (int u = 0; u < 4; u++)
    sg[u] = (__byte_perm(sgn[2 * u], sgn[2 * u + 1], 0x7632) & 0x80008000u) | Slice2<T>::kOnes;  // +-1 each
  slice_levels<T, S, 0>(w0, w1, sg, dst, slice_stride);
}

// Complex elements (CPLX): the real product's A tile is [Ar, -Ai] (inner index kk' < q
// takes the real part of column kk', kk' >= q the negated imaginary part of column kk' - q)
// and its B tile [[Br, Bi], [Bi, -Br]] (row half and column half pick the part and the
// sign); q and c below are the doubled sizes, the stored complex tile is q/2 and c/2 wide.
__device__ __forceinline__ double neg_if(double v, bool n) {  // sign flip as bits (no FP64 op)
  return n ? __longlong_as_double(__double_as_longlong(v) ^ (long long)0x8000000000000000ull) : v;
}

// A CTA packs a group of 128 lines at one or several inner blocks: the rows of one A block,
// or the columns of four B blocks that follow each other in the plan's list. It looks every
// line up once (four dependent loads) and then makes passes of 256 pieces of 8 inner
// elements: half a 32-deep chunk of the A block, or two chunks of a B block. A pass's loads
// are in flight while the pass before is sliced. Groups are dealt to `ny` CTAs each, pass
// by pass, when they are too few to fill the machine. Four neighbouring threads take one
// line's 32 inner elements and a warp 8 lines, so every store instruction writes 512
// contiguous bytes of the packed image, and loads read whole 32-byte sectors in either
// storage order: 64 bytes of a line (in 16-byte loads where the line starts are aligned),
// or 8 neighbouring lines' elements.
constexpr int kPackThreads = 256;
constexpr int kPackLines = 128;                             // lines of a group
constexpr int kPackEntries = kPackLines / 32;               // B blocks of a group (32 columns each)
constexpr int kPackMaxY = 8;
constexpr int kPackResident = 3 * 152;                      // CTAs on the machine at once
static_assert(kPackLines == kSplitBM, "an A group is one A block");

// What a CTA looks up once per line ...
struct PackLine {
  int64_t base;   // the line's first element (real: E units; complex: doubles), -1: zeros
  int32_t step;   // elements (doubles) from one inner index to the next
  int32_t e;      // the line's exponent
  int32_t cpart;  // complex B: 1 for the second half of the doubled columns
};
// ... and once per block
struct PackEntry {
  int64_t out;    // byte offset of the packed block
  int32_t q, nkc; // inner elements, 32-deep chunks (0: no block)
};

struct PackGrid {
  int ncls, ranges, every;  // CTAs for the scale classes, per block of lines, and their spacing
  int ny;                   // CTAs per group of lines to pack
};

template <typename T, int S, typename E, bool CPLX = false>
__global__ void __launch_bounds__(kPackThreads, 3) split_pack_kernel(const __grid_constant__ SplitArgs a, PackGrid g) {
  __shared__ union {
    ClassShared cls;
    struct {
      PackLine lines[kPackLines];
      PackEntry entries[kPackEntries];
      int passes_of[kPackEntries];
    } pk;
  } sm;
  grid_wait();
  const int turn = blockIdx.x / g.every;  // every g.every-th CTA: offsets and scale classes
  if (turn < g.ncls && blockIdx.x % g.every == 0) {
    scale_classes(a, sm.cls, turn, g.ranges, g.ncls);
    return;
  }
  auto& lines = sm.pk.lines;
  auto& entries = sm.pk.entries;
  auto& passes_of = sm.pk.passes_of;
  const int bid = blockIdx.x - min(g.ncls, turn + 1);
  const int ny = g.ny;
  constexpr int VE = 16 / (int)sizeof(E);
  const int tid = threadIdx.x;
  const int grp = bid / ny;
  const bool isA = grp < a.n_a_blocks;
  const bool contig = isA ? !a.transa : a.transb != 0;  // a line's inner elements are contiguous
  if (tid < kPackLines) {
    const int en = isA ? 0 : tid >> 5, ln = isA ? tid : tid & 31;
    const int at = isA ? grp : (grp - a.n_a_blocks) * kPackEntries + en;
    PackLine l{-1, 1, 0, 0};
    PackEntry pe{0, 0, 0};
    if (isA || at < a.n_b_blocks) {
      const int blk = isA ? a.a_blocks[at] : a.b_blocks[at];
      const int kt = isA ? blk % a.K : blk / a.CB;
      const int64_t x = (isA ? (int64_t)(blk / a.K) * kSplitBM : (int64_t)(blk % a.CB) * 32) + ln;
      const int q = a.q[kt];
      pe.out = isA ? a.apk_off[blk] : a.bpk_off[blk];
      pe.q = q;
      pe.nkc = (q + kSplitKC - 1) / kSplitKC;
      if (x < (isA ? a.Mtot : a.Ntot)) {
        const int t = isA ? a.row_tile[x] : a.col_tile[x];
        const int64_t tile = isA ? (int64_t)t * a.K + kt : (int64_t)kt * a.N + t;
        const int64_t off = isA ? (a.transa ? a.a_off[(int64_t)kt * a.M + t] : a.a_off[tile])
                                : (a.transb ? a.b_off[(int64_t)t * a.K + kt] : a.b_off[tile]);
        const int width = isA ? a.r[t] : a.c[t];  // lines of the tile
        int64_t lx = x - (isA ? a.ro[t] : a.co[t]);
        if (!isA && CPLX && lx >= (width >> 1)) {
          l.cpart = 1;
          lx -= width >> 1;
        }
        if (isA ? a.am[tile] : a.bm[tile]) {
          // (an offset off the 16-byte grid is reported, never read with 16-byte loads)
          if (off < 0 || (!CPLX && contig && q % VE == 0 && off % VE != 0)) {
            atomicOr(a.err, kErrBadOffset);
          } else if (CPLX) {
            const int64_t tw = isA ? width : width >> 1;
            l.base = 2 * (off + (contig ? lx * (q >> 1) : lx));
            l.step = contig ? 2 : (int)(2 * tw);
          } else {
            l.base = off + (contig ? lx * q : lx);
            l.step = contig ? 1 : width;
          }
        }
        l.e = a.rowscale ? (isA ? a.eArow[(int64_t)kt * a.Mtot + x] : a.eBcol[(int64_t)kt * a.Ntot + x])
                         : (isA ? a.eA[tile] : a.eB[tile]);
      }
    }
    lines[tid] = l;
    if (ln == 0) {
      entries[en] = pe;
      passes_of[en] = isA ? 2 * pe.nkc : (pe.nkc + 1) >> 1;
    }
  }
  __syncthreads();
  int total = 0;
  for (int en = 0; en < (isA ? 1 : kPackEntries); en++) total += passes_of[en];

  const E* const src = isA ? reinterpret_cast<const E*>(std::is_same<E, float>::value ? (const void*)a.Af : (const void*)a.A)
                           : reinterpret_cast<const E*>(std::is_same<E, float>::value ? (const void*)a.Bf : (const void*)a.B);
  // (a pair of column blocks packed together: the other block's part lies between the slices)
  int slice_stride = isA ? kSplitBM * kSplitKC * 2 : 32 * kSplitKC * 2;
  if constexpr (S <= kWidePairsMaxS) slice_stride <<= !isA && a.pairs;
  uint8_t* const pk = isA ? a.apk : a.bpk;
  const int ch = tid & 3;

  struct Piece {  // a thread's 8 elements of a pass
    E x[8];
    int line;  // -1: none
    int k0;    // first inner index, or past the end: zeros
    uint8_t* dst;
  };
  auto load = [&](Piece& pc, int pass) {
    int en = 0, p = pass;
    while (p >= passes_of[en]) p -= passes_of[en++];
    const PackEntry pe = entries[en];
    // A: pass p is half p & 1 of chunk p >> 1; B: chunks 2p and 2p + 1
    const int ln = isA ? (p & 1) * 64 + (tid >> 2) : (tid >> 2) & 31;
    const int kc = isA ? p >> 1 : 2 * p + (tid >> 7);
    pc.line = kc < pe.nkc ? (isA ? ln : en * 32 + ln) : -1;
    pc.dst = pk + pe.out + (size_t)kc * S * slice_stride + swz64(ln, ch * 8);
    const int q = pe.q;
    int k0 = kc * kSplitKC + ch * 8;
    const PackLine l = lines[isA ? ln : en * 32 + ln];
    if (l.base < 0) k0 = 1 << 30;
    pc.k0 = k0 < q ? k0 : 1 << 30;
    if constexpr (CPLX) {
      // inner index kk takes part (kk >= q/2) of the complex inner index; its sign and part
      // follow the block form above
      const int qc = q >> 1;
#pragma unroll
      for (int u = 0; u < 8; u++) {
        const int kk = k0 + u, part = kk >= qc;
        const bool neg = isA ? part : (part & l.cpart);
        pc.x[u] = kk < q ? neg_if(__ldg(src + l.base + (int64_t)(kk - part * qc) * l.step + (part ^ l.cpart)), neg) : 0.0;
      }
    } else if (contig && q % VE == 0) {
      // lines of whole 16-byte vectors (tiles start on 16 bytes)
      const uint4* const v4 = reinterpret_cast<const uint4*>(src + l.base + k0);
#pragma unroll
      for (int v = 0; v < 8 / VE; v++) {
        uint4 r = make_uint4(0u, 0u, 0u, 0u);
        if (k0 + v * VE < q) r = __ldg(v4 + v);
        *reinterpret_cast<uint4*>(&pc.x[v * VE]) = r;
      }
    } else {
      const E* const v = src + l.base + (int64_t)k0 * l.step;
      const int64_t step = l.step;
#pragma unroll
      for (int u = 0; u < 8; u++) pc.x[u] = k0 + u < q ? __ldg(v + u * step) : E(0);
    }
  };
  auto store = [&](const Piece& pc) {
    if (pc.line < 0) return;
    if (pc.k0 < 1 << 30) {
      slice_store8<T, S>(pc.x, lines[pc.line].e, pc.dst, slice_stride);
    } else {  // an absent tile's line, or past the inner block's end
#pragma unroll
      for (int t = 0; t < S; t++)
        *reinterpret_cast<uint4*>(pc.dst + (size_t)t * slice_stride) = make_uint4(0u, 0u, 0u, 0u);
    }
  };
  int pass = bid % ny;
  if (pass >= total) return;
  Piece cur, nxt;
  load(cur, pass);
  for (;;) {
    pass += ny;
    const bool more = pass < total;
    if (more) load(nxt, pass);
    store(cur);
    if (!more) break;
    cur = nxt;
  }
}

}  // namespace

template <typename E, bool C = false>
cudaError_t launch_pack(const SplitArgs& a, PackGrid pg, cudaStream_t st, bool after) {
  // CTAs per group: one, or as many (up to a pass each) as fill the resident grid, where a
  // group's passes one after the other would be most of a small product's time
  const int groups = a.n_a_blocks + (a.n_b_blocks + kPackEntries - 1) / kPackEntries;
  const int passes = 2 * ((a.qmax + kSplitKC - 1) / kSplitKC);
  const int ny = std::max(1, std::min({kPackMaxY, passes, kPackResident / std::max(1, groups)}));
  const unsigned g = (unsigned)(pg.ncls + groups * ny);
  if (g == 0) return cudaSuccess;
  pg.ny = ny;
  pg.every = std::max(1, pg.ncls ? (int)(g / pg.ncls) * 3 / 4 : 1);
  auto launch = [&](void (*kernel)(SplitArgs, PackGrid)) {
    return launch_kernel(after, kernel, dim3(g), kPackThreads, 0, st, 1, a, pg);
  };
  switch (a.s * 2 + (a.fp16 ? 1 : 0)) {
    case 2: return launch(split_pack_kernel<__nv_bfloat16, 1, E, C>);
    case 3: return launch(split_pack_kernel<__half, 1, E, C>);
    case 4: return launch(split_pack_kernel<__nv_bfloat16, 2, E, C>);
    case 5: return launch(split_pack_kernel<__half, 2, E, C>);
    case 6: return launch(split_pack_kernel<__nv_bfloat16, 3, E, C>);
    case 7: return launch(split_pack_kernel<__half, 3, E, C>);
    case 8: return launch(split_pack_kernel<__nv_bfloat16, 4, E, C>);
    case 9: return launch(split_pack_kernel<__half, 4, E, C>);
    case 10: return launch(split_pack_kernel<__nv_bfloat16, 5, E, C>);
    case 11: return launch(split_pack_kernel<__half, 5, E, C>);
    case 12: return launch(split_pack_kernel<__nv_bfloat16, 6, E, C>);
    case 13: return launch(split_pack_kernel<__half, 6, E, C>);
    default: return cudaErrorInvalidValue;
  }
}

// CTAs of the pack launch that write offsets and scale classes: the blocks of lines, each in
// as many ranges of inner blocks (of 8 at least) as make about two of a resident grid
static PackGrid class_grid(const SplitArgs& a) {
  PackGrid g{0, 1, 1, 1};
  const int blocks = a.RB + a.CB;
  if (!(a.urow || !a.rowscale) || a.K == 0 || blocks == 0) return g;
  g.ranges = std::max(1, std::min({kClassMaxRanges, (a.K + 7) / 8, 2 * kPackResident / blocks}));
  g.ncls = blocks * g.ranges;
  return g;
}

int split_prep_kernels(const SplitArgs& a) {  // the kernels launch_split_prep launches
  int n = 0;
  if (a.n_a_tiles + a.n_b_tiles > 0) n++;
  if (a.rowscale && a.Mtot + a.Ntot > 0) n++;
  if (class_grid(a).ncls + a.n_a_blocks + a.n_b_blocks > 0) n++;
  return n;
}

cudaError_t launch_split_prep(const SplitArgs& a, cudaStream_t st, cudaEvent_t* ev, int* k, bool after) {
  const int tiles = a.n_a_tiles + a.n_b_tiles;
  cudaError_t e = cudaSuccess;
  if (tiles > 0 && a.rowscale) {
    const dim3 grid(tiles, kLinesY);
    e = a.f32 ? launch_kernel(after, split_exp_lines_kernel<float>, grid, 256, 0, st, 1, a)
              : launch_kernel(after, split_exp_lines_kernel<double>, grid, 256, 0, st, 1, a);
    after = true;
  } else if (tiles > 0) {
    int nz = 1;  // CTAs per tile: up to a resident grid's worth of CTAs in all
    while (nz < kExpCluster && 2 * nz * tiles <= kExpResident) nz *= 2;
    e = launch_kernel(after, split_exp_kernel, dim3(tiles * nz), kExpThreads, 0, st, nz, a);
    after = true;
  }
  if (e != cudaSuccess) return e;
  if (a.rowscale && a.Mtot + a.Ntot > 0) {  // the line maxima, and rowexp/colexp
    e = launch_kernel(after, split_scale_lines_kernel, dim3((unsigned)((a.Mtot + a.Ntot + 31) / 32)), 256, 0, st, 1, a);
    after = true;
  }
  if (ev) cudaEventRecord(ev[++*k], st), after = false;
  if (e != cudaSuccess) return e;
  const PackGrid pg = class_grid(a);
  e = a.f32 ? launch_pack<float>(a, pg, st, after)
            : a.cplx ? launch_pack<double, true>(a, pg, st, after) : launch_pack<double>(a, pg, st, after);
  if (e != cudaSuccess) return e;
  if (ev) cudaEventRecord(ev[++*k], st);
  return cudaGetLastError();
}

}  // namespace bsmm
