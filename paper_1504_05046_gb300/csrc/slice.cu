// Split-precision operands: exponents, scale classes and slices (the error-free slicing of
// split.cu's method; kernels 1 and 2 of its launch order). Everything here works on the
// operands' bit patterns with integer instructions: GB300's FP64 pipe takes 2 lanes per
// clock.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <climits>
#include <cstdint>
#include <type_traits>

#include "bsmm_internal.h"

namespace bsmm {

namespace {

constexpr int kAChunk = kSplitBM * kSplitKC * 2;  // bytes of one slice of a 128x32 A chunk

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
  return -126 - (__clz((int)m) - 8);  // subnormal: leading one at bit 31 - clz
}

__global__ void __launch_bounds__(256) split_exp_kernel(SplitArgs a) {
  const int b = blockIdx.x;
  const bool isA = b < a.n_a_tiles;
  const int t = isA ? a.a_tiles[b] : a.b_tiles[b - a.n_a_tiles];
  int rows, cols;
  int64_t off;
  tile_geometry(a, isA, t, rows, cols, off);
  // complex elements: the tile's doubles (both parts) at twice its complex offset; an A
  // tile holds r x q' doubles (q' = 2q), a B tile q' x c' / 2 (c' = 2c)
  const double* x = (isA ? a.A : a.B) + (off < 0 ? 0 : (a.cplx ? 2 * off : off));
  const int64_t n = (int64_t)rows * cols / (a.cplx && !isA ? 2 : 1);
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
      const int64_t bd = blockDim.x;
      for (int64_t e = threadIdx.x; e < n4; e += 4 * bd) {  // four loads in flight
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; u++) v[u] = e + u * bd < n4 ? __ldg(x4 + e + u * bd) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < 4; u++)
          m32 = max(m32, max(max(v[u].x & 0x7FFFFFFFu, v[u].y & 0x7FFFFFFFu),
                             max(v[u].z & 0x7FFFFFFFu, v[u].w & 0x7FFFFFFFu)));
      }
      for (int64_t e = (n4 << 2) + threadIdx.x; e < n; e += blockDim.x)
        m32 = max(m32, __float_as_uint(__ldg(xf + e)) & 0x7FFFFFFFu);
    }
    // as a double's magnitude bits: equal exponent of the top bit, so exponent_above agrees
    if (m32 >= kInfBits32)
      mx = kInfBits;
    else if (m32)
      mx = (unsigned long long)(exponent_above32(m32) + 1022) << 52;
  } else if (off >= 0) {
    // tiles start 16-byte aligned (even offsets): pairs of doubles, four pairs in flight
    const longlong2* x2 = reinterpret_cast<const longlong2*>(x);
    const int64_t n2 = n >> 1;
    const int64_t bd = blockDim.x;
    for (int64_t e = threadIdx.x; e < n2; e += 4 * bd) {
      longlong2 v[4];
#pragma unroll
      for (int u = 0; u < 4; u++) v[u] = e + u * bd < n2 ? __ldg(x2 + e + u * bd) : make_longlong2(0, 0);
#pragma unroll
      for (int u = 0; u < 4; u++) {
        mx = max(mx, (unsigned long long)v[u].x & kAbsMask);
        mx = max(mx, (unsigned long long)v[u].y & kAbsMask);
      }
    }
    if ((n & 1) && threadIdx.x == 0) mx = max(mx, mag_bits(__ldg(x + n - 1)));
  }
  __shared__ unsigned long long red[8];
  for (int o = 16; o; o >>= 1) mx = max(mx, (unsigned long long)__shfl_xor_sync(0xffffffffu, (long long)mx, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long m = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) m = max(m, red[w]);
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
// stored B tile (kZeroLine for an all-zero line); a non-finite value is reported by
// split_exp_kernel. One block per tile, one thread per line.
__global__ void __launch_bounds__(256) split_exp_lines_kernel(SplitArgs a) {
  const int b = blockIdx.x;
  const bool isA = b < a.n_a_tiles;
  const int t = isA ? a.a_tiles[b] : a.b_tiles[b - a.n_a_tiles];
  int rows, cols;
  int64_t off;
  tile_geometry(a, isA, t, rows, cols, off);
  if (off < 0) return;
  const double* x = (isA ? a.A : a.B) + off;
  const int i_or_k = isA ? t / a.K : t / a.N;
  const int k_or_j = isA ? t % a.K : t % a.N;
  const int nl = isA ? rows : cols;   // lines
  const int len = isA ? cols : rows;  // elements per line
  const bool tr = isA ? a.transa != 0 : a.transb != 0;
  // element u of line l: A row l is (l, u), B column l is (u, l); stored transposed or not
  const int64_t lstep = isA ? (tr ? 1 : cols) : (tr ? rows : 1);
  const int64_t ustep = isA ? (tr ? rows : 1) : (tr ? 1 : cols);
  if (a.cplx) {
    // complex elements: the plan's inner and column tilings count both parts, so an A tile
    // is rows x (2 qc) and a B tile (2 qc) x (2 cc) of the real product; a line's exponent
    // is that of the complex row (column) over both parts, and the B column cl and its
    // partner cl + cc (the same complex column's other part) share it
    const int qc = (isA ? cols : rows) >> 1;
    const int nlc = isA ? rows : cols >> 1;  // complex lines
    const int64_t cl_step = isA ? (tr ? 1 : qc) : (tr ? qc : 1);           // between lines
    const int64_t cu_step = isA ? (tr ? rows : 1) : (tr ? 1 : (cols >> 1));  // along a line
    const double* xc = (isA ? a.A : a.B) + 2 * off;
    for (int l = threadIdx.x; l < nlc; l += blockDim.x) {
      unsigned long long lm = 0;
      const double* line = xc + 2 * (l * cl_step);
      for (int u = 0; u < qc; u++) {
        lm = max(lm, mag_bits(__ldg(line + 2 * u * cu_step)));
        lm = max(lm, mag_bits(__ldg(line + 2 * u * cu_step + 1)));
      }
      const int e = (lm > 0 && lm < kInfBits) ? exponent_above(lm) : kZeroLine;
      if (isA) {
        a.eArow[(int64_t)k_or_j * a.Mtot + a.ro[i_or_k] + l] = e;
      } else {
        a.eBcol[(int64_t)i_or_k * a.Ntot + a.co[k_or_j] + l] = e;
        a.eBcol[(int64_t)i_or_k * a.Ntot + a.co[k_or_j] + nlc + l] = e;
      }
    }
    return;
  }
  for (int l = threadIdx.x; l < nl; l += blockDim.x) {
    int e = kZeroLine;
    if (a.f32) {
      uint32_t lm = 0;
      const float* line = (isA ? a.Af : a.Bf) + off + l * lstep;
      for (int u = 0; u < len; u++) lm = max(lm, __float_as_uint(__ldg(line + u * ustep)) & 0x7FFFFFFFu);
      if (lm > 0 && lm < kInfBits32) e = exponent_above32(lm);
    } else {
      unsigned long long lm = 0;
      const double* line = x + l * lstep;
      for (int u = 0; u < len; u++) lm = max(lm, mag_bits(__ldg(line + u * ustep)));
      if (lm > 0 && lm < kInfBits) e = exponent_above(lm);
    }
    if (isA)
      a.eArow[(int64_t)k_or_j * a.Mtot + a.ro[i_or_k] + l] = e;
    else
      a.eBcol[(int64_t)i_or_k * a.Ntot + a.co[k_or_j] + l] = e;
  }
}

// ---------------------------------------------------------------- kernel 1b: largest exponents
// Per row block i: Emax_A(i) = the largest exponent of its stored A tiles (0 when none);
// the same per column block for B. One block per row or column block, its threads
// spread over the K inner blocks. The contraction adds each tile pair's exact integer at
// the binary position GUARD + rowexp + colexp of a 128-bit accumulator whose unit is
// 2^(Emax_A(i) + Emax_B(j) - 7(s+1) - GUARD); the class kernel writes rowexp and colexp.
__global__ void __launch_bounds__(256) split_emax_kernel(SplitArgs a) {
  const bool isA = (int)blockIdx.x < a.M;
  const int t = isA ? blockIdx.x : blockIdx.x - a.M;
  int em = INT_MIN;
  if (isA ? a.r[t] > 0 : a.c[t] > 0) {
    for (int k = threadIdx.x; k < a.K; k += blockDim.x) {
      if (a.q[k] <= 0) continue;
      if (isA) {
        if (a.am[(int64_t)t * a.K + k]) em = max(em, a.eA[(int64_t)t * a.K + k]);
      } else {
        if (a.bm[(int64_t)k * a.N + t]) em = max(em, a.eB[(int64_t)k * a.N + t]);
      }
    }
  }
  __shared__ int red[8];
  for (int o = 16; o; o >>= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = em;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); w++) em = max(em, red[w]);
    if (em == INT_MIN) em = 0;
    if (isA)
      a.eAmax[t] = em;
    else
      a.eBmax[t] = em;
  }
}

// ---------------------------------------------------------------- kernel 1b': line scales
// Row/column scaling: one thread per row m of A (per column n of B): Emax = the largest
// exponent of that line over its stored tiles (all-zero lines excluded; 0 when none), and
// rowexp[k][m] = e(m, k) - Emax (colexp likewise), 0 where there is no tile or the line is
// zero there (its slices are zero).
__global__ void __launch_bounds__(256) split_scale_lines_kernel(SplitArgs a) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < a.Mtot) {
    const int64_t m = t;
    const int i = a.row_tile[m];
    int em = INT_MIN;
    for (int k = 0; k < a.K; k++) {
      const int e = a.eArow[(int64_t)k * a.Mtot + m];
      if (a.am[(int64_t)i * a.K + k] && a.q[k] > 0 && e != kZeroLine) em = max(em, e);
    }
    if (em == INT_MIN) em = 0;
    a.eAmaxr[m] = em;
    for (int k = 0; k < a.K; k++) {
      const int e = a.eArow[(int64_t)k * a.Mtot + m];
      const bool pres = a.am[(int64_t)i * a.K + k] && a.q[k] > 0 && e != kZeroLine;
      a.rowexp[(int64_t)k * a.Mtot + m] = (int16_t)(pres ? e - em : 0);
    }
  } else if (t < a.Mtot + a.Ntot) {
    const int64_t n = t - a.Mtot;
    const int j = a.col_tile[n];
    int em = INT_MIN;
    for (int k = 0; k < a.K; k++) {
      const int e = a.eBcol[(int64_t)k * a.Ntot + n];
      if (a.bm[(int64_t)k * a.N + j] && a.q[k] > 0 && e != kZeroLine) em = max(em, e);
    }
    if (em == INT_MIN) em = 0;
    a.eBmaxc[n] = em;
    for (int k = 0; k < a.K; k++) {
      const int e = a.eBcol[(int64_t)k * a.Ntot + n];
      const bool pres = a.bm[(int64_t)k * a.N + j] && a.q[k] > 0 && e != kZeroLine;
      a.colexp[(int64_t)k * a.colexp_ld + n] = (int16_t)(pres ? e - em : 0);
    }
  }
}

// ---------------------------------------------------------------- kernel 1c: offsets and scale classes
// One warp per (k block, row block) and per (k block, column block). With one scale per
// tile it first writes the offsets of its rows, rowexp[k][m] = e_A(i,k) - Emax_A(i) for a
// stored tile (0 for an absent one), or of its columns (colexp); with one scale per row
// and column the line kernel wrote them.
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
__global__ void __launch_bounds__(256) split_class_kernel(SplitArgs a) {
  // one warp per (k block, row block) and per (k block, column block); lanes over the lines
  const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t nr = (int64_t)a.K * a.RB, nc = (int64_t)a.K * a.CB;
  int lo = INT_MAX, hi = INT_MIN, emx = INT_MIN;
  if (wid < nr) {
    const int k = (int)(wid / a.RB), rb = (int)(wid % a.RB);
    const int64_t m0 = (int64_t)rb * kSplitBM;
    const int64_t m1 = m0 + kSplitBM < a.Mtot ? m0 + kSplitBM : a.Mtot;
    for (int64_t m = m0 + lane; m < m1; m += 32) {
      const int i = a.row_tile[m];
      const int emax_m = a.rowscale ? a.eAmaxr[m] : a.eAmax[i];
      emx = max(emx, emax_m);
      bool pres = a.q[k] > 0 && a.am[(int64_t)i * a.K + k];
      int eabs = 0;
      if (!a.rowscale) {
        eabs = pres ? a.eA[(int64_t)i * a.K + k] : 0;
        a.rowexp[(int64_t)k * a.Mtot + m] = (int16_t)(pres ? eabs - emax_m : 0);
      } else if (pres) {
        eabs = a.eArow[(int64_t)k * a.Mtot + m];
        pres = eabs != kZeroLine;
      }
      if (pres) {
        lo = min(lo, eabs);
        hi = max(hi, eabs);
      }
    }
    for (int o = 16; o; o >>= 1) {
      lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      emx = max(emx, __shfl_xor_sync(0xffffffffu, emx, o));
    }
    if (k == 0)
      for (int64_t m = m0 + lane; m < m1; m += 32) {
        const int e = a.rowscale ? a.eAmaxr[m] : a.eAmax[a.row_tile[m]];
        a.emaxr[m] = e;
        if (a.urow) a.rowadj[m] = (int16_t)(emx - e);
      }
    if (a.urow && lane == 0) a.urow[wid] = (int16_t)(lo > hi ? 0 : lo == hi ? lo - emx : kNonUniform);
  } else if (wid < nr + nc) {
    const int64_t u = wid - nr;
    const int k = (int)(u / a.CB), cb = (int)(u % a.CB);
    const int64_t n0 = (int64_t)cb * a.tn;
    const int64_t n1 = n0 + a.tn < a.Ntot ? n0 + a.tn : a.Ntot;
    for (int64_t n = n0 + lane; n < n1; n += 32) {
      const int j = a.col_tile[n];
      const int emax_n = a.rowscale ? a.eBmaxc[n] : a.eBmax[j];
      emx = max(emx, emax_n);
      bool pres = a.q[k] > 0 && a.bm[(int64_t)k * a.N + j];
      int eabs = 0;
      if (!a.rowscale) {
        eabs = pres ? a.eB[(int64_t)k * a.N + j] : 0;
        a.colexp[(int64_t)k * a.colexp_ld + n] = (int16_t)(pres ? eabs - emax_n : 0);
      } else if (pres) {
        eabs = a.eBcol[(int64_t)k * a.Ntot + n];
        pres = eabs != kZeroLine;
      }
      if (pres) {
        lo = min(lo, eabs);
        hi = max(hi, eabs);
      }
    }
    for (int o = 16; o; o >>= 1) {
      lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      emx = max(emx, __shfl_xor_sync(0xffffffffu, emx, o));
    }
    if (k == 0)
      for (int64_t n = n0 + lane; n < n1; n += 32) {
        const int e = a.rowscale ? a.eBmaxc[n] : a.eBmax[a.col_tile[n]];
        a.emaxc[n] = e;
        if (a.ucol) a.coladj[n] = (int16_t)(emx - e);
      }
    if (a.ucol && lane == 0) a.ucol[u] = (int16_t)(lo > hi ? 0 : lo == hi ? lo - emx : kNonUniform);
  }
}

// ---------------------------------------------------------------- kernel 2: slices
// Slice 8 consecutive inner elements (one 16-byte chunk of a swizzled row) of one
// packed row and store the s chunks.
// The slicing recurrence N_t = rint(rho_{t-1} 2^(7t)), rho_t = rho_{t-1} - N_t 2^(-7t)
// telescopes: with Z_t = sum_{u<=t} N_u 2^(7(t-u)) one has Z_t = rint(x 2^(7t-e)) (the
// subtracted 128 Z_{t-1} is even, so round-half-even commutes with it), hence
// N_t = Z_t - 128 Z_{t-1}. Each Z_t is computed exactly from the mantissa with integer
// shifts and a round-half-even step; no floating-point operation is involved.
// All Z_t of one element come from one window of its significand: x 2^-e = +-m 2^ex with
// an integer m < 2^53; at the finest level t = S the window is W = floor(m 2^-k),
// k = -(ex + 7S), with the round bit R (bit k-1 of m) and the sticky flag (any lower bit
// set); level t < S drops a = 7(S-t) more bits of W, rounding with bit a-1 of W and the
// bits below it (the finest level's fraction included). The window's shifts are
// compile-time constants. Only the low 32 bits of Z_t are kept: N_t is small, so
// Z_t - 128 Z_(t-1) is exact in 32-bit wrap-around arithmetic.
struct SliceWindow {
  unsigned long long W;  // floor(m 2^-k)
  bool R, T, F;          // round bit and sticky bits at the finest level; F = any bit below W
  __device__ __forceinline__ void init(unsigned long long m, int k) {
    if (k <= 0) {  // exact (a subnormal tile's elements, or a non-finite input already reported)
      W = -k >= 63 ? 0ull : m << -k;
      R = T = F = false;
    } else if (k >= 64) {
      W = 0ull;
      R = false;
      T = F = m != 0ull;
    } else {
      W = m >> k;
      R = (m >> (k - 1)) & 1ull;
      T = (m & ((1ull << (k - 1)) - 1ull)) != 0ull;
      F = R || T;
    }
  }
  // low 32 bits of Z at the level a bits coarser than the finest. For A > 0 the rounding
  // is one addition: with h = 2^(A-1) and b = (bit A of W) | F, W + h - 1 + b carries into
  // bit A exactly when the dropped part exceeds h, or equals h with an odd quotient or a
  // nonzero fraction below W (round half to even).
  template <int A>
  __device__ __forceinline__ uint32_t z() const {
    if constexpr (A == 0) {
      return (uint32_t)W + ((R && (T || (W & 1ull))) ? 1u : 0u);
    } else {
      const unsigned long long b = ((W >> A) & 1ull) | (F ? 1ull : 0ull);
      return (uint32_t)((W + ((1ull << (A - 1)) - 1ull) + b) >> A);
    }
  }
};

template <typename T>
__device__ __forceinline__ uint16_t small_int_bits(int n) {  // |n| <= 256, exact in bf16/fp16
  const float f = __int_as_float(0x4B400000 + n) - 12582912.0f;  // exact for |n| < 2^22
  if constexpr (std::is_same<T, __nv_bfloat16>::value) {
    return (uint16_t)(__float_as_uint(f) >> 16);  // <= 8 significant bits: truncation is exact
  } else {
    return __half_as_ushort(__float2half_rn(f));
  }
}

template <typename T, int S, int t>
__device__ __forceinline__ void slice_level(const SliceWindow (&w)[8], const bool (&neg)[8], uint32_t (&zp)[8],
                                            uint8_t* base, int slice_stride, uint32_t soff) {
  if constexpr (t <= S) {
    uint16_t h[8];
#pragma unroll
    for (int u = 0; u < 8; u++) {
      uint32_t zt = w[u].template z<kSplitBeta * (S - t)>();
      if (neg[u]) zt = 0u - zt;
      h[u] = small_int_bits<T>((int)(zt - (zp[u] << kSplitBeta)));
      zp[u] = zt;
    }
    *reinterpret_cast<uint4*>(base + (size_t)(t - 1) * slice_stride + soff) = *reinterpret_cast<uint4*>(h);
    slice_level<T, S, t + 1>(w, neg, zp, base, slice_stride, soff);
  }
}

// x 2^-e = +-m 2^ex with an integer significand m, from the bits of a double or a float
__device__ __forceinline__ void decode(double x, int e, bool& neg, unsigned long long& m, int& ex) {
  const long long b = __double_as_longlong(x);
  neg = b < 0;
  const int be = (int)((b >> 52) & 0x7FF);
  const unsigned long long frac = (unsigned long long)b & ((1ull << 52) - 1ull);
  m = be ? (frac | (1ull << 52)) : frac;
  ex = (be ? be : 1) - 1075 - e;
}
__device__ __forceinline__ void decode(float x, int e, bool& neg, unsigned long long& m, int& ex) {
  const uint32_t b = __float_as_uint(x);
  neg = (b >> 31) != 0;
  const int be = (int)((b >> 23) & 0xFF);
  const uint32_t frac = b & 0x7FFFFFu;
  m = be ? (frac | 0x800000u) : frac;
  ex = (be ? be : 1) - 150 - e;
}

template <typename T, int S, typename E>
__device__ __forceinline__ void slice_store8(const E (&x)[8], int e, uint8_t* base, int slice_stride, uint32_t soff) {
  SliceWindow w[8];
  bool neg[8];
  uint32_t zp[8];
#pragma unroll
  for (int u = 0; u < 8; u++) {
    unsigned long long m;
    int ex;
    decode(x[u], e, neg[u], m, ex);
    w[u].init(m, -(ex + kSplitBeta * S));
    zp[u] = 0u;
  }
  slice_level<T, S, 1>(w, neg, zp, base, slice_stride, soff);
}

// Complex elements (CPLX): the real product's A tile is [Ar, -Ai] (inner index kk' < q
// takes the real part of column kk', kk' >= q the negated imaginary part of column kk' - q)
// and its B tile [[Br, Bi], [Bi, -Br]] (row half and column half pick the part and the
// sign); q and c below are the doubled sizes, the stored complex tile is q/2 and c/2 wide.
__device__ __forceinline__ double neg_if(double v, bool n) {  // sign flip as bits (no FP64 op)
  return n ? __longlong_as_double(__double_as_longlong(v) ^ (long long)0x8000000000000000ull) : v;
}

template <typename T, int S, typename E, bool CPLX = false>
__global__ void __launch_bounds__(256) split_pack_kernel(SplitArgs a) {
  constexpr int s = S;
  const E* Ae = reinterpret_cast<const E*>(std::is_same<E, float>::value ? (const void*)a.Af : (const void*)a.A);
  const E* Be = reinterpret_cast<const E*>(std::is_same<E, float>::value ? (const void*)a.Bf : (const void*)a.B);
  if ((int)blockIdx.x < a.n_a_blocks) {
    // A block (rb, kt): chunks of 128 rows x 32 inner elements
    const int blk = a.a_blocks[blockIdx.x];
    const int rb = blk / a.K, kt = blk % a.K;
    const int q = a.q[kt];
    const int nkc = (q + kSplitKC - 1) / kSplitKC;
    uint8_t* out = a.apk + a.apk_off[blk];
    for (int item = threadIdx.x; item < nkc * kSplitBM * 4; item += blockDim.x) {
      const int ch = item & 3, rr = (item >> 2) % kSplitBM, kc = (item >> 2) / kSplitBM;
      const int64_t m = (int64_t)rb * kSplitBM + rr;
      E x[8];
      int e = 0;
      bool present = false;
      int64_t off = -1;
      int i = 0;
      if (m < a.Mtot) {
        i = a.row_tile[m];
        present = a.am[(int64_t)i * a.K + kt] != 0;
        off = a.transa ? a.a_off[(int64_t)kt * a.M + i] : a.a_off[(int64_t)i * a.K + kt];
        if (present && off < 0) {
          atomicOr(a.err, kErrBadOffset);
          present = false;
        }
        e = a.rowscale ? a.eArow[(int64_t)kt * a.Mtot + m] : a.eA[(int64_t)i * a.K + kt];
      }
      const int64_t lr = m - (m < a.Mtot ? a.ro[i] : 0);
      // element (lr, k) of A_ik at line + k * step, stored transposed or not
      const int64_t step = a.transa ? (m < a.Mtot ? a.r[i] : 0) : 1;
      const int k0 = kc * kSplitKC + ch * 8;
      if constexpr (CPLX) {
        // complex element (lr, kc) of the tile at row + 2 kc cstep (cstep = 1, or the tile's
        // row count when stored transposed); part 0 real, 1 imaginary
        const int qc = q >> 1;
        const int64_t cstep = a.transa ? step : 1;
        const double* row = a.A + 2 * (off + (a.transa ? lr : lr * qc));
#pragma unroll
        for (int u = 0; u < 8; u++) {
          const int kk = k0 + u, part = kk >= qc;
          x[u] = (present && kk < q) ? neg_if(__ldg(row + 2 * (kk - part * qc) * cstep + part), part) : 0.0;
        }
      } else {
        const E* line = Ae + off + (a.transa ? lr : lr * q);
#pragma unroll
        for (int u = 0; u < 8; u++) x[u] = (present && k0 + u < q) ? __ldg(line + (k0 + u) * step) : E(0);
      }
      slice_store8<T, S>(x, e, out + (size_t)kc * s * kAChunk, kAChunk, swz64(rr, ch * 8));
    }
  } else {
    // B block (kt, cb): chunks of tn rows (columns of B) x 32 inner elements, transposed
    const int blk = a.b_blocks[blockIdx.x - a.n_a_blocks];
    const int kt = blk / a.CB, cb = blk % a.CB;
    const int q = a.q[kt];
    const int tn = a.tn;
    const int nkc = (q + kSplitKC - 1) / kSplitKC;
    const int bchunk = tn * kSplitKC * 2;
    uint8_t* out = a.bpk + a.bpk_off[blk];
    for (int item = threadIdx.x; item < nkc * tn * 4; item += blockDim.x) {
      const int nn = item % tn, ch = (item / tn) & 3, kc = (item / tn) >> 2;
      const int64_t n = (int64_t)cb * tn + nn;
      E x[8];
      int e = 0;
      bool present = false;
      int64_t off = -1;
      int j = 0, cj = 0;
      if (n < a.Ntot) {
        j = a.col_tile[n];
        cj = a.c[j];
        present = a.bm[(int64_t)kt * a.N + j] != 0;
        off = a.transb ? a.b_off[(int64_t)j * a.K + kt] : a.b_off[(int64_t)kt * a.N + j];
        if (present && off < 0) {
          atomicOr(a.err, kErrBadOffset);
          present = false;
        }
        e = a.rowscale ? a.eBcol[(int64_t)kt * a.Ntot + n] : a.eB[(int64_t)kt * a.N + j];
      }
      const int64_t lc = n - (n < a.Ntot ? a.co[j] : 0);
      // element (k, lc) of B_kj at line + k * step, stored transposed or not
      const int64_t step = a.transb ? 1 : cj;
      const int k0 = kc * kSplitKC + ch * 8;
      if constexpr (CPLX) {
        // complex element (kc, c) of the tile at col + 2 kc kstep: kstep = the tile's complex
        // column count, or 1 when stored transposed (then column c starts c * qc in)
        const int qc = q >> 1, cc = cj >> 1;
        const int cpart = lc >= cc;
        const int64_t kstep = a.transb ? 1 : cc;
        const double* col = a.B + 2 * (off + (lc - cpart * cc) * (a.transb ? qc : 1));
#pragma unroll
        for (int u = 0; u < 8; u++) {
          const int kk = k0 + u, rpart = kk >= qc;
          x[u] = (present && kk < q)
                     ? neg_if(__ldg(col + 2 * (int64_t)(kk - rpart * qc) * kstep + (rpart ^ cpart)), rpart & cpart)
                     : 0.0;
        }
      } else {
        const E* line = Be + off + (a.transb ? lc * q : lc);
#pragma unroll
        for (int u = 0; u < 8; u++) x[u] = (present && k0 + u < q) ? __ldg(line + (k0 + u) * step) : E(0);
      }
      slice_store8<T, S>(x, e, out + (size_t)kc * s * bchunk, bchunk, swz64(nn, ch * 8));
    }
  }
}

}  // namespace

template <typename E, bool C = false>
cudaError_t launch_pack(const SplitArgs& a, unsigned g, cudaStream_t st) {
  switch (a.s * 2 + (a.fp16 ? 1 : 0)) {
    case 2: split_pack_kernel<__nv_bfloat16, 1, E, C><<<g, 256, 0, st>>>(a); break;
    case 3: split_pack_kernel<__half, 1, E, C><<<g, 256, 0, st>>>(a); break;
    case 4: split_pack_kernel<__nv_bfloat16, 2, E, C><<<g, 256, 0, st>>>(a); break;
    case 5: split_pack_kernel<__half, 2, E, C><<<g, 256, 0, st>>>(a); break;
    case 6: split_pack_kernel<__nv_bfloat16, 3, E, C><<<g, 256, 0, st>>>(a); break;
    case 7: split_pack_kernel<__half, 3, E, C><<<g, 256, 0, st>>>(a); break;
    case 8: split_pack_kernel<__nv_bfloat16, 4, E, C><<<g, 256, 0, st>>>(a); break;
    case 9: split_pack_kernel<__half, 4, E, C><<<g, 256, 0, st>>>(a); break;
    case 10: split_pack_kernel<__nv_bfloat16, 5, E, C><<<g, 256, 0, st>>>(a); break;
    case 11: split_pack_kernel<__half, 5, E, C><<<g, 256, 0, st>>>(a); break;
    case 12: split_pack_kernel<__nv_bfloat16, 6, E, C><<<g, 256, 0, st>>>(a); break;
    case 13: split_pack_kernel<__half, 6, E, C><<<g, 256, 0, st>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

int split_prep_kernels(const SplitArgs& a) {  // the kernels launch_split_prep launches
  int n = 0;
  if (a.n_a_tiles + a.n_b_tiles > 0) n += a.rowscale ? 2 : 1;
  if (a.rowscale ? a.Mtot + a.Ntot > 0 : a.M + a.N > 0) n++;
  if ((a.urow || !a.rowscale) && (int64_t)a.K * (a.RB + a.CB) > 0) n++;
  if (a.n_a_blocks + a.n_b_blocks > 0) n++;
  return n;
}

cudaError_t launch_split_prep(const SplitArgs& a, cudaStream_t st, cudaEvent_t* ev, int* k) {
  if (a.n_a_tiles + a.n_b_tiles > 0) {
    split_exp_kernel<<<a.n_a_tiles + a.n_b_tiles, 256, 0, st>>>(a);
    if (a.rowscale) split_exp_lines_kernel<<<a.n_a_tiles + a.n_b_tiles, 256, 0, st>>>(a);
  }
  if (a.rowscale) {
    // the per-tile maxima (eAmax/eBmax) are not used in this mode; the line kernel writes
    // rowexp/colexp and the line maxima
    const int64_t lines = a.Mtot + a.Ntot;
    if (lines > 0) split_scale_lines_kernel<<<(unsigned)((lines + 255) / 256), 256, 0, st>>>(a);
  } else if (a.M + a.N > 0) {
    split_emax_kernel<<<a.M + a.N, 256, 0, st>>>(a);
  }
  // tile scaling: the offsets rowexp/colexp; both: the scale classes (when kept)
  const int64_t ncls = (int64_t)a.K * (a.RB + a.CB);
  if ((a.urow || !a.rowscale) && ncls > 0) split_class_kernel<<<(unsigned)((ncls * 32 + 255) / 256), 256, 0, st>>>(a);
  if (ev) cudaEventRecord(ev[++*k], st);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (a.n_a_blocks + a.n_b_blocks > 0) {
    const unsigned g = (unsigned)(a.n_a_blocks + a.n_b_blocks);
    cudaError_t pe = a.f32 ? launch_pack<float>(a, g, st)
                           : a.cplx ? launch_pack<double, true>(a, g, st) : launch_pack<double>(a, g, st);
    if (pe != cudaSuccess) return pe;
  }
  if (ev) cudaEventRecord(ev[++*k], st);
  return cudaGetLastError();
}

}  // namespace bsmm
