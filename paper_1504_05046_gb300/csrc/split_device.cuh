// Device code shared by the contraction kernels: bounded waits, bulk copies, tcgen05, the
// exact 128-bit accumulation and its rounding, the C store, and the walk over a unit's inner
// blocks with the accumulation-group rule. (split.cu describes the method.)
#pragma once

#include <cstdint>
#include <type_traits>

#include "bsmm_internal.h"
#include "overlap.cuh"

namespace bsmm {

namespace {

constexpr int64_t kWaitNs = 4000000000LL;  // bounded waits: 4 s, then error + abort
constexpr int kEpiThreads = kSplitEpiWarps * 32;
constexpr uint32_t kTmemCols = 512;
constexpr int kAChunk = kSplitBM * kSplitKC * 2;  // bytes of one slice of a 128x32 A chunk

__device__ __forceinline__ int64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return (int64_t)t;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Single-thread bounded wait. False on timeout (sets the error word and the abort
// flag) or when another role aborted.
__device__ bool wait1(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int32_t* err,
                      int64_t limit = kWaitNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const int64_t t0 = gtimer();
  for (uint32_t spin = 1;; spin++) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if ((spin & 63) == 0 && gtimer() - t0 > limit) {
      *abort_flag = 1;
      atomicOr(err, kErrTimeout);
      return false;
    }
  }
}

constexpr uint32_t kGroupPollNs = 128;  // the epilogue's sleep between polls for the next group

// Warp-uniform bounded wait (every lane polls; the decision is taken by the warp). A warp
// whose wait is not on the critical path passes sleep_ns > 0: it sleeps between polls,
// leaving the issue slots to the warps that are.
__device__ bool wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int32_t* err,
                          int64_t limit = kWaitNs, uint32_t sleep_ns = 0) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const int64_t t0 = gtimer();
  for (uint32_t spin = 1;; spin++) {
    if (sleep_ns) __nanosleep(sleep_ns);
    const bool ok = mbar_try_wait(bar, parity);
    if (__all_sync(0xffffffffu, ok)) return true;
    int stop = *abort_flag;
    if ((spin & 63) == 0 && gtimer() - t0 > limit) stop = 2;
    if (__any_sync(0xffffffffu, stop != 0)) {
      if (stop == 2 && (threadIdx.x & 31) == 0) {
        *abort_flag = 1;
        atomicOr(err, kErrTimeout);
      }
      __syncwarp();
      return false;
    }
  }
}

// ---------------------------------------------------------------- bulk copy
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}


// ---------------------------------------------------------------- tcgen05
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem]^T, kind::f16 (bf16 or fp16 in, fp32 accumulate)
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_zero4(uint32_t taddr) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%1,%1,%1};" ::"r"(taddr), "r"(0u) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_zero8(uint32_t taddr) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr), "r"(0u) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// One lane of a converged warp. Code that a whole warp runs up to this choice keeps its
// addresses and descriptors in uniform registers, which tcgen05.mma takes them from.
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(r));
  return r != 0;
}

// Shared-memory matrix descriptor: K-major operand, 64-byte swizzle, 8-row groups of
// 64-byte rows (stride between 8-row groups = 512 bytes).
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);  // start address (16-byte units)
  d |= (uint64_t)0 << 16;                   // leading byte offset: unused (one swizzle atom along K)
  d |= (uint64_t)(512u >> 4) << 32;         // stride byte offset
  d |= (uint64_t)1 << 46;                   // descriptor version for tcgen05
  d |= (uint64_t)4 << 61;                   // layout: 64-byte swizzle
  return d;
}

// Instruction descriptor, kind::f16: D fp32, A and B bf16 (or fp16), both K-major.
__device__ __forceinline__ uint32_t idesc_f16(int M, int N, bool fp16) {
  const uint32_t fmt = fp16 ? 0u : 1u;
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ---------------------------------------------------------------- exact accumulation
// The exact integer of an element's accumulation group from its diagonal sums (integers of
// magnitude <= 2^24 as floats): T = sum_d S_d 2^(7(S-1-d)), |T| < 2^59.
// Bound by the float-to-integer conversions: 16 lanes per clock and SM, so six of them hold
// two warps of a scheduler for 96 cycles, and all else an element needs fits beside them.
// Two neighbouring diagonals a, b are therefore joined into a 2^7 + b (below 2^31 from 3
// slices on) with one conversion where kMagic: b's part above 7 bits moves over to a (both
// exact: |a| <= 2^24 (S+1)/(S+2), the carry <= 2^17), and the small rest is read off the bits
// of rest + 1.5 2^23. Two of the three joins of 6 slices that way balance the conversions
// with the other instructions: 112 to 90 cycles per element of two warps (128 when every
// diagonal was converted and shifted on its own).
__device__ __forceinline__ int to_int(float x) {  // an integer's value
  int r;
  asm("cvt.rni.s32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}
template <bool kMagic>
__device__ __forceinline__ int join_pair(float a, float b) {
  if constexpr (!kMagic) return to_int(a) * 128 + to_int(b);
  constexpr float kM = 12582912.0f;                     // 1.5 2^23: adding it rounds to an integer
  const float h = fmaf(b, 1.0f / 128, kM) - kM;         // the carry into a
  const float rest = fmaf(h, -128.0f, b);               // |rest| <= 64
  return to_int(a + h) * 128 + (__float_as_int(rest + kM) - __float_as_int(kM));
}
template <int S, int CW, bool kMagic>
__device__ __forceinline__ long long diagonal_sum(const uint32_t (&v)[S][CW], int c) {
  auto f = [&](int d) { return __uint_as_float(v[d][c]); };
  if constexpr (S == 1) {
    return to_int(f(0));
  } else if constexpr (S == 2) {
    return (long long)to_int(f(0)) * 128 + to_int(f(1));
  } else {
    long long T = join_pair<kMagic>(f(S - 2), f(S - 1));
    if constexpr (S >= 4) T += (long long)join_pair<kMagic && (S >= 5)>(f(S - 4), f(S - 3)) * (1ll << 14);
    if constexpr (S == 3) T += (long long)to_int(f(0)) * (1ll << 14);
    if constexpr (S == 5) T += (long long)to_int(f(0)) * (1ll << 28);
    if constexpr (S == 6) T += (long long)join_pair<false>(f(0), f(1)) * (1ll << 28);
    return T;
  }
}

// w (four 32-bit words, two's complement) += T * 2^sh, with floor(T / 2^-sh) for sh < 0.
// |T| < 2^59 and sh <= kSplitGuard for every accumulation group (its depth keeps each FP32
// partial sum below 2^24); an absent tile pair has T = 0.
__device__ __forceinline__ void acc_add(uint32_t (&w)[4], long long T, int sh) {
  const int sl = min(max(sh, 0), 63);
  long long lo = T << sl;
  long long hi = sl ? (T >> (64 - sl)) : (T >> 63);
  if (sh < 0) {
    lo = T >> min(-sh, 63);
    hi = T >> 63;
  }
  asm("add.cc.u32 %0, %0, %4;\n\t"
      "addc.cc.u32 %1, %1, %5;\n\t"
      "addc.cc.u32 %2, %2, %6;\n\t"
      "addc.u32 %3, %3, %7;"
      : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3])
      : "r"((uint32_t)lo), "r"((uint32_t)((unsigned long long)lo >> 32)), "r"((uint32_t)hi),
        "r"((uint32_t)((unsigned long long)hi >> 32)));
}

// w += T
__device__ __forceinline__ void acc_add_plain(uint32_t (&w)[4], long long T) {
  const uint32_t s = (uint32_t)(T >> 63);
  asm("add.cc.u32 %0, %0, %4;\n\t"
      "addc.cc.u32 %1, %1, %5;\n\t"
      "addc.cc.u32 %2, %2, %6;\n\t"
      "addc.u32 %3, %3, %6;"
      : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3])
      : "r"((uint32_t)T), "r"((uint32_t)((unsigned long long)T >> 32)), "r"(s));
}

// w *= 2^sh (0 <= sh < 64)
__device__ __forceinline__ void acc_shl(uint32_t (&w)[4], int sh) {
  const bool word = sh >= 32;
  const uint32_t w3 = word ? w[2] : w[3], w2 = word ? w[1] : w[2], w1 = word ? w[0] : w[1], w0 = word ? 0u : w[0];
  w[3] = __funnelshift_l(w2, w3, sh);  // (shifts by sh mod 32)
  w[2] = __funnelshift_l(w1, w2, sh);
  w[1] = __funnelshift_l(w0, w1, sh);
  w[0] = __funnelshift_l(0u, w0, sh);
}

// 64-bit window of a 128-bit magnitude shifted right by r (0 <= r < 128)
__device__ __forceinline__ unsigned long long shr128(unsigned long long hi, unsigned long long lo, int r) {
  if (r == 0) return lo;
  if (r < 64) return (lo >> r) | (hi << (64 - r));
  return hi >> (r - 64);
}

// |w| of the 128-bit two's-complement integer w shifted left until its leading one is bit
// 31 of t[0] (t[0] is the most significant of the window's 96 bits; the bits below the
// window are or-ed into the last bit of t[2], which only ever serves as sticky bits): no
// branch, so a warp whose 32 sums differ in magnitude runs every instruction once. Returns
// the leading one's position; w = 0 gives t[0] = 0.
__device__ __forceinline__ int acc_normalise(const uint32_t (&w)[4], uint32_t (&t)[3]) {
  const uint32_t s = (uint32_t)((int32_t)w[3] >> 31);
  uint32_t h0 = w[0] ^ s, h1 = w[1] ^ s, h2 = w[2] ^ s, h3 = w[3] ^ s;
  asm("sub.cc.u32 %0, %0, %4;\n\t"  // minus -1 = plus one for a negative w
      "subc.cc.u32 %1, %1, %4;\n\t"
      "subc.cc.u32 %2, %2, %4;\n\t"
      "subc.u32 %3, %3, %4;"
      : "+r"(h0), "+r"(h1), "+r"(h2), "+r"(h3)
      : "r"(s));
  int msb = 127;
  const bool z64 = (h3 | h2) == 0u;
  h3 = z64 ? h1 : h3;
  h2 = z64 ? h0 : h2;
  h1 = z64 ? 0u : h1;
  h0 = z64 ? 0u : h0;
  msb = z64 ? 63 : msb;
  const bool z32 = h3 == 0u;
  h3 = z32 ? h2 : h3;
  h2 = z32 ? h1 : h2;
  h1 = z32 ? h0 : h1;
  h0 = z32 ? 0u : h0;
  const int c = __clz((int)h3);  // 32 only when w = 0
  msb -= (z32 ? 32 : 0) + c;
  t[0] = __funnelshift_lc(h2, h3, c);
  t[1] = __funnelshift_lc(h1, h2, c);
  t[2] = __funnelshift_lc(h0, h1, c) | (h0 != 0u ? 1u : 0u);
  return msb;
}

// Bit b of the 128-bit magnitude (hi, lo), and whether any of its bits below b is set.
__device__ __forceinline__ bool bit128(unsigned long long hi, unsigned long long lo, int b) {
  return b < 64 ? (lo >> b) & 1 : (hi >> (b - 64)) & 1;
}
__device__ __forceinline__ bool low128(unsigned long long hi, unsigned long long lo, int b) {  // bits [0, b)
  if (b <= 0) return false;
  if (b <= 64) return (b == 64 ? lo : lo & ((1ull << b) - 1)) != 0;
  if (b >= 128) return (lo | hi) != 0;
  return lo != 0 || (hi & ((1ull << (b - 64)) - 1)) != 0;
}

// A result below the smallest normal number (rare): w * 2^L rounded once, ties to even,
// to a multiple of the format's smallest subnormal 2^emin_sub, returned as that multiple
// (at most 2^P-1: the next normal number's pattern when it rounds up). Callers pass only
// values below the smallest normal, so |w| < 2^(emin_sub - L + P - 1). Out of line, with
// the words passed by value (no address of the caller's accumulators is taken). The sign
// bit of the result's pattern is added by the caller.
template <int P>
__device__ __noinline__ unsigned long long acc_round_subnormal(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3,
                                                               int L, int emin_sub) {
  unsigned long long lo = ((unsigned long long)w1 << 32) | w0;
  unsigned long long hi = ((unsigned long long)w3 << 32) | w2;
  const bool neg = (long long)hi < 0;
  if (neg) {
    lo = ~lo;
    hi = ~hi;
    lo += 1;
    if (lo == 0) hi += 1;
  }
  const int sh = emin_sub - L;  // the grid step in units of w
  if (sh <= 0) return lo << (-sh);  // exact (then |w| < 2^(P-1+sh), so hi = 0)
  if (sh > 128) return 0;           // |w| < 2^128 <= half a step
  unsigned long long q = sh < 128 ? shr128(hi, lo, sh) : 0ull;
  const bool round = bit128(hi, lo, sh - 1);
  if (round && (low128(hi, lo, sh - 1) || (q & 1))) q += 1;
  return q;
}

// The integer w times 2^L rounded to the nearest double, as its bits: the 53-bit significand
// and the exponent are assembled into the double's bit pattern (GB300's FP64 pipe is narrow,
// so no FP64 instruction is spent per element). A result below the normal range is rounded
// once on the subnormal grid (not first to 53 bits); one beyond it is an infinity.
// The significand with its leading one is added to the exponent field less one, so a
// rounding that carries out of it moves the exponent (and 2046 to an infinity) by itself.
// No branch, so that a thread's values overlap: the two rare ranges set `rare` (the value
// returned is then not the result) and are formed by acc_bits_any. A unit's 16 sums per
// thread took 11700 cycles when every sum chose among shift cases by branches (banded 32768
// product), 4400 with only the rare ranges branching.
template <bool F32>
__device__ __forceinline__ unsigned long long acc_bits(const uint32_t (&w)[4], int L, bool& rare) {
  uint32_t t[3];
  const int msb = acc_normalise(w, t);
  const uint32_t sign = w[3] & 0x80000000u;
  const bool nonzero = t[0] != 0u;
  if constexpr (F32) {  // 24-bit significand
    const int biased = msb + L + 127;
    rare |= nonzero && (uint32_t)(biased - 1) > 253u;
    const uint32_t low = (t[0] & 0x7Fu) | t[1] | t[2];
    const uint32_t inc = (t[0] >> 7) & 1u & ((low != 0u ? 1u : 0u) | (t[0] >> 8));
    const uint32_t v = (sign | ((uint32_t)(biased - 1) << 23)) + (t[0] >> 8) + inc;
    return nonzero ? v : 0u;
  } else {
    const int biased = msb + L + 1023;
    rare |= nonzero && (uint32_t)(biased - 1) > 2045u;
    const unsigned long long mant = (((unsigned long long)t[0] << 32) | t[1]) >> 11;
    const uint32_t low = (t[1] & 0x3FFu) | t[2];
    const uint32_t inc = (t[1] >> 10) & 1u & ((low != 0u ? 1u : 0u) | (t[1] >> 11));
    const unsigned long long v =
        ((unsigned long long)(sign | ((uint32_t)(biased - 1) << 20)) << 32) + mant + inc;
    return nonzero ? v : 0ull;
  }
}
template <bool F32>
__device__ __noinline__ unsigned long long acc_bits_any(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, int L) {
  const uint32_t w[4] = {w0, w1, w2, w3};
  bool rare = false;
  const unsigned long long v = acc_bits<F32>(w, L, rare);
  if (!rare) return v;
  uint32_t t[3];
  const int biased = acc_normalise(w, t) + L + (F32 ? 127 : 1023);
  const unsigned long long sign = F32 ? (w3 & 0x80000000u) : (unsigned long long)(w3 & 0x80000000u) << 32;
  if (biased > 0) return sign | (F32 ? 0x7F800000ull : 0x7FF0000000000000ull);
  return sign | (F32 ? acc_round_subnormal<24>(w0, w1, w2, w3, L, -149) : acc_round_subnormal<53>(w0, w1, w2, w3, L, -1074));
}

// w += v, 128-bit two's complement
__device__ __forceinline__ void add128(uint32_t (&w)[4], const uint4& v) {
  asm("add.cc.u32 %0, %0, %4;\n\t"
      "addc.cc.u32 %1, %1, %5;\n\t"
      "addc.cc.u32 %2, %2, %6;\n\t"
      "addc.u32 %3, %3, %7;"
      : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3])
      : "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w));
}

template <int R>
__device__ __forceinline__ void regs_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R));
}
template <int R>
__device__ __forceinline__ void regs_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R));
}

// True when v is true in every thread of the kEpiThreads epilogue threads (named barrier 1
// with an AND reduction; all of them must call it).
__device__ __forceinline__ bool epi_all(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, 1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(kEpiThreads)
      : "memory");
  return r != 0;
}

// Multiplication by alpha or beta. FP64 multiplications run at 2 lanes per clock and SM, 4096 of
// them per unit and factor; by +-2^k (1, -1, 0.5, ...) the product is the value with another
// exponent and sign, so those are formed on the bits, and only zeros aside from a value or
// result outside the normal range take the multiplication. C store of one tile with alpha
// -0.5 and beta 0.5: 12000 cycles as two multiplications and an addition per element.
struct Factor {
  double v;
  int32_t k;       // v = +-2^k when pow2
  uint32_t sign;   // its sign bit
  bool one, pow2;
  __device__ __forceinline__ explicit Factor(double f) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(f);
    const int e = (int)((b >> 52) & 0x7FF);
    v = f;
    k = e - 1023;
    sign = (uint32_t)(b >> 32) & 0x80000000u;
    one = b == 0x3FF0000000000000ull;
    pow2 = (b & 0xFFFFFFFFFFFFFull) == 0 && e > 0 && e < 0x7FF;
  }
  __device__ __forceinline__ double times(double x) const {  // fl(v x)
    if (one) return x;
    if (pow2) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(x);
      const uint32_t hi = (uint32_t)(b >> 32);
      const int e = (int)((hi >> 20) & 0x7FF);
      if ((uint32_t)(e - 1) < 2046u && (uint32_t)(e + k - 1) < 2046u)
        return __hiloint2double((int)((hi + ((uint32_t)k << 20)) ^ sign), (int)(uint32_t)b);
    }
    return __dmul_rn(v, x);
  }
};

// Where one lane's column of a unit goes in C: its tile column, and its element within a
// row of a tile. Looked up before the unit's results are waited for.
struct StoreCol {
  int j;             // tile column (-1: beyond the last column)
  int64_t first;     // element of a tile's row 0 (complex elements: double) the column is
  int64_t row_step;  // elements (complex: doubles) from one row of the tile to the next
  template <int ELEM>
  __device__ __forceinline__ void init(const SplitArgs& P, int64_t n) {
    j = -1;
    first = row_step = 0;
    if (n >= P.Ntot) return;
    j = P.col_tile[n];
    const int64_t lc = n - P.co[j], cj = P.c[j];
    if constexpr (ELEM == 2) {
      // column lc of the doubled tile: the real part of complex column lc, or the
      // imaginary part of column lc - c_j / 2
      const int64_t cc = cj >> 1, part = lc >= cc;
      first = 2 * (lc - part * cc) + part;
      row_step = 2 * cc;
    } else {
      first = lc;
      row_step = cj;
    }
  }
};

// C = alpha*v + beta*C for a 128 x TN region staged in shared memory as bit patterns (row
// stride TN + 1), on the elements that lie in S_C tiles. Warp w of NW stores rows
// w*(128/NW) .. with lane = column (TN == 32), so a store instruction writes one or two
// contiguous row segments. The rows are taken tile by tile: per tile one offset per lane
// (the next tile's is loaded while this one's rows are stored), then rows a constant step
// apart, with alpha and beta tested once per region, as bits: per row the loop holds a
// shared load, a store and an address addition. A unit takes the four store warps 4300
// cycles (banded 32768 product); testing alpha and beta per row as doubles (the FP64 pipe
// takes 2 lanes per clock) and looking every row's tile up took 31000, half of the unit's
// time. With the branch-free rounding above the contraction went from 6.00 to 4.32 ms
// (2048 uniform product: 169 to 77 us).
template <int TN, int NW, int ELEM>  // ELEM: 0 float64, 1 float32, 2 complex (one part per column)
__device__ __forceinline__ void store_region(const SplitArgs& P, const unsigned long long* cstage, int rb,
                                             const StoreCol& col, int w, int lane, int32_t* err) {
  static_assert(TN == 32, "one column per lane");
  using E = std::conditional_t<ELEM == 1, float, double>;
  constexpr int kRowsPerWarp = kSplitBM / NW;
  constexpr int kBatch = 8;  // rows whose loads are in flight together
  const E alpha = (E)P.alpha, beta = (E)P.beta;  // float32 elements: exact (given as floats)
  const Factor fa(P.alpha), fb(P.beta);
  const bool scale = !fa.one;
  const bool accum = (__double_as_longlong(P.beta) & 0x7FFFFFFFFFFFFFFFll) != 0;
  E* const C = reinterpret_cast<E*>(ELEM == 1 ? (void*)P.Cf : (void*)P.C);
  const int64_t* const ro = P.ro;
  const int64_t* const c_off = P.c_off;
  const uint8_t* const cs = P.cs;
  const int N = P.N;
  const int64_t m_end = min((int64_t)rb * kSplitBM + (w + 1) * kRowsPerWarp, P.Mtot);
  int64_t m = (int64_t)rb * kSplitBM + w * kRowsPerWarp;
  if (m >= m_end) return;
  const unsigned long long* src = cstage + w * kRowsPerWarp * (TN + 1) + lane;
  int i = P.row_tile[m];
  // the offset of tile (i, col.j): -2 when it is not in S_C (nothing to store)
  auto offset = [&](int i_) -> int64_t {
    if (col.j < 0) return -2;
    const int64_t tile = (int64_t)i_ * N + col.j;
    return cs[tile] ? c_off[tile] : -2;
  };
  int64_t off = offset(i), lr = m - ro[i], next = ro[i + 1];
  for (;;) {
    // the next tile with rows (zero-height tiles hold none), looked up ahead
    const int64_t seg = min(next, m_end);
    int i2 = i;
    int64_t off2 = -2, next2 = next;
    if (next < m_end) {
      do {
        i2++;
        next2 = ro[i2 + 1];
      } while (next2 == next);
      off2 = offset(i2);
    }
    if (off == -1) atomicOr(err, kErrBadOffset);
    const int rows = (int)(seg - m);
    if (off >= 0) {
      E* dst = C + (ELEM == 2 ? 2 * off : off) + lr * col.row_step + col.first;
      const int64_t step = col.row_step;
      auto bits = [](unsigned long long v) -> E {
        if constexpr (ELEM == 1)
          return __uint_as_float((uint32_t)v);
        else
          return __longlong_as_double((long long)v);
      };
      if (!scale && !accum) {
#pragma unroll 1
        for (int r = 0; r < rows; r += kBatch) {
          unsigned long long v[kBatch];
#pragma unroll
          for (int u = 0; u < kBatch; u++) v[u] = r + u < rows ? src[(r + u) * (TN + 1)] : 0ull;
#pragma unroll
          for (int u = 0; u < kBatch; u++) {
            if (r + u < rows) *dst = bits(v[u]);
            dst += step;
          }
        }
      } else {
#pragma unroll 1
        for (int r = 0; r < rows; r += kBatch) {
          E v[kBatch], old[kBatch];
#pragma unroll
          for (int u = 0; u < kBatch; u++) {
            v[u] = bits(r + u < rows ? src[(r + u) * (TN + 1)] : 0ull);
            old[u] = accum && r + u < rows ? dst[u * step] : E(0);
          }
#pragma unroll
          for (int u = 0; u < kBatch; u++) {
            if constexpr (ELEM == 1) {
              if (scale) v[u] = __fmul_rn(alpha, v[u]);
              if (accum) v[u] = __fadd_rn(v[u], __fmul_rn(beta, old[u]));
            } else {
              v[u] = fa.times(v[u]);
              if (accum) v[u] = __dadd_rn(v[u], fb.times(old[u]));
            }
            if (r + u < rows) *dst = v[u];
            dst += step;
          }
        }
      }
    }
    src += rows * (TN + 1);
    m = seg;
    if (m >= m_end) break;
    i = i2;
    off = off2;
    next = next2;
    lr = 0;
  }
}

// store_region for the product's element type, the column looked up here or before
__device__ __forceinline__ void store_col(const SplitArgs& P, int cb, int lane, StoreCol& col) {
  const int64_t n = (int64_t)cb * 32 + lane;
  if (P.cplx)
    col.init<2>(P, n);
  else
    col.init<0>(P, n);
}
template <int TN, int NW>
__device__ __forceinline__ void store_unit(const SplitArgs& P, const unsigned long long* cstage, int rb,
                                           const StoreCol& col, int w, int lane, int32_t* err) {
  if (P.f32)
    store_region<TN, NW, 1>(P, cstage, rb, col, w, lane, err);
  else if (P.cplx)
    store_region<TN, NW, 2>(P, cstage, rb, col, w, lane, err);
  else
    store_region<TN, NW, 0>(P, cstage, rb, col, w, lane, err);
}

// The TH columns' largest exponents, with a few 16-byte loads (n0 is a multiple of TH).
template <int TH>
__device__ __forceinline__ void load_emaxc(const SplitArgs& P, int64_t n0, int (&emc)[TH]) {
#pragma unroll
  for (int w = 0; w < TH / 4; w++) {
    const int4 v = __ldg(reinterpret_cast<const int4*>(P.emaxc + n0) + w);
    emc[4 * w] = v.x;
    emc[4 * w + 1] = v.y;
    emc[4 * w + 2] = v.z;
    emc[4 * w + 3] = v.w;
  }
}

// One thread's row of a unit's sums rounded into the staging buffer: the doubles' or (for
// float32 elements) floats' bit patterns. Elements outside the product are not stored, so
// what is staged for them does not matter (their sums are zero).
template <int TH, bool F32>
__device__ __forceinline__ void round_row(const uint32_t (&acc)[TH][4], unsigned long long* srow,
                                          const int (&emc)[TH], int Lrow) {
  bool rare = false;
#pragma unroll
  for (int c = 0; c < TH; c++) srow[c] = acc_bits<F32>(acc[c], Lrow + emc[c], rare);
  if (rare) {
#pragma unroll
    for (int c = 0; c < TH; c++)
      srow[c] = acc_bits_any<F32>(acc[c][0], acc[c][1], acc[c][2], acc[c][3], Lrow + emc[c]);
  }
}


// ---------------------------------------------------------------- kernel 3: contraction
// Ascending k blocks of one unit (a 128-row block times a group of cl column blocks):
// presA[rb] & presBg[group], within the unit's inner-block range [k0, k1) (all of it, or
// one piece under split k). Each CTA of the group takes from it, with next_own(), the k
// blocks where its own column block has a B tile.
struct UnitIter {
  const uint64_t* pa;
  const uint64_t* pb;
  const uint64_t* po;  // this CTA's own column block (null: beyond the last one)
  int kwords, wd, kend;
  uint64_t bits;
  __device__ void init(const SplitArgs& a, const SplitUnit& un, int cb) {
    pa = a.presA + (size_t)un.rb * a.kwords;
    pb = a.presBg + (size_t)un.cb * a.kwords;
    po = cb < a.CB ? a.presB + (size_t)cb * a.kwords : nullptr;
    kwords = a.kwords;
    kend = un.k1;
    wd = un.k0 >> 6;
    bits = wd < kwords ? (pa[wd] & pb[wd]) & (~0ull << (un.k0 & 63)) : 0ull;
  }
  __device__ bool own_b(int k) const { return po && ((po[k >> 6] >> (k & 63)) & 1); }
  __device__ int next_own() {  // next k block that also has a B tile in this CTA's column block
    for (int k = next(); k >= 0; k = next())
      if (own_b(k)) return k;
    return -1;
  }
  __device__ int next() {  // -1 when done
    while (!bits) {
      if (++wd >= kwords) return -1;
      bits = pa[wd] & pb[wd];
    }
    const int k = wd * 64 + __ffsll((long long)bits) - 1;
    if (k >= kend) {  // past the unit's range
      bits = 0;
      wd = kwords;
      return -1;
    }
    bits &= bits - 1;
    return k;
  }
};

// Accumulation groups: consecutive k blocks of a CTA's own list (those where its column
// block has a B tile) share one TMEM accumulation when each has a uniform scale class
// for the unit, the classes add up to the same binary position, and the total inner depth
// keeps every FP32 partial sum exact. The MMA warps and the epilogue apply the same rule
// to the same list, so they agree on where the accumulator is drained.
// The scale class of k block k for the unit's row block rb and column block cb: true
// and the binary offset sig of its products when both classes are uniform.
// A class more than kSplitGuard binades below the unit's largest scale is not uniform
// either: its products enter the accumulator rounded down (floor) to its unit, and the
// floor of a sum is not the sum of the floors, so such k blocks are drained one by one,
// each product taking its own floor as the exact sum's definition states.
__device__ __forceinline__ bool scale_class(const SplitArgs& P, int k, int rb, int cb, int& sig) {
  if (!P.urow) return false;
  const int u = P.urow[(size_t)k * P.RB + rb], v = P.ucol[(size_t)k * P.CB + cb];
  if (u == kNonUniform || v == kNonUniform || u + v < -kSplitGuard) return false;
  sig = u + v;
  return true;
}

struct GroupRule {
  bool uni;
  int sig, depth, kdepth;
  __device__ void start(bool uni_, int sig_, int q, int kdepth_) {
    uni = uni_;
    sig = sig_;
    depth = q;
    kdepth = kdepth_;
  }
  __device__ bool joins(bool uni_, int sig_, int q) {  // true: the k block joins (its depth is added)
    if (!uni || !uni_ || sig_ != sig || depth + q > kdepth) return false;
    depth += q;
    return true;
  }
};

// A group is complete: its descriptor goes to the epilogue (from the first MMA warp),
// then every MMA warp's commit marks the buffer full once its MMAs have finished.
__device__ __forceinline__ void close_group(bool first, int4* gdesc, uint64_t* gready, uint64_t* tfull, uint32_t buf,
                                            int gk0, const GroupRule& grp, bool last) {
  if (elect_one()) {
    if (first) {
      gdesc[buf] = make_int4(gk0, grp.sig, (grp.uni ? 1 : 0) | (last ? 2 : 0), 0);
      mbar_arrive(&gready[buf]);
    }
    umma_commit(&tfull[buf]);
  }
  __syncwarp();
}

// The values of one own k block of a unit's list that the MMA warps need, loaded ahead.
struct KAhead {
  int k, q;
  bool uni;
  int sig;
  __device__ void load(const SplitArgs& P, int k_, int rb, int cb) {  // k_: an own k block, or -1
    k = k_;
    q = 0;
    uni = false;
    sig = 0;
    if (k < 0) return;
    q = P.q[k];
    uni = scale_class(P, k, rb, cb, sig);
  }
};

// The chunks of one CTA's unit list in order: unit by unit, k block by k block
// (ascending; only the k blocks where the CTA's own column block has a B tile), 32-deep
// chunk by chunk.
struct ChunkCursor {
  const SplitArgs* P;  // the product of the current unit (the batch-wide args for one product)
  int idx, uend;
  int rb, cb;  // this CTA's row block and column block
  UnitIter it;
  int kt, kc, nkc;
  bool in_unit;
  const uint8_t* asrc;
  const uint8_t* bsrc;
  __device__ void start(int beg, int end) {
    idx = beg - 1;
    uend = end;
    in_unit = false;
    kc = 0;
    nkc = 0;
  }
  __device__ bool advance(const SplitArgs& a, int cl, int rank) {  // false when exhausted
    if (++kc < nkc) return true;
    for (;;) {
      if (in_unit) {
        kt = it.next_own();
        if (kt >= 0) {
          nkc = (P->q[kt] + kSplitKC - 1) / kSplitKC;  // >= 1: blocks with q = 0 are never present
          kc = 0;
          asrc = P->apk + P->apk_off[(size_t)rb * P->K + kt];
          bsrc = P->bpk + P->bpk_off[(size_t)kt * P->CB + cb];
          return true;
        }
        in_unit = false;
      }
      if (++idx >= uend) return false;
      int g = a.sched_units[idx];
      P = a.prods ? &a.prods[a.unit_prod[g]] : &a;
      if (a.prods) g = a.unit_local[g];
      const SplitUnit un = P->units[g];
      rb = un.rb;
      cb = un.cb * cl + rank;
      it.init(*P, un, cb);
      in_unit = true;
    }
  }
};

}  // namespace

}  // namespace bsmm
