// The 64-column form of the contraction kernel (split.cu), for products of long k lists.
//
// A CTA takes two neighbouring 32-column blocks of its unit at once: the stacked slices of B
// are then 64 rows each, so slice p of A meets slices 1..S+1-p of B in MMAs of up to 256
// columns. Against the 32-column form a slice product costs half the A bytes (copied from L2
// into the ring and read by the tensor core) and half the MMA instructions:
//   cycles per 32-deep chunk and 32 columns, MMAs fed by a ring of copies and nothing else:
//     6 slices: 852 with 32 columns, 698 with 64 (672 at the tensor cores' rate);
//     4 slices: 580 and 345 (320).
// The 32-column form does not reach its own 852 on large products (1090): its three 60 KB
// stages hold less time than an access to DRAM takes. Three 72 KB stages here hold twice
// that time.
// The price: two accumulator buffers of S x 64 columns fit TMEM only up to 4 slices. With 5
// and 6 there is one, and the tensor core waits while a group is drained (3200 cycles of a
// 26000-cycle group of the dense product, 6000 at binary positions), so the form suits
// products whose groups are long. With those slice counts the 32-column form is launched
// behind this one, and one of the two has nothing to do (3 us), chosen from the scale classes
// by the slicing (slice.cu; the limit is plan.cpp's). This kernel finds its lists empty then: a
// test and a return at its top cost it 0.5% (dense 4096: 1948 against 1938 us).
// And the 128-bit sums of 64 columns take 128 registers of each of the 8 epilogue warps, which
// leaves no room for store warps: the epilogue stores a unit itself while the next unit's
// first group runs.
// Contraction, 32-column form against this one: dense 16384, 6 slices, 133.1 to 112.3 ms
// (1645 TFLOP/s of slice products, 0.98 of what cuBLAS sustains in BF16); float32 8192, 4
// slices, 11.68 to 7.64 ms; thin 512 x 524288 4.29 to 3.45 ms. The rule that takes it is the
// planner's (plan.cpp).
//
// Roles: warp 0 producer, warps 1 and 2 MMA issue, warp 3 idle, warps 4 to 11 epilogue. The
// unit list, the k lists, the accumulation groups and the exact sums are those of the
// 32-column form with groups of 2 or 4 CTAs: a plan's units are the same for both (a batch
// runs them with the 32-column form), and so are the result bits.
#include <cstdint>
#include <type_traits>

#include "split_device.cuh"

namespace bsmm {

namespace {

constexpr int kWideN = 64;        // columns per CTA
constexpr int kWideMmaWarps = 2;  // 6 slices, issue alone: 1594 cycles per chunk with one, 1395 with two
constexpr int kWideEpiWarp0 = 4;
constexpr int kWideThreads = 32 * (kWideEpiWarp0 + kSplitEpiWarps);  // 384
constexpr int kWideRegsLaunch = 168;                                // 384 x 168 registers
constexpr int kWideRegsCtl = 72, kWideRegsEpi = 216;
static_assert(4 * 32 * kWideRegsCtl + kSplitEpiWarps * 32 * kWideRegsEpi <= kWideThreads * kWideRegsLaunch,
              "the warpgroups' register shares must fit the launch's registers");

// The MMAs of one 16-deep step: slice p of A against slices 1..S+1-p of B, at most 256 columns each
template <int S>
struct WideList {
  int n = 0;
  int N[2 * S] = {}, dcol[2 * S] = {}, aslice[2 * S] = {}, brow[2 * S] = {};
  constexpr WideList() {
    for (int p = 1; p <= S; p++)
      for (int c = 0, tot = (S + 1 - p) * kWideN; c < tot; c += 256) {
        N[n] = tot - c < 256 ? tot - c : 256;
        dcol[n] = (p - 1) * kWideN + c;
        aslice[n] = p - 1;
        brow[n] = c;
        n++;
      }
  }
};

// The scale class of k block k for the unit's row block and the CTA's two column blocks: one
// binary position when the row class and both column classes are uniform and the latter equal.
__device__ __forceinline__ bool wide_class(const SplitArgs& P, int k, int rb, int cb, int cb1, int& sig) {
  int s1 = 0;
  return scale_class(P, k, rb, cb, sig) && scale_class(P, k, rb, cb1, s1) && s1 == sig;
}

// A warp's 32 rows x TH columns of sums rounded and stored: C = alpha*fl(sum) + beta*C on the
// elements that lie in S_C tiles. The sums (a row per lane) are in units of
// 2^(Lrow + Lcol), Lcol of column n0 + c in lane c. Four columns at a time go
// through a 1 KB slab of the warp's own (XOR-swizzled, so neither side has bank conflicts),
// from which a store instruction takes 8 rows of 32 contiguous bytes: 8-byte stores of 32
// rows each took 83000 cycles per unit. Each lane keeps the addresses of its 4 rows in the
// tile its column lies in, and looks them up again when its column enters another tile.
constexpr int kSlabBytes = 32 * 4 * 8;
template <int TH, int ELEM>  // ELEM: 0 float64, 1 float32, 2 complex (one part per column)
__device__ __forceinline__ void wide_store(const SplitArgs& P, uint32_t (&acc)[TH][4], unsigned long long* slab,
                                           int64_t m0, int lane, int64_t n0, int Lrow, int Lcol) {
  using E = std::conditional_t<ELEM == 1, float, double>;
  if (m0 >= P.Mtot || n0 >= P.Ntot) return;
  const E alpha = (E)P.alpha, beta = (E)P.beta;
  const Factor fa(P.alpha), fb(P.beta);
  const bool scale = !fa.one;
  const bool accum = (__double_as_longlong(P.beta) & 0x7FFFFFFFFFFFFFFFll) != 0;
  E* const C = reinterpret_cast<E*>(ELEM == 1 ? (void*)P.Cf : (void*)P.C);
  int it[4], lrow[4];  // the lane's rows m0 + 8 r + lane / 4: row tile (-1: none) and row in it
#pragma unroll
  for (int r = 0; r < 4; r++) {
    const int64_t m = m0 + 8 * r + (lane >> 2);
    it[r] = m < P.Mtot ? P.row_tile[m] : -1;
    lrow[r] = it[r] >= 0 ? (int)(m - P.ro[it[r]]) : 0;
  }
  int64_t n = n0 + (lane & 3);  // the lane's column of this round
  int j = n < P.Ntot ? P.col_tile[n] : 0;
  int64_t next = n < P.Ntot ? P.co[j + 1] : 0;  // (a column past the last one never enters a tile)
  bool look = true;
  E* dst[4] = {nullptr, nullptr, nullptr, nullptr};
  int64_t flip = 0;  // complex: the column at which the tile's imaginary parts begin
  // (A loop, the sums moving down four columns per round: unrolled, this code runs once per
  // unit out of a cold instruction cache, 49000 cycles per unit against 40000.)
#pragma unroll 1
  for (int c0 = 0; c0 < TH; c0 += 4) {
    const bool in = n < P.Ntot;
    if (in && n >= next) {
      do {
        j++;
        next = P.co[j + 1];
      } while (n >= next);
      look = true;
    }
    if (ELEM == 2 && in && !look && n >= flip && n - 4 < flip) look = true;
    if (in && look) {
      look = false;
      const int64_t lc = n - P.co[j], cj = P.c[j];
      const int64_t cc = cj >> 1, part = ELEM == 2 && lc >= cc;
      flip = P.co[j] + cc;
#pragma unroll
      for (int r = 0; r < 4; r++) {
        const int64_t tile = (int64_t)it[r] * P.N + j;
        const int64_t off = it[r] >= 0 && P.cs[tile] ? P.c_off[tile] : -2;
        if (off == -1) atomicOr(P.err, kErrBadOffset);
        if constexpr (ELEM == 2)
          dst[r] = off < 0 ? nullptr : C + 2 * (off + lrow[r] * cc + lc - part * cc) + part;
        else
          dst[r] = off < 0 ? nullptr : C + off + lrow[r] * cj + lc;
      }
    }
    E old[4];
#pragma unroll
    for (int r = 0; r < 4; r++) old[r] = accum && in && dst[r] ? *dst[r] : E(0);
    // round the lane's own row's four columns into the slab
    unsigned long long bits[4];
    int L[4];
    bool rare = false;
#pragma unroll
    for (int u = 0; u < 4; u++) {
      L[u] = Lrow + __shfl_sync(0xffffffffu, Lcol, c0 + u);
      bits[u] = acc_bits<ELEM == 1>(acc[u], L[u], rare);
    }
    if (rare) {
#pragma unroll
      for (int u = 0; u < 4; u++) bits[u] = acc_bits_any<ELEM == 1>(acc[u][0], acc[u][1], acc[u][2], acc[u][3], L[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; u++) slab[lane * 4 + (u ^ ((lane >> 2) & 3))] = bits[u];
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 4; r++) {
      const int row = 8 * r + (lane >> 2);
      const unsigned long long x = slab[row * 4 + ((lane & 3) ^ ((row >> 2) & 3))];
      E v;
      if constexpr (ELEM == 1) {
        v = __uint_as_float((uint32_t)x);
        if (scale) v = __fmul_rn(alpha, v);
        if (accum) v = __fadd_rn(v, __fmul_rn(beta, old[r]));
      } else {
        v = __longlong_as_double((long long)x);
        v = fa.times(v);
        if (accum) v = __dadd_rn(v, fb.times(old[r]));
      }
      if (in && dst[r]) {
        *dst[r] = v;
        dst[r] += ELEM == 2 ? 8 : 4;
      }
    }
    __syncwarp();
    n += 4;
#pragma unroll
    for (int c = 0; c + 4 < TH; c++)
#pragma unroll
      for (int w = 0; w < 4; w++) acc[c][w] = acc[c + 4][w];
  }
}

// acc += one group's exact integers: the S diagonals of this thread's TH columns, read in
// batches of 4 columns and zeroed behind. PLAIN: in the group's own unit; otherwise at the
// binary positions shr + cx[column].
template <int S, int TH, bool PLAIN>
__device__ __forceinline__ void wide_drain(uint32_t taddr, uint32_t (&acc)[TH][4], int shr, const uint4 (&cx)[TH / 8]) {
  constexpr int CW = 4;
#pragma unroll
  for (int cc = 0; cc < TH / CW; cc++) {
    uint32_t v[S][CW];
#pragma unroll
    for (int d = 0; d < S; d++) tmem_ld4(taddr + d * kWideN + cc * CW, v[d]);
    tmem_ld_wait();
#pragma unroll
    for (int d = 0; d < S; d++) tmem_zero4(taddr + d * kWideN + cc * CW);
#pragma unroll
    for (int c = 0; c < CW; c++) {
      const long long T = diagonal_sum<S, CW, true>(v, c);
      const int col = cc * CW + c;
      if constexpr (PLAIN) {
        acc_add_plain(acc[col], T);
      } else {
        const uint4& w4 = cx[col >> 3];
        const int e = col & 7;
        const uint32_t wd = e < 2 ? w4.x : e < 4 ? w4.y : e < 6 ? w4.z : w4.w;
        acc_add(acc[col], T, shr + (int)(int16_t)(wd >> (16 * (e & 1))));
      }
    }
  }
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

template <int S>
__global__ void __launch_bounds__(kWideThreads, 1) split_mma_wide_kernel(const __grid_constant__ SplitArgs a) {
  constexpr int TH = kWideN / 2;                 // columns per epilogue thread: one column block
  constexpr int A_STAGE = S * kAChunk;
  constexpr int B_HALF = 32 * kSplitKC * 2;      // one slice of a 32-column block's chunk
  constexpr int B_STAGE = S * 2 * B_HALF;
  constexpr bool PAIRS = S <= kWidePairsMaxS;    // column blocks packed in pairs
  constexpr int STAGE = A_STAGE + B_STAGE;
  constexpr int BUF_COLS = S * kWideN;
  constexpr int NB = 2 * BUF_COLS <= (int)kTmemCols ? 2 : 1;  // accumulator buffers
  constexpr int W = kWideMmaWarps;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int stages = a.wstages;
  uint64_t* full = (uint64_t*)(smem + (size_t)stages * STAGE);
  uint64_t* empty = full + stages;
  uint64_t* tfull = empty + stages;
  uint64_t* tempty = tfull + NB;
  uint64_t* drain = tempty + NB;  // one per MMA warp
  uint32_t* tmem_slot = (uint32_t*)(drain + W);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  // per epilogue warp, for the C store
  unsigned long long* const slabs = (unsigned long long*)(smem + (size_t)stages * STAGE + kSplitBarBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int CL = a.cl, WCL = CL >> 1;  // column blocks and CTAs of a group
  const int cta = blockIdx.x / WCL;    // the group: schedules are per group
  const int rank = blockIdx.x % WCL;
  grid_wait();  // before anything of global memory is read, the schedule included
  const int ubeg = a.sched_ptr[cta], uend = a.sched_ptr[cta + 1];

  if (threadIdx.x == 0) {
    for (int st = 0; st < stages; st++) {
      mbar_init(&full[st], 1);
      mbar_init(&empty[st], W);
    }
    for (int b = 0; b < NB; b++) {
      mbar_init(&tfull[b], W);
      mbar_init(&tempty[b], kSplitEpiWarps);
    }
    for (int w = 0; w < W; w++) mbar_init(&drain[w], 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp < kWideEpiWarp0) {
    regs_dec<kWideRegsCtl>();
    if (warp == 0) {
      // ---------------------------------------------------------- producer
      // The whole warp walks the list. With 3 and 4 slices a pair of column blocks is packed as
      // it is read here, 64 rows per slice, and a chunk is two copies. From the 32-column
      // packing it is 2S + 1, about 100 cycles each to issue: with 4 slices the tensor core
      // waited for them a quarter of the time (float32 8192: 9.66 ms, 7.64 with two). With 5
      // and 6 slices it does not: the dense 16384 product took 111.2 ms with 13 copies and
      // 111.7 with two.
      int stage = 0;
      uint32_t phase = 0;
      uint32_t issued = 0, issued_par = 0;  // bit st: stage st holds an issued copy; its parity
      bool ok = true;
      for (int idx = ubeg; idx < uend && ok; idx++) {
        const SplitUnit un = a.units[a.sched_units[idx]];
        const int cb = un.cb * CL + 2 * rank;
        [[maybe_unused]] const int cb1 = cb + 1 < a.CB ? cb + 1 : cb;  // a last, single block stands in for both
        UnitIter it;
        it.init(a, un, cb);
        for (int kt = it.next_own(); kt >= 0 && ok; kt = it.next_own()) {
          const int nkc = (a.q[kt] + kSplitKC - 1) / kSplitKC;
          const uint8_t* asrc = a.apk + a.apk_off[(size_t)un.rb * a.K + kt];
          const uint8_t* bsrc;
          if constexpr (PAIRS)
            bsrc = a.bpk + a.bpk_off[(size_t)kt * a.CB + cb];
          else
            bsrc = a.bpk + a.bpk_off[(size_t)kt * a.CB + (lane & 1 ? cb1 : cb)] + (lane >> 1) * B_HALF;
          for (int kc = 0; kc < nkc; kc++) {
            if (!wait_warp(&empty[stage], phase ^ 1, abort_flag, a.err)) {
              ok = false;
              break;
            }
            uint8_t* sa = smem + (size_t)stage * STAGE;
            if constexpr (PAIRS) {
              if (elect_one()) {
                mbar_arrive_expect_tx(&full[stage], STAGE);
                bulk_g2s(sa, asrc + (size_t)kc * A_STAGE, A_STAGE, &full[stage]);
                bulk_g2s(sa + A_STAGE, bsrc + (size_t)kc * B_STAGE, B_STAGE, &full[stage]);
              }
            } else {  // lane l: slice l / 2 of block l % 2
              if (lane == 0) mbar_arrive_expect_tx(&full[stage], STAGE);
              __syncwarp();
              if (lane == 0) bulk_g2s(sa, asrc + (size_t)kc * A_STAGE, A_STAGE, &full[stage]);
              if (lane < 2 * S)
                bulk_g2s(sa + A_STAGE + lane * B_HALF, bsrc + (size_t)kc * (S * B_HALF), B_HALF, &full[stage]);
            }
            __syncwarp();
            issued |= 1u << stage;
            issued_par = (issued_par & ~(1u << stage)) | (phase << stage);
            if (++stage == stages) {
              stage = 0;
              phase ^= 1;
            }
          }
        }
      }
      // every copy issued has landed before the CTA may exit
      for (int st = 0; st < stages; st++) {
        if (!(issued >> st & 1)) continue;
        const int64_t t0 = gtimer();
        while (!mbar_try_wait(&full[st], issued_par >> st & 1)) {
          if (gtimer() - t0 > kWaitNs) {
            if (lane == 0) atomicOr(a.err, kErrTimeout);
            break;
          }
        }
      }
    } else if (warp <= W) {
      // ---------------------------------------------------------- MMA issue
      // As in the 32-column form: both warps walk the same chunks, each issues its share of
      // a step's MMAs, and every MMA accumulates into buffers the epilogue zeroes.
      const int mw = warp - 1;
      int stage = 0;
      uint32_t phase = 0;
      uint32_t tcount = 0;
      bool ok = true, any = false;
      const uint64_t adesc0 = sdesc_sw64(smem_u32(smem));
      const uint64_t bdesc0 = sdesc_sw64(smem_u32(smem) + A_STAGE);
      const uint32_t idesc0 = idesc_f16(kSplitBM, 0, a.fp16 != 0);
      for (int idx = ubeg; idx < uend && ok; idx++) {
        const SplitUnit un = a.units[a.sched_units[idx]];
        const int cb = un.cb * CL + 2 * rank;
        const int cb1 = cb + 1 < a.CB ? cb + 1 : cb;
        UnitIter it;
        it.init(a, un, cb);
        GroupRule grp;
        bool in_group = false;
        uint32_t buf = 0;
        auto load = [&](int k, int& q, bool& uni, int& sig) {
          q = 0;
          uni = false;
          sig = 0;
          if (k < 0) return;
          q = a.q[k];
          uni = wide_class(a, k, un.rb, cb, cb1, sig);
        };
        int kt = it.next_own(), q, sig;
        bool uni;
        load(kt, q, uni, sig);
        while (kt >= 0 && ok) {
          const int kn = it.next_own();
          int qn, sign;
          bool unin;
          load(kn, qn, unin, sign);  // one k block ahead
          const int nkc = (q + kSplitKC - 1) / kSplitKC;
          if (!(in_group && grp.joins(uni, sig, q))) {
            if (in_group) {
              if (elect_one()) umma_commit(&tfull[buf]);
              __syncwarp();
              tcount++;
            }
            buf = tcount % NB;
            if (!wait_warp(&tempty[buf], (tcount / NB) & 1, abort_flag, a.err)) {
              ok = false;
              in_group = false;
              break;
            }
            tc_fence_after();
            grp.start(uni, sig, q, a.kdepth);
            in_group = true;
          }
          const uint32_t dbase = tmem_base + buf * BUF_COLS;
          for (int kc = 0; kc < nkc; kc++) {
            if (!wait_warp(&full[stage], phase, abort_flag, a.err)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (elect_one()) {
              const uint64_t soff = (uint64_t)((stage * STAGE) >> 4);
              const uint64_t ad = adesc0 + soff, bd = bdesc0 + soff;
              const bool two = q - kc * kSplitKC > 16;  // second 16-deep step of the chunk
              constexpr WideList<S> L{};
#pragma unroll
              for (int h = 0; h < 2; h++) {
                if (h == 1 && !two) break;
#pragma unroll
                for (int m = 0; m < L.n; m++)
                  if (m % W == mw)
                    umma_f16(dbase + L.dcol[m], ad + (uint64_t)((L.aslice[m] * kAChunk) >> 4) + 2 * h,
                             bd + (uint64_t)((L.brow[m] * 64) >> 4) + 2 * h, idesc0 | ((uint32_t)(L.N[m] >> 3) << 17), 1u);
              }
              umma_commit(&empty[stage]);
            }
            __syncwarp();
            any = true;
            if (++stage == stages) {
              stage = 0;
              phase ^= 1;
            }
          }
          kt = kn;
          q = qn;
          uni = unin;
          sig = sign;
        }
        if (in_group && ok) {
          if (elect_one()) umma_commit(&tfull[buf]);
          __syncwarp();
          tcount++;
        }
      }
      // every MMA this warp issued has completed before TMEM is released
      if (any) {
        if (elect_one()) umma_commit(&drain[mw]);
        __syncwarp();
        const int64_t t0 = gtimer();
        while (!mbar_try_wait(&drain[mw], 0)) {
          if (gtimer() - t0 > kWaitNs) {
            if (lane == 0) atomicOr(a.err, kErrTimeout);
            break;
          }
        }
      }
    }
  } else {
    regs_inc<kWideRegsEpi>();
    // ------------------------------------------------------------ epilogue
    const int ew = warp - kWideEpiWarp0;
    const int quad = warp & 3, half = ew >> 2;
    const int row = quad * 32 + lane;
    unsigned long long* const slab = slabs + ew * (kSlabBytes / 8);
    const uint32_t tq = tmem_base + ((uint32_t)(quad * 32) << 16) + half * TH;
#pragma unroll 1
    for (int b = 0; b < NB; b++)
#pragma unroll
      for (int d = 0; d < S; d++)
#pragma unroll
        for (int cc = 0; cc < TH / 8; cc++) tmem_zero8(tq + b * BUF_COLS + d * kWideN + cc * 8);
    tmem_st_wait();
    tc_fence_before();
    __syncwarp();
    if (lane == 0)
      for (int b = 0; b < NB; b++) mbar_arrive(&tempty[b]);
    uint32_t tcount = 0;
    bool ok = true;
    for (int idx = ubeg; idx < uend && ok; idx++) {
      const int u = a.sched_units[idx];
      const SplitUnit un = a.units[u];
      const int cb = un.cb * CL + 2 * rank;
      if (cb >= a.CB) continue;  // past the last column block: no work
      const int cb1 = cb + 1 < a.CB ? cb + 1 : cb;
      const int64_t t_unit = a.timings && ew == 0 && lane == 0 ? gtimer() : 0;
      if (a.timings && rank == 0 && ew == 0 && lane == 0) a.timings[2 * (int64_t)u] = t_unit;
      const int64_t m = (int64_t)un.rb * kSplitBM + row;
      const bool row_ok = m < a.Mtot;
      const int64_t n0 = (int64_t)(cb + half) * TH;  // this thread's column block
      // (a second block past the last one: its columns are loaded from the padded tables'
      // last rows and never stored)
      const int64_t n0t = cb + half < a.CB ? n0 : (int64_t)cb * TH;
      uint32_t acc[TH][4];
#pragma unroll
      for (int c = 0; c < TH; c++) acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = 0u;
      UnitIter it;
      it.init(a, un, cb);
      int kt = it.next_own();
      // While every group so far is of one uniform class, the sums are kept in the class's own
      // unit and a group's integers are added as they are; the binary position is applied once,
      // at the unit's end (or when another class comes). On data of one scale that is every
      // group, and the drain, which the tensor core waits for with 5 and 6 slices, is two
      // thirds of the instructions.
      const int k_first = kt;
      bool plain = false;
      int sig0 = 0;
      int em = 0, ca = 0;  // lane = column: its largest exponent and its part of a class's position
      while (kt >= 0) {
        const uint32_t buf = tcount % NB;
        // the group, by the MMA warps' rule, ahead of them
        GroupRule grp;
        int gsig = 0;
        {
          const bool uni = wide_class(a, kt, un.rb, cb, cb1, gsig);
          grp.start(uni, gsig, a.q[kt], a.kdepth);
        }
        const int gk0 = kt;
        int kn = it.next_own();
        for (; kn >= 0; kn = it.next_own()) {
          int sg = 0;
          const bool uni = wide_class(a, kn, un.rb, cb, cb1, sg);
          if (!grp.joins(uni, sg, a.q[kn])) break;
        }
        kt = kn;
        if (kt < 0) {
          // the unit's last group: what the unit's end looks up (tables that the operand
          // streams have pushed out of L2) is asked for while the tensor core is at work
          em = a.emaxc[n0t + lane];
          ca = a.coladj[n0t + lane];
          const int64_t nl = n0t + lane;
          if (un.slot < 0 && m - lane < a.Mtot && nl < a.Ntot) {
            const int64_t ml = m - lane + 31 < a.Mtot ? m - lane + 31 : a.Mtot - 1;
            const int i0 = a.row_tile[m - lane], i1 = a.row_tile[ml], jl = a.col_tile[nl];
            prefetch_l2(a.ro + i0);
            prefetch_l2(a.co + jl);
            prefetch_l2(a.c + jl);
            prefetch_l2(a.cs + (int64_t)i0 * a.N + jl);
            prefetch_l2(a.cs + (int64_t)i1 * a.N + jl);
            prefetch_l2(a.c_off + (int64_t)i0 * a.N + jl);
            prefetch_l2(a.c_off + (int64_t)i1 * a.N + jl);
            prefetch_l2(a.emaxr + (row_ok ? m : 0));
          }
        }
        const bool first = gk0 == k_first;
        if (first) {
          plain = grp.uni;
          sig0 = gsig;
        } else if (plain && !(grp.uni && gsig == sig0)) {
          // from here on at binary positions: what there is moves to them
          plain = false;
          const int sh = kSplitGuard + sig0 + (row_ok ? (int)a.rowadj[m] : 0);
#pragma unroll
          for (int w = 0; w < TH / 8; w++) {
            const uint4 ca = __ldg(reinterpret_cast<const uint4*>(a.coladj + n0t) + w);
#pragma unroll
            for (int e = 0; e < 8; e++) {
              const uint32_t wd = e < 2 ? ca.x : e < 4 ? ca.y : e < 6 ? ca.z : ca.w;
              acc_shl(acc[w * 8 + e], sh + (int)(int16_t)(wd >> (16 * (e & 1))));
            }
          }
        }
        int shr = kSplitGuard;
        uint4 cx[TH / 8];
        if (!plain) {
          const uint4* csrc;
          if (grp.uni) {
            shr += gsig + (row_ok ? (int)a.rowadj[m] : 0);
            csrc = reinterpret_cast<const uint4*>(a.coladj + n0t);
          } else {
            shr += row_ok ? (int)a.rowexp[(int64_t)gk0 * a.Mtot + m] : 0;
            csrc = reinterpret_cast<const uint4*>(a.colexp + (int64_t)gk0 * a.colexp_ld + n0t);
          }
#pragma unroll
          for (int w = 0; w < TH / 8; w++) cx[w] = __ldg(csrc + w);
        }
        if (!wait_warp(&tfull[buf], (tcount / NB) & 1, abort_flag, a.err)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t taddr = tq + buf * BUF_COLS;
        if (plain)
          wide_drain<S, TH, true>(taddr, acc, shr, cx);
        else
          wide_drain<S, TH, false>(taddr, acc, shr, cx);
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[buf]);
        tcount++;
      }
      const int adj = plain ? kSplitGuard + sig0 + (row_ok ? (int)a.rowadj[m] : 0) : 0;
      if (ok && un.slot < 0) {
        const int Lrow = (row_ok ? a.emaxr[m] - kSplitBeta * (S + 1) - kSplitGuard : 0) + adj;
        if (a.f32)
          wide_store<TH, 1>(a, acc, slab, m - lane, lane, n0, Lrow, em + (plain ? ca : 0));
        else if (a.cplx)
          wide_store<TH, 2>(a, acc, slab, m - lane, lane, n0, Lrow, em + (plain ? ca : 0));
        else
          wide_store<TH, 0>(a, acc, slab, m - lane, lane, n0, Lrow, em + (plain ? ca : 0));
      } else if (ok && cb + half < a.CB) {
        // a piece of a split k-list: the same layout as from a group of 32-column CTAs
        uint4* dst = a.part + ((size_t)un.slot * CL + 2 * rank + half) * (TH * kSplitBM) + row;
#pragma unroll
        for (int c = 0; c < TH; c++) {
          if (plain) acc_shl(acc[c], adj + __shfl_sync(0xffffffffu, ca, c));
          dst[(size_t)c * kSplitBM] = make_uint4(acc[c][0], acc[c][1], acc[c][2], acc[c][3]);
        }
      }
      ok = epi_all(ok);
      if (!ok) break;
      if (a.timings && ew == 0 && lane == 0) {
        atomicMax(reinterpret_cast<unsigned long long*>(&a.timings[2 * (int64_t)u + 1]),
                  (unsigned long long)(gtimer() - t_unit));
        if (rank == 0) a.unit_cta[u] = cta;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
}

template <int S>
cudaError_t launch_wide(const SplitArgs& a, int groups, cudaStream_t st, bool after) {
  const size_t smem = split_wide_smem_bytes(S, a.wstages);
  cudaError_t e = cudaFuncSetAttribute(split_mma_wide_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // the register split assumes kWideRegsLaunch registers per thread at launch (a smaller
  // allocation could not satisfy the epilogue's setmaxnreg.inc): refuse otherwise
  cudaFuncAttributes fa{};
  e = cudaFuncGetAttributes(&fa, split_mma_wide_kernel<S>);
  if (e != cudaSuccess) return e;
  if (fa.numRegs != kWideRegsLaunch) return cudaErrorInvalidConfiguration;
  return launch_kernel(after, split_mma_wide_kernel<S>, dim3(groups * (a.cl / 2)), kWideThreads, smem, st, 1, a);
}

}  // namespace

size_t split_wide_smem_bytes(int s, int stages) {
  return 1024 /*alignment slack*/ + (size_t)stages * s * (kAChunk + kWideN * kSplitKC * 2) + kSplitBarBytes +
         (size_t)kSplitEpiWarps * kSlabBytes;
}

int split_wide_stages(int s) {
  int st = 8;
  while (st > 2 && split_wide_smem_bytes(s, st) > kMaxSmemPerCta) st--;
  return st;
}

cudaError_t launch_split_wide(const SplitArgs& a, int groups, cudaStream_t st, bool after) {
  if (a.cl != 2 && a.cl != 4) return cudaErrorInvalidValue;
  switch (a.s) {
    case 3: return launch_wide<3>(a, groups, st, after);
    case 4: return launch_wide<4>(a, groups, st, after);
    case 5: return launch_wide<5>(a, groups, st, after);
    case 6: return launch_wide<6>(a, groups, st, after);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace bsmm
