// Split-precision tile tasks on the tcgen05 tensor cores.
//
// The tile tasks C_ij += A_ik B_kj (paper Sec. 2.1) are computed with
// error-free Ozaki-style slicing (Ozaki, Ogita, Oishi, Rump, Numer. Algorithms
// 59, 2012), one power-of-two scale per tile:
//   e = smallest integer with max|x| < 2^e over the tile, rho_0 = x 2^-e,
//   N_t = rint(rho_{t-1} 2^(7t)), rho_t = rho_{t-1} - N_t 2^(-7t),  t = 1..s,
// so every slice is an integer of at most 8 bits, exact in bfloat16 and float16.
// For one tile pair the diagonal sums S_d = sum_{p+q=d} NA_p NB_q (d = 2..s+1)
// are integer matrices; with |S_d| <= 2^24 (inner blocks up to 512 elements for
// s = 6) the FP32 tensor-core accumulator holds them exactly. The epilogue forms
// T = sum_d S_d 2^(7(s+1-d)) exactly in int64 and adds T, shifted to its binary
// position e_A + e_B - 7(s+1), into an exact 128-bit integer accumulator per C
// element (no floating-point rounding and no FP64 instruction in the k loop; GB300's
// FP64 pipe is narrow). The sum is rounded once to FP64 at the end of the unit, so
// the result is fixed bit for bit, independent of schedule, unit order and k order.
//
// Kernels, in launch order (1 and 2 in slice.cu, the others here):
//   1. split_exp_kernel   per stored tile: the exponent e (integer max reduction);
//                         with one scale per line, split_exp_lines_kernel and
//                         split_scale_lines_kernel in its place.
//   2. split_pack_kernel  per (128-row block, k block) of A and (k block, tn-column
//                         block) of B: the s slices, stored as bf16/fp16 in the
//                         exact shared-memory image the tensor core reads (K-major,
//                         64-byte swizzle, 32-element chunks), so the contraction
//                         kernel moves them with plain 1-D bulk copies. The same
//                         launch writes, per (k block, row block / column block), the
//                         per-row / per-column offsets from the block's largest
//                         exponent and the scale classes.
//   3. split_mma_kernel   persistent, one CTA per SM, warp-specialised:
//                         warp 0 streams packed chunks into an S-stage shared-memory
//                         ring with cp.async.bulk (several k panels in flight -- the
//                         on-chip form of the paper's multiple-issue SUMMA
//                         iterations, Sec. 3.2); warps 1..3 share the issue of the
//                         tcgen05.mma slice products into double-buffered TMEM
//                         accumulators; warps 4..11 drain TMEM (zeroing it behind
//                         them), recombine in integer arithmetic and store
//                         C = alpha*fl(sum) + beta*C.
//                         split_mma_wide_kernel (wide.cu) in its place for products of
//                         long k lists.
//   4. split_reduce_kernel only for a plan that cut k-lists (split k, Sec. 3.2, Fig. 2):
//                         adds each cut region's exact partial sums and stores C.
// A work unit is a 128-row x tn-column block of the global C index space over its
// k-list (or one piece of it); the CTA that owns it runs its inner blocks in ascending
// order. Float32 and complex elements use the same kernels: the exponent and pack
// kernels read the element type, the epilogue rounds and stores it.
// wait_selftest_kernel exercises the bounded waits and the abort protocol (diagnostics).

#include <nvtx3/nvToolsExt.h>

#include <cstdint>
#include <type_traits>

#include "split_device.cuh"

namespace bsmm {

namespace {

// MMA issue: one thread issues tcgen05.mma instructions about one per 100 cycles, whatever
// their N, so the slice products of a step are spread over kMmaWarps issuing warps.
constexpr int kMmaWarps = 3;
constexpr int kEpiWarp0 = 1 + kMmaWarps;                 // first epilogue warp (warpgroups 1 and 2)
constexpr int kStoreWarps = 4;                           // C store warps (warpgroup 3), when present
constexpr int kStoreWarp0 = kEpiWarp0 + kSplitEpiWarps;  // first store warp
// Two forms of the contraction kernel: without store warps (the epilogue warps store each
// unit's C themselves) and with them (the C store of a unit runs while the epilogue drains
// the next one; it pays off when units are short).
template <bool SW>
constexpr int threads_of() {
  return 32 * (kStoreWarp0 + (SW ? kStoreWarps : 0));
}
// Register split with setmaxnreg (form with store warps): the CTA is launched with
// kThreadsSW x kRegsLaunch registers (the whole register file); the producer and MMA warps
// (warpgroup 0) and the store warps (warpgroup 3) give registers back and the epilogue warps
// take them. The shares add up to the launch's total exactly, so every setmaxnreg.inc is
// satisfiable.
constexpr int kThreadsSW = threads_of<true>();  // 512
constexpr int kRegsLaunch = 65536 / kThreadsSW;  // 128
constexpr int kRegsCtl = 80, kRegsEpi = 168, kRegsStore = 96;
static_assert(kEpiWarp0 % 4 == 0 && kStoreWarp0 % 4 == 0, "roles start on warpgroup boundaries");
static_assert(4 * 32 * kRegsCtl + kSplitEpiWarps * 32 * kRegsEpi + kStoreWarps * 32 * kRegsStore ==
                  kThreadsSW * kRegsLaunch,
              "the warpgroups' register shares must add up to the launch's registers");

// a.cl consecutive CTAs form a column-block group: they take the same units (a 128-row
// block times cl column blocks), each its own column block, at about the same time, so
// the A panel they all read is served from L2. Every CTA loads its own operands; no CTA
// reads or signals another's shared memory.
// WALK: the epilogue finds the accumulation groups on its own k list (products of long
// k lists) instead of taking the MMA warps' descriptors; the two ways share no code path,
// so each form keeps its own register allocation.
// DEEP: some inner block is deeper than the exact FP32 depth; such a block (it always
// starts a group of its own) is cut into groups of kdepth / 32 whole 32-deep chunks, the
// last of which may take the following blocks. A form of its own, because any extra work
// in the MMA-issuing loop slows every product.
template <int S, int TN, bool SW, bool WALK, bool DEEP>
__global__ void __launch_bounds__(threads_of<SW>(), 1) split_mma_kernel(const __grid_constant__ SplitArgs a) {
  constexpr int TH = TN / 2;                    // columns per epilogue thread
  constexpr int A_STAGE = S * kAChunk;          // bytes of A per stage
  constexpr int B_STAGE = S * TN * kSplitKC * 2;
  constexpr int STAGE = A_STAGE + B_STAGE;
  constexpr int BUF_COLS = S * TN;              // TMEM columns per accumulator buffer
  constexpr int W = S < kMmaWarps ? S : kMmaWarps;  // MMA warps with work: warp 1+w issues slices p = w+1, w+1+W, ...
  static_assert(A_STAGE % 16 == 0 && B_STAGE % 16 == 0, "bulk copies move multiples of 16 bytes");
  static_assert(TN == 32, "the coalesced C store maps one column to each lane");

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int stages = a.stages;
  uint64_t* bars = (uint64_t*)(smem + (size_t)stages * STAGE);
  uint64_t* full = bars;
  uint64_t* empty = bars + stages;
  uint64_t* tfull = bars + 2 * stages;
  uint64_t* tempty = tfull + 2;
  uint64_t* gready = tempty + 2;  // a group's descriptor is in gdesc[buf]
  uint64_t* cready = gready + 2;  // the unit's rounded results are in cstage
  uint64_t* cfree = cready + 1;   // the store warps are done with cstage
  uint64_t* drain = cfree + 1;    // one per MMA warp
  uint32_t* tmem_slot = (uint32_t*)(drain + kMmaWarps);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  // the accumulation group in TMEM buffer b: first k block, binary offset of a uniform
  // group, flags (1: uniform scale class, 2: the unit's last group); written by the first
  // MMA warp when it closes the group
  int4* gdesc = (int4*)(((uintptr_t)(tmem_slot + 2) + 15) & ~(uintptr_t)15);
  // the unit's results on their way to C: 128 rows x (TN + 1) bit patterns (padded rows)
  unsigned long long* cstage = (unsigned long long*)(smem + (size_t)stages * STAGE + kSplitBarBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int CL = a.cl;
  const int cta = blockIdx.x / CL;   // the group: schedules are per group
  const int rank = blockIdx.x % CL;  // this CTA's column block within the group's units
  grid_wait();  // before anything of global memory is read, the schedule included
  if constexpr (S > kWidePairsMaxS && SW && !DEEP)
    if (a.changes && a.changes[3]) return;  // the 64-column form ran
  const int ubeg = a.sched_ptr[cta], uend = a.sched_ptr[cta + 1];

  if (threadIdx.x == 0) {
    for (int st = 0; st < stages; st++) {
      mbar_init(&full[st], 1);
      mbar_init(&empty[st], W);  // released by every MMA warp
    }
    for (int b = 0; b < 2; b++) {
      mbar_init(&tfull[b], W);
      mbar_init(&tempty[b], kSplitEpiWarps);
      mbar_init(&gready[b], 1);
    }
    mbar_init(cready, kEpiThreads);         // every epilogue thread, after its row
    mbar_init(cfree, kStoreWarps * 32);     // every store thread, after its rows
    for (int w = 0; w < kMmaWarps; w++) mbar_init(&drain[w], 1);
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

  // Roles by warpgroup; with store warps each warpgroup first takes its register share
  // (every warp of the warpgroup executes the setmaxnreg, and it dominates the role's code).
  if (warp < kEpiWarp0) {
    if constexpr (SW) regs_dec<kRegsCtl>();
  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      uint32_t issued = 0;  // bit st: stage st holds an issued copy; its parity in issued_par
      uint32_t issued_par = 0;
      bool ok = true;
      ChunkCursor cur;
      cur.start(ubeg, uend);
      while (ok && cur.advance(a, CL, rank)) {
        if (!wait1(&empty[stage], phase ^ 1, abort_flag, a.err)) {
          ok = false;
          break;
        }
        uint8_t* sa = smem + (size_t)stage * STAGE;
        mbar_arrive_expect_tx(&full[stage], STAGE);
        bulk_g2s(sa, cur.asrc + (size_t)cur.kc * A_STAGE, A_STAGE, &full[stage]);
        bulk_g2s(sa + A_STAGE, cur.bsrc + (size_t)cur.kc * B_STAGE, B_STAGE, &full[stage]);
        issued |= 1u << stage;
        issued_par = (issued_par & ~(1u << stage)) | (phase << stage);
        if (++stage == stages) {
          stage = 0;
          phase ^= 1;
        }
      }
      // drain: every copy this thread issued has landed before the CTA may exit
      for (int st = 0; st < stages; st++) {
        if (!(issued >> st & 1)) continue;
        const uint32_t par = issued_par >> st & 1;
        const int64_t t0 = gtimer();
        while (!mbar_try_wait(&full[st], par)) {
          if (gtimer() - t0 > kWaitNs) {
            atomicOr(a.err, kErrTimeout);
            break;
          }
        }
      }
    }
  } else if (warp <= W) {
    // ------------------------------------------------------------ MMA issuers
    // Every MMA warp walks the same chunks and issues its share of each step's slice
    // products; all of them accumulate (the epilogue zeroes a buffer once drained), and
    // the order in which the tensor core applies them does not matter: every partial sum
    // is an integer below 2^24, exact in FP32.
    // The whole warp walks the list and one elected lane issues: every partial product's
    // descriptors then come from uniform registers. (With lane 0 alone in the loop each had
    // to be moved there first: 837 against 753 cycles per 6-slice chunk, issue alone.)
    {
      const int mw = warp - 1;
      int stage = 0;
      uint32_t phase = 0;
      uint32_t tcount = 0;
      bool ok = true;
      bool any = false;
      // Descriptors are built once: within a stage, slice p of A starts (p-1)*kAChunk bytes
      // in and the second 16-deep step 32 bytes in, i.e. fixed additions to the 16-byte
      // start-address field (which cannot carry: shared addresses are below 256 KB).
      const uint64_t adesc0 = sdesc_sw64(smem_u32(smem));
      const uint64_t bdesc0 = sdesc_sw64(smem_u32(smem) + A_STAGE);
      constexpr int NP = (S + W - 1) / W;  // slices per warp (upper bound)
      uint32_t idp[NP];
      uint32_t dcol[NP];
      uint64_t aoff[NP];
#pragma unroll
      for (int j = 0; j < NP; j++) {
        const int p = mw + 1 + j * W;
        idp[j] = idesc_f16(kSplitBM, (S + 1 - (p <= S ? p : S)) * TN, a.fp16 != 0);
        dcol[j] = (uint32_t)((p - 1) * TN);
        aoff[j] = (uint64_t)((p - 1) * (kAChunk >> 4));
      }
      for (int idx = ubeg; idx < uend && ok; idx++) {
        int g = a.sched_units[idx];
        const SplitArgs& P = a.prods ? a.prods[a.unit_prod[g]] : a;
        if (a.prods) g = a.unit_local[g];
        const SplitUnit un = P.units[g];
        const int cb = un.cb * CL + rank;
        UnitIter it;
        it.init(P, un, cb);
        GroupRule grp;
        bool in_group = false;
        uint32_t buf = 0;
        int gk0 = 0;  // the current group's first k block
        // per-k values are loaded one k block ahead, so their latency hides behind the
        // current block's MMAs; a group is closed when the next own k block does not join
        KAhead cur, nxt;
        cur.load(P, it.next_own(), un.rb, cb);
        while (cur.k >= 0 && ok) {
          nxt.load(P, it.next_own(), un.rb, cb);
          const int kt = cur.k;
          const int q = cur.q;
          const int nkc = (q + kSplitKC - 1) / kSplitKC;
          if (!(in_group && grp.joins(cur.uni, cur.sig, cur.q))) {
            if (in_group) {  // the previous group is complete
              close_group(mw == 0, gdesc, gready, tfull, buf, gk0, grp, false);
              tcount++;
            }
            buf = tcount & 1;
            const uint32_t use = tcount >> 1;
            // the buffer was drained and zeroed by the epilogue (use 0: zeroed at start)
            if (!wait_warp(&tempty[buf], use & 1, abort_flag, a.err)) {
              ok = false;
              in_group = false;
              break;
            }
            tc_fence_after();
            grp.start(cur.uni, cur.sig, cur.q, P.kdepth);
            gk0 = kt;
            in_group = true;
          }
          uint32_t dbase = tmem_base + buf * BUF_COLS;
          for (int kc = 0; kc < nkc; kc++) {
            if constexpr (DEEP) {
              const int cpg = P.kdepth >= kSplitKC ? P.kdepth / kSplitKC : 1;
              if (kc > 0 && q > P.kdepth && kc % cpg == 0) {  // the block's next group
                close_group(mw == 0, gdesc, gready, tfull, buf, gk0, grp, false);
                tcount++;
                buf = tcount & 1;
                if (!wait_warp(&tempty[buf], (tcount >> 1) & 1, abort_flag, a.err)) {
                  ok = false;
                  break;
                }
                tc_fence_after();
                dbase = tmem_base + buf * BUF_COLS;
              }
            }
            if (!wait_warp(&full[stage], phase, abort_flag, a.err)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (elect_one()) {
              const uint64_t soff = (uint64_t)((stage * STAGE) >> 4);
              const uint64_t ad = adesc0 + soff, bd = bdesc0 + soff;
              const bool two = q - kc * kSplitKC > 16;  // second 16-deep step of the 32-deep chunk
#pragma unroll
              for (int j = 0; j < NP; j++) {
                if (mw + 1 + j * W > S) break;
                umma_f16(dbase + dcol[j], ad + aoff[j], bd, idp[j], 1u);
                if (two) umma_f16(dbase + dcol[j], ad + aoff[j] + 2, bd + 2, idp[j], 1u);
              }
              umma_commit(&empty[stage]);  // the stage is free once these MMAs have finished
            }
            __syncwarp();
            any = true;
            if (++stage == stages) {
              stage = 0;
              phase ^= 1;
            }
          }
          if constexpr (DEEP) {
            const int cpg = P.kdepth >= kSplitKC ? P.kdepth / kSplitKC : 1;
            if (q > P.kdepth) grp.depth = q - kSplitKC * cpg * ((nkc - 1) / cpg);  // its last group's depth
          }
          cur = nxt;
        }
        if (in_group && ok) {  // the unit's last group
          close_group(mw == 0, gdesc, gready, tfull, buf, gk0, grp, true);
          tcount++;
        }
      }
      // drain: every MMA this warp issued has completed before TMEM is released
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
  }
  } else if (warp < kStoreWarp0) {
    if constexpr (SW) regs_inc<kRegsEpi>();
    // ------------------------------------------------------------ epilogue warps
    const int ew = warp - kEpiWarp0;   // 0..7
    const int quad = warp & 3;         // TMEM lane quadrant this warp may access
    const int half = ew >> 2;          // which half of the tn columns
    const int row = quad * 32 + lane;  // row inside the unit
    const uint32_t tq = tmem_base + ((uint32_t)(quad * 32) << 16) + half * TH;  // this warp's lanes and columns
    // both accumulator buffers start at zero; the MMA warps only ever accumulate
#pragma unroll 1
    for (int b = 0; b < 2; b++)
#pragma unroll
      for (int d = 0; d < S; d++)
#pragma unroll
        for (int cc = 0; cc < TH / 8; cc++) tmem_zero8(tq + b * BUF_COLS + d * TN + cc * 8);
    tmem_st_wait();
    tc_fence_before();
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(&tempty[0]);
      mbar_arrive(&tempty[1]);
    }
    uint32_t tcount = 0;
    uint32_t ncs = 0;  // uses of cstage so far
    bool ok = true;
    for (int idx = ubeg; idx < uend && ok; idx++) {
      int u = a.sched_units[idx];
      const SplitArgs& P = a.prods ? a.prods[a.unit_prod[u]] : a;
      if (a.prods) u = a.unit_local[u];
      const SplitUnit un = P.units[u];
      const int cb = un.cb * CL + rank;
      if (cb >= P.CB) continue;  // a group's CTA past the last column block has no work
      // timing record: the unit's start (the group's first CTA) and the longest time any CTA
      // of the group spends on it
      const int64_t t_unit = a.timings && ew == 0 && lane == 0 ? gtimer() : 0;
      if (a.timings && rank == 0 && ew == 0 && lane == 0) a.timings[2 * (int64_t)u] = t_unit;
      const int64_t m = (int64_t)un.rb * kSplitBM + row;
      const bool row_ok = m < P.Mtot;
      const int64_t n0 = (int64_t)cb * TN + half * TH;
      uint32_t acc[TH][4];  // exact 128-bit two's-complement sums, unit 2^L per column
#pragma unroll
      for (int c = 0; c < TH; c++) acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = 0u;
      // The unit's accumulation groups, in the order the MMA warps fill them. With WALK the
      // epilogue walks the CTA's own k list with the MMA warps' rule, ahead of them;
      // otherwise it takes each group's descriptor when the first MMA warp closes it (none
      // when this CTA's column block has no B tile in the unit's inner range: the planner's
      // own mask). Either way the groups are the same, in the same order.
      UnitIter it;
      int kt = -1;
      [[maybe_unused]] int sub = 0;  // DEEP: groups already taken from k block kt
      if constexpr (WALK) {
        it.init(P, un, cb);
        kt = it.next_own();
      }
      bool more = WALK ? kt >= 0 : ((un.own >> rank) & 1) != 0;
      while (more) {
        const uint32_t buf = tcount & 1, use = tcount >> 1;
        int gk0, gsig;  // the group's first k block and, for a uniform group, its class
        bool guni;
        if constexpr (WALK) {
          GroupRule grp;
          {
            int sg = 0;
            const bool uni = scale_class(P, kt, un.rb, cb, sg);
            grp.start(uni, sg, P.q[kt], P.kdepth);
          }
          gk0 = kt;
          guni = grp.uni;
          gsig = grp.sig;
          bool whole = true;  // DEEP: a deep block's groups but its last take no other block
          if constexpr (DEEP) {
            const int qk = P.q[kt];
            if (qk > P.kdepth) {
              const int cpg = P.kdepth >= kSplitKC ? P.kdepth / kSplitKC : 1;
              const int nsub = ((qk + kSplitKC - 1) / kSplitKC + cpg - 1) / cpg;
              if (++sub < nsub) {
                whole = false;
              } else {
                grp.depth = qk - kSplitKC * cpg * (nsub - 1);
                sub = 0;
              }
            }
          }
          if (whole) {
            int kn = it.next_own();
            for (; kn >= 0; kn = it.next_own()) {
              int sg = 0;
              const bool uni = scale_class(P, kn, un.rb, cb, sg);
              if (!grp.joins(uni, sg, P.q[kn])) break;
            }
            kt = kn;
          }
          more = kt >= 0;
        } else {
          // (the epilogue warps sleep between polls here: while the MMA warps fill a group
          // they would otherwise take issue slots from the producer and MMA threads)
          if (!wait_warp(&gready[buf], use & 1, abort_flag, a.err, kWaitNs, kGroupPollNs)) {
            ok = false;
            break;
          }
          const int4 gd = gdesc[buf];
          more = (gd.z & 2) == 0;
          gk0 = gd.x;
          guni = (gd.z & 1) != 0;
          gsig = gd.y;
        }
        // the binary position of the group's integers: one shift for a uniform group (its
        // common class plus the row's and the columns' parts), per-row and per-column
        // offsets for a lone k block; loaded while the tensor core finishes the group
        int shr = kSplitGuard;
        uint4 cx[TH / 8];
        if (guni) {
          shr += gsig + (row_ok ? (int)P.rowadj[m] : 0);
          const uint4* src = reinterpret_cast<const uint4*>(P.coladj + n0);
#pragma unroll
          for (int w = 0; w < TH / 8; w++) cx[w] = __ldg(src + w);
        } else {
          shr += row_ok ? (int)P.rowexp[(int64_t)gk0 * P.Mtot + m] : 0;
          const uint4* src = reinterpret_cast<const uint4*>(P.colexp + (int64_t)gk0 * P.colexp_ld + n0);
#pragma unroll
          for (int w = 0; w < TH / 8; w++) cx[w] = __ldg(src + w);
        }
        if (!wait_warp(&tfull[buf], use & 1, abort_flag, a.err)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t taddr = tq + buf * BUF_COLS;
        // columns in batches of CW (4 for s >= 5 keeps the TMEM values and the 128-bit
        // sums within the register budget)
        constexpr int CW = S >= 5 ? 4 : 8;
#pragma unroll
        for (int cc = 0; cc < TH / CW; cc++) {
          uint32_t v[S][CW];
#pragma unroll
          for (int d = 0; d < S; d++) {
            if constexpr (CW == 8)
              tmem_ld8(taddr + d * TN + cc * CW, v[d]);
            else
              tmem_ld4(taddr + d * TN + cc * CW, v[d]);
          }
          tmem_ld_wait();
#pragma unroll
          for (int d = 0; d < S; d++) {  // ready for the buffer's next use
            if constexpr (CW == 8)
              tmem_zero8(taddr + d * TN + cc * CW);
            else
              tmem_zero4(taddr + d * TN + cc * CW);
          }
#pragma unroll
          for (int c = 0; c < CW; c++) {
            const long long T = diagonal_sum<S, CW, false>(v, c);  // exact: the tensor core's FP32 sums are integers
            const int col = cc * CW + c;  // column within this thread's TH
            const uint4& w4 = cx[col >> 3];
            const int e = col & 7;
            const uint32_t wd = e < 2 ? w4.x : e < 4 ? w4.y : e < 6 ? w4.z : w4.w;
            acc_add(acc[col], T, shr + (int)(int16_t)(wd >> (16 * (e & 1))));
          }
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[buf]);
        tcount++;
      }
      // (a warp whose wait gave up still passes the barriers below, so that no other
      // epilogue warp waits at them for it; every wait before them is bounded and sees the
      // abort flag, so all eight warps reach them, and the last one agrees on the outcome,
      // so all eight leave the unit loop together)
      if (un.slot < 0) {
        // C = alpha*fl(sum) + beta*C on the unit's elements that lie in S_C tiles: each
        // thread rounds its row's sums to doubles into the staging buffer (with store warps,
        // once they are done with the previous unit's); then whole rows are stored, lane =
        // column, so a store instruction writes one or two contiguous row segments. With
        // store warps the store runs while this warp drains the next unit.
        // the accumulator's unit 2^L: per row block and column block of tiles, or per row
        // and column with row/column scaling (loaded before the wait for the staging buffer)
        int emc[TH];
        load_emaxc<TH>(P, n0, emc);
        const int Lrow = row_ok ? P.emaxr[m] - kSplitBeta * (S + 1) - kSplitGuard : 0;
        if constexpr (SW)
          if (ok && !wait_warp(cfree, (ncs & 1) ^ 1, abort_flag, a.err)) ok = false;
        if (ok) {
          unsigned long long* srow = cstage + row * (TN + 1) + half * TH;
          if (P.f32)
            round_row<TH, true>(acc, srow, emc, Lrow);
          else
            round_row<TH, false>(acc, srow, emc, Lrow);
        }
        if constexpr (SW) {
          mbar_arrive(cready);  // every thread: its row is in cstage (release)
          ncs++;
        } else {
          StoreCol col;
          store_col(P, cb, lane, col);
          asm volatile("bar.sync 1, %0;" ::"r"(kEpiThreads) : "memory");
          if (ok && !*abort_flag) store_unit<TN, kSplitEpiWarps>(P, cstage, un.rb, col, ew, lane, a.err);
        }
      } else if (ok) {
        // a piece of a split k-list: its exact partial sums go to the workspace (column-
        // major, so the 32 rows of a warp write 512 contiguous bytes per column)
        uint4* dst = P.part + ((size_t)un.slot * CL + rank) * (TN * kSplitBM) + (size_t)half * TH * kSplitBM + row;
#pragma unroll
        for (int c = 0; c < TH; c++) dst[(size_t)c * kSplitBM] = make_uint4(acc[c][0], acc[c][1], acc[c][2], acc[c][3]);
      }
      ok = epi_all(ok);  // every epilogue warp has the same outcome (and, without store warps,
                         // cstage is free again)
      if (!ok) break;
      if (a.timings && ew == 0 && lane == 0) {
        atomicMax(reinterpret_cast<unsigned long long*>(&a.timings[2 * (int64_t)u + 1]),
                  (unsigned long long)(gtimer() - t_unit));
        if (rank == 0) a.unit_cta[u] = cta;
      }
    }
  } else if constexpr (SW) {
    regs_dec<kRegsStore>();
    // ------------------------------------------------------------ C store warps
    // The units' rounded results from the staging buffer to C, in the epilogue's unit
    // order, while the epilogue warps drain the next unit.
    const int sw = warp - kStoreWarp0;
    uint32_t ncs = 0;
    for (int idx = ubeg; idx < uend; idx++) {
      int u = a.sched_units[idx];
      const SplitArgs& P = a.prods ? a.prods[a.unit_prod[u]] : a;
      if (a.prods) u = a.unit_local[u];
      const SplitUnit un = P.units[u];
      const int cb = un.cb * CL + rank;
      if (cb >= P.CB || un.slot >= 0) continue;  // units that do not use the staging buffer
      StoreCol col;
      store_col(P, cb, lane, col);  // its loads run while the unit is still being computed
      if (!wait_warp(cready, ncs & 1, abort_flag, a.err, kWaitNs, 200)) break;
      if (!*abort_flag) store_unit<TN, kStoreWarps>(P, cstage, un.rb, col, sw, lane, a.err);
      mbar_arrive(cfree);  // every thread: done reading cstage (release)
      ncs++;
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
}

// ---------------------------------------------------------------- kernel 4: split-k reduction
// The reduction task of a region whose k-list was cut into pieces (Sec. 3.2, Fig. 2).
// The pieces' partial sums are exact 128-bit integers in the same unit 2^L, so adding
// them is exact in any order and the rounded result equals the unsplit one bit for bit;
// it is rounded once and stored like the contraction's epilogue. One CTA of 256 threads
// per 32 rows of a (region, column block of the region's group); thread = (row, 4 columns).
// Bound by HBM (16 bytes per element and piece): a CTA per 128 rows left most SMs idle on
// few regions, and its loads ran one piece after the other (thin 512 x 524288 product, 78 MB
// of partials: 62 us; 31 us this way).
constexpr int kRedRows = 32;
template <int TN>
__global__ void __launch_bounds__(256) split_reduce_kernel(const __grid_constant__ SplitArgs a) {
  constexpr int kCols = TN * kRedRows / 256;  // columns per thread
  constexpr int kParts = kSplitBM / kRedRows;
  __shared__ unsigned long long cstage[kRedRows * (TN + 1)];
  grid_wait();
  const int unit = blockIdx.x / kParts, part = blockIdx.x % kParts;
  const SplitRed rd = a.red[unit / a.cl];
  const int rank = unit % a.cl;
  const int cb = rd.cb * a.cl + rank;
  if (cb >= a.CB) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = part * kRedRows + lane;  // a warp reads 32 rows of a column: 512 contiguous bytes
  const int64_t m = (int64_t)rd.rb * kSplitBM + row;
  const bool row_ok = m < a.Mtot;
  const int Lrow =
      row_ok ? a.emaxr[m] - kSplitBeta * (a.s + 1) - kSplitGuard : 0;
  const int64_t n0 = (int64_t)cb * TN + warp * kCols;
  const size_t piece_stride = (size_t)a.cl * TN * kSplitBM;
  const uint4* src =
      a.part + ((size_t)rd.slot0 * a.cl + rank) * (TN * kSplitBM) + (size_t)warp * kCols * kSplitBM + row;
  uint32_t w[kCols][4];
#pragma unroll
  for (int c = 0; c < kCols; c++) w[c][0] = w[c][1] = w[c][2] = w[c][3] = 0u;
#pragma unroll 4
  for (int p = 0; p < rd.n; p++)
#pragma unroll
    for (int c = 0; c < kCols; c++) add128(w[c], __ldg(src + p * piece_stride + (size_t)c * kSplitBM));
  StoreCol col;
  store_col(a, cb, lane, col);
#pragma unroll
  for (int c = 0; c < kCols; c++) {
    const int64_t n = n0 + c;
    unsigned long long v = 0ull;
    if (row_ok && n < a.Ntot) {
      const int L = Lrow + a.emaxc[n];
      v = a.f32 ? acc_bits_any<true>(w[c][0], w[c][1], w[c][2], w[c][3], L)
                : acc_bits_any<false>(w[c][0], w[c][1], w[c][2], w[c][3], L);
    }
    cstage[lane * (TN + 1) + warp * kCols + c] = v;
  }
  __syncthreads();
  constexpr int kWarps = kSplitBM / (kRedRows / 8);  // 4 rows per warp over the whole 128-row block
  store_unit<TN, kWarps>(a, cstage - part * kRedRows * (TN + 1), rd.rb, col, part * 8 + warp, lane, a.err);
}

// ---------------------------------------------------------------- bounded-wait self-test
// Two mbarriers that no thread ever arrives at. Warp 0 (one thread) waits on the first
// with the given limit, runs out, sets the error word and the abort flag; warps 1 and 2
// wait on the second (warp-uniform waits, a 20x longer limit) and leave as soon as they
// see the abort flag. The kernel then exits normally: the contraction's wait functions
// and its abort protocol, exercised without a hang.
__global__ void __launch_bounds__(96) wait_selftest_kernel(int32_t* err, int64_t limit_ns) {
  __shared__ uint64_t bars[2];
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    if (threadIdx.x == 0) wait1(&bars[0], 0, &abort_flag, err, limit_ns);
  } else {
    wait_warp(&bars[1], 0, &abort_flag, err, 20 * limit_ns);
  }
  __syncthreads();
}

template <int S, int TN, bool SW, bool WALK, bool DEEP = false>
cudaError_t launch_mma(const SplitArgs& a, int groups, cudaStream_t st, bool after) {
  const size_t smem = split_smem_bytes(S, TN, a.stages);
  cudaError_t e = cudaFuncSetAttribute(split_mma_kernel<S, TN, SW, WALK, DEEP>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if constexpr (SW) {
    // the register split assumes exactly kRegsLaunch registers per thread at launch (a
    // smaller allocation could not satisfy the epilogue's setmaxnreg.inc): refuse otherwise
    cudaFuncAttributes fa{};
    e = cudaFuncGetAttributes(&fa, split_mma_kernel<S, TN, SW, WALK, DEEP>);
    if (e != cudaSuccess) return e;
    if (fa.numRegs != kRegsLaunch) return cudaErrorInvalidConfiguration;
  }
  return launch_kernel(after, split_mma_kernel<S, TN, SW, WALK, DEEP>, dim3(groups * a.cl), threads_of<SW>(), smem, st, 1,
                       a);
}

template <int S>
cudaError_t launch_mma_sw(const SplitArgs& a, int groups, cudaStream_t st, bool after) {
  if (a.cl != 1 && a.cl != 2 && a.cl != 4) return cudaErrorInvalidValue;
  // the walking epilogue is built for the forms with store warps and 3 to 6 slices (the
  // dense products' default); other forms take the descriptors whatever epi_walk says
  if (a.deep) {  // products with inner blocks deeper than the exact depth: store-warp forms
    if (!a.sw) return cudaErrorInvalidConfiguration;
    if constexpr (S >= 3)
      if (a.epi_walk) return launch_mma<S, 32, true, true, true>(a, groups, st, after);
    return launch_mma<S, 32, true, false, true>(a, groups, st, after);
  }
  if constexpr (S >= 3)
    if (a.sw && a.epi_walk) return launch_mma<S, 32, true, true>(a, groups, st, after);
  return a.sw ? launch_mma<S, 32, true, false>(a, groups, st, after) : launch_mma<S, 32, false, false>(a, groups, st, after);
}

// Groups of cl CTAs that are resident at once: the persistent grid (one CTA per SM at
// this shared-memory size) divided into groups.
template <int S, bool SW>
int max_groups_for(int cl, int stages) {
  const size_t smem = split_smem_bytes(S, 32, stages);
  if (cudaFuncSetAttribute(split_mma_kernel<S, 32, SW, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return 0;
  int per_sm = 0, dev = 0, sms = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, split_mma_kernel<S, 32, SW, false, false>, threads_of<SW>(), smem) !=
      cudaSuccess)
    return 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  return cl > 0 ? per_sm * sms / cl : 0;
}

template <int S>
int max_groups_s(int cl, int stages, bool sw) {
  return sw ? max_groups_for<S, true>(cl, stages) : max_groups_for<S, false>(cl, stages);
}

}  // namespace

// NVTX ranges name the phases of a product for a timeline tool (host-side enqueue spans).
cudaError_t launch_split(const SplitArgs& a, int ctas, cudaStream_t st, cudaEvent_t* ev, int* nk, bool after) {
  int k = 0;
  if (ev) cudaEventRecord(ev[0], st);
  nvtxRangePushA("bsmm split: exponents, scales, slices");
  cudaError_t e = launch_split_prep(a, st, ev, &k, after);
  nvtxRangePop();
  if (e != cudaSuccess) return e;
  nvtxRangePushA("bsmm split: contraction");
  after = !ev && split_prep_kernels(a) > 0;
  if (a.wide && !a.prods && a.changes) {  // both forms, of which the scale classes chose one
    SplitArgs b = a;
    b.sched_ptr = a.sched_sel;
    e = launch_split_wide(b, ctas, st, after);
    b.sched_ptr = a.sched_ptr2;
    b.sched_units = a.sched_units2;
    if (e == cudaSuccess) e = launch_split_mma(b, (ctas + 1) / 2, st, true);
  } else {
    e = a.wide && !a.prods ? launch_split_wide(a, ctas, st, after) : launch_split_mma(a, ctas, st, after);
  }
  nvtxRangePop();
  if (ev) cudaEventRecord(ev[++k], st);
  if (e == cudaSuccess && !a.prods && a.n_red > 0) {  // a batch launches its products' reductions
    nvtxRangePushA("bsmm split: split-k reduction");
    e = launch_split_reduce(a, st, !ev);
    nvtxRangePop();
    if (ev) cudaEventRecord(ev[++k], st);
  }
  if (nk) *nk = k;
  return e;
}

cudaError_t launch_wait_selftest(int32_t* err, int64_t limit_ns, cudaStream_t st) {
  wait_selftest_kernel<<<1, 96, 0, st>>>(err, limit_ns);
  return cudaGetLastError();
}

cudaError_t launch_split_reduce(const SplitArgs& a, cudaStream_t st, bool after) {
  if (a.n_red <= 0) return cudaSuccess;
  return launch_kernel(after, split_reduce_kernel<32>, dim3(a.n_red * a.cl * (kSplitBM / kRedRows)), 256, 0, st, 1, a);
}

cudaError_t launch_split_mma(const SplitArgs& a, int ctas, cudaStream_t st, bool after) {
  cudaError_t e;
  switch (a.s) {  // `ctas` counts groups of a.cl CTAs
    case 1: e = launch_mma_sw<1>(a, ctas, st, after); break;
    case 2: e = launch_mma_sw<2>(a, ctas, st, after); break;
    case 3: e = launch_mma_sw<3>(a, ctas, st, after); break;
    case 4: e = launch_mma_sw<4>(a, ctas, st, after); break;
    case 5: e = launch_mma_sw<5>(a, ctas, st, after); break;
    case 6: e = launch_mma_sw<6>(a, ctas, st, after); break;
    default: e = cudaErrorInvalidValue;
  }
  return e;
}

int split_max_clusters(int s, int cl, int stages, bool sw) {
  switch (s) {
    case 1: return max_groups_s<1>(cl, stages, sw);
    case 2: return max_groups_s<2>(cl, stages, sw);
    case 3: return max_groups_s<3>(cl, stages, sw);
    case 4: return max_groups_s<4>(cl, stages, sw);
    case 5: return max_groups_s<5>(cl, stages, sw);
    case 6: return max_groups_s<6>(cl, stages, sw);
    default: return 0;
  }
}

}  // namespace bsmm
