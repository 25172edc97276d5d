// Token-importance scoring on the Blackwell tensor cores (Eqs. 3, 14, 15), bf16 inputs.
//
// One persistent kernel, one CTA per SM.  K is streamed from HBM exactly once:
//
//   pass 1 (statistics)  tile = 128 tokens.  D[query row, token] = Q K^T on tcgen05 with the
//                        accumulator in TMEM.  Query rows sit on TMEM lanes, so the softmax
//                        denominator of a row (Eq. 3) is an in-thread sum: every row keeps a
//                        reference exponent and a running sum of 2^(logit - reference).
//   exchange             a run of RT consecutive tiles of one (layer, sequence, KV head) unit
//                        yields one (reference, sum) per row.  The short way: every row has a
//                        fixed reference (its logit against token 0, from a small kernel that
//                        runs first) and one 64-bit word; the run's sum is rescaled to that
//                        reference, converted to fixed point (2^-20) and added, together with an
//                        arrival count in the top byte, with one integer reduction.  Integer
//                        addition makes the total independent of the order of arrival, and sum
//                        and count travel in one word, so a reader of the sum needs no fence: the
//                        word is complete when its count equals the unit's runs.  That is two round
//                        trips to L2 between the last pass-1 tile of a unit and its first pass-2
//                        tile.  The long way, for a run's sum that does not fit the fixed-point
//                        range (a token about 14 nats above token 0): the run writes its
//                        (reference, sum) of that row to global memory, marks itself in the row's
//                        bitmap of such runs, and only then counts itself into the word, with
//                        release semantics (the runs that fit add relaxed and write nothing
//                        else); a pass-2 thread whose word shows such runs acquires the complete
//                        word and folds their records, in run order (the same order for every
//                        reader), into the fixed-point sum of the others.
//   pass 2 (emit)        the same CTA revisits its tiles as soon as their unit's statistics are
//                        complete, when their K rows are still in L2.  D[token, query row] = K Q^T (operands swapped:
//                        tokens on TMEM lanes), so the max over the window rows (Eq. 14) and the
//                        mean/max over the query heads of the group (Eq. 15) are in-thread and
//                        the score store is coalesced.  max_m exp(s_m - lse_m) is evaluated as
//                        exp(max_m(s_m - lse_m)): one exponential per query head, not per row.
//
// A unit is a (layer, sequence, KV head, row tile): the G x w window rows of a KV head are cut
// into row tiles of at most 128 rows: whole query heads where w <= 128 (w = 8, 16, 32, 64, 128 as
// compile-time specialisations, any other length through one variant that reads it at run time),
// pieces of one query head for longer windows, so that any GQA group and window runs here; with
// more than one row tile the pass-2 results are partial aggregates that the Eq. 16 kernel combines
// in a fixed order.
//
// The two passes of a CTA are two pipelines of their own (copies -> K stages and Q slots -> MMAs ->
// accumulators -> epilogue) over the same list of runs; they share nothing but the issue slots, the
// tensor pipe and shared memory.  Pass 1 has its Q, the row operand, in TMEM (copied there once per run) and one
// accumulator, which its epilogue empties at once.  Pass 2 goes as fast as the statistics arrive; pass 1 is held to at most
// `lead` tiles ahead of it (two runs where a unit has no more runs than there are CTAs: 38 MB of K at
// 148 CTAs, which L2 still holds), exactly what the statistics need: they need every run of a unit, and
// the other CTAs' runs of it lie that far ahead at most, so the CTAs cannot wait for each other in a
// circle while all of them are resident (the host checks that they can be).  Windows longer than 128 rows get
// two runs more: 77 MB of copies, but the row tiles of a KV head follow one another and copy the same rows (a group of 4 with 500 rows
// 16 times: 5 MB of K, or one head's where the context is long, 34 MB at 128K).  Every wait (mbarrier or
// global word) is bounded; on expiry the kernel records KVC_ERR_TIMEOUT, stops computing and drains.
//
// Warp roles (512 threads): warp 0 = TMA producer of pass 1 (K, Q, L2 prefetch), warp 3 = of pass 2; warp
// 1 = MMA issuer of pass 1 and TMEM owner, warp 2 = of pass 2; warps 4-7 = pass-2 epilogue; warps 8-15 = pass-1
// epilogue, two groups of four warps.  The four single warps
// run their loops with all lanes and elect a lane for each MMA, commit or copy: from one lane of a diverged
// warp every such instruction first moves its operands to uniform registers, about 50 clocks per MMA.
//
// What bounds it (waits counted in an instrumented copy, heads of 128, clocks per pair of tiles = 128 rows x 128 tokens in both
// passes): the two epilogues.  Tensor pipe and special-function pipe have 1024 clocks of work each, DRAM, L2 and the data banks of
// shared memory are at half or less.  With one row tile per unit a pair took 1890: pass 1's epilogue was busy for 1700 of them
// (1150 to 1250 of exponentials, both warps of a scheduler at once, and the rest, barrier, TMEM load, the exchange of the halves,
// at once as well), pass 2's for 1540, because each of its 32-column chunks waited for an accumulator load and for eight
// 16-byte reads of -log-sum-exps, which queue behind pass 1's exponentials (all lanes reading one address: 2.1 clocks of the
// SM each, 270 per tile).  Hence:
//   - one row tile per unit: the pass-2 epilogue keeps a run's 128 -log-sum-exps in registers (216 per thread, taken from the
//     single warps and from pass 1 by setmaxnreg), reads them once per run, and loads a chunk while it works on the one before:
//     8B shape at 32K 1078 -> 1060 us per pass, 4 sequences of 5003 with heads of 64 442 -> 430 (8K and less within 1 %).  Pass 1's epilogue
//     is what is left: 1750 of 1800 clocks.
//   - several row tiles: a work unit has two of them, which share every K tile in shared memory.  Pass 1's
//     two groups then take a row tile each, a tile's 128 columns at once in registers (168 per thread): half of the rounds of
//     barrier and load, and the groups are out of phase, where with one row tile each takes half of the columns of every tile.
//     Pass 2 takes 16 columns at a time, the next 16 in flight.  Window 64, GQA group 7 at 128K 4400 -> 4280 us per pass, 500-row
//     windows 1203 -> 1158; 1690 clocks per pair, of which pass 2's epilogue is busy for 1530.
// Registers decide the rest: a warp's 128 exponentials take 1134 clocks when the compiler has room to overlap them and 2125
// when it has not (it then waits for every pair), so in the second form the logits die in their exponentials.
// Power is the rest: the 8B shape's scoring at 32K takes 573 us for 50 ms from rest and 690 to 710 back to back, where the clock reads 1.17 to
// 1.21 GHz: 830 K clocks, 435 us at 1.9 GHz.  (The same clocks in 573 us are 1.45 GHz; the reading, 1.965, lags by 0.1 s.)
#include <cuda.h>

#include <atomic>
#include <mutex>

#include "kvc_internal.cuh"
#include "value_norm.cuh"

namespace kvc {
namespace {

constexpr int kTile = 128;            // tokens per tile = MMA M = MMA N
constexpr int kFastThreads = 512;
// Registers per thread of the warpgroups, out of the 128 that the kernel starts with: the single warps, the pass-2 epilogue
// and the pass-1 epilogue's two groups.  With one row tile pass 2 keeps a run's -log-sum-exps, with two pass 1 a whole tile's logits.
// (A kernel that moves registers must not call functions out of line: ptxas 12.9 crashes on it, so the cold paths are inlined.)
constexpr int kRegsStart = 128;
template <int kRT> struct Regs;
template <> struct Regs<1> { static constexpr int kSingle = 56, kP2 = 216, kP1 = 120; };
template <> struct Regs<2> { static constexpr int kSingle = 64, kP2 = 112, kP1 = 168; };

constexpr int kRows = 128;            // query rows per unit handled by one MMA (R <= 128)
constexpr int kMinRunTiles = 4;       // tiles per run; runs are longer only where a unit would otherwise have more than 255
constexpr int kPrefetch = 2;          // pass-1 tiles prefetched into L2 ahead of their load
constexpr float kLog2eF = 1.4426950408889634f;
constexpr float kRescaleLimit = 1.8446744e19f;               // 2^64: a chunk sum beyond it restarts with a new reference
constexpr unsigned long long kDefaultWaitLimitNs = 2000000000ull;   // 2 s: far beyond any healthy wait

constexpr int kMaxFastLayers = 112;   // 2 tensor maps per layer must fit the 32 KB kernel-parameter space

struct FastParams {
  CUtensorMap k_maps[kMaxFastLayers];   // K^(l) as (64, N, d / 64, Hkv, Bt), box 64 x 128 x d / 64 x 1 x 1, 128-byte swizzle:
                                        // a tile arrives as d / 64 blocks of 128 rows of 128 bytes with one copy
  CUtensorMap q_maps[kMaxFastLayers];   // Q^(l) as (d, w, Hq, Bt), box 64 x w x G x 1
  float2* partial;             // [U][RPU][128]: (ref, sum) of a row over one run, written only where the sum
                               // does not fit the row's word
  unsigned long long* ovf;     // [U][128][4], preset to 0: per row, the runs (bit j) that wrote such a record
  unsigned long long* acc;     // [U][128], preset to 0: per row  arrivals << 56 | overflows << 48 | sum in units
                               // of 2^-20 of 2^(logit - ref[row]), added to by every run of the unit
  const float* ref;            // [U][128]: the row's reference exponent (its scaled logit against token 0)
  int* status;                 // device status word (may be null)
  float* scores;               // [L*Bt*Hkv][N], or with QT > 1 the partial aggregates [QT][L*Bt*Hkv][N]
  int L, Bt, Hkv, G;
  int HPT, QT, w;              // query heads per row tile, row tiles per KV head, window rows per query head
  int QP;                      // work units per KV head: QT, or with two row tiles per unit ceil(QT / 2)
  int CH;                      // row tiles per query head: 1, or ceil(w / 128) for windows longer than 128 rows
                               // (then HPT = 1 and row tile q holds rows (q % CH) * 128 .. of query head q / CH)
  long long N, q_pos0;
  int U, NT, RPU, grid;        // units, tiles per unit, runs per unit, CTAs
  int RT;                      // tiles per run
  int step_u, step_j;          // grid = step_u * RPU + step_j: how a CTA's next run moves (unit, run in unit)
  int step_l, step_b, step_h, step_q;  // step_u = ((step_l * Bt + step_b) * Hkv + step_h) * QP + step_q
  unsigned int total_runs;     // runs of all work units
  int lead;                    // tiles by which pass 1 may be ahead of pass 2 (their K copies)
  float sl2e;                  // scale * log2(e)
  int agg_group;
  unsigned long long wait_limit_ns;   // bound of every device-side wait
  // the value norms, by the CTAs from `grid` on (see value_norm_cta): V^(l), their place, V's strides in elements
  LayerPtrs v;
  float* vnorm;
  long long vs0, vs1, vs2;
  int norm_ctas;               // 0: none
  int withhold_unit;           // test hook: the statistics of this unit are never sent (-1: none), so that
                               // the waits for them run into their bound
};

// ------------------------------------------------------------------------------------------------
// PTX wrappers
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Per-CTA control block in shared memory.
struct Ctl {
  int abort;                       // set by the first wait of this CTA that gives up
  int p2_tiles;                    // pass-2 tiles whose copies have been issued
  unsigned long long limit_ns;     // bound of every wait
  const int* grid_status;          // the device status word (may be null): non-zero once any CTA gave up
};
// Called from the slow part of every wait loop: has this CTA, or any other, given up, or has this
// wait lasted longer than the bound?  (Then it marks the CTA as aborted.)
__device__ __forceinline__ bool give_up(volatile Ctl* ctl, unsigned long long t0) {
  if (ctl->abort) return true;
  const int* gs = ctl->grid_status;
  if (gs != nullptr && *reinterpret_cast<const volatile int*>(gs) != 0) { ctl->abort = 1; return true; }
  if (globaltimer_ns() - t0 > ctl->limit_ns) { ctl->abort = 1; return true; }
  return false;
}
// Bounded wait.  Returns false when the CTA has given up (see give_up).  The retry loop is for
// the rare case.
__device__ __forceinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile Ctl* ctl) {
  const unsigned long long t0 = globaltimer_ns();
  uint32_t spins = 0;
  while (!mbar_try(bar, parity)) {
    if ((++spins & 1023u) == 0 && give_up(ctl, t0)) return false;
  }
  return true;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile Ctl* ctl) {
  if (mbar_try(bar, parity)) return true;
  return mbar_wait_slow(bar, parity, ctl);
}
// The same by a whole warp, with one answer for all lanes: a role that runs warp-uniformly keeps its ring
// positions, descriptors and barrier addresses in uniform registers, which is where tcgen05.mma, tcgen05.commit and
// the TMA copies take them from.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile Ctl* ctl) {
  if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
  return __all_sync(0xffffffffu, mbar_wait_slow(bar, parity, ctl));
}
// Pass 1 may copy tile `pos` once fewer than `lead` tiles lie between it and pass 2 (bounded; one answer per warp).
__device__ __forceinline__ bool wait_lead_slow(int pos, int lead, volatile Ctl* ctl) {
  const unsigned long long t0 = globaltimer_ns();
  uint32_t spins = 0;
  while (pos - ctl->p2_tiles >= lead) {
    __nanosleep(20);
    if ((++spins & 1023u) == 0 && give_up(ctl, t0)) return false;
  }
  return true;
}
__device__ __forceinline__ bool wait_lead(int pos, int lead, volatile Ctl* ctl) {
  if (__all_sync(0xffffffffu, pos - ctl->p2_tiles < lead)) return true;
  return __all_sync(0xffffffffu, wait_lead_slow(pos, lead, ctl));
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
// The same for a copy or an MMA that has been issued and therefore completes whatever the rest
// of the grid does: only the time bound ends this wait early, not the abort flag.
__device__ __forceinline__ bool mbar_wait_issued(uint32_t bar, uint32_t parity, volatile Ctl* ctl) {
  const unsigned long long t0 = globaltimer_ns();
  uint32_t spins = 0;
  while (!mbar_try(bar, parity)) {
    if ((++spins & 1023u) == 0 && globaltimer_ns() - t0 > ctl->limit_ns) { ctl->abort = 1; return false; }
  }
  return true;
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c0, int c1, int c2, int c3, unsigned long long policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(policy) : "memory");
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c0, int c1, int c2, int c3, int c4, unsigned long long policy) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%3, %4, %5, %6, %7}], [%2], %8;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "l"(policy) : "memory");
}
__device__ __forceinline__ void tma_prefetch_5d(const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4) {
  asm volatile("cp.async.bulk.prefetch.tensor.5d.L2.global.tile [%0, {%1, %2, %3, %4, %5}];"
               ::"l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// The same with A in TMEM (lane = row, 16 elements of a row in 8 columns).
__device__ __forceinline__ void tc_mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// One K step (128 rows x 32 bytes) of a K-major operand tile from shared memory to 8 TMEM columns.
__device__ __forceinline__ void tc_cp_256b(uint32_t d_tmem, uint64_t desc) {
  asm volatile("tcgen05.cp.cta_group::1.128x256b [%0], %1;" ::"r"(d_tmem), "l"(desc) : "memory");
}
// 32 consecutive accumulator columns of this thread's TMEM lane; the caller waits for the load.
__device__ __forceinline__ void tc_ld32_nowait(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
// Wait for a TMEM load, tied to the registers it filled: the compiler may not use them before it.
__device__ __forceinline__ void tc_wait_ld(uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
        "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
        "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
        "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
      :: "memory");
}
// The same for 16 columns.
__device__ __forceinline__ void tc_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc_wait_ld(uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
        "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
      :: "memory");
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Two fp32 lanes in one 64-bit register (Blackwell packed fp32 arithmetic).
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ unsigned long long pack2u(uint32_t a, uint32_t b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ void unpack2(unsigned long long p, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// The registers per thread of the calling warpgroup.
template <int N> __device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void regs_set() {
  if constexpr (N > kRegsStart) regs_inc<N>(); else if constexpr (N < kRegsStart) regs_dec<N>();
}
__device__ __forceinline__ void named_bar(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// (release: what this thread wrote before -- the run's record of the row -- is visible to whoever
// acquires a value of the word that includes this addition)
__device__ __forceinline__ void red_add_release_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void red_add_relaxed_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void red_or_relaxed_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.or.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float lg2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows 128 B apart,
// 8-row groups 1024 B apart; `addr` may be advanced by 32 B per 16-element K step.
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3ffffu) >> 4);        // start address
  d |= (uint64_t)1 << 16;                          // leading byte offset (unused with swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset
  d |= (uint64_t)1 << 46;                          // descriptor version (sm_100)
  d |= (uint64_t)2 << 61;                          // SWIZZLE_128B
  return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t umma_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
}

// (reference, sum) pairs of the same row: fold (m, l) into (M, Ls).  Exponents are base 2.
__device__ __forceinline__ void combine(float& M, float& Ls, float m, float l) {
  const float Mn = fmaxf(M, m);
  if (Mn > -INFINITY) Ls = Ls * ex2(M - Mn) + l * ex2(m - Mn);
  M = Mn;
}

// ------------------------------------------------------------------------------------------------
// The runs of a CTA.  A run is RT consecutive tiles of one unit (the last run of a unit may be
// shorter); run k of the CTA is the global run blockIdx.x + k * grid.  The cursor moves from run to run
// by additions only (the increments come from the host): a division would queue behind the
// exponentials in the special-function pipe.
// ------------------------------------------------------------------------------------------------
struct RunCursor {
  int j;            // run inside the work unit
  int l, b, h, q;   // the work unit's layer, sequence, KV head, and which of the KV head's work units it is
  __device__ __forceinline__ void init(const FastParams& P) {
    const int u = (int)(blockIdx.x / (unsigned int)P.RPU);
    j = (int)(blockIdx.x - (unsigned int)u * (unsigned int)P.RPU);
    const int uh = u / P.QP;
    q = u - uh * P.QP;
    const int lb = uh / P.Hkv;
    h = uh - lb * P.Hkv;
    l = lb / P.Bt;
    b = lb - l * P.Bt;
  }
  // row tiles of this work unit (kRT, but for a KV head's last one)
  template <int kRT>
  __device__ __forceinline__ int row_tiles(const FastParams& P) const { return kRT == 1 ? 1 : min(kRT, P.QT - q * kRT); }
  // window rows of its row tile rt (whole query heads; the last tile of a KV head may be short)
  // (kLong: the instantiation that also handles windows longer than 128 rows, CH > 1; everywhere else
  // that case is compiled out of the hot loops)
  template <bool kLong, int kRT>
  __device__ __forceinline__ int rows(const FastParams& P, int rt) const {
    const int qt = q * kRT + rt;
    return (!kLong || P.CH == 1) ? min(P.HPT, P.G - qt * P.HPT) * P.w : min(kRows, P.w - (qt % P.CH) * kRows);
  }
  // first window row of the row tile inside its query head, and the tile's first query head in the group
  template <bool kLong, int kRT>
  __device__ __forceinline__ int row0(const FastParams& P, int rt) const {
    return (!kLong || P.CH == 1) ? 0 : ((q * kRT + rt) % P.CH) * kRows;
  }
  template <bool kLong, int kRT>
  __device__ __forceinline__ int head0(const FastParams& P, int rt) const {
    return (!kLong || P.CH == 1) ? (q * kRT + rt) * P.HPT : (q * kRT + rt) / P.CH;
  }
  // index of the (layer, sequence, KV head), and of the unit (layer, sequence, KV head, row tile)
  __device__ __forceinline__ int kv_unit(const FastParams& P) const { return (l * P.Bt + b) * P.Hkv + h; }
  template <int kRT>
  __device__ __forceinline__ int unit(const FastParams& P, int rt) const { return kv_unit(P) * P.QT + q * kRT + rt; }
  __device__ __forceinline__ int tiles(const FastParams& P) const { return min(P.RT, P.NT - j * P.RT); }
  __device__ __forceinline__ int first_token(const FastParams& P) const { return j * P.RT * kTile; }
  __device__ __forceinline__ void next(const FastParams& P) {
    j += P.step_j;
    int c = 0;
    if (j >= P.RPU) { j -= P.RPU; c = 1; }
    q += P.step_q + c; c = 0;
    if (q >= P.QP) { q -= P.QP; c = 1; }
    h += P.step_h + c; c = 0;
    if (h >= P.Hkv) { h -= P.Hkv; c = 1; }
    b += P.step_b + c; c = 0;
    if (b >= P.Bt) { b -= P.Bt; c = 1; }
    l += P.step_l + c;
  }
};

// A ring position with its mbarrier phase bit.
struct Ring {
  int i, phase;
  __device__ __forceinline__ void next(int n) { if (++i == n) { i = 0; phase ^= 1; } }
};

// K stages and Q slots per pass: what 227 KB hold, and pass 1, whose rows come from HBM, gets the odd stage.  (With two
// and two stages and another Q slot for either pass, or with two and three, the kernel takes the same time within 1 %;
// with three and one it is 5 % slower.)
template <int K1, int K2, int Q1, int Q2>
struct RingSizes {
  static constexpr int kK1 = K1, kK2 = K2, kQ1 = Q1, kQ2 = Q2;
};
template <int D, int kRT> struct Rings;
template <> struct Rings<128, 1> : RingSizes<3, 2, 1, 1> {};
template <> struct Rings<64, 1> : RingSizes<5, 5, 2, 2> {};
template <> struct Rings<128, 2> : RingSizes<2, 2, 1, 2> {};
template <> struct Rings<64, 2> : RingSizes<4, 4, 2, 4> {};

template <int D, int kRT>
struct SmemLayout : Rings<D, kRT> {
  using R = Rings<D, kRT>;
  static constexpr int kHalves = D / 64;
  static constexpr int kTileBytes = kTile * D * 2;
  static constexpr int kStages = R::kK1 + R::kK2, kSlots = R::kQ1 + R::kQ2;
  static constexpr int kQ = 0;                                 // Q slots, pass 1's first
  static constexpr int kK = kSlots * kTileBytes;               // K stages, pass 1's first
  static constexpr int kMisc = kK + kStages * kTileBytes;
  static constexpr int kBarKFull = kMisc;                      // kStages x 8
  static constexpr int kBarKEmpty = kBarKFull + 8 * kStages;
  static constexpr int kBarTFull = kBarKEmpty + 8 * kStages;   // 4 x 8
  static constexpr int kBarTEmpty = kBarTFull + 32;
  static constexpr int kBarQFull = kBarTEmpty + 32;            // kSlots x 8
  static constexpr int kBarQFree = kBarQFull + 8 * kSlots;
  static constexpr int kBarMmaDone = kBarQFree + 8 * kSlots;   // 2 x 8
  static constexpr int kTmemSlot = kBarMmaDone + 16;           // 4 B (+ padding)
  static constexpr int kCtl = kTmemSlot + 8;                   // Ctl, 24 B
  static constexpr int kNegLse = (kCtl + 24 + 15) / 16 * 16;   // kRT x 128 floats, read as 16-byte vectors:
                                                               // -log-sum-exp of the pass-2 unit's rows
  static constexpr int kStats = kNegLse + kRT * kRows * 4;     // one row tile: 2 x 128 rows x float2: the upper half's statistics
  static constexpr int kTotal = kStats + (kRT == 1 ? 2 * kRows * 8 : 0);
  // TMEM columns: the accumulator of pass 1, the two of pass 2, pass 1's Q (two sets)
  static constexpr int kAcc1 = 0, kAcc2 = kTile, kQt = 3 * kTile;
  static_assert(kQt + 2 * (D / 2) <= 512, "TMEM columns");
  static_assert(kCtl % 8 == 0 && kNegLse % 16 == 0 && kStats % 8 == 0 && kTotal <= 232448, "shared-memory layout");
};

// The pushed statistics of one row (see FastParams::acc).
constexpr int kAccFracBits = 20;                              // the sum counts units of 2^-20
constexpr float kAccLimitLog2 = 20.f;                         // a run's contribution must stay below 2^20
constexpr unsigned long long kAccArrival = 1ull << 56, kAccOverflow = 1ull << 48;
constexpr unsigned long long kAccSumMask = kAccOverflow - 1;

// Bounded poll of a row's pushed statistics until all `runs` runs of the unit have arrived.
__device__ __forceinline__ unsigned long long poll_acc_slow(const unsigned long long* src, unsigned int runs,
                                                         volatile Ctl* ctl) {
  const unsigned long long t0 = globaltimer_ns();
  uint32_t spins = 0;
  unsigned long long v;
  while ((unsigned int)((v = ld_relaxed_u64(src)) >> 56) != runs) {
    __nanosleep(100);
    if ((++spins & 255u) == 0 && give_up(ctl, t0)) break;
  }
  return v;
}

// Pass 1: a run's sum of one row, 2^(logit - M) over its tokens = Ls.  The short way: rescaled to the row's fixed
// reference and added to the row's 64-bit word (integer addition: the total does not depend on the order).
__device__ __forceinline__ void send_sum(const FastParams& P, int unit, int run, int row, float row_ref, float M, float Ls) {
  unsigned long long* word = P.acc + (long long)unit * kRows + row;
  const float lv = lg2(Ls) + (M - row_ref);                     // log2 of the contribution
  if (!(Ls > 0.f)) {
    red_add_relaxed_u64(word, kAccArrival);
  } else if (lv < kAccLimitLog2) {
    red_add_relaxed_u64(word, kAccArrival + __float2ull_rn(ex2(lv + (float)kAccFracBits)));
  } else {
    // it does not fit: the run's record and its bit in the row's bitmap, then the arrival with
    // release semantics, so that both are visible to whoever acquires the complete word
    P.partial[((long long)unit * P.RPU + run) * kRows + row] = make_float2(M, Ls);
    red_or_relaxed_u64(P.ovf + ((long long)unit * kRows + row) * 4 + (run >> 6), 1ull << (run & 63));
    red_add_release_u64(word, kAccArrival + kAccOverflow);
  }
}

// ------------------------------------------------------------------------------------------------
// Cold paths: tiles that touch the causal boundary or the end of the context, and
// the aggregator variants other than the paper's defaults.
// ------------------------------------------------------------------------------------------------

// Pass 1, 64 columns (tokens c_first ..) of this thread's query row, with masking: the row's
// (reference, sum) follows the running maximum.  Reads the accumulator itself.
__device__ __forceinline__ void p1_masked_half(uint32_t taddr, long long c_first, long long row_vis, float sl2e,
                                            float* mref_io, float* lsum_io) {
  float mref = *mref_io, lsum = *lsum_io;
#pragma unroll 1
  for (int part = 0; part < 2; ++part) {
    uint32_t r[32];
    tc_ld32_nowait(taddr + part * 32, r);
    tc_wait_ld(r);
    float v[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      v[i] = __uint_as_float(r[i]);
      if (c_first + part * 32 + i > row_vis) v[i] = -INFINITY;
    }
    float x0 = v[0], x1 = v[1];
#pragma unroll
    for (int i = 2; i < 32; i += 2) { x0 = max3(x0, v[i], v[i + 1]); }
    const float m_new = fmaxf(mref, fmaxf(x0, x1) * sl2e);
    if (m_new > -INFINITY) {
      float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        a0 += ex2(fmaf(v[i + 0], sl2e, -m_new));
        a1 += ex2(fmaf(v[i + 1], sl2e, -m_new));
        a2 += ex2(fmaf(v[i + 2], sl2e, -m_new));
        a3 += ex2(fmaf(v[i + 3], sl2e, -m_new));
      }
      lsum = lsum * ex2(mref - m_new) + ((a0 + a1) + (a2 + a3));
      mref = m_new;
    }
  }
  *mref_io = mref;
  *lsum_io = lsum;
}

// Pass 2, one token (this thread's TMEM lane) against all query rows, any aggregator, with
// masking.  Returns the group aggregate before the division of the mean.  W is the window length
// where it is one of the specialised powers of two, 0 where it is only known at run time (`w`).
template <int W, bool kTaskMean>
__device__ __forceinline__ float p2_generic_tile(uint32_t taddr, const float* neg_lse, int n_chunks, int R, float sl2e,
                                              bool full, long long m_min, int agg_group, int w) {
  float gacc = (agg_group == KVC_AGG_MAX) ? -INFINITY : 0.f;
  float hacc = kTaskMean ? 0.f : -INFINITY;
  int m = 0;                                                             // row inside its query head (W == 0)
#pragma unroll 1
  for (int j = 0; j < n_chunks; ++j) {
    uint32_t r[32];
    tc_ld32_nowait(taddr + j * 32, r);
    tc_wait_ld(r);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const int col = j * 32 + i;
      if (W == 0 && i > 0 && i % 8 == 0 && col >= R) break;              // (one row per head and few heads: most columns are nobody's)
      float xi = fmaf(__uint_as_float(r[i]), sl2e, neg_lse[col]);       // log2 of the attention weight
      bool head_done;
      if (W > 0) {
        constexpr int Wd = W > 0 ? W : 1;
        if (!full && (col % Wd) < m_min) xi = -INFINITY;
        head_done = (col + 1) % Wd == 0;
      } else {
        if (!full && m < m_min) xi = -INFINITY;
        head_done = ++m == w;
        if (head_done) m = 0;
      }
      if (kTaskMean) hacc += ex2(xi); else hacc = fmaxf(hacc, xi);
      if (head_done) {                                                   // a query head is complete
        if (col < R) {
          const float s_task = kTaskMean ? hacc / (float)w : ex2(hacc);
          gacc = (agg_group == KVC_AGG_MAX) ? fmaxf(gacc, s_task) : gacc + s_task;
        }
        hacc = kTaskMean ? 0.f : -INFINITY;
      }
    }
  }
  return gacc;
}

// kC consecutive accumulator columns of this thread's TMEM lane, loaded.
template <int kC>
__device__ __forceinline__ void tc_ld_cols(uint32_t taddr, uint32_t (&r)[kC]) {
  static_assert(kC == 8 || kC == 16 || kC == 32, "columns");
  if constexpr (kC == 32) {
    tc_ld32_nowait(taddr, r);
    tc_wait_ld(r);
  } else if constexpr (kC == 16) {
    tc_ld16_nowait(taddr, r);
    tc_wait_ld(r);
  } else {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr) : "memory");
  }
}

// Pass 2, one token, max over a window of w <= 128 rows that is no power of two, on a tile no mask touches.  A query
// head's columns are taken kC at a time (kC <= w, the largest of 8, 16, 32), the last kC ending with the head and
// overlapping the ones before: a maximum does not mind.  (Column by column with a run-time count of the rows, as the
// masked tiles still are, the scoring of the 8B shape at 16K takes 886 us with w = 24, 2071 with 49 and 4097 with 100; so it
// takes 386, 649 and 1240.)  Returns the group aggregate before the division of the mean.
template <int kC>
__device__ __forceinline__ float p2_odd_tile(uint32_t taddr, const float* neg_lse, int R, int w, float sl2e, bool gmax) {
  float gacc = gmax ? -INFINITY : 0.f;
#pragma unroll 1
  for (int h0 = 0; h0 < R; h0 += w) {
    float hacc = -INFINITY;
#pragma unroll 1
    for (int c = 0; c < w; c += kC) {
      const int col = h0 + min(c, w - kC);
      uint32_t r[kC];
      tc_ld_cols<kC>(taddr + col, r);
#pragma unroll
      for (int i = 0; i < kC; i += 2)
        hacc = max3(hacc, fmaf(__uint_as_float(r[i]), sl2e, neg_lse[col + i]),
                    fmaf(__uint_as_float(r[i + 1]), sl2e, neg_lse[col + i + 1]));
    }
    const float s_task = ex2(hacc);
    gacc = gmax ? fmaxf(gacc, s_task) : gacc + s_task;
  }
  return gacc;
}

// The same out of line, for windows of 9 to 15 rows: where pass 2 bounds the kernel they are 1 to 3 % faster so (20000 tokens, heads of 64:
// at worst 1.05 of the time before all of these went into the kernel's body, 1.025 called), longer windows 1 to 2 % slower.
template <int kC>
__device__ __noinline__ float p2_odd_tile_called(uint32_t taddr, const float* neg_lse, int R, int w, float sl2e, bool gmax) {
  return p2_odd_tile<kC>(taddr, neg_lse, R, w, sl2e, gmax);
}

// Pass 2, one token against the R rows of one query head that this row tile holds (windows longer
// than 128 rows), with masking: rows below m_min do not see the token.  Returns the tile's part of
// Eq. 14 for the token: the largest attention weight, or the sum of the weights, over these rows.
template <bool kTaskMean>
__device__ __forceinline__ float p2_long_tile(uint32_t taddr, const float* neg_lse, int n_chunks, int R, float sl2e,
                                           bool full, long long m_min) {
  float hacc = kTaskMean ? 0.f : -INFINITY;
#pragma unroll 1
  for (int j = 0; j < n_chunks; ++j) {
    uint32_t r[32];
    tc_ld32_nowait(taddr + j * 32, r);
    tc_wait_ld(r);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const int col = j * 32 + i;
      float xi = fmaf(__uint_as_float(r[i]), sl2e, neg_lse[col]);       // log2 of the attention weight
      if (col >= R || (!full && col < m_min)) xi = -INFINITY;
      if (kTaskMean) hacc += ex2(xi); else hacc = fmaxf(hacc, xi);
    }
  }
  return kTaskMean ? hacc : ex2(hacc);
}

// ------------------------------------------------------------------------------------------------
// Value norms (App. A.1.3) on CTAs of their own in the scoring launch: they wait for HBM, the scoring CTAs for their SMs, so the
// two overlap where a kernel before the scoring had to be waited for (see norm_share).  A lane's pieces of the rows go through
// shared memory, kNormStages blocks of rows ahead: 192 KB in flight per SM (two blocks in registers reach half of the rate: the
// loads of both are waited for together).
// ------------------------------------------------------------------------------------------------
constexpr int kNormStages = 3;
template <int D>
__device__ __forceinline__ void value_norm_cta(const FastParams& P, uint32_t sbase) {
  constexpr int kLpr = D / 8, kGroups = 32 / kLpr, kBlock = kNormBlock<kLpr>, kWarps = kFastThreads / 32;
  static_assert(kNormStages * kNormRows * kFastThreads * 16 <= 14 * 16384, "shared memory");
  unsigned long long policy;                               // (V goes through L2 once; K has to stay there)
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  const int lane = threadIdx.x & 31, sub = lane & (kLpr - 1), grp = lane / kLpr;
  const int segs = P.L * P.Bt * P.Hkv, per_seg = (int)((P.N + kBlock - 1) / kBlock);
  const int stride = P.norm_ctas * kWarps, step_seg = stride / per_seg, step_blk = stride % per_seg;
  const int id = (int)(blockIdx.x - P.grid) * kWarps + (int)(threadIdx.x >> 5);
  struct At {
    int seg, blk;
    __device__ __forceinline__ void next(int step_seg, int step_blk, int per_seg) {
      blk += step_blk;
      seg += step_seg;
      if (blk >= per_seg) { blk -= per_seg; ++seg; }
    }
  } ahead = {id / per_seg, id % per_seg}, at = ahead;
  const uint32_t mine = sbase + threadIdx.x * 16;          // piece u of stage s: + (s * kNormRows + u) * kFastThreads * 16
  auto fetch = [&](int stage) {
    if (ahead.seg < segs) {
      const int h = ahead.seg % P.Hkv, lb = ahead.seg / P.Hkv, b = lb % P.Bt, l = lb / P.Bt;
      const __nv_bfloat16* base = reinterpret_cast<const __nv_bfloat16*>(P.v.p[l]) + b * P.vs0 + h * P.vs1 + sub * 8;
      const int first = ahead.blk * kBlock + grp, last = (int)P.N - 1;     // (N < 2^30)
#pragma unroll
      for (int u = 0; u < kNormRows; ++u) {
        const __nv_bfloat16* src = base + min(first + u * kGroups, last) * P.vs2;
        asm volatile("cp.async.cg.shared.global.L2::cache_hint.L2::256B [%0], [%1], 16, %2;"
                     ::"r"(mine + (uint32_t)(stage * kNormRows + u) * (kFastThreads * 16)), "l"(src), "l"(policy) : "memory");
      }
      ahead.next(step_seg, step_blk, per_seg);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");   // (empty behind the end: the count of groups stays that of the stages)
  };
#pragma unroll
  for (int s = 0; s < kNormStages; ++s) fetch(s);
  for (int stage = 0; at.seg < segs; at.next(step_seg, step_blk, per_seg)) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kNormStages - 1) : "memory");
    uint4 w[kNormRows];                                    // (a lane reads back what it copied itself)
#pragma unroll
    for (int u = 0; u < kNormRows; ++u)
      asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[u].x), "=r"(w[u].y), "=r"(w[u].z), "=r"(w[u].w)
                   : "r"(mine + (uint32_t)(stage * kNormRows + u) * (kFastThreads * 16)) : "memory");
    norm_store<__nv_bfloat16, kLpr>(w, P.vnorm + (long long)at.seg * P.N, (long long)at.blk * kBlock, P.N);
    fetch(stage);
    if (++stage == kNormStages) stage = 0;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// ------------------------------------------------------------------------------------------------
// The kernel
// ------------------------------------------------------------------------------------------------
template <int D, int W, bool kTaskMean, int kRT, bool kKeep>
__device__ __forceinline__ void score_cta(const FastParams& P, uint8_t* smem) {
  using SL = SmemLayout<D, kRT>;
  const uint32_t sbase = smem_u32(smem);
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  volatile Ctl* ctl = reinterpret_cast<volatile Ctl*>(smem + SL::kCtl);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + SL::kTmemSlot);

  auto bar_kfull = [&](int s) { return sbase + SL::kBarKFull + 8 * s; };
  auto bar_kempty = [&](int s) { return sbase + SL::kBarKEmpty + 8 * s; };
  auto bar_tfull = [&](int b) { return sbase + SL::kBarTFull + 8 * b; };
  auto bar_tempty = [&](int b) { return sbase + SL::kBarTEmpty + 8 * b; };
  auto bar_qfull = [&](int q) { return sbase + SL::kBarQFull + 8 * q; };
  auto bar_qfree = [&](int q) { return sbase + SL::kBarQFree + 8 * q; };
  auto bar_mma_done = [&](int p) { return sbase + SL::kBarMmaDone + 8 * p; };

  const bool aligned = (sbase & 1023u) == 0;     // the swizzled tiles need a 1024-byte aligned base
  if (threadIdx.x == 0) {
    for (int s = 0; s < SL::kStages; ++s) { mbar_init(bar_kfull(s), 1); mbar_init(bar_kempty(s), 1); }
    // the accumulators of pass 1 are read by eight warps (two column halves), those of pass 2 by four
    for (int b = 0; b < 3; ++b) { mbar_init(bar_tfull(b), 1); mbar_init(bar_tempty(b), b == 0 && kRT == 1 ? 8 : 4); }
    if (kRT == 2) mbar_init(bar_tfull(3), 1);
    for (int q = 0; q < SL::kSlots; ++q) { mbar_init(bar_qfull(q), 1); mbar_init(bar_qfree(q), 1); }
    mbar_init(bar_mma_done(0), 1); mbar_init(bar_mma_done(1), 1);
    ctl->abort = 0;
    ctl->p2_tiles = 0;
    ctl->limit_ns = P.wait_limit_ns;
    ctl->grid_status = P.status;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dependency_wait();      // everything above overlapped the end of the kernel before this one

  // this CTA's share of the runs
  int my_runs = (P.total_runs > blockIdx.x) ? (int)((P.total_runs - blockIdx.x + P.grid - 1) / P.grid) : 0;
  if (!aligned) {
    if (threadIdx.x == 0 && P.status) atomicCAS(P.status, 0, (int)KVC_ERR_CUDA);
    my_runs = 0;               // nothing is computed; the teardown below still frees the TMEM columns
  }
  static_assert(!kKeep || (kRT == 1 && W > 0 && !kTaskMean), "pass 2 keeps a run's -log-sum-exps in registers");
  constexpr bool kLong = (W == 0);   // only the run-time window variant has windows longer than 128 rows
  // the whole box arrives (rows outside the tensor as zeros)
  const uint32_t q_bytes = (uint32_t)((!kLong || P.CH == 1) ? P.HPT * P.w : kRows) * D * 2;
  const long long vis_all = min(P.N - 1, P.q_pos0);          // tokens up to here are seen by every row

  static_assert(Regs<kRT>::kSingle + Regs<kRT>::kP2 + 2 * Regs<kRT>::kP1 <= 4 * kRegsStart, "registers");
  if constexpr (kRT == 2 || kKeep) { if (warp < 4) regs_set<Regs<kRT>::kSingle>(); }
  if (kRT == 2 && warp >= 8) {
    if constexpr (kRT == 2) {
    // ============================== pass-1 epilogue, two row tiles =============================
    // A group per row tile, the tiles of the two in turn.  A tile's 128 columns go to registers at once and the accumulator is free.
    regs_set<Regs<kRT>::kP1>();
    const int group = (warp - 8) >> 2;                // which of a work unit's row tiles
    const int quarter = warp & 3;                     // TMEM lane quarter this warp may read
    const int row = quarter * 32 + lane;              // TMEM lane = query row
    const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + SL::kAcc1;
    const int row_m = row % (W > 0 ? W : P.w);        // the row inside its query head (windows of up to 128 rows)
    const unsigned long long scale2 = pack2(P.sl2e, P.sl2e);
    const int bar = group * 3;
    uint32_t n1 = 0;
    bool ok = true;
    const int vis_plain = (int)vis_all - (kTile - 1); // a tile whose first token is at most this has no mask (N < 2^30)
    RunCursor c;
    c.init(P);
    for (int k = 0; k < my_runs; ++k, c.next(P)) {
      if (group >= c.template row_tiles<kRT>(P)) continue;
      const int unit = c.template unit<kRT>(P, group);
      const bool row_used = row < c.template rows<kLong, kRT>(P, group);
      const float row_ref = __ldg(P.ref + (long long)unit * kRows + row);
      float mref[2] = {-INFINITY, -INFINITY}, lsum[2] = {0.f, 0.f};    // per half of the columns: sum over the run so far of 2^(logit - mref)
      // 32 logits against a reference: packed arithmetic, four partial sums
      auto sum_chunk = [&](const uint32_t (&r)[32], const float ref) {
        const unsigned long long neg_ref = pack2(-ref, -ref);
        unsigned long long acc0 = 0ull, acc1 = 0ull;        // +0.0f twice
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const unsigned long long y0 = fma2(pack2u(r[i], r[i + 1]), scale2, neg_ref);
          const unsigned long long y1 = fma2(pack2u(r[i + 2], r[i + 3]), scale2, neg_ref);
          float a, b, c, d;
          unpack2(y0, a, b);
          unpack2(y1, c, d);
          acc0 = add2(acc0, pack2(ex2(a), ex2(b)));
          acc1 = add2(acc1, pack2(ex2(c), ex2(d)));
        }
        float s0, s1, s2, s3;
        unpack2(acc0, s0, s1);
        unpack2(acc1, s2, s3);
        return (s0 + s1) + (s2 + s3);
      };
      auto max_chunk = [&](const uint32_t (&r)[32]) {
        float a = __uint_as_float(r[0]), b = __uint_as_float(r[1]);
#pragma unroll
        for (int i = 2; i < 30; i += 4) {
          a = max3(a, __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
          b = max3(b, __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3]));
        }
        a = max3(a, __uint_as_float(r[30]), __uint_as_float(r[31]));
        return fmaxf(a, b);
      };
      const int nt = c.tiles(P);
      int tok0 = c.first_token(P);
      for (int t = 0; t < nt; ++t, tok0 += kTile) {
        ok = __all_sync(0xffffffffu, ok && mbar_wait(bar_tfull(bar), n1 & 1u, ctl));
        ++n1;
        if (!ok) continue;
        tc_fence_after();
        if (tok0 <= vis_plain) {
          uint32_t r0[32], r1[32], r2[32], r3[32];
          tc_ld32_nowait(taddr, r0);
          tc_ld32_nowait(taddr + 32, r1);
          tc_ld32_nowait(taddr + 64, r2);
          tc_ld32_nowait(taddr + 96, r3);
          tc_wait_ld(r0); tc_wait_ld(r1); tc_wait_ld(r2); tc_wait_ld(r3);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_tempty(0));
          if (mref[0] == -INFINITY) { mref[0] = __uint_as_float(r0[0]) * P.sl2e; mref[1] = __uint_as_float(r2[0]) * P.sl2e; }
          const float top = fmaxf(fmaxf(max_chunk(r0), max_chunk(r1)), fmaxf(max_chunk(r2), max_chunk(r3)));
          if (!__any_sync(0xffffffffu, row_used && !(fmaf(top, P.sl2e, -fminf(mref[0], mref[1])) < 58.5f))) {
            lsum[0] += sum_chunk(r0, mref[0]);
            lsum[0] += sum_chunk(r1, mref[0]);
            lsum[1] += sum_chunk(r2, mref[1]);
            lsum[1] += sum_chunk(r3, mref[1]);
          } else {
            uint32_t copy[128];
#pragma unroll
            for (int i = 0; i < 32; ++i) { copy[i] = r0[i]; copy[32 + i] = r1[i]; copy[64 + i] = r2[i]; copy[96 + i] = r3[i]; }
#pragma unroll 1
            for (int ch = 0; ch < 4; ++ch) {
              float m = ch < 2 ? mref[0] : mref[1], l = ch < 2 ? lsum[0] : lsum[1];
#pragma unroll 1
              for (int attempt = 0; attempt < 8; ++attempt) {
                float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 1
                for (int i = 0; i < 32; i += 4) {
                  const uint32_t* p = copy + ch * 32 + i;
                  s0 += ex2(fmaf(__uint_as_float(p[0]), P.sl2e, -m));
                  s1 += ex2(fmaf(__uint_as_float(p[1]), P.sl2e, -m));
                  s2 += ex2(fmaf(__uint_as_float(p[2]), P.sl2e, -m));
                  s3 += ex2(fmaf(__uint_as_float(p[3]), P.sl2e, -m));
                }
                const float sum = (s0 + s1) + (s2 + s3);
                if (sum < kRescaleLimit) { l += sum; break; }    // (false for inf / NaN as well)
                m += 64.f;
                l *= 5.421010862427522e-20f;                     // 2^-64
              }
              if (ch < 2) { mref[0] = m; lsum[0] = l; } else { mref[1] = m; lsum[1] = l; }
            }
          }
        } else {
          const long long row_vis = min(P.N - 1, P.q_pos0 + ((!kLong || P.CH == 1) ? row_m : c.template row0<kLong, kRT>(P, group) + row));
#pragma unroll 1
          for (int h = 0; h < 2; ++h) {
            float m2 = h == 0 ? mref[0] : mref[1], l2 = h == 0 ? lsum[0] : lsum[1];
            p1_masked_half(taddr + h * 64, (long long)tok0 + h * 64, row_vis, P.sl2e, &m2, &l2);
            if (h == 0) { mref[0] = m2; lsum[0] = l2; } else { mref[1] = m2; lsum[1] = l2; }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_tempty(0));
        }
      }
      if (ok && unit != P.withhold_unit) {
        float M = row_used ? mref[0] : -INFINITY, Ls = row_used ? lsum[0] : 0.f;
        combine(M, Ls, row_used ? mref[1] : -INFINITY, row_used ? lsum[1] : 0.f);
        send_sum(P, unit, c.j, row, row_ref, M, Ls);
      }
    }
    }
  } else if (kRT == 1 && warp >= 8) {
    // ============================== pass-1 epilogue, one row tile ==============================
    if constexpr (kKeep) regs_set<Regs<1>::kP1>();
    const int half = (warp - 8) >> 2;                 // which 64 columns (tokens) of every tile
    const int quarter = warp & 3;                     // TMEM lane quarter this warp may read
    const int row = quarter * 32 + lane;              // TMEM lane = query row
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    float2* const stage = reinterpret_cast<float2*>(smem + SL::kStats) + row;
    const int row_m = row % (W > 0 ? W : P.w);        // the row inside its query head (windows of up to 128 rows)
    const unsigned long long scale2 = pack2(P.sl2e, P.sl2e);

    uint32_t n1 = 0;
    float mref = -INFINITY, lsum = 0.f;               // sum over the run so far of 2^(logit - mref)
    bool ok = true;

    // 32 unmasked logits against the row's current reference: no maximum, packed arithmetic.
    // Any logit of the row will do as a reference; if a chunk's sum leaves the range of fp32
    // the reference is moved up by 64 and the chunk is summed again.
    auto fast_chunk = [&](const uint32_t (&r)[32]) {
      if (mref == -INFINITY) mref = __uint_as_float(r[0]) * P.sl2e;
#pragma unroll 1
      for (int attempt = 0; attempt < 8; ++attempt) {
        const unsigned long long neg_ref = pack2(-mref, -mref);
        unsigned long long acc0 = 0ull, acc1 = 0ull;      // +0.0f twice
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const unsigned long long y0 = fma2(pack2u(r[i], r[i + 1]), scale2, neg_ref);
          const unsigned long long y1 = fma2(pack2u(r[i + 2], r[i + 3]), scale2, neg_ref);
          float a, b, c, d;
          unpack2(y0, a, b);
          unpack2(y1, c, d);
          acc0 = add2(acc0, pack2(ex2(a), ex2(b)));
          acc1 = add2(acc1, pack2(ex2(c), ex2(d)));
        }
        float s0, s1, s2, s3;
        unpack2(acc0, s0, s1);
        unpack2(acc1, s2, s3);
        const float sum = (s0 + s1) + (s2 + s3);
        if (sum < kRescaleLimit) { lsum += sum; break; }   // (false for inf / NaN as well)
        mref += 64.f;
        lsum *= 5.421010862427522e-20f;                    // 2^-64
      }
    };

    // The end of a run: the two halves of every row meet through shared memory (two buffers in turn); the lower
    // half's warps send the run's sum of every row, the upper half's go on.  n: runs before this one.
    auto exchange = [&](const int n, const bool row_used, const float row_ref, const int unit, const int run) {
      const int par = n & 1;
      if (half == 1) {
        if (n >= 2) named_bar(5 + par, 256);              // the buffer has been read
        stage[par * kRows] = make_float2(row_used ? mref : -INFINITY, row_used ? lsum : 0.f);
        named_bar_arrive(3 + par, 256);
      } else {
        named_bar(3 + par, 256);
        const float2 other = stage[par * kRows];
        if (n + 2 < my_runs) named_bar_arrive(5 + par, 256);
        if (ok && unit != P.withhold_unit) {
          float M = row_used ? mref : -INFINITY, Ls = row_used ? lsum : 0.f;
          combine(M, Ls, other.x, other.y);
          send_sum(P, unit, run, row, row_ref, M, Ls);
        }
      }
      mref = -INFINITY; lsum = 0.f;
    };

    const int vis_plain = (int)vis_all - (kTile - 1);     // a tile whose first token is at most this has no mask (N < 2^30)
    RunCursor c;
    c.init(P);
    for (int k = 0; k < my_runs; ++k, c.next(P)) {
      const int unit = c.template unit<1>(P, 0);
      const bool row_used = row < c.template rows<kLong, 1>(P, 0);
      float row_ref = 0.f;                              // the row's reference exponent for the pushed sum: used at the run's end
      if (half == 0) row_ref = __ldg(P.ref + (long long)unit * kRows + row);
      const int nt = c.tiles(P);
      int tok0 = c.first_token(P);                      // first token of the tile
      for (int t = 0; t < nt; ++t, tok0 += kTile) {
        // (the TMEM loads below are warp-wide instructions: the decision has to be the warp's)
        ok = __all_sync(0xffffffffu, ok && mbar_wait(bar_tfull(0), n1 & 1u, ctl));
        ++n1;
        if (ok) {
          tc_fence_after();
          const uint32_t taddr = lane_addr + SL::kAcc1 + half * 64;
          if (tok0 <= vis_plain) {
            uint32_t ra[32], rb[32];
            tc_ld32_nowait(taddr, ra);
            tc_ld32_nowait(taddr + 32, rb);
            tc_wait_ld(ra);
            tc_wait_ld(rb);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_tempty(0));  // the accumulator is in registers now
            if (row_used) { fast_chunk(ra); fast_chunk(rb); }
          } else {
            float m2 = mref, l2 = lsum;                 // (the whole warp takes part in the TMEM loads)
            const long long row_vis = min(P.N - 1, P.q_pos0 + ((!kLong || P.CH == 1) ? row_m : c.template row0<kLong, 1>(P, 0) + row));   // last key this row sees
            p1_masked_half(taddr, (long long)tok0 + half * 64, row_vis, P.sl2e, &m2, &l2);
            if (row_used) { mref = m2; lsum = l2; }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_tempty(0));
          }
        }
      }
      exchange(k, row_used, row_ref, unit, c.j);
    }
  } else if (warp >= 4 && warp < 8) {
    // ============================== pass-2 epilogue ============================================
    if constexpr (kRT == 2 || kKeep) regs_set<Regs<kRT>::kP2>();
    const int quarter = warp & 3;
    const int trow = quarter * 32 + lane;             // TMEM lane = token inside the tile; also 0..127 in the group
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    float* neg_lse_of = reinterpret_cast<float*>(smem + SL::kNegLse);
    const unsigned long long scale2 = pack2(P.sl2e, P.sl2e);
    int n2 = 0;
    bool ok = true;
    // per-tile work is kept to a minimum here: this group's instruction stream is what the kernel waits for
    const bool gmax = P.agg_group == KVC_AGG_MAX;
    const float inv_g = (P.QT == 1 && !gmax) ? 1.f / (float)P.G : 1.f;   // one row tile: the mean of Eq. 15 is finished here
    const int vis_all_i = (int)vis_all;                // (N < 2^30)
    const int n_ctx = (int)P.N;
    RunCursor cu;
    cu.init(P);
    unsigned long long early_word[kRT];               // a coming run's pushed words and references, fetched ahead
    float early_ref[kRT];
    auto fetch_early = [&]() {
#pragma unroll
      for (int rt = 0; rt < kRT; ++rt) {
        early_word[rt] = 0ull; early_ref[rt] = 0.f;
        if (kRT == 1 || rt < cu.template row_tiles<kRT>(P)) {
          const long long at = (long long)cu.template unit<kRT>(P, rt) * kRows + trow;
          early_word[rt] = ld_relaxed_u64(P.acc + at);
          early_ref[rt] = __ldg(P.ref + at);
        }
      }
    };
    if (my_runs > 0) fetch_early();
    for (int k = 0; k < my_runs; ++k) {
      const int nrt = cu.template row_tiles<kRT>(P);
      int rows_of[kRT], row0_of[kRT];
      float* score_row_of[kRT];                        // where the units' scores (or partial aggregates) go
#pragma unroll
      for (int rt = 0; rt < kRT; ++rt) {
        const int r1 = kRT == 1 ? 0 : min(rt, nrt - 1);
        rows_of[rt] = cu.template rows<kLong, kRT>(P, r1);
        row0_of[rt] = cu.template row0<kLong, kRT>(P, r1);
        score_row_of[rt] = P.scores + ((long long)(cu.q * kRT + r1) * ((long long)P.L * P.Bt * P.Hkv) + cu.kv_unit(P)) * P.N;
      }
      const int nt = cu.tiles(P);
      int tok0 = cu.first_token(P);                    // first token of the tile
      ulonglong2 nl_regs[kKeep ? 32 : 1];           // one row tile: its rows' -log-sum-exps
      {
        // a new run: its units' log-sum-exps.  The short way: the row's pushed word, complete once
        // every run of the unit has arrived (fetched a tile or two ago; polled if it was not
        // complete then).  If a run's sum did not fit, the runs' records decide.
        float lse_of[kRT];
#pragma unroll
        for (int rt = 0; rt < kRT; ++rt) {
          float lse = 0.f;
          if (ok && (kRT == 1 || rt < nrt) && trow < rows_of[rt]) {
            const int unit = cu.template unit<kRT>(P, rt);
            bool pushed = false;
            {
              unsigned long long word = early_word[rt];
              if ((unsigned int)(word >> 56) != (unsigned int)P.RPU)
                word = poll_acc_slow(P.acc + (long long)unit * kRows + trow, (unsigned int)P.RPU, ctl);
              const unsigned long long sum = word & kAccSumMask;
              if (((word >> 48) & 0xffull) == 0 && sum != 0) {
                lse = early_ref[rt] + lg2((float)sum) - (float)kAccFracBits;
                pushed = true;
              }
            }
            if (!pushed) {
              // the long way: all runs have arrived (the count in the word); those whose sum did not fit
              // wrote a record and set their bit before their release.  Fold them, in run order (the same
              // order for every reader), into the fixed-point sum of the others.
              asm volatile("fence.acq_rel.gpu;" ::: "memory");
              const unsigned long long word = ld_relaxed_u64(P.acc + (long long)unit * kRows + trow);
              const unsigned long long sum = word & kAccSumMask;
              float M = -INFINITY, Ls = 0.f;
              if (sum != 0) { M = early_ref[rt]; Ls = (float)sum * 9.5367431640625e-07f; }       // 2^-20
              const float2* rec = P.partial + (long long)unit * P.RPU * kRows + trow;
              const unsigned long long* bits_of = P.ovf + ((long long)unit * kRows + trow) * 4;
#pragma unroll 1
              for (int wi = 0; wi < 4; ++wi) {
                unsigned long long bits = __ldcg(bits_of + wi);
                while (bits) {
                  const int j = wi * 64 + __ffsll((long long)bits) - 1;
                  bits &= bits - 1;
                  const float2 v = __ldcg(rec + (long long)j * kRows);
                  combine(M, Ls, v.x, v.y);
                }
              }
              lse = M + log2f(Ls);
            }
          }
          lse_of[rt] = lse;
        }
        named_bar(1, 128);                             // everyone is done with the previous unit's values
#pragma unroll
        for (int rt = 0; rt < kRT; ++rt)               // (a row that is not there never wins a maximum)
          neg_lse_of[rt * kRows + trow] = (trow < rows_of[rt]) ? -lse_of[rt] : -INFINITY;
        named_bar(1, 128);
        if constexpr (kKeep) {
          const ulonglong2* l2 = reinterpret_cast<const ulonglong2*>(neg_lse_of);
#pragma unroll
          for (int i = 0; i < 32; ++i) nl_regs[i] = l2[i];
        }
        ok = !__any_sync(0xffffffffu, ctl->abort != 0) && ok;
      }
      cu.next(P);
      for (int t = 0; t < nt; ++t, tok0 += kTile) {
      // the next run's words and references: in flight while the rest of this run (two accumulators) is computed
      if (t == max(nt - 2 / kRT, 0) && k + 1 < my_runs) fetch_early();
      for (int rt = 0; rt < nrt; ++rt) {
      const int rows_u = kRT == 1 || rt == 0 ? rows_of[0] : rows_of[kRT - 1];
      const int n_chunks = (rows_u + 31) / 32;
      const float* const neg_lse = neg_lse_of + rt * kRows;
      const int buf = 1 + (n2 & 1);
      const uint32_t tmem_col = SL::kAcc2 + (uint32_t)(n2 & 1) * kTile;
      // (the TMEM loads below are warp-wide instructions: the decision has to be the warp's)
      ok = __all_sync(0xffffffffu, ok && mbar_wait(bar_tfull(buf), (uint32_t)((n2 >> 1) & 1), ctl));
      ++n2;
      if (!ok) continue;
      tc_fence_after();
      const int c = tok0 + trow;                                     // this thread's token
      const bool full = tok0 + kTile - 1 <= vis_all_i;
      float gacc;
      if (!kTaskMean && full && (W > 0 || P.CH > 1)) {
        // the paper's default (max over the window) on a tile no mask touches: every 32-column chunk belongs to
        // one query head, or holds whole query heads (W = 8, 16); a row tile of a window longer than 128 rows
        // belongs to one head throughout (a window of 500 rows at 4K: 1849 -> 1036 us for the scoring against the
        // column-by-column loop of the masked tiles)
        gacc = gmax ? -INFINITY : 0.f;
        float hacc = -INFINITY;
        const uint32_t acc = lane_addr + tmem_col;
        // 16 columns: the largest log2 of their weights goes to hacc; with W = 16 a head ends here
        auto part = [&](const uint32_t* r, const ulonglong2* nl, const int col) {
          float x[16];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const unsigned long long y0 = fma2(pack2u(r[4 * i], r[4 * i + 1]), scale2, nl[i].x);
            const unsigned long long y1 = fma2(pack2u(r[4 * i + 2], r[4 * i + 3]), scale2, nl[i].y);
            unpack2(y0, x[4 * i], x[4 * i + 1]);
            unpack2(y1, x[4 * i + 2], x[4 * i + 3]);
          }
          if (W == 16) {
            float a = fmaxf(x[0], x[1]);
#pragma unroll
            for (int i = 2; i < 16; i += 2) a = max3(a, x[i], x[i + 1]);
            if (col < rows_u) {
              const float s_task = ex2(a);
              gacc = gmax ? fmaxf(gacc, s_task) : gacc + s_task;
            }
          } else {
            float a = max3(x[0], x[1], x[2]), b = max3(x[3], x[4], x[5]);
            a = max3(a, x[6], x[7]); b = max3(b, x[8], x[9]);
            a = max3(a, x[10], x[11]); b = max3(b, x[12], x[13]);
            a = max3(a, x[14], x[15]);
            hacc = max3(hacc, a, b);
          }
        };
        auto head_end = [&](const int j) {                               // behind chunk j of 32 columns
          if (W > 16 && ((j + 1) * 32) % (W > 0 ? W : 1) == 0) {
            const float s_task = ex2(hacc);
            gacc = gmax ? fmaxf(gacc, s_task) : gacc + s_task;
            hacc = -INFINITY;
          }
        };
        auto emptied = [&]() {                                           // the accumulator has been read
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_tempty(buf));
        };
        if constexpr (kKeep) {
          // a chunk of 32 columns is fetched while the one before it is worked on
          uint32_t ra[32], rb[32];
          tc_ld32_nowait(acc, ra);
          auto chunk = [&](const int j, uint32_t (&r)[32], uint32_t (&r_next)[32]) {
            tc_wait_ld(r);
            if (j + 1 < n_chunks) tc_ld32_nowait(acc + j * 32 + 32, r_next); else emptied();
            part(r, nl_regs + 8 * j, j * 32);
            part(r + 16, nl_regs + 8 * j + 4, j * 32 + 16);
            head_end(j);
          };
          chunk(0, ra, rb);
          if (n_chunks > 1) chunk(1, rb, ra);
          if (n_chunks > 2) chunk(2, ra, rb);
          if (n_chunks > 3) chunk(3, rb, ra);
        } else if constexpr (W == 8) {
          // whole chunks, the next one behind the arithmetic: every head ends with an exponential, which half chunks, and the form
          // above (it spills), only put off (heads of 128, 128 rows, 20000 tokens, 6 layers: 84.3 us kept, 85.5 in halves, 81.0 so)
          uint32_t r[32];
          tc_ld32_nowait(acc, r);
#pragma unroll 1
          for (int j = 0; j < n_chunks; ++j) {
            ulonglong2 nl[8];
            const ulonglong2* l2 = reinterpret_cast<const ulonglong2*>(neg_lse + j * 32);
#pragma unroll
            for (int i = 0; i < 8; ++i) nl[i] = l2[i];
            tc_wait_ld(r);
            float x[32];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              unpack2(fma2(pack2u(r[4 * i], r[4 * i + 1]), scale2, nl[i].x), x[4 * i], x[4 * i + 1]);
              unpack2(fma2(pack2u(r[4 * i + 2], r[4 * i + 3]), scale2, nl[i].y), x[4 * i + 2], x[4 * i + 3]);
            }
            if (j + 1 < n_chunks) tc_ld32_nowait(acc + j * 32 + 32, r); else emptied();
#pragma unroll
            for (int h0 = 0; h0 < 32; h0 += 8) {
              float a = fmaxf(x[h0], x[h0 + 1]);
#pragma unroll
              for (int i = 2; i < 8; i += 2) a = max3(a, x[h0 + i], x[h0 + i + 1]);
              if (j * 32 + h0 < rows_u) {
                const float s_task = ex2(a);
                gacc = gmax ? fmaxf(gacc, s_task) : gacc + s_task;
              }
            }
          }
        } else {
          // the same with half chunks, whose -log-sum-exps come from shared memory
          uint32_t ra[16], rb[16];
          ulonglong2 na[4], nb[4];
          auto load_nl = [&](ulonglong2 (&nl)[4], const int col) {
            const ulonglong2* l2 = reinterpret_cast<const ulonglong2*>(neg_lse + col);
#pragma unroll
            for (int i = 0; i < 4; ++i) nl[i] = l2[i];
          };
          tc_ld16_nowait(acc, ra);
          load_nl(na, 0);
#pragma unroll 1
          for (int j = 0; j < n_chunks; ++j) {
            load_nl(nb, j * 32 + 16);
            tc_wait_ld(ra);
            tc_ld16_nowait(acc + j * 32 + 16, rb);
            part(ra, na, j * 32);
            if (j + 1 < n_chunks) load_nl(na, j * 32 + 32);
            tc_wait_ld(rb);
            if (j + 1 < n_chunks) tc_ld16_nowait(acc + j * 32 + 32, ra); else emptied();
            part(rb, nb, j * 32 + 16);
            head_end(j);
          }
        }
        if (W == 0) gacc = ex2(hacc);                                  // the head's maximum over these rows
      } else if (!kTaskMean && W == 0 && full && P.w >= 8) {
        // (row tiles in pairs never come here, yet their kernel with heads of 64 is 15 % slower where ptxas does not see it)
        const auto short_blocks = [&]() {
          if constexpr (kRT == 1) return p2_odd_tile_called<8>(lane_addr + tmem_col, neg_lse, rows_u, P.w, P.sl2e, gmax);
          else return p2_odd_tile<8>(lane_addr + tmem_col, neg_lse, rows_u, P.w, P.sl2e, gmax);
        };
        gacc = P.w >= 32 ? p2_odd_tile<32>(lane_addr + tmem_col, neg_lse, rows_u, P.w, P.sl2e, gmax)
             : P.w >= 16 ? p2_odd_tile<16>(lane_addr + tmem_col, neg_lse, rows_u, P.w, P.sl2e, gmax)
                         : short_blocks();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tempty(buf));
      } else if (W == 0 && P.CH > 1) {
        // a window longer than 128 rows: the tile holds rows row0 .. of one query head and yields
        // that head's partial Eq. 14 (the maximum, or the sum, over these rows)
        gacc = p2_long_tile<kTaskMean>(lane_addr + tmem_col, neg_lse, n_chunks, rows_u, P.sl2e, full,
                                       (long long)c - P.q_pos0 - (kRT == 1 || rt == 0 ? row0_of[0] : row0_of[kRT - 1]));
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tempty(buf));
      } else {
        gacc = p2_generic_tile<W, kTaskMean>(lane_addr + tmem_col, neg_lse, n_chunks, rows_u, P.sl2e, full,
                                             (long long)c - P.q_pos0, P.agg_group, P.w);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tempty(buf));
      }
      // one row tile: the group aggregate itself; several: this tile's part of it
      if (c < n_ctx) (kRT == 1 || rt == 0 ? score_row_of[0] : score_row_of[kRT - 1])[c] = gacc * inv_g;
      }
      }
    }
  } else if (warp == 1 || warp == 2) {
    // ============================== MMA issuers ================================================
    // One warp per pass, the same code: it walks its pass's runs, all lanes together.
    const int pass = warp - 1;
    const int stage0 = pass == 0 ? 0 : SL::kK1, stages = pass == 0 ? SL::kK1 : SL::kK2;
    const int slot0 = pass == 0 ? 0 : SL::kQ1, slots = pass == 0 ? SL::kQ1 : SL::kQ2;
    const int bufs = pass == 0 ? 1 : 2;
    Ring kr = {0, 0}, qr = {0, 0}, tb = {0, 0};        // K stage, Q slot, accumulator
    bool ok = true, issued = false;
    RunCursor c;
    c.init(P);
    int visits = 0;                                    // row tiles begun
    for (int k = 0; k < my_runs && ok; ++k, c.next(P)) {
      const int nt = c.tiles(P), nrt = c.template row_tiles<kRT>(P);
      int slot_of[kRT];
      uint64_t dq_of[kRT];
      uint32_t idesc_of[kRT], q_tmem_of[kRT];
      // a row tile's Q has arrived; for pass 1 it moves on to TMEM
      auto begin_q = [&](const int rt) {
        const int slot = slot0 + qr.i;
        ok = mbar_wait_warp(bar_qfull(slot), (uint32_t)qr.phase, ctl);
        const uint64_t dq = umma_desc(sbase + SL::kQ + slot * SL::kTileBytes);
        qr.next(slots);
        const uint32_t q_tmem = tmem_base + SL::kQt + (uint32_t)(visits & 1) * (D / 2);   // pass 1
        ++visits;
        slot_of[rt] = slot; dq_of[rt] = dq; q_tmem_of[rt] = q_tmem;
        idesc_of[rt] = umma_idesc(pass == 0 ? kTile : (c.template rows<kLong, kRT>(P, rt) + 31) / 32 * 32);
        if (pass == 0 && ok) {
          // Its slot is free again then.  Two sets of columns in turn: PTX runs an MMA behind the copies issued
          // before it (tcgen05.cp -> tcgen05.mma), but promises nothing for a copy issued behind an MMA, and the MMAs of the row
          // tile before may still read their set.  Those of the one before that, which read this set, are complete: an MMA of
          // another row tile has been issued since, and only when the epilogue had emptied the accumulator of their last tile.
          // (One set, and a wait for the last MMAs in front of the copy: 448 rows per token at 128K 4457 -> 4491 us per pass,
          // 500-row windows 1225 -> 1234.)
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
              tc_cp_256b(q_tmem + kk * 8, dq + (uint64_t)(((kk >> 2) * (kTile * 128) + (kk & 3) * 32) >> 4));
            tc_commit(bar_qfree(slot));
          }
          __syncwarp();
          issued = true;
        }
      };
      begin_q(0);
      for (int t = 0; t < nt && ok; ++t) {
        const int st = stage0 + kr.i;
        ok = mbar_wait_warp(bar_kfull(st), (uint32_t)kr.phase, ctl);
        const uint64_t dk = umma_desc(sbase + SL::kK + st * SL::kTileBytes);
        for (int rt = 0; rt < nrt && ok; ++rt) {
          // (the second row tile's Q only now: its TMEM columns are those of the run before until the MMAs above are issued)
          if (kRT == 2 && rt == 1 && t == 0) begin_q(kRT - 1);
          const int buf = pass + tb.i;
          if (ok) ok = mbar_wait_warp(bar_tempty(buf), (uint32_t)(tb.phase ^ 1), ctl);
          if (!ok) break;
          tc_fence_after();
          const bool first = kRT == 1 || rt == 0;
          const uint64_t dq = first ? dq_of[0] : dq_of[kRT - 1];
          const uint32_t q_tmem = first ? q_tmem_of[0] : q_tmem_of[kRT - 1];
          const uint32_t idesc = first ? idesc_of[0] : idesc_of[kRT - 1];
          const uint32_t d_tmem = tmem_base + (uint32_t)buf * kTile;
          if (elect_one()) {
            // pass 1: rows = query rows (A = Q, in TMEM), columns = tokens (B = K); pass 2: A = K, B = Q
            // (the start-address field counts 16-byte units: 64-element half, then 32 B per K step)
            if (pass == 0) {
#pragma unroll
              for (int kk = 0; kk < D / 16; ++kk) {
                const uint64_t off = (uint64_t)(((kk >> 2) * (kTile * 128) + (kk & 3) * 32) >> 4);
                tc_mma_bf16_ts(d_tmem, q_tmem + kk * 8, dk + off, idesc, kk > 0);
              }
            } else {
#pragma unroll
              for (int kk = 0; kk < D / 16; ++kk) {
                const uint64_t off = (uint64_t)(((kk >> 2) * (kTile * 128) + (kk & 3) * 32) >> 4);
                tc_mma_bf16(d_tmem, dk + off, dq + off, idesc, kk > 0);
              }
            }
            if (rt + 1 == nrt) tc_commit(bar_kempty(st));   // the K stage may be refilled once these MMAs are done
            tc_commit(bar_tfull(kRT == 2 && pass == 0 && rt == 1 ? 3 : buf));   // ... and the accumulator is then complete
            if (pass != 0 && t + 1 == nt) tc_commit(bar_qfree(first ? slot_of[0] : slot_of[kRT - 1]));
          }
          __syncwarp();
          issued = true;
          tb.next(bufs);
        }
        kr.next(stages);
      }
    }
    // no MMA may be in flight when the TMEM columns and the shared memory are given back
    if (issued) {
      if (elect_one()) tc_commit(bar_mma_done(pass));
      __syncwarp();
      mbar_wait_issued(bar_mma_done(pass), 0u, ctl);
    }
  } else {
    // ============================== TMA producers =============================================
    // Warp 0 for pass 1, warp 3 for pass 2, the same code.  Pass 1 leaves the rows in L2 for pass 2; pass 2 is
    // their last use.  Pass 1's producer stays at most P.lead tiles ahead of pass 2's.
    const int pass = warp == 0 ? 0 : 1;
    const int stage0 = pass == 0 ? 0 : SL::kK1, stages = pass == 0 ? SL::kK1 : SL::kK2;
    const int slot0 = pass == 0 ? 0 : SL::kQ1, slots = pass == 0 ? SL::kQ1 : SL::kQ2;
    unsigned long long pol_stream, pol_keep;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol_stream));
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_keep));
    const unsigned long long pol_k = pass == 0 ? pol_keep : pol_stream;
    Ring kr = {0, 0}, qr = {0, 0};
    int pos = 0, nq = 0;               // K tiles and Q tiles issued
    bool ok = true;
    RunCursor c, nx;
    c.init(P);
    for (int k = 0; k < my_runs && ok; ++k) {
      nx = c;
      nx.next(P);
      const int nt = c.tiles(P);
      const int ntn = k + 1 < my_runs ? nx.tiles(P) : 0;
      const int tok0 = c.first_token(P);
      for (int t = 0; t < nt; ++t) {
        if (pass == 0) ok = wait_lead(pos, P.lead, ctl);
        const int st = stage0 + kr.i;
        if (ok) ok = mbar_wait_warp(bar_kempty(st), (uint32_t)(kr.phase ^ 1), ctl);
        if (!ok) break;
        if (elect_one()) {
          mbar_expect_tx(bar_kfull(st), SL::kTileBytes);
          // (one copy for the whole tile: the 64-element halves of the rows are a dimension of the map)
          tma_load_5d(sbase + SL::kK + st * SL::kTileBytes, P.k_maps + c.l, bar_kfull(st), 0, tok0 + t * kTile, 0, c.h, c.b,
                      pol_k);
          if (pass == 0) {
            const int ta = t + kPrefetch;
            if (ta < nt) tma_prefetch_5d(P.k_maps + c.l, 0, tok0 + ta * kTile, 0, c.h, c.b);
            else if (ta - nt < ntn) tma_prefetch_5d(P.k_maps + nx.l, 0, nx.first_token(P) + (ta - nt) * kTile, 0, nx.h, nx.b);
          } else {
            ctl->p2_tiles = pos + 1;
          }
        }
        __syncwarp();
        kr.next(stages);
        ++pos;
        if (t == 0) {
          // the run's Q (after its first K tile: with a single slot it has to wait for the MMAs of the run before)
          const int nrt = c.template row_tiles<kRT>(P);
          for (int rt = 0; rt < nrt; ++rt) {
            const int slot = slot0 + qr.i;
            ok = mbar_wait_warp(bar_qfree(slot), (uint32_t)(qr.phase ^ 1), ctl);
            if (!ok) break;
            if (elect_one()) {
              mbar_expect_tx(bar_qfull(slot), q_bytes);
              for (int hf = 0; hf < SL::kHalves; ++hf)
                tma_load_4d(sbase + SL::kQ + slot * SL::kTileBytes + hf * (kTile * 128), P.q_maps + c.l, bar_qfull(slot), hf * 64,
                            c.template row0<kLong, kRT>(P, rt), c.h * P.G + c.template head0<kLong, kRT>(P, rt), c.b, pol_keep);
            }
            __syncwarp();
            qr.next(slots);
            ++nq;
          }
          if (!ok) break;
        }
      }
      c = nx;
    }
    // drain: every issued copy must have landed before the CTA's shared memory is released
    // (an issued copy always completes, so these waits do not take the abort shortcut).
    // The last fill of a stage is complete once its full barrier has left the phase of that fill.
    for (int n = 0; n < min(pos, stages); ++n) {
      // walk the ring backwards from the slot before kr
      int i2 = kr.i - 1 - n, ph = kr.phase;
      if (i2 < 0) { i2 += stages; ph ^= 1; }
      mbar_wait_issued(bar_kfull(stage0 + i2), (uint32_t)ph, ctl);
    }
    for (int n = 0; n < min(nq, slots); ++n) {
      int i2 = qr.i - 1 - n, ph = qr.phase;
      if (i2 < 0) { i2 += slots; ph ^= 1; }
      mbar_wait_issued(bar_qfull(slot0 + i2), (uint32_t)ph, ctl);
    }
  }

  // ---------------- teardown ----------------
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && ctl->abort && P.status) atomicCAS(P.status, 0, (int)KVC_ERR_TIMEOUT);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// The value norms' code stands behind the roles': in front of them it cost every launch, with norms or without, the instruction
// fetches of the jump over it (a run-time window of 24 rows at 40 to 20000 tokens 3.5 % of the scoring, the others 1 %).
template <int D, int W, bool kTaskMean, int kRT, bool kKeep>
__global__ void __launch_bounds__(kFastThreads, 1)
score_sm100_kernel(const __grid_constant__ FastParams P) {
  extern __shared__ __align__(1024) uint8_t smem[];
  if (blockIdx.x < (unsigned int)P.grid) {
    score_cta<D, W, kTaskMean, kRT, kKeep>(P, smem);
  } else {
    grid_dependency_wait();
    value_norm_cta<D>(P, smem_u32(smem));
  }
}

// ------------------------------------------------------------------------------------------------
// The rows' reference exponents: the scaled logit (base 2) of every window row against token 0 of
// its KV head, which every row sees.  Only a common scale for the pushed sums: a row's sum of
// 2^(logit - ref) is then at least about 1, so fixed point with 20 fractional bits keeps it.
// Bound by reading Q once.  A row's products are added in order, by one thread, so the rows go through shared memory: a
// thread that loads its own row touches 32 lines per warp load, and L1 takes those one by one.  (4096 units of 128 rows
// x 128, 155 MB: 42 -> 28.6 us, 5.4 TB/s; 256 units, one wave: 6.6 -> 4.8 us.)
// ------------------------------------------------------------------------------------------------
struct RefParams {
  int Bt, Hkv, G, HPT, QT, CH, w;
  unsigned long long* acc;     // [U][128]: cleared here
  unsigned long long* ovf;     // [U][128][4]: cleared here
  int* status;                 // the device status word (may be null): cleared here
  long long qs0, qs1, qs2, kvs0, kvs1;
  float sl2e;
};

template <int D>
__global__ void __launch_bounds__(kRows)
score_ref_kernel(RefParams P, LayerPtrs qp, LayerPtrs kp, float* __restrict__ ref) {
  constexpr int kVec = D / 8;                                // 16-byte pieces of a row
  constexpr int kRowsAtOnce = 32 / kVec;
  __shared__ __align__(16) uint4 k_row[kVec];                // token 0's key
  __shared__ __align__(16) uint4 q_row[kRows * kVec];        // piece t of row r in slot t ^ (r & 7): no bank conflicts either way
  grid_dependency_wait();
  const int u = blockIdx.x, row = threadIdx.x, lane = threadIdx.x & 31;
  const int uh = u / P.QT, qt = u - uh * P.QT;
  const int lb = uh / P.Hkv, h = uh - lb * P.Hkv;
  const int l = lb / P.Bt, b = lb - l * P.Bt;
  const int rows_u = P.CH == 1 ? min(P.HPT, P.G - qt * P.HPT) * P.w : min(kRows, P.w - (qt % P.CH) * kRows);
  {
    // a warp copies its 32 rows, neighbouring lanes neighbouring pieces, all in flight at once
    const int j = P.CH == 1 ? h * P.G + qt * P.HPT + row / P.w : h * P.G + qt / P.CH;
    const int m = P.CH == 1 ? row % P.w : (qt % P.CH) * kRows + row;
    const long long own = row < rows_u ? j * P.qs1 + m * P.qs2 : -1;      // (strides of a readable tensor are not negative)
    const __nv_bfloat16* q = reinterpret_cast<const __nv_bfloat16*>(qp.p[l]) + b * P.qs0;
    const int piece = lane % kVec;
#pragma unroll
    for (int i = 0; i < kVec; ++i) {
      const int from = i * kRowsAtOnce + lane / kVec, r = row - lane + from;
      const long long at = __shfl_sync(0xffffffffu, own, from);
      if (at >= 0) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(q_row + r * kVec + (piece ^ (r & 7)));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(q + at + piece * 8) : "memory");
      }
    }
  }
  if (row < kVec)
    k_row[row] = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(kp.p[l]) + b * P.kvs0 + h * P.kvs1) + row);
  // the unit's exchange state: empty words
  if (P.status != nullptr && u == 0 && row == 0) *P.status = 0;
  P.acc[(long long)u * kRows + row] = 0ull;
  {
    ulonglong2* o = reinterpret_cast<ulonglong2*>(P.ovf + ((long long)u * kRows + row) * 4);
    o[0] = make_ulonglong2(0ull, 0ull);
    o[1] = make_ulonglong2(0ull, 0ull);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  float r = 0.f;
  if (row < rows_u) {
    float acc = 0.f;                                         // products added in order
#pragma unroll
    for (int t = 0; t < kVec; ++t) {
      const uint4 a = q_row[row * kVec + (t ^ (row & 7))], k4 = k_row[t];
      const uint32_t aw[4] = {a.x, a.y, a.z, a.w}, bw[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        // a bf16 is the upper half of the fp32 with the same value
        acc = fmaf(__uint_as_float(aw[i] << 16), __uint_as_float(bw[i] << 16), acc);
        acc = fmaf(__uint_as_float(aw[i] & 0xffff0000u), __uint_as_float(bw[i] & 0xffff0000u), acc);
      }
    }
    r = acc * P.sl2e;
  }
  ref[(long long)u * kRows + row] = r;
}

// ------------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

bool encode_map(CUtensorMap* m, const void* base, int rank, const long long* dims, const long long* strides_bytes,
                const unsigned* box) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t gd[5]; cuuint64_t gs[4]; cuuint32_t bx[5]; cuuint32_t es[5] = {1, 1, 1, 1, 1};
  for (int i = 0; i < rank; ++i) { gd[i] = (cuuint64_t)dims[i]; bx[i] = box[i]; }
  for (int i = 0; i < rank - 1; ++i) gs[i] = (cuuint64_t)strides_bytes[i];
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), gd, gs, bx, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct FastPlan {
  int U, NT, RPU, grid, RT;
  int HPT, QT, CH;             // query heads per row tile, row tiles per KV head, row tiles per query head
  int RTU, QP;                 // row tiles per work unit, work units per KV head
  long long total_runs;
  int lead, norm_ctas;
  bool keep;                   // pass 2 keeps a run's -log-sum-exps in registers
  size_t off_partial, off_parts, off_acc, off_ovf, off_ref, off_total;
};

// Window lengths with a specialisation of their own.
constexpr bool window_special(int w) { return w == 8 || w == 16 || w == 32 || w == 64 || w == 128; }

// Clocks of a scoring CTA per pair of tiles, by what its pass 2 does with the rows of a row tile.  The maximum over a specialised
// window, or a long one, is bound by pass 1; every other way costs clocks per row.  (Scoring of 98304 tokens x 8 heads of 128, clocks per
// pair at 1.9 GHz, start included, times 0.74, which makes the first of them 1800: window 32 x 4 heads 1800, 32 x 1 1510, 7 x 4 2290, 7 x
// 16 5040, 13 x 9 3540, 24 x 4 2530, 49 x 2 2140; mean 32 x 4 2940, 32 x 2 2110, 24 x 4 7930, 13 x 9 9840, 500 rows 2840; a masked tile
// 2300 to 3800 more.  Heads of 64: 1550, 1390, and 100 to 300 less than heads of 128 elsewhere.)
constexpr double kMaskedClocks = 3000.;
double pair_clocks(const Problem& P, const FastPlan& pl) {
  const bool mean = P.agg_task == KVC_AGG_MEAN;
  const double rows = P.w > kRows ? kRows : pl.HPT * P.w;
  double least = P.d == 128 ? 1410. + 3. * rows : 1470. + 0.6 * rows;
  if (mean && least < 1600.) least = 1600.;
  double per_row = 0.;
  if (P.w > kRows) per_row = mean ? 12. : 0.;
  else if (window_special(P.w)) per_row = mean ? 14. : 0.;
  else if (mean) per_row = 70.;
  else per_row = P.w < 8 ? 32. : P.w < 16 ? 20. : P.w < 32 ? 14. : 7.;
  const double clocks = 1250. + per_row * rows;
  return clocks > least ? clocks : least;
}

// How many of the SMs take the value norms: as many as make both parts take the same time, in clocks: a scoring CTA has whole
// runs; an SM that only reads gets kNormBytes per clock.  (8B shape with value norms, us per pass
// with the norms before the scoring, and beside it at 25, 32, 40, 50 bytes per clock: 1000 tokens 86.6, 80.6, 81.7, 76.1, 75.4;
// 4096: 219, 218, 208, 206, 209; 16384 with the other options 805, 760, 735, 755, 781; 32768: 1542, 1488, 1453, 1491, 1535; two
// sequences of 8192 with heads of 64: 525, 521, 494, 487, 517.  With the prices above, at 36, 34, 32: 4096 tokens 211, 209, 207; 16384 761,
// 748, 745; 32768 1489, 1464, 1451; 16 layers of GQA group 7, window 64, 20000 tokens 519, 508, 511.)
// 0, for the kernel of their own, where that is expected to be as fast: it reads 25 bytes per clock and SM and takes 2 to 3 us besides.
// A unit's masked tiles are its last; a CTA's runs are `grid` apart, so with a common divisor g of grid and runs per unit it meets every
// g-th run of a unit only, and some CTA the masked ones all the time (500 rows at the end of 4096 tokens, value norms, 16 layers: 635
// us at a grid without such a divisor, 1214 at one of a multiple of eight).  The worst CTA counts.
// Windows longer than 128 rows, whose row tiles find their K in L2 for longer, lose 4 % to V going through it (300 rows behind 65536
// tokens, 3 layers: 1158 us with the kernel of its own, 1224 with six SMs beside the scoring).
constexpr double kNormBytes = 32., kNormAloneBytes = 25., kNormAloneClocks = 4500.;
int norm_share(const Problem& P, const FastPlan& pl, int sms, long long masked) {
  const long long block = P.d == 128 ? kNormBlock<16> : kNormBlock<8>;            // (rows are read by whole blocks)
  const double bytes = (double)P.L * P.Bt * P.Hkv * (double)((P.N + block - 1) / block * block) * P.d * P.elem_bytes;
  const double plain = pl.RTU * pair_clocks(P, pl) * pl.NT / pl.RPU;              // of a run
  auto score = [&](int grid) {
    int g = grid, b = pl.RPU;
    while (b != 0) { const int r = g % b; g = b; b = r; }
    // the masked tiles of the runs j = RPU - 1 - c, RPU - 1 - c - g, ...: the last run's class c = 0 has the most, or c = 1 where the
    // last run is a short one
    long long worst = 0;
    for (int c = 0; c < 2 && c < g; ++c) {
      long long sum = 0;
      for (int j = pl.RPU - 1 - c; j >= 0; j -= g) {
        const long long first = (long long)j * pl.RT, end = first + pl.RT < pl.NT ? first + pl.RT : pl.NT, from = pl.NT - masked;
        if (end <= from) break;
        sum += end - (first > from ? first : from);
      }
      worst = sum > worst ? sum : worst;
    }
    return (double)((pl.total_runs + grid - 1) / grid) * (plain + pl.RTU * kMaskedClocks * (double)worst * g / pl.RPU);
  };
  // where an even scoring and the norms would take the same time; the best whole number is next to it, or the largest that costs no
  // CTA another run
  const double all = (double)pl.total_runs * (plain + pl.RTU * kMaskedClocks * (double)masked / pl.RPU);
  const int even = (int)(sms / (1. + all * kNormBytes / bytes));
  int best = 0;
  double best_t = score(sms) + bytes / (sms * kNormAloneBytes) + kNormAloneClocks;
  auto consider = [&](int n) {
    if (n < 1 || n >= sms) return;
    const double beside = score(sms - n), norm = bytes / (n * kNormBytes), t = (beside > norm ? beside : norm) * (P.w > kRows ? 1.04 : 1.01);
    if (t < best_t) { best_t = t; best = n; }
  };
  for (int n = even - 3; n <= even + 12; ++n) consider(n);
  const long long most = (pl.total_runs + sms - even - 1) / (sms - even);
  for (long long k = most > 2 ? most - 2 : 1; k <= most + 1; ++k) consider(sms - (int)((pl.total_runs + k - 1) / k));
  return best;
}

// sms <= 0: no device yet (host-only size query) -- the workspace does not depend on it
void make_plan(const Problem& P, int sms, FastPlan* pl) {
  const int G = P.Hq / P.Hkv;
  if (P.w <= kRows) {
    pl->HPT = kRows / P.w < G ? kRows / P.w : G;
    pl->CH = 1;
    pl->QT = (G + pl->HPT - 1) / pl->HPT;
  } else {                      // a window longer than one accumulator: several row tiles per query head
    pl->HPT = 1;
    pl->CH = (P.w + kRows - 1) / kRows;
    pl->QT = G * pl->CH;
  }
  pl->U = P.L * P.Bt * P.Hkv * pl->QT;
  pl->NT = (int)((P.N + kTile - 1) / kTile);
  pl->RT = kMinRunTiles;
  if ((pl->NT + pl->RT - 1) / pl->RT > 255) pl->RT = (pl->NT + 254) / 255;   // the arrivals of a unit are counted in 8 bits
  pl->RPU = (pl->NT + pl->RT - 1) / pl->RT;
  // Tiles that some row does not see whole: the causal mask runs through them, or the context ends in them.
  const long long masked = pl->NT - ((P.q_pos0 < P.N - 1 ? P.q_pos0 : P.N - 1) + 1) / kTile;
  // Two row tiles per work unit share every K tile, but a run takes twice as long until its sums are out, and so do the first
  // run's and the last one's lead: 5 to 7 us, which have to be earned back.  (Scoring of 28 layers with 2 KV heads of 128, window 64,
  // GQA group 4: 6 pairs of runs per CTA 68.3 us one row tile at a time, 75.9 in pairs; 12: 127.2 and 126.9; 24: 246.4 and
  // 240.3; 16 layers of one KV head, window 300: 10 pairs 101 and 106, 21 187 and 186, 42 366 and 355.)  With heads of 64 pairs are
  // slower (32K tokens of the first shape 201 and 213 us) except for windows longer than 128 rows
  // (window 200: 7 pairs per CTA 68 and 67, 14 125 and 114, 55 443 and 399).  A run-time window of up to 128 rows gains
  // nothing (49 rows, 24 pairs: 276 and 276).  Of few row tiles an odd one left over costs what the pairs gain (us per pass one at a time
  // and in pairs: 7 row tiles 2306 and 2336, 9 1411 and 1425, 11 1685 and 1695, 13 1007 and 1021, 9 of 300 rows 724 and 736; 21 of 300 rows 772
  // and 749; heads of 64, 9 of 300 rows 300 and 292, 21 619 and 576).  The task mean, whose pass 2 goes column by column, stays one row tile
  // at a time.
  // So do contexts of whose tiles more than a fiftieth is masked: masked tiles go column by column as well, and a run of them on two
  // row tiles holds its whole unit up.  (us per pass of 32 layers, 8 KV heads, one at a time and in pairs: 500 rows at the end of
  // 4096 tokens 408 and 481, 16384 1231 and 1250, behind 3000 tokens, whose last tile is partial, 1025 and 1062, group 9 behind 1155
  // tokens, 16 layers, 523 and 622; window 150, heads of 64, behind 3000 tokens 238 and 248; window 128, group 8, 1787 tokens, one
  // tile masked by the window, 324 and 387.  With less: window 64 at 8192 tokens 470 and 466, at 32768 1772 and 1732; 500 rows
  // behind 65536 tokens, 4 layers, 1923 and 1824.)
  pl->RTU = 1;
  if (pl->QT > 1 && (pl->QT % 2 == 0 || pl->QT > (P.d == 128 ? 16 : 8)) && P.agg_task == KVC_AGG_MAX && (P.w > kRows || (P.d == 128 && window_special(P.w)))) {
    const long long pair_runs = (long long)P.L * P.Bt * P.Hkv * ((pl->QT + 1) / 2) * pl->RPU;
    if (pair_runs >= (long long)sms * (P.d == 128 ? 20 : 8) && sms > 0 && masked * 50 <= pl->NT) pl->RTU = 2;
  }
  // Keeping the -log-sum-exps pays on tiles that are not masked; where more than an eighth of them is, the other form is faster
  // (GQA group 7: window 128, heads of 64, 704 tokens 47.9 and 42.3 us, window 64, 795 tokens 33.7 and 32.2; the 8B shape at 1000
  // tokens, one of eight, 30.5 and 31.4).
  pl->keep = pl->RTU == 1 && P.agg_task == KVC_AGG_MAX && window_special(P.w) && P.w > 8 && masked * 8 <= pl->NT;
  pl->QP = (pl->QT + pl->RTU - 1) / pl->RTU;
  pl->total_runs = (long long)P.L * P.Bt * P.Hkv * pl->QP * pl->RPU;
  pl->norm_ctas = P.value_norm && sms > 1 ? norm_share(P, *pl, sms, masked) : 0;
  pl->grid = sms > 0 ? (int)(pl->total_runs < sms - pl->norm_ctas ? pl->total_runs : sms - pl->norm_ctas) : 1;
  // Pass 2 of a run starts once every run of its unit has been through pass 1: at other CTAs these lie at most
  // (grid + RPU - 2) / grid runs later in their order.  Pass 1 must be allowed that far ahead of pass 2 (or the CTAs
  // would wait for each other), and further only there: the rows in between should still be in L2 when pass 2 reads them.  Two runs further
  // for windows longer than 128 rows: a head's row tiles read the same rows anyway, and the runs are uneven (the short last row tile of
  // a head, masked tiles).  (500 rows: 65536 tokens 692 -> 583 us, 60000 615 -> 512, one row tile at a time 579 -> 528; 4096 tokens without a
  // mask the same.  Window 64, GQA group 7 at 128K 1 % slower with one run more, so not there.)
  pl->lead = (1 + (pl->grid + pl->RPU - 2) / pl->grid) * pl->RT + (pl->CH > 1 ? 2 * pl->RT : 0);
  size_t off = 0;
  pl->off_partial = off; off += align_up((size_t)pl->U * pl->RPU * kRows * sizeof(float2));
  pl->off_acc = off; off += align_up((size_t)pl->U * kRows * sizeof(unsigned long long));
  pl->off_ovf = off; off += align_up((size_t)pl->U * kRows * 4 * sizeof(unsigned long long));
  pl->off_ref = off; off += align_up((size_t)pl->U * kRows * sizeof(float));
  pl->off_parts = off;         // partial group aggregates [QT][L*Bt*Hkv][N], only with several row tiles
  if (pl->QT > 1) off += align_up((size_t)pl->U * P.N * sizeof(float));
  pl->off_total = off;
}

int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return sms;
}

// Test hooks (kvc_debug_score_hooks): the bound of the device-side waits and a unit whose
// statistics are withheld.
std::atomic<unsigned long long> g_wait_limit_ns{kDefaultWaitLimitNs};
std::atomic<int> g_withhold_unit{-1};

constexpr int kMaxDevices = 64;
std::mutex g_launch_mutex;

// The kernel's CTAs wait for one another, so all of them have to be resident at once: one per
// SM with the opt-in amount of shared memory.  Checked once per device and instantiation (the
// attribute is per device); KVC_ERR_UNSUPPORTED sends the caller to the CUDA-core path.
template <int D, int W, bool M, int kRT, bool kKeep>
kvc_status prepare_t(int grid) {
  using SL = SmemLayout<D, kRT>;
  static signed char state[kMaxDevices];      // 0: not looked at, 1: fits, -1: does not
  int dev = 0;
  KVC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return KVC_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_launch_mutex);
  if (state[dev] == 0) {
    KVC_CUDA(cudaFuncSetAttribute(score_sm100_kernel<D, W, M, kRT, kKeep>, cudaFuncAttributeMaxDynamicSharedMemorySize, SL::kTotal));
    int per_sm = 0, sms = 0;
    KVC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, score_sm100_kernel<D, W, M, kRT, kKeep>, kFastThreads,
                                                           (size_t)SL::kTotal));
    KVC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    state[dev] = (per_sm >= 1 && sms >= 1) ? 1 : -1;
  }
  (void)grid;                                 // grid <= SM count by construction (make_plan)
  return state[dev] == 1 ? KVC_OK : KVC_ERR_UNSUPPORTED;
}

template <int D, int W, bool M, int kRT, bool kKeep>
kvc_status launch_t(const FastParams& fp, int grid, cudaStream_t st) {
  using SL = SmemLayout<D, kRT>;
  const kvc_status s = prepare_t<D, W, M, kRT, kKeep>(grid);
  if (s != KVC_OK) return s;
  KVC_CUDA(launch_dependent(score_sm100_kernel<D, W, M, kRT, kKeep>, dim3(grid + fp.norm_ctas), dim3(kFastThreads), (size_t)SL::kTotal, st, fp));
  KVC_LAUNCH_CHECK("score_sm100_kernel");
  return KVC_OK;
}

template <int D, bool M, int kRT, bool kKeep>
kvc_status launch_w(int W, const FastParams& fp, int grid, cudaStream_t st) {
  switch (W) {
    case 8: return launch_t<D, 8, M, kRT, false>(fp, grid, st);
    case 16: return launch_t<D, 16, M, kRT, kKeep>(fp, grid, st);
    case 32: return launch_t<D, 32, M, kRT, kKeep>(fp, grid, st);
    case 64: return launch_t<D, 64, M, kRT, kKeep>(fp, grid, st);
    case 128: return launch_t<D, 128, M, kRT, kKeep>(fp, grid, st);
    default: return launch_t<D, 0, M, kRT, false>(fp, grid, st);      // any other window length: known at run time only
  }
}

// (two row tiles: only what make_plan sends here)
template <int D>
kvc_status launch_d(bool mean, int row_tiles, bool keep, int W, const FastParams& fp, int grid, cudaStream_t st) {
  if (row_tiles == 1) {
    if (mean) return launch_w<D, true, 1, false>(W, fp, grid, st);
    return keep ? launch_w<D, false, 1, true>(W, fp, grid, st) : launch_w<D, false, 1, false>(W, fp, grid, st);
  }
  if constexpr (D == 128) return launch_w<D, false, 2, false>(W, fp, grid, st);
  else return launch_t<D, 0, false, 2, false>(fp, grid, st);
}

}  // namespace

// The descriptor alone: is this a shape the tensor-core kernel handles?
bool score_sm100_shape_ok(const Problem& P) {
  if (P.dtype != KVC_BF16 || !P.contiguous_groups) return false;
  if (P.w < 1) return false;
  if (P.L > kMaxFastLayers) return false;
  if (P.N >= (1LL << 30)) return false;
  FastPlan pl;
  make_plan(P, 0, &pl);
  if ((long long)P.L * P.Bt * P.Hkv * pl.QT > (1 << 24)) return false;
  if (((long long)pl.U * pl.RPU + 8192) * pl.RT >= (1LL << 31)) return false;   // 32-bit sequence indices
  return true;
}

// ... and can its tensor maps be encoded here (a driver with the encoder is present)?
bool score_sm100_supported(const Problem& P) { return score_sm100_shape_ok(P) && encode_fn() != nullptr; }

size_t score_sm100_workspace_bytes(const Problem& P) {
  FastPlan pl;
  make_plan(P, 0, &pl);
  return pl.off_total;
}

// Returns KVC_ERR_UNSUPPORTED (without setting an error) when the tensor maps cannot be encoded
// for these strides; the caller then uses the CUDA-core path.
kvc_status launch_score_sm100(const Problem& P, const LayerPtrs& q, const LayerPtrs& k, const LayerPtrs* v, float* scores,
                              float* vnorm, int* device_status, void* ws, size_t ws_bytes, cudaStream_t st,
                              const float** parts_out, int* row_tiles_out, int* tiles_per_head_out) {
  const int sms = sm_count();
  if (sms < 1) return KVC_ERR_UNSUPPORTED;
  FastPlan pl;
  make_plan(P, sms, &pl);
  if (ws_bytes < pl.off_total) { set_error("score: workspace too small"); return KVC_ERR_WORKSPACE; }
  const int G = P.Hq / P.Hkv;
  static thread_local FastParams fp;
  for (int l = 0; l < P.L; ++l) {
    const long long kd[5] = {64, P.N, P.d / 64, P.Hkv, P.Bt};
    const long long ks[4] = {P.kvs[2] * 2, 128, P.kvs[1] * 2, P.kvs[0] * 2};
    const unsigned kb[5] = {64, (unsigned)kTile, (unsigned)(P.d / 64), 1, 1};
    const long long qd[4] = {P.d, P.w, P.Hq, P.Bt};
    const long long qs[3] = {P.qs[2] * 2, P.qs[1] * 2, P.qs[0] * 2};
    const unsigned qb[4] = {64, (unsigned)(pl.CH == 1 ? P.w : kRows), (unsigned)pl.HPT, 1};
    if (!encode_map(&fp.k_maps[l], k.p[l], 5, kd, ks, kb)) return KVC_ERR_UNSUPPORTED;
    if (!encode_map(&fp.q_maps[l], q.p[l], 4, qd, qs, qb)) return KVC_ERR_UNSUPPORTED;
  }
  char* w = reinterpret_cast<char*>(ws);

  fp.partial = reinterpret_cast<float2*>(w + pl.off_partial);
  fp.acc = reinterpret_cast<unsigned long long*>(w + pl.off_acc);
  fp.ovf = reinterpret_cast<unsigned long long*>(w + pl.off_ovf);
  float* ref = reinterpret_cast<float*>(w + pl.off_ref);
  fp.ref = ref;
  {
    RefParams rp;
    rp.acc = fp.acc;
    rp.ovf = fp.ovf;
    rp.status = device_status;
    rp.Bt = P.Bt; rp.Hkv = P.Hkv; rp.G = G; rp.HPT = pl.HPT; rp.QT = pl.QT; rp.CH = pl.CH; rp.w = P.w;
    rp.qs0 = P.qs[0]; rp.qs1 = P.qs[1]; rp.qs2 = P.qs[2]; rp.kvs0 = P.kvs[0]; rp.kvs1 = P.kvs[1];
    rp.sl2e = P.scale * kLog2eF;
    KVC_CUDA(launch_dependent(P.d == 128 ? score_ref_kernel<128> : score_ref_kernel<64>, dim3(pl.U), dim3(kRows), 0, st, rp, q, k, ref));
    KVC_LAUNCH_CHECK("score_ref_kernel");
  }
  fp.status = device_status;
  float* parts = pl.QT > 1 ? reinterpret_cast<float*>(w + pl.off_parts) : nullptr;
  fp.scores = pl.QT > 1 ? parts : scores;
  *parts_out = parts;
  *row_tiles_out = pl.QT;
  *tiles_per_head_out = pl.CH;
  fp.L = P.L; fp.Bt = P.Bt; fp.Hkv = P.Hkv; fp.G = G;
  fp.HPT = pl.HPT; fp.QT = pl.QT; fp.QP = pl.QP; fp.CH = pl.CH; fp.w = P.w;
  fp.N = P.N; fp.q_pos0 = P.q_pos0;
  fp.U = pl.U; fp.NT = pl.NT; fp.RPU = pl.RPU; fp.RT = pl.RT; fp.grid = pl.grid;
  fp.total_runs = (unsigned int)pl.total_runs; fp.lead = pl.lead;
  fp.step_u = pl.grid / pl.RPU; fp.step_j = pl.grid % pl.RPU;
  fp.step_q = fp.step_u % pl.QP;
  fp.step_h = (fp.step_u / pl.QP) % P.Hkv;
  fp.step_b = (fp.step_u / pl.QP / P.Hkv) % P.Bt;
  fp.step_l = fp.step_u / pl.QP / P.Hkv / P.Bt;
  fp.sl2e = P.scale * kLog2eF;
  fp.agg_group = P.agg_group;
  fp.norm_ctas = vnorm != nullptr ? pl.norm_ctas : 0;
  if (vnorm != nullptr && fp.norm_ctas == 0) {         // (see norm_share)
    const kvc_status s = launch_value_norm(P, *v, vnorm, st);
    if (s != KVC_OK) return s;
  }
  if (fp.norm_ctas > 0) {
    fp.v = *v;
    fp.vnorm = vnorm;
    fp.vs0 = P.kvs[0]; fp.vs1 = P.kvs[1]; fp.vs2 = P.kvs[2];
  }
  fp.wait_limit_ns = g_wait_limit_ns.load();
  fp.withhold_unit = g_withhold_unit.load();
  const bool mean = P.agg_task == KVC_AGG_MEAN;
  return P.d == 128 ? launch_d<128>(mean, pl.RTU, pl.keep, P.w, fp, pl.grid, st) : launch_d<64>(mean, pl.RTU, pl.keep, P.w, fp, pl.grid, st);
}

}  // namespace kvc


// Test hook: the bound of the scoring kernel's device-side waits (<= 0: the default of 2 s) and a
// unit (layer, sequence, KV head, row tile in that order) whose statistics are never sent, so
// that the waits for them expire (-1: none).  Process-wide; takes effect at the next launch.
extern "C" __attribute__((visibility("default"))) void kvc_debug_score_hooks(int64_t wait_limit_ns,
                                                                             int32_t withhold_unit) {
  kvc::g_wait_limit_ns.store(wait_limit_ns > 0 ? (unsigned long long)wait_limit_ns : kvc::kDefaultWaitLimitNs);
  kvc::g_withhold_unit.store(withhold_unit);
}

// Test hook: how the scoring of this problem is laid out on a device of `sms` SMs (none needed here): out[0] row tiles per work unit,
// [1] scoring CTAs, [2] CTAs of the value norms, [3] whether pass 2 keeps a run's -log-sum-exps, [4] work units' runs, [5] tiles by
// which pass 1 may be ahead.  KVC_ERR_UNSUPPORTED for a problem of the CUDA-core kernels.
extern "C" __attribute__((visibility("default"))) int kvc_debug_score_plan(const kvc_desc* d, int32_t sms, int64_t* out) {
  kvc::Problem P;
  const kvc_status s = kvc::resolve_desc(d, &P);
  if (s != KVC_OK) return s;
  if (sms < 1 || !kvc::score_sm100_shape_ok(P)) {
    kvc::set_error("score plan: not a problem of the tensor-core kernel");
    return KVC_ERR_UNSUPPORTED;
  }
  kvc::FastPlan pl;
  kvc::make_plan(P, sms, &pl);
  out[0] = pl.RTU; out[1] = pl.grid; out[2] = pl.norm_ctas; out[3] = pl.keep; out[4] = pl.total_runs; out[5] = pl.lead;
  return KVC_OK;
}
