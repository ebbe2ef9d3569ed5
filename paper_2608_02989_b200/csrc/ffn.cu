// Stage 4: grouped SwiGLU expert FFN over the activated experts with weighted combine,
//   y_t = sum_e w_{t,e} * W_down_e ( silu(W_gate_e x_t) * (W_up_e x_t) ),
// the step whose cost is the number of distinct expert weights touched (Section 1; Section 3.1).
//
// bf16 path (sm_100a): one persistent kernel, one CTA per SM, eight specialised warps:
//   warp 0      weight producer: one TMA copy per operand and stage (32 KB of weights = 128 rows x 128 K
//               in two 128-byte-swizzled atoms, plus the x chunk of gate/up stages) into a 3-stage ring
//   warp 1      issues tcgen05.mma (M=128 weight rows, N=node columns, fp32 accumulators in TMEM)
//   warps 2..5  epilogue: tcgen05.ld, SwiGLU / combine; only TMEM and shared memory are touched here
//   warp 6      helper: waits for other CTAs' partial sums and copies them into shared memory ahead of
//               need; adds the activation chunk to down stages once their experts are complete
//   warp 7      publisher: moves staged fragments / activation tiles to global memory (bulk reduce-add,
//               TMA store), waits for completion, then raises the counter other CTAs wait on
// The weights are the M operand ("swap-AB"): every activated expert's weights are read from HBM
// exactly once for all nodes of the block.  Work plan of a launch (plan_lane):
//   gate/up  tile = 64 gate rows + the 64 matching up rows of one expert, K = hidden.  The
//            n_tiles mod grid leftover tiles come first, cut into equal contiguous ranges of (tile,
//            K-chunk) units over all CTAs; the CTA that owns a tile's last chunk receives the others'
//            partial sums (added into its pre-zeroed global buffer), applies w * silu(g) * u and
//            stores the activation tile.  Then whole tiles, one per CTA and round.
//   down     tile = 128 output rows, K = (activated expert, intermediate) concatenated, cut evenly;
//            experts complete early first.  Partial tiles are added to the output with fp32
//            reductions in L2 (the caller zeroes the output).
// The down phase reads activations written by other CTAs in the gate/up phase; one finished-tile counter
// per expert orders them (a CTA waits for the experts its share of the K range reads).  Every wait is
// bounded; on expiry the kernel raises a status and drains.
//
// Small blocks (bf16, up to 32 node columns): k_ffn_bf16_small below, whose CTAs keep their activation tiles.
//
// f32 path: plain FMA kernels (the fp32 toy configuration is a few MFLOP).
#include <cuda_bf16.h>

#include <mutex>

#include "acm_internal.h"
#include "ffn_plan.h"
#include "mx_act.cuh"

namespace acm {
namespace {

#ifndef ACM_FFN_MX
#define ACM_FFN_MX 0
#endif
constexpr int kMaxStages = 3;                            // pipeline stages of the weight ring (see Geo)
constexpr int kAcc = 4;                                  // TMEM accumulators in flight (power of two)
constexpr int kBK = 64;                                  // K elements of one 128-byte swizzle atom
constexpr int kAtoms = 2;                                // atoms per pipeline stage: a stage covers 128 K
constexpr int kTileM = 128;
constexpr int kAtomABytes = kTileM * kBK * 2;            // 16 KB: 128 weight rows x one atom
constexpr int kABytes = kAtoms * kAtomABytes;            // 32 KB weight tile, one TMA copy
// The epilogue handles node columns kMaxNodes = 64 at a time: one fragment, one activation tile.  A wide tile (a
// batch of blocks with more than 64 nodes in all, up to kWideNodes = 128 accumulator columns) goes in two halves.
constexpr int kOutStageBytes = kTileM * kMaxNodes * 4;   // 32 KB: outgoing fragment (also the gate/up exchange buffer)
// One finished activation tile (64 features x 64 nodes): 8 KB of bf16, or three e5m2 pieces per element and 256 bytes of
// scales (MXFP4, see below).
constexpr int kHStages = ACM_FFN_MX ? 1 : 2;             // of them in shared memory
constexpr int kHPieceBytes = kMaxNodes * 64 * (ACM_FFN_MX ? kMxPieces : 2);
constexpr int kHStageBytes = kHPieceBytes + (ACM_FFN_MX ? kMxActScaleBytes : 0);
// ACM_FFN_MX = 1 (set by ffn_mx.cu, which includes this file) builds the same kernel for MXFP4 expert weights on the
// block-scaled tensor-core instruction (tcgen05.mma kind::mxf8f6f4: 8-bit operands, an E8M0 scale per row and 32 K).
//   Weights.  A pipeline stage of a tile is one contiguous 8704-byte record (128 rows x 64 bytes of E2M1 codes, 128 x 4
//   scale bytes).  Eight unpacking warps give every code a byte of its own -- two bits up, it is the same value as an
//   e2m3: sign | 2 exponent bits | 3 mantissa bits, of which the lower two are zero -- four instructions for eight codes
//   (an e4m3 would take seven), and store them in tensor memory, from where the MMAs take their A operand.  (4-bit
//   operands as they are would do without the moves, but have to lie in shared memory, 16 bytes for 16 codes: written
//   there and read again by the MMAs they made shared-memory bandwidth the bound, 670 of 720 clocks a stage.)
//   Activations.  A bf16 has 8 significand bits, an e5m2 three: x is the sum of three of them under one scale per node
//   and 32 K and its 2^-4 and 2^-8 (mx_act.cuh), exact unless another value of those 32 is more than 2^31 times larger and
//   then off by at most 2^-39 of that one.  Each piece has MMAs of its own into the same accumulator.  (Two e4m3 pieces as
//   node columns of their own, one MMA for both, are exact down to 2^-13 only.  Weights that are zero wherever a feature is
//   2^14 times the others then leave a result with three times the error; at 2^20 times it is 31 % off.)
//   The features are stored in the order the moves leave the weights in (mx_act.cuh).
// What bounds it: at 64 node columns the MMAs (a launch of 103 us takes 90 with a third of them) and what an SM takes in, 34 KB a
// stage of 0.45 us.  Up to 32 columns a stage takes 0.35 us where HBM would deliver one every 0.20, and no part of it by itself
// is the reason: with a third of the MMAs, an eighth of the tensor-memory stores, no activations or 512 bytes a record copied, or
// three unpacking groups, a launch of 85.7 us takes 82 to 86.
// A layer of 2048 x 768, 64 nodes, 22 experts: 42.5 us; 49.0 with the weights expanded to bf16 by four warps (0.56 us a
// stage) for eight kind::f16 MMAs.
constexpr int kThreads = ACM_FFN_MX ? 512 : 256;         // producer, MMA, 4 epilogue warps, helper, publisher (+ 2 x 4 unpacking warps)
[[maybe_unused]] constexpr int kMxCodeBytes = kTileM * 64;                // 128 rows x 128 four-bit codes
[[maybe_unused]] constexpr int kMxStageBytes = kMxCodeBytes + kTileM * 4; // + one scale byte per row and 32 K
[[maybe_unused]] constexpr int kMxACols = 32;                             // an unpacked stage in tensor memory: 4 weights a column
[[maybe_unused]] constexpr int kMxScaleCols = 16;                         // its scales: 4 columns the weights', 4 each piece's (2 used)
// Stages in flight behind the packed records: tensor-memory slots and activation stages, one ring.
constexpr int kMxA = 5;
static_assert(!ACM_FFN_MX || kAcc * kMaxNodes + kMxA * (kMxACols + kMxScaleCols) <= 512, "tensor memory: accumulators + unpacked stages");
// Shared memory of the MXFP4 kernel's rings: kMxA activation stages of 384 n_pad bytes and their scales, and packed records in
// what they leave (6 beside 64 node columns, 12 beside up to 32: mx_raw_stages).  Either is 1.5 us from request to arrival
// under load, from L2 and from HBM.
[[maybe_unused]] constexpr int kMaxRaw = 12;
[[maybe_unused]] constexpr int kMxRingBytes = 178 * 1024;
constexpr int kFragBytes = ACM_FFN_MX ? 0 : kTileM * kMaxNodes * 4;   // contributor fragments pre-summed in shared memory (MXFP4: no cut tiles)
constexpr int kFragFloats = kTileM * kMaxNodes;

using plan::FastDiv;
using plan::make_fastdiv;
using plan::fdiv;
using plan::Segment;
using plan::SegRange;
using plan::Plan;
using plan::Sched;
using plan::SmallWalk;
using plan::make_range;
using plan::cut_begin;
using plan::plan_lane;

// Every wait in this kernel is bounded.  What a role needs when one runs out lives in shared memory (GiveUp,
// touched on slow paths only): the limit, where to raise the status, and this CTA's diagnostic word, which
// names the wait that gave up first (acm_wait_report reads it).
enum WaitSite : int {
  kSiteNone = 0,
  kSiteAnchorWords = 1,     // prologue: the anchors' tagged words (router kernel's root CTAs)
  kSiteEligibleWords = 2,   // prologue / helper: the eligible set's tagged words (selection kernel)
  kSiteStageEmpty = 3,      // weight producer: a ring stage the MMAs have not released
  kSiteAccEmpty = 4,        // MMA issuer: an accumulator the epilogue has not drained
  kSiteStageFull = 5,       // MMA issuer: a stage whose copies have not landed
  kSiteFragFree = 6,        // helper: the fragment buffer in shared memory is still being read
  kSiteFragArrivals = 7,    // helper: other CTAs' partial sums of a cut tile
  kSiteFragCopy = 8,        // helper: its own bulk copy of the summed fragment
  kSiteExpertReady = 9,     // helper: finished-tile counters of the experts a down stage reads
  kSiteStageArmed = 10,     // helper: the weight producer has not armed the stage
  kSiteOutStaged = 11,      // publisher: an outgoing fragment from the epilogue
  kSiteActStaged = 12,      // publisher (small blocks: MMA issuer): a finished activation tile from the epilogue
  kSiteAccFull = 13,        // epilogue: an accumulator's MMAs
  kSiteOutFree = 14,        // epilogue: the outgoing-fragment buffer
  kSiteFragFull = 15,       // epilogue: the summed fragments of a cut tile
  kSiteActFree = 16,        // epilogue: an activation staging buffer
  kSitePlanReady = 17,      // any role: the rest of the plan (anchor start)
  kSitePackedStage = 18,    // MXFP4 unpacking warps: the packed weight stage
  kSitePackedFree = 19,     // MXFP4 weight producer: a record slot the unpacking warps have not read
  kSiteActStage = 20,       // MXFP4 unpacking warps: the stage's activations
  kSiteActSlot = 21,        // MXFP4 activation producer: a ring stage the MMAs have not released
  kSiteXPieces = 22         // MXFP4 activation producer: the hidden states' pieces
};
struct GiveUp {
  volatile int flag;             // set once this CTA has given up: every role then leaves at its next slow path
  unsigned long long limit_ns;   // the longest any single wait may last
  int32_t* status;               // the context's sticky status word
  int32_t* where;                // this CTA's diagnostic word: (launch number << 8) | WaitSite
  int32_t tag;                   // launch number << 8
};

// stages of the ring that the MMAs take their operands from
constexpr int kMaxRing = ACM_FFN_MX ? kMxA : kMaxStages;
template <int kN>
struct __align__(8) BarriersT {
  unsigned long long full[kMaxRing];
  unsigned long long empty[kMaxRing];
  unsigned long long tfull[kAcc];
  unsigned long long tempty[kAcc];
  unsigned long long drained;
#if !ACM_FFN_MX
  unsigned long long frag_full;      // helper -> epilogue: the pre-summed fragments of the next cut tile (half) are in smem
  unsigned long long frag_free;      // epilogue -> helper: the fragment buffer may be overwritten
  unsigned long long helper;         // completion of the helper warp's bulk copy
  unsigned long long ost_full, ost_free;   // epilogue <-> publisher: outgoing fragment staged / copied out
#endif
  unsigned long long hst_full[kHStages], hst_free[kHStages];   // epilogue <-> publisher: activation tile staged / stored
#if ACM_FFN_MX
  unsigned long long raw[kMaxRaw], raw_empty[kMaxRaw];   // packed records: landed (-> unpacking warps) / read (-> producer)
  unsigned long long act[kMaxRing];      // activation stages landed (-> unpacking warps)
#else
  volatile uint32_t armed;           // stages whose barrier the weight producer has armed so far
#endif
  volatile int32_t n_routed_slots;   // routed experts in this launch's work list (known with the complete list)
  uint32_t tmem_base;
  GiveUp give_up;
  float wd[kN];                 // combine weights of the expert being finalised
  int32_t entry[kMaxSlots];     // this launch's work list: make_entry(source, index) of every activated slot
  int16_t expert[kMaxSlots];    // routed expert id of the slot (-1: shared expert)
  uint32_t sel_half[4 * kMaskWords];   // early start: the eligible mask in 16-bit pieces (second half: blocks 4..7 of a batch)
  Plan plan;                    // this launch's work plan
  unsigned long long plan_ready;     // anchors' pre-segment: the rest of the plan and of the work list is in place
  uint32_t anc_part[4 * kMaskWords];   // early start on the anchors: their mask in 16-bit pieces (by the two polling warps)
};

// Geometry of the kernel for accumulator tiles of kN node columns: 64 (one block, three 48 KB stages) or 128 (a
// batch, two 64 KB stages -- as many bytes in flight -- and all of tensor memory).
template <int kN>
struct Geo {
  static constexpr int kStages = kN > kMaxNodes ? 2 : 3;
  static constexpr int kBBytes = kAtoms * kN * kBK * 2;          // activation chunk of a stage, one TMA copy
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kTmemCols = ACM_FFN_MX ? 512 : kAcc * kN;    // MXFP4: accumulators, unpacked weights, scales
  static constexpr int kRingBytes = ACM_FFN_MX ? kMxRingBytes : kStages * kStageBytes;
  static constexpr size_t kSmemBytes =
      1024 + static_cast<size_t>(kRingBytes) + kOutStageBytes + kFragBytes + kHStages * kHStageBytes + sizeof(BarriersT<kN>);
  static_assert(kSmemBytes <= 232448, "shared memory: ring + staging buffers + control block exceed 227 KB");
  static constexpr int kRing = ACM_FFN_MX ? kMxA : kStages;
  static_assert(kRing <= kMaxRing, "barrier arrays");
};

// ---------------------------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ unsigned long long global_timer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Has a wait that began at t0 outlasted the limit?  The clock is read twice before the answer is yes: a single
// reading that lies outside [t0, t0 + limit] (a value caught while the counter's halves roll over would) must
// not end a healthy launch.
__device__ __forceinline__ bool limit_passed(unsigned long long t0, unsigned long long limit_ns) {
  const long long d1 = static_cast<long long>(global_timer() - t0);
  if (d1 >= 0 && static_cast<unsigned long long>(d1) <= limit_ns) return false;
  const long long d2 = static_cast<long long>(global_timer() - t0);
  return d2 < 0 ? false : static_cast<unsigned long long>(d2) > limit_ns;
}
__device__ __noinline__ void give_up(GiveUp* g, int site) {
  if (atomicExch(const_cast<int*>(&g->flag), 1) == 0 && g->where) *g->where = g->tag | site;
  atomicCAS(g->status, 0, static_cast<int32_t>(ACM_ERR_TIMEOUT));
}
// Returns false if the limit ran out (the status is raised once) or the CTA has already given up; callers
// then skip the rest of their work.
// The wait for the rest of the plan is each thread's own, and the threads of a role must agree on its outcome -- one that
// left alone would strand the others at their next vote.  So it looks at the barrier only, not at the flag, and its limit
// is eight times that of the two polls behind which the barrier is opened, found or not.
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, GiveUp* g, int site) {
  const bool for_plan = site == kSitePlanReady;
  if (g->flag && !for_plan) return false;
  for (int i = 0; i < 1024; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_timer();
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (g->flag && !for_plan) return false;
    if (limit_passed(t0, for_plan ? 8 * g->limit_ns : g->limit_ns)) {
      give_up(g, site);
      return false;
    }
  }
}
// One inlined poll for the common case (the phase is already complete), the bounded loop out of line: the
// single-thread roles pay every instruction of their per-stage loop.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, GiveUp* g, int site) {
  if (mbar_try_wait(bar, parity)) return true;
  return mbar_wait_slow(bar, parity, g, site);
}
__device__ __forceinline__ int ld_acquire(const int32_t* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_add(int32_t* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Bounded wait until *p >= target (p written by other CTAs with release semantics).
__device__ bool flag_wait_ge(const int32_t* p, int target, GiveUp* g, int site) {
  if (g->flag) return false;
  for (int i = 0; i < 256; ++i)
    if (ld_acquire(p) >= target) return true;
  const unsigned long long t0 = global_timer();
  for (;;) {
    for (int i = 0; i < 16; ++i) {
      if (ld_acquire(p) >= target) return true;
      __nanosleep(64);
    }
    if (g->flag) return false;
    if (limit_passed(t0, g->limit_ns)) {
      give_up(g, site);
      return false;
    }
  }
}
// Bounded poll of one self-validating word (16 payload bits under a 16-bit tag) written by an earlier kernel
// of the same stream: returns the payload, or sets `seen` to false when the limit ran out.
__device__ __forceinline__ uint32_t poll_tagged_word(const uint32_t* word, uint32_t tag, unsigned long long limit_ns, bool& seen) {
  uint32_t v = 0;
  const unsigned long long t0 = global_timer();
  do {
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(word) : "memory");
    seen = (v >> 16) == tag;
  } while (!seen && !limit_passed(t0, limit_ns));
  return seen ? (v & 0xffffu) : 0u;
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
#if ACM_FFN_MX
__device__ __forceinline__ void bulk_load_hint(uint32_t smem_dst, const void* gmem_src, uint32_t bytes, uint32_t bar, uint64_t policy) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
               ::"r"(smem_dst), "l"(gmem_src), "r"(bytes), "r"(bar), "l"(policy) : "memory");
}
#endif
#if ACM_FFN_MX
__device__ __forceinline__ void bulk_store(void* gmem_dst, uint32_t smem_src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gmem_dst), "r"(smem_src), "r"(bytes) : "memory");
}
#endif
__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// Barrier over the 128 epilogue threads that also ANDs a predicate, so that all of them take the
// same decision after a bounded wait (a thread that left alone would strand the others at a barrier).
__device__ __forceinline__ bool epi_vote_all(bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 1, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r) : "r"(static_cast<uint32_t>(pred)) : "memory");
  return r != 0;
}

// The same over the 128 threads of one of several epilogue teams (named barriers 1, 2).
__device__ __forceinline__ bool team_vote_all(int team, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, %2, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r) : "r"(static_cast<uint32_t>(pred)), "r"(1 + team) : "memory");
  return r != 0;
}
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                            int c2, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4}], [%5], %6;"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar), "l"(policy) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                            int c2, int c3, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar), "l"(policy) : "memory");
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                            int c2, int c3, int c4, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4, %5, %6}], [%7], %8;"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar), "l"(policy) : "memory");
}
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t slot_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
      ::"r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// One lane of a converged warp (always the same one).
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(r));
  return r != 0;
}
// The end of a CTA in which a role has given up, so that any other may have left with work in flight: waits (bounded) for the
// MMAs before tensor memory is released -- a commit covers those of the lane that makes it, hence the issuer's election --
// and for copies to land before the CTA's shared memory is.  By the issuing warp.  (Out of line: in line it put 0.14 us
// on a launch that never runs it.)
__device__ __noinline__ void drain_cta(uint32_t drained) {
  if (elect_one()) umma_commit(drained);
  const unsigned long long t0 = global_timer();
  while (!mbar_try_wait(drained, 0) && global_timer() - t0 < 1000000ull) {}
  while (global_timer() - t0 < 200000ull) {}
  __syncwarp();
}
// Loads of this thread's lane from column taddr on.  The registers hold the values only behind tmem_arrived, which therefore names
// them: arithmetic on a register keeps its place beside volatile statements only if they name it, so behind a wait that names none
// it could be moved ahead of the wait.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);      // (a name for the same register)
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld1(uint32_t taddr, uint32_t& r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr) : "memory");
}
template <int kCount>
__device__ __forceinline__ void tmem_arrived(float (&v)[kCount]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < kCount; ++i) asm volatile("" : "+f"(v[i]));
}
template <int kCount>
__device__ __forceinline__ void tmem_arrived(uint32_t (&r)[kCount], float (&v)[kCount]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < kCount; ++i) {
    asm volatile("" : "+r"(r[i]));
    v[i] = __uint_as_float(r[i]);
  }
}

// Shared-memory matrix descriptor: K-major operand, rows of 128 bytes, 128-byte swizzle, groups of
// 8 rows 1024 bytes apart.  The tile base is 1024-byte aligned; stepping K by 16 elements adds 32 bytes.
__device__ __forceinline__ uint64_t umma_smem_desc(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((smem_addr & 0x3ffffu) >> 4);       // start address
  d |= static_cast<uint64_t>(1) << 16;                           // leading byte offset (unused here)
  d |= static_cast<uint64_t>(1024 >> 4) << 32;                   // stride byte offset
  d |= static_cast<uint64_t>(1) << 46;                           // descriptor version
  d |= static_cast<uint64_t>(2) << 61;                           // 128-byte swizzle
  return d;
}
#if ACM_FFN_MX
// Block-scaled MMA over 32 K: unpacked weights (128 rows, e2m3, in tensor memory: row = lane, four K a column) x e5m2
// activation pieces (K-major in shared memory), with their E8M0 scales in tensor memory (row or column j: lane j % 32 of
// every quarter, column j / 32).
__device__ __forceinline__ void umma_mx(uint32_t tmem_d, uint32_t tmem_a, uint64_t desc_b, uint32_t idesc, uint32_t accumulate,
                                        uint32_t tmem_sfa, uint32_t tmem_sfb) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], [%1], %2, %3, [%5], [%6], p;\n\t}\n"
      ::"r"(tmem_d), "r"(tmem_a), "l"(desc_b), "r"(idesc), "r"(accumulate), "r"(tmem_sfa), "r"(tmem_sfb) : "memory");
}
// Its instruction descriptor: A = E2M3, B = E5M2, E8M0 scales, fp32 accumulator, M = 128, N = n (bits 29, 30 and 4, 5: which
// byte of the scales' words).
__device__ __forceinline__ uint32_t umma_mx_idesc(int n) {
  return (3u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | (1u << 23) | (static_cast<uint32_t>(kTileM >> 7) << 27);
}
// Descriptor of an activation half-stage: rows of 64 bytes (64 K e5m2), 64-byte swizzle, groups of 8 rows 512 bytes apart.
__device__ __forceinline__ uint64_t umma_smem_desc_64(uint32_t smem_addr) {
  return static_cast<uint64_t>((smem_addr & 0x3ffffu) >> 4) | (static_cast<uint64_t>(1) << 16) |
         (static_cast<uint64_t>(512 >> 4) << 32) | (static_cast<uint64_t>(1) << 46) | (static_cast<uint64_t>(4) << 61);
}
// 4 consecutive columns of this thread's lane
__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void tmem_st2(uint32_t taddr, uint32_t a, uint32_t b) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1,%2};" ::"r"(taddr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]),
        "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]),
        "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
#endif
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t umma_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(kTileM >> 4) << 24);
}

// Optional time stamps (acm_stage_timing): per CTA, slot 0 = the roles start, 10 / 11 = its last gate/up / down tile is done.
#define ACM_STAMP(slot) do { if (p.trace) p.trace[static_cast<size_t>(blockIdx.x) * 32 + (slot)] = global_timer(); } while (0)

struct FfnArgs {
  int T, H, I, n_pad;
  FastDiv d_grid, d_kc1, d_tpe, d_kpe;   // reciprocals of the grid size and of the per-tile / per-expert chunk counts
  const uint32_t* act_mask;
  const uint32_t* resident;
  int li, n_shared;
  uint32_t only[4];
  const int32_t* slot_of;
  const float* wtab;
  acm_block_stats* stats;
  int32_t* ready;
#if !ACM_FFN_MX
  float* frag;
  int32_t* frag_flag;
#endif
  const uint32_t* sel_flag;
  int32_t sel_epoch;
  int sel_blocks;
  const uint32_t* anc_flag;    // non-null: eight tagged words with the anchor experts (Eq. 5), published before sel_flag
  float* out;
  int32_t* status;
  unsigned long long wait_limit_ns;   // the longest any single device-side wait may last
  int32_t* wait_diag;          // [grid] per-CTA diagnostic words (see GiveUp) or null
  int32_t launch_tag;          // launch number << 8
  unsigned long long* trace;   // optional [grid][32] time stamps (acm_stage_timing) or null
#if ACM_FFN_MX
  const unsigned char* mx_gate_up;   // [E][I/64][H/128][8704]
  const unsigned char* mx_down;      // [E][H/128][I/128][8704]
  const unsigned char* xq;           // hidden states in pieces: [H/64][3 n_pad][64], 64-byte swizzled
  const unsigned char* xq_scale;     // [H/64][256] (mx_scale_at)
  unsigned char* hq;                 // activations alike: [slot][I/64][3 n_pad][64]
  unsigned char* hq_scale;           // [slot][I/64][256]
  const int32_t* xq_count;           // CTAs that have stored their part of the pieces
  int32_t xq_target;                 // ... and how many there are
  int n_raw;                         // packed records in flight
#endif
};

__device__ __forceinline__ const CUtensorMap* pick_map(int src, const CUtensorMap* routed, const CUtensorMap* shared,
                                                       const CUtensorMap* staged) {
  return src == kSrcRouted ? routed : src == kSrcShared ? shared : staged;
}

// The plan (ffn_plan.h) lives in shared memory: a private copy indexed at run time would live in local memory,
// whose first touch costs every role a trip to DRAM at the start of the kernel.
#if ACM_FFN_MX
#define ACM_FFN_KERNEL k_ffn_mxfp4
#else
#define ACM_FFN_KERNEL k_ffn_bf16
#endif
// One kernel for both starts (on the anchors' pre-segment, or with the whole work list at hand): a launch bracketed
// by events then runs the same code as the launches around it, which keeps its instructions warm in the caches.
// kN = node columns of an accumulator tile (see Geo).
template <int kN>
__global__ void __launch_bounds__(kThreads, 1)
#if ACM_FFN_MX      // (every copy of it is a plain bulk one: no tensor maps)
ACM_FFN_KERNEL(const FfnArgs p) {
#else
ACM_FFN_KERNEL(const __grid_constant__ FfnMaps maps, const __grid_constant__ CUtensorMap x_map,
           const __grid_constant__ CUtensorMap h_map, const __grid_constant__ CUtensorMap hs_map,
           const FfnArgs p) {
#endif
  constexpr int kRing = Geo<kN>::kRing, kAccCols = kN, kTmemCols = Geo<kN>::kTmemCols;
#if !ACM_FFN_MX
  constexpr int kStageBytes = Geo<kN>::kStageBytes;
#endif
  using Barriers = BarriersT<kN>;
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
#if !ACM_FFN_MX
  unsigned char* stage_base = smem;
#endif
  unsigned char* after_ring = smem + static_cast<size_t>(Geo<kN>::kRingBytes);
#if ACM_FFN_MX
  // the ring area: activation pieces, their scales, packed records
  const int act_bytes = p.n_pad * (kMxPieces * 128);      // of a stage: two half-stages of 64 K
  unsigned char* act_base = smem;
  unsigned char* act_scale_base = act_base + kMxA * act_bytes;
  unsigned char* raw_base = act_scale_base + kMxA * 2 * kMxActScaleBytes;
#endif
  float* ostage = reinterpret_cast<float*>(after_ring);           // outgoing fragment [node][128 rows]
#if !ACM_FFN_MX
  float* ex = ostage;                                             // gate/up exchange aliases it (never used at once)
  float* sfrag = reinterpret_cast<float*>(after_ring + kOutStageBytes);
#endif
  unsigned char* hstage = after_ring + kOutStageBytes + kFragBytes;   // 2 x [node][64 features] bf16, swizzled
  Barriers* bars = reinterpret_cast<Barriers*>(after_ring + kOutStageBytes + kFragBytes + kHStages * kHStageBytes);
  GiveUp* const quit = &bars->give_up;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = blockIdx.x, G = gridDim.x;
  griddep_launch_dependents();
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRing; ++s) {
      mbar_init(smem_u32(&bars->full[s]), ACM_FFN_MX ? 4 : 1);   // MXFP4: one arrival per unpacking warp
      mbar_init(smem_u32(&bars->empty[s]), 1);
    }
#if ACM_FFN_MX
    for (int s = 0; s < p.n_raw; ++s) {
      mbar_init(smem_u32(&bars->raw[s]), 1);
      mbar_init(smem_u32(&bars->raw_empty[s]), 4);
    }
    for (int s = 0; s < kRing; ++s) mbar_init(smem_u32(&bars->act[s]), 1);
#endif
    for (int b = 0; b < kAcc; ++b) {
      mbar_init(smem_u32(&bars->tfull[b]), 1);
      mbar_init(smem_u32(&bars->tempty[b]), 128);
    }
    mbar_init(smem_u32(&bars->drained), 1);
    mbar_init(smem_u32(&bars->plan_ready), 1);
#if !ACM_FFN_MX
    mbar_init(smem_u32(&bars->frag_full), 1);
    mbar_init(smem_u32(&bars->frag_free), 128);
    mbar_init(smem_u32(&bars->helper), 1);
    mbar_init(smem_u32(&bars->ost_full), 128);
    mbar_init(smem_u32(&bars->ost_free), 1);
#endif
    for (int b = 0; b < kHStages; ++b) {
      mbar_init(smem_u32(&bars->hst_full[b]), 128);
      mbar_init(smem_u32(&bars->hst_free[b]), 1);
    }
    bars->give_up.flag = 0;
    bars->give_up.limit_ns = p.wait_limit_ns;
    bars->give_up.status = p.status;
    bars->give_up.where = p.wait_diag ? p.wait_diag + blockIdx.x : nullptr;
    bars->give_up.tag = p.launch_tag;
    if (p.wait_diag) p.wait_diag[blockIdx.x] = p.launch_tag;      // "this CTA of that launch has started"
#if !ACM_FFN_MX
    bars->armed = 0;
#endif
    fence_barrier_init();
  }
#if !ACM_FFN_MX
  if (warp == 0 && lane == 0) {
    prefetch_tensormap(&maps.gate_up);
    prefetch_tensormap(&maps.down);
    prefetch_tensormap(&x_map);
    prefetch_tensormap(&h_map);
  }
#endif
  if (warp == 1) {
    tmem_alloc(smem_u32(&bars->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  // Everything above touched only this CTA's own resources; global memory written by the kernels
  // before this one is read only from here on.  Early start: wait for the eligible set only.
  const bool early = p.sel_flag != nullptr;
  // Early start on the ANCHORS (Eq. 5: the root's natural top-k, always eligible): the router kernel publishes
  // them microseconds before the selection is done.  Their gate/up tiles become segment 0 of the plan, one
  // whole tile per CTA, and the roles start on it at once; the helper warp meanwhile waits for the eligible
  // set, completes the work list (the pre-streamed experts keep the first slots) and the plan, and opens
  // `plan_ready`, which every other role passes before its second segment.
  const bool pre = p.anc_flag != nullptr && p.sel_flag != nullptr;
  if (pre || early) {
    // Eight tagged words per block (16 mask bits under the 16-bit tag of this call; a batch has eight per block
    // and takes their union), each polled by its own thread of warps 2 and 3 -- four blocks per warp -- which have
    // nothing else to do yet, so that the poll runs beside the set-up above.  With the anchor start these are the
    // anchors' words, else the eligible set's.
    bool timed_out = false;
    if (threadIdx.x >= 64 && threadIdx.x < 128) {
      const int j = threadIdx.x - 64;
      const uint32_t* words = pre ? p.anc_flag : p.sel_flag;
      bool seen = true;
      uint32_t bits = 0u;
      if (j < 2 * kMaskWords * p.sel_blocks)
        bits = poll_tagged_word(words + j, static_cast<uint32_t>(p.sel_epoch) & 0xffffu, p.wait_limit_ns, seen);
      timed_out = !seen;
      bits |= __shfl_xor_sync(0xffffffffu, bits, 8);
      bits |= __shfl_xor_sync(0xffffffffu, bits, 16);
      if (lane < 2 * kMaskWords) (pre ? bars->anc_part : bars->sel_half)[(j >> 5) * 2 * kMaskWords + lane] = bits;
    }
    __syncthreads();
    if (timed_out) give_up(quit, pre ? kSiteAnchorWords : kSiteEligibleWords);
  } else {
    griddep_wait();
  }
  // The work list of this launch: slot a = the a-th activated expert of this list in ascending id
  // order (list 0: the resident ones, then the shared experts; list 1: the non-resident ones, which
  // the host has copied into staging slot a).
  uint32_t am[kMaskWords];
  int n_routed = 0;
#pragma unroll
  for (int wd = 0; wd < kMaskWords; ++wd) {
    uint32_t act;
    if (pre) {
      act = (bars->anc_part[2 * wd] | bars->anc_part[2 * kMaskWords + 2 * wd]) |
            ((bars->anc_part[2 * wd + 1] | bars->anc_part[2 * kMaskWords + 2 * wd + 1]) << 16);      // for now: the anchors only
    } else if (early) {
      act = (bars->sel_half[2 * wd] | bars->sel_half[2 * kMaskWords + 2 * wd]) |
            ((bars->sel_half[2 * wd + 1] | bars->sel_half[2 * kMaskWords + 2 * wd + 1]) << 16);
    } else {
      act = p.act_mask[wd];
    }
    const uint32_t res = p.resident ? p.resident[wd] : 0xffffffffu;
    am[wd] = (p.li == 0 ? act & res : act & ~res) & p.only[wd];
    n_routed += __popc(am[wd]);
  }
  const int tpe = p.I / 64;          // gate/up tiles per expert = K-chunks per expert in the down phase
  const int n_halves = (kN > kMaxNodes && p.n_pad > kMaxNodes) ? 2 : 1;   // the epilogue takes 64 node columns at a time
  // pre-segment: as many of the anchors (in ascending id) as give every CTA at most one whole tile
  const int n_pre = pre ? min(n_routed, static_cast<int>(fdiv(static_cast<unsigned>(G), p.d_tpe))) : 0;
  if (pre) {
    // keep the first n_pre anchors only
    int left = n_pre;
#pragma unroll
    for (int wd = 0; wd < kMaskWords; ++wd) {
      uint32_t m = am[wd], kept = 0u;
      while (m && left > 0) {
        const uint32_t bit = m & (0u - m);
        kept |= bit;
        m ^= bit;
        --left;
      }
      am[wd] = kept;
    }
    n_routed = n_pre;
  }
  const int n_act = n_routed + ((p.li == 0 && !pre) ? p.n_shared : 0);
  const int kc1 = p.H / (kBK * kAtoms);   // K-chunks (stages) of a gate/up tile
  const int kpe = (tpe + kAtoms - 1) / kAtoms;   // K-chunks (stages) per expert in the down phase
  const int h_tiles = p.H / kTileM;  // output tiles of the down phase
#if !ACM_FFN_MX
  const uint32_t b_atom_bytes = static_cast<uint32_t>(p.n_pad) * kBK * 2;   // one atom of the activation chunk
  const uint32_t b_bytes = kAtoms * b_atom_bytes;
#endif
  if (pre) {
    if (threadIdx.x == 7 * 32) {            // segment 0: the pre-streamed experts' tiles, one whole tile per CTA
      Segment sg0 = Segment{1, 1, 0, n_pre * tpe, 0, 0, 0, p.d_kc1, 0};
      bars->plan.seg[0] = sg0;
      bars->plan.range[0] = make_range(sg0, cta, p.d_grid, h_tiles);
      bars->plan.n_pre = n_pre;
      bars->plan.n_seg = 1;
    }
  } else if (warp == 7 && lane < 4) {      // (the publisher warp has nothing else to do yet)
    if (lane == 0) bars->n_routed_slots = n_routed;
    plan_lane<ACM_FFN_MX>(bars->plan, lane, cta, n_act, tpe, G, p.d_kc1, kpe, p.d_grid, p.d_tpe, h_tiles);
  }
  int32_t* s_entry = bars->entry;
  if (threadIdx.x < kMaxExperts) {
    const int e = threadIdx.x, wd = e >> 5;
    const uint32_t mine = wd == 0 ? am[0] : wd == 1 ? am[1] : wd == 2 ? am[2] : am[3];
    if ((mine >> (e & 31)) & 1u) {
      int slot = __popc(mine & ((1u << (e & 31)) - 1u));
#pragma unroll
      for (int v = 0; v < kMaskWords; ++v) slot += v < wd ? __popc(am[v]) : 0;
      // where the expert's weights are: the layer's own tensors (resident), staging slot `slot` (copied in
      // for this block), or -- with an expert pool -- whichever pool slot holds it
      s_entry[slot] = p.slot_of ? make_entry(kSrcStaged, p.slot_of[e])
                                : p.li == 0 ? make_entry(kSrcRouted, e) : make_entry(kSrcStaged, slot);
      bars->expert[slot] = e;
    }
  } else if (p.li == 0 && !pre && threadIdx.x - kMaxExperts < p.n_shared) {
    const int i = threadIdx.x - kMaxExperts;
    s_entry[n_routed + i] = make_entry(kSrcShared, i);
    bars->expert[n_routed + i] = -1;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const Segment* seg = bars->plan.seg;
  const uint32_t tmem_base = bars->tmem_base;
  if (threadIdx.x == 0) ACM_STAMP(0);
  // Does segment si exist?  With a pre-segment the plan behind segment 0 arrives later (the helper warp opens
  // plan_ready); n_seg is read from shared memory every time.
  const int n_seg_fixed = bars->plan.n_seg;
  auto have_seg = [&](int si, bool wait_for_plan) -> bool {
    if (pre) {
      if (si == 1 && wait_for_plan && !mbar_wait(smem_u32(&bars->plan_ready), 0u, quit, kSitePlanReady)) return false;
      return si < bars->plan.n_seg;
    } else {
      return si < n_seg_fixed;
    }
  };

  // The rest of the plan behind the anchors' pre-segment, by a warp that has nothing to do before it is there: the bf16
  // helper, the MXFP4 publisher (no tile is finalised before the routing kernel has completed).
  auto complete_plan = [&]() -> bool {
    // While the others run the anchors' pre-segment: wait for the eligible set, give the other experts the
    // slots behind the pre-streamed ones (ascending id), append the shared experts, work out the rest of the
    // plan, and let everyone on.
    // eight words per block; lane l takes words l and l + 32 (blocks 0-3 and 4-7), the union goes to lanes 0..7
    bool seen = true;
    uint32_t half = 0u;
    {
      const uint32_t tag = static_cast<uint32_t>(p.sel_epoch) & 0xffffu;
      const int n_words = 2 * kMaskWords * p.sel_blocks;
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        const int j = lane + 32 * part;
        if (j < n_words) {
          bool got = true;
          half |= poll_tagged_word(p.sel_flag + j, tag, p.wait_limit_ns, got);
          seen = seen && got;
        }
      }
      half |= __shfl_xor_sync(0xffffffffu, half, 8);
      half |= __shfl_xor_sync(0xffffffffu, half, 16);
    }
    const bool good = __all_sync(0xffffffffu, seen);
    uint32_t rest[kMaskWords];
    int n_rest = 0;
#pragma unroll
    for (int wd = 0; wd < kMaskWords; ++wd) {
      const uint32_t lo = __shfl_sync(0xffffffffu, half, 2 * wd), hi = __shfl_sync(0xffffffffu, half, 2 * wd + 1);
      rest[wd] = ((lo | (hi << 16)) & p.only[wd]) & ~am[wd];
      n_rest += __popc(rest[wd]);
    }
    if (good) {
      for (int e = lane; e < kMaxExperts; e += 32) {
        const int wd = e >> 5;
        const uint32_t mine = wd == 0 ? rest[0] : wd == 1 ? rest[1] : wd == 2 ? rest[2] : rest[3];
        if ((mine >> (e & 31)) & 1u) {
          int slot = n_pre + __popc(mine & ((1u << (e & 31)) - 1u));
#pragma unroll
          for (int w2 = 0; w2 < kMaskWords; ++w2) slot += w2 < wd ? __popc(rest[w2]) : 0;
          s_entry[slot] = make_entry(kSrcRouted, e);
          bars->expert[slot] = e;
        }
      }
      if (lane < p.n_shared) {
        s_entry[n_pre + n_rest + lane] = make_entry(kSrcShared, lane);
        bars->expert[n_pre + n_rest + lane] = -1;
      }
      if (lane == 0) bars->n_routed_slots = n_pre + n_rest;
      if (lane < 4)
        plan_lane<ACM_FFN_MX>(bars->plan, lane, cta, n_pre + n_rest + p.n_shared, tpe, G, p.d_kc1, kpe, p.d_grid, p.d_tpe, h_tiles,
                  n_pre, 1);
    } else if (lane == 0) {
      give_up(quit, kSiteEligibleWords);
    }
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(smem_u32(&bars->plan_ready));
    }
    return good;
  };
  // The CTAs walk the K-chunks of their (whole) tiles from different ones on: in step, all of them would fetch the same
  // chunk of the hidden states at the same time, from the same few slices of L2.
  const int k_first = cta % kc1;
  auto k_rot = [&](int kc) { return kc + k_first < kc1 ? kc + k_first : kc + k_first - kc1; };

  if (warp == 0) {
    // ------------------------------------------------------------------ weight producer
    // Streams every weight tile of this CTA (and the x chunk of gate/up stages).  It arms each
    // stage's barrier with the bytes of both operands; the activation chunk of a down stage is
    // added by the helper warp once that expert group is complete, so this stream never stalls on
    // it.  The loop is kept to a few instructions per stage: one thread pays every one of them.
    if (lane == 0) {
      const uint64_t pol_w = policy_evict_first();
      uint32_t s = 0, par = 0;
#if !ACM_FFN_MX
      const uint64_t pol_x = policy_evict_last();
      uint32_t n_armed = 0;
#endif
      bool ok = true;
      for (int si = 0; ok && have_seg(si, true); ++si) {
        const Segment sg = seg[si];
        if (sg.phase == 1) {
          Sched sc(bars->plan.range[si]);
          int tile, k0, k1;
          while (ok && sc.next(tile, k0, k1)) {
            const int a_of = static_cast<int>(fdiv(static_cast<unsigned>(sg.t0 + tile), p.d_tpe));
            const int32_t ent = s_entry[a_of];
            const int r0 = (sg.t0 + tile - a_of * tpe) * 64, eidx = entry_idx(ent);
#if !ACM_FFN_MX
            const CUtensorMap* gu = pick_map(entry_src(ent), &maps.gate_up, &maps.shared_gate_up, &maps.staged_gate_up);
#endif
#if !ACM_FFN_MX
            int kk = (k0 == 0 && k1 == kc1) ? k_rot(0) : k0;      // the K-chunk of stage kc
#endif
            for (int kc = k0; kc < k1; ++kc) {
#if ACM_FFN_MX
              if (!(ok = mbar_wait(smem_u32(&bars->raw_empty[s]), par ^ 1u, quit, kSitePackedFree))) break;
              const uint32_t rawb = smem_u32(&bars->raw[s]);
              mbar_expect_tx(rawb, kMxStageBytes);
              bulk_load_hint(smem_u32(raw_base) + s * kMxStageBytes,
                             p.mx_gate_up + (static_cast<size_t>(eidx * tpe + (r0 >> 6)) * kc1 + k_rot(kc)) * kMxStageBytes,
                             kMxStageBytes, rawb, pol_w);
              if (++s == static_cast<uint32_t>(p.n_raw)) { s = 0; par ^= 1u; }
#else
              if (!(ok = mbar_wait(smem_u32(&bars->empty[s]), par ^ 1u, quit, kSiteStageEmpty))) break;
              const uint32_t full = smem_u32(&bars->full[s]);
              const uint32_t sa = smem_u32(stage_base) + s * kStageBytes;
              mbar_expect_tx(full, kABytes + b_bytes);
              tma_load_5d(sa, gu, full, 0, r0, 0, kk * kAtoms, eidx, pol_w);   // 64 gate + 64 up rows, 2 atoms
              tma_load_3d(sa + kABytes, &x_map, full, 0, 0, kk * kAtoms, pol_x);
              if (++kk == kc1) kk = 0;
              ++n_armed;
              if (++s == kRing) { s = 0; par ^= 1u; }
#endif
            }
          }
        } else {
          Sched sc(bars->plan.range[si]);
          int ht, k0, k1;
          while (ok && sc.next(ht, k0, k1)) {
            const int q0 = static_cast<int>(fdiv(static_cast<unsigned>(k0), p.d_kpe));
            int a = sg.a0 + q0, ic = k0 - q0 * kpe;
            int32_t ent = s_entry[a];
#if !ACM_FFN_MX
            const CUtensorMap* dn = pick_map(entry_src(ent), &maps.down, &maps.shared_down, &maps.staged_down);
#endif
            int eidx = entry_idx(ent);
            for (int kc = k0; kc < k1; ++kc) {
#if ACM_FFN_MX
              if (!(ok = mbar_wait(smem_u32(&bars->raw_empty[s]), par ^ 1u, quit, kSitePackedFree))) break;
              const uint32_t rawb = smem_u32(&bars->raw[s]);
              mbar_expect_tx(rawb, kMxStageBytes);
              bulk_load_hint(smem_u32(raw_base) + s * kMxStageBytes,
                             p.mx_down + (static_cast<size_t>(eidx * h_tiles + ht) * kpe + ic) * kMxStageBytes,
                             kMxStageBytes, rawb, pol_w);
              if (++s == static_cast<uint32_t>(p.n_raw)) { s = 0; par ^= 1u; }
              if (++ic == kpe && kc + 1 < k1) {
                ic = 0;
                ent = s_entry[++a];
                eidx = entry_idx(ent);
              }
#else
              if (!(ok = mbar_wait(smem_u32(&bars->empty[s]), par ^ 1u, quit, kSiteStageEmpty))) break;
              const uint32_t full = smem_u32(&bars->full[s]);
              const uint32_t sa = smem_u32(stage_base) + s * kStageBytes;
              mbar_expect_tx(full, kABytes + b_bytes);
              tma_load_4d(sa, dn, full, 0, ht * kTileM, ic * kAtoms, eidx, pol_w);
              bars->armed = ++n_armed;      // the helper warp may now add this stage's activation chunk
              if (++s == kRing) { s = 0; par ^= 1u; }
              if (++ic == kpe && kc + 1 < k1) {
                ic = 0;
                ent = s_entry[++a];
                dn = pick_map(entry_src(ent), &maps.down, &maps.shared_down, &maps.staged_down);
                eidx = entry_idx(ent);
              }
#endif
            }
          }
        }
      }
      // The block's activated-expert counts, by the thread that is done first (its copies are all issued
      // microseconds before the last epilogue): off the kernel's tail.
      if (p.stats && p.li == 0 && blockIdx.x == 0) {
        griddep_wait();                       // early start: the routing kernel is long complete
        int n_all = 0, n_stg = 0;
#pragma unroll
        for (int wd = 0; wd < kMaskWords; ++wd) {
          const uint32_t act = __ldcg(p.act_mask + wd);
          n_all += __popc(act);
          n_stg += p.resident ? __popc(act & ~p.resident[wd]) : 0;
        }
        p.stats->n_activated = n_all;
        p.stats->n_staged = n_stg;
        p.stats->n_streamed = bars->n_routed_slots;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // The whole warp walks the stages and one elected lane issues: the operands of an MMA are uniform registers, and
    // in code that only lane 0 runs every one of them is moved there from a vector register first (four MMAs of an
    // MXFP4 stage: 370 clocks to issue, 110 this way).
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem_base, 0);
#if ACM_FFN_MX
    const uint32_t idesc = umma_mx_idesc(p.n_pad);
    const uint64_t act_hi = umma_smem_desc_64(0);
    // (in 16-byte units) from one half-stage to the other, from one piece to the next
    const uint32_t half_step = static_cast<uint32_t>(act_bytes) >> 5, piece_step = static_cast<uint32_t>(p.n_pad) * 4;
    const uint32_t act0 = (smem_u32(act_base) & 0x3ffffu) >> 4;
#else
    const uint32_t idesc = umma_idesc(p.n_pad);
    const uint64_t desc_hi = umma_smem_desc(0);
    const uint32_t stage0 = (smem_u32(stage_base) & 0x3ffffu) >> 4;
#endif
    uint32_t s = 0, par = 0, b = 0, bpar = 1;
    bool ok = true;
    for (int si = 0; ok && __all_sync(0xffffffffu, have_seg(si, true)); ++si) {
      Sched sc(bars->plan.range[si]);
      int tile, k0 = 0, k1 = 0;
      while (ok && __any_sync(0xffffffffu, sc.next(tile, k0, k1))) {
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->tempty[b]), bpar, quit, kSiteAccEmpty));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tm + b * kAccCols;
        const int nk = __shfl_sync(0xffffffffu, k1 - k0, 0);
        for (int kc = 0; kc < nk; ++kc) {
          ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->full[s]), par, quit, kSiteStageFull));
          if (!ok) break;
          tc_fence_after();
#if ACM_FFN_MX
          const uint32_t ta = tm + kAcc * kAccCols + s * kMxACols;
          const uint32_t sf = tm + kAcc * kAccCols + kMxA * kMxACols + s * kMxScaleCols;
          const uint64_t db = act_hi | (act0 + s * (static_cast<uint32_t>(act_bytes) >> 4));
          if (elect_one()) {
            // 32 K = one scale each (byte kb of the scales' words); two half-stages of 64 K of activations
#pragma unroll
            for (int pc = 0; pc < kMxPieces; ++pc) {
#pragma unroll
              for (int kb = 0; kb < 4; ++kb)
                umma_mx(d_tmem, ta + 8 * kb, db + pc * piece_step + (kb >> 1) * half_step + (kb & 1) * 2,
                        idesc | (static_cast<uint32_t>(kb) << 29) | (static_cast<uint32_t>(kb) << 4), (kc > 0 || pc > 0 || kb > 0) ? 1u : 0u,
                        sf, sf + 4 + 4 * pc);
            }
            umma_commit(smem_u32(&bars->empty[s]));
            if (kc + 1 == nk) umma_commit(smem_u32(&bars->tfull[b]));
          }
#else
          // descriptors: only the address field changes from stage to stage and atom to atom
          const uint64_t da0 = desc_hi | (stage0 + s * (kStageBytes >> 4));
          const uint64_t db0 = desc_hi | (stage0 + s * (kStageBytes >> 4) + (kABytes >> 4));
          if (elect_one()) {
#pragma unroll
            for (int at = 0; at < kAtoms; ++at) {
#pragma unroll
              for (int kk = 0; kk < kBK / 16; ++kk)
                umma_bf16(d_tmem, da0 + (at * (kAtomABytes >> 4) + 2 * kk), db0 + (at * (b_atom_bytes >> 4) + 2 * kk), idesc,
                          (kc > 0 || at > 0 || kk > 0) ? 1u : 0u);
            }
            umma_commit(smem_u32(&bars->empty[s]));
            if (kc + 1 == nk) umma_commit(smem_u32(&bars->tfull[b]));
          }
#endif
          __syncwarp();
          if (++s == kRing) { s = 0; par ^= 1u; }
        }
        if (++b == kAcc) { b = 0; bpar ^= 1u; }
      }
    }
#if ACM_FFN_MX
  } else if (warp == 6) {
    // ------------------------------------------------------------------ activation producer
    // Fetches the activation pieces of every stage, a stage of 128 K = two half-stages of 64: the hidden states' once
    // the router kernel's CTAs have stored them all, an expert's activations once all its tiles have been stored.
    bool ok = true, x_seen = false;
    const uint64_t pol_x = policy_evict_last();
    uint32_t ai = 0, apar = 0;
    auto fetch = [&](const unsigned char* pieces, const unsigned char* scales) -> bool {
      if (!mbar_wait(smem_u32(&bars->empty[ai]), apar ^ 1u, quit, kSiteActSlot)) return false;
      const uint32_t full = smem_u32(&bars->act[ai]);
      mbar_expect_tx(full, static_cast<uint32_t>(act_bytes) + 2 * kMxActScaleBytes);
      bulk_load_hint(smem_u32(act_base) + ai * act_bytes, pieces, act_bytes, full, pol_x);
      bulk_load_hint(smem_u32(act_scale_base) + ai * 2 * kMxActScaleBytes, scales, 2 * kMxActScaleBytes, full, pol_x);
      if (++ai == kRing) { ai = 0; apar ^= 1u; }
      return true;
    };
    for (int si = 0; ok && have_seg(si, true); ++si) {
      const Segment sg = seg[si];
      const SegRange& rg = bars->plan.range[si];
      if (sg.phase == 1) {
        if (lane == 0) {
          if (!x_seen) {
            ok = flag_wait_ge(p.xq_count, p.xq_target, quit, kSiteXPieces);
            fence_proxy_async();
            x_seen = true;
          }
          Sched sc(rg);
          int tile, k0, k1;
          while (ok && sc.next(tile, k0, k1))
            for (int kc = k0; ok && kc < k1; ++kc)
              ok = fetch(p.xq + static_cast<size_t>(k_rot(kc)) * act_bytes, p.xq_scale + static_cast<size_t>(k_rot(kc)) * 2 * kMxActScaleBytes);
        }
      } else {
        bool good = true;
        const unsigned n_units = rg.u_end - rg.u;
        if (n_units > 0) {      // the experts this CTA's share reads (as in the bf16 build's helper warp)
          int q_lo = 0, q_hi = sg.a1 - sg.a0 - 1;
          if (static_cast<unsigned>(rg.k00) + n_units <= static_cast<unsigned>(rg.kc)) {
            q_lo = static_cast<int>(fdiv(static_cast<unsigned>(rg.k00), p.d_kpe));
            q_hi = static_cast<int>(fdiv(static_cast<unsigned>(rg.k00) + n_units - 1u, p.d_kpe));
          }
          for (int q = q_lo + lane; q <= q_hi && good; q += 32)
            good = flag_wait_ge(&p.ready[sg.a0 + q], tpe, quit, kSiteExpertReady);
        }
        ok = __all_sync(0xffffffffu, good);
        if (ok && lane == 0) {
          Sched sc(rg);
          int ht, k0, k1;
          fence_proxy_async();
          while (ok && sc.next(ht, k0, k1)) {
            const int q0 = static_cast<int>(fdiv(static_cast<unsigned>(k0), p.d_kpe));
            // (an expert's K-chunks lie one after the other, and so do the experts of a segment)
            size_t at = static_cast<size_t>(sg.a0 + q0) * kpe + (k0 - q0 * kpe);
            for (int kc = k0; ok && kc < k1; ++kc, ++at) ok = fetch(p.hq + at * act_bytes, p.hq_scale + at * 2 * kMxActScaleBytes);
          }
        }
      }
      ok = __all_sync(0xffffffffu, ok);
    }
#else
  } else if (warp == 6) {
    // ------------------------------------------------------------------ helper warp
    // Keeps slow global round trips off the other roles' paths: (a) for each gate/up segment whose
    // last fragment is the head of a tile shared with later CTAs, waits for their fragments and sums
    // them into shared memory; (b) for each down segment, waits until every activation tile of its
    // expert group has been stored, then tells the producer.
    bool ok = true;
    int frag_uses = 0;
    uint32_t hs = 0, hidx = 0;   // ring slot and running index of the next stage, tracked through the gate/up stages too
    if (pre) ok = complete_plan();
    for (int si = 0; ok && have_seg(si, false); ++si) {
      const Segment sg = seg[si];
      const int n_exp = sg.a1 - sg.a0;
      if (sg.phase == 1) {
        hidx += bars->plan.range[si].n_stages;
        hs = hidx % kRing;
        if (sg.whole) continue;          // whole tiles: nothing to exchange
        const unsigned ub = cut_begin(sg, cta, p.d_grid), ue = cut_begin(sg, cta + 1, p.d_grid);
        if (ue <= ub) continue;
        const unsigned last_tile = fdiv(ue - 1, p.d_kc1);
        const unsigned tile_end = (last_tile + 1) * kc1;
        const bool head = (last_tile * kc1 >= ub) && (ue < tile_end);   // starts at chunk 0, ends before the tile does
        if (!head) continue;
        int n_contrib = 0;
        for (int c2 = cta + 1; c2 < G; ++c2) {
          const unsigned b2 = cut_begin(sg, c2, p.d_grid), e2 = cut_begin(sg, c2 + 1, p.d_grid);
          if (b2 >= tile_end) break;
          if (e2 > b2) ++n_contrib;
        }
        // one fragment buffer and one arrival counter per column half of the tile (a wide tile has two)
        for (int h = 0; h < n_halves && ok; ++h) {
          if (frag_uses > 0) {   // the buffer in shared memory still holds the previous sum until the epilogue has read it
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->frag_free), (frag_uses - 1) & 1u, quit, kSiteFragFree));
            if (!ok) break;
          }
          float* frag = p.frag + ((static_cast<size_t>(sg.p1_index) * G + cta) * 2 + h) * kFragFloats;   // this CTA's buffer
          int32_t* arrived = p.frag_flag + (sg.p1_index * G + cta) * 2 + h;
          const int n_el = min(p.n_pad - h * kMaxNodes, kMaxNodes) * kTileM;
          // every CTA holding a later part of the tile has reduce-added its fragment: one bulk copy
          bool got = true;
          if (lane == 0) got = flag_wait_ge(arrived, n_contrib, quit, kSiteFragArrivals);
          ok = __all_sync(0xffffffffu, got);
          if (!ok) break;
          if (lane == 0) {
            fence_proxy_async();
            const uint32_t hb = smem_u32(&bars->helper);
            mbar_expect_tx(hb, static_cast<uint32_t>(n_el) * 4u);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(smem_u32(sfrag)), "l"(frag), "r"(static_cast<uint32_t>(n_el) * 4u), "r"(hb) : "memory");
          }
          ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->helper), frag_uses & 1u, quit, kSiteFragCopy));
          if (!ok) break;
          if (lane == 0) mbar_arrive(smem_u32(&bars->frag_full));
          // leave the buffer and its counter zero for the next launch
          float4* z4 = reinterpret_cast<float4*>(frag);
          for (int i = lane; i < n_el / 4; i += 32) z4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (lane == 0) *arrived = 0;
          ++frag_uses;
        }
        if (!ok) break;
      } else {
        // activation producer: once every activation tile of this expert group is stored, add the
        // activation chunk of each down stage to the barrier the weight producer has armed (or will arm)
        bool good = true;
        {
          // The experts whose activation tiles this CTA's share of the segment reads (one finished-tile counter
          // per expert), polled side by side, one lane each: from the first to the last K-chunk of the share, or
          // the whole group if the share runs on into the next output tile.
          const SegRange& rg = bars->plan.range[si];
          const unsigned n_units = rg.u_end - rg.u;
          if (n_units > 0) {
            int q_lo = 0, q_hi = n_exp - 1;
            if (static_cast<unsigned>(rg.k00) + n_units <= static_cast<unsigned>(rg.kc)) {
              q_lo = static_cast<int>(fdiv(static_cast<unsigned>(rg.k00), p.d_kpe));
              q_hi = static_cast<int>(fdiv(static_cast<unsigned>(rg.k00) + n_units - 1u, p.d_kpe));
            }
            for (int q = q_lo + lane; q <= q_hi && good; q += 32)
              good = flag_wait_ge(&p.ready[sg.a0 + q], tpe * n_halves, quit, kSiteExpertReady);
          }
          good = __all_sync(0xffffffffu, good);
        }
        if (good && lane == 0) {
          const uint64_t pol_x = policy_evict_last();
          Sched sc(bars->plan.range[si]);
          int ht, k0, k1;
          fence_proxy_async();
          while (good && sc.next(ht, k0, k1)) {
            const int q0 = static_cast<int>(fdiv(static_cast<unsigned>(k0), p.d_kpe));
            int a = sg.a0 + q0, ic = k0 - q0 * kpe;
            for (int kc = k0; kc < k1; ++kc) {
              // never ahead of the weight producer: it has found the slot free and armed the barrier
              if (bars->armed <= hidx) {
                const unsigned long long t0 = global_timer();
                while (bars->armed <= hidx) {
                  if (quit->flag) { good = false; break; }
                  if (limit_passed(t0, p.wait_limit_ns)) {
                    give_up(quit, kSiteStageArmed);
                    good = false;
                    break;
                  }
                }
                if (!good) break;
              }
              tma_load_4d(smem_u32(stage_base) + hs * kStageBytes + kABytes, &h_map, smem_u32(&bars->full[hs]),
                          0, 0, ic * kAtoms, a, pol_x);
              ++hidx;
              if (++hs == kRing) hs = 0;
              if (++ic == kpe) { ic = 0; ++a; }
            }
          }
        }
        ok = __all_sync(0xffffffffu, good);
      }
    }
#endif
  } else if (warp == 7) {
    // ------------------------------------------------------------------ publisher
    // Moves what the epilogue staged in shared memory to global memory with bulk copies, waits for
    // them to complete and only then announces them (fragment flag / finished-tile counter).
#if ACM_FFN_MX
    const bool planned = !pre || complete_plan();
#else
    constexpr bool planned = true;
#endif
    if (lane == 0) {
      uint32_t fin_n = 0;
#if !ACM_FFN_MX
      uint32_t ost_n = 0;
#endif
      bool ok = planned;
      for (int si = 0; ok && have_seg(si, true); ++si) {
        const Segment sg = seg[si];
        if (sg.phase != 1) continue;
#if !ACM_FFN_MX
        float* frag = p.frag + static_cast<size_t>(sg.p1_index) * G * 2 * kFragFloats;
        int32_t* frag_flag = p.frag_flag + sg.p1_index * G * 2;
#endif
        Sched sc(bars->plan.range[si]);
        int tile, k0, k1;
        while (ok && sc.next(tile, k0, k1)) {
         for (int h = 0; h < n_halves && ok; ++h) {          // a wide tile comes in two column halves
#if !ACM_FFN_MX
          if (k0 > 0) {
            if (!(ok = mbar_wait(smem_u32(&bars->ost_full), ost_n & 1u, quit, kSiteOutStaged))) break;
            const uint32_t bytes = static_cast<uint32_t>(min(p.n_pad - h * kMaxNodes, kMaxNodes)) * kTileM * 4u;
            // All CTAs that hold a tail part of this tile add into ONE global buffer, that of the CTA
            // which owns the tile's first chunks and will finish it.  The buffers are zero between
            // launches (the finishing CTA clears its own after reading), so nobody waits for anybody.
            const unsigned tile_begin = static_cast<unsigned>(tile) * kc1;
            int c_head = cta - 1;
            while (c_head > 0 && cut_begin(sg, c_head, p.d_grid) > tile_begin) --c_head;   // owner of the tile's first chunk
            asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;"
                         ::"l"(frag + static_cast<size_t>(c_head * 2 + h) * kFragFloats), "r"(smem_u32(ostage)), "r"(bytes) : "memory");
            bulk_commit();
            bulk_wait_all();
            red_release_add(&frag_flag[c_head * 2 + h], 1);
            mbar_arrive(smem_u32(&bars->ost_free));
            ++ost_n;
          } else
#endif
          {
            const uint32_t hb = fin_n % kHStages;
            if (!(ok = mbar_wait(smem_u32(&bars->hst_full[hb]), (fin_n / kHStages) & 1u, quit, kSiteActStaged))) break;
            const int a = static_cast<int>(fdiv(static_cast<unsigned>(sg.t0 + tile), p.d_tpe)), ti = sg.t0 + tile - a * tpe;
#if ACM_FFN_MX
            const size_t tile_at = static_cast<size_t>(a) * tpe + ti;
            bulk_store(p.hq + tile_at * (act_bytes / 2), smem_u32(hstage + hb * kHStageBytes), act_bytes / 2);
            bulk_store(p.hq_scale + tile_at * kMxActScaleBytes, smem_u32(hstage + hb * kHStageBytes) + kHPieceBytes,
                       kMxActScaleBytes);
#else
            asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];"
                         ::"l"(&hs_map), "r"(0), "r"(h * kMaxNodes), "r"(ti), "r"(a), "r"(smem_u32(hstage + hb * kHStageBytes)) : "memory");
#endif
            bulk_commit();
            bulk_wait_all();
            red_release_add(&p.ready[a], 1);
            mbar_arrive(smem_u32(&bars->hst_free[hb]));
            ++fin_n;
          }
         }
        }
      }
    }
#if ACM_FFN_MX
  } else if (warp >= 8) {
    // ------------------------------------------------------------------ unpacking warps
    // Two groups of four warps take the stages in turn.  Thread r of a group unpacks row r = lane r of tensor memory;
    // every warp stores the stage's scales, both operands', into its quarter (rows i, i + 32, i + 64, i + 96 and nodes i,
    // i + 32 in lane i; copies by tcgen05.cp instead took 260 clocks a stage out of the MMAs' pipe).  A group's next
    // record is loaded while the stage at hand is being stored, and given back behind it.
    const int r = threadIdx.x & 127, group = (warp - 8) >> 2;
    const uint32_t my_lane = static_cast<uint32_t>((warp & 3) * 32) << 16;
    bool ok = true;
    unsigned it = static_cast<unsigned>(group), total = 0;
    uint32_t ri = static_cast<uint32_t>(group), rpar = 0, s = static_cast<uint32_t>(group), par = 0;
    uint4 q[4];
    uint32_t sa[4];
    auto wait_raw = [&]() -> bool {
      return __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->raw[ri]), rpar, quit, kSitePackedStage));
    };
    auto load_raw = [&]() {
      const unsigned char* R = raw_base + static_cast<size_t>(ri) * kMxStageBytes;
      // (the record keeps the row's four 16-byte pieces rotated by the row number, so that a warp's loads
      // spread over all banks)
#pragma unroll
      for (int b = 0; b < 4; ++b) q[b] = *reinterpret_cast<const uint4*>(R + r * 64 + 16 * (b ^ ((r >> 1) & 3)));
#pragma unroll
      for (int g = 0; g < 4; ++g) sa[g] = *reinterpret_cast<const uint32_t*>(R + kMxCodeBytes + (lane + 32 * g) * 4);
    };
    auto next_raw = [&]() {
      ri += 2u;
      if (ri >= static_cast<uint32_t>(p.n_raw)) { ri -= static_cast<uint32_t>(p.n_raw); rpar ^= 1u; }
    };
    bool fetched = false;
    for (int si = 0; ok && have_seg(si, true); ++si) {
     total += bars->plan.range[si].n_stages;
     for (; it < total; it += 2) {
      if (!fetched) {
        if (!(ok = wait_raw())) break;
        load_raw();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars->raw_empty[ri]));
        next_raw();
      }
      uint32_t o[32], so[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const uint32_t words[4] = {q[b].x, q[b].y, q[b].z, q[b].w};
#pragma unroll
        for (int w = 0; w < 4; ++w) {      // the low nibbles of a word's bytes, then the high ones
          o[8 * b + 2 * w] = (words[w] << 2) & 0x3c3c3c3cu;
          o[8 * b + 2 * w + 1] = (words[w] >> 2) & 0x3c3c3c3cu;
        }
      }
      // (scale bytes above the limit, which no registered tensor holds, count as the limit)
#pragma unroll
      for (int g = 0; g < 4; ++g) so[g] = __vminu4(sa[g], 0x80808080u);
      if (!(ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->empty[s]), par ^ 1u, quit, kSiteStageEmpty)))) break;
      tc_fence_after();
      tmem_st32(tmem_base + my_lane + kAcc * kAccCols + s * kMxACols, o);
      const uint32_t sf = tmem_base + my_lane + kAcc * kAccCols + kMxA * kMxACols + s * kMxScaleCols;
      tmem_st4(sf, so[0], so[1], so[2], so[3]);
      fetched = it + 2 < total;
      {      // the next record and this stage's activations: polled side by side, one vote
        const uint32_t raw_bar = smem_u32(&bars->raw[ri]), act_bar = smem_u32(&bars->act[s]);
        bool raw_there = !fetched || mbar_try_wait(raw_bar, rpar), act_there = mbar_try_wait(act_bar, par);
        if (!raw_there) raw_there = mbar_wait_slow(raw_bar, rpar, quit, kSitePackedStage);
        if (!act_there) act_there = mbar_wait_slow(act_bar, par, quit, kSiteActStage);
        if (!(ok = __all_sync(0xffffffffu, raw_there && act_there))) break;
      }
      if (fetched) load_raw();
      const uint2* S = reinterpret_cast<const uint2*>(act_scale_base + s * 2 * kMxActScaleBytes) + lane;
      const uint2 lo = S[0], hi = S[kMxActScaleBytes / 8];      // two half-stages, two bytes of a word each
      const uint32_t s0 = __byte_perm(lo.x, hi.x, 0x5410), s1 = __byte_perm(lo.y, hi.y, 0x5410);
#pragma unroll
      for (int pc = 0; pc < kMxPieces; ++pc)      // (no scale is below 8; that of a block that is not finite has to be NaN once)
        tmem_st2(sf + 4 + 4 * pc, s0 - pc * (kMxPieceShift * 0x01010101u), s1 - pc * (kMxPieceShift * 0x01010101u));
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();                     // (the loads above have arrived, too)
      if (lane == 0) {
        mbar_arrive(smem_u32(&bars->full[s]));
        if (fetched) mbar_arrive(smem_u32(&bars->raw_empty[ri]));
      }
      if (fetched) next_raw();
      s += 2u;
      if (s >= kRing) { s -= kRing; par ^= 1u; }
     }
    }
    if (!ok) tmem_st_wait();      // (left between a stage's stores and its wait: tensor memory is released behind this)
#endif
  } else {
    // ------------------------------------------------------------------ epilogue (128 threads)
    // On-chip work only: accumulators -> registers -> shared memory.  Everything that has to reach
    // global memory and be announced to other CTAs (fragments, activation tiles) is staged in shared
    // memory and handed to the publisher warp, so these warps never sit in a memory fence.
    const int quarter = warp & 3;               // TMEM lanes this warp may read
    const int row = quarter * 32 + lane;        // accumulator row = weight-tile row
    const uint32_t lane_addr = static_cast<uint32_t>(quarter * 32) << 16;
    uint32_t f = 0, fin_count = 0;
#if !ACM_FFN_MX
    uint32_t ost_uses = 0, frag_reads = 0;
#endif
    bool ok = true, waited = !early;
#if ACM_FFN_MX
    // 32 node columns from column c on (the last 16 only if there are that many)
    auto load_32 = [&](uint32_t b, int c, int np, float (&v)[32]) {
      const uint32_t at = tmem_base + lane_addr + b * kAccCols + c;
      tmem_ld16(at, v);
      if (c + 16 < np) tmem_ld16(at + 16, v + 16);
      tmem_arrived(v);
    };
    auto release_acc = [&](uint32_t b) {
      tc_fence_before();
      mbar_arrive(smem_u32(&bars->tempty[b]));
    };
#else
    float v[kMaxNodes];
    // one half (up to 64 columns from column `cb` on) of accumulator b; the accumulator is released with its last half
    auto load_half = [&](uint32_t b, int cb, int np, bool release) {
#pragma unroll
      for (int c = 0; c < kMaxNodes; c += 16)
        if (c < np) tmem_ld16(tmem_base + lane_addr + b * kAccCols + cb + c, v + c);
      tmem_arrived(v);
      if (release) {
        tc_fence_before();
        mbar_arrive(smem_u32(&bars->tempty[b]));
      }
    };
#endif
#if !ACM_FFN_MX
    // the outgoing-fragment buffer (and the exchange buffer aliasing it) is free once the publisher
    // has copied the previous fragment out
    auto wait_ostage = [&]() -> bool {
      if (ost_uses == 0) return true;
      return epi_vote_all(mbar_wait(smem_u32(&bars->ost_free), (ost_uses - 1) & 1u, quit, kSiteOutFree));
    };
#endif
    for (int si = 0; ok && have_seg(si, true); ++si) {
      const Segment sg = seg[si];
      if (sg.phase == 1) {
        Sched sc(bars->plan.range[si]);
        int tile, k0, k1;
        while (ok && sc.next(tile, k0, k1)) {
          const uint32_t b = f % kAcc;
          // A tile this CTA will finish needs its expert's combine weights: fetch them (one L2 round
          // trip) while the tile's MMAs run, not after them.  They are the routing kernel's last output.
          float wd_mine = 0.0f;
          const int a = static_cast<int>(fdiv(static_cast<unsigned>(sg.t0 + tile), p.d_tpe));
          if (k0 == 0) {
            if (!waited) {
              griddep_wait();
              waited = true;
            }
            if (row < p.n_pad) {
              const int ex_id = bars->expert[a];      // the table row of a routed expert, 1 for a shared one
              wd_mine = ex_id >= 0 ? __ldcg(p.wtab + static_cast<size_t>(ex_id) * kWtabStride + row) : (row < p.T ? 1.0f : 0.0f);
            }
          }
          ok = epi_vote_all(mbar_wait(smem_u32(&bars->tfull[b]), (f / kAcc) & 1u, quit, kSiteAccFull));
          if (!ok) break;
          tc_fence_after();
          ++f;
          if (k0 == 0 && row < p.n_pad) bars->wd[row] = wd_mine;
          for (int h = 0; h < n_halves && ok; ++h) {
            const int cb = h * kMaxNodes;                              // first node column of this half
            const int np = min(p.n_pad - cb, kMaxNodes);               // its columns (a multiple of 16)
            // (all have read the half before out of the exchange buffer before this one is written to it)
            if (kN > kMaxNodes && h > 0 && !(ok = epi_vote_all(true))) break;
#if ACM_FFN_MX
            // The tile goes through the exchange buffer, [node][64 gate rows, 64 up rows] with the rows rotated by the
            // node, and a thread then takes up the 32 features of one node, i.e. one scale block, so that the block's
            // maximum and its packed pieces never leave the thread.  (A thread per feature, which needs a warp reduction
            // per node, took 2.7-4.6 us a tile in a rolled loop and 5-8 us unrolled -- 40 KB of instructions, fetched
            // anew through the busy L2.)
#pragma unroll 1
            for (int c = 0; c < np; c += 32) {
              float v[32];
              load_32(b, c, np, v);
              float* dst = ostage + c * kTileM;
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (j < 16 || c + 16 < np) dst[j * kTileM + (row ^ j)] = v[j];
            }
            release_acc(b);
            bool hst_ok = true;
            if (fin_count >= 1) hst_ok = mbar_wait(smem_u32(&bars->hst_free[0]), (fin_count - 1) & 1u, quit, kSiteActFree);
            ok = epi_vote_all(hst_ok);      // also orders the writes above before the reads below
            if (!ok) break;
            {
              unsigned char* hs = hstage;
              const int t = row & 63, half = row >> 6;        // this thread's node and 32 features
              if (t < np) {
                const float wgt = bars->wd[t];
                const float* gate = ostage + t * kTileM;
                uint32_t h2[16];
#pragma unroll
                for (int i = 0; i < 32; i += 2) {
                  float hval[2];
#pragma unroll
                  for (int j = 0; j < 2; ++j) {
                    // w * u * silu(g), silu(g) = g/2 * (1 + tanh(g/2))
                    const int at = 32 * half + ((i + j) ^ (t & 31));
                    const float g = gate[at], u = gate[64 + at];
                    const float hg = 0.5f * g;
                    float th;
                    asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(hg));
                    const float q = wgt * u * hg;
                    hval[j] = fmaf(q, th, q);
                  }
                  const __nv_bfloat162 pair = __floats2bfloat162_rn(hval[0], hval[1]);
                  h2[i / 2] = *reinterpret_cast<const uint32_t*>(&pair);
                }
                mx_store_block(hs, hs + kHPieceBytes, h2, t, p.n_pad, half);
              }
              fence_proxy_async_smem();
              mbar_arrive(smem_u32(&bars->hst_full[0]));
              ++fin_count;
            }
#else
            load_half(b, cb, np, h == n_halves - 1);
            if (k0 > 0) {
              // tail part of a tile whose first chunks belong to an earlier CTA: stage the fragment
              if (!(ok = wait_ostage())) break;
#pragma unroll
              for (int c = 0; c < kMaxNodes; ++c)
                if (c < np) ostage[c * kTileM + row] = v[c];
              fence_proxy_async_smem();
              mbar_arrive(smem_u32(&bars->ost_full));
              ++ost_uses;
              continue;
            }
            if (k1 < kc1) {
              // head part: the helper warp has summed the other CTAs' fragments of this tile (half) into smem
              ok = epi_vote_all(mbar_wait(smem_u32(&bars->frag_full), frag_reads & 1u, quit, kSiteFragFull));
              if (!ok) break;
#pragma unroll
              for (int c = 0; c < kMaxNodes; ++c)
                if (c < np) v[c] += sfrag[c * kTileM + row];
              mbar_arrive(smem_u32(&bars->frag_free));
              ++frag_reads;
            }
            // rows 0..63 hold gate, rows 64..127 the matching up projections.  Each pair of threads
            // (i, i+64) splits the node columns: the gate thread finishes columns [0, 32), the up
            // thread columns [32, 64); they swap the halves they do not finish through smem.
            constexpr int kHalf = kMaxNodes / 2;
            const int feat = row & 63;
            if (!(ok = wait_ostage())) break;
            if (quarter >= 2) {
#pragma unroll
              for (int c = 0; c < kHalf; ++c)
                if (c < np) ex[c * 64 + feat] = v[c];
            } else {
#pragma unroll
              for (int c = kHalf; c < kMaxNodes; ++c)
                if (c < np) ex[c * 64 + feat] = v[c];
            }
            const uint32_t hb = fin_count & 1u;
            bool hst_ok = true;
            if (fin_count >= 2) hst_ok = mbar_wait(smem_u32(&bars->hst_free[hb]), ((fin_count >> 1) - 1) & 1u, quit, kSiteActFree);
            ok = epi_vote_all(hst_ok);      // also orders the exchange writes above before the reads below
            if (!ok) break;
            {
              unsigned char* hs = hstage + hb * kHStageBytes;
              const int c0 = quarter < 2 ? 0 : kHalf;
#pragma unroll
              for (int j0 = 0; j0 < kHalf; j0 += 8) {
                if (c0 + j0 < np) {           // np is a multiple of 16: a block of 8 columns is all in or all out
                  float other[8], wgt[8], hval[8];
#pragma unroll
                  for (int j = 0; j < 8; ++j) {
                    other[j] = ex[(c0 + j0 + j) * 64 + feat];
                    wgt[j] = bars->wd[cb + c0 + j0 + j];
                  }
#pragma unroll
                  for (int j = 0; j < 8; ++j) {
                    const float mine = quarter < 2 ? v[j0 + j] : v[kHalf + j0 + j];
                    const float g = quarter < 2 ? mine : other[j];
                    const float u = quarter < 2 ? other[j] : mine;
                    // w * u * silu(g), silu(g) = g/2 * (1 + tanh(g/2))
                    const float hg = 0.5f * g;
                    float th;
                    asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(hg));
                    const float q = wgt[j] * u * hg;
                    hval[j] = fmaf(q, th, q);
                  }
                  // activation tile [node][64 features] bf16 in the 128-byte-swizzled layout of its TMA store
#pragma unroll
                  for (int j = 0; j < 8; ++j) {
                    const int t = c0 + j0 + j;
                    const int off = t * 128 + ((((feat >> 3) ^ (t & 7))) << 4) + ((feat & 7) << 1);
                    *reinterpret_cast<__nv_bfloat16*>(hs + off) = __float2bfloat16_rn(hval[j]);
                  }
                }
              }
              fence_proxy_async_smem();
              mbar_arrive(smem_u32(&bars->hst_full[hb]));
              ++fin_count;
            }
#endif
          }
        }
        if (row == 0) ACM_STAMP(10);
      } else {
        Sched sc(bars->plan.range[si]);
        int ht, k0, k1;
        while (ok && sc.next(ht, k0, k1)) {
          const uint32_t b = f % kAcc;
          ok = epi_vote_all(mbar_wait(smem_u32(&bars->tfull[b]), (f / kAcc) & 1u, quit, kSiteAccFull));
          if (!ok) break;
          tc_fence_after();
          ++f;
#if ACM_FFN_MX
#pragma unroll 1
          for (int c = 0; c < p.n_pad; c += 32) {
            float v[32];
            load_32(b, c, p.n_pad, v);
            float* dst = p.out + static_cast<size_t>(c) * p.H + static_cast<size_t>(ht) * kTileM + row;
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (c + j < p.T) atomicAdd(dst + static_cast<size_t>(j) * p.H, v[j]);
          }
          release_acc(b);
#else
          for (int h = 0; h < n_halves; ++h) {
            const int cb = h * kMaxNodes;
            load_half(b, cb, min(p.n_pad - cb, kMaxNodes), h == n_halves - 1);
            float* dst = p.out + static_cast<size_t>(cb) * p.H + static_cast<size_t>(ht) * kTileM + row;
#pragma unroll
            for (int c = 0; c < kMaxNodes; ++c)
              if (cb + c < p.T) atomicAdd(dst + static_cast<size_t>(c) * p.H, v[c]);
          }
#endif
        }
        if (row == 0) ACM_STAMP(11);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    if (__any_sync(0xffffffffu, quit->flag)) drain_cta(smem_u32(&bars->drained));
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

#if !ACM_FFN_MX
// ---------------------------------------------------------------------------------- bf16, up to 32 node columns
// The kernel above sends every activation tile through L2 to whichever CTAs take the down projection's work on that expert:
// finalise, store, announce, poll, load, about 4 us of a launch in which a small block streams for 11 us.  With few nodes
// that trip can be left out.  A unit of work here is a gate/up tile (64 features) AND its part of the down projection,
//   out[:, all H] += w * h[:, these 64 features] W_down[:, these 64 features]^T,
// by the same CTA: the activation tile goes from the epilogue into shared memory and from there into the MMAs, and no CTA
// waits for another one.  What that costs is reductions into the output: H per unit and routed node instead of about one
// output tile a CTA (an expert's combine weight is applied to them, and a node that has none takes no part).  An SM issues a
// warp's reduction in 5 clocks at best and all of them together reach 5 to 6 TB/s: 2.7 us a unit of 16 nodes, 10.8 of 64,
// beside 9 to 17 us of its weights (64 nodes of 2048 x 768, 8 / 20 / 80 experts: 44 / 53 / 123 us a layer against 31 / 44 /
// 122 with the kernel above; small_block_nodes has the line).
//   roles    warp 0 weights and hidden states, warp 1 MMAs, warps 2-9 epilogue (two teams of four: of a gate/up tile each takes
//            half the columns, of the down phase every other node), warp 10 the list behind the anchors
//   stages   gate/up: 128 rows x 128 K and the matching hidden states; down: 256 output rows x 64 features (the activations
//            are there already).  Five of them, or three (small_kernel).
//   tiles    number i of the list (anchors first, as above) to CTA i mod grid, whole.  HBM serves the CTAs in proportion to
//            what they have in flight, so one that has less to do than others keeps fewer stages in flight and all end
//            together: with 21 experts on 2048 x 768 40.4 us instead of 44.2, with 40 experts 63.8 instead of 66.0.
// What bounds it: HBM, 5.8 to 6.7 TB/s from the roles' start to the last copy.  us a layer, the kernel above -> this one, with
// 8 / 12 / 20 / 40 experts: 2048 x 768, 1 node 28.0 / 35.8 / 42.1 / 67.3 -> 21.9 / 29.1 / 38.4 / 65.5, 16 nodes 29.2 / 35.9 /
// 42.7 / 68.1 -> 24.9 / 31.4 / 39.1 / 66.0; 1024 x 512, 1 node 23.7 / 27.6 / 29.7 / 38.2 -> 16.8 / 21.2 / 24.4 / 33.1;
// 4096 x 1536, 1 node 64.7 / 80.2 / 124 / 234 -> 59.9 / 77.8 / 123 / 229, 16 nodes 66.4 / 81.2 / 124 / 238 -> 68.1 / 82.5 / 125 / 233.
constexpr int kEpiTeams = 2;                                       // of four epilogue warps
constexpr int kSmallThreads = 96 + 128 * kEpiTeams;
constexpr int kHeadStart = 16;                                     // stages of an anchor tile that are through when the rest of the list comes
template <int kN, int kR>
struct SmallGeo {
  static constexpr int kRing = kR;
  static constexpr int kStageBytes = kABytes + kAtoms * kN * kBK * 2;
  static constexpr int kSlotCols = 128;                            // columns of an accumulator slot, of kAcc
  static constexpr int kSlotTiles = kSlotCols / kN;                // output tiles of the down phase in a slot
  static constexpr int kExBytes = kN * 64 * 4;                     // gate/up exchange
  static constexpr int kHBytes = kN * 64 * 2;                      // an activation tile: [node][64 features] bf16, swizzled
};
template <int kN, int kR>
struct __align__(8) SmallBars {
  unsigned long long full[SmallGeo<kN, kR>::kRing], empty[SmallGeo<kN, kR>::kRing];
  unsigned long long tfull[kAcc], tempty[kAcc];
  unsigned long long h_full[2], h_free[2];     // epilogue -> MMAs: an activation tile is in place / MMAs -> epilogue: it has been read
  unsigned long long drained, plan_ready;
  volatile int32_t n_slots, n_routed_slots;    // length of the work list, routed experts in it (as far as it is known)
  uint32_t tmem_base;
  GiveUp give_up;
  float wd[kEpiTeams][2][kN];                  // combine weights of this and the next unit's expert
  float2 list[4 * kEpiTeams][kN];              // per epilogue warp: (weight, node) of the nodes that have one
  int32_t entry[kMaxSlots];                    // the work list, as above
  int16_t expert[kMaxSlots];
  uint32_t words[4 * kMaskWords];              // the mask the launch starts on, in 16-bit pieces (second half: blocks 4..7 of a batch)
};
template <int kN, int kR>
constexpr size_t small_smem_bytes() {
  return 1024 + static_cast<size_t>(SmallGeo<kN, kR>::kRing) * SmallGeo<kN, kR>::kStageBytes + 2 * SmallGeo<kN, kR>::kHBytes + SmallGeo<kN, kR>::kExBytes +
         sizeof(SmallBars<kN, kR>);
}
static_assert(small_smem_bytes<16, 5>() <= 232448 && small_smem_bytes<32, 5>() <= 232448, "shared memory");

template <int kN, int kR>
__global__ void __launch_bounds__(kSmallThreads, 1)
k_ffn_bf16_small(const __grid_constant__ FfnMaps maps, const __grid_constant__ CUtensorMap x_map, const FfnArgs p) {
  using Geom = SmallGeo<kN, kR>;
  constexpr int kRing = Geom::kRing, kStageBytes = Geom::kStageBytes, kSlotCols = Geom::kSlotCols, kSlotTiles = Geom::kSlotTiles;
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  unsigned char* hstage = smem + kRing * kStageBytes;
  float* ex = reinterpret_cast<float*>(hstage + 2 * Geom::kHBytes);
  SmallBars<kN, kR>* bars = reinterpret_cast<SmallBars<kN, kR>*>(hstage + 2 * Geom::kHBytes + Geom::kExBytes);
  GiveUp* const quit = &bars->give_up;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = blockIdx.x, G = gridDim.x;
  griddep_launch_dependents();
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRing; ++s) {
      mbar_init(smem_u32(&bars->full[s]), 1);
      mbar_init(smem_u32(&bars->empty[s]), 1);
    }
    for (int b = 0; b < kAcc; ++b) {
      mbar_init(smem_u32(&bars->tfull[b]), 1);
      mbar_init(smem_u32(&bars->tempty[b]), 128 * kEpiTeams);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bars->h_full[b]), 128 * kEpiTeams);
      mbar_init(smem_u32(&bars->h_free[b]), 1);
    }
    mbar_init(smem_u32(&bars->drained), 1);
    mbar_init(smem_u32(&bars->plan_ready), 1);
    bars->give_up.flag = 0;
    bars->give_up.limit_ns = p.wait_limit_ns;
    bars->give_up.status = p.status;
    bars->give_up.where = p.wait_diag ? p.wait_diag + blockIdx.x : nullptr;
    bars->give_up.tag = p.launch_tag;
    if (p.wait_diag) p.wait_diag[blockIdx.x] = p.launch_tag;      // "this CTA of that launch has started"
    fence_barrier_init();
  }
  if (warp == 0 && lane == 0) {
    prefetch_tensormap(&maps.gate_up);
    prefetch_tensormap(&maps.down);
    prefetch_tensormap(&x_map);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&bars->tmem_base), 512);
    tmem_relinquish();
  }
  // (Starts as above: on the anchors' words, on the eligible set's, or behind the kernels before.)
  const bool early = p.sel_flag != nullptr;
  const bool pre = p.anc_flag != nullptr && early;
  if (early) {
    bool timed_out = false;
    if (threadIdx.x >= 64 && threadIdx.x < 128) {
      const int j = threadIdx.x - 64;
      const uint32_t* words = pre ? p.anc_flag : p.sel_flag;
      bool seen = true;
      uint32_t bits = 0u;
      if (j < 2 * kMaskWords * p.sel_blocks)
        bits = poll_tagged_word(words + j, static_cast<uint32_t>(p.sel_epoch) & 0xffffu, p.wait_limit_ns, seen);
      timed_out = !seen;
      bits |= __shfl_xor_sync(0xffffffffu, bits, 8);
      bits |= __shfl_xor_sync(0xffffffffu, bits, 16);
      if (lane < 2 * kMaskWords) bars->words[(j >> 5) * 2 * kMaskWords + lane] = bits;
    }
    __syncthreads();
    if (timed_out) give_up(quit, pre ? kSiteAnchorWords : kSiteEligibleWords);
  } else {
    griddep_wait();
  }
  uint32_t am[kMaskWords];
  int n_first = 0;          // routed experts of the list known so far (anchor start: the anchors)
#pragma unroll
  for (int wd = 0; wd < kMaskWords; ++wd) {
    uint32_t act;
    if (early)
      act = (bars->words[2 * wd] | bars->words[2 * kMaskWords + 2 * wd]) |
            ((bars->words[2 * wd + 1] | bars->words[2 * kMaskWords + 2 * wd + 1]) << 16);
    else
      act = p.act_mask[wd];
    const uint32_t res = p.resident ? p.resident[wd] : 0xffffffffu;
    am[wd] = (p.li == 0 ? act & res : act & ~res) & p.only[wd];
    n_first += __popc(am[wd]);
  }
  static_assert(kBK * kAtoms == 128 && kTileM == 128, "SmallWalk");
  const SmallWalk walk(p.H, p.I, cta);
  const int tpe = walk.tpe, kc1 = walk.kc1, n_down = walk.n_down;
  const uint32_t b_atom_bytes = static_cast<uint32_t>(p.n_pad) * kBK * 2;
  int32_t* s_entry = bars->entry;
  // slots of the experts in m behind slot `base`, in ascending id
  auto list_experts = [&](const uint32_t (&m)[kMaskWords], int base, int e) {
    const int wd = e >> 5;
    const uint32_t mine = wd == 0 ? m[0] : wd == 1 ? m[1] : wd == 2 ? m[2] : m[3];
    if ((mine >> (e & 31)) & 1u) {
      int local = __popc(mine & ((1u << (e & 31)) - 1u));
#pragma unroll
      for (int v = 0; v < kMaskWords; ++v) local += v < wd ? __popc(m[v]) : 0;
      s_entry[base + local] = p.slot_of ? make_entry(kSrcStaged, p.slot_of[e])
                                        : p.li == 0 ? make_entry(kSrcRouted, e) : make_entry(kSrcStaged, local);
      bars->expert[base + local] = e;
    }
  };
  auto list_shared = [&](int base, int i) {
    s_entry[base + i] = make_entry(kSrcShared, i);
    bars->expert[base + i] = -1;
  };
  if (threadIdx.x < kMaxExperts) {
    list_experts(am, 0, threadIdx.x);
  } else if (p.li == 0 && !pre && static_cast<int>(threadIdx.x) - kMaxExperts < p.n_shared) {
    list_shared(n_first, threadIdx.x - kMaxExperts);
  }
  if (threadIdx.x == 0) {
    bars->n_slots = n_first + ((p.li == 0 && !pre) ? p.n_shared : 0);
    bars->n_routed_slots = n_first;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = bars->tmem_base;
  if (threadIdx.x == 0) ACM_STAMP(0);
  const int n_first_tiles = pre ? n_first * tpe : bars->n_slots * tpe;
  // Is there a tile `tile`?  With the anchor start the list behind the anchors comes later.
  int limit = n_first_tiles;
  bool more = pre;
  auto have = [&](int tile) -> bool {
    if (tile < limit) return true;
    if (!more) return false;
    more = false;
    if (!mbar_wait(smem_u32(&bars->plan_ready), 0u, quit, kSitePlanReady)) return false;
    limit = bars->n_slots * tpe;
    return tile < limit;
  };

  if (warp == 0) {
    // ------------------------------------------------------------------ weights and hidden states
    if (lane == 0) {
      const uint64_t pol_w = policy_evict_first(), pol_x = policy_evict_last();
      uint32_t s = 0, par = 0;
      bool ok = true;
      // Stages in flight, as soon as the list is known: in proportion to the stages that this CTA has left, against the one with
      // the most (of the CTAs with an anchor tile, or of the others).
      const int tile_stages = kc1 + n_down;
      auto ring_depth = [&]() -> int {
        auto left = [&](int c) {
          const int n = c < limit ? tile_stages * (static_cast<int>(fdiv(static_cast<unsigned>(limit - 1 - c), p.d_grid)) + 1) : 0;
          return pre && c < n_first_tiles ? n - min(tile_stages - 1, kHeadStart) : n;
        };
        const int most = max(left(0), left(min(n_first_tiles, G - 1)));
        const int d = (2 * kRing * left(cta) + most - 1) / (2 * most);
        return min(max(d, 2), kRing);
      };
      int depth = kRing;
      bool depth_open = true;
      if (!pre && cta < limit) depth = ring_depth();
      for (int tile = cta; ok && have(tile); tile += G) {
        const int a = static_cast<int>(fdiv(static_cast<unsigned>(tile), p.d_tpe)), ti = tile - a * tpe;
        const int32_t ent = s_entry[a];
        const int eidx = entry_idx(ent);
        const CUtensorMap* gu = pick_map(entry_src(ent), &maps.gate_up, &maps.shared_gate_up, &maps.staged_gate_up);
        const CUtensorMap* dn = pick_map(entry_src(ent), &maps.down, &maps.shared_down, &maps.staged_down);      // (slices: DownSlices)
        int kk = walk.k_first;
        if (pre && depth_open && !more) {
          depth_open = false;
          depth = ring_depth();
        }
        // (the stage `depth` back has been read: at full depth that is the one whose place this stage takes)
        auto wait_room = [&]() -> bool {
          if (more && mbar_try_wait(smem_u32(&bars->plan_ready), 0u)) {
            more = depth_open = false;
            limit = bars->n_slots * tpe;
            depth = ring_depth();
          }
          const int back = static_cast<int>(s) - depth;
          const uint32_t at = back < 0 ? back + kRing : back, at_par = back < 0 ? par ^ 1u : par;
          return mbar_wait(smem_u32(&bars->empty[at]), at_par, quit, kSiteStageEmpty);
        };
        for (int kc = 0; kc < kc1; ++kc) {
          if (!(ok = wait_room())) break;
          const uint32_t full = smem_u32(&bars->full[s]);
          const uint32_t sa = smem_u32(smem) + s * kStageBytes;
          mbar_expect_tx(full, kABytes + kAtoms * b_atom_bytes);
          tma_load_5d(sa, gu, full, 0, ti * 64, 0, kk * kAtoms, eidx, pol_w);
          tma_load_3d(sa + kABytes, &x_map, full, 0, 0, kk * kAtoms, pol_x);
          kk = walk.next_k(kk);
          if (++s == kRing) { s = 0; par ^= 1u; }
        }
        int jj = walk.j_first;
        for (int j = 0; ok && j < n_down; ++j) {
          if (!(ok = wait_room())) break;
          const uint32_t full = smem_u32(&bars->full[s]);
          mbar_expect_tx(full, kABytes);
          tma_load_4d(smem_u32(smem) + s * kStageBytes, dn, full, 0, walk.first_tile(jj) * kTileM, ti, eidx, pol_w);
          jj = walk.next_j(jj);
          if (++s == kRing) { s = 0; par ^= 1u; }
        }
      }
      if (p.stats && p.li == 0 && blockIdx.x == 0) {
        griddep_wait();
        int n_all = 0, n_stg = 0;
#pragma unroll
        for (int wd = 0; wd < kMaskWords; ++wd) {
          const uint32_t act = __ldcg(p.act_mask + wd);
          n_all += __popc(act);
          n_stg += p.resident ? __popc(act & ~p.resident[wd]) : 0;
        }
        p.stats->n_activated = n_all;
        p.stats->n_staged = n_stg;
        p.stats->n_streamed = bars->n_routed_slots;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (see above)
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem_base, 0);
    const uint32_t idesc = umma_idesc(p.n_pad);
    const uint64_t desc_hi = umma_smem_desc(0);
    const uint32_t stage0 = (smem_u32(smem) & 0x3ffffu) >> 4, h0 = (smem_u32(hstage) & 0x3ffffu) >> 4;
    uint32_t s = 0, par = 0, b = 0, bpar = 1, hb = 0, hpar = 0;
    bool ok = true;
    auto vote = [&](bool v) { return __all_sync(0xffffffffu, v); };
    for (int tile = cta; ok && vote(have(tile)); tile += G) {
      if (!(ok = vote(mbar_wait(smem_u32(&bars->tempty[b]), bpar, quit, kSiteAccEmpty)))) break;
      tc_fence_after();
      for (int kc = 0; kc < kc1; ++kc) {
        if (!(ok = vote(mbar_wait(smem_u32(&bars->full[s]), par, quit, kSiteStageFull)))) break;
        tc_fence_after();
        const uint64_t da0 = desc_hi | (stage0 + s * (kStageBytes >> 4));
        const uint64_t db0 = da0 + (kABytes >> 4);
        if (elect_one()) {
#pragma unroll
          for (int at = 0; at < kAtoms; ++at) {
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
              umma_bf16(tm + b * kSlotCols, da0 + (at * (kAtomABytes >> 4) + 2 * kk), db0 + (at * (b_atom_bytes >> 4) + 2 * kk), idesc,
                        (kc > 0 || at > 0 || kk > 0) ? 1u : 0u);
          }
          umma_commit(smem_u32(&bars->empty[s]));
          if (kc + 1 == kc1) umma_commit(smem_u32(&bars->tfull[b]));
        }
        __syncwarp();
        if (++s == kRing) { s = 0; par ^= 1u; }
      }
      if (!ok) break;
      if (++b == kAcc) { b = 0; bpar ^= 1u; }
      if (!(ok = vote(mbar_wait(smem_u32(&bars->h_full[hb]), hpar, quit, kSiteActStaged)))) break;
      tc_fence_after();
      const uint64_t dh0 = desc_hi | (h0 + hb * (Geom::kHBytes >> 4));
      for (int j = 0; j < n_down; ++j) {
        const int first = (2 * j) % kSlotTiles;      // place of the stage's first output tile in its slot
        if (first == 0) {
          if (!(ok = vote(mbar_wait(smem_u32(&bars->tempty[b]), bpar, quit, kSiteAccEmpty)))) break;
          tc_fence_after();
        }
        if (!(ok = vote(mbar_wait(smem_u32(&bars->full[s]), par, quit, kSiteStageFull)))) break;
        tc_fence_after();
        const uint64_t da0 = desc_hi | (stage0 + s * (kStageBytes >> 4));
        const bool last = j + 1 == n_down;
        const bool slot_done = first + 2 == kSlotTiles || last;
        // (rows beyond the tensor, in the last stage of an odd number of tiles, arrive as zeros)
        if (elect_one()) {
#pragma unroll
          for (int half = 0; half < 2; ++half) {
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
              umma_bf16(tm + b * kSlotCols + (first + half) * kN, da0 + (half * (kAtomABytes >> 4) + 2 * kk), dh0 + 2 * kk, idesc, kk > 0 ? 1u : 0u);
          }
          umma_commit(smem_u32(&bars->empty[s]));
          if (last) umma_commit(smem_u32(&bars->h_free[hb]));
          if (slot_done) umma_commit(smem_u32(&bars->tfull[b]));
        }
        __syncwarp();
        if (++s == kRing) { s = 0; par ^= 1u; }
        if (slot_done && ++b == kAcc) { b = 0; bpar ^= 1u; }
      }
      if (++hb == 2) { hb = 0; hpar ^= 1u; }
    }
  } else if (warp == 2 + 4 * kEpiTeams) {
    // ------------------------------------------------------------------ the list behind the anchors
    if (pre) {
      bool seen = true;
      uint32_t half = 0u;
      const uint32_t tag = static_cast<uint32_t>(p.sel_epoch) & 0xffffu;
      const int n_words = 2 * kMaskWords * p.sel_blocks;
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        const int j = lane + 32 * part;
        if (j < n_words) {
          bool got = true;
          half |= poll_tagged_word(p.sel_flag + j, tag, p.wait_limit_ns, got);
          seen = seen && got;
        }
      }
      half |= __shfl_xor_sync(0xffffffffu, half, 8);
      half |= __shfl_xor_sync(0xffffffffu, half, 16);
      const bool good = __all_sync(0xffffffffu, seen);
      uint32_t rest[kMaskWords];
      int n_rest = 0;
#pragma unroll
      for (int wd = 0; wd < kMaskWords; ++wd) {
        const uint32_t lo = __shfl_sync(0xffffffffu, half, 2 * wd), hi = __shfl_sync(0xffffffffu, half, 2 * wd + 1);
        rest[wd] = ((lo | (hi << 16)) & p.only[wd]) & ~am[wd];
        n_rest += __popc(rest[wd]);
      }
      if (good) {
        for (int e = lane; e < kMaxExperts; e += 32) list_experts(rest, n_first, e);
        if (lane < p.n_shared) list_shared(n_first + n_rest, lane);
        __syncwarp();
        if (lane == 0) {
          bars->n_routed_slots = n_first + n_rest;
          bars->n_slots = n_first + n_rest + p.n_shared;
        }
      } else if (lane == 0) {
        give_up(quit, kSiteEligibleWords);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->plan_ready));
    }
  } else {
    // ------------------------------------------------------------------ epilogue
    const int team = (warp - 2) >> 2, quarter = warp & 3, row = quarter * 32 + lane, feat = row & 63;
    const uint32_t lane_addr = static_cast<uint32_t>(quarter * 32) << 16;
    uint32_t b = 0, bpar = 0, n_tile = 0;
    bool ok = true, waited = !early;
    auto acc_wait = [&]() -> bool { return team_vote_all(team, mbar_wait(smem_u32(&bars->tfull[b]), bpar, quit, kSiteAccFull)); };
    auto acc_next = [&]() {
      tc_fence_before();
      mbar_arrive(smem_u32(&bars->tempty[b]));
      if (++b == kAcc) { b = 0; bpar ^= 1u; }
    };
    for (int tile = cta; ok && have(tile); tile += G, ++n_tile) {
      const int a = static_cast<int>(fdiv(static_cast<unsigned>(tile), p.d_tpe));
      const uint32_t hb = n_tile & 1u;
      const int ex_id = bars->expert[a];
      auto load_weight = [&]() -> float {
        return row >= p.T ? 0.0f : ex_id >= 0 ? __ldcg(p.wtab + static_cast<size_t>(ex_id) * kWtabStride + row) : 1.0f;
      };
      float wd_mine = 0.0f;
      const bool ready = waited;
      if (ready) wd_mine = load_weight();
      if (!(ok = acc_wait())) break;
      tc_fence_after();
      {
        // a team's share of the columns; the gate thread finishes the first half of them, the up thread the other
        constexpr int kCols = kN / kEpiTeams, kHalf = kCols / 2;
        const int c_team = team * kCols;
        uint32_t r[kCols];
        float v[kCols];
#pragma unroll
        for (int c = 0; c < kCols; c += 8) tmem_ld8(tmem_base + lane_addr + b * kSlotCols + c_team + c, r + c);
        tmem_arrived(r, v);
        acc_next();
        if (quarter >= 2) {
#pragma unroll
          for (int c = 0; c < kHalf; ++c) ex[(c_team + c) * 64 + feat] = v[c];
        } else {
#pragma unroll
          for (int c = kHalf; c < kCols; ++c) ex[(c_team + c) * 64 + feat] = v[c];
        }
        bool h_ok = true;
        if (n_tile >= 2) h_ok = mbar_wait(smem_u32(&bars->h_free[hb]), ((n_tile >> 1) - 1) & 1u, quit, kSiteActFree);
        if (!(ok = team_vote_all(team, h_ok))) break;
        unsigned char* hs = hstage + hb * Geom::kHBytes;
        const int c0 = c_team + (quarter < 2 ? 0 : kHalf);
#pragma unroll
        for (int j = 0; j < kHalf; ++j) {
          if (c0 + j < p.T) {
            const float other = ex[(c0 + j) * 64 + feat];
            const float mine = quarter < 2 ? v[j] : v[kHalf + j];
            const float g = quarter < 2 ? mine : other, u = quarter < 2 ? other : mine;
            // u * silu(g), silu(g) = g/2 * (1 + tanh(g/2))
            const float hg = 0.5f * g;
            float th;
            asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(hg));
            const float q = u * hg;
            const int t = c0 + j;
            *reinterpret_cast<__nv_bfloat16*>(hs + t * 128 + (((feat >> 3) ^ (t & 7)) << 4) + ((feat & 7) << 1)) =
                __float2bfloat16_rn(fmaf(q, th, q));
          }
        }
        fence_proxy_async_smem();
        mbar_arrive(smem_u32(&bars->h_full[hb]));
      }
      if (row == 0 && team == 0) ACM_STAMP(10);
      // The routing kernel's weights, which only the sums need, and the cleared output.
      if (!ready) {
        griddep_wait();
        waited = true;
        wd_mine = load_weight();
      }
      if (row < kN) bars->wd[team][hb][row] = wd_mine;
      // Every warp lists the nodes that the expert has a weight for and takes their columns alone out of the accumulators:
      // eight values at a time, kNodes nodes of all of a slot's tiles; the teams take turns.  (The list is filled up with
      // weights of zero.)
      constexpr int kNodes = 8 / kSlotTiles;
      float2* list = bars->list[warp - 2];
      int n_list = 0, jj = walk.j_first;
      for (int j0 = 0; j0 < n_down; j0 += kSlotTiles / 2) {
        if (!(ok = acc_wait())) break;
        tc_fence_after();
        if (j0 == 0) {
#pragma unroll
          for (int c = 0; c < kN; c += 32) {
            const float w = c + lane < kN ? bars->wd[team][hb][c + lane] : 0.0f;
            const unsigned has = __ballot_sync(0xffffffffu, w != 0.0f);
            if (w != 0.0f) list[n_list + __popc(has & ((1u << lane) - 1u))] = make_float2(w, __int_as_float(c + lane));
            n_list += __popc(has);
          }
          if (kNodes > 1 && lane < (-n_list & (kNodes - 1))) list[n_list + lane] = make_float2(0.0f, 0.0f);
          __syncwarp();
        }
        float* dst[kSlotTiles / 2];
        bool whole = j0 + kSlotTiles / 2 <= n_down;
        int last_at = 2 * n_down;      // (at an odd number of tiles the last stage holds one)
#pragma unroll
        for (int st = 0; st < kSlotTiles / 2; ++st) {
          dst[st] = p.out + walk.first_tile(jj) * kTileM + row;
          if (j0 + st < n_down) {
            if (walk.out_tiles(jj) == 1) { whole = false; last_at = st; }
            jj = walk.next_j(jj);
          }
        }
        const uint32_t at = tmem_base + lane_addr + b * kSlotCols;
        uint32_t nv[8];
        float v[8];
        float2 en[kNodes], ne[kNodes];
        auto fetch = [&](int q, float2 (&e)[kNodes], uint32_t (&x)[8]) {
#pragma unroll
          for (int m = 0; m < kNodes; ++m) {
            e[m] = list[q + m];
#pragma unroll
            for (int i = 0; i < kSlotTiles; ++i) tmem_ld1(at + i * kN + __float_as_int(e[m].y), x[m * kSlotTiles + i]);
          }
        };
        if (team * kNodes < n_list) fetch(team * kNodes, ne, nv);
#pragma unroll 1
        for (int q = team * kNodes; q < n_list; q += kEpiTeams * kNodes) {
          tmem_arrived(nv, v);
#pragma unroll
          for (int m = 0; m < kNodes; ++m) en[m] = ne[m];
          if (q + kEpiTeams * kNodes < n_list) fetch(q + kEpiTeams * kNodes, ne, nv);
#pragma unroll
          for (int m = 0; m < kNodes; ++m) {
            const size_t to = static_cast<size_t>(__float_as_int(en[m].y)) * p.H;
            if (kNodes == 1 || en[m].x != 0.0f) {
              if (whole) {
#pragma unroll
                for (int i = 0; i < kSlotTiles; ++i) atomicAdd(dst[i / 2] + to + (i & 1) * kTileM, en[m].x * v[m * kSlotTiles + i]);
              } else {
#pragma unroll
                for (int i = 0; i < kSlotTiles; ++i)
                  if (j0 + i / 2 < n_down && !(i / 2 == last_at && (i & 1))) atomicAdd(dst[i / 2] + to + (i & 1) * kTileM, en[m].x * v[m * kSlotTiles + i]);
              }
            }
          }
        }
        acc_next();
      }
      if (row == 0 && team == 0) ACM_STAMP(11);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    if (__any_sync(0xffffffffu, quit->flag)) drain_cta(smem_u32(&bars->drained));
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}
#endif

#if !ACM_FFN_MX
// ---------------------------------------------------------------------------------- f32 path
// A few MFLOP in L2: what counts is the chain of latencies, so both kernels are dependent launches in the fused call (the
// second one's CTAs are resident before the first is done), a warp has the loads of four rows in flight, and rows are
// read 16 bytes a lane where shapes and pointers allow (kVec).  8 nodes, 256 x 512, top-2 of 16, the whole layer:
// 22.9 -> 18.5 us a call, the binding's cheaper stream handle included; 14.8 of them are the host's launches.
constexpr int kF32Rows = 4;      // weight rows (of gate and of up; of down) a warp works on at a time

// (four products by themselves before they join the running sum: a quarter of its roundings)
__device__ __forceinline__ float dot4(const float4& a, const float4& b) {
  return fmaf(a.x, b.x, a.y * b.y) + fmaf(a.z, b.z, a.w * b.w);
}
// Four sums, one per row, over the warp's lanes: lane r < 4 returns that of row r (exchanges of two rows' halves instead of
// a full reduction per row).
__device__ __forceinline__ float reduce_rows(const float (&a)[kF32Rows], int lane) {
  const bool up2 = lane & 2, up1 = lane & 1;
  const float s0 = (up2 ? a[2] : a[0]) + __shfl_xor_sync(0xffffffffu, up2 ? a[0] : a[2], 2);
  const float s1 = (up2 ? a[3] : a[1]) + __shfl_xor_sync(0xffffffffu, up2 ? a[1] : a[3], 2);
  float v = (up1 ? s1 : s0) + __shfl_xor_sync(0xffffffffu, up1 ? s0 : s1, 1);
#pragma unroll
  for (int s = 16; s >= 4; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
  return v;
}

// h[t][j][i] = silu(g) * u for routed slot j < k (expert idx[t][j]) and shared slot j >= k.
template <bool kVec>
__global__ void __launch_bounds__(256)
k_ffn_f32_gate_up(const float* x, const float* __restrict__ gate_up,
                  const float* __restrict__ shared_gate_up, const int32_t* idx,
                  float* __restrict__ hbuf, int T, int H, int I, int E, int k, int n_shared) {
  const int slots = k + n_shared, groups = (I + kF32Rows - 1) / kF32Rows;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  griddep_wait();
  griddep_launch_dependents();      // (behind the wait: what the next kernel waits for then includes the routes)
  if (warp >= T * slots * groups) return;
  const int i0 = (warp % groups) * kF32Rows, j = (warp / groups) % slots, t = warp / (groups * slots);
  int e = j < k ? idx[t * k + j] : j - k;
  if (j < k && e >= E) e = -1;                 // an id outside the layer is an empty slot, like -1
  float g[kF32Rows] = {}, u[kF32Rows] = {};
  if (e >= 0) {
    const float* base = (j < k ? gate_up : shared_gate_up) + static_cast<size_t>(e) * 2 * I * H;
    const float* xr = x + static_cast<size_t>(t) * H;
    const float* g_row[kF32Rows];
#pragma unroll
    for (int r = 0; r < kF32Rows; ++r) g_row[r] = base + static_cast<size_t>(min(i0 + r, I - 1)) * H;
    const size_t to_up = static_cast<size_t>(I) * H;
    if constexpr (kVec) {
#pragma unroll 2
      for (int hh = 4 * lane; hh < H; hh += 128) {
        const float4 xv = *reinterpret_cast<const float4*>(xr + hh);
#pragma unroll
        for (int r = 0; r < kF32Rows; ++r) {
          const float4 gv = *reinterpret_cast<const float4*>(g_row[r] + hh), uv = *reinterpret_cast<const float4*>(g_row[r] + to_up + hh);
          g[r] += dot4(gv, xv);
          u[r] += dot4(uv, xv);
        }
      }
    } else {
      for (int hh = lane; hh < H; hh += 32) {
        const float xv = xr[hh];
#pragma unroll
        for (int r = 0; r < kF32Rows; ++r) {
          g[r] = fmaf(g_row[r][hh], xv, g[r]);
          u[r] = fmaf(g_row[r][to_up + hh], xv, u[r]);
        }
      }
    }
  }
  const float gs = reduce_rows(g, lane), us = reduce_rows(u, lane);
  if (lane < kF32Rows && i0 + lane < I)
    hbuf[(static_cast<size_t>(t) * slots + j) * I + i0 + lane] = e >= 0 ? (gs / (1.0f + expf(-gs))) * us : 0.0f;
}

template <bool kVec>
__global__ void __launch_bounds__(256)
k_ffn_f32_down(const float* __restrict__ down, const float* __restrict__ shared_down, const int32_t* idx, const float* w,
               const float* hbuf, float* __restrict__ out, int T, int H, int I, int E, int k, int n_shared) {
  const int slots = k + n_shared, groups = (H + kF32Rows - 1) / kF32Rows;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  griddep_launch_dependents();
  griddep_wait();
  if (warp >= T * groups) return;
  const int h0 = (warp % groups) * kF32Rows, t = warp / groups;
  // the node's experts and weights, a lane per slot (at most kMaxTopK + kMaxShared)
  int my_e = -1;
  float my_w = 1.0f;
  if (lane < slots) {
    my_e = lane < k ? idx[t * k + lane] : lane - k;
    if (lane < k) {
      my_w = w[t * k + lane];
      if (my_e >= E) my_e = -1;
    }
  }
  float y = 0.f;
#pragma unroll 2
  for (int j = 0; j < slots; ++j) {
    const int e = __shfl_sync(0xffffffffu, my_e, j);
    if (e < 0) continue;
    const float* base = (j < k ? down : shared_down) + static_cast<size_t>(e) * H * I;
    const float* hr = hbuf + (static_cast<size_t>(t) * slots + j) * I;
    float acc[kF32Rows] = {};
    if constexpr (kVec) {
#pragma unroll 4
      for (int i = 4 * lane; i < I; i += 128) {
        const float4 hv = *reinterpret_cast<const float4*>(hr + i);
#pragma unroll
        for (int r = 0; r < kF32Rows; ++r) {
          const float4 dv = *reinterpret_cast<const float4*>(base + static_cast<size_t>(min(h0 + r, H - 1)) * I + i);
          acc[r] += dot4(dv, hv);
        }
      }
    } else {
      for (int i = lane; i < I; i += 32) {
        const float hv = hr[i];
#pragma unroll
        for (int r = 0; r < kF32Rows; ++r) acc[r] = fmaf(base[static_cast<size_t>(min(h0 + r, H - 1)) * I + i], hv, acc[r]);
      }
    }
    y = fmaf(__shfl_sync(0xffffffffu, my_w, j), reduce_rows(acc, lane), y);
  }
  if (lane < kF32Rows && h0 + lane < H) out[static_cast<size_t>(t) * H + h0 + lane] = y;
}

#endif   // !ACM_FFN_MX

}  // namespace

#if ACM_FFN_MX
namespace {
// Packed records in flight in a launch of n_pad node columns.
int mx_raw_stages(int n_pad) {
  return min(kMaxRaw, (kMxRingBytes - kMxA * (n_pad * (kMxPieces * 128) + 2 * kMxActScaleBytes)) / kMxStageBytes);
}
}  // namespace
cudaError_t ffn_mx_configure() {
  return cudaFuncSetAttribute(ACM_FFN_KERNEL<kMaxNodes>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(Geo<kMaxNodes>::kSmemBytes));
}
cudaError_t launch_ffn_mxfp4(const FfnLaunch& L, cudaStream_t s) {
#else

namespace {
// The small blocks' kernel for a launch.  Up to 1152 hidden features with three stages (120 KB): a CTA of the next call's router
// kernel then fits beside it and has its weights by the time this launch is done, which such short launches gain more from than
// from stages in flight.  Three stages against five, mean / highest over 13 sets of 4 to 40 experts, 1 to 16 nodes, inter 512 to 1408:
// hidden 768 0.92 to 0.98 / 1.02, 1024 0.91 to 0.99 / 1.05, 1152 0.92 to 0.99 / 1.04; beyond the line 1280 0.93 to 0.99 / 1.05, 1536
// 0.96 to 1.00 / 1.06.  us a layer, five -> three, with 8 / 21 / 40 experts: 1024 x 512, 1 node 17.0 / 24.4 / 33.7 -> 15.4 / 22.8 / 31.6;
// 1024 x 1408, 16 nodes 29.2 / 40.1 / 63.3 -> 26.1 / 39.1 / 62.0; 2048 x 768, 1 node 21.3 / 39.4 / 64.0 -> 22.3 / 41.8 / 66.4.
// (Six stages: 22.1 / 40.6 / 67.4 there.  The router kernel's CTAs without their request for 104 KB, so that they fit beside five
// stages: they pile up on the SMs that are free first, 22.7 / 42.3 / 66.7.)
struct SmallKernel {
  const void* fn;
  size_t smem;
};
SmallKernel small_kernel(int n_pad, int hidden) {
  if (n_pad > 16) return {reinterpret_cast<const void*>(k_ffn_bf16_small<kSmallNodes, 5>), small_smem_bytes<kSmallNodes, 5>()};
  if (hidden <= 1152) return {reinterpret_cast<const void*>(k_ffn_bf16_small<16, 3>), small_smem_bytes<16, 3>()};
  return {reinterpret_cast<const void*>(k_ffn_bf16_small<16, 5>), small_smem_bytes<16, 5>()};
}
}  // namespace
cudaError_t ffn_configure() {
  cudaError_t err = cudaFuncSetAttribute(ACM_FFN_KERNEL<kMaxNodes>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(Geo<kMaxNodes>::kSmemBytes));
  if (err != cudaSuccess) return err;
  for (const SmallKernel& k : {small_kernel(16, 128), small_kernel(16, 2048), small_kernel(kSmallNodes, 128)}) {
    err = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(k.smem));
    if (err != cudaSuccess) return err;
  }
  return cudaFuncSetAttribute(ACM_FFN_KERNEL<kWideNodes>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(Geo<kWideNodes>::kSmemBytes));
}

cudaError_t launch_ffn_bf16(const FfnLaunch& L, const FfnMaps& maps, const CUtensorMap& x_map,
                            const CUtensorMap& h_map, const CUtensorMap& hs_map, cudaStream_t s) {
#endif
  {
    // the schedules count (tile, K-chunk) units times the grid in 32 bits
    const unsigned long long u1 = static_cast<unsigned long long>(kMaxSlots) * (L.I / 64) * (L.H / (kBK * kAtoms));
    const unsigned long long u2 = static_cast<unsigned long long>(L.H / kTileM) * kMaxSlots * ((L.I / 64 + kAtoms - 1) / kAtoms);
    if ((u1 > u2 ? u1 : u2) * (static_cast<unsigned long long>(L.grid) + 1) >= (1ull << 32)) return cudaErrorInvalidValue;
  }
  FfnArgs a;
  {
    const int tpe = L.I / 64;
    a.d_grid = make_fastdiv(static_cast<unsigned>(L.grid));
    a.d_kc1 = make_fastdiv(static_cast<unsigned>(L.H / (kBK * kAtoms)));
    a.d_tpe = make_fastdiv(static_cast<unsigned>(tpe));
    a.d_kpe = make_fastdiv(static_cast<unsigned>((tpe + kAtoms - 1) / kAtoms));
  }
  a.T = L.T; a.H = L.H; a.I = L.I; a.n_pad = L.n_pad;
  a.act_mask = L.act_mask; a.resident = L.resident; a.li = L.li; a.n_shared = L.n_shared; a.slot_of = L.slot_of; a.wtab = L.wtab;
  for (int w = 0; w < 4; ++w) a.only[w] = L.only[w];
  a.stats = L.stats; a.ready = L.ready;
  a.sel_flag = L.sel_flag; a.sel_epoch = L.sel_epoch; a.sel_blocks = L.sel_blocks;
  a.anc_flag = (L.sel_blocks < 1 || L.sel_blocks > kMaxEarlyBlocks || L.li != 0 || L.resident || L.slot_of) ? nullptr : L.anc_flag;
  a.out = L.out; a.status = L.status; a.trace = L.trace;
  a.wait_limit_ns = L.wait_limit_ns; a.wait_diag = L.wait_diag; a.launch_tag = L.launch_tag;
#if ACM_FFN_MX
  if (!L.mx_gate_up || !L.mx_down || L.I % 128 != 0 || L.n_shared != 0) return cudaErrorInvalidValue;
  a.mx_gate_up = static_cast<const unsigned char*>(L.mx_gate_up);
  a.mx_down = static_cast<const unsigned char*>(L.mx_down);
  if (!L.xq || L.n_pad > kMaxNodes) return cudaErrorInvalidValue;
  a.xq = static_cast<const unsigned char*>(L.xq);
  a.xq_scale = a.xq + mx_act_scale_offset(L.H);
  a.xq_count = L.xq_count; a.xq_target = L.xq_target;
  // (a slot's share of the activation buffer is 256 I bytes: up to 192 I of pieces; the scales lie behind all pieces)
  a.hq = static_cast<unsigned char*>(L.hbuf);
  a.hq_scale = a.hq + static_cast<size_t>(kMaxSlots) * (kMxPieces * 64) * L.I;
  a.n_raw = mx_raw_stages(L.n_pad);
  void* args[] = {&a};
#else
  a.frag = L.frag; a.frag_flag = L.frag_flag;
  void* args[] = {const_cast<FfnMaps*>(&maps), const_cast<CUtensorMap*>(&x_map), const_cast<CUtensorMap*>(&h_map),
                  const_cast<CUtensorMap*>(&hs_map), &a};
#endif
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(L.grid);
  cfg.blockDim = dim3(kThreads);
#if ACM_FFN_MX
  if (L.n_pad > kMaxNodes) return cudaErrorInvalidValue;
  const bool wide = false;
#else
  const bool wide = L.n_pad > kMaxNodes;       // a batch with more than 64 nodes: 128-column accumulators
  if (L.n_pad > kWideNodes) return cudaErrorInvalidValue;
#endif
  cfg.dynamicSmemBytes = wide ? Geo<kWideNodes>::kSmemBytes : Geo<kMaxNodes>::kSmemBytes;
#if !ACM_FFN_MX
  const bool small = small_block(L.T, L.H, L.I, L.n_shared);
  void* small_args[] = {const_cast<FfnMaps*>(&maps), const_cast<CUtensorMap*>(&x_map), &a};
  if (small) {
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = small_kernel(L.n_pad, L.H).smem;
  }
#endif
  cfg.stream = s;
  // The CTAs wait on one another, so all of them must be resident: one CTA per SM on an otherwise
  // idle GPU is, and a cooperative launch makes the driver check it.  A dependent launch cannot be
  // cooperative (its CTAs trickle in behind the previous kernel's); there the waits' limits, which
  // end in an error status instead of a hang, are the guard.
  cudaLaunchAttribute attr[1];
  if (L.pdl) {
    set_pdl_attr(&attr[0]);
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = 1;
#if ACM_FFN_MX
  return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(ACM_FFN_KERNEL<kMaxNodes>), args);
#else
  if (small) return cudaLaunchKernelExC(&cfg, small_kernel(L.n_pad, L.H).fn, small_args);
  return cudaLaunchKernelExC(&cfg, wide ? reinterpret_cast<const void*>(ACM_FFN_KERNEL<kWideNodes>)
                                        : reinterpret_cast<const void*>(ACM_FFN_KERNEL<kMaxNodes>), args);
#endif
}

#if !ACM_FFN_MX
cudaError_t launch_ffn_f32(const float* x, const float* gate_up, const float* down,
                           const float* shared_gate_up, const float* shared_down, int n_shared,
                           const int32_t* idx, const float* w, float* hbuf, float* out, int T, int H,
                           int I, int E, int k, bool pdl, cudaStream_t s) {
  const int slots = k + n_shared;
  auto aligned = [](const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; };
  const bool vec = H % 4 == 0 && I % 4 == 0 && aligned(x) && aligned(gate_up) && aligned(down) && aligned(hbuf) &&
                   (n_shared == 0 || (aligned(shared_gate_up) && aligned(shared_down)));
  cudaLaunchAttribute attr[1];
  set_pdl_attr(attr);
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  auto blocks = [](long long warps) { return dim3(static_cast<unsigned>((warps * 32 + 255) / 256)); };
  cfg.gridDim = blocks(static_cast<long long>(T) * slots * ((I + kF32Rows - 1) / kF32Rows));
  cudaError_t err = cudaLaunchKernelEx(&cfg, vec ? k_ffn_f32_gate_up<true> : k_ffn_f32_gate_up<false>, x, gate_up, shared_gate_up,
                                       idx, hbuf, T, H, I, E, k, n_shared);
  if (err != cudaSuccess) return err;
  cfg.gridDim = blocks(static_cast<long long>(T) * ((H + kF32Rows - 1) / kF32Rows));
  return cudaLaunchKernelEx(&cfg, vec ? k_ffn_f32_down<true> : k_ffn_f32_down<false>, down, shared_down, idx, w,
                            static_cast<const float*>(hbuf), out, T, H, I, E, k, n_shared);
}

#endif   // !ACM_FFN_MX

}  // namespace acm

#if !ACM_FFN_MX
// ------------------------------------------------------------------------------------------------
// Allocation-free variant of the f32 expert FFN.  The per-(node, slot) intermediate activations that
// the context-based call keeps in its cudaMalloc'ed workspace live here in a fixed array that is part
// of the library image, so the call never allocates.
// ------------------------------------------------------------------------------------------------
namespace {
constexpr size_t kNoAllocScratchFloats = ACM_NOALLOC_MAX_FLOATS;
static __device__ __align__(256) float g_noalloc_scratch[kNoAllocScratchFloats];

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mutex;
float* g_noalloc_ptr[kNoAllocMaxDevices];   // device address of the array above, per device (0 = not looked up yet)
}  // namespace

extern "C" acm_status acm_expert_ffn_f32_noalloc(const float* x, int T, int hidden, int inter, int n_experts, int top_k,
                                                 const int32_t* idx, const float* w, const float* w_gate_up,
                                                 const float* w_down, float* out, acm_stream stream) {
  if (!x || !idx || !w || !w_gate_up || !w_down || !out) return ACM_ERR_INVALID;
  if (T < 1 || hidden < 1 || inter < 1 || n_experts < 1 || top_k < 1 || top_k > n_experts) return ACM_ERR_INVALID;
  if (T > acm::kMaxNodes || top_k > acm::kMaxTopK || n_experts > acm::kMaxExperts) return ACM_ERR_UNSUPPORTED;
  // the scratch holds one float per (node, slot, intermediate feature): refuse what does not fit
  if (static_cast<size_t>(T) * top_k * inter > kNoAllocScratchFloats) return ACM_ERR_UNSUPPORTED;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return ACM_ERR_CUDA;
  if (dev < 0 || dev >= kNoAllocMaxDevices) return ACM_ERR_UNSUPPORTED;
  float* scratch = nullptr;
  {
    // First call on this device: ask the runtime where this device's copy of the array lives.  In host
    // code the array's name is only a handle; a kernel must be given the address obtained here.
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return ACM_ERR_CUDA;
      g_noalloc_ptr[dev] = static_cast<float*>(p);
    }
    scratch = g_noalloc_ptr[dev];
  }
  const cudaError_t err = acm::launch_ffn_f32(x, w_gate_up, w_down, nullptr, nullptr, 0, idx, w, scratch, out, T, hidden,
                                              inter, n_experts, top_k, false, static_cast<cudaStream_t>(stream));
  return err == cudaSuccess ? ACM_OK : ACM_ERR_CUDA;
}
#endif   // !ACM_FFN_MX
