// FP8 GEMM for sm_100a: D[M,N] = (A[M,Kc] . B[N,Kc]^T) * alpha, A and B bytes (E4M3 or E5M2, mixed freely), each
// stored contraction-major ([rows, Kc]) or MN-major ([Kc, rows]: the transposed view of a row-major tensor, read by the
// tensor cores directly), FP32 accumulation in tensor memory.
//
// Structure: persistent clusters of two CTAs on neighbouring SMs, 320, 352 or 384 threads each, that compute one tile of 256 rows
// and 256, 128 or 64 columns together with tcgen05.mma.cta_group::2:
//   warp 0      TMA producer: cp.async.bulk.tensor boxes into a shared-memory ring (six stages of a 128-byte K block, or four
//               of two blocks for tiles of 128 or 64 columns); each CTA loads its own 128 rows of A and its own half of the
//               tile's B rows
//   warp 1      allocates tensor memory, then one elected lane of the even CTA issues tcgen05.mma (256 x tile_n x 32 per
//               instruction) and tcgen05.commit, which multicasts stage-free / accumulator-ready arrivals to both CTAs
//   8 warps     epilogue: tcgen05.ld the CTA's 128 x tile_n FP32 accumulator (two warps per 32-lane quadrant, half of
//               the columns each) in 32 x 32 blocks, scale, write each block into a swizzled per-warp shared-memory
//               tile and hand it to the bulk-store unit: a bulk tensor store for bf16 (+ max|D| reduced by warp
//               shuffles, one atomicMax per warp and tile) and for FP32 overwrite; a bulk tensor reduction (.add) for
//               FP32 accumulation straight into the destination (direct gradient placement): the addition is done in
//               L2, one per element and launch, and the destination tile is prefetched into L2 while the tile's
//               main loop runs.  The reduction is a plain round-to-nearest FP32 addition (subnormal values kept).
//   The launch may also carry up to fifty-six independent problems (grouped launch): tiles are numbered problem after
//   problem and a warp of its own tells the roles what each tile is, so that one set of persistent CTAs packs them all.
//   A problem may be the sum of several products (the deferred weight gradients of several microbatches): each gets an
//   accumulator of its own, the epilogue adds them up in registers, and a warp of its own stores the result.
//   A launch of one GEMM with an odd number of 128-row tiles may run without clusters, a CTA to a tile of 128 x 256
//   (gemm_fp8_kernel: the same roles, four stages of 128 rows of A and 256 of B, tcgen05.mma.cta_group::1; see one_cta).
// Rows beyond M (M is a multiple of 128; a pair's tile has 256) are read as zeros by TMA and never stored.
// Scale commits (fold a pending amax into its history, update the scale) ride along, so that no extra launch is needed:
// classes whose amax an earlier kernel completed (X of a forward, G of an input gradient) are committed by an idle
// epilogue warp while the first tile is being computed; only the class the epilogue itself reduces (Y) waits for the
// last CTA to finish.  With all of them in the tail, every launch of a chain of sixteen 1024 x 1024 linears (T = 512)
// ended with a ticket and a chain of dependent loads: 3270 us per step, 2979 us with the early commits.
// Two accumulators (2 x 256 tensor-memory columns) let the epilogue of tile i overlap the main loop of tile i+1.
//
// No TMA multicast is used.
// Each output element is produced by exactly one thread with a fixed contraction order and reaches its destination
// by exactly one store or one addition per launch, so results do not depend on the grid size or on how tiles are
// scheduled, nor on how wide they are or how many CTAs compute one (no split-K; launches that add to the same destination are ordered by their stream).
//
// Every wait on an mbarrier is bounded by a clock budget; on expiry the thread ORs an error bit into the status
// word, raises a CTA-wide abort flag that all other waits observe, and the CTA falls through to its common exit
// where tensor memory is released.
#include <cuda_bf16.h>
#include <type_traits>
#include <cuda_fp8.h>

#include <cstddef>
#include <cstring>

#include "commit.cuh"
#include "kernels.h"
#include "tile_count.h"

namespace qe {
namespace {

constexpr uint32_t BM = 128, BK = 128;  // rows per CTA; bytes (= FP8 elements) per stage along the contraction
constexpr uint32_t ACC_COLS = 256;      // tensor-memory columns between the two accumulators (the widest tile)
constexpr uint32_t UMMA_K = 32;
constexpr uint32_t A_BYTES = BM * BK;
// CTAs that work on one tile, and what follows from it.
template <bool PAIR>
struct Form {
  static constexpr uint32_t CTAS = PAIR ? 2 : 1;
  static constexpr uint32_t TILE_M = CTAS * BM;  // rows of D per tile
};
// The ring of operand stages: A and this CTA's rows of B, for one K block of 128 bytes (tiles of 256 columns) or two of them
// (narrower tiles of a pair).  A stage costs the producer about 270 clocks and the issuer of the MMAs about 130 whatever its size
// (barrier operations; 45 to 90 for another load), while the MMAs of a K block take 240 to 260 clocks at up to 128 columns: with
// stages of one K block, tiles of 64 columns ran at 387 clocks a block, now at 339 (256 x 2048 x 8192: 15.9 -> 14.1 us).  There
// shared memory bounds them: 20 KB written and 20 to 24 KB read a block at 128 bytes a clock.
constexpr uint32_t EPI_BUF_BYTES = 4096;                     // per epilogue warp: one FP32 or two bf16 32 x 32 output tiles
                                                             // (1 KB-aligned, swizzled) that the bulk-store unit reads
constexpr uint32_t RING_AND_BUFS = 14 * A_BYTES;
constexpr int MAX_STAGES = 6;
template <bool PAIR, uint32_t BUFS>
struct Ring {
  static constexpr uint32_t BYTES = RING_AND_BUFS - 8 * BUFS * EPI_BUF_BYTES;
  uint32_t blocks, stages, stage_bytes;  // K blocks of a stage, stages, bytes of one
  __device__ __forceinline__ explicit Ring(uint32_t tile_n)
      : blocks(PAIR && tile_n < 256u ? 2u : 1u),
        stages(PAIR && tile_n == 256u ? BYTES / (2 * A_BYTES) : BYTES / (3 * A_BYTES)),
        stage_bytes(PAIR && tile_n == 256u ? 2 * A_BYTES : 3 * A_BYTES) {}
  __device__ __forceinline__ uint32_t b_offset() const { return blocks * A_BYTES; }
};
static_assert(2 * A_BYTES + 2 * 64 * BK <= 3 * A_BYTES && Ring<true, 1>::BYTES / (2 * A_BYTES) <= MAX_STAGES, "");
constexpr uint32_t TMEM_COLS = 512;
constexpr int EPI_WARPS = 8, EPI_THREADS = EPI_WARPS * 32;
// Threads of a CTA: warps 0 and 1, then the epilogue's eight, and where a launch has several problems one for the tile records.
// The variant that sums several products keeps a tile row of 128 FP32 per epilogue thread: its epilogue warps are two whole
// warpgroups (warps 2 and 3 make records and store results), which take over registers that the first warpgroup hands back
// (launched with 168 a thread; 56 + 2 * 224 <= 3 * 168).
constexpr int threads_of(bool sums, bool several) { return sums ? 384 : several ? 352 : 320; }
static_assert(EPI_WARPS == 8, "shared-memory budget below assumes 8 epilogue warps");
// Launches of several problems: what the roles need to know of a tile is put into a small ring of records by a warp of its own,
// some tiles ahead.  Looked up by each role, it is a chain of reads of the parameter block, which no constant cache holds: 800
// to 2300 clocks a tile and role, where the MMAs of a tile of eight K blocks take 4100 (the records: 300 to 450).
constexpr uint32_t INFO_SLOTS = 4, INFO_BYTES = 128;
constexpr uint32_t BARS_BYTES = 512;
// (What the SM has left has to hold a block of the casts that run beside these launches: 1 KB that the system takes and 36 bytes.)
constexpr uint32_t SMEM_BYTES = RING_AND_BUFS + BARS_BYTES /*barriers, flags*/ + INFO_SLOTS * INFO_BYTES;
static_assert(SMEM_BYTES + 1024 + 2048 <= 228 * 1024, "no room for a cast beside a GEMM launch");
constexpr long long WAIT_BUDGET_CYCLES = 4000000000ll;  // ~2 s at the maximum SM clock

constexpr uint32_t ERR_PRODUCER = 1u, ERR_MMA = 2u, ERR_EPILOGUE = 4u;

// ------------------------------------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false if the budget ran out or another thread of the CTA already gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                          uint32_t* status, uint32_t err_bit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (clock64() - t0 > WAIT_BUDGET_CYCLES) {
      *abort_flag = 1u;
      atomicOr(status, err_bit);
      return false;
    }
  }
}

// The same wait by a whole warp (converged), as every role makes it.  Its lanes leave it together and with one answer: in the
// roles that issue from an elected lane, a lane that was still polling while that one went on could find the barrier a phase
// further, take that for the phase it waits for not being over, and wait on; and where one lane gives up (the launch is being
// abandoned) while another finds the phase complete, the warp may not go on to its next aligned instruction in parts.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t* status,
                                               uint32_t err_bit) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, status, err_bit));
}

// Whether `count` CTAs have said that they have stored their part of some rows (chained problems).  What they stored is then there for
// bulk loads too.
__device__ __forceinline__ bool rows_there(const uint32_t* done, uint32_t count) {
  const bool there = ld_acquire(done) >= count;
  asm volatile("fence.proxy.async;" ::: "memory");
  return __all_sync(0xffffffffu, there);
}

// Wait of a warp until they have, bounded like the others.
__device__ __forceinline__ bool rows_wait(const uint32_t* done, uint32_t count, volatile uint32_t* abort_flag, uint32_t* status) {
  const long long t0 = clock64();
  bool there = ld_acquire(done) >= count;
  while (!there) {
    there = ld_acquire(done) >= count;
    if (there || *abort_flag) break;
    if (clock64() - t0 > WAIT_BUDGET_CYCLES) {
      *abort_flag = 1u;
      atomicOr(status, ERR_PRODUCER);
      break;
    }
  }
  asm volatile("fence.proxy.async;" ::: "memory");
  return __all_sync(0xffffffffu, there);
}

// ... and how they say it: the last warp of a CTA to have stored its part (last_of_tile), for all of them.  (By an addition of
// each warp's own, behind a fence of each lane, sixteen linears of 1024 x 1024 at 512 tokens took 1636 us a step; 1500 now.)
__device__ __forceinline__ uint32_t add_acq_rel_cta(uint32_t* count /* shared */) {
  uint32_t before;
  asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(before) : "r"(smem_u32(count)) : "memory");
  return before;
}
// Whether a CTA is the last of the grid to say so.  What any of them did before is visible to who learns that it is.
__device__ __forceinline__ bool last_of_grid(uint32_t* ticket, uint32_t ctas) {
  uint32_t before;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(before) : "l"(ticket) : "memory");
  if (before != ctas - 1) return false;
  *ticket = 0u;  // ready for the next kernel that uses it
  return true;
}
__device__ __forceinline__ void add_release(uint32_t* p, uint32_t v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Of a role that loads into shared memory, when the launch is being abandoned: gives copies already in flight a bounded chance to
// land before the CTA's shared memory goes away.
__device__ __forceinline__ void let_copies_land() {
  const long long t0 = clock64();
  while (clock64() - t0 < 2000000ll) { }
}

// Arrival on a barrier that may live in the peer CTA.  What it announces are tensor-memory reads, ordered by the
// tcgen05 fences on both sides, so it need not be a release at cluster scope: that waits for the thread's outstanding
// stores too, ~1000 clocks per drained accumulator.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Address of the same shared-memory location in CTA `rank` of the cluster (shared::cluster window).
__device__ __forceinline__ uint32_t map_to_cta(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// TMA load of a box of an operand; in a pair its completion may be credited to a barrier of the peer CTA.
template <bool PAIR>
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, int c3) {
  if (PAIR)
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cta.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
// One lane of a converged warp, the same one every time.  The producer's and the issuer's loops run on whole warps, so that
// addresses and descriptors stay in uniform registers, and this lane issues: on one lane of a divergent warp the same loops
// took 65 clocks an MMA instead of 48 (64 columns) and twice as long a load (8192 x 256 x 2048: 21.1 us, now 15.9).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {  // arrives on `bar` in both CTAs of the pair
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"((uint16_t)3)
               : "memory");
}
__device__ __forceinline__ void tc_mma_f8_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tc_commit_one(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma_f8_one(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                              uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
template <bool PAIR>
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  if (PAIR) tc_commit_pair(bar);
  else tc_commit_one(bar);
}
template <bool PAIR>
__device__ __forceinline__ void tc_mma_f8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  if (PAIR) tc_mma_f8_pair(d_tmem, adesc, bdesc, idesc, accumulate);
  else tc_mma_f8_one(d_tmem, adesc, bdesc, idesc, accumulate);
}

// Load of a 32 x 32 block of an output.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
               ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1)
               : "memory");
}

__device__ __forceinline__ void tma_prefetch(const CUtensorMap* map, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile [%0, {%1, %2, %3, %4}];" ::"l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}

// Bulk tensor store of a shared-memory tile (issued by one lane), with group tracking.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
               ::"l"(map), "r"(c0), "r"(c1), "r"(src)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Bulk tensor reduction: global tile += shared-memory tile, added element by element where the data lives (L2).
__device__ __forceinline__ void tma_reduce_add_2d(const CUtensorMap* map, uint32_t src, int c0, int c1) {
  asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2}], [%3];"
               ::"l"(map), "r"(c0), "r"(c1), "r"(src)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void tma_store_wait_read() {  // at most N groups may still be reading shared memory
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: start address (>>4) in bits 0-13; leading byte offset (>>4) in bits 16-29: from one swizzle
// atom of an MN-major tile's rows to the next, 1 (unused) where there is only one; the high word (stride byte offset >>4 in bits 32-45, descriptor version 1 in bits
// 46-47, swizzle mode in bits 61-63) comes from the host: desc_hi() below.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t hi, uint32_t leading = 1u) {
  return (uint64_t)((saddr & 0x3ffffu) >> 4) | ((uint64_t)leading << 16) | ((uint64_t)hi << 32);
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// One row of a 32 x 32 FP32 tile for the bulk-store unit: 128-byte rows, 128-byte swizzle (chunk c of row r sits at
// c ^ (r & 7)).
__device__ __forceinline__ void st_tile_f32(uint32_t buf, uint32_t row, const float (&v)[32]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const uint32_t dst = buf + row * 128u + (((uint32_t)c ^ (row & 7u)) << 4);
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "f"(v[4 * c]), "f"(v[4 * c + 1]), "f"(v[4 * c + 2]),
                 "f"(v[4 * c + 3])
                 : "memory");
  }
}

// Two FP32 values at a time.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(uint32_t lo, uint32_t hi) {
  f32x2 v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(lo), "r"(hi));
  return v;
}
// a * b, rounded by itself.  (Written as mul.rn, ptxas makes a multiply-add of it and the addition that follows, which rounds
// once.  So it is one already, with a -0 that ptxas cannot see: that changes no product, not even the sign of a zero.)
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b, f32x2 minus_zero) {
  f32x2 v;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(minus_zero));
  return v;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 v;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}
__device__ __forceinline__ void st_tile_f32x2(uint32_t buf, uint32_t row, const f32x2 (&v)[16]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const uint32_t dst = buf + row * 128u + (((uint32_t)c ^ (row & 7u)) << 4);
    asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(dst), "l"(v[2 * c]), "l"(v[2 * c + 1]) : "memory");
  }
}
__device__ __forceinline__ void ld_tile_f32x2(uint32_t buf, uint32_t row, f32x2 (&v)[16]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const uint32_t src = buf + row * 128u + (((uint32_t)c ^ (row & 7u)) << 4);
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v[2 * c]), "=l"(v[2 * c + 1]) : "r"(src) : "memory");
  }
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);  // .x = a in the low half
  return *reinterpret_cast<uint32_t*>(&v);
}

// Tile order.  The CTAs running at the same time take consecutive tiles.  Walking the dimension of the SMALLER
// operand fastest means that operand is swept again and again (from L2, where it fits) while the larger one is
// streamed from HBM once.
template <uint32_t TILE_M>
__device__ __forceinline__ void tile_coords(uint32_t tile, uint32_t tiles_m, uint32_t tiles_n, bool m_fastest,
                                            uint32_t tile_n, uint32_t& m0, uint32_t& n0) {
  if (m_fastest) {
    m0 = (tile % tiles_m) * TILE_M;
    n0 = (tile / tiles_m) * tile_n;
  } else {
    n0 = (tile % tiles_n) * tile_n;
    m0 = (tile / tiles_n) * TILE_M;
  }
}

__device__ __forceinline__ void epi_bar_sync() { asm volatile("bar.sync 1, %0;" ::"n"(EPI_THREADS) : "memory"); }

// High word of the descriptor of a tile whose rows are `row` bytes (128, 64 or 32), swizzled over the row: eight rows
// make up the stride; swizzle mode 2 / 4 / 6 for 128 / 64 / 32 bytes.
__host__ __device__ constexpr uint32_t desc_hi(uint32_t row) {
  return (8u * row >> 4) | (1u << 14) | ((row == 128u ? 2u : row == 64u ? 4u : 6u) << 29);
}
constexpr uint32_t A_DESC_HI = desc_hi(128u);  // an A tile always has 128-byte rows

// Which tile cluster `first` of `step` clusters takes in wave w: the clusters walk the tile list back and forth, so
// that with tiles sorted by decreasing duration the cluster that got the longest tile of one wave gets the shortest
// of the next (a static approximation of longest-processing-time-first).
__device__ __forceinline__ uint32_t snake_tile(uint32_t w, uint32_t first, uint32_t step) {
  return w * step + ((w & 1u) ? step - 1u - first : first);
}

// ------------------------------------------------------------------------------------------------ problem lookup
// A launch computes one GEMM, or (grouped launch) several independent ones whose tiles are numbered one after the
// other, so that one set of persistent CTAs packs them into common waves and the launch overhead is paid once.
template <int NP, bool SEVERAL, uint32_t EPI_BUFS = 1, bool CHAINED = false>
struct Problems {
  static constexpr bool CHAIN = CHAINED;                // each problem's A is the result of the one before
  static constexpr bool ONE = NP == 1, SUMS = SEVERAL;  // one problem; problems may have several products
  static constexpr uint32_t BUFS = EPI_BUFS;            // output buffers of an epilogue warp
  const GemmLaunchParams<NP>& g;
  __device__ __forceinline__ uint32_t count() const { return NP == 1 ? 1u : g.n; }
  __device__ __forceinline__ uint32_t total_tiles() const { return g.tile_end[count() - 1]; }
  // `i`: the problem of an earlier tile of the same role (its tiles come in ascending order), from which the search goes on
  __device__ __forceinline__ const GemmParams& at(uint32_t tile, uint32_t& i, uint32_t& local) const {
    if constexpr (NP == 1) {
      local = tile;
      return g.prob[0];
    } else {
      while (i + 1 < g.n && tile >= g.tile_end[i]) ++i;
      local = tile - (i ? g.tile_end[i - 1] : 0u);
      return g.prob[i];
    }
  }
  __device__ __forceinline__ const GemmParams& problem(uint32_t i) const { return g.prob[NP == 1 ? 0u : i]; }
  __device__ __forceinline__ const GemmParams& first() const { return g.prob[0]; }
  __device__ __forceinline__ const CommitParams& commit(uint32_t i) const { return g.prob[i].commit; }
  __device__ __forceinline__ uint32_t* ticket() const { return g.ticket; }
  __device__ __forceinline__ uint32_t* commits() const { return g.commits; }
  __device__ __forceinline__ uint32_t commits_op() const { return g.commits_op; }
  __device__ __forceinline__ const CommitParams& before() const { return g.before; }
  __device__ __forceinline__ uint32_t* status_of(uint32_t i) const { return g.prob[i].status; }
};

// What the roles need to know of a tile (INFO_BYTES of shared memory at most; written 16 bytes at a time up to amax_bits).  `alpha` is filled in later than the rest: scales
// come from kernels before this one.
struct alignas(16) TileInfo {
  uint32_t problem, m0, n0, num_kb;
  uint32_t nseg, epi, a_mn, b_mn;
  uint32_t idesc, b_desc_hi, b_step, ldo;
  uint32_t M, N;
  unsigned long long out;
  unsigned long long amax_bits;
  uint8_t slot_a[kMaxSegments], slot_b[kMaxSegments];
  float alpha[kMaxSegments];
  uint32_t minus_zero;  // see mul2; 0 where the tile is no sum
};
static_assert(sizeof(TileInfo) <= INFO_BYTES && INFO_BYTES % alignof(TileInfo) == 0 && BARS_BYTES % alignof(TileInfo) == 0 &&
              offsetof(TileInfo, amax_bits) % 16 == 0, "");
// The same value in every lane, and known to be: kept in a uniform register, as the instructions of the issuing roles want it.
__device__ __forceinline__ uint32_t uniform(uint32_t v) { return __reduce_or_sync(0xffffffffu, v); }

// ------------------------------------------------------------------------------------------------ kernel
template <bool PAIR, class PS>
__device__ __forceinline__ void gemm_body(const PS& ps) {
  constexpr uint32_t CTAS = Form<PAIR>::CTAS, TILE_M = Form<PAIR>::TILE_M;
  constexpr bool SUMS = PS::SUMS, ONE = PS::ONE, CHAIN = PS::CHAIN;
  constexpr int EPI_WARP0 = SUMS ? 4 : 2;    // first epilogue warp
  constexpr int INFO_WARP = SUMS ? 2 : 10;  // (launches of several problems)
  constexpr int STORE_WARP = 3;             // (sums)
  constexpr uint32_t BUFS = PS::BUFS, RING_BYTES = Ring<PAIR, BUFS>::BYTES;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t smem_base = smem_u32(smem_raw);
  const uint32_t epi_base = smem_base + RING_BYTES;  // 1 KB-aligned
  const uint32_t bar_base = smem_base + RING_AND_BUFS;
  // barrier block: full[MAX_STAGES], empty[MAX_STAGES], tmem_full[2], tmem_empty[2], tmem address + abort flag + last-CTA flag + counts
  // of warps, of the tile records full, scales and empty[INFO_SLOTS], of the buffers of sums ready and result[2][BUFS]
  auto full_bar = [&](uint32_t s) { return bar_base + 8u * s; };
  auto empty_bar = [&](uint32_t s) { return bar_base + 8u * (MAX_STAGES + s); };
  auto tfull_bar = [&](int a) { return bar_base + 8u * (2 * MAX_STAGES + a); };
  auto tempty_bar = [&](int a) { return bar_base + 8u * (2 * MAX_STAGES + 2 + a); };
  uint8_t* const gen_base = smem_raw;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gen_base + RING_AND_BUFS + 8 * (2 * MAX_STAGES + 4));
  constexpr uint32_t INFO_BARS = 8 * (2 * MAX_STAGES + 4) + (4 * (3 + kTileCounters) + 7) / 8 * 8;
  constexpr uint32_t BUF_BARS = INFO_BARS + 8 * 3 * INFO_SLOTS;
  static_assert(BUF_BARS + 8 * 4 * BUFS <= BARS_BYTES, "barrier block too large");
  // sums: buffer b of a half of the tile's columns (128 rows x 32 columns) is the epilogue's again (free, or holding what the
  // tile is added to) / is the storing warp's
  auto ready_bar = [&](uint32_t h, uint32_t b) { return bar_base + BUF_BARS + 8u * (h * BUFS + b); };
  auto result_bar = [&](uint32_t h, uint32_t b) { return ready_bar(h, b) + 16u * BUFS; };
  auto info_bar = [&](uint32_t n) { return bar_base + INFO_BARS + 8u * (n % INFO_SLOTS); };  // of the CTA's n-th tile
  auto scales_bar = [&](uint32_t n) { return info_bar(n) + 8u * INFO_SLOTS; };
  auto taken_bar = [&](uint32_t n) { return info_bar(n) + 16u * INFO_SLOTS; };
  auto info_of = [&](uint32_t n) { return reinterpret_cast<TileInfo*>(gen_base + RING_AND_BUFS + BARS_BYTES + INFO_BYTES * (n % INFO_SLOTS)); };
  auto info_parity = [](uint32_t n) { return n / INFO_SLOTS & 1u; };
  volatile uint32_t* abort_flag = tmem_slot + 1;
  uint32_t* last_flag = tmem_slot + 2;
  uint32_t* warps_done = tmem_slot + 3;  // [kTileCounters]: epilogue warps that have come to where a tile, or the CTA, is counted

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;  // position in the CTA pair; rank 0 issues the MMAs
  const uint32_t num_tiles = ps.total_tiles();
  const Ring<PAIR, BUFS> ring(ps.first().tile_n);  // (one tile width per launch)
  const uint32_t first_tile = blockIdx.x / CTAS, tile_step = gridDim.x / CTAS;
  uint32_t* const status = ps.first().status;
  // the n-th tile of this cluster.  (Chained problems: in order, so that what a tile waits for is on its way before it.)
  auto tile_of = [&](uint32_t n) { return CHAIN ? first_tile + n * tile_step : snake_tile(n, first_tile, tile_step); };
  const uint32_t tile_n = ps.first().tile_n;  // (of the whole launch)
  // which problem a tile belongs to and where it lies in it; `at_problem` as in Problems::at
  auto look_up = [&](uint32_t tile, uint32_t& at_problem, TileInfo& t) -> const GemmParams& {
    uint32_t local_tile;
    const GemmParams& p = ps.at(tile, at_problem, local_tile);
    tile_coords<TILE_M>(local_tile, (p.M + TILE_M - 1) / TILE_M, (p.N + tile_n - 1) / tile_n, !CHAIN && p.M <= p.N, tile_n, t.m0, t.n0);
    t.problem = at_problem;
    t.num_kb = p.Kc / BK;
    t.nseg = SUMS ? p.nseg : 1u;
    t.epi = (uint32_t)p.epi;
    t.a_mn = p.a_mn;
    t.b_mn = p.b_mn;
    t.idesc = p.idesc;
    t.b_desc_hi = p.b_desc_hi;
    t.b_step = p.b_step;
    t.ldo = p.ldo;
    t.M = p.M;
    t.N = p.N;
    t.out = (unsigned long long)p.out;
    t.amax_bits = (unsigned long long)p.amax_bits;
    return p;
  };
  // ... from the records that the info warp makes of it, for the CTA's n-th tile: one role's reading of it, and that it has
  auto await = [&](uint32_t bar, uint32_t parity, uint32_t err_bit) { return mbar_wait_warp(bar, parity, abort_flag, status, err_bit); };
  auto await_tile = [&](uint32_t n, uint32_t err_bit) { return await(info_bar(n), info_parity(n), err_bit); };
  auto took_tile = [&](uint32_t n) {
    __syncwarp();
    if (lane == 0) mbar_arrive(taken_bar(n));
  };
  // info warp: makes the record of the CTA's n-th tile
  auto announce = [&](uint32_t n, uint32_t tile, uint32_t& at_problem) {
    const uint32_t before = at_problem;
    TileInfo t;
    const GemmParams& p = look_up(tile, at_problem, t);
    if ((n == 0 || at_problem != before) && lane < 3)
      asm volatile("prefetch.tensormap [%0];" ::"l"(lane == 0 ? &p.tmA : lane == 1 ? &p.tmB : &p.tmD) : "memory");
    TileInfo* const to = info_of(n);
    if (lane == 0) {
      uint4* const w = reinterpret_cast<uint4*>(to);
      const uint4* const v = reinterpret_cast<const uint4*>(&t);
#pragma unroll
      for (uint32_t i = 0; i < offsetof(TileInfo, amax_bits) / 16; ++i) w[i] = v[i];
      to->amax_bits = t.amax_bits;
      if (SUMS) to->minus_zero = p.sum ? 0x80000000u : 0u;
    }
    if (SUMS && (uint32_t)lane < kMaxSegments) to->slot_a[lane] = p.slot_a[lane], to->slot_b[lane] = p.slot_b[lane];
    if (!SUMS && lane == 0) to->slot_a[0] = p.slot_a[0], to->slot_b[0] = p.slot_b[0];
    __syncwarp();
    if (lane == 0) mbar_arrive(info_bar(n));
  };

  if (threadIdx.x == 32) {  // descriptor fetch overlaps the rest of the prologue (and the predecessor's tail)
    const GemmParams& q = ps.first();  // (a group's other descriptors are fetched on first use)
    asm volatile("prefetch.tensormap [%0];" ::"l"(&q.tmA) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&q.tmB) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&q.tmD) : "memory");
  }
  if (threadIdx.x == 0) {
    for (uint32_t s = 0; s < MAX_STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull_bar(a), 1);
      mbar_init(tempty_bar(a), EPI_WARPS * CTAS);  // the epilogue warps of every CTA of the tile
    }
    if (SUMS)
      for (uint32_t i = 0; i < 2 * BUFS; ++i) {
        mbar_init(ready_bar(0, 0) + 8u * i, 1);
        mbar_init(result_bar(0, 0) + 8u * i, EPI_WARPS / 2);
      }
    if (!ONE)
      for (uint32_t i = 0; i < INFO_SLOTS; ++i) {
      mbar_init(info_bar(i), 1);
      mbar_init(scales_bar(i), 1);
      mbar_init(taken_bar(i), EPI_WARPS + 1 + (SUMS ? 1u : 0u) + (rank == 0 ? 1u : 0u));  // epilogue, producer, storing warp, MMA issuer
    }
    *abort_flag = 0u;
    for (uint32_t i = 0; i < kTileCounters; ++i) warps_done[i] = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    if (PAIR) {  // same warp in both CTAs of the pair
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();  // the peer's barriers are initialised before anything signals them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (warp == (ONE ? 0 : INFO_WARP) && first_tile < num_tiles) {
    // While the predecessor drains: pull the first ring-full of B tiles of this CTA's first tile towards L2.  A
    // prefetch moves no data into the SM, so it is harmless even if the predecessor is still writing that operand.
    uint32_t at_problem = 0;
    TileInfo t;
    const GemmParams& p = look_up(first_tile, at_problem, t);
    if (lane == 0) {
      const int rb = (int)(t.n0 + rank * (tile_n / 2));
      const CUtensorMap* tmB = &p.tmB;
      for (uint32_t kb = 0; kb < t.num_kb && kb < ring.blocks * ring.stages; kb += ring.blocks)
        for (int b = 0; b < (PAIR ? 1 : 2); ++b)
          tma_prefetch(tmB, p.b_mn ? rb + b * (int)BM : 0, p.b_mn ? 0 : rb + b * (int)BM, (int)kb, p.slot_b[0]);
    }
    // (and the first records)
    if (!ONE)
      for (uint32_t n = 0, tile = first_tile, from = 0; n < INFO_SLOTS && tile < num_tiles; ++n, tile = tile_of(n))
        announce(n, tile, from);
  }
  // Everything above (barriers, tensor memory) touched no data a predecessor produces and may overlap the previous
  // kernel's tail; operands, scales and the destination may come from it, so wait for it here.
  grid_dep_wait();
  const bool hold = blockIdx.x < ps.count() && ps.commits_op() == 1u;
  if (!hold) grid_dep_launch();
  if (blockIdx.x == 0 && warp == EPI_WARP0 && (uint32_t)lane < (CHAIN ? ps.count() : 1u)) {  // FP8 hand-off: the consumer's tape snapshot of its inverse scale
    const GemmParams& q = ps.problem((uint32_t)lane);
    if (q.epi == 3 && q.sinv_dst) *q.sinv_dst = *q.sinv_src;
  }
  if (!CHAIN && warp == EPI_WARP0 + 7 && blockIdx.x < ps.count()) {  // (a launch with early commits has a CTA per problem at least: most_committing)
    // The classes whose amax an EARLIER kernel reduced (the cast that made this GEMM's A operand) are committed here,
    // by an epilogue warp that has nothing to drain yet: nothing this launch computes reads their scale (its alphas
    // are snapshots), so only the output's class is left for the launch's tail.
    const CommitParams& c = ps.commit(blockIdx.x);
    if (c.st && c.early_mask) commit_class<false>(c, c.early_mask, c.bump_token != 0, true, lane);
    if (ps.commits_op() && lane == 0) {
      if (!hold) *ps.commits() = 0u;
      else {
        __threadfence();
        atomicAdd(ps.commits(), 1u);
      }
    }
    if (hold) {
      __syncwarp();
      grid_dep_launch();
    }
  }

  // The output's class of a chained forward before this one: its amax is complete too, and no tail of its own was spent on it.
  if (PS::ONE && warp == EPI_WARP0 + 6 && blockIdx.x == 0 && ps.before().st)
    commit_class<false>(ps.before(), ps.before().class_mask, false, true, lane);

  // (The roles are one flat choice: with producer and issuer nested under a choice of their own, or written as lambdas, the
  // same code ran 4 % slower, small launches and large ones alike.)
  if (SUMS) {
    __syncwarp();
    if (warp < EPI_WARP0) asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
  }
  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    const bool elected = elect_one();
    const bool several_waves = num_tiles > ps.count() * tile_step;  // (of each of the problems, on an average)
    uint32_t s = 0, ph = 0;
    bool ok = true;
    for (uint32_t n = 0, tile = first_tile; ok && tile < num_tiles; ++n, tile = tile_of(n)) {
      TileInfo t;
      unsigned long long slots_a = 0, slots_b = 0;  // a byte per product
      if (ONE) {
        uint32_t at_problem = 0;
        const GemmParams& p = look_up(tile, at_problem, t);
        slots_a = p.slot_a[0], slots_b = p.slot_b[0];
      } else {
        if (!(ok = await_tile(n, ERR_PRODUCER))) break;
        const TileInfo& r = *info_of(n);
        t.problem = uniform(r.problem), t.m0 = uniform(r.m0), t.n0 = uniform(r.n0), t.num_kb = uniform(r.num_kb);
        t.nseg = SUMS ? uniform(r.nseg) : 1u, t.a_mn = uniform(r.a_mn), t.b_mn = uniform(r.b_mn);
        if (SUMS) {
          slots_a = *reinterpret_cast<const unsigned long long*>(r.slot_a), slots_b = *reinterpret_cast<const unsigned long long*>(r.slot_b);
        } else {
          slots_a = uniform(r.slot_a[0]), slots_b = uniform(r.slot_b[0]);
        }
        took_tile(n);
      }
      const GemmParams& p = ps.problem(t.problem);
      // contraction-major operand: box = 128 K-bytes x rows x blocks at (0, row, block); MN-major operand (stored as [Kc, rows]):
      // box = row-bytes x 128 K-rows x blocks at (row, 0, block).  Either way 128 bytes per row and block land in shared memory.
      const int ra = (int)(t.m0 + rank * BM), rb = (int)(t.n0 + rank * (tile_n / 2));
      const int a0 = t.a_mn ? ra : 0, a1 = t.a_mn ? 0 : ra, b0 = t.b_mn ? rb : 0, b1 = t.b_mn ? 0 : rb;
      // both CTAs of a pair credit the even CTA's barrier, which expects the bytes of the whole pair (blocks beyond the
      // contraction are filled with zeros and counted)
      const uint32_t bytes = ring.blocks * (CTAS * A_BYTES + tile_n * BK);
      for (uint32_t seg = 0; ok && seg < t.nseg; ++seg, slots_a >>= 8, slots_b >>= 8) {
        const CUtensorMap *tmA = &p.tmA, *tmB = &p.tmB;
        const int sa = SUMS ? (int)uniform((uint32_t)slots_a & 255u) : (int)slots_a, sb = SUMS ? (int)uniform((uint32_t)slots_b & 255u) : (int)slots_b;
        uint32_t kb = 0;
        auto rows_before = [&](auto ask) {  // of the result that A is
          const GemmParams& q = ps.problem(t.problem - 1);
          return ask(&q.commit.st->rows_done[t.m0 / TILE_M], (q.N + tile_n - 1) / tile_n * CTAS);
        };
        if (CHAIN && t.problem && !(several_waves && rows_before(rows_there))) {
          // A is being made by other CTAs: B first, as far as the ring goes, then A when its rows are there.  (Where they are there
          // already, A and B go together: the first A would wait until the tile before had freed the whole ring.  Linears of several
          // waves meet few rows that they have to wait for: four of 4096 x 4096 at 8192 tokens 448 -> 408 us, at 4096 213 -> 199.
          // Linears of one wave find none there, and to ask holds up B: sixteen of 1024 x 1024 at 512 tokens 1497 -> 1516 a step.)
          const uint32_t s0 = s;
          for (uint32_t j = 0; ok && j < ring.stages && kb < t.num_kb; ++j, kb += ring.blocks) {
            if (!(ok = await(empty_bar(s), ph ^ 1u, ERR_PRODUCER))) break;
            if (elected) {
              if (rank == 0) mbar_expect_tx(full_bar(s), bytes);
              tma_load<PAIR>(smem_base + s * ring.stage_bytes + ring.b_offset(), tmB, PAIR ? map_to_cta(full_bar(s), 0) : full_bar(s), b0, b1, (int)kb, sb);
            }
            if (++s == ring.stages) { s = 0; ph ^= 1u; }
          }
          ok = ok && rows_before([&](const uint32_t* done, uint32_t count) { return rows_wait(done, count, abort_flag, status); });
          if (!ok) break;
          for (uint32_t j = s0, at = 0; at < kb; at += ring.blocks) {
            if (elected) tma_load<PAIR>(smem_base + j * ring.stage_bytes, tmA, PAIR ? map_to_cta(full_bar(j), 0) : full_bar(j), a0, a1, (int)at, sa);
            if (++j == ring.stages) j = 0;
          }
        }
        for (; kb < t.num_kb; kb += ring.blocks) {
          if (!(ok = mbar_wait_warp(empty_bar(s), ph ^ 1u, abort_flag, status, ERR_PRODUCER))) break;
          const uint32_t a_dst = smem_base + s * ring.stage_bytes, b_dst = a_dst + ring.b_offset();
          if (elected) {
            if (rank == 0) mbar_expect_tx(full_bar(s), bytes);
            const uint32_t bar = PAIR ? map_to_cta(full_bar(s), 0) : full_bar(s);
            tma_load<PAIR>(a_dst, tmA, bar, a0, a1, (int)kb, sa);
            tma_load<PAIR>(b_dst, tmB, bar, b0, b1, (int)kb, sb);
            // (a CTA on its own loads the tile's 256 rows of B as two boxes of 128, one behind the other)
            if (!PAIR) tma_load<PAIR>(b_dst + A_BYTES, tmB, bar, t.b_mn ? rb + (int)BM : 0, t.b_mn ? 0 : rb + (int)BM, (int)kb, sb);
          }
          if (++s == ring.stages) { s = 0; ph ^= 1u; }
        }
      }
    }
    if (!ok) let_copies_land();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (rank == 0) {
      const bool elected = elect_one();
      uint32_t s = 0, ph = 0, acc = 0, acc_ph = 0;
      bool ok = true;
      for (uint32_t n = 0, tile = first_tile; ok && tile < num_tiles; ++n, tile = tile_of(n)) {
        TileInfo t;
        if (ONE) {
          uint32_t at_problem = 0;
          look_up(tile, at_problem, t);
        } else {
          if (!(ok = await_tile(n, ERR_MMA))) break;
          const TileInfo& r = *info_of(n);
          t.num_kb = uniform(r.num_kb), t.nseg = SUMS ? uniform(r.nseg) : 1u;
          t.idesc = uniform(r.idesc), t.b_desc_hi = uniform(r.b_desc_hi), t.b_step = uniform(r.b_step);
          t.a_mn = uniform(r.a_mn), t.b_mn = uniform(r.b_mn);
          took_tile(n);
        }
        const uint32_t idesc = t.idesc, b_hi = t.b_desc_hi, a_step = t.a_mn ? 256u : 2u, b_step = t.b_step, num_kb = t.num_kb;
        const uint32_t b_block = tile_n / CTAS * BK / 16u;  // from one block of B in a stage to the next
        for (uint32_t seg = 0; ok && seg < t.nseg; ++seg) {  // an accumulator of its own for each product
          if (!(ok = mbar_wait_warp(tempty_bar(acc), acc_ph ^ 1u, abort_flag, status, ERR_MMA))) break;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + acc * ACC_COLS;
          for (uint32_t kb = 0; kb < num_kb; kb += ring.blocks) {
            if (!(ok = mbar_wait_warp(full_bar(s), ph, abort_flag, status, ERR_MMA))) break;
            tc_fence_after();
            const uint32_t a_src = smem_base + s * ring.stage_bytes, b_src = a_src + ring.b_offset();
            const uint64_t adesc = make_desc(a_src, A_DESC_HI);
            const uint64_t bdesc = make_desc(b_src, b_hi, PAIR || !t.b_mn ? 1u : A_BYTES / 16u);
            if (elected) {
#pragma unroll
              for (uint32_t k = 0; k < BK / UMMA_K; ++k)
                // advancing 32 along the contraction: 32 bytes inside the 128-byte swizzle row for a contraction-major
                // tile (+2 in the address field), 32 rows for an MN-major one (+256 with rows of 128 bytes)
                tc_mma_f8<PAIR>(d_tmem, adesc + a_step * k, bdesc + b_step * k, idesc, k ? 1u : kb);
              if (PAIR && ring.blocks == 2 && kb + 1 < num_kb) {
#pragma unroll
                for (uint32_t k = 0; k < BK / UMMA_K; ++k)
                  tc_mma_f8<PAIR>(d_tmem, adesc + A_BYTES / 16u + a_step * k, bdesc + b_block + b_step * k, idesc, 1u);
              }
              tc_commit<PAIR>(empty_bar(s));  // stage reusable (in both CTAs) once these MMAs have read it
            }
            if (++s == ring.stages) { s = 0; ph ^= 1u; }
          }
          if (!ok) break;
          if (elected) tc_commit<PAIR>(tfull_bar(acc));  // accumulator complete (each CTA holds its 128 rows)
          if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
        }
      }
    }
  } else if (!ONE && warp == INFO_WARP) {
    // ---------------------------------------------------------------- tile records
    uint32_t at_problem = 0, announced = 0, fetched_to = 0, last = 0;
    bool ok = true;
    auto fetch_rows = [&](uint32_t tile, uint32_t& from) {
      TileInfo t;
      look_up(tile, from, t);
      if (t.epi != 2 || !ps.problem(from).sum) return;
      const uint32_t rows = min(BM, t.M - min(t.M, t.m0 + rank * BM)), lines = min(tile_n, t.N - t.n0) / 32u;
      const char* d = reinterpret_cast<const char*>(reinterpret_cast<const float*>(t.out) + (size_t)(t.m0 + rank * BM) * t.ldo + t.n0);
      for (uint32_t i = (uint32_t)lane; i < rows * lines; i += 32)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(d + (size_t)(i / lines) * t.ldo * 4u + 128u * (i % lines)));
    };
    for (uint32_t n = 0, tile = first_tile; ok && tile < num_tiles; ++n, tile = tile_of(n)) {
      if (n >= INFO_SLOTS) {
        if (!(ok = await(taken_bar(n), info_parity(n) ^ 1u, ERR_PRODUCER))) break;
        announce(n, tile, announced);
      }
      uint32_t local_tile;
      const GemmParams& p = ps.at(tile, at_problem, local_tile);
      // (of the products' scales a lane each)
      if (CHAIN) {  // (the tape's copy of A's scale is being made; its source stays as it is until the launch's last commits)
        const bool later = at_problem > 0;
        const GemmParams& q = ps.problem(later ? at_problem - 1 : 0u);
        if (lane == 0) info_of(n)->alpha[0] = __fmul_rn(later ? *q.sinv_src : p.alpha_a[p.slot_a[0]], p.alpha_b[p.slot_b[0]]);
        if (lane == 1 && p.epi == 3) info_of(n)->alpha[1] = *p.out_scale;
      } else if ((uint32_t)lane < (SUMS ? p.nseg : 1u)) {
        info_of(n)->alpha[lane] = __fmul_rn(p.alpha_a[p.slot_a[lane]], p.alpha_b[p.slot_b[lane]]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(scales_bar(n));
      // Sums that start from what is there: towards L2, two tiles ahead (this warp is four ahead).
      if (SUMS && n >= INFO_SLOTS / 2) fetch_rows(tile_of(n - INFO_SLOTS / 2), fetched_to);
      last = n;
    }
    for (uint32_t n = last < INFO_SLOTS / 2 ? 0 : last - INFO_SLOTS / 2 + 1; SUMS && ok && n <= last && first_tile < num_tiles; ++n)
      fetch_rows(tile_of(n), fetched_to);
  } else if (SUMS && warp == STORE_WARP) {
    // ---------------------------------------------------------------- stores of sums
    // An SM writes 32 bytes a clock to L2 at most, by whichever unit: the 128 KB of a tile take 4130 clocks, and after a few
    // stores the thread that issues them waits for that.  So that is this warp's and not the epilogue's, which goes on to the next
    // tile: 11000 by 4096 gradients of 256 tokens, five products overwriting, 13000 -> 11500 clocks a tile.  Boxes of 16 KB: by
    // boxes of 4 KB the warp's own 500 clocks for each would bound it.  It also loads what a tile is added to into the buffers,
    // as they come free (by the epilogue's threads, a row each, that took as long as the stores).
    uint32_t result_ph = 0;    // a bit per buffer, the same for both halves
    bool ok = true, first = true;
    const uint32_t all = tile_n / 64u;
    struct Place {
      uint32_t sum, epi, problem, row, col;
      bool rows;  // not beyond M
      uint32_t N;
    };
    auto place_of = [&](uint32_t n) {
      const TileInfo& r = *info_of(n);
      const uint32_t row = r.m0 + rank * BM;
      return Place{r.minus_zero, r.epi, r.problem, row, r.n0, row < r.M, r.N};
    };
    auto result = [&](uint32_t h, uint32_t b) {
      const bool got = await(result_bar(h, b), result_ph >> b & 1u, ERR_EPILOGUE);
      if (h) result_ph ^= 1u << b;
      return got;
    };
    auto buf_of = [&](uint32_t h, uint32_t b) { return epi_base + (h * BUFS + b) * (4 * EPI_BUF_BYTES); };
    auto hand_on = [&](const Place& t, uint32_t h, uint32_t block) {  // block's buffer, for that block of tile t
      const uint32_t b = block % BUFS, col = t.col + h * (tile_n / 2) + block * 32u;
      if (t.sum && t.epi == 2 && t.rows && col < t.N) {
        fence_async_smem();
        mbar_expect_tx(ready_bar(h, b), 4 * EPI_BUF_BYTES);
        tma_load_2d(buf_of(h, b), &ps.problem(t.problem).tmD, ready_bar(h, b), (int)col, (int)t.row);
      } else {
        mbar_arrive(ready_bar(h, b));
      }
    };
    Place t{}, next{};
    if (first_tile < num_tiles && (ok = await_tile(0, ERR_EPILOGUE))) next = place_of(0);
    for (uint32_t n = 0, tile = first_tile; ok && tile < num_tiles; ++n) {
      tile = tile_of(n + 1);
      t = next;
      took_tile(n);
      next.sum = 0;
      if (tile < num_tiles) {
        if (!(ok = await_tile(n + 1, ERR_EPILOGUE))) break;
        next = place_of(n + 1);
      }
      if (!t.sum) continue;
      for (uint32_t i = 0; ok && first && i < 2 * min(BUFS, all); ++i)
        if ((ok = result(i & 1u, i / 2)) && lane == 0) hand_on(t, i & 1u, i / 2);
      first = false;
      for (uint32_t i = 0; ok && t.epi == 2 && i / 2 + BUFS < all; ++i)
        if ((ok = result(i & 1u, i / 2 % BUFS)) && lane == 0) hand_on(t, i & 1u, i / 2 + BUFS);
      auto stored = [&](uint32_t i) {  // the i-th block has been read out of its buffer
        const uint32_t block = i / 2;
        if (block + BUFS < all) mbar_arrive(ready_bar(i & 1u, block % BUFS));
        else hand_on(next, i & 1u, block % BUFS);
      };
      for (uint32_t i = 0; i < 2 * all; ++i) {
        const uint32_t h = i & 1u, block = i / 2;
        if (!(ok = ok && result(h, block % BUFS))) break;
        if (lane == 0) {
          const uint32_t col = t.col + h * (tile_n / 2) + block * 32u;
          if (t.rows && col < t.N) tma_store_2d(&ps.problem(t.problem).tmD, buf_of(h, block % BUFS), (int)col, (int)t.row);
          else asm volatile("cp.async.bulk.commit_group;" ::: "memory");  // (a group for every block)
          if (i) {
            tma_store_wait_read<1>();
            stored(i - 1);
          }
        }
      }
      if (ok && lane == 0) {
        tma_store_wait_read<0>();
        stored(2 * all - 1);
      }
    }
    if (lane == 0) tma_store_wait_read<0>();
    if (!ok) let_copies_land();
  } else if (!SUMS || warp >= EPI_WARP0) {
    // ---------------------------------------------------------------- epilogue
    if (SUMS) asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    const uint32_t quad = (uint32_t)warp & 3u;          // tensor-memory lane quadrant this warp may read
    const uint32_t half = (uint32_t)(warp - EPI_WARP0) >> 2;   // which half of the tile's columns
    const int etid = (int)threadIdx.x - EPI_WARP0 * 32;
    // this warp's output tiles; sums: the first of its quarters of its half's buffers
    const uint32_t epi_smem = epi_base + ((uint32_t)half * 4 * BUFS + (uint32_t)(warp - EPI_WARP0) % 4u) * EPI_BUF_BYTES;
    uint32_t n_groups = 0;  // bulk-store groups this warp has committed (buffer parity)
    const uint32_t ready = ready_bar(half, 0), result = result_bar(half, 0);
    uint32_t ready_ph = 0;  // a bit per buffer
    auto give_buf = [&](uint32_t b) {  // sums: to the storing warp
      __syncwarp();
      if (lane == 0) mbar_arrive(result + 8u * b);
    };
    auto await_buf = [&](uint32_t b) {  // ... and back
      const bool got = await(ready + 8u * b, ready_ph >> b & 1u, ERR_EPILOGUE);
      ready_ph ^= 1u << b;
      return got;
    };
    uint32_t acc = 0, acc_ph = 0;
    bool ok = true;
    const uint32_t tempty_leader0 = PAIR ? map_to_cta(tempty_bar(0), 0) : tempty_bar(0);
    const uint32_t tempty_leader1 = PAIR ? map_to_cta(tempty_bar(1), 0) : tempty_bar(1);
    // Of a tile: this warp's part of it.
    struct Part {
      uint32_t problem, epi, nseg, row, col, blocks;  // 32 x 32 blocks: none in rows beyond M, fewer in a ragged last column tile
      float* dst;                                     // FP32 results: this thread's row
      uint32_t* amax_bits;
      float alpha;                                    // SUMS: lane i has the scale of product i
      float out_scale;                                // hand-off
      uint8_t* dst8;                                  // chained problems: this thread's row, its format, the count of its rows
      int32_t out_fmt;
      uint32_t* done;
      uint32_t minus_zero;
    };
    auto part_of = [&](const TileInfo& r) {
      Part t;
      t.problem = r.problem;
      t.epi = r.epi;
      t.nseg = SUMS ? r.nseg : 1u;
      t.row = r.m0 + rank * BM + quad * 32u;
      t.col = r.n0 + half * (tile_n / 2);
      t.blocks = t.row >= r.M || t.col >= r.N ? 0u : min(tile_n / 64u, (r.N - t.col) / 32u);
      t.dst = reinterpret_cast<float*>(r.out) + (size_t)(t.row + lane) * r.ldo + t.col;
      t.amax_bits = reinterpret_cast<uint32_t*>(r.amax_bits);
      return t;
    };
    auto take_part = [&](uint32_t n, Part& t) {  // of the CTA's n-th tile
      if (ONE) {
        uint32_t at_problem = 0;
        TileInfo r;
        const GemmParams& p = look_up(tile_of(n), at_problem, r);
        t = part_of(r);
        t.alpha = __fmul_rn(p.alpha_a[p.slot_a[0]], p.alpha_b[p.slot_b[0]]);
        if (t.epi == 3) t.out_scale = *p.out_scale;
        return true;
      }
      if (!await(scales_bar(n), info_parity(n), ERR_EPILOGUE)) return false;
      const TileInfo& r = *info_of(n);
      t = part_of(r);
      t.alpha = r.alpha[SUMS ? (uint32_t)lane % kMaxSegments : 0u];
      t.minus_zero = r.minus_zero;
      if (CHAIN) {
        t.out_scale = r.alpha[1];
        t.dst8 = reinterpret_cast<uint8_t*>(r.out) + (size_t)(t.row + lane) * r.ldo + t.col;
        t.out_fmt = ps.problem(r.problem).out_fmt;
        t.done = &ps.problem(r.problem).commit.st->rows_done[r.m0 / TILE_M];
      }
      took_tile(n);
      return true;
    };
    auto prefetch_rows = [&](const Part& t) {  // what this thread's row will be added to, towards L2
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j)
        if (j < t.blocks) asm volatile("prefetch.global.L2 [%0];" ::"l"(t.dst + 32 * j));
    };
    RingState ring_of_Y;  // (the class that the tail commits)
    if (ONE && ps.ticket()) ring_of_Y = ring_state(ps.commit(0), __ffs(ps.commit(0).class_mask) - 1);
    Part now;
    ok = first_tile < num_tiles && take_part(0, now);
    uint32_t n = 0, tile = first_tile;
    for (; ok && tile < num_tiles && !(SUMS && now.minus_zero); ++n) {  // (sums come after all others)
      tile = tile_of(n + 1);
      const Part t = now;
      const uint32_t nch = t.blocks, blk_row0 = t.row, col0 = t.col;
      const GemmParams& p = ps.problem(t.problem);
      const uint32_t ln = (uint32_t)lane;
      const float alpha = SUMS ? __shfl_sync(0xffffffffu, t.alpha, 0) : t.alpha;
      // accumulate: pull this thread's destination row segment into L2, where the reduction will add to it, while the MMAs of
      // the tile run
      if (t.epi == 2) prefetch_rows(t);
      uint32_t r[2][32];
      if (!(ok = mbar_wait_warp(tfull_bar(acc), acc_ph, abort_flag, status, ERR_EPILOGUE))) break;
      tc_fence_after();
      const uint32_t t_row = tmem_base + ((quad * 32u) << 16) + acc * ACC_COLS + half * (tile_n / 2);
      uint32_t amax_bits = 0;
      // Software pipeline over the warp's (up to four) 32 x 32 blocks: the tensor-memory load of block ch+1 is in flight
      // while block ch is scaled, written to shared memory and handed to the bulk-store unit.
      if (nch) tmem_ld32(t_row, r[0]);
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        if ((uint32_t)ch >= nch) break;
        const uint32_t col = col0 + ch * 32u;
        tmem_ld_wait();
        if ((uint32_t)ch + 1 < nch) tmem_ld32(t_row + (ch + 1) * 32u, r[(ch + 1) & 1]);
        const uint32_t(&rc)[32] = r[ch & 1];
        // Each lane (= row) writes its 32 columns into a swizzled shared-memory tile (conflict-free); one lane hands
        // the 32 x 32 tile to the bulk-store unit, which writes full rows to global memory (bf16, FP32 overwrite) or
        // adds them to the destination where it lives, in L2 (FP32 accumulate: one addition per element and launch).
        if (t.epi == 0) {
          const uint32_t buf = epi_smem + (n_groups & 1u) * 2048u;  // two tiles: the previous store may still read
          if (lane == 0) {  // (a tile before this one may have used the buffer as a whole)
            if (ch == 0) tma_store_wait_read<0>();
            else tma_store_wait_read<1>();
          }
          __syncwarp();
          uint32_t o[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            o[j] = pack_bf16(__fmul_rn(__uint_as_float(rc[2 * j]), alpha), __fmul_rn(__uint_as_float(rc[2 * j + 1]), alpha));
            amax_bits = __vmaxu2(amax_bits, o[j] & 0x7fff7fffu);  // packed magnitudes of the rounded values stored
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {  // 64-byte rows, 64-byte swizzle: 16-byte chunk c of row r sits at c ^ ((r >> 1) & 3)
            const uint32_t dst = buf + ln * 64u + (((uint32_t)c ^ ((ln >> 1) & 3u)) << 4);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(o[4 * c]), "r"(o[4 * c + 1]),
                         "r"(o[4 * c + 2]), "r"(o[4 * c + 3])
                         : "memory");
          }
          fence_async_smem();
          __syncwarp();
          if (lane == 0) tma_store_2d(&p.tmD, buf, (int)col, (int)blk_row0);
        } else if ((ONE || CHAIN) && t.epi == 3) {
          // FP8 hand-off to the consuming linear: round to bf16 (the value that linear would have read), take its
          // magnitude for the amax, multiply by the consumer's scale in FP32 and convert -- the consumer's cast
          // kernel, applied to registers.  32 bytes per row; two 1 KB tiles per warp.
          const uint32_t buf = epi_smem + (n_groups & 1u) * 1024u;
          if (!CHAIN) {
            if (lane == 0) tma_store_wait_read<1>();
            __syncwarp();
          }
          const float qs = t.out_scale;
          const int32_t out_fmt = CHAIN ? t.out_fmt : p.out_fmt;
          uint32_t q[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            uint32_t w[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              w[h] = pack_bf16(__fmul_rn(__uint_as_float(rc[4 * j + 2 * h]), alpha), __fmul_rn(__uint_as_float(rc[4 * j + 2 * h + 1]), alpha));
              amax_bits = __vmaxu2(amax_bits, w[h] & 0x7fff7fffu);
            }
            const float2 f01 = make_float2(__fmul_rn(__uint_as_float(w[0] << 16), qs), __fmul_rn(__uint_as_float(w[0] & 0xffff0000u), qs));
            const float2 f23 = make_float2(__fmul_rn(__uint_as_float(w[1] << 16), qs), __fmul_rn(__uint_as_float(w[1] & 0xffff0000u), qs));
            const uint32_t lo = out_fmt == 0 ? __nv_cvt_float2_to_fp8x2(f01, __NV_SATFINITE, __NV_E4M3)
                                               : __nv_cvt_float2_to_fp8x2(f01, __NV_SATFINITE, __NV_E5M2);
            const uint32_t hi = out_fmt == 0 ? __nv_cvt_float2_to_fp8x2(f23, __NV_SATFINITE, __NV_E4M3)
                                               : __nv_cvt_float2_to_fp8x2(f23, __NV_SATFINITE, __NV_E5M2);
            q[j] = lo | (hi << 16);
          }
          if (CHAIN) {  // (whole sectors by plain stores: they are there a bulk store's 500 clocks sooner)
            asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(t.dst8 + ch * 32),
                         "r"(q[0]), "r"(q[1]), "r"(q[2]), "r"(q[3]), "r"(q[4]), "r"(q[5]), "r"(q[6]), "r"(q[7])
                         : "memory");
          } else {
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const uint32_t dst = buf + ln * 32u + ((uint32_t)c << 4);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(q[4 * c]), "r"(q[4 * c + 1]),
                         "r"(q[4 * c + 2]), "r"(q[4 * c + 3])
                         : "memory");
          }
          fence_async_smem();
          __syncwarp();
          if (lane == 0) tma_store_2d(&p.tmD, buf, (int)col, (int)blk_row0);
          }
        } else {
          // one tile: waiting for the previous block's store to have read it paces the FP32 traffic, which measured
          // faster than two tiles in flight per warp
          const uint32_t buf = epi_smem;
          if (lane == 0) tma_store_wait_read<0>();
          __syncwarp();
          float o[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) o[j] = __fmul_rn(__uint_as_float(rc[j]), alpha);
          st_tile_f32(buf, ln, o);
          fence_async_smem();
          __syncwarp();
          if (lane == 0) {
            if (t.epi == 2) tma_reduce_add_2d(&p.tmD, buf, (int)col, (int)blk_row0);
            else tma_store_2d(&p.tmD, buf, (int)col, (int)blk_row0);
          }
        }
        ++n_groups;
      }
      // accumulator drained: hand it back to the MMA warp
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {  // the MMA issuer of a pair waits in the even CTA
        if (PAIR) mbar_arrive_cluster(acc ? tempty_leader1 : tempty_leader0);
        else mbar_arrive(acc ? tempty_leader1 : tempty_leader0);
      }
      if (CHAIN && t.epi == 3) {  // the next problem's loads of these rows wait for this
        __syncwarp();
        if (lane == 0 && last_of_tile(n, EPI_WARPS, [&](uint32_t i) { return add_acq_rel_cta(warps_done + i); })) add_release(t.done, 1u);
      }
      uint32_t* const also = ONE || CHAIN ? p.amax_bits2 : nullptr;  // (hand-off)
      if ((t.epi == 0 || ((ONE || CHAIN) && t.epi == 3)) && (t.amax_bits || also)) {
        // two packed bf16 magnitudes -> FP32 bit pattern of the larger
        const uint32_t w = __reduce_max_sync(0xffffffffu, max(amax_bits & 0xffffu, amax_bits >> 16) << 16);
        if (lane == 0 && w) {
          if (t.amax_bits) atomicMax(t.amax_bits, w);
          if (also) atomicMax(also, w);
        }
      }
      if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
      if (tile < num_tiles && !(ok = take_part(n + 1, now))) break;
    }
    if constexpr (SUMS) {
      // A tile's running value stays in registers and every product (the weight gradient of a microbatch) is added to it in
      // order, each with its own scale -- the additions that launches of their own would have done in L2, at one read and one
      // write of the destination instead of one per product.  (A loop of its own behind the other tiles': in one loop with them
      // the values did not fit the registers, and the few bytes of them in local memory, for which shared memory leaves no L1,
      // cost more than all that is saved here.  12 bytes a thread are still there.)
      f32x2 v[4][16];                    // this thread's row
      const uint32_t all = tile_n / 64u;  // blocks of a tile that is not ragged: what buffers are handed on for
      if (lane == 0) tma_store_wait_read<0>();
      for (uint32_t b = 0; b < BUFS && b < all; ++b) give_buf(b);
      for (; ok && tile < num_tiles; ++n) {
          const uint32_t nch = now.blocks, nseg = now.nseg;
          const bool adds = now.epi == 2;
          const f32x2 minus_zero = pack2(now.minus_zero, now.minus_zero);
          auto take = [&](uint32_t seg, auto first) {
            const float alpha = __shfl_sync(0xffffffffu, now.alpha, (int)seg);
            const f32x2 alpha2 = pack2(__float_as_uint(alpha), __float_as_uint(alpha));
            if (!(ok = await(tfull_bar(acc), acc_ph, ERR_EPILOGUE))) return;
            tc_fence_after();
            const uint32_t t_row = tmem_base + ((quad * 32u) << 16) + acc * ACC_COLS + half * (tile_n / 2);
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
              if ((uint32_t)ch >= nch) break;
              uint32_t r[32];
              tmem_ld32(t_row + ch * 32u, r);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const f32x2 d = mul2(pack2(r[2 * j], r[2 * j + 1]), alpha2, minus_zero);
                v[ch][j] = decltype(first)::value ? d : add2(v[ch][j], d);
              }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(acc ? tempty_leader1 : tempty_leader0);
            if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
          };
          if (!adds) {
            take(0, std::true_type{});
          } else {
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
              if ((uint32_t)ch >= all || !(ok = await_buf(ch % BUFS))) break;
              if ((uint32_t)ch < nch) ld_tile_f32x2(epi_smem + (ch % BUFS) * (4 * EPI_BUF_BYTES), (uint32_t)lane, v[ch]);
              if (ch + BUFS < all) give_buf(ch % BUFS);
            }
            if (ok) take(0, std::false_type{});
          }
          for (uint32_t seg = 1; ok && seg < nseg; ++seg) take(seg, std::false_type{});
          if (!ok) break;
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) {
            if ((uint32_t)ch >= all) break;
            if ((!adds || ch >= (int)BUFS) && !(ok = await_buf(ch % BUFS))) break;
            if ((uint32_t)ch < nch) st_tile_f32x2(epi_smem + (ch % BUFS) * (4 * EPI_BUF_BYTES), (uint32_t)lane, v[ch]);
            fence_async_smem();
            give_buf(ch % BUFS);
          }
          if (!ok) break;
          tile = tile_of(n + 1);
          if (tile < num_tiles && !(ok = take_part(n + 1, now))) break;
      }
    }
    // Every epilogue thread of every CTA gets here (also after a timeout); the last CTA commits the scale state of
    // every problem that asks for it.  The commit needs the amax atomics only, so it runs while this CTA's last
    // bulk stores are still draining.
    // (Of one problem by a warp: the last of its CTA to get here, of the last CTA.  It has read ahead what it needs beside the amax.
    // Counted by all threads behind a fence and two barriers, the commit read and made after that, the tail was 0.7 us longer:
    // a 2048 / 8192 layer of 256 tokens action by action 992 -> 980 us a step, 512 to 2048 at 640 tokens 1190 -> 1164.)
    if (ONE && ps.ticket()) {
      __syncwarp();
      const bool last = lane == 0 && add_acq_rel_cta(warps_done) == EPI_WARPS - 1 && last_of_grid(ps.ticket(), gridDim.x);
      if (__shfl_sync(0xffffffffu, last ? 1 : 0, 0)) {
        __syncwarp();
        commit_class<false>(ps.commit(0), ps.commit(0).class_mask, false, true, lane, &ring_of_Y);
      }
    }
    if (!ONE && ps.ticket() && last_block(ps.ticket(), gridDim.x, etid, last_flag, epi_bar_sync)) {
      // (the token is counted by the early part)
      const uint32_t ew = (uint32_t)(warp - EPI_WARP0);
      if (ew < ps.count()) {  // a lane per problem, dealt to the epilogue's warps
        static_assert(kMaxProblems <= EPI_WARPS * 32, "a lane for every problem");
        const uint32_t i = ew + EPI_WARPS * (uint32_t)lane;
        const CommitParams& c = ps.commit(i < ps.count() ? i : 0u);
        if (CHAIN) {  // all classes of all problems; and nobody waits for rows any more
          commit_class<true>(c, c.early_mask, true, i < ps.count(), lane);
          for (uint32_t r = 0; i < ps.count() && r < (ps.problem(i).M + TILE_M - 1) / TILE_M; ++r) c.st->rows_done[r] = 0u;
        }
        commit_class<true>(c, c.class_mask, false, i < ps.count() && c.st && c.class_mask, lane);
      }
    }
    // The bulk-store unit has read this warp's last tiles out of shared memory; that the bytes are in global memory
    // before a dependent kernel passes its griddepcontrol.wait is part of this grid's completion.
    if (lane == 0) tma_store_wait_read<0>();
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    // a wait gave up in this CTA: the error bits went to the first problem's status word; every other problem of a
    // shared launch gets them too, since any of their tiles may be missing
    const uint32_t bits = atomicOr(status, 0u);
    for (uint32_t i = 1; i < ps.count(); ++i)
      if (ps.status_of(i) && ps.status_of(i) != status) atomicOr(ps.status_of(i), bits);
  }
  if (PAIR) cluster_sync_all();  // no arrival may still be on its way to a CTA that has left
  if (warp == 1) {
    tc_fence_after();
    if (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(threads_of(false, false), 1)
    gemm_fp8_pair_kernel(const __grid_constant__ GemmLaunchParams<1> p) {
  gemm_body<true>(Problems<1, false>{p});
}

// One GEMM with an odd number of 128-row tiles, a CTA to a tile.
__global__ void __launch_bounds__(threads_of(false, false), 1) gemm_fp8_kernel(const __grid_constant__ GemmLaunchParams<1> p) {
  gemm_body<false>(Problems<1, false>{p});
}

// The whole-step call's casts may run beside these launches (quantize_multi_kernel, Announce), a block of eight warps of 40
// registers on each SM: three GEMM warps share a sub-partition's 16384 registers with two of the cast's, which leaves each 144.
// The bound is that of 448 threads (128 registers taken, none spilled; 168 without it).  us a step with the casts between the
// GEMMs / with their blocks starting on SMs that a GEMM launch has left (168 registers) / beside its CTAs, under the power limit:
// a block of hidden 2048 at 2048 tokens 2620 / 2575 / 2510, 48 linears of 1024 4990 / 4910 / 4880, a 4096 / 11008 layer at 256
// tokens 1564 / 1536 / 1536.
constexpr int SHARED_SM_THREADS = 448;

// Several independent GEMMs in one launch: up to eight (a parameter block of 5 KB), or what the parameter space holds.
template <int NP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(SHARED_SM_THREADS, 1)
    gemm_fp8_pair_group_kernel(const __grid_constant__ GemmLaunchParams<NP> g) {
  gemm_body<true>(Problems<NP, false>{g});
}

// Chained problems: each one's A is the result of the one before, handed on in FP8, in one launch.  Its CTAs wait on one another
// (a cooperative launch): a tile's loads of A for its rows of the problem before, which are counted as they are stored; those
// of B do not wait, up to a ring-full, and a tile waits behind earlier ones only.  The scales are committed when all is done.  Of the
// 7800 clocks from one 512 x 1024 x 1024 to the next (tiles of 64 columns, half of the CTAs) the loads of A take 2560, the MMAs
// behind them 680, the epilogue 670, the count among a CTA's warps 300, and some 3600 pass until the next linear's loads are let
// go: the release, 1050 of them, and the poll (16 layers: 66 us a launch, 88 as launches of their own).
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(threads_of(false, true), 1)
    gemm_fp8_pair_chain_kernel(const __grid_constant__ GemmLaunchParams<kMaxChained> g) {
  gemm_body<true>(Problems<kMaxChained, false, 1, true>{g});
}

// The same where problems have several products each.
template <uint32_t EPI_BUFS>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(threads_of(true, true), 1)
    gemm_fp8_pair_wide_kernel(const __grid_constant__ GemmLaunchParams<kMaxProblems> g) {
  gemm_body<true>(Problems<kMaxProblems, true, EPI_BUFS>{g});
}

constexpr uint32_t PAIR_M = Form<true>::TILE_M;
uint32_t ceil_div(uint32_t a, uint32_t b) { return (a + b - 1) / b; }
uint32_t tiles_of(const GemmDesc& d, uint32_t tile_n) { return ceil_div(d.M, PAIR_M) * ceil_div(d.N, tile_n); }

// Columns per tile of a launch's problems (index into kTileWidths).  A tile's main loop takes 340, 460 or 530 clocks per 128-byte
// K block at 64, 128 or 256 columns (shared memory is read and written for A whatever the width; an MMA of up to 64 columns
// takes 48 clocks, one of 128 takes 64), so narrower tiles gain nothing unless every CTA pair has one: a launch that leaves
// pairs idle takes narrower ones, which also shortens its epilogue.  us at 256 / 128 / 64 columns, back to back: 256 x 256 x
// 256 4.5 / 3.7 / 3.2, 512 x 1024 x 1024 6.4 / 4.8 / 4.1, 256 x 2048 x 8192 22.4 / 15.6 / 13.9, 512 x 4096 x 4096 13.8 / 10.8
// (two waves of 64: 14.6).  The narrowest only up to half the pairs: beyond, the next launch's CTAs find no free SM to start on
// before this one ends, which costs what the width gains (1024 x 1024 x 1024 6.5 / 4.96 / 5.01, 768 x 1536 x 1536 7.7 / 5.63 /
// 5.76, 512 x 2048 x 2048 9.0 / 6.4 / 6.2).  More tiles than pairs lose at once (256 x 8192 x 4096 14.9 / 12.0 / 15.2).
uint32_t choose_width(const GemmDesc* d, uint32_t n, uint32_t pairs) {
  uint32_t w = 0;
  while (w + 1 < kNumTileWidths) {
    uint32_t tiles = 0;
    for (uint32_t i = 0; i < n; ++i) tiles += tiles_of(d[i], kTileWidths[w + 1]);
    if (tiles > (w == 0 ? pairs : pairs / 2)) break;
    ++w;
  }
  return w;
}

// Whether a GEMM goes out with a CTA to a 128 x 256 tile instead of a pair to a 256-row one.  With an odd number of 128-row
// tiles the pairs' last row tile is half empty, and the launch may need a wave more; a CTA on its own loads half as much
// again per K block, so that its waves take up to a fifth longer (M x N x contraction, one CTA to a tile against pairs):
//   1 wave for 2    1152 x 4096 x 4096 15.0 us for 24.7, 384 x 11008 x 4096 14.6 for 24.6, 3712 x 1280 x 1024 8.2 for 11.5
//   2 for 3         640 x 12800 x 4096 29.1 for 34.7, 3712 x 2560 x 1024 12.2 for 13.5
//   3 for 4         3968 x 3584 x 4096 43.5 for 47.6;  4 for 5: 1152 x 15360 x 4096 61.9 for 62.8
//   5 for 6         3712 x 6400 x 4096 74.6 for 74.5;  7 for 8: 3968 x 8448 x 4096 104.7 for 101.5;  4 for 4: 64.8 for 60.8
// With one wave either way the CTAs, which wait for no peer, start and finish 1 us earlier (384 x 9472 x 4096 14.5 for 15.3),
// which the loads of a long contraction eat up (1920 x 2176, cast included: 23.7 for 25.3 at 4096, 31.6 for 32.3 at 6528,
// 39.2 for 38.8 at 8192); at 128 rows the pair's empty half still shares the loads of B (128 x 16384 x 4096, FP32: 17.6
// for 16.9).  Even row counts have no empty half.
bool saves_a_wave(const GemmDesc& d, int num_sms) {
  const uint32_t waves_pairs = ceil_div(tiles_of(d, 256), (uint32_t)num_sms / 2u);
  const uint32_t waves_ctas = ceil_div((d.M / BM) * ceil_div(d.N, 256), (uint32_t)num_sms);
  return 6 * waves_ctas < 5 * waves_pairs;
}
bool one_cta(const GemmDesc& d, int num_sms) {
  const uint32_t pairs = (uint32_t)num_sms / 2u;
  if (d.M % PAIR_M == 0 || choose_width(&d, 1, pairs) != 0) return false;
  return saves_a_wave(d, num_sms) || (tiles_of(d, 256) <= pairs && d.M > BM && d.Kc <= 6144);
}

// The device's parameter block of one problem at a tile width.
GemmParams problem_of(const GemmDesc& d, uint32_t w, uint32_t tile_m) {
  GemmParams p = d;
  const uint32_t tile_n = kTileWidths[w], per_cta = tile_n / 2;
  p.tmA = d.mapA[a_map_of(w)];
  p.tmB = d.mapB[w];
  p.tile_n = tile_n;
  // bits 4-5: accumulator format (1 = FP32); 7-9 / 10-12: A / B format (0 = E4M3, 1 = E5M2); 15 / 16: A / B major
  // (0 = contraction-major); 17-22: N >> 3; 24-28: M >> 4 (of the whole tile).
  p.idesc = (1u << 4) | (d.a_fmt << 7) | (d.b_fmt << 10) | (d.a_mn << 15) | (d.b_mn << 16) | ((tile_n >> 3) << 17) | ((tile_m >> 4) << 24);
  // An MN-major B tile has rows of per_cta bytes (a CTA alone: two boxes of 128), swizzled over exactly that width; a
  // contraction-major one rows of 128.
  const uint32_t row = d.b_mn ? per_cta : 128u;
  p.b_desc_hi = desc_hi(row);
  p.b_step = d.b_mn ? 32u * row / 16u : 2u;
  return p;
}

// Whether chained problems go out as one launch.  What that saves is a launch's start and end between two of them, about
// 1.3 us, and a layer's last wave, which the next one's tiles fill; what it costs is a launch whose blocks all have to be there at
// once, which starts some us later, one tile width for all, and tiles that go row by row, so that a linear's weights are read again
// with every wave.  One by one / in one launch, us of a forward chain and of an input-gradient chain:
//   one width       not where linears want different ones: 512 tokens, 2048 - 8192 - 2048 - 8192 - 2048 67 / 78 and 64 / 75; 256 tokens,
//                   4096 - 16384 - 4096 - 16384 - 4096 107 / 129 and 104 / 125; 2048 tokens, 512 - 2048 - ... 40.4 / 43.0 and 37.9 / 42.0
//   few and small   four to seven linears pay for the later start only where each fills three fifths of the pairs: 512 tokens, four of 1024
//                   28.2 / 29.2 and 26.1 / 27.6, of 4096 56.8 / 53.3 and 55.3 / 51.2; 2048 tokens, four of 256 32.3 / 36.3 and 29.7 / 35.3,
//                   of 1024 36.4 / 34.3 and 33.8 / 32.8; 384 tokens, four of 2560 (40 tiles) 41.1 / 41.0 and 37.9 / 38.9
//   eight or more   512 tokens, 1024 46.6 / 44.6 and 44.5 / 44.0; 2048 tokens, 256 41.4 / 39.9 and 37.9 / 37.9, 512 50.3 / 44.6 and 46.1 / 43.0
//   waves           in part-filled ones the gain is largest (eight linears: 4096 tokens, 4096 (3.5 waves) 501 / 431; 2048 tokens, 6144 (2.6)
//                   549 / 476; 4096 tokens, 6144 (5.2) 1028 / 940); at seven little is left to fill (8192 tokens, 4096 (6.9) 859 / 867)
//   weights         of more than the L2 cache keeps: bytes times waves 3072 tokens, four of 8192 (348 MB) 661 / 643, 1024 tokens, four of
//                   10240 (227 MB) 406 / 347, 512 tokens, four of 16384 (464 MB) 423 / 436, 1024 tokens (929 MB) 862 / 1008; 4096 tokens, four
//                   of 8192 (464 MB) 738 / 842
// Half-filled row tiles are not avoided there: where that saved a wave (one_cta) the launches stay (us a step of four
// microbatches: 1152 tokens, four of 4096 x 4096 1112 / 1136; 1920 tokens, six of 2304 x 2304, one wave, 1007 / 950).
constexpr uint32_t kManyChained = 8;
bool launch_chained(const GemmDesc* d, uint32_t n, int num_sms) {
  if (n < kLaunchChained || n > kMaxChained || d->M > PAIR_M * (sizeof(DevState::rows_done) / sizeof(uint32_t))) return false;
  const uint32_t pairs = (uint32_t)num_sms / 2u, w = choose_width(d, 1, pairs);
  for (uint32_t i = 0; i < n; ++i) {
    const uint32_t tiles = tiles_of(d[i], kTileWidths[w]);
    if (choose_width(d + i, 1, pairs) != w || (n < kManyChained && 5 * tiles < 3 * pairs) || 2 * tiles > 13 * pairs) return false;
    if ((uint64_t)d[i].N * d[i].Kc * tiles > 400000000ull * pairs) return false;
    if (d[i].M % PAIR_M && saves_a_wave(d[i], num_sms)) return false;
  }
  return true;
}

template <int NP>
Launch make_launch(const GemmDesc* probs, uint32_t n, int num_sms, const void* func, bool sums, bool alone = false) {
  using P = GemmLaunchParams<NP>;
  static_assert(sizeof(P) <= sizeof(Launch::Block) && sizeof(P) <= 32764, "parameter block too large");
  static_assert(NP > 1 || sizeof(P) <= ParamBytes::kInline, "a launch of one problem takes no heap memory");
  Launch l;
  l.nbytes = sizeof(P);
  l.params.resize(offsetof(P, prob) + n * sizeof(GemmParams));  // (no unused problems)
  unsigned char* at = l.params.data();
  const uint32_t tile_m = alone ? BM : PAIR_M, ctas = alone ? 1u : 2u, most = (uint32_t)num_sms / ctas;
  const uint32_t w = choose_width(probs, probs->chained ? 1 : n, (uint32_t)num_sms / 2u);  // (alone: 0, see one_cta)
  uint32_t tiles = 0;
  uint32_t* ticket = nullptr;
  for (uint32_t i = 0; i < n; ++i) {
    if (!ticket && probs[i].commit.st && (probs[i].commit.class_mask || probs[i].chained)) ticket = &probs[i].commit.st->ticket;
    tiles += ceil_div(probs[i].M, tile_m) * ceil_div(probs[i].N, kTileWidths[w]);
    std::memcpy(at + offsetof(P, tile_end) + i * sizeof(uint32_t), &tiles, sizeof(tiles));
    const GemmParams p = problem_of(probs[i], w, tile_m);
    std::memcpy(at + offsetof(P, prob) + i * sizeof(GemmParams), &p, sizeof(p));
  }
  std::memcpy(at + offsetof(P, n), &n, sizeof(n));
  std::memcpy(at + offsetof(P, ticket), &ticket, sizeof(ticket));
  if (NP == 1) std::memcpy(at + offsetof(P, before), &probs->before, sizeof(CommitParams));
  l.func = func;
  l.grid = dim3(ctas * (tiles < most ? tiles : most), 1, 1);
  l.block = dim3(threads_of(sums, NP > 1), 1, 1);
  l.smem = SMEM_BYTES;
  return l;
}

// Problems of a launch with a parameter block of 5 KB instead of 32, whose copies cost the host 2 to 3 us a launch: two problems of
// 256 x 256 x 256 by qe_gemm_fp8_group 12.9 us for 15.3, eight 24 for 27; F, dI and dW of four such linears, their calls sharing
// launches, 123 for 132 (a graph keeps its blocks: 114 either way).  Blocks of up to sixteen gain nothing over eight, nor do
// small blocks for sums, which go out a few times a step: 5 KB and 32 within 1 % on steps of 2 to 64 linears.
constexpr uint32_t kFew = 8;


Launch make_any(const GemmDesc* probs, uint32_t n, int num_sms) {
  const bool sums = probs[n - 1].sum;  // (they are the last ones)
  if (n == 1 && !sums) {
    const bool alone = one_cta(*probs, num_sms);
    return make_launch<1>(probs, n, num_sms, alone ? (const void*)gemm_fp8_kernel : (const void*)gemm_fp8_pair_kernel, false, alone);
  }
  if (!sums && n <= kFew) return make_launch<kFew>(probs, n, num_sms, (const void*)gemm_fp8_pair_group_kernel<kFew>, false);
  if (!sums) return make_launch<kMaxProblems>(probs, n, num_sms, (const void*)gemm_fp8_pair_group_kernel<kMaxProblems>, false);
  // Output buffers of a sum's epilogue warps, for each of which there is one operand stage less than six.  Short products are as
  // good as never short of operands and want to be rid of their results, long ones the other way round: us a step with four / three / one,
  // 256 tokens 1294 / 1313 / 1446 (4096 / 11008 layer) and 451 / 456 / 498 (2048 / 8192), 512 tokens 4638 / 4597 / 4723 (48 linears of 1024),
  // 768 748 / 734 / 747 (eight of 2048), 1024 740 / 746 / 722 (six of 2048), 2048 2331 / 2122 / 2120 (block of hidden 2048).
  uint32_t longest = 0;
  for (uint32_t i = 0; i < n; ++i)
    if (probs[i].sum && probs[i].Kc > longest) longest = probs[i].Kc;
  return make_launch<kMaxProblems>(probs, n, num_sms, longest <= 256 ? (const void*)gemm_fp8_pair_wide_kernel<4>
                                   : longest <= 768 ? (const void*)gemm_fp8_pair_wide_kernel<3> : (const void*)gemm_fp8_pair_wide_kernel<1>, true);
}

}  // namespace

bool whole_row_tiles(uint32_t M) { return M % 256 == 0; }

cudaError_t gemm_prepare() {
  for (const void* f : {(const void*)gemm_fp8_pair_chain_kernel, (const void*)gemm_fp8_kernel, (const void*)gemm_fp8_pair_kernel, (const void*)gemm_fp8_pair_group_kernel<kFew>,
                        (const void*)gemm_fp8_pair_group_kernel<kMaxProblems>, (const void*)gemm_fp8_pair_wide_kernel<1>,
                        (const void*)gemm_fp8_pair_wide_kernel<3>, (const void*)gemm_fp8_pair_wide_kernel<4>}) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

bool chained_fit(int num_sms, cudaStream_t stream) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((uint32_t)num_sms / 2u * 2u, 1, 1);
  cfg.blockDim = dim3(threads_of(false, true), 1, 1);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim = {2, 1, 1};
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, (const void*)gemm_fp8_pair_chain_kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();  // (the question's, not a call's)
    return false;
  }
  return clusters >= num_sms / 2;
}

bool make_gemm_group(const GemmDesc* probs, uint32_t n, int num_sms, Launch* out) {
  if (n && probs->chained) {
    if (!launch_chained(probs, n, num_sms)) return false;
    *out = make_launch<kMaxChained>(probs, n, num_sms, (const void*)gemm_fp8_pair_chain_kernel, false);
    out->cooperative = true;
    return true;
  }
  if (n < 2 || n > kMaxProblems) return false;
  for (uint32_t i = 0; i < n && n > most_committing(num_sms); ++i)
    if (probs[i].commit.st && probs[i].commit.early_mask) return false;
  *out = make_any(probs, n, num_sms);
  return true;
}

// (the fields stand at the front of every launch's parameter block)
static void set_commits(Launch* l, uint32_t* word, uint32_t op) {
  using P = GemmLaunchParams<1>;
  static_assert(offsetof(P, commits) == 0 && offsetof(P, n) == offsetof(GemmLaunchParams<kMaxProblems>, n), "");
  std::memcpy(l->params.data() + offsetof(P, commits), &word, sizeof(word));
  std::memcpy(l->params.data() + offsetof(P, commits_op), &op, sizeof(op));
}
uint32_t announce_commits(Launch* gemm, uint32_t* word) {
  set_commits(gemm, word, 1u);
  uint32_t n;
  std::memcpy(&n, gemm->params.data() + offsetof(GemmLaunchParams<1>, n), sizeof(n));
  return n;
}
void withdraw_commits(Launch* gemm, uint32_t* word) { set_commits(gemm, word, 2u); }

uint32_t gemm_width(const GemmDesc* probs, uint32_t n, int num_sms) { return choose_width(probs, n, (uint32_t)num_sms / 2u); }

Launch make_gemm(const GemmDesc& d, int num_sms) { return make_any(&d, 1, num_sms); }

}  // namespace qe
