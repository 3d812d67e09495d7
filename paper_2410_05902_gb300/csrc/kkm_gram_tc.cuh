#pragma once
// tcgen05 / TMA form of the two Gram passes (BF16, split-BF16 and TF32 products).
//
// One persistent CTA per SM walks the work items round-robin. For each item
//   G = A B^T            tcgen05.mma kind::f16 (BF16) or kind::tf32 (TF32),
//                        FP32 in TMEM; operands streamed by TMA through a
//                        192 KB ring of 128B-swizzled shared-memory slices
//   K = kernel(||a||^2 + ||b||^2 - 2G)      in registers after tcgen05.ld
//   weighted row sums of K                  FP32 per row, see below
// The split form (x = hi + lo) runs the K loop three times over the slice
// pairs (hi,hi), (hi,lo), (lo,hi) into the same accumulator.
//
// Distance pass (mode 0): an item is (128-row batch tile, TNV-row support tile
// of one center; TNV = 256 by default, 64 or 128 on request), and it writes
// part[tile][x] = sum_y w_y K(x, y), one partial per row and tile.
// Window pass (mode 1, the norm recurrence of Sec. 4 with the drops of
// Eq. (1)): an item is (128 support rows, 128 support rows) of one center,
// rows from the dropped prefix D (kind 0) or the new block B (kind 1), and it
// writes four sums:
//   kind 0: A = sum_{p in D, q in W} w_p w_q K, Bdd = sum_{p, q in D} w_p w_q K,
//           E = sum_{p in D, q in B} w_p K          (W: the old window)
//   kind 1: M = sum_{p, q in B} K.
// Mode 2 runs the window items of the previous step's update and the distance
// items of this step in one launch.
//
// Roles: warp 0 issues the operand tiles' TMA copies; warp 1 issues the MMAs
// (one elected lane) and owns the TMEM allocation (up to four accumulators);
// warps 2-17 are the epilogue, four groups of four warps, one warp per TMEM
// lane quadrant; warp 18 stages each item's metadata (norms, weights, data
// indices, and the item's row and column ranges) into a ring of slots with
// per-lane 16-byte asynchronous copies; warp 19 (modes 1 and 2) carries the
// norm of every center whose last window item has finished. A copy through the
// TMA unit costs the issuing thread a few hundred cycles, so an item takes as
// few of them as possible: its B tile, and its A tile only when the row tile
// changes (the batch tile stays resident while consecutive items share it).
//
// Teams: with four accumulators (64- and 128-column tiles, window items) each
// group is a team and takes every fourth item whole; with two (256-column
// tiles) two groups form a team, take every other item and split its columns,
// each writing its own partial. Either way every waiter on a barrier sees each
// of its phases in order. A run with fewer than NTEAM items per SM runs every
// item on all four groups, each on a quarter of the columns, and the groups'
// sums meet in shared memory (chosen per run, so that a run's results do not
// depend on how a launch splits its items).
//
// CTA pairs (PAIR, distance pass of 128- or 256-column tiles whose operands stream):
// two CTAs of a cluster take two row tiles against the same support tile, and
// the tcgen05 pair form multiplies both at once: each CTA stages its own A rows
// and half of the B rows, so a 128-byte slice costs 32 KB of operand traffic per
// CTA where a CTA alone takes 48 KB. Alone, operands arrived at about 42 bytes per
// clock and SM while the MMAs could use 96, which is what bounded rows of
// more than 128 BF16 columns.
// The even CTA's MMA warp issues for both; its full barriers count both CTAs' copies,
// its commits arrive on both CTAs' stage and accumulator barriers, and both
// epilogues release an accumulator at the even CTA. With 128-column tiles two
// items of a row tile share one pass over its slices. Row tiles, partials and
// their sums are those of the single-CTA form, bit for bit.
//
// Gaussian kernel values without a per-element row term: with rc = -log2(e)
// ||x||^2 / kappa and t = (2 log2(e) / kappa) g - log2(e) ||y||^2 / kappa,
//   K(x, y) = 2^(rc + t) = 2^rc 2^t,
// so a row's weighted sum is 2^rc sum_y w_y 2^t: one FMA for t, one MUFU ex2
// and one FMA into the sum per element. t <= -rc, so 2^t stays finite while
// -rc <= 100; a warp whose rows pass that bound uses the full exponent.
//
// Every mbarrier wait is bounded. A wait that runs out sets ST_TIMEOUT and
// makes the role stop. On the way out the producer waits for its last copies
// to land and the MMA warp waits for its last MMAs, so TMEM is freed only once
// nothing is in flight.
#include <algorithm>
#include <cstddef>
#include <cuda.h>
#include <cudaTypedefs.h>

#include <type_traits>

#include "kkm_internal.cuh"

namespace kkm {
namespace {

constexpr int TM = 128;                         // A rows per tile = TMEM lanes
constexpr int KS = 64;                          // BF16 columns per slice (one 128-byte swizzle row)
constexpr int A_BYTES = TM * KS * 2;            // 16 KB: the A tile of one slice
// operand formats: BF16 (one product), split BF16 (hi.hi + hi.lo + lo.hi), TF32
// (FP32 rows rounded to TF32; a 128-byte slice row holds 32 of them)
constexpr int OP_BF16 = 0, OP_X3 = 1, OP_TF32 = 2;
constexpr int RING_BYTES = 192 * 1024;          // shared memory for the operands
constexpr int STAGES = 16;                      // most stages any layout uses
constexpr int A_RES_MAX = 96 * 1024;            // largest batch tile kept resident (all its slices)
// Operand layout, per launch (Layout below). A slice is 128 bytes of every
// operand row: 64 BF16 or 32 TF32 values. The split form holds hi and lo
// tiles of each operand and runs 12 MMAs per slice (hi.hi, hi.lo, lo.hi).
//   resident A: the A tile's slices stay in shared memory while consecutive
//               items share it (same batch or support row tile); a stage
//               holds one slice of the B tile. A is reloaded only when the
//               row tile changes.
//   streaming:  (A too large to keep) a stage holds one slice of A and B.
constexpr int NEPI = 16;                         // epilogue warps (2 .. 17): four on each scheduler
constexpr int NGRP = 4;                          // epilogue groups, one warp per TMEM lane quadrant each
constexpr int MWARP = 2 + NEPI;                  // the metadata warp
// TMA warp, MMA warp, epilogue, metadata warp and, where there are window items, the norm warp
template <int MODE> constexpr int nthreads() { return 32 * (MWARP + (MODE == 0 ? 1 : 2)); }
constexpr int WSUM_BYTES = 16;                   // a window sum in shared memory (FixedSum, or one FP64)
constexpr int NSLOT = 4;                         // finished window items waiting for the norm warp
constexpr uint64_t WAIT_LIMIT_NS = 2000000000ull;   // 2 s per wait
constexpr float ROW_EXP_FLOOR = -100.0f;        // Gaussian: rc at or above it keeps 2^t finite

// TMEM accumulators (TNV columns each, at most 512 columns), teams of
// groups (one per accumulator), groups per team (= partials per tile), and
// metadata slots
template <int TNV> struct Geo {
  static constexpr int NACC = 512 / TNV < 4 ? 512 / TNV : 4;
  static constexpr int NTEAM = NACC < NGRP ? NACC : NGRP;
  static constexpr int GPT = NGRP / NTEAM;
  static constexpr int MS = TNV == 256 ? 5 : TNV == 128 ? 6 : 8;
  static constexpr uint32_t TMEM_COLS = (uint32_t)(NACC * TNV);
};
using WG = Geo<WPASS_TNV>;                       // window items' accumulators and teams, whatever the distance tile
constexpr uint32_t META_ARRIVALS = 33;           // 32 lanes' asynchronous arrivals + lane 0's release

__device__ __forceinline__ void tma_load_2d(bool lead, void* dst, const CUtensorMap* map, uint64_t* bar, int x,
                                            int y);

// Operand layout of one launch (identical in every role). Byte offsets are
// from the 1024-aligned start of the operand region; every tile starts on a
// multiple of 1024 bytes, as the 128-byte swizzle needs. A tile's slices are
// laid out hi slices first, then (split form) lo slices.
struct Layout {
  bool res;            // A resident; a stage holds one item's whole B tile
  int nsl;             // slices of one operand tile (nks, twice that for the split form)
  int a_bytes;         // resident A region (res), else 0
  int sb;              // bytes per stage
  int nst;             // stages
};
template <bool X3, int TNV>
__device__ __forceinline__ Layout layout(int nks) {
  constexpr int BT = TNV * KS * 2;              // one B slice (TNV rows x 128 bytes)
  Layout L;
  L.nsl = nks * (X3 ? 2 : 1);
  const int a = L.nsl * A_BYTES, sbr = L.nsl * BT;
  // resident only if the A tile fits and at least two whole B tiles fit beside it
  L.res = a <= A_RES_MAX && (RING_BYTES - a) / sbr >= 2;
  L.a_bytes = L.res ? a : 0;
  L.sb = L.res ? sbr : (X3 ? 2 : 1) * (A_BYTES + BT);   // streaming: one slice of A and B
  const int n = (RING_BYTES - L.a_bytes) / L.sb;
  L.nst = n < STAGES ? n : STAGES;
  return L;
}

// CTA pairs always stream: a stage holds one slice of A and of this CTA's half of
// B: 128 rows of one 256-column tile, or 64 of each of two 128-column tiles.
template <bool X3>
__device__ __forceinline__ Layout pair_layout(int nks) {
  Layout L;
  L.nsl = nks * (X3 ? 2 : 1);
  L.res = false;
  L.a_bytes = 0;
  L.sb = (X3 ? 2 : 1) * 2 * A_BYTES;
  const int n = RING_BYTES / L.sb;
  L.nst = n < STAGES ? n : STAGES;
  return L;
}

// The slices of a whole tile (hi slices, then lo slices at column dp) into dst + t * tb.
__device__ __forceinline__ void tile_issue(bool lead, int n, int nks, int dp, int kse, uint8_t* dst, int tb,
                                           const CUtensorMap* tm, uint64_t* bar, int y) {
  for (int t = 0; t < n; ++t)
    tma_load_2d(lead, dst + t * tb, tm, bar, t < nks ? t * kse : dp + (t - nks) * kse, y);
}

// Instruction descriptor of tcgen05.mma kind::f16 / kind::tf32: D FP32
// (bits 4-5 = 1), A and B BF16 (type 1) or TF32 (type 2) in bits 7-9 and
// 10-12, both K-major (bits 15, 16 = 0), N >> 3 in bits 17-22, M >> 4 in
// bits 24-28.
template <int OP>
__device__ __forceinline__ uint32_t idesc(uint32_t n, uint32_t m = TM) {
  constexpr uint32_t t = OP == OP_TF32 ? 2u : 1u;
  return (1u << 4) | (t << 7) | (t << 10) | ((n >> 3) << 17) | ((m >> 4) << 24);
}

// An item's ranges. Distance item: only tnew, the tile's columns. Window item:
// row and column ranges relative to the item's first row and column (both
// 4-aligned positions of the center's region).
struct ItemDesc {
  int32_t kind;        // 0: rows of D against W and B; 1: rows of B against B
  int32_t rlo, rhi;    // rows [rlo, rhi) of the tile are in the row range
  int32_t dnew;        // columns below dnew are dropped rows (D)
  int32_t told;        // columns below told are the old window W (D included)
  int32_t tnew;        // columns in [told, tnew) are the new block B
  int32_t j;           // center
  int32_t pad0;
};

// Metadata of one item, copied by the metadata warp. col[0] = ||y||^2, col[1] = w,
// col[2] = data index (bits) of the TNV B rows; row[0] = ||a||^2, row[1] =
// data index, row[2] = w (window pass) of the 128 A rows.
template <int TNV> struct MetaSlot {
  float col[3][TNV];
  float row[3][TM];
  ItemDesc desc;
};

template <int TNV> struct Shared {
  uint64_t full[STAGES];
  uint64_t empty[STAGES];
  uint64_t afull;                // resident A tile landed
  uint64_t afree;                // the MMAs on the previous resident A tile are done
  uint32_t mark[STAGES];         // 1: the stage's item brings a new resident A tile
  uint64_t tfull[4];
  uint64_t tempty[4];
  uint64_t wfull[4];             // the same for window items
  uint64_t wempty[4];
  uint64_t mfull[8];
  uint64_t mempty[8];
  uint64_t mma_done;
  uint64_t nfull[NSLOT];         // window items finished, for the norm warp
  uint64_t nempty[NSLOT];
  int32_t nj[NSLOT];             // their centers (-1: the item was skipped)
  uint32_t tmem_base;
  uint32_t pad;
  long long gtot;                // run groups: the class's weighted item total
  int gseg[4];                   // run groups: the next segment (run, first item, end item), whole CTAs per run
  alignas(16) Dev gdev;          // run groups: the segment's run (a shared copy: no reloads after global stores)
  alignas(16) MetaSlot<TNV> ring[Geo<TNV>::MS];   // 16-byte asynchronous copies land here
  float red[2][NGRP][4][32];     // distance items, all-groups mode: row sums (item parity, group, quadrant, row)
  alignas(16) unsigned char wq[NGRP][2][3 * 4 * WSUM_BYTES];   // window items: sums (group, parity; class, quadrant)
};

template <int TNV> constexpr int smem_bytes() { return 1024 + RING_BYTES + (int)sizeof(Shared<TNV>); }
// the metadata slots take 16-byte cp.async copies: each slot, and every array in it, on a 16-byte boundary
static_assert(offsetof(Shared<64>, ring) % 16 == 0 && offsetof(Shared<128>, ring) % 16 == 0 &&
                  offsetof(Shared<256>, ring) % 16 == 0 && sizeof(MetaSlot<64>) % 16 == 0 &&
                  sizeof(MetaSlot<128>) % 16 == 0 && sizeof(MetaSlot<256>) % 16 == 0,
              "metadata ring misaligned for 16-byte copies");
static_assert(smem_bytes<128>() <= 232448 && smem_bytes<256>() <= 232448 && smem_bytes<64>() <= 232448,
              "shared memory per CTA");

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_inval(uint64_t* b) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(b)) : "memory");
}

// dist_tc_body's lifecycle flags: allocate TMEM on entry, free it on exit,
// invalidate the barriers before initialising them (a later segment)
constexpr int TC_ALLOC = 1, TC_FREE = 2, TC_REINIT = 4;

__device__ __forceinline__ void mbar_expect_tx(bool lead, uint64_t* b, uint32_t bytes) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t"
      "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(smem_u32(b)), "r"(bytes),
      "r"((uint32_t)lead)
      : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b, uint32_t count = 1) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Waits for the phase of parity `parity` to complete; false after WAIT_LIMIT_NS.
__device__ bool mbar_wait(uint64_t* b, uint32_t parity, uint64_t limit_ns = WAIT_LIMIT_NS) {
  if (mbar_try_wait(b, parity)) return true;
  const uint64_t t0 = globaltimer();
  while (true) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(b, parity)) return true;
    if (globaltimer() - t0 > limit_ns) return false;
  }
}

// The producer and MMA warps run converged, all lanes computing the same
// values, and one lane (`lead`) issues: the copy and MMA instructions take their
// operands from uniform registers, which the compiler can use only for values
// that are the same over a converged warp. Issued from a one-lane branch every
// operand went through a register move first, about 170 cycles an MMA.
__device__ __forceinline__ void tma_load_2d(bool lead, void* dst, const CUtensorMap* map, uint64_t* bar, int x,
                                            int y) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n\t}"
      ::"r"(smem_u32(dst)), "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"((uint32_t)lead)
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile stored as rows of
// 128 bytes with the 128-byte swizzle (the layout TMA writes with
// CU_TENSOR_MAP_SWIZZLE_128B): start address >> 4 in bits 0-13, leading byte
// offset 16 (unused by swizzled K-major layouts), stride byte offset 1024
// (8 rows x 128 B) in bits 32-45, descriptor version 1 in bits 46-47,
// swizzle mode 2 (128B) in bits 61-63. The low word changes with the tile (a
// 32-byte K step adds 2 to it), the high word never.
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return ((saddr >> 4) & 0x3FFFu) | (1u << 16); }
constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);

// One MMA on a 32-byte K step of the 128-byte swizzled rows: K = 16 BF16
// values (kind::f16) or K = 8 TF32 values (kind::tf32).
// PAIR: M = 256, rows 0-127 in this CTA and 128-255 in its peer (the addresses
// hold in both).
template <int OP, bool PAIR = false>
__device__ __forceinline__ void mma_op(bool lead, uint32_t d_tmem, uint32_t alo, uint32_t blo, uint32_t idesc,
                                       uint32_t accum) {
#define KKM_MMA(group, kind)                                                                     \
  asm volatile(                                                                                  \
      "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %6, 0;\n\t" \
      "mov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\t"                                       \
      "@q tcgen05.mma.cta_group::" group "." kind " [%0], da, db, %3, p;\n\t}"                   \
      ::"r"(d_tmem), "r"(alo), "r"(blo), "r"(idesc), "r"(accum), "r"(DESC_HI), "r"((uint32_t)lead) \
      : "memory")
  if constexpr (OP == OP_TF32 && PAIR) KKM_MMA("2", "kind::tf32");
  else if constexpr (OP == OP_TF32) KKM_MMA("1", "kind::tf32");
  else if constexpr (PAIR) KKM_MMA("2", "kind::f16");
  else KKM_MMA("1", "kind::f16");
#undef KKM_MMA
}

template <bool PAIR = false>
__device__ __forceinline__ void mma_commit(bool lead, uint64_t* bar) {
#define KKM_COMMIT(group)                                                                          \
  asm volatile(                                                                                    \
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"                                            \
      "@q tcgen05.commit.cta_group::" group ".mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" \
      ::"r"(smem_u32(bar)), "r"((uint32_t)lead)                                                    \
      : "memory")
  if constexpr (PAIR) KKM_COMMIT("2");
  else KKM_COMMIT("1");
#undef KKM_COMMIT
}

// CTA pairs. The address of a shared variable in the pair's even CTA:
__device__ __forceinline__ uint32_t lead_addr(const void* p) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(smem_u32(p)));
  return a;
}
// both CTAs' threads meet here
__device__ __forceinline__ void pair_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// a copy into this CTA's shared memory that counts at a barrier of the even CTA
__device__ __forceinline__ void tma_load_2d_pair(bool lead, void* dst, const CUtensorMap* map, uint32_t bar, int x,
                                                 int y) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%3, %4}], [%2];\n\t}"
      ::"r"(smem_u32(dst)), "l"((uint64_t)map), "r"(bar), "r"(x), "r"(y), "r"((uint32_t)lead)
      : "memory");
}
// arrives on the barrier at bar's address in both CTAs once the pair's MMAs so far are done
__device__ __forceinline__ void mma_commit_pair(bool lead, uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t.reg .b16 both;\n\tsetp.ne.b32 q, %1, 0;\n\tmov.b16 both, 3;\n\t"
      "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], both;\n\t}"
      ::"r"(smem_u32(bar)), "r"((uint32_t)lead)
      : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}

// One thread's hand-over of a value through a slot: waits for the slot to be
// free (phase `parity` of empty), writes and arrives on full. On a wait that
// runs out the slot and its barrier stay untouched, since the reader may not
// have taken the value before; the caller gives up handing over.
__device__ __forceinline__ bool slot_put(uint64_t* empty, uint32_t parity, int32_t* slot, int32_t v, uint64_t* full,
                                         uint64_t limit_ns = WAIT_LIMIT_NS) {
  if (!mbar_wait(empty, parity, limit_ns)) return false;
  *slot = v;
  mbar_arrive(full);
  return true;
}

// A whole warp's wait, the same answer on every lane.
__device__ __forceinline__ bool warp_wait(uint64_t* b, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(b, parity));
}

// tcgen05.ld .16x256b.xNB: 16 TMEM lanes starting at the address's lane, NB
// blocks of 8 consecutive FP32 columns. Thread t receives, for block j,
//   v[4j]   = (lane t/4,     column 8j + 2(t%4)),  v[4j+1] = the next column,
//   v[4j+2] = (lane t/4 + 8, column 8j + 2(t%4)),  v[4j+3] = the next column.
// Each column value is needed by 4 threads instead of 32 (the 32x32b shape
// gives a thread one lane and all columns), which cuts the per-column
// metadata the epilogue reads from shared memory by 4x.
template <int NB>
__device__ __forceinline__ void tmem_ld16x256(uint32_t taddr, float (&v)[4 * NB]) {
  uint32_t r[4 * NB];
  if constexpr (NB == 8) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
          "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
          "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
  } else if constexpr (NB == 4) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
  } else {
    static_assert(NB == 2, "tmem_ld16x256: 2, 4 or 8 blocks");
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr));
  }
#pragma unroll
  for (int i = 0; i < 4 * NB; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Kernel values of one row against two columns from their Gram entries g, for
// the kernels without the factored Gaussian form: the Laplacian, the linear
// and the polynomial kernel, and the Gaussian with its full exponent.
// Gaussian: rc = ||x||^2 * negc and cc = ||y||^2 * negc (negc = -log2(e)/kappa),
//           K = 2^(rc + cc - 2 negc g).
// Laplacian: rc = ||x||^2, cc = ||y||^2, K = 2^(negc * sqrt(max(D^2, 0))).
// Both give exactly 1 when the two rows are the same data point (K(x,x) = 1).
template <int KIND>
__device__ __forceinline__ float2 kernel_pair(float2 g, float rc, float2 cc, int xi, int2 yi, float negc,
                                              float coef0, int degree) {
  float2 k;
  if constexpr (KIND == K_GAUSS) {
    const float2 a = __ffma2_rn(g, make_float2(-2.0f * negc, -2.0f * negc), __fadd2_rn(make_float2(rc, rc), cc));
    k.x = xi == yi.x ? 1.0f : ex2_approx(a.x);
    k.y = xi == yi.y ? 1.0f : ex2_approx(a.y);
  } else if constexpr (KIND == K_LAPLACE) {
    const float2 d2 = __ffma2_rn(g, make_float2(-2.0f, -2.0f), __fadd2_rn(make_float2(rc, rc), cc));
    k.x = xi == yi.x ? 1.0f : ex2_approx(sqrt_approx(fmaxf(d2.x, 0.0f)) * negc);
    k.y = xi == yi.y ? 1.0f : ex2_approx(sqrt_approx(fmaxf(d2.y, 0.0f)) * negc);
  } else if constexpr (KIND == K_LINEAR) {
    k.x = yi.x == -2 ? 0.0f : g.x;
    k.y = yi.y == -2 ? 0.0f : g.y;
  } else {
    float rx = 1.0f, ry = 1.0f;
    for (int p = 0; p < degree; ++p) { rx *= g.x + coef0; ry *= g.y + coef0; }
    k.x = yi.x == -2 ? 0.0f : rx;
    k.y = yi.y == -2 ? 0.0f : ry;
  }
  return k;
}


// 16-byte asynchronous copy global -> shared through the LSU (not the TMA
// unit), and the asynchronous arrive that follows this thread's earlier ones.
__device__ __forceinline__ void cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_arrive_noinc(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// A chunk is 8 NB accumulator columns of a warp's 32 rows: two 16-lane loads.
// Thread t receives, for block j (8 columns), rows g4 = t/4 and g4 + 8 from
// the first load (v0[4j..4j+3]) and g4 + 16, g4 + 24 from the second (v1),
// columns 8j + 2(t%4) and the next one. Row u of the thread (0..3) is
// g4 + 8u: u = 0, 1 in v0 at offset 4j + 2u, u = 2, 3 in v1 at 4j + 2(u-2).
template <int NB>
__device__ __forceinline__ void chunk_load(uint32_t taddr, float (&v0)[4 * NB], float (&v1)[4 * NB]) {
  tmem_ld16x256<NB>(taddr, v0);                 // rows g4, g4 + 8
  tmem_ld16x256<NB>(taddr + (16u << 16), v1);   // rows g4 + 16, g4 + 24
  tmem_wait_ld();
}

template <int NB>
__device__ __forceinline__ float2 gram2(const float (&v0)[4 * NB], const float (&v1)[4 * NB], int j, int u) {
  const int o = 4 * j + 2 * (u & 1);
  return u < 2 ? make_float2(v0[o], v0[o + 1]) : make_float2(v1[o], v1[o + 1]);
}

// Distance pass, Gaussian: acc[u] += w_y 2^t over the chunk's columns, with
// t = C2 g + cc (FAST, the row term 2^rc applied to the row sum later) or
// t = C2 g + cc + rc (full exponent). c is this thread's first column.
template <int NB, bool FAST>
__device__ __forceinline__ void gauss_chunk(const float (&v0)[4 * NB], const float (&v1)[4 * NB],
                                            const float* __restrict__ yn, const float* __restrict__ w, int c,
                                            float negc, float2 C2, const float (&rc)[4], float2 (&acc)[4]) {
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    const float2 y2 = *reinterpret_cast<const float2*>(yn + c + 8 * j);
    const float2 w2 = *reinterpret_cast<const float2*>(w + c + 8 * j);
    const float2 cc = __fmul2_rn(y2, make_float2(negc, negc));
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float2 bias = FAST ? cc : __fadd2_rn(cc, make_float2(rc[u], rc[u]));
      const float2 t = __ffma2_rn(gram2<NB>(v0, v1, j, u), C2, bias);
      acc[u] = __ffma2_rn(w2, make_float2(ex2_approx(t.x), ex2_approx(t.y)), acc[u]);
    }
  }
}

// Distance pass, other kernels: acc[u] += w_y K(x_u, y) by kernel_pair.
template <int KIND, int NB>
__device__ __forceinline__ void generic_chunk(const float (&v0)[4 * NB], const float (&v1)[4 * NB],
                                              const float* __restrict__ yn, const float* __restrict__ w,
                                              const float* __restrict__ yi, int c, float negc, float coef0,
                                              int degree, const float (&rc)[4], const int (&xi)[4],
                                              float2 (&acc)[4]) {
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    const float2 y2 = *reinterpret_cast<const float2*>(yn + c + 8 * j);
    const float2 w2 = *reinterpret_cast<const float2*>(w + c + 8 * j);
    const int2 i2 = *reinterpret_cast<const int2*>(yi + c + 8 * j);
    const float2 cc = (KIND == K_GAUSS) ? __fmul2_rn(y2, make_float2(negc, negc)) : y2;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      acc[u] = __ffma2_rn(w2, kernel_pair<KIND>(gram2<NB>(v0, v1, j, u), rc[u], cc, xi[u], i2, negc, coef0,
                                                degree), acc[u]);
  }
}

__device__ __forceinline__ float pick4(const float (&v)[4], int u) {
  return u == 0 ? v[0] : (u == 1 ? v[1] : (u == 2 ? v[2] : v[3]));
}

// Sum of a row's values over the four lanes that hold it (lanes 4r .. 4r+3).
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v;
}

// The window pass's sums where kernel values are at most 1 (Gaussian,
// Laplacian). FP64 issues at 1/64 of the FP32 rate on this chip (2 lane
// operations per clock and SM): the 24 FP64 instructions that each of the 16
// epilogue warps took per item (conversions, products and three 32-lane
// reductions) were about 6100 cycles of it, more than the rest of an item. Yet
// the sums feed a recurrence and keep more than FP64's bits: a row's sum is
// three FP32 words (Trip32: the errors of the first two words' sums are carried
// exactly), and the 32 rows of a warp are added as fixed-point numbers of 66
// bits below the largest row's exponent, three 22-bit limbs each, by integer
// warp reductions (FixedSum), so that the sum is off by no more than 2^-60 of
// itself. Only classes of columns that an item has are summed. 90 % of 8192 rows
// in one of 10 centers, BF16: 213 us a step with sums of two FP32 words (48 bits)
// for all three classes, 188 now; even batches of 4096 in 50 centers 53.4 and 54.9.
struct Trip32 {
  float h, m, l;
};
// (l0 + 2^-22 l1 + 2^-44 l2) 2^e
struct FixedSum {
  int l0, l1, l2, e;
};
constexpr int NOT_FINITE = 1 << 20;              // e of a sum with a value that is not finite
// x, |x| < 2^22, as an integer, and what it leaves
__device__ __forceinline__ int limb(float x, float& rest) {
  constexpr float MAGIC = 12582912.0f;           // 1.5 * 2^23: the sum's last bit is 1
  const float t = __fadd_rn(x, MAGIC);
  rest = __fsub_rn(x, __fsub_rn(t, MAGIC));
  return __float_as_int(t) - __float_as_int(MAGIC);
}

// zero; addf adds an FP32 quarter sum to a row's sum; rows gives the sum of w r
// over a warp's 32 rows, value that sum in FP64.
template <int KIND> struct WindowSum {
  using Row = Trip32;
  using Sum = FixedSum;
  static __device__ __forceinline__ Row zero() { return Row{0.0f, 0.0f, 0.0f}; }
  static __device__ __forceinline__ Row addf(Row a, float b) {
    float e, g;
    const float h = two_sum(a.h, b, e), m = two_sum(a.m, e, g);
    return Row{h, m, __fadd_rn(a.l, g)};
  }
  static __device__ __forceinline__ Sum rows(Row r, float w) {
    // w r = h + m + l, m and l at most 2^-23 and 2^-46 or so of h
    const float h = __fmul_rn(r.h, w), e = __fmaf_rn(r.h, w, -h);
    const float q = __fmul_rn(r.m, w), f = __fmaf_rn(r.m, w, -q);
    float g;
    const float m = two_sum(q, e, g), l = __fadd_rn(__fmaf_rn(r.l, w, f), g);
    const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(h) & 0x7fffffffu) >> 23;
    if (top >= 255u) return Sum{0, 0, 0, NOT_FINITE};
    // every |h| is below 2^21 times 2^e (nothing under 2^-100 needs a unit of its own)
    const unsigned ex = top < 27u ? 27u : top;
    const float inv = __uint_as_float((274u - ex) << 23);
    float r1, r2, r3, r4, r5;
    Sum s;
    s.l0 = limb(__fmul_rn(h, inv), r1);
    s.l1 = limb(__fmul_rn(r1, 0x1p22f), r2) + limb(__fmul_rn(__fmul_rn(m, inv), 0x1p22f), r3);
    s.l2 = limb(__fmul_rn(__fadd_rn(r2, r3), 0x1p22f), r4) + limb(__fmul_rn(__fmul_rn(l, inv), 0x1p44f), r5);
    s.l0 = __reduce_add_sync(0xffffffffu, s.l0);
    s.l1 = __reduce_add_sync(0xffffffffu, s.l1);
    s.l2 = __reduce_add_sync(0xffffffffu, s.l2);
    s.e = (int)ex - 147;
    return s;
  }
  static __device__ __forceinline__ double value(Sum s) {
    if (s.e == NOT_FINITE) return __longlong_as_double(0x7ff8000000000000ll);
    // l0 and l1 (together below 2^50) and l2 as the last bits of doubles of known
    // exponents: one FP64 subtraction each and one addition
    const long long q = ((long long)s.l0 << 22) + s.l1 + (1ll << 51);
    const int k = (s.e - 22) << 20, k2 = (s.e - 44) << 20;
    const double a = __hiloint2double(0x43300000 + (int)(q >> 32) + k, (int)q);
    const double b = __hiloint2double(0x43300000 + k2, s.l2 ^ (int)0x80000000);
    return (a - __hiloint2double(0x43380000 + k, 0)) + (b - __hiloint2double(0x43300000 + k2, (int)0x80000000));
  }
};
// FP64 where kernel values have FP32's whole range.
struct WindowSum64 {
  using Row = double;
  using Sum = double;
  static __device__ __forceinline__ Row zero() { return 0.0; }
  static __device__ __forceinline__ Row addf(Row a, float b) { return a + (double)b; }
  static __device__ __forceinline__ Sum rows(Row r, float w) { return warp_sum_f64(r * (double)w); }
  static __device__ __forceinline__ double value(Sum a) { return a; }
};
template <> struct WindowSum<K_LINEAR> : WindowSum64 {};
template <> struct WindowSum<K_POLY> : WindowSum64 {};

struct Range {
  int lo, hi;
};

// What an epilogue warp knows about its place: its group, its row quadrant and
// its share of an item (teams, column halves and the all-groups mode of the
// header comment).
template <int TNV> struct Place {
  static constexpr int GPT = Geo<TNV>::GPT, QPP = NGRP / GPT;
  int g, q, team, h, lane;
  bool all;
  __device__ Place(int warp, int lane_, bool all_)
      : g((warp - 2) >> 2), q(warp & 3), team(g / GPT), h(g % GPT), lane(lane_), all(all_) {}
  __device__ bool mine(uint32_t local) const { return all || (int)(local % Geo<TNV>::NTEAM) == team; }
  __device__ void arrive(uint64_t* b, uint32_t count = 1) const {
    __syncwarp();
    if (lane == 0) mbar_arrive(b, count);
  }
  // the accumulator's barrier: the even CTA's, where the pair's MMAs are issued
  template <bool PAIR> __device__ void arrive_acc(uint64_t* b) const {
    if constexpr (PAIR) {
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(lead_addr(b));
    } else {
      arrive(b);
    }
  }
  __device__ void sync_all() const { asm volatile("bar.sync 1, %0;" ::"n"(32 * NEPI) : "memory"); }
  __device__ void sync_group() const { asm volatile("bar.sync %0, 128;" ::"r"(2 + g) : "memory"); }
};

// One distance-pass item: group h of the team takes the columns [h TNV / GPT,
// (h+1) TNV / GPT), written as partial h of the tile (in the all-groups mode
// every group a quarter of the columns, and the quarters of each partial meet
// in shared memory). Columns from the tile's width on carry weight 0: the
// chunks past it are skipped, and the last partial may be plain 0. A warp
// covers its quadrant's 32 rows; it releases the accumulator once its last
// chunk is in registers and the metadata slot once its arithmetic is done.
template <int KIND, int TNV, bool PAIR>
__device__ __forceinline__ void dist_item(const Dev& s, Shared<TNV>& sh, uint32_t tmem, const Place<TNV>& pl,
                                          uint32_t local, uint32_t buf, int tile, int row0, int rows, bool dead) {
  constexpr int MS = Geo<TNV>::MS, GPT = Geo<TNV>::GPT, QPP = Place<TNV>::QPP;
  const int g = pl.g, q = pl.q, lane = pl.lane;
  const bool all = pl.all;
  const int g4 = lane >> 2, us = lane & 3, c2 = 2 * us;
  const int rq = g4 + 8 * us;                   // the row this lane reports
  const float negc = s.negc;
  const float2 C2 = make_float2(-2.0f * negc, -2.0f * negc);
  const float coef0 = (float)s.coef0;
  const int degree = s.degree;
  const int ncols = all ? TNV / NGRP : TNV / GPT;
  const int cbeg = all ? g * ncols : pl.h * ncols;
  const int ph = all ? g / QPP : pl.h;          // this group's partial
  const bool lead = !all || g % QPP == 0;       // writes the partial
  const uint32_t ms = local % MS;
  const MetaSlot<TNV>& m = sh.ring[ms];
  float f = 0.0f;
  if (!dead) {
    float rc[4];
    int xi[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = q * 32 + g4 + 8 * u;
      rc[u] = (KIND == K_GAUSS) ? m.row[0][r] * negc : m.row[0][r];
      xi[u] = __float_as_int(m.row[1][r]);
    }
    float2 acc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] = make_float2(0.0f, 0.0f);
    const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + buf * TNV + cbeg;
    bool fast = false;
    if constexpr (KIND == K_GAUSS)
      fast = __all_sync(0xffffffffu, fminf(fminf(rc[0], rc[1]), fminf(rc[2], rc[3])) >= ROW_EXP_FLOOR);
    auto release = [&]() {                      // the accumulator is free again
      if (!all) {
        tc_fence_before();
        pl.template arrive_acc<PAIR>(&sh.tempty[buf]);
      }
    };
    // Whole 16-column blocks of the live columns (the MMA's N ends there): 32 at
    // a time, then a last 16. A chunk's TMEM load takes about 30 cycles; what a warp waits
    // for is its own chain of shared-memory reads, FMAs and exponentials, so
    // the wide chunk (32 elements a lane in flight) does as well as two 16-column
    // ones loaded ahead of each other where items are many (1e6 x 128, b = 4096: 79 us
    // an iteration both ways), and better where a CTA has one or two (70000 x 784,
    // b = 1024: 36.9 -> 34.3 to 35.7 us).
    const int live = min(ncols, m.desc.tnew - cbeg);
    const int n16 = live > 0 ? (live + 15) >> 4 : 0;
    auto math = [&](auto nb, const auto& w0, const auto& w1, int col) {
      constexpr int NB = decltype(nb)::value;
      const int c = cbeg + col + c2;
      if constexpr (KIND == K_GAUSS) {
        if (fast) gauss_chunk<NB, true>(w0, w1, m.col[0], m.col[1], c, negc, C2, rc, acc);
        else gauss_chunk<NB, false>(w0, w1, m.col[0], m.col[1], c, negc, C2, rc, acc);
      } else {
        generic_chunk<KIND, NB>(w0, w1, m.col[0], m.col[1], m.col[2], c, negc, coef0, degree, rc, xi, acc);
      }
    };
    static_assert(TNV / NGRP % 16 == 0, "whole 16-column blocks per group");
    if (n16 == 0) release();
    int q16 = 0;
#pragma unroll 1
    for (; q16 + 2 <= n16; q16 += 2) {
      float v0[16], v1[16];
      chunk_load<4>(tq + q16 * 16, v0, v1);
      if (q16 + 2 == n16) release();
      math(std::integral_constant<int, 4>{}, v0, v1, q16 * 16);
    }
    if (q16 < n16) {
      float v0[8], v1[8];
      chunk_load<2>(tq + q16 * 16, v0, v1);
      release();
      math(std::integral_constant<int, 2>{}, v0, v1, q16 * 16);
    }
    float fr[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) fr[u] = quad_sum(acc[u].x + acc[u].y);
    f = pick4(fr, us);
    if (KIND == K_GAUSS && fast) f *= ex2_approx(pick4(rc, us));   // the row term 2^rc
  }
  const int row = row0 + q * 32 + rq;
  float* out = s.part + ((int64_t)tile * GPT + ph) * s.bpad + row;
  if (!all) {
    if (!dead) {
      pl.arrive(&sh.mempty[ms]);                // this warp is done with the slot
      if (row < rows) *out = f;
    }
  } else {
    float (*red)[4][32] = sh.red[local & 1u];
    red[g][q][rq] = f;
    tc_fence_before();
    pl.sync_all();
    if (lead) {
      if (!dead && row < rows) {
        float v = red[g][q][rq];
        for (int o = 1; o < QPP; ++o) v += red[g + o][q][rq];
        *out = v;
      }
      if (!dead) {
        pl.template arrive_acc<PAIR>(&sh.tempty[buf]);
        pl.arrive(&sh.mempty[ms]);
      }
    }
  }
}

// One window-pass item: per element K(a, b) (its full exponent) into the row's
// sum over one of three classes of columns (w_q on D, w_q on the rest of W, 1 on
// B), then per row the weight w_p (kind 0) or 1 (kind 1) and the sum over the 128
// rows (WindowSum). A row meeting its own copy (same data index) gets K = 1.
//
// The columns are four quarters of 32; a row's FP32 sum of each quarter is taken
// by one thread quad. A group alone takes all four and adds them in order before
// the sum over the rows; in the all-groups mode each group takes one, with a sum
// over the rows of its own, and the first group adds those. Which of the two
// depends on the run's items alone (all_w), so that a run's norms come out the
// same however its launches are grouped. `turn` counts the group's items (buffer
// parity). norms: finished items go to the norm warp (cleared once a hand-over's
// wait has run out).
// Window items have four accumulators and four teams whatever the launch's
// distance tile, as in a launch of their own; beside 256-column tiles two teams
// of two groups met twice an item to exchange their column sums.
// One copy of every part, in loops: as straight-line code for the three classes,
// or with a second copy of the chunk's arithmetic that needs no masks, the
// epilogue of a launch with both kinds of items outgrew the instruction cache.
// 90 % of 8192 rows in one of 10 centers, split BF16: 295 and 249 us a step that
// way, 231 in loops with the same sums.
template <int KIND, int TNV>
__device__ __forceinline__ void window_item(const Dev& s, Shared<TNV>& sh, uint32_t tmem,
                                            const Place<WPASS_TNV>& pl, uint32_t local, uint32_t turn, int item,
                                            bool& norms, bool dead) {
  constexpr int MS = Geo<TNV>::MS;
  constexpr uint32_t SLOT_ARRIVALS = Geo<TNV>::GPT;   // a warp's share of a metadata slot's release
  static_assert(WG::NACC == 4 && WG::GPT == 1 && WPASS_TNV == 128, "four quarters, a group each or one group's");
  using WS = WindowSum<KIND>;
  using Row = typename WS::Row;
  using Sum = typename WS::Sum;
  static_assert(sizeof(Sum) <= WSUM_BYTES, "a shared-memory slot holds one sum");
  const int q = pl.q, lane = pl.lane;
  const int g4 = lane >> 2, us = lane & 3, c2 = 2 * us, rq = g4 + 8 * us;
  const bool all = pl.all;
  const float negc = s.negc;
  const float2 C2 = make_float2(-2.0f * negc, -2.0f * negc);
  const float coef0 = (float)s.coef0;
  const int degree = s.degree;
  const uint32_t buf = local % WG::NACC, ms = local % MS;
  const MetaSlot<TNV>& m = sh.ring[ms];
  const int nq = all ? 1 : NGRP, qlo = all ? pl.g : 0;     // this group's quarters
  const bool lead = qlo == 0;
  ItemDesc dsc{};                                // a dead warp's item has no columns
  float wrow = 0.0f;
  bool rows_here = false;
  float rc[4] = {};
  int xi[4] = {};
  if (!dead) {
    dsc = m.desc;
    rows_here = dsc.rlo < q * 32 + 32 && dsc.rhi > q * 32;   // a quadrant may hold no row of the item
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = q * 32 + g4 + 8 * u;
      rc[u] = (KIND == K_GAUSS) ? __fmul_rn(m.row[0][r], negc) : m.row[0][r];
      xi[u] = __float_as_int(m.row[1][r]);
    }
    const int r = q * 32 + rq;
    wrow = r >= dsc.rlo && r < dsc.rhi ? (dsc.kind == 0 ? m.row[2][r] : 1.0f) : 0.0f;
  }
  // Columns by class: 0 dropped rows D, 1 the rest of the old window W, 2 the new
  // block B (columns from tnew on are in none; a new block's item needs only B).
  // Most items have columns of one class alone, and the others cost nothing.
  auto from = [&](int cls) { return cls == 0 ? 0 : max(cls == 1 ? dsc.dnew : dsc.told, 0); };
  auto to = [&](int cls) { return min(cls == 0 ? dsc.dnew : cls == 1 ? dsc.told : dsc.tnew, WPASS_TNV); };
  auto has = [&](int cls) { return (dsc.kind == 0 || cls == 2) && to(cls) > from(cls); };
  auto release = [&]() {                         // the accumulator and the slot are free again
    tc_fence_before();
    pl.arrive(&sh.wempty[buf]);
    pl.arrive(&sh.mempty[ms], SLOT_ARRIVALS);
  };
  const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + buf * WPASS_TNV;
  auto sum_at = [&](int grp, int cls, int p) -> Sum& {
    return *reinterpret_cast<Sum*>(sh.wq[grp][turn & 1u] + (cls * 4 + p) * WSUM_BYTES);
  };
  const int last = has(2) ? 2 : has(1) ? 1 : 0;
  bool held = !all && !dead;
#pragma unroll 1
  for (int cls = 0; cls < 3; ++cls) {
    if (!has(cls)) continue;
    Row r = WS::zero();
#pragma unroll 1
    for (int t = 0; t < nq; ++t) {
      const int cb = (qlo + t) * 32, lo = max(cb, from(cls)), hi = rows_here ? min(cb + 32, to(cls)) : 0;
      float2 acc[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] = make_float2(0.0f, 0.0f);
      constexpr int NB = 2, CW = 8 * NB;
#pragma unroll 1
      for (int c0 = lo & ~(CW - 1); c0 < hi; c0 += CW) {
        float v0[4 * NB], v1[4 * NB];
        chunk_load<NB>(tq + c0, v0, v1);
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          const int c = c0 + 8 * j + c2;
          const float2 y2 = *reinterpret_cast<const float2*>(&m.col[0][c]);
          float2 w2 = *reinterpret_cast<const float2*>(&m.col[1][c]);
          const int2 i2 = *reinterpret_cast<const int2*>(&m.col[2][c]);
          if (cls == 2) w2 = make_float2(1.0f, 1.0f);
          const unsigned o = (unsigned)(c - lo), span = (unsigned)(hi - lo);
          const bool in0 = o < span, in1 = o + 1u < span;
          w2 = make_float2(in0 ? w2.x : 0.0f, in1 ? w2.y : 0.0f);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float2 gg = gram2<NB>(v0, v1, j, u);
            float2 kv;
            if constexpr (KIND == K_GAUSS) {
              // every rounding spelled out: a run's norms must not depend on which
              // kernel's compilation fuses a product into a sum
              const float2 a = __ffma2_rn(gg, C2, __ffma2_rn(y2, make_float2(negc, negc),
                                                             make_float2(rc[u], rc[u])));
              kv.x = ex2_approx(xi[u] == i2.x ? 0.0f : a.x);
              kv.y = ex2_approx(xi[u] == i2.y ? 0.0f : a.y);
            } else {
              kv = kernel_pair<KIND>(gg, rc[u], y2, xi[u], i2, negc, coef0, degree);
            }
            if constexpr (KIND == K_LINEAR || KIND == K_POLY) {   // unbounded outside the class
              kv.x = in0 ? kv.x : 0.0f;
              kv.y = in1 ? kv.y : 0.0f;
            }
            acc[u] = __ffma2_rn(w2, kv, acc[u]);
          }
        }
      }
      float v = 0.0f;
      if (hi > lo) {
        float f4[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) f4[u] = quad_sum(acc[u].x + acc[u].y);
        v = pick4(f4, us);
      }
      r = WS::addf(r, v);
    }
    if (held && cls == last) {
      release();
      held = false;
    }
    const Sum t = WS::rows(r, wrow);
    if (lane == 0) sum_at(pl.g, cls, q) = t;
  }
  if (held) release();
  const int kind = dsc.kind, center = dsc.j;
  if (all) {
    tc_fence_before();
    pl.sync_all();                               // every warp, dead or not
    if (!lead) return;                           // (their next sums go to the other parity)
    if (!dead) release();
  } else {
    pl.sync_group();                             // every warp of the group, dead or not
  }
  if (q == 2) {                                  // the group's first warp
    if (!dead) {                                 // lane 4 cls + p: quadrant p's sum of class cls
      double v = 0.0;
      if (lane < 12 && has(lane >> 2)) {
        v = WS::value(sum_at(pl.g, lane >> 2, lane & 3));
        if (all)
          v = (v + WS::value(sum_at(1, lane >> 2, lane & 3))) +
              (WS::value(sum_at(2, lane >> 2, lane & 3)) + WS::value(sum_at(3, lane >> 2, lane & 3)));
      }
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      const double vd = __shfl_sync(0xffffffffu, v, 0), vw = __shfl_sync(0xffffffffu, v, 4),
                   vb = __shfl_sync(0xffffffffu, v, 8);
      // A over W (D and the rest), Bdd over D, E (kind 0) or M (kind 1) over B
      if (lane < 4)
        s.wpart[(int64_t)item * 4 + lane] =
            lane == 0 ? vd + vw : lane == 1 ? vd : lane == (kind == 0 ? 2 : 3) ? vb : 0.0;
    }
    if (norms) {                                 // hand the item to the norm warp
      __syncwarp();
      const uint32_t ns = local % NSLOT;
      bool ok = true;
      if (lane == 0)
        ok = slot_put(&sh.nempty[ns], ((local / NSLOT) & 1u) ^ 1u, &sh.nj[ns], dead ? -1 : center, &sh.nfull[ns]);
      if (!__shfl_sync(0xffffffffu, (int)ok, 0)) {   // the norm warp has given up: so does this one, at once
        if (lane == 0) atomicOr(s.status, ST_TIMEOUT);
        norms = false;
      }
    }
  }
}

// The epilogue warps (2-17): window items [rw.lo, rw.hi) first (MODE 1, 2),
// then distance items [rd.lo, rd.hi) (MODE 0, 2).
template <int KIND, int MODE, int TNV, bool PAIR>
__device__ __forceinline__ void epilogue(const Dev& s, Shared<TNV>& sh, uint32_t tmem, Range rw, Range rd, int T,
                                         int rows, int warp, int lane, bool all_w, bool all_d, bool norms,
                                         int rank) {
  constexpr int NACC = Geo<TNV>::NACC, MS = Geo<TNV>::MS;
  // part[] must hold GPT partials per tile, as the host sized it (Dev::ppt)
  bool dead = MODE != 1 && s.ppt != Geo<TNV>::GPT;
  if (dead && lane == 0 && warp == 2) atomicOr(s.status, ST_CAPACITY);
  const int nw = MODE == 0 ? 0 : rw.hi - rw.lo;
  const int n = nw + (MODE == 1 ? 0 : rd.hi - rd.lo);
  // item `local`, whose accumulator's barrier is in its phase `turn`
  auto wait = [&](uint32_t local, uint64_t* full, uint32_t turn) {
    const uint32_t ms = local % MS;
    const bool ok = dead || (mbar_wait(&sh.mfull[ms], (local / MS) & 1u) && mbar_wait(full, turn & 1u));
    if (__any_sync(0xffffffffu, !ok)) {
      if (lane == 0 && !dead) atomicOr(s.status, ST_TIMEOUT);
      dead = true;
    }
    if (!dead) tc_fence_after();
  };
  uint32_t local = 0;
  if constexpr (MODE != 0) {
    const Place<WPASS_TNV> pl(warp, lane, all_w);
    uint32_t turn = 0;                           // window items this team has taken
    for (; (int)local < nw; ++local) {
      if (!pl.mine(local)) continue;
      wait(local, &sh.wfull[local % WG::NACC], local / WG::NACC);
      window_item<KIND, TNV>(s, sh, tmem, pl, local, turn++, rw.lo + (int)local, norms, dead);
    }
  }
  if constexpr (MODE != 1) {
    const Place<TNV> pl(warp, lane, all_d);
    for (; (int)local < n; ++local) {
      const uint32_t l = local - (uint32_t)nw, buf = l % NACC;
      if (!pl.mine(l)) continue;
      wait(local, &sh.tfull[buf], l / NACC);
      const int item = rd.lo + (int)l;
      dist_item<KIND, TNV, PAIR>(s, sh, tmem, pl, local, buf, item % T,
                                 (PAIR ? 2 * (item / T) + rank : item / T) * TM, rows, dead);
    }
  }
}

// The norm warp (a launch with norms): reports every finished window item of
// this CTA (items lo, lo + 1, ..). The item's sums were written by the epilogue
// before its arrival on nfull.
template <int TNV>
__device__ __forceinline__ void norm_warp(const Dev& s, Shared<TNV>& sh, int lo, int nw, int lane) {
  NormReports reports(lo + nw);
  for (uint32_t i = 0; (int)i < nw; ++i) {
    const uint32_t ns = i % NSLOT;
    reports.next(s, lo + (int)i);                // its reads overlap the wait
    const bool ok = mbar_wait(&sh.nfull[ns], (i / NSLOT) & 1u);
    if (__any_sync(0xffffffffu, !ok)) {
      if (lane == 0) atomicOr(s.status, ST_TIMEOUT);
      return;
    }
    const int j = sh.nj[ns];
    __syncwarp();
    if (lane == 0) mbar_arrive(&sh.nempty[ns]);
    reports.done(s, j >= 0);
  }
}

// A window-pass item from the pair list: the first rows of its A and B tiles
// (global support rows, both 4-aligned) and its ranges. Row and column tiles
// start at the range starts rounded down to a multiple of 4 rows; rows and
// columns outside the ranges are masked by position.
__device__ __forceinline__ void pair_item(const Dev& s, int w, int& ya, int& yb, ItemDesc& d) {
  const WPair pr = s.wpairs[w];
  const Plan P = s.plan[pr.j];
  int r0, r1, c0;
  if (pr.kind == 0) { r0 = P.head_c; r1 = P.head_c + P.ndrop; c0 = P.head_c; }
  else { r0 = P.tail_c; r1 = P.tail_new; c0 = P.tail_c; }
  const int ra = (r0 & ~3) + pr.rt * TM;
  const int ca = (c0 & ~3) + pr.ct * WPASS_TNV;
  const int base = pr.j * s.cap;
  ya = base + ra;
  yb = base + ca;
  d.kind = pr.kind;
  d.rlo = r0 - ra;
  d.rhi = r1 - ra;
  d.dnew = P.head_new - ca;
  d.told = P.tail_c - ca;
  d.tnew = P.tail_new - ca;
  d.j = pr.j;
  d.pad0 = 0;
}

// This CTA's items: a contiguous range of the launch's items, in row-tile-
// major order (distance pass: item = row tile * tiles + support tile; window
// pass: the pair list's order, row tiles outer within each center), so that
// consecutive items mostly share their A tile.
__device__ __forceinline__ Range my_range(int total, int cta, int ncta) {
  Range r;
  r.lo = (int)((int64_t)cta * total / ncta);
  r.hi = (int)((int64_t)(cta + 1) * total / ncta);
  return r;
}

// MODE 0: distance pass (A = batch tile, B = support tile, one FP32 partial per row).
// MODE 1: window pass (A and B = support rows of one center, four FP64 sums per item).
// MODE 2: both, every CTA's share of the previous step's window items first. An
//         evenly split batch has a few hundred of a few dozen rows each, which
//         by themselves leave the chip waiting on their latency; as one or two
//         more items per CTA they cost their work. With the window pass and the
//         weight update as launches of their own 16 iterations and a scoring call
//         took 1307 us on evenly split batches of 1e6 x 128 (k = 100, b = 4096)
//         and 468 us at 2000 x 16 (b = 256), now 1266 and 407.
// norms (MODE 1, 2): the norm warp carries ||C_j||^2 once a center's items are done.
//
// Both passes only sum over columns, so a tile can be split along its columns
// with no merge. Columns past a tile's width are neither multiplied (the MMA's
// N is the width rounded up to 16) nor read back.
//
// Metadata: distance-pass tiles start on a multiple of 4 support rows and
// support weights are 0 outside the windows, so an item's column metadata
// (||y||^2, w, data index) and row metadata (||x||^2, data index) are plain
// contiguous, 16-byte aligned ranges; window-pass tiles start 4-aligned by
// construction. The metadata warp copies them into a ring of slots next to
// the operands, so nothing on the epilogue's path waits on a global load.
// Item descriptors are fetched 32 at a time, one per lane.
template <int KIND, int MODE, int OP, int TNV, bool PAIR = false>
__device__ __forceinline__ void dist_tc_body(const Dev& s, int rows, const CUtensorMap* tmA, const CUtensorMap* tmB,
                                             const CUtensorMap* tmW, const CUtensorMap* tmN, int cta, int ncta,
                                             bool norms = false,
                                             Range ovr = Range{-1, -1}, int flags = TC_ALLOC | TC_FREE) {
  static_assert(!PAIR || (MODE == 0 && TNV >= 128), "CTA pairs take distance items of 128 or 256 columns");
  constexpr bool X3 = OP == OP_X3;
  constexpr int KSE = OP == OP_TF32 ? 32 : KS;   // operand elements per slice row
  constexpr int NACC = Geo<TNV>::NACC, MS = Geo<TNV>::MS;
  const int rank = PAIR ? cta & 1 : 0;           // the CTA's place in its pair
  // one B slice: the rows its live columns need (a box of 64, 128 or TNV rows) x 128 bytes
  auto slice_bytes = [](uint32_t ncol) {
    return (TNV > 64 && ncol > 64u ? (TNV > 128 && ncol > 128u ? TNV : 128) : 64) * KS * 2;
  };
  // the MMA's N: an item's live columns, whole 16s
  auto live_cols = [](bool win, int wd) {
    const int most = win ? WPASS_TNV : TNV;
    return (uint32_t)(wd <= 0 ? 16 : wd >= most ? most : (wd + 15) & ~15);
  };
  // a pair's N: whole 32s, half of the columns from each CTA's B rows
  constexpr int GRP = PAIR && TNV == 128 ? 2 : 1;   // items that share a pass over their row tile
  constexpr int HB = TNV / 2 * KS * 2;              // bytes of half a tile's B slice
  auto pair_cols = [](int wd) { return (uint32_t)(wd <= 0 ? 32 : wd >= TNV ? TNV : (wd + 31) & ~31); };
  constexpr int AH = X3 ? 2 : 1;                 // hi (and lo) tiles per operand
  static_assert(MODE == 0 || TNV >= WPASS_TNV, "a stage holds a window item's B tile");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  Shared<TNV>& sh = *reinterpret_cast<Shared<TNV>*>(smem + RING_BYTES);
  constexpr uint32_t TMEM_COLS = Geo<TNV>::TMEM_COLS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nks = s.dp / KSE;
  const Layout L = PAIR ? pair_layout<X3>(nks) : layout<X3, TNV>(nks);
  uint8_t* const ring = smem + L.a_bytes;        // stages (resident A sits below them)

  if (threadIdx.x == 0) {
    if (flags & TC_REINIT) {
      // a later segment of a group CTA: every barrier initialised below is
      // quiescent (the previous segment ended on a CTA barrier after all its
      // waits), so it is invalidated before it is initialised again
      for (int i = 0; i < STAGES; ++i) {
        mbar_inval(&sh.full[i]);
        mbar_inval(&sh.empty[i]);
      }
      mbar_inval(&sh.afull);
      mbar_inval(&sh.afree);
      for (int i = 0; i < NACC; ++i) {
        mbar_inval(&sh.tfull[i]);
        mbar_inval(&sh.tempty[i]);
      }
      for (int i = 0; i < MS; ++i) {
        mbar_inval(&sh.mfull[i]);
        mbar_inval(&sh.mempty[i]);
      }
      for (int i = 0; i < NSLOT; ++i) {
        mbar_inval(&sh.nfull[i]);
        mbar_inval(&sh.nempty[i]);
      }
      for (int i = 0; i < WG::NACC && MODE != 0; ++i) {
        mbar_inval(&sh.wfull[i]);
        mbar_inval(&sh.wempty[i]);
      }
      mbar_inval(&sh.mma_done);
    }
    // every stage's pair, not only the layout's L.nst: a later segment may use more
    for (int i = 0; i < STAGES; ++i) {
      mbar_init(&sh.full[i], 1);
      mbar_init(&sh.empty[i], 1);
    }
    mbar_init(&sh.afull, 1);
    mbar_init(&sh.afree, 1);
    for (int i = 0; i < NACC; ++i) {
      mbar_init(&sh.tfull[i], 1);
      mbar_init(&sh.tempty[i], (PAIR ? 2 : 1) * 4 * Geo<TNV>::GPT);   // the warps of one team (of both CTAs)
    }
    for (int i = 0; i < WG::NACC && MODE != 0; ++i) {
      mbar_init(&sh.wfull[i], 1);
      mbar_init(&sh.wempty[i], 4);               // the warps of one group
    }
    for (int i = 0; i < MS; ++i) {
      mbar_init(&sh.mfull[i], META_ARRIVALS);
      mbar_init(&sh.mempty[i], 4 * Geo<TNV>::GPT);
    }
    for (int i = 0; i < NSLOT; ++i) {
      mbar_init(&sh.nfull[i], 1);
      mbar_init(&sh.nempty[i], 1);
    }
    mbar_init(&sh.mma_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1 && (flags & TC_ALLOC)) {
    if constexpr (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(&sh.tmem_base)), "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(&sh.tmem_base)), "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  if constexpr (PAIR) {
    __syncwarp();
    pair_sync();                                 // the peer's barriers are initialised too
  } else {
    __syncthreads();
  }
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;
  const int R = (rows + TM - 1) / TM;

  // Streaming stage for slice sl: A_hi, A_lo (split form), B_hi, B_lo.
  auto stream_issue = [&](bool lead, uint8_t* st, uint64_t* bar, int sl, const CUtensorMap* ta, int ya,
                          const CUtensorMap* tb, int yb, int bt) {
    const int x = sl * KSE;
    tma_load_2d(lead, st, ta, bar, x, ya);
    if (X3) tma_load_2d(lead, st + A_BYTES, ta, bar, s.dp + x, ya);
    tma_load_2d(lead, st + AH * A_BYTES, tb, bar, x, yb);
    if (X3) tma_load_2d(lead, st + AH * A_BYTES + bt, tb, bar, s.dp + x, yb);
  };

  // Metadata of one item, 16 bytes per lane and copy: the column arrays
  // (||y||^2, w, data index of the B rows; the second 128 of them only where
  // the item has that many) and the row arrays (distance item ||x||^2, data
  // index; window item ||y||^2, data index, w). Window items read the weights
  // before the update (wwin). Straight-line on purpose: as a loop that worked out
  // each chunk's array by division this took one warp about as long as an
  // item's arithmetic takes the epilogue.
  auto meta_copy = [&](MetaSlot<TNV>& m, int ya, int yb, int ncol, bool win) {
    const float *c0 = s.yn + yb, *c1 = (win ? s.wwin : s.w32) + yb, *c2 = (const float*)s.yi + yb;
    const float *r0 = (win ? s.yn : s.xbn) + ya, *r1 = (const float*)(win ? s.yi : s.xbi) + ya;
    const int o = 4 * lane;
    if (TNV >= 128 || lane < TNV / 4) {
      cp16(m.col[0] + o, c0 + o);
      cp16(m.col[1] + o, c1 + o);
      cp16(m.col[2] + o, c2 + o);
    }
    if (TNV > 128 && ncol > 128) {
      cp16(m.col[0] + (TNV - 128) + o, c0 + 128 + o);
      cp16(m.col[1] + (TNV - 128) + o, c1 + 128 + o);
      cp16(m.col[2] + (TNV - 128) + o, c2 + 128 + o);
    }
    cp16(m.row[0] + o, r0 + o);
    cp16(m.row[1] + o, r1 + o);
    if (MODE != 0 && win) cp16(m.row[2] + o, s.wwin + ya + o);
  };
  static_assert(TNV == 64 || TNV == 128 || TNV == 256, "meta_copy covers these tiles");

  // The CTA's items: window items, then distance items. With s.pre_b (set per
  // launch when the kernel just ahead writes neither the tile and pair lists
  // nor the plans: the batch gather, the row moves or this pass itself) the
  // lists are read, and the descriptors of the first 32 items fetched, one per
  // lane, before the grid-dependency wait.
  int T = 1, total = 0, np = 0;                  // support tiles, distance items, window items
  Range rw{0, 0}, rd{0, 0};
  auto ranges = [&]() {
    if constexpr (MODE != 0) np = *s.nwpairs;
    if constexpr (MODE != 1) {
      T = *s.ntiles;
      total = R * T;
    }
    if (ovr.lo >= 0) {
      (MODE == 1 ? rw : rd) = ovr;
    } else if (MODE == 2 && np > 0 && ncta == s.nsplit) {
      const int2 lo = s.split[cta], hi = s.split[cta + 1];   // by work (the sort/plan)
      rw = Range{lo.x, hi.x};
      rd = Range{lo.y, hi.y};
    } else if (PAIR) {                           // pairs of row tiles; both CTAs walk the same items
      rd = my_range((R + 1) / 2 * T, cta >> 1, ncta >> 1);
    } else {
      rw = my_range(np, cta, ncta);
      rd = my_range(R * T, cta, ncta);
    }
  };
  int pya = 0, pyb = 0;                          // this lane's prefetched item: A and B rows
  ItemDesc pd{};
  // descriptors of items local .. local + 31, one per lane; a distance item's
  // width goes in tnew
  auto fetch_desc = [&](int local) {
    const int nw = rw.hi - rw.lo, mine = local + lane;
    if (MODE != 0 && mine < nw) {
      pair_item(s, rw.lo + mine, pya, pyb, pd);
    } else if (MODE != 1 && rd.lo + mine - nw < rd.hi) {
      const int item = rd.lo + mine - nw;
      const Tile t = s.tiles[item % T];
      pya = (PAIR ? 2 * (item / T) + rank : item / T) * TM;
      pyb = t.row0;
      pd.tnew = t.ncols;
    }
  };
  const bool desc_pre = s.pre_b != 0;
  if (desc_pre) {
    ranges();
    if (warp <= 1 || warp == MWARP) fetch_desc(0);
    if (warp == 0 && lane < 4)   // the first copy does not wait for its descriptor
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)(lane == 0 ? tmA : lane == 1 ? tmB : lane == 2 ? tmW : tmN))
                   : "memory");
  }
  KKM_GRID_DEP_WAIT();       // everything above reads only data of earlier steps
  KKM_LAUNCH_DEPENDENTS();   // the next kernel may set itself up; it waits before reading our output
  if (!desc_pre) ranges();
  const int nw = rw.hi - rw.lo, n = nw + rd.hi - rd.lo;
  // All epilogue groups on each item (instead of a team per item) when the run
  // has fewer than NTEAM distance items, or fewer than one window item, per SM.
  // The choice depends on the run alone, never on how a launch splits its items,
  // so an item's sums come out the same in a run's own launch and in a run
  // group's. (Window items on all groups up to NTEAM per SM: single steps with
  // half of 1024 rows in one of 100 centers 53.7 and 51.5 us; never: 2000 x 16,
  // b = 256, 34.0 and 34.9.)
  const bool all_d = total < Geo<TNV>::NTEAM * s.num_sms, all_w = np < s.num_sms;

  if (warp == 0) {
    // ------------------------------------------------- operand producer (one warp)
    const bool lead = lane == 0;
    bool ok = true;
    uint32_t it = 0, na = 0;                     // stage fills, A tiles
    int cur_ya = -1;                             // the resident A tile's first row (window items: support rows)
    bool cur_win = false;
    for (int local = 0; local < n && ok; ++local) {
      if ((local & 31) == 0 && !(local == 0 && desc_pre)) fetch_desc(local);
      const int src = local & 31;
      const int ya = __shfl_sync(0xffffffffu, pya, src);
      const int yb = __shfl_sync(0xffffffffu, pyb, src);
      const int wd = __shfl_sync(0xffffffffu, pd.tnew, src);
      const bool win = MODE != 0 && local < nw;
      const uint32_t ncol = live_cols(win, wd);
      const CUtensorMap* ta = win ? tmW : tmA;
      const CUtensorMap* tb = TNV == 64 || ncol <= 64u ? tmN : TNV > 128 && ncol > 128u ? tmB : tmW;
      const int bt = slice_bytes(ncol);
      const bool new_a = L.res && (ya != cur_ya || win != cur_win);
      if (L.res) {
        // one stage: the item's whole B tile
        const int st = it % L.nst;
        ok = warp_wait(&sh.empty[st], ((it / L.nst) & 1u) ^ 1u);
        if (!ok) break;
        if (lead) sh.mark[st] = new_a ? 1u : 0u;   // published by the arrive below
        mbar_expect_tx(lead, &sh.full[st], (uint32_t)(L.nsl * bt));
        tile_issue(lead, L.nsl, nks, s.dp, KSE, ring + st * L.sb, bt, tb, &sh.full[st], yb);
        ++it;
        if (new_a) {
          // the item's B tile is queued (the MMA warp sees the new-A mark on it
          // and releases the old A tile); then the new A tile
          ok = na == 0 || warp_wait(&sh.afree, (na - 1) & 1u);
          if (!ok) break;
          mbar_expect_tx(lead, &sh.afull, (uint32_t)L.a_bytes);
          tile_issue(lead, L.nsl, nks, s.dp, KSE, smem, A_BYTES, ta, &sh.afull, ya);
          ++na;
          cur_ya = ya;
          cur_win = win;
        }
      } else if constexpr (PAIR) {
        // this CTA's A rows (past the last row tile: zeros) and its half of the
        // MMA's B rows, for one or two items; the even CTA's barrier counts the
        // bytes of both CTAs
        const bool two = GRP == 2 && local + 1 < n && src < 31 && __shfl_sync(0xffffffffu, pya, (src + 1) & 31) == ya;
        const int half = (int)pair_cols(wd) / 2;
        const CUtensorMap* th = half <= 64 ? tmN : tmW;
        const int hb = (half <= 64 ? 64 : 128) * KS * 2, yh = yb + rank * half;
        const int yh2 = __shfl_sync(0xffffffffu, pyb, (src + 1) & 31) +
                        rank * ((int)pair_cols(__shfl_sync(0xffffffffu, pd.tnew, (src + 1) & 31)) / 2);
        for (int sl = 0; sl < nks; ++sl, ++it) {
          const int st = it % L.nst, x = sl * KSE;
          ok = warp_wait(&sh.empty[st], ((it / L.nst) & 1u) ^ 1u);
          if (!ok) break;
          if (rank == 0)
            mbar_expect_tx(lead, &sh.full[st], (uint32_t)(2 * AH * (A_BYTES + (two ? 2 * hb : hb))));
          const uint32_t bar = lead_addr(&sh.full[st]);
          uint8_t *sp = ring + st * L.sb, *sb = sp + AH * A_BYTES;
          tma_load_2d_pair(lead, sp, ta, bar, x, ya);
          if (X3) tma_load_2d_pair(lead, sp + A_BYTES, ta, bar, s.dp + x, ya);
          tma_load_2d_pair(lead, sb, th, bar, x, yh);
          if (X3) tma_load_2d_pair(lead, sb + HB, th, bar, s.dp + x, yh);
          if (two) {
            tma_load_2d_pair(lead, sb + AH * HB, th, bar, x, yh2);
            if (X3) tma_load_2d_pair(lead, sb + (AH + 1) * HB, th, bar, s.dp + x, yh2);
          }
        }
        if (two) ++local;
      } else {
        for (int sl = 0; sl < nks; ++sl, ++it) {
          const int st = it % L.nst;
          ok = warp_wait(&sh.empty[st], ((it / L.nst) & 1u) ^ 1u);
          if (!ok) break;
          mbar_expect_tx(lead, &sh.full[st], (uint32_t)(AH * (A_BYTES + bt)));
          stream_issue(lead, ring + st * L.sb, &sh.full[st], sl, ta, ya, tb, yb, bt);
        }
      }
    }
    // the copies in flight must land before the CTA may exit: the last fill
    // of every stage and the last A tile. A pair's copies count at the even CTA,
    // and both CTAs meet before they exit; the odd one waits for the last
    // arrivals that the even CTA's commits send it.
    for (uint32_t q = (it > (uint32_t)L.nst ? it - L.nst : 0u); q < it && (ok || !PAIR); ++q)
      if (!warp_wait(rank == 0 ? &sh.full[q % L.nst] : &sh.empty[q % L.nst], (q / L.nst) & 1u)) ok = false;
    if (na > 0 && !warp_wait(&sh.afull, (na - 1) & 1u)) ok = false;
    if (lead && !ok) atomicOr(s.status, ST_TIMEOUT);
  } else if (warp == MWARP) {
    // ------------------------------------------------------ metadata (one warp)
    // Every lane copies its share of an item's metadata and arrives on the
    // slot's barrier once its copies have landed; lane 0 also arrives after
    // writing the item's ranges, which publishes them.
    bool ok = true;
    for (int local = 0; local < n; ++local) {
      if ((local & 31) == 0 && !(local == 0 && desc_pre)) fetch_desc(local);
      const int src = local & 31;
      const int ya = __shfl_sync(0xffffffffu, pya, src);
      const int yb = __shfl_sync(0xffffffffu, pyb, src);
      const bool win = MODE != 0 && local < nw;
      const int ms = local % MS;
      if (lane == 0 && !mbar_wait(&sh.mempty[ms], (((uint32_t)local / MS) & 1u) ^ 1u)) ok = false;
      if (!__shfl_sync(0xffffffffu, (int)ok, 0)) break;
      MetaSlot<TNV>& m = sh.ring[ms];
      ItemDesc d{};
      d.tnew = __shfl_sync(0xffffffffu, pd.tnew, src);
      if constexpr (MODE != 0) {
        d.kind = __shfl_sync(0xffffffffu, pd.kind, src);
        d.rlo = __shfl_sync(0xffffffffu, pd.rlo, src);
        d.rhi = __shfl_sync(0xffffffffu, pd.rhi, src);
        d.dnew = __shfl_sync(0xffffffffu, pd.dnew, src);
        d.told = __shfl_sync(0xffffffffu, pd.told, src);
        d.j = __shfl_sync(0xffffffffu, pd.j, src);
      }
      if (lane == 0) m.desc = d;
      // the last pair's second row tile may lie past the batch: nothing of it is written
      meta_copy(m, PAIR ? min(ya, (R - 1) * TM) : ya, yb, d.tnew, win);
      cp_arrive_noinc(&sh.mfull[ms]);
      if (lane == 0) mbar_arrive(&sh.mfull[ms]);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");   // nothing in flight when the CTA exits
    if (lane == 0 && !ok) atomicOr(s.status, ST_TIMEOUT);
  } else if (warp == 1) {
    // ---------------------------------------------------- MMA issuer (one warp)
    const bool lead = lane == 0;
    bool ok = true;
    uint32_t it = 0, na = 0;
    const uint32_t abase = smem_u32(smem), rbase = smem_u32(ring);
    // the four K steps of a slice
    auto mma_slice = [&](uint32_t d, uint32_t id, uint32_t ahi, uint32_t alo, uint32_t bhi, uint32_t blo,
                         bool first) {
      const uint32_t ah = desc_lo(ahi), bh = desc_lo(bhi), al = desc_lo(alo), bl = desc_lo(blo);
#pragma unroll
      for (uint32_t k = 0; k < 4; ++k) {
        mma_op<OP, PAIR>(lead, d, ah + 2u * k, bh + 2u * k, id, (first && k == 0) ? 0u : 1u);
        if constexpr (X3) {
          mma_op<OP, PAIR>(lead, d, ah + 2u * k, bl + 2u * k, id, 1u);
          mma_op<OP, PAIR>(lead, d, al + 2u * k, bh + 2u * k, id, 1u);
        }
      }
    };
    if constexpr (PAIR) {
      for (int local = 0; local < n && ok && rank == 0; ++local) {
        if ((local & 31) == 0 && !(local == 0 && desc_pre)) fetch_desc(local);
        const int src = local & 31, nx = (src + 1) & 31;
        const bool two = GRP == 2 && local + 1 < n && src < 31 &&
                         __shfl_sync(0xffffffffu, pya, nx) == __shfl_sync(0xffffffffu, pya, src);
        const uint32_t id = idesc<OP>(pair_cols(__shfl_sync(0xffffffffu, pd.tnew, src)), 2 * TM);
        const uint32_t id2 = idesc<OP>(pair_cols(__shfl_sync(0xffffffffu, pd.tnew, nx)), 2 * TM);
        const uint32_t buf = local % NACC, buf2 = (local + 1) % NACC;
        ok = warp_wait(&sh.tempty[buf], (((uint32_t)local / NACC) & 1u) ^ 1u) &&
             (!two || warp_wait(&sh.tempty[buf2], (((uint32_t)(local + 1) / NACC) & 1u) ^ 1u));
        if (!ok) break;
        asm volatile("fence.acq_rel.cluster;" ::: "memory");   // the peer's releases
        tc_fence_after();
        for (int sl = 0; sl < nks; ++sl, ++it) {
          const int st = it % L.nst;
          ok = warp_wait(&sh.full[st], (it / L.nst) & 1u);
          if (!ok) break;
          tc_fence_after();
          const uint32_t a0 = rbase + (uint32_t)(st * L.sb), b0 = a0 + AH * A_BYTES;
          mma_slice(tmem + buf * TNV, id, a0, a0 + A_BYTES, b0, b0 + HB, sl == 0);
          if (two) mma_slice(tmem + buf2 * TNV, id2, a0, a0 + A_BYTES, b0 + AH * HB, b0 + (AH + 1) * HB, sl == 0);
          mma_commit_pair(lead, &sh.empty[st]);
        }
        if (!ok) break;
        mma_commit_pair(lead, &sh.tfull[buf]);
        if (two) {
          mma_commit_pair(lead, &sh.tfull[buf2]);
          ++local;
        }
      }
    }
    for (int local = 0; local < n && ok && !PAIR; ++local) {
      if ((local & 31) == 0 && !(local == 0 && desc_pre)) fetch_desc(local);
      const int wd = __shfl_sync(0xffffffffu, pd.tnew, local & 31);
      const bool win = MODE != 0 && local < nw;
      const uint32_t ncol = live_cols(win, wd);
      const uint32_t id = idesc<OP>(ncol);
      const int bt = slice_bytes(ncol);
      const uint32_t l = win ? local : local - nw, nacc = win ? WG::NACC : NACC, buf = l % nacc;
      uint64_t* const full = win ? &sh.wfull[buf] : &sh.tfull[buf];
      const uint32_t d = tmem + buf * (win ? WPASS_TNV : TNV);
      // the window items whose accumulators this one's first use covers
      if (MODE == 2 && !win && l < (uint32_t)NACC)
        for (int wb = (int)buf * (TNV / WPASS_TNV); wb < (int)(buf + 1) * (TNV / WPASS_TNV) && ok; ++wb) {
          const int uses = nw > wb ? (nw - wb + WG::NACC - 1) / WG::NACC : 0;
          if (uses > 0) ok = warp_wait(&sh.wempty[wb], (uint32_t)(uses - 1) & 1u);
        }
      if (!ok) break;
      ok = warp_wait(win ? &sh.wempty[buf] : &sh.tempty[buf], ((l / nacc) & 1u) ^ 1u);
      if (!ok) break;
      tc_fence_after();
      if (L.res) {
        const int st = it % L.nst;
        ok = warp_wait(&sh.full[st], (it / L.nst) & 1u);
        if (!ok) break;
        tc_fence_after();
        if (__any_sync(0xffffffffu, sh.mark[st])) {
          // a new resident A tile: release the old one once its MMAs are done, wait for the new one
          if (na > 0) mma_commit(lead, &sh.afree);
          ok = warp_wait(&sh.afull, na & 1u);
          if (!ok) break;
          tc_fence_after();
          ++na;
        }
        const uint32_t b0 = rbase + (uint32_t)(st * L.sb);
        for (int sl = 0; sl < nks; ++sl)
          mma_slice(d, id, abase + sl * A_BYTES, abase + (nks + sl) * A_BYTES, b0 + sl * bt, b0 + (nks + sl) * bt,
                    sl == 0);
        mma_commit(lead, &sh.empty[st]);
        ++it;
      } else {
        for (int sl = 0; sl < nks; ++sl, ++it) {
          const int st = it % L.nst;
          ok = warp_wait(&sh.full[st], (it / L.nst) & 1u);
          if (!ok) break;
          tc_fence_after();
          const uint32_t a0 = rbase + (uint32_t)(st * L.sb), b0 = a0 + AH * A_BYTES;
          mma_slice(d, id, a0, a0 + A_BYTES, b0, b0 + bt, sl == 0);
          mma_commit(lead, &sh.empty[st]);
        }
        if (!ok) break;
      }
      mma_commit(lead, full);
    }
    if (rank == 0) {                             // a pair's MMAs are all the even CTA's
      mma_commit<PAIR>(lead, &sh.mma_done);
      if (!warp_wait(&sh.mma_done, 0)) ok = false;
    }
    if (lead && !ok) atomicOr(s.status, ST_TIMEOUT);
  } else if (warp < MWARP) {
    epilogue<KIND, MODE, TNV, PAIR>(s, sh, tmem, rw, rd, T, rows, warp, lane, all_w, all_d, norms, rank);
  } else if constexpr (MODE != 0) {
    if (norms) norm_warp<TNV>(s, sh, rw.lo, nw, lane);
  }
  tc_fence_before();
  if constexpr (PAIR) {
    __syncwarp();
    pair_sync();                                 // every copy, MMA, arrival and read of both CTAs is done
    if (warp == 1) {
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
    return;
  }
  __syncthreads();
  if (warp == 1 && (flags & TC_FREE)) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS)
                 : "memory");
  }
}

template <int KIND, int MODE, int OP, int TNV>
__global__ void __launch_bounds__(nthreads<MODE>(), 1)
    k_dist_tc(Dev s, int rows, int norms, const __grid_constant__ CUtensorMap tmA,
              const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmW,
              const __grid_constant__ CUtensorMap tmN) {
  dist_tc_body<KIND, MODE, OP, TNV>(s, rows, &tmA, &tmB, &tmW, &tmN, blockIdx.x, gridDim.x, norms != 0);
}

template <int KIND, int MODE, int OP, int TNV>
cudaError_t launch_form(const Dev& s, const CUtensorMap* m, int rows, bool norms, cudaStream_t st) {
  static std::atomic<uint64_t> attr{0};
  {
    const cudaError_t e = smem_limit_once(k_dist_tc<KIND, MODE, OP, TNV>, smem_bytes<TNV>(), attr);
    if (e != cudaSuccess) return e;
  }
  // one CTA per SM, but never more CTAs than the most items this launch can
  // have: small runs then leave SMs free for the kernels of other runs
  const int64_t most = (MODE != 1 ? (int64_t)((rows + TM - 1) / TM) * s.max_tiles : 0) +
                       (MODE != 0 ? (int64_t)s.max_pairs : 0);
  const int grid = MODE == 2 ? s.nsplit : (int)(most < s.num_sms ? (most > 0 ? most : 1) : s.num_sms);
  // maps: [0] batch rows, 128-row boxes; support rows with [1] 128-row, [2] 64-row, [3] 256-row boxes
  return launch_pdl(k_dist_tc<KIND, MODE, OP, TNV>, dim3(grid), dim3(nthreads<MODE>()), smem_bytes<TNV>(), st, s,
                    rows, norms ? 1 : 0, m[0], m[3], m[1], m[2]);
}

// The distance pass on CTA pairs.
template <int KIND, int OP, int TNV>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(nthreads<0>(), 1)
    k_dist_pair(Dev s, int rows, const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmN) {
  dist_tc_body<KIND, 0, OP, TNV, true>(s, rows, &tmA, &tmB, &tmW, &tmN, blockIdx.x, gridDim.x);
}

template <int KIND, int OP, int TNV>
cudaError_t launch_pair_form(const Dev& s, const CUtensorMap* m, int rows, cudaStream_t st) {
  static std::atomic<uint64_t> attr{0};
  const cudaError_t e = smem_limit_once(k_dist_pair<KIND, OP, TNV>, smem_bytes<TNV>(), attr);
  if (e != cudaSuccess) return e;
  const int64_t most = (int64_t)((rows + 2 * TM - 1) / (2 * TM)) * s.max_tiles;
  const int pairs = (int)std::max<int64_t>(1, std::min<int64_t>(most, s.num_sms / 2));
  return launch_pdl(k_dist_pair<KIND, OP, TNV>, dim3(2 * pairs), dim3(nthreads<0>()), smem_bytes<TNV>(), st, s, rows,
                    m[0], m[3], m[1], m[2]);
}

template <int OP, int TNV>
cudaError_t launch_pair_kind(const Dev& s, const CUtensorMap* m, int rows, cudaStream_t st) {
  switch (s.kind) {
    case K_GAUSS: return launch_pair_form<K_GAUSS, OP, TNV>(s, m, rows, st);
    case K_LAPLACE: return launch_pair_form<K_LAPLACE, OP, TNV>(s, m, rows, st);
    case K_LINEAR: return launch_pair_form<K_LINEAR, OP, TNV>(s, m, rows, st);
    default: return launch_pair_form<K_POLY, OP, TNV>(s, m, rows, st);
  }
}

template <int MODE, int OP, int TNV>
cudaError_t launch_kind(const Dev& s, const CUtensorMap* m, int rows, bool norms, cudaStream_t st) {
  switch (s.kind) {
    case K_GAUSS: return launch_form<K_GAUSS, MODE, OP, TNV>(s, m, rows, norms, st);
    case K_LAPLACE: return launch_form<K_LAPLACE, MODE, OP, TNV>(s, m, rows, norms, st);
    case K_LINEAR: return launch_form<K_LINEAR, MODE, OP, TNV>(s, m, rows, norms, st);
    default: return launch_form<K_POLY, MODE, OP, TNV>(s, m, rows, norms, st);
  }
}

template <int MODE, int TNV>
cudaError_t launch_mode(const Dev& s, const void* maps, int rows, bool norms, cudaStream_t st) {
  const CUtensorMap* m = static_cast<const CUtensorMap*>(maps);
  switch (s.form) {
    case FORM_BF16X3: return launch_kind<MODE, OP_X3, TNV>(s, m, rows, norms, st);
    case FORM_TF32: return launch_kind<MODE, OP_TF32, TNV>(s, m, rows, norms, st);
    default: return launch_kind<MODE, OP_BF16, TNV>(s, m, rows, norms, st);
  }
}

// Run groups. A launch covers the runs of one class (same form, kernel kind
// and tile width; their d may differ). Each run's items (distance pass:
// row tiles x support tiles; window pass: its pair list) are laid end to end
// in one weighted item space, an item of run r weighing
// max(5, 2 nks_r m_r) (m = 3 for the split form: the MMA share next to the
// epilogue's fixed share). Where the shares allow it each CTA belongs to one run
// (group_whole_ctas); otherwise CTA c takes the items whose start falls in
// [c W / G, (c + 1) W / G) and walks its range run by run: each stretch of
// one run's items is a segment, run with that run's Dev and TMA descriptors
// (read from device memory; the host wrote them before the group's first
// launch, and the acquire fence orders that write before the tensor-map
// proxy's reads). TMEM is allocated for the first segment and freed after the
// last; the barriers are invalidated and initialised again between segments.
// Item counts are read after the grid-dependency wait, so no data of this
// step is staged before it (the runs' copies carry pre_b = 0).
template <int MODE>
__device__ __forceinline__ int group_items(const Dev& s) {
  return MODE == 0 ? ((s.b + TM - 1) / TM) * (*s.ntiles) : *s.nwpairs;
}

__device__ __forceinline__ int group_weight(const Dev& s) {
  const int kse = s.form == FORM_TF32 ? 32 : KS;
  const int m = s.form == FORM_BF16X3 ? 3 : 1;
  const int w = 2 * (s.dp / kse) * m;
  return w > 5 ? w : 5;
}

__device__ __forceinline__ long long ceil_div_ll(long long a, long long b) {
  return a >= 0 ? (a + b - 1) / b : -((-a) / b);
}

// Warp-wide: the first run r >= rnext whose items intersect the weighted
// range [A, B), with that intersection [lo, hi) of its items; -1 if none.
// With A = B = -1, returns -1 and sets lo to the low and hi to the high word
// of the total weight instead.
template <int MODE>
__device__ __forceinline__ int group_find(const GroupPhase& g, long long A, long long B, int rnext, int& lo,
                                          int& hi, long long& total) {
  const int lane = threadIdx.x & 31;
  long long carry = 0;
  for (int base = 0; base < g.nruns; base += 32) {
    const int r = base + lane;
    int n = 0, om = 1;
    if (r < g.nruns) {
      const Dev& s = g.runs[r].s;
      n = group_items<MODE>(s);
      om = group_weight(s);
    }
    const long long W = (long long)n * om;
    long long incl = W;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const long long P = carry + incl - W;
    int mlo = 0, mhi = 0;
    if (A >= 0 && r < g.nruns && r >= rnext && n > 0) {
      mlo = (int)min((long long)n, max(0LL, ceil_div_ll(A - P, om)));
      mhi = (int)min((long long)n, max(0LL, ceil_div_ll(B - P, om)));
    }
    const unsigned hit = __ballot_sync(0xffffffffu, mlo < mhi);
    if (hit) {
      const int src = __ffs(hit) - 1;
      lo = __shfl_sync(0xffffffffu, mlo, src);
      hi = __shfl_sync(0xffffffffu, mhi, src);
      return base + src;
    }
    carry += __shfl_sync(0xffffffffu, incl, 31);
  }
  total = carry;
  return -1;
}

// Whole CTAs per run (up to 32 runs, a lane each, warp-wide): the runs'
// boundaries in the weighted item space rounded to CTA boundaries, a run's
// items dealt evenly to its CTAs. A CTA then has one segment: filling and draining
// the pass's pipeline a second time costs as much as several items. Four steps of
// eight runs (k 5-100, d 16-256, b 256-2048): 740 -> 693 us.
// False, for the split by exact weight, where a run would get no CTA or
// the rounding would give some CTA over an eighth more than its share. r = -1: no items.
template <int MODE>
__device__ __forceinline__ bool group_whole_ctas(const GroupPhase& g, int cta, int ncta, int& r, int& lo, int& hi) {
  if (g.nruns > 32) return false;
  const int lane = threadIdx.x & 31;
  int n = 0, om = 1;
  if (lane < g.nruns) {
    const Dev& s = g.runs[lane].s;
    n = group_items<MODE>(s);
    om = group_weight(s);
  }
  const long long w = (long long)n * om;
  long long incl = w;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const long long W = __shfl_sync(0xffffffffu, incl, 31);
  r = -1;
  lo = hi = 0;
  if (W == 0) return true;
  const int c0 = (int)((2 * (incl - w) * ncta + W) / (2 * W)), c1 = (int)((2 * incl * ncta + W) / (2 * W));
  // w / (c1 - c0) <= (9 / 8) W / ncta
  const bool fits = n == 0 || (c1 > c0 && 8 * w * ncta <= 9 * W * (c1 - c0));
  if (!__all_sync(0xffffffffu, fits)) return false;
  const unsigned own = __ballot_sync(0xffffffffu, n > 0 && cta >= c0 && cta < c1);
  if (own) {
    r = __ffs(own) - 1;
    const int nr = __shfl_sync(0xffffffffu, n, r), a = __shfl_sync(0xffffffffu, c0, r),
              b = __shfl_sync(0xffffffffu, c1, r);
    lo = (int)((long long)nr * (cta - a) / (b - a));
    hi = (int)((long long)nr * (cta - a + 1) / (b - a));
    if (lo == hi) r = -1;
  }
  return true;
}

template <int KIND, int MODE, int OP, int TNV>
__global__ void __launch_bounds__(nthreads<MODE>(), 1) k_group_tc(GroupPhase g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  Shared<TNV>& sh = *reinterpret_cast<Shared<TNV>*>(smem + RING_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  KKM_GRID_DEP_WAIT();
  KKM_LAUNCH_DEPENDENTS();
  if (warp == 0) {
    int r = -1, lo = 0, hi = 0;
    long long total = 0;
    const bool whole = group_whole_ctas<MODE>(g, blockIdx.x, gridDim.x, r, lo, hi);
    if (lane == 0) {
      sh.gseg[0] = r;
      sh.gseg[1] = lo;
      sh.gseg[2] = hi;
      sh.gseg[3] = whole;
    }
    if (!whole) group_find<MODE>(g, -1, -1, 0, lo, hi, total);
    if (lane == 0) sh.gtot = total;
  }
  __syncthreads();
  const long long W = sh.gtot;
  const bool whole = sh.gseg[3] != 0;
  const long long A = W * (long long)blockIdx.x / gridDim.x, B = W * (long long)(blockIdx.x + 1) / gridDim.x;
  int flags = TC_ALLOC, rnext = 0;
  for (;;) {
    if (warp == 0 && !whole) {
      int lo = 0, hi = 0;
      long long total = 0;
      const int r = A < B ? group_find<MODE>(g, A, B, rnext, lo, hi, total) : -1;
      if (lane == 0) {
        sh.gseg[0] = r;
        sh.gseg[1] = lo;
        sh.gseg[2] = hi;
      }
    }
    __syncthreads();
    const int r = sh.gseg[0];
    if (r < 0) break;
    const Range seg{sh.gseg[1], sh.gseg[2]};
    const GroupRun& gr = g.runs[r];
    {
      // the run's Dev into shared memory (the previous segment ended on a CTA
      // barrier, so nobody reads the old copy any more)
      static_assert(sizeof(Dev) % 16 == 0, "Dev copied in 16-byte words");
      const int4* src = reinterpret_cast<const int4*>(&gr.s);
      int4* dst = reinterpret_cast<int4*>(&sh.gdev);
      for (int i = threadIdx.x; i < (int)(sizeof(Dev) / 16); i += nthreads<MODE>()) dst[i] = src[i];
    }
    __syncthreads();
    const CUtensorMap* m = reinterpret_cast<const CUtensorMap*>(gr.maps);
    if (warp == 0) {
      for (int i = 0; i < 4; ++i)
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"((uint64_t)&m[i]) : "memory");
    }
    // the body starts and ends on CTA barriers, so gseg is read by every
    // thread before warp 0 writes the next segment
    dist_tc_body<KIND, MODE, OP, TNV>(sh.gdev, sh.gdev.b, &m[0], &m[3], &m[1], &m[2], 0, 1, false, seg, flags);
    flags = TC_REINIT;
    if (whole) break;
    rnext = r + 1;
  }
  if (flags == TC_REINIT && warp == 1) {   // TMEM was allocated by the first segment
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sh.tmem_base),
                 "r"(Geo<TNV>::TMEM_COLS)
                 : "memory");
  }
}

}  // namespace
}  // namespace kkm
