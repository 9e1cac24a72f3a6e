// Packed-varlen prefill attention for sm_100a (Sections 2.1 and 3.2 of the prepacking paper):
//   o_i = sum_j softmax_j(q'_i . k'_j * scale) v_j   over keys j of the same prompt with j <= i.
// The independent mask M' (a lower-triangular block per prompt span) is never built: every query
// row carries the key range [start row of its prompt, its own row], and the host work list
// restricts each query tile to the key tiles that can intersect such a range.
//
// Persistent kernel, one CTA per SM, 640 threads (768 in the independent mode), two 128-row query-tile slots per CTA. CTAs draw
// work from a global counter (items are listed KV-head-major, longest first). Two modes, chosen on
// the host from the mean number of key tiles per query tile:
//
// Shared-stream mode (long items). A work item has two slots that share one stream of 128-row
// key/value tiles: two query heads of one KV head over the same rows (even GQA group), or two
// consecutive row tiles of one head.
//   warp 0       draws and decodes items, TMA-loads the K / V tile rings
//   warp 1       issues tcgen05.mma: S_t = Q_t K^T into TMEM, O_t += P_t V with P_t read from TMEM;
//                the two slots alternate so that one slot's MMAs run while the other's softmax works
//   warps 2-3    TMA-load Q of slot 0 / slot 1
//   warps 4-11   softmax and epilogue of slot 0: two threads per query row (TMEM lane = row), one per
//                64-key half of a tile; the row maximum is exchanged through shared memory
//   warps 12-19  the same for slot 1
// Independent mode (short items). Every slot draws its own items (one query tile each) and walks
// their 64-row key tiles on its own; S_t has two 64-column buffers so that the scores of tile k+1
// and the product P(k) V(k) are computed while the softmax threads work on tile k.
// With several query heads per KV head (GQA) the heads are folded into the rows of a query tile:
// 128 / f bin rows x f heads (tile row m = bin row m / f, head m % f; f = 2, 4 or 8 dividing the
// group), loaded and stored as one TMA box over (row, head). One stream of key tiles then serves
// the f heads, a short prompt fills a tile with heads instead of empty rows, and an item's key
// tiles start at the first row of the first prompt it touches rather than at a tile boundary.
//   warps 0-1    issue the tcgen05.mma of the scores of slot 0 / slot 1
//   warps 2-3    draw items and TMA-load Q (two tiles: the next item's is there early), K, V of slot 0 / slot 1
//   warps 4-7    softmax threads of slot 0, one per query row; they never leave the tile loop
//   warps 8-11   helper threads of slot 0, one per row: find the first key of each row of the next item,
//                rotate its Q in shared memory (fused path) and run the previous item's epilogue
//   warps 12-19  the same for slot 1
//   warps 20-21  (kFill) write the V rows of the slots' own query tiles from shared memory to the caches
//   warps 22-23  issue the tcgen05.mma of the products P V of slot 0 / slot 1
// Softmax: tcgen05.ld the thread's scores, mask to the row's key range, lazy running maximum (O is
// rescaled only when the maximum grows by more than 2^8, or 2^90 in the shared-stream mode, where rows
// whose scores are bounded drop the maximum altogether), exp2, P written as bf16 over the S
// columns. Epilogue: O / l goes through a swizzled staging buffer and a TMA store.
// TMEM: S0 | S1 | O0 | O1 = 512 columns. Every wait is an mbarrier wait with a time limit, also the
// rendezvous between warps (no named barriers), so a failed wait ends the kernel with a status code.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdlib>
#include <type_traits>

#include "pp_device_once.h"
#include "pp_internal.h"

namespace pp {
namespace {

constexpr int BM = kTileM;
constexpr int kAttnThreads = 640;
constexpr int kAttnThreadsIndep = 768;     // independent mode: one warpgroup more
constexpr int kSoftmaxThreads = 256;       // per slot: two threads per query row
constexpr uint32_t kTmemCols = 512;
constexpr int kRegsSoftmax = 104;          // setmaxnreg budgets, shared-stream mode: 640 threads start with 96 registers
constexpr int kRegsOther = 64;             //   each; warps 0-3 give back 32 each, the 512 softmax threads take 8 each
constexpr int kRegsSoftmaxIndep = 112;     // independent mode: 768 threads start with 80 each; the 256 softmax threads take
constexpr int kRegsOtherIndep = 56;        //   32 each from warps 0-3 (24 each) and 20-23 (40 each); the 256 helper
constexpr int kRegsLast = 40;              //   threads keep their 80
// Shared-stream mode, when a row needs no maximum any more. Its running maximum is lazy: it stays at the
// maximum of the row's first visible tile until a score exceeds it by more than kLazyLog2 (log2 units).
// Probabilities, sums and O have 8 exponent bits, so a common factor of up to 2^90 costs no precision, and
// it leaves 2^37 for the number of keys times |v|: that much room there must be (kValueRoomLog2, with a bit to
// spare; the largest |v| of the batch is found on the way), or the factor is kept to 2^kLazyLog2Wide and every row
// has its maximum found. Where |q| |k| scale <= kBoundLog2 for every key
// (Cauchy-Schwarz, norms taken before the rotation's rounding to bf16), two scores of a row differ by at
// most 2 * 44 * (1 + 2^-7) < 90, so from its second tile on the row's maximum cannot move: neither the
// 64 comparisons nor the exchange between the two threads of a row are needed, and the exponentials start
// on the first 32 scores while the other 32 are still being loaded. The result does not depend on
// whether the bound was known, so all routes give the same bits. Q and K of N(0, 1) values reach 17-30 (D = 64 / 128). Measured, whole step:
// 16 prompts of up to 22 861 tokens, 32 heads, D = 128: 14.69 -> 12.2 ms (attention 14.1 -> 11.15 ms, 1156
// TFLOP/s, from then on at the power cap: SM clock ~1620 MHz); 256 prompts of up to 3991, 32 / 8 heads:
// 7.22 -> 6.48 ms. A wait for S took a softmax warp 2570 cycles per 128-key tile, now ~1250, of ~2900 in all.
constexpr float kLazyLog2 = 90.f;
constexpr float kBoundLog2 = 44.f;
constexpr float kLazyLog2Wide = 8.f;
constexpr int kValueRoomLog2 = 36;
constexpr uint32_t kRing = 3;               // decoded work items in flight between the fetching thread and its readers
constexpr int kRingInts = 20;              // ints per ring entry

// BN: key rows per tile. 128 in shared-stream mode: one Q tile per slot, rings of K and V tiles that both
// slots read, an O staging buffer per slot. 64 in independent mode: per slot two Q tiles (that of the
// next item is loaded and rotated while the current item is computed) and one ring in which K and V tiles
// alternate; at D = 128, where there is no room for a staging buffer, O is staged in the Q tile of its own
// item. At D = 128 both modes come to exactly 227 KB.
template <int D, int BN> struct AttnCfg {
  static constexpr bool kIndep = BN == kTileNShort;
  static constexpr int kKStages = D == 128 ? 2 : 4, kVStages = kKStages;   // shared-stream mode
  static constexpr int kKVStages = D == 128 ? 3 : 4;         // independent mode, per slot
  static constexpr bool kStageInQ = D == 128;                // independent mode
  static constexpr int kQBytes = BM * D * 2;                 // one Q tile
  static constexpr int kKVBytes = BN * D * 2;
  // barriers + work ring (1024) and the row-maximum exchange buffer [slot][half][row] (2048), placed
  // in front of the 1024-byte-aligned tiles
  static constexpr int kMiscBytes = 3072;
  static constexpr int kStageOBytes = BM * 128;              // per slot: one 64-column box of O
  static constexpr int kTileBytes = kIndep ? 2 * (2 * kQBytes + kKVStages * kKVBytes + (kStageInQ ? 0 : kStageOBytes))
                                           : 2 * kQBytes + (kKStages + kVStages) * kKVBytes + 2 * kStageOBytes;
  static constexpr int kSmemBytes = kMiscBytes + kTileBytes;
  static constexpr uint32_t kTmemS = 0;                      // S_t at 128 * t
  static constexpr uint32_t kTmemO = 256;                    // O_t at 256 + D * t
};

// ------------------------------------------------------------------------------------------
// PTX wrappers
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes, uint32_t issue) {
  asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %2, 0;\n@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}"
               ::"r"(bar), "r"(bytes), "r"(issue) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// A value that is the same in all lanes, said so to the compiler (all 32 lanes call).
__device__ __forceinline__ int uniform(int x) { return __shfl_sync(0xffffffffu, x, 0); }

// Every wait in the kernel goes through here or through the two forms for a warp below: it gives up after `limit`, leaving
// why in the CTA-wide abort word, so that all roles leave their loops; the code goes to the device status word at the end
// of the kernel at the latest. A kernel of this file has some forty waits, inlined, and the warps of a scheduler run three
// to five roles: what they execute has to fit its instruction cache (a straight line of code takes 1.0 cycles an
// instruction up to 32 KB, 3.1 to 128 KB, 6 beyond, one scheduler at work). In the independent mode, with a 64-bit clock,
// a global atomic and a poll counter in each wait 1.1 of the 6 warps of a scheduler stood without an instruction at any
// time; in this form, and with each load of the producer loop at one place, 0.18 (64 prompts on a 7B layer: attention
// 194 -> 158 us under ncu with the changes around them, whole steps 285 -> 258). (As calls of one function the waits do not
// fit the softmax threads' registers.)
struct WaitCtx {
  uint32_t abort;               // address in shared memory, 0: go on
  uint32_t limit;               // in units of 1024 ns
  int32_t* status;              // global, may be null
};
// (A poll parks the thread for about 20 us, so the clock, which starts at the first failed one, is read seldom.)
template <int kCode>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const WaitCtx& w) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n.reg .b32 t0, t1, x;\n.reg .b64 g;\n"
      "mov.b32 t0, 0;\n"
      "AGAIN_%=:\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "@p bra DONE_%=;\n"
      "ld.volatile.shared.b32 x, [%3];\n"
      "setp.ne.b32 p, x, 0;\n"
      "@p bra DONE_%=;\n"
      "mov.u64 g, %%globaltimer;\n"
      "shr.u64 g, g, 10;\n"
      "cvt.u32.u64 t1, g;\n"
      "or.b32 t1, t1, 1;\n"
      "setp.eq.b32 p, t0, 0;\n"
      "selp.b32 t0, t1, t0, p;\n"
      "sub.u32 t1, t1, t0;\n"
      "setp.le.u32 p, t1, %4;\n"
      "@p bra AGAIN_%=;\n"
      "st.volatile.shared.b32 [%3], %5;\n"
      "DONE_%=:\n}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(w.abort), "r"(w.limit), "n"(kCode) : "memory");
  return ok != 0;
}
// The same for a whole warp in uniform control flow: every lane polls, the vote decides.
template <int kCode>
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, const WaitCtx& w) {
  return __all_sync(0xffffffffu, mbar_wait<kCode>(bar, parity, w));
}

// For the warps of the shared-stream mode that load and issue: one loop of the whole warp, which reads the clock at every
// eighth failed poll and writes the code to the status word itself. There the instruction cache is not the limit, and the
// form above made the issuing warp slower: one prompt of 16 000 tokens on 8 / 4 heads of 64 367 us a step with it, 353 in
// this form; six of 9000 on 32 / 8 heads of 64 2790 -> 2690; 16 prompts of up to 22 861 tokens on 32 heads of 128 12.18 ->
// 12.01 ms. (The softmax threads' waits take the same time in either form.)
template <int kCode>
__device__ __forceinline__ bool mbar_wait_issuer(uint32_t bar, uint32_t parity, const WaitCtx& w) {
  uint32_t t0 = 0, polls = 0;
  while (true) {
    uint32_t ok;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (__all_sync(0xffffffffu, ok != 0)) return true;
    if ((++polls & 7u) == 0) {
      uint32_t gone;
      asm volatile("ld.volatile.shared.b32 %0, [%1];" : "=r"(gone) : "r"(w.abort) : "memory");
      const uint32_t now = (uint32_t)(global_ns() >> 10) | 1u;
      if (t0 == 0) t0 = now;
      if (gone == 0 && now - t0 > w.limit) {
        asm volatile("st.volatile.shared.b32 [%0], %1;" ::"r"(w.abort), "n"(kCode) : "memory");
        if (w.status) atomicCAS(w.status, 0, kCode);
        gone = 1;
      }
      if (__any_sync(0xffffffffu, gone != 0)) return false;
    }
  }
}

// The warps that issue TMA loads and MMAs run in uniform control flow: all 32 lanes execute the loop, the waits
// and the address arithmetic, and a predicate (`issue`, set on one lane by elect.sync) picks the lane that
// issues. With a branch on the lane index instead, every tcgen05.mma takes ~50 cycles to issue whatever its size
// (a group of 8: 400 cycles against 101-136 in this form, one CTA per SM, with or without 16 busy warps
// beside it), which held the tensor pipe below its rate of one 128 x 128 x 16 product per 64 cycles. A TMA
// load with its expect_tx and the wait for an earlier one takes a warp 307 ns with the branch and 259 ns in this
// form, for any box from 2 to 32 KB, so a tile is one load: whole steps 3.5 % faster for 256 prompts of up to
// 3991 tokens on 32 / 8 heads, 2.7 % for 2048 short ones, 1 to 2 % for the others.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(r));
  return r;
}
// Coordinates: column (0), head, row, chunk (0), bin; see make_map. Issued, like the MMAs below, by one lane of a
// warp in uniform control flow.
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* map, uint32_t bar, int head, int row, int bin,
                                         uint32_t issue) {
  asm volatile(
      "{\n.reg .pred q;\nsetp.ne.b32 q, %6, 0;\n"
      "@q cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%7, %3, %4, %7, %5}], [%2];\n}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(head), "r"(row), "r"(bin), "r"(issue), "r"(0)
      : "memory");
}
__device__ __forceinline__ void tma_store(const CUtensorMap* map, uint32_t src, int head, int row, int chunk, int bin) {
  asm volatile(
      "cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%6, %2, %3, %4, %5}], [%1];"
      ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(head), "r"(row), "r"(chunk), "r"(bin), "r"(0)
      : "memory");
}
__device__ __forceinline__ void tma_store_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar, uint32_t issue) {
  asm volatile(
      "{\n.reg .pred q;\nsetp.ne.b32 q, %1, 0;\n"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(bar), "r"(issue) : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { __syncwarp(); asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { __syncwarp(); asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptors (tcgen05), 128-byte swizzle, rows of 128 bytes, 8-row groups
// 1024 bytes apart. Low word: start address >> 4 and (MN-major operands only) the distance between
// 64-element spans of the MN dimension >> 4. High word: constant (8-row group stride, descriptor
// version, swizzle mode). Stepping along a tile only ever adds a small constant to the low word.
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr, uint32_t lbo_bytes) {
  return ((saddr & 0x3FFFFu) >> 4) | ((lbo_bytes >> 4) << 16);
}
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);

// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc,
                                       uint32_t accumulate, uint32_t issue) {
  asm volatile(
      "{\n.reg .pred p, q;\n.reg .b64 da, db;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 q, %6, 0;\n"
      "mov.b64 da, {%1, %5};\nmov.b64 db, {%2, %5};\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHi), "r"(issue) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t idesc,
                                       uint32_t accumulate, uint32_t issue) {
  asm volatile(
      "{\n.reg .pred p, q;\n.reg .b64 db;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 q, %6, 0;\n"
      "mov.b64 db, {%2, %5};\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p;\n}"
      ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHi), "r"(issue) : "memory");
}

// 32 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  __syncwarp();
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
// tcgen05.wait::ld with the loaded registers passed through it, so that nothing can be moved between
// the load and the wait (used where other work stands between the two).
__device__ __forceinline__ void tc_wait_ld32(uint32_t (&r)[32]) {
  __syncwarp();
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
        "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
        "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
        "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
      :: "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  __syncwarp();
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};"
      ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(taddr) : "memory");
}

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}
// Packed pairs of fp32 (sm_100 f32x2 arithmetic): halves the FMA-pipe instruction count of the
// softmax inner loop.
__device__ __forceinline__ uint64_t pack_f2(uint32_t lo, uint32_t hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
  return d;
}
__device__ __forceinline__ void unpack_f2(uint64_t x, float& lo, float& hi) {
  uint32_t a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(x));
  lo = __uint_as_float(a);
  hi = __uint_as_float(b);
}
__device__ __forceinline__ uint64_t fma_f2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add_f2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul_f2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float sum_f2x2(uint64_t a, uint64_t b) {
  float x, y, z, w;
  unpack_f2(a, x, y);
  unpack_f2(b, z, w);
  return (x + z) + (y + w);
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);     // .x (low 16 bits) = lo
  return *reinterpret_cast<uint32_t*>(&h);
}

// Probabilities of 32 scores: p = exp2(s * c - m), added up in sum_a / sum_b (two packed accumulators)
// and packed to bf16.
__device__ __forceinline__ void exp_chunk(const uint32_t* v, uint64_t c2, uint64_t negm2, uint64_t& sum_a, uint64_t& sum_b,
                                          uint32_t (&pk)[16]) {
#pragma unroll
  for (int i = 0; i < 32; i += 4) {
    float p0, p1, p2, p3;
    unpack_f2(fma_f2(pack_f2(v[i], v[i + 1]), c2, negm2), p0, p1);
    unpack_f2(fma_f2(pack_f2(v[i + 2], v[i + 3]), c2, negm2), p2, p3);
    p0 = fast_exp2(p0); p1 = fast_exp2(p1); p2 = fast_exp2(p2); p3 = fast_exp2(p3);
    sum_a = add_f2(sum_a, pack_f2(__float_as_uint(p0), __float_as_uint(p1)));
    sum_b = add_f2(sum_b, pack_f2(__float_as_uint(p2), __float_as_uint(p3)));
    pk[i >> 1] = pack_bf16(p0, p1);
    pk[(i >> 1) + 1] = pack_bf16(p2, p3);
  }
}

// Largest of 64 scores.
__device__ __forceinline__ float max64(const uint32_t (&v)[64]) {
  float m0 = fmax3(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]));
  float m1 = fmax3(__uint_as_float(v[3]), __uint_as_float(v[4]), __uint_as_float(v[5]));
  float m2 = fmax3(__uint_as_float(v[6]), __uint_as_float(v[7]), __uint_as_float(v[8]));
  float m3 = fmax3(__uint_as_float(v[9]), __uint_as_float(v[10]), __uint_as_float(v[11]));
#pragma unroll
  for (int i = 12; i + 7 < 64; i += 8) {
    m0 = fmax3(m0, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
    m1 = fmax3(m1, __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]));
    m2 = fmax3(m2, __uint_as_float(v[i + 4]), __uint_as_float(v[i + 5]));
    m3 = fmax3(m3, __uint_as_float(v[i + 6]), __uint_as_float(v[i + 7]));
  }
  m0 = fmax3(m0, __uint_as_float(v[60]), __uint_as_float(v[61]));      // 12 + 8 * 6 = 60
  m1 = fmax3(m1, __uint_as_float(v[62]), __uint_as_float(v[63]));
  return fmaxf(fmax3(m0, m1, m2), m3);
}

// Bits [c_lo, c_hi] of a 64-bit word set (none if the interval is empty); c_hi <= 63, c_lo >= 0.
__device__ __forceinline__ uint64_t visible_mask64(int c_lo, int c_hi) {
  if (c_hi < c_lo) return 0ull;
  return (~0ull << c_lo) & (~0ull >> (63 - c_hi));
}

// Instruction descriptor: fp32 accumulate, bf16 A and B, A K-major, M = 128.
__host__ __device__ constexpr uint32_t instr_desc(uint32_t n, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((n >> 3) << 17) |
         ((128u >> 4) << 24);
}

struct AttnArgs {
  int32_t* counter;              // global work counter (a header word of the table)
  int32_t off_seg_start, off_items;
  int32_t n_items;               // geometry entries in the work list
  int32_t subs;                  // work indices per (KV head, geometry entry)
  int32_t pair_heads;            // 1: slots are two query heads; 0: two row tiles of one head
  int32_t group;                 // query heads per KV head
  int32_t fold;                  // independent mode: query heads folded into a query tile (tile row m is
  int32_t fold_shift;            //   bin row q_row0 + (m >> fold_shift) of head head[0] + (m & (fold - 1)))
  int32_t capacity;              // rows per bin
  int32_t total_work;            // n_kv_heads * n_items * subs
  int32_t tail_head0;            // KV heads from here on are drawn together (launch_attention_t says why):
  int32_t tail_start, tail_cols; //   work indices from tail_start on, tail_cols of them per geometry entry
  float scale_log2;              // softmax scale * log2(e)
  float bound2;                  // (kBoundLog2 / scale_log2)^2: |q|^2 |k|^2 up to which scores are bounded
  const float2* rope_table;      // [D/4][capacity][2] (cos, sin) pairs, or null: Q arrives already rotated
  const uint32_t* k_norm2;       // shared-stream mode: [Hkv] largest |k|^2 (float bits); null: no bound on the scores
  const uint32_t* q_norm2;       // [Hq] largest |q|^2; used when Q arrives already rotated
  const uint32_t* v_max;         // shared-stream mode: largest |v| (bf16 bits); null: not known
  float v_room;                  // 2^kValueRoomLog2 / capacity: |v| up to which kLazyLog2 holds
  int32_t* status;
  uint32_t wait_limit;           // in units of 1024 ns
  __nv_bfloat16* v_cache;                         // kFill: the V caches
  int32_t off_true_len, off_cap, off_cache_off;   // per-segment arrays in the table, for them
};

// What one work index means for a CTA.
struct Work {
  int bin, kv_row0, n, q_row0[2], jb[2], je[2], head[2], kv_head;
  int bin_used, seg_end, key_lo[2], seg_first[2], single_seg;
};

template <class Table>
__device__ __forceinline__ void decode_work(const AttnArgs& a, const Table& tab, int w, Work& wk) {
  // KV head, entry, sub (outermost first); in the tail entry, KV head, sub
  const bool tail = w >= a.tail_start;
  const uint32_t wr = (uint32_t)(tail ? w - a.tail_start : w), cols = (uint32_t)(tail ? a.tail_cols : a.subs);
  const uint32_t q = wr / cols, c = wr - q * cols;
  const uint32_t num = tail ? c : q, den = (uint32_t)(tail ? a.subs : a.n_items);
  const uint32_t d = num / den, m = num - d * den;
  const int gi = (int)(tail ? q : m), sub = (int)(tail ? m : c);
  wk.kv_head = (int)d + (tail ? a.tail_head0 : 0);
  const int at = a.off_items + kItemInts * gi;
  const int4 x = tab.i128(at), y = tab.i128(at + 4);
  wk.bin = x.x; wk.kv_row0 = x.y; wk.n = x.z; wk.q_row0[0] = x.w; wk.q_row0[1] = y.x;
  wk.jb[0] = 0; wk.je[0] = y.z;
  wk.jb[1] = y.y; wk.je[1] = (y.x >= 0) ? x.z : y.y;       // unused slot: empty range
  const int4 r = tab.i128(at + 8), z = tab.i128(at + 12);    // what the softmax threads need to place their rows
  wk.bin_used = r.x; wk.seg_end = r.y; wk.key_lo[0] = r.z; wk.key_lo[1] = r.w;
  wk.seg_first[0] = z.x; wk.seg_first[1] = z.y; wk.single_seg = z.z;
  if (a.pair_heads) {
    wk.head[0] = wk.kv_head * a.group + 2 * sub;
    wk.head[1] = wk.head[0] + 1;
  } else {
    wk.head[0] = wk.head[1] = wk.kv_head * a.group + sub * a.fold;
  }
}

// The next work index of a CTA or slot, -1 when there is none left (a whole warp calls). The first one is the
// drawer's own number, of `drawers` (no round trip to the counter in front of the first loads).
__device__ __forceinline__ int draw_work(const AttnArgs& a, int lane, int drawers) {
  int w = 0;
  if (lane == 0) w = drawers + atomicAdd(a.counter, 1);
  w = __shfl_sync(0xffffffffu, w, 0);
  return w < a.total_work ? w : -1;
}

// The fetching thread decodes an item once and publishes it in shared memory; every other role
// reads it from there instead of going back to global memory.
__device__ __forceinline__ void ring_write(volatile int* e, int w, const Work& wk) {
  e[0] = w; e[1] = wk.bin; e[2] = wk.kv_row0; e[3] = wk.n;
  e[4] = wk.q_row0[0]; e[5] = wk.q_row0[1]; e[6] = wk.jb[1]; e[7] = wk.je[0];
  e[8] = wk.je[1]; e[9] = wk.head[0]; e[10] = wk.head[1]; e[11] = wk.kv_head;
  e[12] = wk.bin_used; e[13] = wk.seg_end; e[14] = wk.key_lo[0]; e[15] = wk.key_lo[1];
  e[16] = wk.seg_first[0]; e[17] = wk.seg_first[1]; e[18] = wk.single_seg;
}

enum WaitCode { kWaitItemFull = 1, kWaitItemEmpty, kWaitQFull, kWaitQEmpty, kWaitKFull, kWaitKEmpty,
                kWaitVFull, kWaitVEmpty, kWaitS, kWaitP, kWaitOFull, kWaitOEmpty, kWaitPair, kWaitRowSum };

// Start row of the prompt that holds bin-local row `i_row`, among the prompts seg_begin .. seg_end-1
// of a bin whose start rows (ascending) are in the table from `starts` on; `lo` if none of them starts at or before the
// row. All 32 lanes call it with the same range and with row_max = the largest row of the warp: the
// starts are loaded 32 at a time, one per lane, and handed round with shuffles, so the walk costs one
// memory round trip per 32 prompts.
template <class Table>
__device__ __forceinline__ int seg_start_at(const Table& tab, int starts, int seg_begin, int seg_end, int i_row, int row_max,
                                            int lo, int lane) {
  for (int base = seg_begin; base < seg_end; base += 32) {
    const int cnt = min(32, seg_end - base);
    const int mine = (lane < cnt) ? tab.i32(starts + base + lane) : 0x7fffffff;
    for (int sg = 0; sg < cnt; ++sg) {
      const int st = __shfl_sync(0xffffffffu, mine, sg);
      if (st > row_max) return lo;                     // warp-uniform: no later prompt starts in these rows
      if (st <= i_row) lo = st;
    }
  }
  return lo;
}

// Independent mode: place in the slot's K / V ring sequence K0 K1 V0 K2 V1 K3 V2 ... of the k-th key tile of the slot.
// With three stages K(k+3) then follows V(k) and V(k+2) follows K(k+2) in a stage: either load has more than a
// tile's time (in the sequence K0 V0 K1 V1 ..., K(k+3) followed V(k+1), and its load was waited for every time).
__device__ __forceinline__ uint32_t kv_index_k(uint32_t k) { return k ? 2u * k - 1u : 0u; }
__device__ __forceinline__ uint32_t kv_index_v(uint32_t k) { return 2u * k + 2u; }

// kIndep = false: the two slots of a CTA work on one item and share its K/V stream (long
//   sequences, GQA head pairs). kIndep = true: every slot draws its own single-tile items and loads
//   its own K/V tiles (64 rows each), so neither slot ever waits for the other (short prompts, where
//   pairing two row tiles of different length would leave one slot idle for a tile per item).
// kFill (independent mode): two more warps write the V rows to the caches.
template <int D, bool kIndep, bool kFill, class Table>
__global__ void __launch_bounds__(kIndep ? kAttnThreadsIndep : kAttnThreads, 1)
attention_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                 const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o,
                 const __grid_constant__ AttnArgs args, const __grid_constant__ Table tab) {
  constexpr int BN = kIndep ? kTileNShort : kTileN;
  using Cfg = AttnCfg<D, BN>;
  constexpr int NK = Cfg::kKStages, NV = Cfg::kVStages;

  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t s_misc = smem_u32(smem_raw);
  uint8_t* misc = smem_raw;
  const uint32_t s_q = (s_misc + 3072u + 1023u) & ~1023u;       // tiles need 1024-byte alignment
  const uint32_t s_kv = s_q + 4 * Cfg::kQBytes;                 // independent mode: [2 slots][kKVStages] behind [2][2] Q tiles
  const uint32_t s_k = s_q + 2 * Cfg::kQBytes;                  // shared-stream mode: [NK] behind [2] Q tiles
  const uint32_t s_v = s_k + NK * Cfg::kKVBytes;                // [NV]
  const uint32_t s_stage_o = kIndep ? s_kv + 2 * Cfg::kKVStages * Cfg::kKVBytes : s_v + NV * Cfg::kKVBytes;   // [2] slots, epilogue staging
  {
    uint32_t dyn_bytes;
    asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_bytes));
    if (s_q + Cfg::kTileBytes > s_misc + dyn_bytes) {           // base less aligned than expected
      if (threadIdx.x == 0 && args.status) atomicCAS(args.status, 0, 100);
      return;
    }
  }
  // mbarriers, 8 bytes each
  const uint32_t bar_item_full = s_misc + 0;     // [2 rings][kRing]
  const uint32_t bar_item_empty = s_misc + 64;   // [2 rings][kRing]
  const uint32_t bar_q_full = s_misc + (kIndep ? 896 : 128);    // [2]; independent mode: [2 slots][2 Q tiles]
  const uint32_t bar_q_empty = s_misc + (kIndep ? 128 : 144);   // [2]; independent mode: [2 slots][2 Q tiles]
  const uint32_t bar_s_full = s_misc + 160;      // [2 slots][2 S buffers]; shared mode uses [t][0]
  const uint32_t bar_p_full = s_misc + 192;      // [2 slots][2 S buffers]
  const uint32_t bar_o_full = s_misc + (kIndep ? 384 : 224);    // [2]
  const uint32_t bar_o_empty = s_misc + (kIndep ? 224 : 240);   // [2]; independent mode: [2 slots][item & 1]
  const uint32_t bar_k_full = s_misc + 256;      // [4]
  const uint32_t bar_k_empty = s_misc + 288;     // [4]
  const uint32_t bar_v_full = s_misc + (kIndep ? 288 : 320);    // [4]; independent mode: bar_k_full, bar_v_full [2 slots][k & 1]
  const uint32_t bar_v_empty = s_misc + 352;     // [4]
  const uint32_t bar_pv_done = s_misc + 320;     // [2 slots][2] independent mode: P(k) V(k) has been computed ([k & 1])
  const uint32_t bar_v_read = s_misc + 352;      // [2 slots][2] and the rows of V(k) have been read for the caches
  const uint32_t bar_q_rot = s_misc + (kIndep ? 928 : 384);     // [2] Q_t has been rotated in place (fused path);
                                                 // independent mode: [2 slots][2 Q tiles], its rows' first keys are there too
  const uint32_t bar_pair0 = s_misc + 896;       // [2 slots][4 quadrants] shared-stream mode: rendezvous of the two warps that share rows
  const uint32_t bar_v_seen0 = s_misc + 960, bar_v_seen1 = s_misc + 1008;   // [2] each, independent mode: V(k) is there, said the slot's warp 22 / 23
  const uint32_t bar_l_ready = s_misc + 976;     // [2][2] independent mode: the slot's row sums of item i are in shared memory ([slot][i & 1])
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(misc + 400);
  volatile int* s_abort = reinterpret_cast<volatile int*>(misc + 404);
  volatile int* s_ring = reinterpret_cast<volatile int*>(misc + 416);   // [2 rings][kRing][kRingInts]
  volatile uint8_t* s_bounded = misc + 1008;     // [2 slots][4 quadrants][2 halves] shared-stream mode: the warp's rows are bounded
  volatile float* s_xchg = reinterpret_cast<volatile float*>(misc + 1024);   // [2 slots][2 halves][128 rows]
  static_assert(416 + 2 * kRing * kRingInts * 4 <= 896, "ring does not fit");
  static_assert(NK <= 4 && NV <= 4 && Cfg::kKVStages <= 4, "barrier slots");

  const int warp = uniform((int)(threadIdx.x >> 5));
  const int lane = threadIdx.x & 31;
  const WaitCtx wctx{s_misc + 404u, args.wait_limit, args.status};

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2 * (int)kRing; ++i) {
      mbar_init(bar_item_full + 8 * i, 1);
      // readers of a ring entry: the MMA warp(s) and the softmax threads of the slot(s) it feeds;
      // in shared mode also the two Q loaders
      // (and in independent mode the slot's cache writer, where caches are filled)
      mbar_init(bar_item_empty + 8 * i, kIndep ? 2 + kSoftmaxThreads + (kFill ? 1 : 0) : 1 + 2 + 2 * kSoftmaxThreads);
    }
    for (int i = 0; i < 2; ++i) {
      for (int b = 0; b < 2; ++b) {
        mbar_init(bar_s_full + 8 * (2 * i + b), 1);
        mbar_init(bar_p_full + 8 * (2 * i + b), kIndep ? kSoftmaxThreads / 2 : kSoftmaxThreads);
        mbar_init(bar_l_ready + 8 * (2 * i + b), kSoftmaxThreads / 2);
      }
      mbar_init(bar_o_full + 8 * i, 1);
      mbar_init(bar_o_empty + 8 * i, kIndep ? kSoftmaxThreads / 2 : kSoftmaxThreads);
      if (kIndep) mbar_init(bar_o_empty + 16 + 8 * i, kSoftmaxThreads / 2);
    }
    if constexpr (kIndep) {
      for (int i = 0; i < 4; ++i) {
        mbar_init(bar_q_full + 8 * i, 1);
        mbar_init(bar_q_empty + 8 * i, Cfg::kStageInQ ? 4 : 1);   // one lane of each helper warp, or a commit
        mbar_init(bar_q_rot + 8 * i, kSoftmaxThreads / 2);
      }
      for (int i = 0; i < 4; ++i) {
        mbar_init(bar_k_full + 8 * i, 1);
        mbar_init(bar_v_full + 8 * i, 1);
        mbar_init(bar_pv_done + 8 * i, 1);
        mbar_init(bar_v_read + 8 * i, 1);
      }
      for (int i = 0; i < 2; ++i) if (kFill) { mbar_init(bar_v_seen0 + 8 * i, 1); mbar_init(bar_v_seen1 + 8 * i, 1); }
    } else {
      for (int i = 0; i < 2; ++i) {
        mbar_init(bar_q_full + 8 * i, 1);
        mbar_init(bar_q_empty + 8 * i, 1);
        mbar_init(bar_q_rot + 8 * i, kSoftmaxThreads);
        for (int qd = 0; qd < 4; ++qd) mbar_init(bar_pair0 + 8 * (4 * i + qd), 64);
      }
      for (int s = 0; s < NK; ++s) { mbar_init(bar_k_full + 8 * s, 1); mbar_init(bar_k_empty + 8 * s, 1); }
      for (int s = 0; s < NV; ++s) { mbar_init(bar_v_full + 8 * s, 1); mbar_init(bar_v_empty + 8 * s, 1); }
    }
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(s_tmem_base)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = (uint32_t)uniform((int)*s_tmem_base);
  // Everything above is set-up that touches no tensor: with a programmatic dependent launch it runs
  // while the kernel before this one (rotation / cache scatter) is still finishing.
  pdl_wait();
  // The next call's table upload may read host memory as SMs run out of work here (2048 short prompts 193 -> 186 us a
  // step, 64 on a 7B layer 282 -> 278). Not before this wait: the next kernel may count on all that was queued before
  // this one. Not where tables are parameters: the rotation kernel, which is next then, would fill the first SMs to
  // become idle with its blocks (16 prompts on a 7B layer 49.5 -> 53.6).
  if (Table::kUploaded) pdl_launch_dependents();

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIndep ? kRegsOtherIndep : kRegsOther));
    if constexpr (kIndep) {
      if (warp >= 2) {
        // -------------------------------------------------------------- producer of slot t:
        // draws the slot's own items, loads Q and the item's K / V tiles. The next item is drawn and announced
        // at the start of the current one and its Q loaded behind the first two key tiles, so that the helper
        // threads rotate it under the current item (loaded behind the last scores of an item and rotated
        // then, Q kept the slot waiting 5500 cycles per item of 5.3 key tiles, 2000 without the rotation; whole
        // steps: 34 bins of a stream 1197 -> 1116 us, 64 prompts 315 -> 307, both 32 heads, D = 128). K runs
        // one tile ahead of V, over the end of the item too: the order in which the MMAs want them.
        const int t = warp - 2;
        constexpr int NS = Cfg::kKVStages;
        const uint32_t issue = elect_one();
        const uint32_t ring_bar = 8 * (uint32_t)t * kRing;
        volatile int* ring_base = s_ring + t * (int)kRing * kRingInts;
        auto announce = [&](const uint32_t it, const int w, Work& wk) -> bool {      // w < 0: there is no item `it`
          if (w >= 0) decode_work(args, tab, w, wk);
          const uint32_t ring = it % kRing;
          if (!mbar_wait_warp<kWaitItemEmpty>(bar_item_empty + ring_bar + 8 * ring, ((it / kRing) & 1u) ^ 1u, wctx)) return false;
          if (issue) {
            if (w >= 0) ring_write(ring_base + ring * kRingInts, w, wk);
            else ring_base[ring * kRingInts] = -1;
            mbar_arrive(bar_item_full + ring_bar + 8 * ring);
          }
          return true;
        };
        auto load_q = [&](const uint32_t it, const Work& wk) -> bool {
          // O of the item before the previous one must have left this Q tile (or, where O is staged
          // elsewhere, its last scores must have been computed)
          const uint32_t qb = 2u * (uint32_t)t + (it & 1u);
          if (!mbar_wait_warp<kWaitQEmpty>(bar_q_empty + 8 * qb, ((it >> 1) & 1u) ^ 1u, wctx)) return false;
          mbar_expect_tx(bar_q_full + 8 * qb, Cfg::kQBytes, issue);
          tma_load(s_q + qb * Cfg::kQBytes, &map_q, bar_q_full + 8 * qb, wk.head[0], wk.q_row0[0], wk.bin, issue);
          return true;
        };
        // A stage is free when what it held has been used: K(k) when S(k) is there, V(k) when P(k) V(k) is, and, where
        // caches are filled, its rows have been read. These are barriers that others wait on anyway: a commit
        // of its own behind each group of MMAs takes the issuing warp ~140 cycles. None can complete the next phase
        // before this warp has seen the one it waits for: that takes K(k) where K(k) waits (S(k), or P(k - 1) V(k - 1), whose
        // V comes after it), V(k) or K(k + 2) where V(k) waits.
        static_assert(NS == 3 || NS == 4, "which tile a stage held is worked out for these");
        auto wait_s = [&](const uint32_t k) -> bool {
          return mbar_wait_warp<kWaitKEmpty>(bar_s_full + 8 * (2u * (uint32_t)t + (k & 1u)), (k >> 1) & 1u, wctx);
        };
        auto wait_pv = [&](const uint32_t k) -> bool {
          const uint32_t bar = 8 * (2u * (uint32_t)t + (k & 1u));
          return mbar_wait_warp<kWaitVEmpty>(bar_pv_done + bar, (k >> 1) & 1u, wctx) &&
                 (!kFill || mbar_wait_warp<kWaitVEmpty>(bar_v_read + bar, (k >> 1) & 1u, wctx));
        };
        auto load_kv = [&](const CUtensorMap* map, const uint32_t idx, const uint32_t bar, const int head, const int row, const int bin) {
          mbar_expect_tx(bar, Cfg::kKVBytes, issue);
          tma_load(s_kv + ((uint32_t)t * NS + idx % NS) * Cfg::kKVBytes, map, bar, head, row, bin, issue);
        };
        // K(k): of four stages, after K(k - 2), whose barrier this is again too; of three, after V(k - 3), or K(0) where k = 2
        auto load_k = [&](const uint32_t k, const int head, const int row, const int bin) -> bool {
          if (NS == 4 ? k >= 2u && !wait_s(k - 2u) : k >= 3u ? !wait_pv(k - 3u) : k == 2u && !wait_s(0u)) return false;
          load_kv(&map_k, kv_index_k(k), bar_k_full + 8 * (2u * (uint32_t)t + (k & 1u)), head, row, bin);
          return true;
        };
        // V(k): of four stages, after V(k - 2), or K(0) where k = 1 (S(1) comes after S(0)); of three, after K(k)
        auto load_v = [&](const uint32_t k, const int head, const int row, const int bin) -> bool {
          if (NS == 4 ? (k >= 2u ? !wait_pv(k - 2u) : k == 1u && !wait_s(1u)) : k >= 1u && !wait_s(k)) return false;
          load_kv(&map_v, kv_index_v(k), bar_v_full + 8 * (2u * (uint32_t)t + (k & 1u)), head, row, bin);
          return true;
        };
        const int drawers = 2 * (int)gridDim.x;
        int w = (int)blockIdx.x + t * (int)gridDim.x;
        if (w >= args.total_work) w = -1;
        Work wk, wk_next;
        bool ok = announce(0, w, wk);
        if (ok && w >= 0) ok = load_q(0, wk) && load_k(0u, wk.kv_head, wk.kv_row0, wk.bin);
        uint32_t kc = 0;                      // key tiles of the slot's stream whose V has been loaded
        for (uint32_t it_n = 0; ok && w >= 0; ++it_n) {
          const int w_next = draw_work(args, lane, drawers);
          if (!(ok = announce(it_n + 1u, w_next, wk_next))) break;
          for (int j = 0; ok && j < wk.n; ++j, ++kc) {
            const bool here = j + 1 < wk.n;             // K of this item, or the first of the next
            if (here || w_next >= 0)
              ok = load_k(kc + 1u, here ? wk.kv_head : wk_next.kv_head, here ? wk.kv_row0 + (j + 1) * BN : wk_next.kv_row0,
                          here ? wk.bin : wk_next.bin);
            if (ok) ok = load_v(kc, wk.kv_head, wk.kv_row0 + j * BN, wk.bin);
            if (ok && j == min(1, wk.n - 1) && w_next >= 0) ok = load_q(it_n + 1u, wk_next);
          }
          w = w_next;
          wk = wk_next;
        }
      } else if (warp < 2) {
        // -------------------------------------------------------------- scores of slot t: S(k) = Q K(k)^T
        // The slot's tiles form one stream across items; tile k uses S buffer k & 1. S(k) is issued as soon as its
        // K tile is there and P(k - 2) V(k - 2), which reads the same buffer, is done: while the softmax
        // threads work on tile k - 1, also when tile k opens the slot's next item (its Q has been loaded and rotated
        // under this one). The products P V have a warp of their own (22, 23): one warp that issued both took 1400 cycles
        // of its own per tile, besides the ~1200 it waited (2048 short prompts on 32 / 8 heads of 64 174 -> 167 us a step, 64
        // prompts on a 7B layer 237.3 -> 235.6, 34 bins of a stream 896 -> 889).
        const int t = warp;
        const uint32_t issue = elect_one();
        constexpr uint32_t idesc_qk = instr_desc(BN, false);
        constexpr int NS = Cfg::kKVStages;
        const uint32_t q_lo = desc_lo(s_q, 0) + 2u * (uint32_t)t * (Cfg::kQBytes >> 4);
        const uint32_t k_lo = desc_lo(s_kv, 0) + (uint32_t)(t * NS) * (Cfg::kKVBytes >> 4);
        const uint32_t tm_s = tmem_base + Cfg::kTmemS + 128u * (uint32_t)t;
        uint32_t kc = 0;
        bool ok = true;
        for (uint32_t it_n = 0; ok; ++it_n) {
          const uint32_t ring = (uint32_t)t * kRing + it_n % kRing, it2 = 2u * (uint32_t)t + (it_n & 1u);
          if (!mbar_wait_warp<kWaitItemFull>(bar_item_full + 8 * ring, (it_n / kRing) & 1u, wctx)) break;
          const volatile int* e = s_ring + ring * kRingInts;
          const int w = uniform(e[0]), n = uniform(e[3]);
          if (issue) mbar_arrive(bar_item_empty + 8 * ring);
          if (w < 0) break;
          // The epilogue of the item before the previous one has read O_t, and the row sums: the softmax threads must not
          // get further ahead of it, also where every item is one tile.
          if (it_n >= 2u && !mbar_wait_warp<kWaitOEmpty>(bar_o_empty + 8 * it2, ((it_n - 2u) >> 1) & 1u, wctx)) break;
          if (!mbar_wait_warp<kWaitQFull>(bar_q_rot + 8 * it2, (it_n >> 1) & 1u, wctx)) break;
          const uint32_t a_lo = q_lo + (it_n & 1u) * (Cfg::kQBytes >> 4);
          for (int j = 0; j < n; ++j, ++kc) {
            const uint32_t st = kv_index_k(kc) % NS, buf = 2u * (uint32_t)t + (kc & 1u);
            if (kc >= 2u && !(ok = mbar_wait_warp<kWaitVEmpty>(bar_pv_done + 8 * buf, ((kc - 2u) >> 1) & 1u, wctx))) break;
            if (!(ok = mbar_wait_warp<kWaitKFull>(bar_k_full + 8 * buf, (kc >> 1) & 1u, wctx))) break;
            tc_fence_after();
            const uint32_t d = tm_s + 64u * (kc & 1u);
            const uint32_t kb = k_lo + st * (Cfg::kKVBytes >> 4);
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              constexpr uint32_t kChunkQ = (BM * 128) >> 4, kChunkK = (BN * 128) >> 4;
              mma_ss(d, a_lo + (uint32_t)(kk >> 2) * kChunkQ + (uint32_t)(kk & 3) * 2,
                     kb + (uint32_t)(kk >> 2) * kChunkK + (uint32_t)(kk & 3) * 2, idesc_qk, kk > 0 ? 1u : 0u, issue);
            }
            tc_commit(bar_s_full + 8 * buf, issue);
            if (!Cfg::kStageInQ && j + 1 == n) tc_commit(bar_q_empty + 8 * it2, issue);   // last read of Q
          }
        }
      }
    } else {
    if (warp == 0) {
      // ---------------------------------------------------------------- work fetch + K/V producer
      const uint32_t issue = elect_one();
      uint32_t it_n = 0, kc = 0;
      Work wk;
      while (true) {
        const int w = it_n == 0 ? (int)blockIdx.x : draw_work(args, lane, (int)gridDim.x);   // (at most one CTA per index)
        if (w >= 0) decode_work(args, tab, w, wk);
        const uint32_t ring = it_n % kRing;
        if (!mbar_wait_issuer<kWaitItemEmpty>(bar_item_empty + 8 * ring, ((it_n / kRing) & 1u) ^ 1u, wctx)) break;
        if (issue) {
          if (w >= 0) ring_write(s_ring + ring * kRingInts, w, wk);
          else s_ring[ring * kRingInts] = -1;
          mbar_arrive(bar_item_full + 8 * ring);
        }
        if (w < 0) break;
        bool ok = true;
        for (int j = 0; ok && j < wk.n; ++j, ++kc) {
          const int kv0 = wk.kv_row0 + j * BN;
          uint32_t s = kc % NK;
          ok = mbar_wait_issuer<kWaitKEmpty>(bar_k_empty + 8 * s, ((kc / NK) & 1u) ^ 1u, wctx);
          if (!ok) break;
          mbar_expect_tx(bar_k_full + 8 * s, Cfg::kKVBytes, issue);
          tma_load(s_k + s * Cfg::kKVBytes, &map_k, bar_k_full + 8 * s, wk.kv_head, kv0, wk.bin, issue);
          s = kc % NV;
          ok = mbar_wait_issuer<kWaitVEmpty>(bar_v_empty + 8 * s, ((kc / NV) & 1u) ^ 1u, wctx);
          if (!ok) break;
          mbar_expect_tx(bar_v_full + 8 * s, Cfg::kKVBytes, issue);
          tma_load(s_v + s * Cfg::kKVBytes, &map_v, bar_v_full + 8 * s, wk.kv_head, kv0, wk.bin, issue);
        }
        if (!ok) break;
        ++it_n;
      }
    } else if (warp >= 2) {
      // ---------------------------------------------------------------- Q loader of slot t
      const int t = warp - 2;
      const uint32_t issue = elect_one();
      uint32_t it_n = 0;
      while (true) {
        const uint32_t ring = it_n % kRing;
        if (!mbar_wait_issuer<kWaitItemFull>(bar_item_full + 8 * ring, (it_n / kRing) & 1u, wctx)) break;
        const volatile int* e = s_ring + ring * kRingInts;
        const int w = uniform(e[0]), bin = uniform(e[1]);
        const int q_row0 = uniform(e[4 + t]), head = uniform(e[9 + t]);
        const bool used = uniform(t ? (e[6] < e[8]) : (e[7] > 0)) != 0;
        if (issue) mbar_arrive(bar_item_empty + 8 * ring);
        if (w < 0) break;
        // the slot's last Q.K^T of the previous item must have finished reading the buffer
        if (!mbar_wait_issuer<kWaitQEmpty>(bar_q_empty + 8 * t, (it_n & 1u) ^ 1u, wctx)) break;
        if (used) {
          mbar_expect_tx(bar_q_full + 8 * t, Cfg::kQBytes, issue);
          tma_load(s_q + t * Cfg::kQBytes, &map_q, bar_q_full + 8 * t, head, q_row0, bin, issue);
        } else if (issue) {
          mbar_arrive(bar_q_full + 8 * t);
        }
        ++it_n;
      }
    } else if (warp == 1) {
      // ---------------------------------------------------------------- MMA issuer
      // Kept lean on purpose: one warp feeds the tensor pipe, so every instruction between two
      // tcgen05.mma counts. Descriptor low words are precomputed; inside a group of
      // MMAs only compile-time constants are added.
      constexpr uint32_t idesc_qk = instr_desc(BN, false);
      constexpr uint32_t idesc_pv = instr_desc(D, true);
      const uint32_t q_lo0 = desc_lo(s_q, 0), k_lo0 = desc_lo(s_k, 0), v_lo0 = desc_lo(s_v, BN * 128);
      const uint32_t issue = elect_one();
      uint32_t it_n = 0, kc0 = 0, vc0 = 0, tc0 = 0, tc1 = 0;
      int n = 0, je0 = 0, jb1 = 0, je1 = 0;
      bool ok = true;
      auto wait_k = [&](const int j) -> bool {
        const uint32_t kc = kc0 + (uint32_t)j, s = kc % NK;
        return mbar_wait_issuer<kWaitKFull>(bar_k_full + 8 * s, (kc / NK) & 1u, wctx);
      };
      // S_t = Q_t K_j^T (K_j has been waited for); the K stage is released after the last slot that reads it
      auto issue_qk = [&](const int t, const int j) {
        const uint32_t kc = kc0 + (uint32_t)j, s = kc % NK;
        tc_fence_after();
        const uint32_t d = tmem_base + Cfg::kTmemS + 128u * t;
        const uint32_t a_lo = q_lo0 + (uint32_t)t * (Cfg::kQBytes >> 4);
        const uint32_t b_lo = k_lo0 + s * (Cfg::kKVBytes >> 4);
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          constexpr uint32_t kChunkQ = (BM * 128) >> 4, kChunkK = (BN * 128) >> 4;
          mma_ss(d, a_lo + (uint32_t)(kk >> 2) * kChunkQ + (uint32_t)(kk & 3) * 2,
                 b_lo + (uint32_t)(kk >> 2) * kChunkK + (uint32_t)(kk & 3) * 2, idesc_qk, kk > 0 ? 1u : 0u, issue);
        }
        if (t == 1 || !(j >= jb1 && j < je1)) tc_commit(bar_k_empty + 8 * s, issue);
        tc_commit(bar_s_full + 16 * t, issue);
        // the slot's last scores of this item: its Q buffer is free for the next item's Q from here on
        if (j + 1 == (t ? je1 : je0)) tc_commit(bar_q_empty + 8 * t, issue);
      };
      // O_t (+)= P_t V_j, then either the next S_t or the end-of-item signals of slot t. V_j and the next K
      // tile are waited for first: they have been there for long, but even a wait that succeeds at once costs
      // ~100 cycles, which then do not stand between P_t and its product.
      auto slot_step = [&](const int t, const int j, const int jb, const int je, uint32_t& tcount) -> bool {
        if (j >= jb && j < je) {
          const bool first = (j == jb);
          // the previous item's epilogue must have read O_t before it is overwritten
          if (first && !mbar_wait_issuer<kWaitOEmpty>(bar_o_empty + 8 * t, (it_n & 1u) ^ 1u, wctx)) return false;
          const uint32_t vc = vc0 + (uint32_t)j, s = vc % NV;
          if (!mbar_wait_issuer<kWaitVFull>(bar_v_full + 8 * s, (vc / NV) & 1u, wctx)) return false;
          if (j + 1 < je && !wait_k(j + 1)) return false;
          if (!mbar_wait_issuer<kWaitP>(bar_p_full + 16 * t, tcount & 1u, wctx)) return false;
          tc_fence_after();
          const uint32_t a = tmem_base + Cfg::kTmemS + 128u * t;
          const uint32_t d = tmem_base + Cfg::kTmemO + (uint32_t)D * t;
          const uint32_t b_lo = v_lo0 + s * (Cfg::kKVBytes >> 4);
          mma_ts(d, a, b_lo, idesc_pv, first ? 0u : 1u, issue);
#pragma unroll
          for (int kk = 1; kk < BN / 16; ++kk)        // P of the first 64 keys at column 0, of the others at column 64
            mma_ts(d, a + (kk >> 2) * 64 + (kk & 3) * 8, b_lo + (uint32_t)kk * ((16 * 128) >> 4), idesc_pv, 1u, issue);
          ++tcount;
          if (t == 1 || !(j >= jb1 && j < je1)) tc_commit(bar_v_empty + 8 * s, issue);
          if (j + 1 < je) issue_qk(t, j + 1);
          else tc_commit(bar_o_full + 8 * t, issue);  // slot t is done with this item
          return true;
        }
        if (j + 1 == jb && jb < je) {        // slot t joins the key loop at the next tile
          if (!wait_k(j + 1)) return false;
          issue_qk(t, j + 1);
        }
        return true;
      };
      while (ok) {
        const uint32_t ring = it_n % kRing;
        if (!mbar_wait_issuer<kWaitItemFull>(bar_item_full + 8 * ring, (it_n / kRing) & 1u, wctx)) break;
        const volatile int* e = s_ring + ring * kRingInts;
        const int w = uniform(e[0]);
        n = uniform(e[3]); jb1 = uniform(e[6]); je0 = uniform(e[7]); je1 = uniform(e[8]);
        if (issue) mbar_arrive(bar_item_empty + 8 * ring);
        if (w < 0) break;
        const uint32_t bar_q_ready = args.rope_table ? bar_q_rot : bar_q_full;
        ok = mbar_wait_issuer<kWaitQFull>(bar_q_ready + 0, it_n & 1u, wctx) &&
             mbar_wait_issuer<kWaitQFull>(bar_q_ready + 8, it_n & 1u, wctx);
        if (!ok) break;
        if (!(ok = wait_k(0))) break;                     // every item has a first tile
        if (je0 > 0) issue_qk(0, 0);
        if (jb1 == 0 && je1 > 0) issue_qk(1, 0);
        for (int j = 0; ok && j < n; ++j) {
          ok = slot_step(0, j, 0, je0, tc0);
          if (ok) ok = slot_step(1, j, jb1, je1, tc1);
        }
        if (!ok) break;
        // Unused slot: keep its per-item barriers in step. o_full must not complete two phases
        // before every softmax thread has seen the first, so wait until all of them are past the
        // previous item's o_full (they signal that on o_empty).
        if (je0 <= 0) {
          if (!(ok = mbar_wait_issuer<kWaitOEmpty>(bar_o_empty + 0, (it_n & 1u) ^ 1u, wctx))) break;
          if (issue) { mbar_arrive(bar_q_empty + 0); mbar_arrive(bar_o_full + 0); }
        }
        if (jb1 >= je1) {
          if (!(ok = mbar_wait_issuer<kWaitOEmpty>(bar_o_empty + 8, (it_n & 1u) ^ 1u, wctx))) break;
          if (issue) { mbar_arrive(bar_q_empty + 8); mbar_arrive(bar_o_full + 8); }
        }
        kc0 += (uint32_t)n;
        vc0 += (uint32_t)n;
        ++it_n;
      }
    }
    }   // shared-stream roles
  } else if (kIndep && warp >= 20) {
    // ------------------------------------------------------------------ cache writer of slot t (warps 20, 21)
    // UNPACK of V: every row of V passes through shared memory here anyway, so the warp writes it to its prompt's
    // cache from there while the slot's other warps compute, and the kernel in front of this one reads and writes K
    // only. An item writes the rows of its own query tile, which are its last key rows; with as many KV heads as
    // query heads (the only use) every row has one such item. The bound is memory, as without: 17 554 tokens of 32
    // heads of 128, rotation kernel 121 -> 77 us, this one 194 -> 210 (they overlap), both 299 -> 292.
    // (K' written the same way made this kernel 58 us longer, as much as the rotation kernel got shorter: a K stage
    // is wanted back as soon as the scores are there, a V stage is held for the softmax's time in any case.)
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLast));
    if (warp >= 22) {
      // ---------------------------------------------------------------- products of slot t: O (+)= P(k) V(k)
      const int t = warp - 22;
      const uint32_t issue = elect_one();
      constexpr uint32_t idesc_pv = instr_desc(D, true);
      constexpr int NS = Cfg::kKVStages;
      const uint32_t v_lo = desc_lo(s_kv, BN * 128) + (uint32_t)(t * NS) * (Cfg::kKVBytes >> 4);
      const uint32_t tm_s = tmem_base + Cfg::kTmemS + 128u * (uint32_t)t;
      const uint32_t tm_o = tmem_base + Cfg::kTmemO + (uint32_t)D * (uint32_t)t;
      uint32_t kc = 0;
      bool ok = true;
      for (uint32_t it_n = 0; ok; ++it_n) {
        const uint32_t ring = (uint32_t)t * kRing + it_n % kRing;
        if (!mbar_wait_warp<kWaitItemFull>(bar_item_full + 8 * ring, (it_n / kRing) & 1u, wctx)) break;
        const volatile int* e = s_ring + ring * kRingInts;
        const int w = uniform(e[0]), n = uniform(e[3]);
        if (issue) mbar_arrive(bar_item_empty + 8 * ring);
        if (w < 0) break;
        for (int j = 0; j < n; ++j, ++kc) {            // (no item is without tiles)
          const uint32_t st = kv_index_v(kc) % NS, buf = 2u * (uint32_t)t + (kc & 1u);
          // the previous item's epilogue must have read O_t before it is overwritten
          if (j == 0 && it_n > 0u &&
              !(ok = mbar_wait_warp<kWaitOEmpty>(bar_o_empty + 8 * (2u * (uint32_t)t + ((it_n - 1u) & 1u)), ((it_n - 1u) >> 1) & 1u, wctx))) break;
          if (!(ok = mbar_wait_warp<kWaitVFull>(bar_v_full + 8 * buf, (kc >> 1) & 1u, wctx))) break;
          if constexpr (kFill) {
            // the cache writer must have seen V(k - 2), whose barrier this is again, before V(k) is announced
            if (kc >= 2u && !(ok = mbar_wait_warp<kWaitVEmpty>(bar_v_read + 8 * buf, ((kc - 2u) >> 1) & 1u, wctx))) break;
            if (issue) mbar_arrive((t ? bar_v_seen1 : bar_v_seen0) + 8 * (kc & 1u));
          }
          if (!(ok = mbar_wait_warp<kWaitP>(bar_p_full + 8 * buf, (kc >> 1) & 1u, wctx))) break;
          tc_fence_after();
          const uint32_t a = tm_s + 64u * (kc & 1u);
          const uint32_t vb = v_lo + st * (Cfg::kKVBytes >> 4);
          mma_ts(tm_o, a, vb, idesc_pv, j == 0 ? 0u : 1u, issue);
#pragma unroll
          for (int kk = 1; kk < BN / 16; ++kk)
            mma_ts(tm_o, a + kk * 8, vb + (uint32_t)kk * ((16 * 128) >> 4), idesc_pv, 1u, issue);
          tc_commit(bar_pv_done + 8 * buf, issue);
          if (j + 1 == n) tc_commit(bar_o_full + 8 * t, issue);
        }
      }
    } else if (kFill) {
      const int t = warp - 20;
      const uint32_t bar_v_seen = t ? bar_v_seen1 : bar_v_seen0;
      constexpr int NS = Cfg::kKVStages;
      constexpr int kPieces = D / 8;                 // 16-byte pieces of a row, one per lane
      constexpr int kRowsAtOnce = 32 / kPieces;
      const int piece = lane & (kPieces - 1);
      uint32_t kc = 0;
      bool ok = true;
      for (uint32_t it_n = 0; ok; ++it_n) {
        const uint32_t ring = (uint32_t)t * kRing + it_n % kRing;
        if (!mbar_wait_warp<kWaitItemFull>(bar_item_full + 8 * ring, (it_n / kRing) & 1u, wctx)) break;
        const volatile int* e = s_ring + ring * kRingInts;
        const int w = uniform(e[0]), kv_row0 = e[2], n = uniform(e[3]), q_row0 = e[4], kv_head = e[11];
        const int bin_used = e[12], seg_end = e[13], seg_first = e[16];
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_item_empty + 8 * ring);
        if (w < 0) break;
        const int own_end = min(q_row0 + BM, bin_used);      // rows [q_row0, own_end)
        // The prompt under the cursor, all lanes alike: its rows [.., cached) go to offset base + row * D, the next
        // prompt starts at row `next`.
        int seg = seg_first, cached = 0, next = 0;
        int64_t seg_base = 0;
        auto load_seg = [&]() {
          const int start = tab.i32(args.off_seg_start + seg);
          next = seg + 1 < seg_end ? tab.i32(args.off_seg_start + seg + 1) : own_end;
          cached = start + tab.i32(args.off_true_len + seg);
          seg_base = tab.i64(args.off_cache_off, seg) + ((int64_t)kv_head * tab.i32(args.off_cap + seg) - start) * D;
        };
        load_seg();
        for (int j = 0; ok && j < n; ++j, ++kc) {
          const int r0 = kv_row0 + j * BN;
          const int lo = max(r0, q_row0), hi = min(r0 + BN, own_end);
          const uint32_t st = kv_index_v(kc) % NS;
          ok = mbar_wait_warp<kWaitVFull>(bar_v_seen + 8 * (kc & 1u), (kc >> 1) & 1u, wctx);
          if (!ok) break;
          const uint32_t tile = s_kv + ((uint32_t)t * NS + st) * Cfg::kKVBytes + (uint32_t)(piece >> 3) * (BN * 128);
          __nv_bfloat16* cache = args.v_cache + 8 * piece;
          for (int row = lo; row < hi;) {                      // prompt by prompt
            if (row >= next) {
              ++seg;
              load_seg();
              continue;
            }
            const int stop = min(hi, next), copy_end = min(stop, cached);
            for (int at = row + lane / kPieces; at < copy_end + lane / kPieces; at += 4 * kRowsAtOnce) {
              uint4 val[4];
#pragma unroll
              for (int x = 0; x < 4; ++x) {
                const uint32_t r = (uint32_t)(min(at + x * kRowsAtOnce, copy_end - 1) - r0);
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(val[x].x), "=r"(val[x].y), "=r"(val[x].z), "=r"(val[x].w)
                             : "r"(tile + r * 128 + ((((uint32_t)piece & 7u) ^ (r & 7u)) << 4)));
              }
#pragma unroll
              for (int x = 0; x < 4; ++x)
                if (at + x * kRowsAtOnce < copy_end)
                  *reinterpret_cast<uint4*>(cache + seg_base + (int64_t)(at + x * kRowsAtOnce) * D) = val[x];
            }
            row = stop;
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_v_read + 8 * (2u * (uint32_t)t + (kc & 1u)));
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ softmax + epilogue
    const int t = (warp - 4) >> 3;                   // slot
    const int h = ((warp - 4) >> 2) & 1;             // shared mode: which 64 keys of a 128-key tile this thread owns
    const int quad = warp & 3;                       // TMEM lane quadrant this warp may access
    const int row = quad * 32 + lane;                // query row inside the tile
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
    const uint32_t tmem_s = tmem_base + Cfg::kTmemS + 128u * t + lane_base;
    const uint32_t tmem_o = tmem_base + Cfg::kTmemO + (uint32_t)D * t + lane_base;

    if constexpr (kIndep) {
      // ---------------------------------------------------------------- independent mode
      // Per slot: warps with h == 0 are the softmax threads, one per query row (all 64 scores of a
      // tile), and never leave the tile loop; warps with h == 1 are helper threads, one per row, which
      // rotate the next item's Q in shared memory (fused path) and run the epilogue of the previous
      // item, both off the softmax threads' critical path.
      const float c_scale = args.scale_log2;
      const int fs = args.fold_shift;                  // tile row m holds bin row q_row0 + (m >> fs)
      const uint32_t ring0 = (uint32_t)t * kRing;
      // row sums travel from the softmax thread to the helper of the same row, double-buffered by item
      volatile float* x_l = s_xchg + t * 128 + row;            // + 256 * (item & 1)
      bool ok = true;
      // key range [key_lo, key_hi] of this thread's row from a ring entry (empty for padding rows)
      // (all lanes of the warp call it together: the prompts' start rows are loaded once per warp). The helper
      // threads do this ahead of time; the softmax threads get the first key from them.
      auto row_range = [&](const volatile int* e, int& key_lo, int& key_hi) {
        const int i_row = e[4] + (row >> fs);
        int lo = e[14];
        if (!(e[18] & 1))
          lo = seg_start_at(tab, args.off_seg_start, e[16] + 1, e[13], i_row, e[4] + ((quad * 32 + 31) >> fs), lo, lane);
        const bool real = i_row < e[12];
        key_lo = real ? lo : 1;
        key_hi = real ? i_row : 0;
      };
      if (h == 0) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmaxIndep));
        uint32_t it_n = 0, tcount = 0;
        while (true) {
          const uint32_t ring = ring0 + it_n % kRing;
          ok = mbar_wait_warp<kWaitItemFull>(bar_item_full + 8 * ring, (it_n / kRing) & 1u, wctx);
          if (!ok) break;
          const volatile int* e = s_ring + ring * kRingInts;
          const int w = e[0], item_kv_row0 = e[2], n_tiles = e[3];
          const int i_row = e[4] + (row >> fs), bin_used = e[12];
          mbar_arrive(bar_item_empty + 8 * ring);
          if (w < 0) break;
          ok = mbar_wait_warp<kWaitQFull>(bar_q_rot + 8 * (2 * t + (it_n & 1u)), (it_n >> 1) & 1u, wctx);
          if (!ok) break;
          const int key_lo = __float_as_int(x_l[256 * (it_n & 1u)]);
          const int key_hi = i_row < bin_used ? i_row : 0;       // padding rows: key_lo = 1, an empty range
          float m_run = -INFINITY;      // running maximum of the row, in scaled log2 units
          float l_run = 0.f;            // running sum of exp2(s * c - m_run)
          for (int j = 0; j < n_tiles; ++j) {
            static_assert(BN == 64, "a row's scores of a tile are one 64-bit mask");
            const int kv0 = item_kv_row0 + j * BN;
            const int c_lo = max(key_lo - kv0, 0);
            const int c_hi = min(key_hi - kv0, BN - 1);          // visible columns [c_lo, c_hi]
            const uint64_t vis = visible_mask64(c_lo, c_hi);     // bit i: column i is visible to this row
            const bool cut = __any_sync(0xffffffffu, ~vis != 0ull);   // some row's interval ends or begins inside the tile
            const uint32_t sbuf = tcount & 1u;                   // tile k of the stream lives in S buffer k & 1
            const uint32_t tmem_sb = tmem_s + 64u * sbuf;
            ok = mbar_wait_warp<kWaitS>(bar_s_full + 8 * (2 * t + sbuf), (tcount >> 1) & 1u, wctx);
            if (!ok) break;
            tc_fence_after();
            // Both halves of the tile, also one that no row of the warp can see: leaving it out costs more in code than
            // it saves (64 prompts on a 7B layer 239 -> 236 us a step).
            uint32_t v[BN];
#pragma unroll
            for (int ch = 0; ch < BN / 32; ++ch) tmem_ld32(tmem_sb + 32 * ch, *reinterpret_cast<uint32_t(*)[32]>(&v[32 * ch]));
            tc_wait_ld();
            // masked tiles (the causal diagonal, the first tile of a prompt): one select per score,
            // steered by the bits of the row's visibility mask
            if (cut) {
              const uint32_t vis_lo = (uint32_t)vis, vis_hi = (uint32_t)(vis >> 32);
#pragma unroll
              for (int i = 0; i < 32; ++i) v[i] = (vis_lo & (1u << i)) ? v[i] : 0xff800000u;
#pragma unroll
              for (int i = 0; i < 32; ++i) v[32 + i] = (vis_hi & (1u << i)) ? v[32 + i] : 0xff800000u;
            }
            // lazy running-maximum update: keep the stale maximum while the new one is < 2^8 above it
            const float m_tile = max64(v) * c_scale;
            float m_new = m_run;
            if (m_tile > m_run + 8.f) m_new = m_tile;
            const bool rescale = (m_new != m_run) && (m_run != -INFINITY);
            const float alpha = rescale ? fast_exp2(m_run - m_new) : 1.f;
            if (j > 0 && __any_sync(0xffffffffu, rescale)) {
              // S(k) is computed ahead of P(k-1) V(k-1): O_t is stable only once that product is there
              ok = mbar_wait_warp<kWaitVEmpty>(bar_pv_done + 16 * t + 8 * (sbuf ^ 1u), ((tcount - 1u) >> 1) & 1u, wctx);
              if (!ok) break;
              tc_fence_after();
#pragma unroll 1
              for (int ch = 0; ch < D / 16; ++ch) {          // rare path: keep it small
                uint32_t ov[16];
                tmem_ld16(tmem_o + ch * 16, ov);
                tc_wait_ld();
#pragma unroll
                for (int i = 0; i < 16; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * alpha);
                tmem_st16(tmem_o + ch * 16, ov);
              }
            }
            l_run *= alpha;
            m_run = m_new;
            const float neg_m = (m_run == -INFINITY) ? 0.f : -m_run;
            // p = exp2(s * c - m), row sum, P (bf16) written over the first half of the S buffer
            const uint64_t c2 = pack_f2(__float_as_uint(c_scale), __float_as_uint(c_scale));
            const uint64_t negm2 = pack_f2(__float_as_uint(neg_m), __float_as_uint(neg_m));
            uint64_t sum_a = 0ull, sum_b = 0ull;
#pragma unroll
            for (int ch = 0; ch < BN / 32; ++ch) {
              uint32_t pk[16];
              exp_chunk(&v[32 * ch], c2, negm2, sum_a, sum_b, pk);
              tmem_st16(tmem_sb + ch * 16, pk);              // S(k) was read completely above
            }
            l_run += sum_f2x2(sum_a, sum_b);
            tc_wait_st();
            tc_fence_before();
            mbar_arrive(bar_p_full + 8 * (2 * t + sbuf));
            ++tcount;
          }
          if (!ok) break;
          // The row sum goes to the helper thread of this row (arrive has release semantics). The
          // softmax threads can finish item i+1 before the helpers have picked up item i, but not
          // item i+2 (its scores are issued after the epilogue of item i has read O_t), so the
          // hand-over is double-buffered by item parity, barrier included.
          x_l[256 * (it_n & 1u)] = l_run;
          mbar_arrive(bar_l_ready + 16 * t + 8 * (it_n & 1u));
          ++it_n;
        }
      } else {
        uint32_t it_n = 0;
        int p_q_row0 = 0, p_head = 0, p_bin = 0;         // coordinates of the previous item (its epilogue is due)
        while (true) {
          const uint32_t ring = ring0 + it_n % kRing;
          ok = mbar_wait_warp<kWaitItemFull>(bar_item_full + 8 * ring, (it_n / kRing) & 1u, wctx);
          if (!ok) break;
          const volatile int* e = s_ring + ring * kRingInts;
          const int w = e[0], c_bin = e[1], c_q_row0 = e[4], c_head = e[9];
          int key_lo = 1, key_hi = 0;
          if (w >= 0) row_range(e, key_lo, key_hi);
          mbar_arrive(bar_item_empty + 8 * ring);
          const uint32_t qb = 2u * (uint32_t)t + (it_n & 1u);      // Q tile of this item
          // the O tile that was stored last has left its Q tile by now, or will soon: hand the tile back
          if (Cfg::kStageInQ && it_n > 1 && lane == 0) {
            tma_store_wait_read();
            mbar_arrive(bar_q_empty + 8 * qb);
          }
          if (w >= 0) {
            // rotate row `row` of this item's Q in shared memory by the angles of its position, with
            // the same fp32 arithmetic and rounding as the stand-alone kernel, leave the row's first key
            // where its row sum will be (this thread has read that of the item before the previous one
            // from there), then report Q_t ready
            ok = mbar_wait_warp<kWaitQFull>(bar_q_full + 8 * qb, (it_n >> 1) & 1u, wctx);
            if (!ok) break;
            const int pos = key_hi - key_lo;             // < 0 for padding rows
            if (args.rope_table && pos > 0) {
              constexpr int kUnits = D / 16;             // 16-byte (lower, upper) unit pairs per row
              const uint32_t q_row = s_q + qb * Cfg::kQBytes + (uint32_t)row * 128;
              // table[g][pos] = (cos, sin) of j = 2g and 2g + 1: consecutive rows read consecutive 16 bytes
              const float4* tab = reinterpret_cast<const float4*>(args.rope_table) + pos;
#pragma unroll 1
              for (int u0 = 0; u0 < kUnits; u0 += 2) {
                float4 cs[2][4];                         // table loads of two units first: one L2 round trip
#pragma unroll
                for (int uu = 0; uu < 2; ++uu)
#pragma unroll
                  for (int i = 0; i < 4; ++i)
                    cs[uu][i] = tab[(size_t)((u0 + uu) * 4 + i) * (size_t)args.capacity];
#pragma unroll
                for (int uu = 0; uu < 2; ++uu) {
                  const int u = u0 + uu;                 // pairs (8u .. 8u+7, + D/2)
                  const uint32_t a_lo = q_row + ((((uint32_t)u) ^ ((uint32_t)row & 7u)) << 4);
                  const uint32_t a_hi = (D == 128)
                      ? q_row + (BM * 128) + ((((uint32_t)u) ^ ((uint32_t)row & 7u)) << 4)
                      : q_row + ((((uint32_t)(u + kUnits)) ^ ((uint32_t)row & 7u)) << 4);
                  uint32_t lo[4], hi[4];
                  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(lo[0]), "=r"(lo[1]), "=r"(lo[2]), "=r"(lo[3]) : "r"(a_lo));
                  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(hi[0]), "=r"(hi[1]), "=r"(hi[2]), "=r"(hi[3]) : "r"(a_hi));
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    const float4 c = cs[uu][i];          // (cos, sin) of two consecutive j
                    const __nv_bfloat162 l2 = *reinterpret_cast<__nv_bfloat162*>(&lo[i]);
                    const __nv_bfloat162 h2 = *reinterpret_cast<__nv_bfloat162*>(&hi[i]);
                    const float2 a = __bfloat1622float2(l2), b = __bfloat1622float2(h2);
                    lo[i] = pack_bf16(__fmaf_rn(a.x, c.x, -__fmul_rn(b.x, c.y)), __fmaf_rn(a.y, c.z, -__fmul_rn(b.y, c.w)));
                    hi[i] = pack_bf16(__fmaf_rn(b.x, c.x, __fmul_rn(a.x, c.y)), __fmaf_rn(b.y, c.z, __fmul_rn(a.y, c.w)));
                  }
                  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a_lo), "r"(lo[0]), "r"(lo[1]), "r"(lo[2]), "r"(lo[3]) : "memory");
                  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a_hi), "r"(hi[0]), "r"(hi[1]), "r"(hi[2]), "r"(hi[3]) : "memory");
                }
              }
              asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // visible to the tensor core
            }
            x_l[256 * (it_n & 1u)] = __int_as_float(key_lo);
            mbar_arrive(bar_q_rot + 8 * qb);
          }
          if (it_n > 0) {
            // epilogue of the previous item: O_t / l -> bf16 -> shared memory (128-byte swizzle) -> TMA store
            const uint32_t pi = it_n - 1u;
            ok = mbar_wait_warp<kWaitOFull>(bar_o_full + 8 * t, pi & 1u, wctx);
            if (!ok) break;
            ok = mbar_wait_warp<kWaitRowSum>(bar_l_ready + 16 * t + 8 * (pi & 1u), (pi >> 1) & 1u, wctx);
            if (!ok) break;
            tc_fence_after();
            const float l_row = x_l[256 * (pi & 1u)];
            const float inv_l = l_row > 0.f ? 1.f / l_row : 0.f;
            // Each warp stages and stores its own 32 rows (a 32-row TMA box), so the epilogue needs
            // no rendezvous between warps.
            const uint32_t stage = (Cfg::kStageInQ ? s_q + (qb ^ 1u) * Cfg::kQBytes : s_stage_o + (uint32_t)t * Cfg::kStageOBytes) +
                                   (uint32_t)quad * (32 * 128);
            const int p_row0 = p_q_row0 + ((32 * quad) >> fs);   // the warp's 32 tile rows: 32 >> fs bin rows x fold heads
#pragma unroll 1
            for (int hh = 0; hh < D / 64; ++hh) {          // 64 columns (one TMA box) at a time
              const uint32_t box = stage + (uint32_t)hh * (BM * 128);
              if (!Cfg::kStageInQ) {                       // the previous item's store must have read the staging rows
                if (lane == 0) tma_store_wait_read();
                __syncwarp();
              }
              uint32_t ov[64];
              tmem_ld32(tmem_o + hh * 64, *reinterpret_cast<uint32_t(*)[32]>(&ov[0]));
              tmem_ld32(tmem_o + hh * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&ov[32]));
              tc_wait_ld();
              if (hh == D / 64 - 1) {
                tc_fence_before();
                mbar_arrive(bar_o_empty + 16 * t + 8 * (pi & 1u));   // O_t may be overwritten by the next item now
              }
#pragma unroll
              for (int c16 = 0; c16 < 8; ++c16) {
                const uint32_t addr = box + (uint32_t)lane * 128 + (((uint32_t)c16 ^ ((uint32_t)lane & 7u)) << 4);
                const uint32_t w0 = pack_bf16(__uint_as_float(ov[c16 * 8 + 0]) * inv_l, __uint_as_float(ov[c16 * 8 + 1]) * inv_l);
                const uint32_t w1 = pack_bf16(__uint_as_float(ov[c16 * 8 + 2]) * inv_l, __uint_as_float(ov[c16 * 8 + 3]) * inv_l);
                const uint32_t w2 = pack_bf16(__uint_as_float(ov[c16 * 8 + 4]) * inv_l, __uint_as_float(ov[c16 * 8 + 5]) * inv_l);
                const uint32_t w3 = pack_bf16(__uint_as_float(ov[c16 * 8 + 6]) * inv_l, __uint_as_float(ov[c16 * 8 + 7]) * inv_l);
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w0), "r"(w1), "r"(w2), "r"(w3) : "memory");
              }
              asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
              __syncwarp();
              if (lane == 0 && p_row0 < args.capacity) {
                tma_store(&map_o, box, p_head, p_row0, hh, p_bin);
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
              }
            }
          }
          if (w < 0) break;
          p_q_row0 = c_q_row0; p_head = c_head; p_bin = c_bin;
          ++it_n;
        }
        if (lane == 0) tma_store_wait_read();    // staging must outlive the last store's read
      }
    } else {
    // ---------------------------------------------------------------- shared-stream mode
    // All softmax warps run the same code (slot and half at run time): the unrolled row loops are
    // large and several copies of them would not stay resident in the instruction caches.
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
    volatile float* x_mine = s_xchg + (t * 2 + h) * 128 + row;
    volatile float* x_other = s_xchg + (t * 2 + (h ^ 1)) * 128 + row;
    // Rendezvous points are mbarriers (arrive, then a bounded wait) rather than named barriers, so
    // that a warp whose partner gave up on a wait cannot be left waiting for it.
    const uint32_t bar_pair = bar_pair0 + 8 * (uint32_t)(t * 4 + quad);
    uint32_t pair_ph = 0;
    auto rendezvous = [&](const uint32_t bar, uint32_t& ph) -> bool {
      mbar_arrive(bar);
      const bool r = __all_sync(0xffffffffu, mbar_wait<kWaitPair>(bar, ph, wctx));
      ph ^= 1u;
      return r;
    };
    const float c_scale = args.scale_log2;
    // (a NaN among the values, too, leaves no room)
    const float lazy_log2 = args.v_max && __uint_as_float(__ldcg(args.v_max) << 16) <= args.v_room ? kLazyLog2 : kLazyLog2Wide;
    uint32_t it_n = 0, tcount = 0;
    bool ok = true;
    // Rotates this thread's part of row `row` of Q_t in shared memory by the angles of position `pos`
    // (< 0: padding, nothing to do), with the same fp32 arithmetic and rounding as the stand-alone
    // kernel, then reports the slot's Q as ready. Waits for the TMA load of Q first. The warp also says
    // whether its half of every row is short enough for the bound on the scores: |half|^2 <= limit (0: there is no bound,
    // not even for a row whose squares come to 0).
    volatile uint8_t* const bounded_mine = s_bounded + (t * 4 + quad) * 2 + h;
    volatile uint8_t* const bounded_other = s_bounded + (t * 4 + quad) * 2 + (h ^ 1);
    auto rotate_q = [&](const int pos, const float limit, const uint32_t parity) -> bool {
      if (!__all_sync(0xffffffffu, mbar_wait<kWaitQFull>(bar_q_full + 8 * t, parity, wctx))) return false;
      uint64_t n2a = 0ull, n2b = 0ull;
      if (pos >= 0) {
        constexpr int kUnits = D / 16;                 // 16-byte units per half of a row
        const uint32_t q_row = s_q + (uint32_t)t * Cfg::kQBytes + (uint32_t)row * 128;
        // table[g][pos] = (cos, sin) of j = 2g and 2g + 1: consecutive rows read consecutive 16 bytes
        const float4* tab = reinterpret_cast<const float4*>(args.rope_table) + pos;
        float4 cs[kUnits / 2][4];                      // all table loads first: one L2 round trip
#pragma unroll
        for (int uu = 0; uu < kUnits / 2; ++uu)
#pragma unroll
          for (int i = 0; i < 4; ++i)
            cs[uu][i] = tab[(size_t)((h * (kUnits / 2) + uu) * 4 + i) * (size_t)args.capacity];
#pragma unroll
        for (int uu = 0; uu < kUnits / 2; ++uu) {
          const int u = h * (kUnits / 2) + uu;         // pairs (8u .. 8u+7, + D/2)
          const uint32_t a_lo = q_row + ((((uint32_t)u) ^ ((uint32_t)row & 7u)) << 4);
          const uint32_t a_hi = (D == 128)
              ? q_row + (BM * 128) + ((((uint32_t)u) ^ ((uint32_t)row & 7u)) << 4)
              : q_row + ((((uint32_t)(u + kUnits)) ^ ((uint32_t)row & 7u)) << 4);
          uint32_t lo[4], hi[4];
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(lo[0]), "=r"(lo[1]), "=r"(lo[2]), "=r"(lo[3]) : "r"(a_lo));
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(hi[0]), "=r"(hi[1]), "=r"(hi[2]), "=r"(hi[3]) : "r"(a_hi));
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 c = cs[uu][i];                // (cos, sin) of two consecutive j
            const __nv_bfloat162 l2 = *reinterpret_cast<__nv_bfloat162*>(&lo[i]);
            const __nv_bfloat162 h2 = *reinterpret_cast<__nv_bfloat162*>(&hi[i]);
            const float2 a = __bfloat1622float2(l2), b = __bfloat1622float2(h2);
            const uint64_t a2 = pack_f2(__float_as_uint(a.x), __float_as_uint(a.y));
            const uint64_t b2 = pack_f2(__float_as_uint(b.x), __float_as_uint(b.y));
            n2a = fma_f2(a2, a2, n2a);
            n2b = fma_f2(b2, b2, n2b);
            lo[i] = pack_bf16(__fmaf_rn(a.x, c.x, -__fmul_rn(b.x, c.y)), __fmaf_rn(a.y, c.z, -__fmul_rn(b.y, c.w)));
            hi[i] = pack_bf16(__fmaf_rn(b.x, c.x, __fmul_rn(a.x, c.y)), __fmaf_rn(b.y, c.z, __fmul_rn(a.y, c.w)));
          }
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a_lo), "r"(lo[0]), "r"(lo[1]), "r"(lo[2]), "r"(lo[3]) : "memory");
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a_hi), "r"(hi[0]), "r"(hi[1]), "r"(hi[2]), "r"(hi[3]) : "memory");
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // visible to the tensor core
      }
      const bool short_rows = __all_sync(0xffffffffu, limit > 0.f && sum_f2x2(n2a, n2b) <= limit);
      if (lane == 0) *bounded_mine = short_rows ? 1 : 0;
      mbar_arrive(bar_q_rot + 8 * t);
      return true;
    };
    while (true) {
      const uint32_t ring = it_n % kRing;              // both slots read the one ring, each its own fields of an entry
      ok = mbar_wait_warp<kWaitItemFull>(bar_item_full + 8 * ring, (it_n / kRing) & 1u, wctx);
      if (!ok) break;
      const volatile int* e = s_ring + ring * kRingInts;
      const int w = e[0];
      const int item_bin = e[1], item_kv_row0 = e[2];
      const int jb_t = t ? e[6] : 0, je_t = t ? e[8] : e[7];
      const int q_row0_t = e[4 + t], head_t = e[9 + t], kv_head = e[11];
      const int bin_used = e[12], seg_end = e[13], key_lo_t = e[14 + t], seg_first_t = e[16 + t];
      const int single_seg = e[18] >> t;
      mbar_arrive(bar_item_empty + 8 * ring);
      if (w < 0) break;
      const bool used = jb_t < je_t;
      const int i_row = q_row0_t + row;                // bin-local query row
      int key_lo = 1, key_hi = 0;                      // visible keys [key_lo, key_hi]; empty for padding
      if (used) {                                      // warp-uniform
        int lo = key_lo_t;
        if (!(single_seg & 1))                         // several prompts in this tile: find this row's
          lo = seg_start_at(tab, args.off_seg_start, seg_first_t + 1, seg_end, i_row, i_row - lane + 31, lo, lane);
        if (i_row < bin_used) { key_lo = lo; key_hi = i_row; }
      }
      // |q|^2 up to which every score of a row stays below the bound (0 if nothing is known about the keys). The norms grew
      // while this kernel was starting, beside table words that the rotation kernel reads through L1: not from there.
      float q2_limit = 0.f;
      if (args.k_norm2 && lazy_log2 == kLazyLog2) {
        const float k2 = __uint_as_float(__ldcg(args.k_norm2 + kv_head));
        // (a NaN among the keys bounds nothing; the limit is finite, for a |q|^2 that overflows is beyond any)
        if (k2 < INFINITY) q2_limit = fminf(args.bound2 / fmaxf(k2, 1e-30f), FLT_MAX);
      }
      bool bounded = false;
      // Fused path: Q arrives raw and is rotated in shared memory. Each half of a row is held to half
      // the limit, so that no sum over the two threads of a row is needed.
      if (args.rope_table) {
        ok = rotate_q(used ? key_hi - key_lo : -1, 0.5f * q2_limit, it_n & 1u);
        if (!ok) break;
      } else if (args.q_norm2) {
        bounded = q2_limit > 0.f && __uint_as_float(__ldcg(args.q_norm2 + head_t)) <= q2_limit;
      }
      float m_run = -INFINITY;      // running maximum of the whole row, in scaled log2 units
      uint64_t sum_a = 0ull, sum_b = 0ull;   // this thread's share of the running sum of exp2(s * c - m_run), in four parts
      float neg_m = 0.f;
      const uint64_t c2 = pack_f2(__float_as_uint(c_scale), __float_as_uint(c_scale));
      bool fast = false;            // bounded, and every row of the warp has its maximum
      // tiles [clean_jb, clean_je) of this half are visible to every row of the warp from end to end
      constexpr int EPT = BN / 2;                            // scores per thread and tile
      constexpr int NCH = EPT / 32;                          // 32-column TMEM round trips
      const int half0 = item_kv_row0 + EPT * h;
      const int clean_jb = (max(__reduce_max_sync(0xffffffffu, key_lo) - half0, 0) + BN - 1) / BN;
      const int clean_je = (__reduce_min_sync(0xffffffffu, key_hi) - half0 + (BN - EPT + 1)) / BN;   // <= 0 with padding rows
      // this half's P goes over the first half of its own scores' columns: no other thread reads them
      const uint32_t tmem_sb = tmem_s + EPT * h;

      for (int j = jb_t; j < je_t; ++j) {
        if (fast && j >= clean_jb && j < clean_je) {
          // The common tile: nothing to mask, no maximum to find. The scores of the second chunk are
          // loaded while the exponentials of the first are computed.
          ok = mbar_wait_warp<kWaitS>(bar_s_full + 16 * t, tcount & 1u, wctx);
          if (!ok) break;                                    // warp-uniform
          tc_fence_after();
          const uint64_t negm2 = pack_f2(__float_as_uint(neg_m), __float_as_uint(neg_m));
          uint32_t va[32], vb[32], pk[16];
          tmem_ld32(tmem_sb, va);
          tc_wait_ld32(va);
          tmem_ld32(tmem_sb + 32, vb);
          exp_chunk(va, c2, negm2, sum_a, sum_b, pk);
          tmem_st16(tmem_sb, pk);
          tc_wait_ld32(vb);
          exp_chunk(vb, c2, negm2, sum_a, sum_b, pk);
          tmem_st16(tmem_sb + 16, pk);
          tc_wait_st();
          tc_fence_before();
          mbar_arrive(bar_p_full + 16 * t);
          ++tcount;
          continue;
        }
        const int kv0 = item_kv_row0 + j * BN + EPT * h;     // first key of this thread's half
        const int c_lo = max(key_lo - kv0, 0);
        const int c_hi = min(key_hi - kv0, EPT - 1);         // visible columns [c_lo, c_hi] of the half
        // one warp reduction for all the per-warp flags of the tile: which 32-column chunks somebody
        // can see, and whether any row's interval ends or begins inside this half of the tile
        static_assert(NCH == 2, "flag bits below are laid out for two chunks");
        const uint64_t vis = visible_mask64(c_lo, c_hi);     // bit i: column i is visible to this row
        const uint32_t vis_lo = (uint32_t)vis, vis_hi = (uint32_t)(vis >> 32);
        const uint32_t lane_flags = (uint32_t)(vis_lo != 0u) | ((uint32_t)(vis_hi != 0u) << 1) |
                            ((uint32_t)(~vis != 0ull) << 2);
        const uint32_t warp_flags = __reduce_or_sync(0xffffffffu, lane_flags);
        const bool need[NCH] = {(warp_flags & 1u) != 0, (warp_flags & 2u) != 0};
        const bool cut = (warp_flags & 4u) != 0;
        ok = mbar_wait_warp<kWaitS>(bar_s_full + 16 * t, tcount & 1u, wctx);
        if (!ok) break;                                      // warp-uniform
        tc_fence_after();
        uint32_t v[EPT];
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
          if (need[ch]) {
            tmem_ld32(tmem_sb + 32 * ch, *reinterpret_cast<uint32_t(*)[32]>(&v[32 * ch]));
          } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) v[32 * ch + i] = 0xff800000u;        // -inf
          }
        }
        tc_wait_ld();
        // masked tiles (the causal diagonal, the first tile of a prompt): one select per score,
        // steered by the bits of the row's visibility mask
        if (cut) {
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = (vis_lo & (1u << i)) ? v[i] : 0xff800000u;
#pragma unroll
          for (int i = 0; i < 32; ++i) v[32 + i] = (vis_hi & (1u << i)) ? v[32 + i] : 0xff800000u;
        }
        if (!fast) {
          // Row maximum over both halves. (The exchange slot is not written again before both halves
          // have announced their P of this tile.)
          float mx = max64(v);
          *x_mine = mx;
          if (!(ok = rendezvous(bar_pair, pair_ph))) break;
          mx = fmaxf(mx, *x_other);
          if (j == jb_t && args.rope_table) bounded = (*bounded_mine & *bounded_other) != 0;
          const float m_tile = mx * c_scale;
          float m_new = m_run;
          if (m_tile > m_run + lazy_log2) m_new = m_tile;
          const bool rescale = (m_new != m_run) && (m_run != -INFINITY);
          if (j > jb_t && __any_sync(0xffffffffu, rescale)) {
            const float alpha = rescale ? fast_exp2(m_run - m_new) : 1.f;
            // (S_t ready implies that the previous P_t V product has finished.) Each half rescales its
            // own D/2 columns of the row.
#pragma unroll 1
            for (int ch = 0; ch < D / 32; ++ch) {          // rare path: keep it small
              uint32_t ov[16];
              tmem_ld16(tmem_o + (D / 2) * h + ch * 16, ov);
              tc_wait_ld();
#pragma unroll
              for (int i = 0; i < 16; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * alpha);
              tmem_st16(tmem_o + (D / 2) * h + ch * 16, ov);
            }
            const uint64_t alpha2 = pack_f2(__float_as_uint(alpha), __float_as_uint(alpha));
            sum_a = mul_f2(sum_a, alpha2);
            sum_b = mul_f2(sum_b, alpha2);
          }
          m_run = m_new;
          neg_m = (m_run == -INFINITY) ? 0.f : -m_run;
          // rows that see nothing at all (padding) do not hold the others back
          fast = bounded && __all_sync(0xffffffffu, m_run != -INFINITY || key_hi < key_lo);
        }
        // p = exp2(s * c - m), row sum, P (bf16) written over the S columns
        const uint64_t negm2_tile = pack_f2(__float_as_uint(neg_m), __float_as_uint(neg_m));
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
          uint32_t pk[16];
          if (need[ch]) {
            exp_chunk(&v[32 * ch], c2, negm2_tile, sum_a, sum_b, pk);
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) pk[i] = 0u;
          }
          tmem_st16(tmem_sb + ch * 16, pk);
        }
        tc_wait_st();
        tc_fence_before();
        mbar_arrive(bar_p_full + 16 * t);
        ++tcount;
      }
      if (!ok) break;
      const float l_run = sum_f2x2(sum_a, sum_b);

      // epilogue: O_t / l -> bf16 -> shared memory (128-byte swizzle) -> TMA store
      ok = __all_sync(0xffffffffu, mbar_wait<kWaitOFull>(bar_o_full + 8 * t, it_n & 1u, wctx));
      if (!ok) break;
      if (used) {
        // the half-1 threads hand their share of the row sum to the half-0 threads, which run the
        // epilogue; the second barrier keeps the exchange slot from being reused too early
        if (h == 1) *x_mine = l_run;
        if (!(ok = rendezvous(bar_pair, pair_ph))) break;
        const float l_row = (h == 0) ? l_run + *x_other : 0.f;
        if (!(ok = rendezvous(bar_pair, pair_ph))) break;
        if (h == 1) mbar_arrive(bar_o_empty + 8 * t);      // this thread is past o_full and never reads O_t
        if (h == 0) {
          tc_fence_after();
          const float inv_l = l_row > 0.f ? 1.f / l_row : 0.f;
          // each warp stages and stores its own 32 rows (a 32-row TMA box): no rendezvous between
          // warps; lane 0 issues the warp's stores and waits for the previous one to have read the rows
          const uint32_t stage = s_stage_o + (uint32_t)t * Cfg::kStageOBytes + (uint32_t)quad * (32 * 128);
          const uint32_t stage_row = stage + (uint32_t)lane * 128;
          const int row0_w = q_row0_t + 32 * quad;
#pragma unroll 1
          for (int hh = 0; hh < D / 64; ++hh) {          // 64 columns (one TMA box) at a time
            if (lane == 0) tma_store_wait_read();
            __syncwarp();
            uint32_t ov[64];
            tmem_ld32(tmem_o + hh * 64, *reinterpret_cast<uint32_t(*)[32]>(&ov[0]));
            tmem_ld32(tmem_o + hh * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&ov[32]));
            tc_wait_ld();
            if (hh == D / 64 - 1) {
              tc_fence_before();
              mbar_arrive(bar_o_empty + 8 * t);        // O_t may be overwritten by the next item now
            }
#pragma unroll
            for (int c16 = 0; c16 < 8; ++c16) {
              const uint32_t addr = stage_row + (((uint32_t)c16 ^ ((uint32_t)lane & 7u)) << 4);
              const uint32_t w0 = pack_bf16(__uint_as_float(ov[c16 * 8 + 0]) * inv_l, __uint_as_float(ov[c16 * 8 + 1]) * inv_l);
              const uint32_t w1 = pack_bf16(__uint_as_float(ov[c16 * 8 + 2]) * inv_l, __uint_as_float(ov[c16 * 8 + 3]) * inv_l);
              const uint32_t w2 = pack_bf16(__uint_as_float(ov[c16 * 8 + 4]) * inv_l, __uint_as_float(ov[c16 * 8 + 5]) * inv_l);
              const uint32_t w3 = pack_bf16(__uint_as_float(ov[c16 * 8 + 6]) * inv_l, __uint_as_float(ov[c16 * 8 + 7]) * inv_l);
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w0), "r"(w1), "r"(w2), "r"(w3) : "memory");
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0 && row0_w < args.capacity) {
              tma_store(&map_o, stage, head_t, row0_w, hh, item_bin);
              asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
          }
        }
      } else {
        mbar_arrive(bar_o_empty + 8 * t);
      }
      if (!ok) break;
      ++it_n;
    }
    if (h == 0 && lane == 0) tma_store_wait_read();    // staging must outlive the last store's read
    }   // shared-stream mode
  }

  tc_fence_before();
  __syncthreads();
  if (*s_abort) {
    if (threadIdx.x == 0 && args.status) atomicCAS(args.status, 0, *s_abort);
    // A wait gave up: TMA loads and MMAs of this CTA may still be in flight. Give them time to land
    // (they take microseconds) before shared memory and TMEM are handed back.
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < 100000ull) {}
    __syncthreads();
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

// Self-test of the bounded-wait mechanism: one thread waits on an mbarrier that nothing ever
// arrives on. The wait must give up after `limit_ns`, write its code to the status word and let
// the kernel return normally.
__global__ void bounded_wait_selftest_kernel(int32_t* status, unsigned long long limit_ns) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  const WaitCtx wctx{smem_u32(&abort_flag), (uint32_t)(limit_ns >> 10), status};
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_wait<77>(smem_u32(&bar), 0, wctx);
  __syncthreads();
  if (threadIdx.x == 0 && abort_flag) atomicCAS(status, 0, abort_flag);
}

// ------------------------------------------------------------------------------------------
// Host side: tensor maps and launch
// ------------------------------------------------------------------------------------------
using EncodeFn = PFN_cuTensorMapEncodeTiled_v12000;

EncodeFn get_encode_fn() {
  static EncodeFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeFn>(p);
  }();
  return fn;
}

// 5-D map (column, head, row, chunk of 64 columns, bin) over a dense [R, M, H, D] bf16 tensor; box = 64 columns x
// `heads` heads x `rows` rows x `chunks` chunks x 1 bin: in shared memory the chunks lie one behind the other, each
// row-major over (row, head) with 128 bytes per row, swizzled. So a whole tile is one load.
int make_map(CUtensorMap* map, const void* ptr, int64_t R, int64_t M, int64_t H, int64_t D, int rows, int heads, int chunks) {
  EncodeFn enc = get_encode_fn();
  if (!enc) return note_cuda_error(-1, "cuTensorMapEncodeTiled entry point not found");
  cuuint64_t dims[5] = {64u, (cuuint64_t)H, (cuuint64_t)M, (cuuint64_t)(D / 64), (cuuint64_t)R};
  cuuint64_t strides[4] = {(cuuint64_t)(D * 2), (cuuint64_t)(H * D * 2), 128u, (cuuint64_t)(M * H * D * 2)};
  cuuint32_t box[5] = {64u, (cuuint32_t)heads, (cuuint32_t)rows, (cuuint32_t)chunks, 1u};
  cuuint32_t estr[5] = {1u, 1u, 1u, 1u, 1u};
  const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(ptr), dims, strides,
                         box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? PP_OK : note_cuda_error((int)r, "cuTensorMapEncodeTiled");
}

unsigned long long wait_limit_ns() {
  // Debug overrides of the device-side wait limit, in milliseconds or microseconds.
  if (const char* e = std::getenv("PP_WAIT_LIMIT_MS")) {
    const long ms = std::atol(e);
    if (ms > 0) return (unsigned long long)ms * 1000000ull;
  }
  if (const char* e = std::getenv("PP_WAIT_LIMIT_US")) {
    const long us = std::atol(e);
    if (us > 0) return (unsigned long long)us * 1000ull;
  }
  return 2000000000ull;   // 2 s
}

int sm_count() {
  static thread_local int cached_dev = -1, cached = 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (dev != cached_dev) {
    if (cudaDeviceGetAttribute(&cached, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    cached_dev = dev;
  }
  return cached;
}

template <int D, bool kIndep, bool kFill, class Table>
int launch_attention_t(const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const Table& tab, const void* q,
                       const void* k, const void* v, void* o, const void* rope_table, bool have_norms,
                       const CacheFill* caches, int32_t* device_status, cudaStream_t stream) {
  constexpr int BN = kIndep ? kTileNShort : kTileN;
  using Cfg = AttnCfg<D, BN>;
  CUtensorMap mq, mk, mv, mo;
  int st;
  const int fold = kIndep ? L.fold : 1;
  int fold_shift = 0;
  while ((1 << fold_shift) < fold) ++fold_shift;
  if ((st = make_map(&mq, q, p.n_bins, p.capacity, p.n_q_heads, D, BM / fold, fold, D / 64)) != PP_OK) return st;
  if ((st = make_map(&mk, k, p.n_bins, p.capacity, p.n_kv_heads, D, BN, 1, D / 64)) != PP_OK) return st;
  if ((st = make_map(&mv, v, p.n_bins, p.capacity, p.n_kv_heads, D, BN, 1, D / 64)) != PP_OK) return st;
  if ((st = make_map(&mo, o, p.n_bins, p.capacity, p.n_q_heads, D, 32 / fold, fold, 1)) != PP_OK) return st;   // one warp's rows per store
  // the shared-memory opt-in of a kernel is a per-device attribute
  static DeviceOnce configured;     // per template instance
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return note_cuda_error(-1, "cudaGetDevice");
  if (!configured.done(dev)) {
    cudaError_t e = cudaFuncSetAttribute(attention_kernel<D, kIndep, kFill, Table>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         Cfg::kSmemBytes);
    if (e != cudaSuccess) return note_cuda_error((int)e, "cudaFuncSetAttribute(smem)");
    configured.mark(dev);
  }
  const int sms = sm_count();
  if (sms <= 0) return note_cuda_error(-1, "multiprocessor count");
  AttnArgs a;
  a.counter = d_table + kHeaderCounter;
  a.v_cache = kFill ? static_cast<__nv_bfloat16*>(caches->v_cache) : nullptr;
  a.off_true_len = caches ? caches->off_true_len : 0;
  a.off_cap = caches ? caches->off_cap : 0;
  a.off_cache_off = caches ? caches->off_cache_off : 0;
  a.off_seg_start = L.seg_start;
  a.off_items = L.items;
  a.n_items = L.n_items;
  a.group = p.n_q_heads / p.n_kv_heads;
  a.pair_heads = (!kIndep && a.group % 2 == 0) ? 1 : 0;
  a.fold = fold;
  a.fold_shift = fold_shift;
  a.subs = a.pair_heads ? a.group / 2 : a.group / fold;
  a.capacity = p.capacity;
  const int64_t total = (int64_t)p.n_kv_heads * L.n_items * a.subs;
  if (total > INT32_MAX) return PP_ERR_UNSUPPORTED;
  a.total_work = (int32_t)total;
  const float scale = p.softmax_scale > 0.f ? p.softmax_scale : 1.0f / sqrtf((float)D);
  a.scale_log2 = scale * 1.4426950408889634f;
  a.bound2 = fminf((kBoundLog2 / a.scale_log2) * (kBoundLog2 / a.scale_log2), FLT_MAX);
  const bool norms = have_norms && tracks_ranges(p, L);
  a.k_norm2 = norms ? reinterpret_cast<const uint32_t*>(d_table + L.norms) : nullptr;
  a.q_norm2 = norms && !rope_table ? a.k_norm2 + p.n_kv_heads : nullptr;
  a.v_max = tracks_ranges(p, L) ? reinterpret_cast<const uint32_t*>(d_table + kHeaderValueMax) : nullptr;
  a.v_room = ldexpf(1.f, kValueRoomLog2) / (float)p.capacity;
  a.rope_table = static_cast<const float2*>(rope_table);
  a.status = device_status;
  a.wait_limit = (uint32_t)std::min<unsigned long long>(wait_limit_ns() >> 10, 0x7fffffffu);
  // The order of the work: KV heads one after another, so that those at work at a time find their K and V in L2, each
  // head's entries longest first. How evenly the CTAs finish is then left to the last head alone, so the last heads are
  // drawn together, the longest entries of all of them first.
  // Independent mode: two heads, or as many as make two entries for every slot (16 prompts on 32 heads, longest finish /
  // mean as replayed 1.41 -> 1.17, whole step 48.8 -> 46.1 us, with four entries per slot 46.7, with one 48.2; 64 prompts
  // 235 -> 231.5, 232.5, 234).
  // Shared-stream mode: as many as make two entries for every CTA, where one head has less (one after another -> together:
  // one prompt of 4000 tokens on 32 heads of 128 192 -> 163 us, of 12 800 1295 -> 1219, two of 12 800 2474 -> 2410, one of 6400 on
  // 32 / 8 heads 342 -> 317, of 3000 on 32 / 8 heads of 64 97 -> 75; 0.998 to 1.01 close to the line). From there on one:
  // two made 0.994 to 1.006 of it on seven batches of up to 1.5 times as many entries, and cost 256 prompts on 32 / 8
  // heads L2 hits (6330 -> 6400).
  const int64_t per_head = (int64_t)L.n_items * a.subs, drawers = (int64_t)(kIndep ? 2 : 1) * sms;
  const int64_t together = std::min<int64_t>(p.n_kv_heads, std::max<int64_t>(kIndep ? 2 : 1, (2 * drawers + per_head - 1) / per_head));
  a.tail_head0 = p.n_kv_heads - (int32_t)together;
  a.tail_start = (int32_t)(a.tail_head0 * per_head);
  a.tail_cols = (int32_t)(together * a.subs);
  const unsigned grid = (unsigned)(total < sms ? total : sms);
  const cudaError_t launch_err = launch_dependent(attention_kernel<D, kIndep, kFill, Table>, dim3(grid), dim3(kIndep ? kAttnThreadsIndep : kAttnThreads),
                                                  (size_t)Cfg::kSmemBytes, stream, mq, mk, mv, mo, a, tab);
  const cudaError_t e = launch_err != cudaSuccess ? launch_err : cudaGetLastError();
  return e == cudaSuccess ? PP_OK : note_cuda_error((int)e, "attention kernel launch");
}

}  // namespace

int launch_bounded_wait_selftest(int32_t* device_status, uint64_t limit_ns, void* stream) {
  bounded_wait_selftest_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(device_status, limit_ns);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? PP_OK : note_cuda_error((int)e, "self-test kernel launch");
}

int launch_attention(const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const int32_t* inline_table, const void* q,
                     const void* k, const void* v, void* o, const void* rope_table, bool have_norms,
                     const CacheFill* caches, int32_t* device_status, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const auto launch = [&](auto d, auto indep, auto fill, const auto& tab) {
    return launch_attention_t<d(), indep(), fill()>(p, d_table, L, tab, q, k, v, o, rope_table, have_norms, caches, device_status, s);
  };
  using D64 = std::integral_constant<int, 64>;
  using D128 = std::integral_constant<int, 128>;
  using Yes = std::true_type;
  using No = std::false_type;
  if (inline_table) {                 // independent mode only
    const TableInline tab = inline_copy(inline_table, caches ? (size_t)caches->off_cache_off + 2 * (size_t)L.n_segments
                                                             : (size_t)L.total_ints);
    if (caches) return launch(D128{}, Yes{}, Yes{}, tab);
    return p.head_dim == 128 ? launch(D128{}, Yes{}, No{}, tab) : launch(D64{}, Yes{}, No{}, tab);
  }
  const TableInMemory tab{d_table};
  if (caches) return launch(D128{}, Yes{}, Yes{}, tab);
  if (L.independent_slots) return p.head_dim == 128 ? launch(D128{}, Yes{}, No{}, tab) : launch(D64{}, Yes{}, No{}, tab);
  return p.head_dim == 128 ? launch(D128{}, No{}, No{}, tab) : launch(D64{}, No{}, No{}, tab);
}

}  // namespace pp
