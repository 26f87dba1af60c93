// Tree-masked attention on the 5th-generation tensor cores (tcgen05.mma, accumulators in tensor
// memory, K/V/Q tiles staged by TMA), for 16-bit inputs.
//
// Work unit: (kv head g, tile of 128 query rows, range of the tile's keys).  A query row is
// a (node, head-in-group) pair, r = i_local * G + hg, so under GQA the G heads that share a kv head
// share every K/V tile.  Per block of 64 keys:
//     S = Q K^T      128x64x128   tcgen05.mma, Q and K K-major in 128-byte-swizzled shared memory
//     P = 2^(scale*S - m) masked  one thread per row: S read from tensor memory, P written back over
//                                 it as packed 16-bit values
//     O += P V       128x128x64   tcgen05.mma, A = P from tensor memory, V MN-major in shared memory
//
// Two chains per CTA, each double-buffered.  Keys are taken in blocks of 64; even blocks of the CTA's
// key range belong to chain A, odd blocks to chain B.  Each chain has two S/P buffers (64 columns
// each) and its own accumulator O in tensor memory (2 x (2*64 + 128) = 512 columns), two K and two V
// stages in shared memory, its own 128 row threads (one warp group), its own MMA-issuing warp and its
// own running (m, l); the chains share Q and the two TMA warps (one for Q and K, one for V: a K stage
// is free once its S is computed, a V stage only after the block's softmax, and K loads must not queue
// behind that).  S of a chain's next block is computed while its row threads still work on the current
// one, so a chain runs at the speed of its softmax, and while one chain exponentiates the tensor pipe
// also works for the other.  Per block a row thread first takes the block maximum (comparisons only),
// settles the reference maximum - it only moves when the block maximum exceeds it by more than 2^8, the
// accumulator row is then rescaled in tensor memory - and then takes the 64 exponentials, which are
// the bottleneck (16 per clock and SM).  Registers are rebalanced with setmaxnreg: 40 for the TMA/MMA
// warp group, 232 for the rows.
//
// Work distribution.  Grid mode: one CTA per (tile, kv head), in as many waves as that takes, or (up to one wave) a
// cluster of 2 to 8 CTAs that split its key range; the thread that arms the barriers requests the Q tile and the
// first K tiles itself, before the CTA-wide barrier.  Stream mode (many units of long tiles): one CTA per SM; the
// 64-key blocks of all units are laid end to end (each tile preceded by a few positions that stand for
// its fixed cost, tiles of a head taken alternately from both ends) and cut into equal ranges.  A CTA
// works through the segments of its range with barrier phases that run on from segment to segment, so
// the next segment's loads and first S are under way while the rows still merge and store.  A tile cut
// by a range boundary is completed by whichever of its CTAs finishes last: the others leave their
// piece (m, l, unnormalised accumulator) in the workspace and count themselves on the tile's counter;
// the pieces are added in CTA order, so the result does not depend on who finishes last.
//
// Merge.  The CTAs that share (tile, kv head) form a thread-block cluster along the key range (cs = 1 .. 8).  Each sends
// its rows' (m, l) into every CTA as soon as its two chains are done; that travels while it reads its accumulators out of
// tensor memory.  Then it knows the rows' common maximum and sum, scales its partial to its share of the final output, and
// sends each slice of 8 output columns to the CTA that owns it (the K/V stages, dead by then, receive them).  After a
// cluster barrier an owner has only additions left.  No workspace, no second kernel.  (Against unscaled pieces, with the
// owner working out every contributor's factor behind the barrier: 64 nodes on 1024 keys of 32 heads 9.95 -> 9.6 us.)
//
// Masking: key j < prefix_len is visible; key prefix_len + t is visible iff bit t of the row's
// ancestor mask; masked scores become -inf before the maximum, so their probability is exactly 0.
// Rows of K/V past prefix_len + n_tree are never fetched: the tensor maps end there and TMA fills
// the rest of a tile with zeros.
//
// Every mbarrier wait is bounded; a wait that runs out raises SEQ_DEV_TIMEOUT and the CTA drains.
//
// The kernel is launched with programmatic stream serialisation: its set-up runs under the previous kernel's tail,
// griddepcontrol.wait precedes its first access to global memory.
#include <cooperative_groups.h>
#include <cstddef>
#include <cuda.h>
#include <stdlib.h>

#include <type_traits>

#include "common.cuh"
#include "tensor_map.cuh"
#include "trace_attention.cuh"

namespace cg = cooperative_groups;

namespace seqtree {

constexpr int kTileM = 128;         // query rows per CTA
constexpr int kBlockN = 64;         // keys per block
constexpr int kUmmaThreads = 384;   // warp group 0: TMA warp, MMA warp, two spare; warp groups 1, 2: rows of chains A, B
constexpr int kRegsLight = 40, kRegsRows = 232;  // after setmaxnreg: 128*40 + 256*232 = 384*168
constexpr int kMaxClusterSplit = 8;
constexpr int kMaxStreamTiles = 128;  // tiles per kv head the stream mode can index
// Stream mode balances cost, not block counts: every tile is laid out with this many extra positions in
// front of its blocks, standing for what starting and finishing a tile costs (about 4 us, in 64-key blocks).
constexpr int kStreamTileCost = 8;

constexpr uint32_t kTileBytes = 128 * 128 * 2;   // the Q tile: 128 rows x 128 elements of 16 bits
constexpr uint32_t kHalfBytes = kTileBytes / 2;  // one 128-row x 64-element sub-tile of Q (128 B rows)
constexpr uint32_t kKvBytes = kBlockN * 128 * 2; // a K or V tile: 64 keys x 128 elements
constexpr uint32_t kKvHalf = kKvBytes / 2;       // one 64-row x 64-element sub-tile of K or V
constexpr float kRescaleThreshold = 8.f;         // log2 units
constexpr float kRescaleLimit = 256.f;           // 2^kRescaleThreshold: no term of a row sum at or below it came from a score above the threshold
constexpr uint32_t kSpinLimit = 1u << 22;

struct UmmaSmem {
  // all tiles 1024-byte aligned (128-byte swizzle atoms are 8 rows x 128 B)
  uint8_t q[kTileBytes];
  uint8_t k[2][2][kKvBytes];  // [chain][stage]; after the last block these 64 KB receive the cluster merge
  uint8_t v[2][2][kKvBytes];  // [chain][stage]
  float2 ml_chain[2][2][kTileM];             // [segment parity][chain]: (m, l) of every row of the two chains of this CTA
  float2 ml_cta[kMaxClusterSplit][kTileM];   // (m, l) of every row of every CTA of the cluster, after its chains are merged
  uint64_t q_full;
  uint64_t k_full[2][2], k_empty[2][2], v_full[2][2], v_empty[2][2], s_full[2][2], p_full[2][2];  // [chain][stage]
  uint64_t pv_done[2];                       // [chain]: one phase per block of the chain
  uint64_t all_done[2];                      // [chain]: every MMA of the chain in this segment has completed (one phase per segment)
  uint64_t o_free;                           // the row threads have read both accumulators (one phase per segment)
  uint32_t tmem_base;
  volatile int abort_flag;
  int32_t abort_seen[2];                     // [segment parity]: abort_flag as one row thread saw it, so that all 256 leave together
  int32_t last_part;                         // stream mode: this CTA completed the tile (broadcast to the row threads)
  // mask from the parent array: the tree, and the ancestor rows of the current tile's nodes (row stride 33 words)
  int32_t parent[SEQ_MAX_TREE];
  uint32_t tile_mask[kTileM][SEQ_MAX_TREE / 32 + 1];
  int32_t tile_prefix[kMaxStreamTiles + 1];  // stream mode: positions of a kv head's layout before its t-th tile
};

static_assert(offsetof(UmmaSmem, v) == offsetof(UmmaSmem, k) + sizeof(UmmaSmem::k), "the cluster merge receives into k and v as one buffer");

struct UmmaArgs {
  int32_t n, L_host, Hq, Hkv, group, mask_wpr, splits, nodes_per_tile, tiles;
  int32_t rows;           // query rows of a full tile: nodes_per_tile * group, 128 when the group divides it
  const int32_t* L_dev;   // nullable: the prefix length in device memory (<= L_host)
  int32_t L_count;        // > 1: one length per request, requests stacked as heads (grid schedule only: a CTA has one kv head)
  int32_t zero_tail;      // the K/V maps cover the whole cache: rows past the tree are cleared in shared memory
  // Stream mode (more (tile, kv head) units than SMs): the 64-key blocks of all units, laid end to end, are
  // cut into gridDim.x equal ranges, one per CTA; a tile cut by a range boundary is completed by whichever
  // of its CTAs finishes last, from partial results in the workspace.
  int32_t stream, blocks_per_head_host;
  int32_t total_blocks_host;  // (a layout of 2^31 positions and more is not streamed)
  int32_t* ws_count;   // [Hkv * tiles] arrivals per tile, zero on entry and on exit
  float2* ws_ml;       // [2 * gridDim.x][128] (m, l) of a partial result
  float4* ws_o;        // [2 * gridDim.x][2][16][128] its unnormalised accumulator, thread-major
  float scale_log2;
  uint32_t idesc_qk, idesc_pv;
  const uint32_t* mask_bits;
  const int32_t* parent;  // used when mask_bits is null
  void* out; int64_t o_stride_tok, o_stride_head;
  float* lse;
  int32_t* dev_status;
};

// ---------------------------------------------------------------- PTX wrappers ------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
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
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false (and raises the CTA-wide abort flag) if the phase never completes.
__device__ __forceinline__ bool mbar_wait(UmmaSmem* sm, uint64_t* bar, uint32_t parity, int32_t* dev_status) {
  for (uint32_t it = 0; it < kSpinLimit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 1023u) == 1023u && sm->abort_flag) return false;
  }
  sm->abort_flag = 1;
  dev_flag(dev_status, SEQ_DEV_TIMEOUT);
  return false;
}

__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1, int c2, int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4) : "memory");
}
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// A value that every lane of the warp holds, so that the compiler knows it is the same: what is derived from it stays on the
// uniform datapath, where the operands of tcgen05.mma have to be (a value it cannot prove uniform is moved there for every
// single instruction).
template <typename T>
__device__ __forceinline__ T uniform(T x) { return __shfl_sync(0xffffffffu, x, 0); }

// True in exactly one lane of a converged warp.  Code that must be issued once per warp (MMAs, commits)
// goes under this predicate while everything around it stays warp-uniform, which keeps descriptors and
// addresses on the uniform datapath.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(pred));
  return pred != 0;
}

__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// The two products of a block, each issued as one run of MMAs.  The operands' descriptors differ in their low words only
// (start address in 16-byte units), which the run itself steps along the contraction: descriptors worked out beside the MMAs
// are hoisted out of the block loop by the compiler and cost the issuing warp its few registers.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);  // 1024 B between groups of 8 rows, version 1, 128-byte swizzle
// low word of a shared-memory descriptor; lbo: bytes between 64-element blocks along MN (MN-major operands)
__device__ __forceinline__ uint32_t desc_lo(uint32_t smem_addr, uint32_t lbo) { return ((smem_addr >> 4) & 0x3FFFu) | (((lbo >> 4) & 0x3FFFu) << 16); }

// S = Q K^T over head_dim = 128: eight steps of 16 elements, 32 bytes apart inside a 64-element sub-tile; kQHalf, kKHalf:
// bytes from the first sub-tile to the second
template <uint32_t kQHalf, uint32_t kKHalf>
__device__ __forceinline__ void mma_qk(uint32_t d_tmem, uint32_t q_lo, uint32_t k_lo, uint32_t idesc) {
#define SEQ_STEP(qs, ks) "add.u32 q, q, " qs ";\n\tadd.u32 k, k, " ks ";\n\tmov.b64 x, {q, %3};\n\tmov.b64 y, {k, %3};\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %4, t;\n\t"
  asm volatile(
      "{\n\t.reg .pred p, t;\n\t.reg .b64 x, y;\n\t.reg .b32 q, k;\n\t"
      "setp.ne.b32 p, 0, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
      "mov.b32 q, %1;\n\tmov.b32 k, %2;\n\t"
      "mov.b64 x, {%1, %3};\n\tmov.b64 y, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %4, p;\n\t"
      SEQ_STEP("2", "2") SEQ_STEP("2", "2") SEQ_STEP("2", "2") SEQ_STEP("%5", "%6") SEQ_STEP("2", "2") SEQ_STEP("2", "2") SEQ_STEP("2", "2")
      "}"
      ::"r"(d_tmem), "r"(q_lo), "r"(k_lo), "r"(kDescHi), "r"(idesc), "n"((kQHalf >> 4) - 6), "n"((kKHalf >> 4) - 6) : "memory");
#undef SEQ_STEP
}
// O (+)= P V over 64 keys: A = 8 packed columns of P, B = 16 key rows of V (2048 bytes) per step
__device__ __forceinline__ void mma_pv(uint32_t d_tmem, uint32_t p_tmem, uint32_t v_lo, uint32_t idesc, uint32_t accumulate) {
#define SEQ_STEP "add.u32 a, a, 8;\n\tadd.u32 v, v, 128;\n\tmov.b64 y, {v, %3};\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [a], y, %4, t;\n\t"
  asm volatile(
      "{\n\t.reg .pred p, t;\n\t.reg .b64 y;\n\t.reg .b32 a, v;\n\t"
      "setp.ne.b32 p, %5, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
      "mov.b32 a, %1;\n\tmov.b32 v, %2;\n\t"
      "mov.b64 y, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], y, %4, p;\n\t"
      SEQ_STEP SEQ_STEP SEQ_STEP "}"
      ::"r"(d_tmem), "r"(p_tmem), "r"(v_lo), "r"(kDescHi), "r"(idesc), "r"(accumulate) : "memory");
#undef SEQ_STEP
}

#define SEQ_R32(a, o) \
  "=r"(a[o + 0]), "=r"(a[o + 1]), "=r"(a[o + 2]), "=r"(a[o + 3]), "=r"(a[o + 4]), "=r"(a[o + 5]), "=r"(a[o + 6]),   \
  "=r"(a[o + 7]), "=r"(a[o + 8]), "=r"(a[o + 9]), "=r"(a[o + 10]), "=r"(a[o + 11]), "=r"(a[o + 12]),               \
  "=r"(a[o + 13]), "=r"(a[o + 14]), "=r"(a[o + 15]), "=r"(a[o + 16]), "=r"(a[o + 17]), "=r"(a[o + 18]),            \
  "=r"(a[o + 19]), "=r"(a[o + 20]), "=r"(a[o + 21]), "=r"(a[o + 22]), "=r"(a[o + 23]), "=r"(a[o + 24]),            \
  "=r"(a[o + 25]), "=r"(a[o + 26]), "=r"(a[o + 27]), "=r"(a[o + 28]), "=r"(a[o + 29]), "=r"(a[o + 30]),            \
  "=r"(a[o + 31])
#define SEQ_W32(a, o) \
  "r"(a[o + 0]), "r"(a[o + 1]), "r"(a[o + 2]), "r"(a[o + 3]), "r"(a[o + 4]), "r"(a[o + 5]), "r"(a[o + 6]),          \
  "r"(a[o + 7]), "r"(a[o + 8]), "r"(a[o + 9]), "r"(a[o + 10]), "r"(a[o + 11]), "r"(a[o + 12]), "r"(a[o + 13]),      \
  "r"(a[o + 14]), "r"(a[o + 15]), "r"(a[o + 16]), "r"(a[o + 17]), "r"(a[o + 18]), "r"(a[o + 19]), "r"(a[o + 20]),   \
  "r"(a[o + 21]), "r"(a[o + 22]), "r"(a[o + 23]), "r"(a[o + 24]), "r"(a[o + 25]), "r"(a[o + 26]), "r"(a[o + 27]),   \
  "r"(a[o + 28]), "r"(a[o + 29]), "r"(a[o + 30]), "r"(a[o + 31])

// 32 consecutive fp32 columns of this thread's tensor-memory lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r, int o) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, "
      "%23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : SEQ_R32(r, o) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r, int o) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, "
      "%23, %24, %25, %26, %27, %28, %29, %30, %31};"
      ::SEQ_W32(r, o), "r"(taddr) : "memory");
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};"
      ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr) : "memory");
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// The Q tile of nodes [i0, i0 + nodes_per_tile) of kv head g.  When the group divides 128 the tile has 128 rows and one
// copy brings both 64-element halves; otherwise it has fewer (the halves of one copy would then lie rows * 128 bytes
// apart, off the swizzle's 1024-byte boundary), and each half is a copy of its own to its fixed place.
__device__ __forceinline__ void load_q(uint8_t* dst, const CUtensorMap* map, uint64_t* bar, int rows, int i0, int g) {
  mbar_expect_tx(bar, (uint32_t)rows * 256u);
  tma_load_5d(dst, map, bar, 0, 0, i0, 0, g);
  if (rows < kTileM) tma_load_5d(dst + kHalfBytes, map, bar, 0, 0, i0, 1, g);
}

// Two single-precision values in one 64-bit register, for the packed fused multiply-add and add: half the issue slots.
__device__ __forceinline__ uint64_t pair_of(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpair(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// The address of a shared-memory word of CTA `rank` of the cluster, and stores to it.
__device__ __forceinline__ uint32_t remote_smem(uint32_t addr, int rank) {
  uint32_t d;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
  return d;
}
__device__ __forceinline__ void st_cluster4(uint32_t addr, const float* x) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]) : "memory");
}
__device__ __forceinline__ void st_cluster2(uint32_t addr, float x, float y) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

template <bool kBf16>
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  if (kBf16) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
  } else {
    __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
  }
}

// What pack2 left of a and b, packed the same way.
template <bool kBf16>
__device__ __forceinline__ uint32_t pack_rest(float a, float b, uint32_t packed) {
  float ra, rb;
  if (kBf16) {
    ra = __uint_as_float(packed << 16); rb = __uint_as_float(packed & 0xFFFF0000u);
  } else {
    const float2 r = __half22float2(*reinterpret_cast<const __half2*>(&packed));
    ra = r.x; rb = r.y;
  }
  return pack2<kBf16>(a - ra, b - rb);
}

// 32 validity bits for tree indices [t, t+32) of one mask row; negative indices are prefix keys (visible)
__device__ __forceinline__ uint32_t mask_window(const uint32_t* row, int wpr, int n, int t) {
  const int w = t >> 5;  // floor
  const uint32_t lo = w < 0 ? 0xFFFFFFFFu : (w < wpr ? row[w] : 0u);
  const uint32_t hi = (w + 1) < 0 ? 0xFFFFFFFFu : ((w + 1) < wpr ? row[w + 1] : 0u);
  uint32_t bits = __funnelshift_r(lo, hi, t & 31);
  const int nvis = n - t;  // tree indices >= n do not exist, whatever the mask words hold there
  if (nvis < 32) bits &= nvis <= 0 ? 0u : ((1u << nvis) - 1u);
  return bits;
}

enum { kGrid, kCluster, kStreamed };  // the schedule: a CTA per unit; a cluster of CTAs per unit; ranges of all units' blocks
// kFineP: P enters its product as two 16-bit pieces, the rounded value and the rest, each in a run of MMAs of its own.  For
// the groups of heads that do not divide 128, whose probabilities are held to single precision (the other groups round P
// to the input type).  Relative error of the output against fp64, 100 nodes on 1501 keys of 40/8 heads: 1.658e-3 in
// bfloat16 and 2.071e-4 in half, which is what rounding the exact output gives; with P rounded once 2.26e-3 and 2.82e-4.
// The second run costs that call 11.6 -> 12.7 us.
template <bool kBf16, int kMode, bool kFineP>
__global__ void __launch_bounds__(kUmmaThreads, 1)
tree_attention_umma_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                           const __grid_constant__ CUtensorMap v_map, const UmmaArgs a) {
  constexpr bool kStream = kMode == kStreamed;
  extern __shared__ uint8_t smem_raw[];
  UmmaSmem* sm = reinterpret_cast<UmmaSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = uniform((int)threadIdx.x >> 5), lane = threadIdx.x & 31;
#ifdef SEQ_TRACE
  int utrace_i = 0;
#endif
  const int split = kMode == kCluster ? blockIdx.z : 0;  // the cluster spans blockIdx.z
  if (kMode == kCluster) cluster_arrive_relaxed();  // "this CTA runs": waited for before the first remote store
  if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 10);
#ifdef SEQ_TRACE
  const unsigned cta_lin = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  if (threadIdx.x == 128 && cta_lin < 1024) g_cta_times[cta_lin][0] = gtimer();
#endif

  // A CTA works through segments: (kv head, tile, range of the tile's 64-key blocks).  Grid mode: the one
  // segment (blockIdx.y, blockIdx.x, this CTA's share of the cluster's key range).  Stream mode: the pieces
  // of the units that its range [range_lo, range_hi) of the flattened block space overlaps.
  // The prefix length: the host's, or - for a step replayed from one CUDA graph while the prefix grows - read from
  // device memory below (the host's value is then the largest it can be, which the launch was planned for).
  int L = a.L_host;
  int blocks_per_head = a.blocks_per_head_host;
  int total_blocks = a.total_blocks_host;
  int range_lo = 0, range_hi = 1;
  struct Seg { int g, tile, slot_in_head, i0, i1, blk_lo, nblk, nblk_tile, next; };
  // Stream mode lays the tiles of a kv head out alternating from both ends (0, T-1, 1, T-2, ...): late tiles
  // have more masked blocks, which cost more, and this way every range gets its share of them.
  auto tile_at = [&](int k) { return (k & 1) ? a.tiles - 1 - (k >> 1) : (k >> 1); };
  auto seg_at = [&](int pos) -> Seg {
    Seg x;
    if (!kStream) {
      x.tile = blockIdx.x; x.g = blockIdx.y; x.slot_in_head = x.tile;
      x.i0 = x.tile * a.nodes_per_tile;
      x.i1 = min(x.i0 + a.nodes_per_tile, a.n);
      // keys this tile can see end at L + i1 (a node sees no later node); blocks of this CTA
      x.nblk_tile = (L + x.i1 + kBlockN - 1) / kBlockN;
      // (rounded up: the CTA of the last keys, which are masked, is not the one with a block more)
      x.blk_lo = kMode == kGrid ? 0 : (split * x.nblk_tile + a.splits - 1) / a.splits;
      x.nblk = kMode == kGrid ? x.nblk_tile : ((split + 1) * x.nblk_tile + a.splits - 1) / a.splits - x.blk_lo;
      x.next = 1;
    } else {
      x.g = pos / blocks_per_head;
      const int rem = pos - x.g * blocks_per_head;
      int lo = 0, hi = a.tiles - 1;  // the last place in the head's layout whose first block is at or before rem
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sm->tile_prefix[mid] <= rem) lo = mid; else hi = mid - 1;
      }
      x.slot_in_head = lo;
      x.tile = tile_at(lo);
      x.i0 = x.tile * a.nodes_per_tile;
      x.i1 = min(x.i0 + a.nodes_per_tile, a.n);
      // the tile's positions are [vs, ve): kStreamTileCost positions of overhead, then its blocks
      const int vs = sm->tile_prefix[lo], ve = sm->tile_prefix[lo + 1];
      const int end = min(ve, rem + (range_hi - pos));  // where this CTA leaves the tile
      const int from = max(rem, vs + kStreamTileCost);
      x.blk_lo = from - (vs + kStreamTileCost);
      x.nblk_tile = ve - vs - kStreamTileCost;
      x.nblk = max(end - from, 0);  // 0: the range ends in the overhead positions, the tile is the next CTA's
      x.next = pos + (end - rem);
    }
    return x;
  };
  // The barriers are armed once.  Their phases run on from segment to segment: a stage barrier counts the
  // blocks its chain has processed so far, q_full / all_done[] / o_free count segments.  So the loads and
  // the first S of the next segment are under way while the row threads still merge and store this one.
  auto init_barriers = [&]() {  // thread 0
    mbar_init(&sm->q_full, 1);
    for (int c = 0; c < 2; ++c) {
      for (int b = 0; b < 2; ++b) {
        mbar_init(&sm->k_full[c][b], 1); mbar_init(&sm->k_empty[c][b], 1);
        mbar_init(&sm->v_full[c][b], 1); mbar_init(&sm->v_empty[c][b], 1);
        mbar_init(&sm->s_full[c][b], 1); mbar_init(&sm->p_full[c][b], 4);
      }
      mbar_init(&sm->pv_done[c], 1);
    }
    mbar_init(&sm->all_done[0], 1); mbar_init(&sm->all_done[1], 1);  // each has one arriver: its chain's MMA warp
    mbar_init(&sm->o_free, 8);    // one arrival per warp of row threads
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  };
  if (threadIdx.x == 0) {
    init_barriers();
    sm->abort_flag = 0;
    // programmatic dependent launch: the next kernel in the stream may be scheduled onto free SMs from now on (it
    // waits, as this one does below, before it touches memory); without the launch attribute this does nothing
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  // ... and everything above ran while the previous kernel in the stream was still finishing.  Nothing before this
  // line reads or writes global memory.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (a.L_dev != nullptr) {
    const int v = a.L_dev[(!kStream && a.L_count > 1) ? ((int)blockIdx.y * a.L_count) / a.Hkv : 0];
    if (v < 0 || v > a.L_host) { if (threadIdx.x == 0) dev_flag(a.dev_status, SEQ_DEV_BAD_LENGTH); }
    L = uniform(min(max(v, 0), a.L_host));
    if (kStream) {  // the flattened block space of this prefix length (every warp for itself)
      int sum = 0;
      for (int t = lane; t < a.tiles; t += 32) sum += kStreamTileCost + (L + min((t + 1) * a.nodes_per_tile, a.n) + kBlockN - 1) / kBlockN;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      blocks_per_head = sum;
      total_blocks = sum * a.Hkv;
    }
  }
  // where the range of CTA x starts: total_blocks * x / gridDim.x
  const int per_cta = kStream ? total_blocks / (int)gridDim.x : 0, left_over = total_blocks - per_cta * (int)gridDim.x;
  auto cta_lo = [&](int x) { return per_cta * x + (left_over * x) / (int)gridDim.x; };
  if (kStream) {
    range_lo = cta_lo(blockIdx.x);
    range_hi = cta_lo(blockIdx.x + 1);
  }
  // Grid schedule: the one segment of this CTA is known from its block index, so the thread that armed the barriers
  // requests the Q tile and the first K tile of each chain right away, before the CTA-wide barrier below and the
  // hand-over to the producer warps (which skip what has been requested here).
  if (!kStream && threadIdx.x == 0) {
    const Seg s0 = seg_at(range_lo);
    if (s0.nblk > 0) {
      load_q(sm->q, &q_map, &sm->q_full, a.rows, s0.i0, s0.g);
      for (int jj = 0; jj < 2 && jj < s0.nblk; ++jj) {
        mbar_expect_tx(&sm->k_full[jj][0], kKvBytes);
        tma_load_4d(sm->k[jj][0], &k_map, &sm->k_full[jj][0], 0, (s0.blk_lo + jj) * kBlockN, 0, s0.g);
      }
    }
  }
  if (a.mask_bits == nullptr)
    for (int t = threadIdx.x; t < a.n; t += kUmmaThreads) sm->parent[t] = a.parent[t];
  if (a.rows < kTileM) {  // rows no copy writes (the group does not divide 128): zeros, so that their scores are finite
    for (int t = a.rows * 8 + (int)threadIdx.x; t < kTileM * 8; t += kUmmaThreads) {
      reinterpret_cast<uint4*>(sm->q)[t] = make_uint4(0u, 0u, 0u, 0u);
      reinterpret_cast<uint4*>(sm->q + kHalfBytes)[t] = make_uint4(0u, 0u, 0u, 0u);
    }
    fence_async_smem();
  }
  if (kStream && warp == 2) {  // blocks of a kv head before each place of its layout: four places per lane, then a warp scan
    const int per = (a.tiles + 31) / 32;
    int local[kMaxStreamTiles / 32], sum = 0;
#pragma unroll
    for (int k = 0; k < kMaxStreamTiles / 32; ++k) {
      const int t = lane * per + k;
      local[k] = (k < per && t < a.tiles) ? kStreamTileCost + (L + min((tile_at(t) + 1) * a.nodes_per_tile, a.n) + kBlockN - 1) / kBlockN : 0;
      sum += local[k];
    }
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += v;
    }
    int run = incl - sum;
#pragma unroll
    for (int k = 0; k < kMaxStreamTiles / 32; ++k) {
      const int t = lane * per + k;
      if (k < per && t < a.tiles) sm->tile_prefix[t] = run;
      run += local[k];
    }
    if (lane == 31) sm->tile_prefix[a.tiles] = incl;
  }
  if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 11);
  if (warp == 1) {  // all 512 tensor-memory columns: per chain two S buffers of 64 (P over them), then O_A, O_B
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&sm->tmem_base)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = uniform(sm->tmem_base);
  if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 0);

  if (warp < 4) {
    // ============================ warp group 0: data movement and MMA issue, few registers =========
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLight));
    int seg_n = 0, base_an = 0, base_bn = 0;  // segments done; blocks chains A, B have processed in them
    uint32_t issued = 0, issued_parity = 0;   // producers: stages (bit 2*chain + stage; bit 4: Q) this warp has requested a tile for, and the phase of the last request
    for (int pos = range_lo; pos < range_hi;) {
    const Seg sg = seg_at(pos);
    if (kStream && sg.nblk == 0) { pos = sg.next; continue; }
    const int g = sg.g, i0 = sg.i0, blk_lo = sg.blk_lo, nblk = sg.nblk;
    const int seg = kStream ? seg_n : 0, base_a = kStream ? base_an : 0, base_b = kStream ? base_bn : 0;  // grid mode: constants
    if (warp == 0 || warp == 3) {
      // ---------------------------------------------------------- TMA producers -----------------
      // Warp 0 loads Q and the K tiles, warp 3 the V tiles.  A K stage is free as soon as its S has been
      // computed, a V stage only after the block's softmax and P.V; in one queue the K loads would wait
      // behind the V stages and arrive just in time instead of a block ahead.
      // The whole warp runs the loop; one elected lane issues the copies (coordinates stay warp-uniform).
      if (nblk > 0) {
        const bool is_v = warp == 3;
        // the Q tile is free when every MMA of the previous segment has completed: the row threads have
        // seen that before they read O (waiting on o_free rather than all_done keeps every waiter of a
        // barrier within one phase of its arrivers)
        if (!is_v && seg > 0 && !mbar_wait(sm, &sm->o_free, (seg - 1) & 1, a.dev_status)) break;
        if (kStream && !is_v && elect_one()) {  // (grid schedule: requested before the roles split, see above)
          load_q(sm->q, &q_map, &sm->q_full, a.rows, i0, g);
        }
        __syncwarp();
        if (kStream && !is_v) { issued |= 16u; issued_parity = (issued_parity & ~16u) | ((uint32_t)(seg & 1) << 4); }
        const CUtensorMap* map = is_v ? &v_map : &k_map;
        for (int jj = (!kStream && !is_v) ? min(2, nblk) : 0; jj < nblk; ++jj) {
          const int c = jj & 1, u = (c ? base_b : base_a) + (jj >> 1);  // chain, the chain's running block count
          const int b = u & 1, w = u >> 1;                              // stage, use count of the stage
          const int row = (blk_lo + jj) * kBlockN;
          uint64_t* full = is_v ? &sm->v_full[c][b] : &sm->k_full[c][b];
          uint64_t* empty = is_v ? &sm->v_empty[c][b] : &sm->k_empty[c][b];
          uint8_t* dst = is_v ? sm->v[c][b] : sm->k[c][b];
          if (w > 0 && !mbar_wait(sm, empty, (w - 1) & 1, a.dev_status)) break;
          if (elect_one()) {
            mbar_expect_tx(full, kKvBytes);
            tma_load_4d(dst, map, full, 0, row, 0, g);  // both 64-element halves by one copy
          }
          __syncwarp();
          issued |= 1u << (2 * c + b);
          issued_parity = (issued_parity & ~(1u << (2 * c + b))) | ((uint32_t)(w & 1) << (2 * c + b));
          if (lane == 0 && !is_v) UTRACE(0, 1);
        }
      }
      __syncwarp();
    } else if (warp <= 2) {
      // ---------------------------------------------------------- MMA issuers -------------------
      // Warp 1 issues for chain A, warp 2 for chain B.  The whole warp runs this code; only the MMAs and
      // commits are issued by one elected lane, so descriptors and addresses stay warp-uniform.
      const int c = warp - 1;
      const int n_c = nblk > c ? (nblk - c + 1) >> 1 : 0;  // blocks of this chain
      // Both MMA warps see every phase of q_full, also in a segment in which their chain has no block: a
      // parity wait must never be two phases behind its barrier.
      const bool q_here = nblk > 0 && mbar_wait(sm, &sm->q_full, seg & 1, a.dev_status);
      if (n_c > 0) {
        const int base = c ? base_b : base_a;
        bool go = q_here;
        const uint32_t q_lo = desc_lo(smem_u32(sm->q), 16);
        const uint32_t tmem_o = tmem + 256u + 128u * c;
        // S of block u of the chain: buffer u & 1
        auto issue_qk = [&](int u) -> bool {
          const int b = (base + u) & 1, w = (base + u) >> 1;
          if (!mbar_wait(sm, &sm->k_full[c][b], w & 1, a.dev_status)) return false;
          tc_fence_after();
          const uint32_t d = tmem + 128u * c + 64u * b;
          if (elect_one()) {
            mma_qk<kHalfBytes, kKvHalf>(d, q_lo, desc_lo(smem_u32(sm->k[c][b]), 16), a.idesc_qk);
            tc_commit(&sm->s_full[c][b]);  // the row threads wait for this one
            tc_commit(&sm->k_empty[c][b]);
          }
          __syncwarp();
          if (lane == 0) UTRACE(c == 0 ? 1 : 3, 2);
          return true;
        };
        // two S in flight before the first P is needed
        if (go) go = issue_qk(0);
        if (go && n_c > 1) go = issue_qk(1);
        for (int u = 0; u < n_c && go; ++u) {
          const int b = (base + u) & 1, w = (base + u) >> 1;
          if (!mbar_wait(sm, &sm->v_full[c][b], w & 1, a.dev_status)) break;
          if (!mbar_wait(sm, &sm->p_full[c][b], w & 1, a.dev_status)) break;
          // the first P.V of a segment overwrites O: the row threads must have read the previous segment's
          if (u == 0 && seg > 0 && !mbar_wait(sm, &sm->o_free, (seg - 1) & 1, a.dev_status)) break;
          if (lane == 0) UTRACE(c == 0 ? 1 : 3, 3);
          if (a.zero_tail) {
            // The tensor maps of this mode cover the whole cache, so a block that reaches past the last tree row has
            // fetched rows that may hold anything; their probabilities are exactly 0, but 0 * NaN is not: the rows are
            // cleared here (whole 128-byte rows of both halves: the swizzle stays inside a row), and the clearing is
            // made visible to the tensor core's reads.
            const int live = L + a.n - (blk_lo + 2 * u + c) * kBlockN;  // rows of this block that exist
            if (live < kBlockN) {
              uint4* vt = reinterpret_cast<uint4*>(sm->v[c][b]);
              for (int i = max(live, 0) * 8 + lane; i < kBlockN * 8; i += 32) {
                vt[i] = make_uint4(0u, 0u, 0u, 0u);
                vt[kKvHalf / 16 + i] = make_uint4(0u, 0u, 0u, 0u);
              }
              fence_async_smem();
              __syncwarp();
            }
          }
          tc_fence_after();
          const uint32_t pa = tmem + 128u * c + 64u * b;
          const uint32_t first = u > 0 ? 1u : 0u;
          if (elect_one()) {
            mma_pv(tmem_o, pa, desc_lo(smem_u32(sm->v[c][b]), kKvHalf), a.idesc_pv, first);
            if (kFineP) mma_pv(tmem_o, pa + 32u, desc_lo(smem_u32(sm->v[c][b]), kKvHalf), a.idesc_pv, 1u);
            tc_commit(&sm->v_empty[c][b]);
            tc_commit(&sm->pv_done[c]);
          }
          __syncwarp();
          if (lane == 0) UTRACE(c == 0 ? 1 : 3, 5);
          // S of block u+2 goes where P of block u lives.  tcgen05.mma operations issued by one thread
          // execute in issue order, so this QK^T cannot overtake the P.V just issued.
          if (u + 2 < n_c && !issue_qk(u + 2)) break;
        }
        if (elect_one()) tc_commit(&sm->all_done[c]);  // arrives when every MMA of this chain has completed
        __syncwarp();
      } else if (nblk > 0) {
        // A chain without blocks in this segment.  Its arrival must not overtake the completion of its own
        // previous segment (an asynchronous commit), nor run a phase ahead of the row threads: it waits
        // until they have taken the previous segment's accumulators.
        const bool go = q_here && (seg == 0 || mbar_wait(sm, &sm->o_free, (seg - 1) & 1, a.dev_status));
        if (go && lane == 0) mbar_arrive(&sm->all_done[c]);
      }
      __syncwarp();
    }
    if (kMode == kCluster) {  // the cluster barriers of the merge (see the row threads)
      cluster_wait();
      cluster_arrive_relaxed();
      cluster_wait();
      cluster_arrive_relaxed();
      cluster_wait();
    }
    if (threadIdx.x == 32) UTRACE(1, 9);
    pos = sg.next;
    ++seg_n; base_an += (nblk + 1) >> 1; base_bn += nblk >> 1;
    if (kStream && sm->abort_flag) break;
    }  // segments
    // A CTA that gives up must not leave while a tile it has requested is still on its way into its shared memory
    // (the next CTA on this SM could get that memory): the producers wait, with a bound of their own, for the last
    // tile requested into each stage.  (Whether its consumer has taken that phase or not, the parity test answers
    // when the bytes have landed.  Tiles requested earlier into the same stage landed before the stage was reused.)
    if (sm->abort_flag && (warp == 0 || warp == 3)) {
      for (int st = 0; st < 5; ++st) {
        if (!((issued >> st) & 1u)) continue;
        uint64_t* full = st == 4 ? &sm->q_full : (warp == 3 ? &sm->v_full[st >> 1][st & 1] : &sm->k_full[st >> 1][st & 1]);
        for (uint32_t it = 0; it < (1u << 16); ++it)
          if (mbar_try_wait(full, (issued_parity >> st) & 1u)) break;
      }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
    return;
  }

  // ============================== warp groups 1, 2: one thread per query row of chain A, B ============
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsRows));
  const int chain = (warp >> 2) - 1;
  const int quad = warp & 3;                  // tensor-memory lane quarter this warp may access
  const int r = quad * 32 + lane;             // row of the tile = tensor-memory lane
  const uint32_t lane_sel = (uint32_t)(quad * 32) << 16;
  const uint32_t tmem_o = tmem + 256u + 128u * chain + lane_sel;
  int seg_n = 0, base_n = 0;  // segments done; blocks this chain has processed in them
  for (int pos = range_lo; pos < range_hi;) {
  const Seg sg = seg_at(pos);
  if (kStream && sg.nblk == 0) { pos = sg.next; continue; }
  const int g = sg.g, i0 = sg.i0, blk_lo = sg.blk_lo, nblk = sg.nblk;
  const int seg = kStream ? seg_n : 0, base = kStream ? base_n : 0;  // grid mode: constants
  const int i = i0 + r / a.group;             // node of this row
  const int h = g * a.group + r % a.group;
  const bool row_valid = i < sg.i1;           // (a row past the tile's nodes may be one of the next tile's)
  // The row's ancestor bits: the caller's mask, or rows derived from the parent array at the start of the
  // segment by the first thread of each node (0 <= parent[j] < j, so a walk ends; anything else is flagged and
  // read as "no parent").  In grid mode the row threads are idle at this point, waiting for the first tiles.
  // (The previous segment's rows are out of use: every row thread has passed that segment's merge barrier.)
  if (a.mask_bits == nullptr && (blk_lo + nblk) * kBlockN > L) {  // (a segment of prefix keys alone needs none)
    if (chain == 0 && r % a.group == 0) {
      uint32_t* row = sm->tile_mask[r / a.group];
      const int wpr = (a.n + 31) >> 5;
      for (int w = 0; w < wpr; ++w) row[w] = 0u;  // (nodes past the last one see no tree key)
      int j = i;
      for (int step = 0; step < a.n && row_valid; ++step) {
        row[j >> 5] |= 1u << (j & 31);
        const int pj = sm->parent[j];
        if (pj == -1) break;
        if (pj < -1 || pj >= j) { dev_flag(a.dev_status, SEQ_DEV_BAD_PARENT); break; }
        j = pj;
      }
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
  }
  const uint32_t* mrow = a.mask_bits != nullptr ? a.mask_bits + (size_t)min(i, a.n - 1) * a.mask_wpr : sm->tile_mask[r / a.group];
  const int mask_wpr = a.mask_bits != nullptr ? a.mask_wpr : (a.n + 31) >> 5;
  const float sc = a.scale_log2;

  float m_used = -INFINITY, l = 0.f;
  bool ok = true;
  const int n_mine = nblk > chain ? (nblk - chain + 1) >> 1 : 0;  // blocks of this chain
  // A warp whose 32 rows all lie past the tile's last node (small trees fill only part of a 128-row tile) leaves
  // the special-function unit and the issue slots to the warps with real rows; its P rows stay whatever they are
  // (rows of the product are independent).
  const bool warp_live = i0 + (quad * 32) / a.group < sg.i1;
  for (int u = 0; u < n_mine && ok; ++u) {
    const int jj = 2 * u + chain, b = (base + u) & 1, w = (base + u) >> 1;
    const uint32_t tmem_s = tmem + 128u * chain + 64u * b + lane_sel;
    if (!mbar_wait(sm, &sm->s_full[chain][b], w & 1, a.dev_status)) { ok = false; break; }
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 1);
    if (!warp_live) {  // 32 padding rows: nothing to compute, only keep in step with the barriers
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm->p_full[chain][b]);
      continue;
    }
    tc_fence_after();
    uint32_t sreg[64];
    tmem_ld32(tmem_s, sreg, 0);
    tmem_ld32(tmem_s + 32u, sreg, 32);
    const int kb = (blk_lo + jj) * kBlockN;
    const bool masked = kb + kBlockN > L;  // the block reaches into the tree keys (or past the end)
    uint32_t vis[2] = {0xFFFFFFFFu, 0xFFFFFFFFu};
    if (masked) {
      vis[0] = mask_window(mrow, mask_wpr, a.n, kb - L);
      vis[1] = mask_window(mrow, mask_wpr, a.n, kb - L + 32);
    }
    tc_wait_ld();
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 2);
    if (masked) {  // masked scores become -inf: probability exactly 0, and they cannot raise the maximum
#pragma unroll
      for (int e = 0; e < 64; ++e)
        if (!(vis[e >> 5] & (1u << (e & 31)))) sreg[e] = __float_as_uint(-INFINITY);
    }
    // P = 2^(scale*s - m) written over S as packed 16-bit values (32 columns, two stores of 16; with kFineP the rests in the
    // 32 columns behind); returns the row sum.
    // (A row without a reference sees nothing in this block: its scores are all -inf and its P are 0.)
    auto exponentials = [&]() -> float {
      const float neg_m = m_used == -INFINITY ? 0.f : -m_used;
      const uint64_t sc2 = pair_of(sc, sc), neg_m2 = pair_of(neg_m, neg_m);
      uint64_t sm2[2] = {pair_of(0.f, 0.f), pair_of(0.f, 0.f)};
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t packed[16], rest[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {  // two scores at a time: one packed multiply-add, two exponentials, one packed add
          float x0, x1;
          unpair(fma2(pair_of(__uint_as_float(sreg[32 * c + 2 * e]), __uint_as_float(sreg[32 * c + 2 * e + 1])), sc2, neg_m2), x0, x1);
          const float p0 = ex2(x0), p1 = ex2(x1);
          sm2[e & 1] = add2(sm2[e & 1], pair_of(p0, p1));
          packed[e] = pack2<kBf16>(p0, p1);
          if (kFineP) rest[e] = pack_rest<kBf16>(p0, p1, packed[e]);
        }
        tmem_st16(tmem_s + 16u * c, packed);
        if (kFineP) tmem_st16(tmem_s + 32u + 16u * c, rest);
      }
      float s0, s1, s2, s3;
      unpair(sm2[0], s0, s1);
      unpair(sm2[1], s2, s3);
      return (s0 + s1) + (s2 + s3);
    };
    // The reference maximum only moves when the block maximum exceeds it by more than the threshold, or when the row
    // has no reference yet: rare after the first blocks.  So the exponentials are taken against the reference as it
    // stands, and their sum tells whether that was right: a score more than the threshold above the reference gives a
    // term, hence a sum, above 2^threshold.  Only then (or without a reference) is the block maximum taken, the
    // reference moved, O rescaled, and the pass repeated (the scores are still in registers).
    float alpha = 1.f, sum;
    bool settle = __any_sync(0xffffffffu, m_used == -INFINITY);
#pragma unroll 1
    for (;;) {  // (a loop, so that the exponentials' code exists once)
      if (settle) {
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int e = 0; e < 64; e += 2)  // three-input maximum: two scores per instruction
          mx[(e >> 1) & 3] = max3(mx[(e >> 1) & 3], __uint_as_float(sreg[e]), __uint_as_float(sreg[e + 1]));
        const float m_blk = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sc;  // scale > 0
        const bool move = m_blk > m_used + kRescaleThreshold || (m_used == -INFINITY && m_blk != -INFINITY);
        if (__any_sync(0xffffffffu, move)) {
          if (move) {
            alpha = m_used == -INFINITY ? 0.f : ex2(m_used - m_blk);
            m_used = m_blk;
          }
          if (u > 0) {
            // O may still be taking the chain's previous block: wait for it, then rescale this warp's rows
            if (!mbar_wait(sm, &sm->pv_done[chain], (base + u - 1) & 1, a.dev_status)) { ok = false; break; }
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
              uint32_t o[32];
              tmem_ld32(tmem_o + 32u * c, o, 0);
              tc_wait_ld();
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
              tmem_st32(tmem_o + 32u * c, o, 0);
            }
          }
        }
      }
      sum = exponentials();
      if (settle) break;
      settle = __any_sync(0xffffffffu, !(sum <= kRescaleLimit));
      if (!settle) break;
    }
    if (!ok) break;
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 3);
    l = l * alpha + sum;
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 4);
    tc_wait_st();
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 12);
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm->p_full[chain][b]);  // one arrival per warp
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 5);
  }
  // Both chains must be done with the tensor pipe before O is read and the K stages are reused.  (A
  // parity wait on pv_done could be fooled here: the other chain may be several phases behind.)
  if (nblk > 0 && ok) ok = mbar_wait(sm, &sm->all_done[0], seg & 1, a.dev_status) && mbar_wait(sm, &sm->all_done[1], seg & 1, a.dev_status);
  tc_fence_after();

  // ---------------------------------------------------------------- merge ------------------------
  // Step 1, inside the CTA: both accumulators live in this CTA's tensor memory and a warp may read
  // any column of its 32 lanes, so the thread of chain c and row r merges columns [64c, 64c+64) of
  // O_A and O_B itself; only (m, l) goes through shared memory.
  if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 6);
  sm->ml_chain[seg & 1][chain][r] = (ok && n_mine > 0) ? make_float2(m_used, l) : make_float2(-INFINITY, 0.f);
  // Whether to stop after this segment is decided once for all row threads: a flag raised between two threads' own
  // reads would send some to the closing barrier and the rest into the next segment's bar.sync, which has no bound.
  if (kStream && threadIdx.x == 128) sm->abort_seen[seg & 1] = sm->abort_flag;
  asm volatile("bar.sync 1, 256;" ::: "memory");  // the 256 row threads only
  const bool stop_here = kStream && sm->abort_seen[seg & 1] != 0;
  float M, Lc;           // reference maximum and denominator of the CTA's merged partial
  float merged[64];      // its columns [64*chain, 64*chain + 64), unnormalised
  {
    const float2 mlA = sm->ml_chain[seg & 1][0][r], mlB = sm->ml_chain[seg & 1][1][r];
    M = fmaxf(mlA.x, mlB.x);
    const float fA = mlA.x == -INFINITY ? 0.f : ex2(mlA.x - M), fB = mlB.x == -INFINITY ? 0.f : ex2(mlB.x - M);
    Lc = mlA.y * fA + mlB.y * fB;
    if (kMode == kCluster) {
      __syncwarp();
      cluster_wait();  // every CTA of the cluster runs
      if (chain == 0 && row_valid) {
        const uint32_t to = smem_u32(&sm->ml_cta[split][r]);
        for (int q = 0; q < a.splits; ++q) st_cluster2(remote_smem(to, q), M, Lc);
      }
      __syncwarp();
      cluster_arrive_release();
    }
    const uint32_t oA = tmem + 256u + lane_sel + 64u * chain, oB = oA + 128u;
    uint64_t* m2 = reinterpret_cast<uint64_t*>(merged);
    if (nblk > 0 && ok) {
      tmem_ld32(oA, reinterpret_cast<uint32_t*>(merged), 0);
      tmem_ld32(oA + 32u, reinterpret_cast<uint32_t*>(merged), 32);
      tc_wait_ld();
      const uint64_t f2 = pair_of(fA, fA);
#pragma unroll
      for (int e = 0; e < 32; ++e) m2[e] = mul2(m2[e], f2);
    } else {
#pragma unroll
      for (int e = 0; e < 64; ++e) merged[e] = 0.f;
    }
    if (nblk > 1 && ok) {  // (a segment of one block has left O_B alone)
      uint32_t o[64];
      tmem_ld32(oB, o, 0);
      tmem_ld32(oB + 32u, o, 32);
      tc_wait_ld();
      const uint64_t f2 = pair_of(fB, fB);
#pragma unroll
      for (int e = 0; e < 32; ++e) m2[e] = fma2(pair_of(__uint_as_float(o[2 * e]), __uint_as_float(o[2 * e + 1])), f2, m2[e]);
    }
  }
  // both accumulators are in registers: the next segment's first P.V may overwrite them
  if (kStream) {
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm->o_free);
  }
  uint8_t* out_row = reinterpret_cast<uint8_t*>(a.out) + 2 * ((int64_t)i * a.o_stride_tok + (int64_t)h * a.o_stride_head);
  if (kStream && nblk < sg.nblk_tile) {
    // A piece of a tile (stream mode).  Every piece is written to this CTA's slot of the workspace (slot 0
    // if the piece opens the CTA's range, else 1), then counted; the CTA whose count completes the tile
    // adds the other pieces to its own and writes the output.  Nobody waits for anybody.
    // positions of the tile's blocks in the layout, and the CTAs whose ranges hold some of them
    const int t0 = g * blocks_per_head + sm->tile_prefix[sg.slot_in_head] + kStreamTileCost, t1 = t0 + sg.nblk_tile;
    int c_first = min((int)((float)t0 / (float)total_blocks * (float)gridDim.x), (int)gridDim.x - 1);  // the CTA whose range holds block t0 ...
    while (cta_lo(c_first + 1) <= t0) ++c_first;                      // ... exactly
    while (cta_lo(c_first) > t0) --c_first;
    int c_last = c_first;
    while (cta_lo(c_last + 1) < t1) ++c_last;
    const int my_slot = 2 * (int)blockIdx.x + (max(t0, range_lo) == range_lo ? 0 : 1);
    int* cnt = a.ws_count + (size_t)g * a.tiles + sg.tile;
    const int parts = c_last - c_first + 1;
    // If every other piece has been counted already (the usual case for the piece that closes a range: the
    // others were finished long ago), this CTA completes the tile without writing its own piece.
    if (threadIdx.x == 128) {
      const int done = *reinterpret_cast<volatile int*>(cnt) == parts - 1;
      if (done) *cnt = 0;  // leave the counter as it was found
      sm->last_part = done;
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (!sm->last_part) {
      if (chain == 0) a.ws_ml[(size_t)my_slot * kTileM + r] = make_float2(M, Lc);
      float4* my_o = a.ws_o + ((size_t)(my_slot * 2 + chain) * 16) * kTileM + r;
#pragma unroll
      for (int j = 0; j < 16; ++j) my_o[(size_t)j * kTileM] = make_float4(merged[4 * j], merged[4 * j + 1], merged[4 * j + 2], merged[4 * j + 3]);
      __threadfence();
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (threadIdx.x == 128) {
        const int last = atomicAdd(cnt, 1) == parts - 1;
        if (last) *cnt = 0;  // every piece has been counted
        sm->last_part = last;
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
    }
    if (sm->last_part) {
      // The pieces are added in the order of their CTAs, this CTA's own (from registers) at its place, with one
      // common reference maximum: the result does not depend on which CTA happened to finish last.
      __threadfence();
      auto slot_of = [&](int c) { return 2 * c + (max(t0, cta_lo(c)) == cta_lo(c) ? 0 : 1); };
      float Mg = M;
      for (int c = c_first; c <= c_last; ++c)
        if (c != (int)blockIdx.x) Mg = fmaxf(Mg, __ldcg(a.ws_ml + (size_t)slot_of(c) * kTileM + r).x);
      float Ls = 0.f;
#pragma unroll
      for (int half = 0; half < 2; ++half) {  // 32 columns at a time: the own piece must stay until its turn
        float acc[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) acc[e] = 0.f;
        for (int c = c_first; c <= c_last; ++c) {
          if (c == (int)blockIdx.x) {
            const float f = M == -INFINITY ? 0.f : ex2(M - Mg);
#pragma unroll
            for (int e = 0; e < 32; ++e) acc[e] = fmaf(merged[32 * half + e], f, acc[e]);
            if (half == 0) Ls = fmaf(Lc, f, Ls);
          } else {
            const int slot = slot_of(c);
            const float2 ml = __ldcg(a.ws_ml + (size_t)slot * kTileM + r);
            const float f = ml.x == -INFINITY ? 0.f : ex2(ml.x - Mg);
            const float4* its = a.ws_o + ((size_t)(slot * 2 + chain) * 16 + 8 * half) * kTileM + r;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float4 x = __ldcg(its + (size_t)j * kTileM);
              acc[4 * j] = fmaf(x.x, f, acc[4 * j]);
              acc[4 * j + 1] = fmaf(x.y, f, acc[4 * j + 1]);
              acc[4 * j + 2] = fmaf(x.z, f, acc[4 * j + 2]);
              acc[4 * j + 3] = fmaf(x.w, f, acc[4 * j + 3]);
            }
            if (half == 0) Ls = fmaf(ml.y, f, Ls);
          }
        }
#pragma unroll
        for (int e = 0; e < 32; ++e) merged[32 * half + e] = acc[e];
      }
      M = Mg;
      Lc = Ls;
    }
  }
  if (kStream && nblk < sg.nblk_tile && !sm->last_part) {
    // not the completing piece: nothing to write
  } else if (kMode != kCluster) {
    if (row_valid) {
      const float inv = 1.f / Lc;  // the row saw at least its own key, so Lc > 0
#pragma unroll
      for (int e = 0; e < 64; e += 8) {
        uint4 val;
        val.x = pack2<kBf16>(merged[e] * inv, merged[e + 1] * inv);
        val.y = pack2<kBf16>(merged[e + 2] * inv, merged[e + 3] * inv);
        val.z = pack2<kBf16>(merged[e + 4] * inv, merged[e + 5] * inv);
        val.w = pack2<kBf16>(merged[e + 6] * inv, merged[e + 7] * inv);
        *reinterpret_cast<uint4*>(out_row + 2 * (64 * chain + e)) = val;
      }
      if (chain == 0 && a.lse != nullptr) a.lse[(size_t)h * a.n + i] = (M + log2f(Lc)) * kLn2;
    }
  } else {
    // Step 2, across the cluster (cs = 2 .. 8 CTAs along the key range).  The 16 slices of 8 output columns are owned
    // round-robin: slice s by CTA s % cs, as its slot s / cs.  An owner receives into its K and V stages (adjacent in
    // shared memory: cs * ceil(16 / cs) * 4 KB <= 84 KB of their 128 KB), as float4 planes [contributor][slot][half][row].
    const int cs = a.splits, slots = (int)((15u + (uint32_t)cs) / (uint32_t)cs);  // (any cs from 2 to 8; the last slots of some CTAs may be empty)
    cluster_wait();  // every CTA's (m, l) is here, and every CTA is done with its K and V stages
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 7);
    float Mg = -INFINITY;
    for (int q = 0; q < cs; ++q) Mg = fmaxf(Mg, sm->ml_cta[q][r].x);
    float Ls = 0.f;
    for (int q = 0; q < cs; ++q) {
      const float2 mlq = sm->ml_cta[q][r];
      if (mlq.x != -INFINITY) Ls += mlq.y * ex2(mlq.x - Mg);
    }
    const uint32_t recv = smem_u32(&sm->k[0][0][0]);
    // (rows past the tile's last node are padding: nothing of theirs is pushed, reduced or stored)
    if (row_valid) {
      const float f = M == -INFINITY ? 0.f : ex2(M - Mg) / Ls;  // some CTA saw the row's own key, so Ls > 0
      const uint64_t f2 = pair_of(f, f);
      uint64_t* m2 = reinterpret_cast<uint64_t*>(merged);
#pragma unroll
      for (int e = 0; e < 32; ++e) m2[e] = mul2(m2[e], f2);
      int slot = (int)(8u * (uint32_t)chain / (uint32_t)cs), owner = 8 * chain - slot * cs;
      const uint32_t to = recv + 16u * (uint32_t)(split * slots * 2 * kTileM + r);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t dst = remote_smem(to + 16u * (uint32_t)(slot * 2 * kTileM), owner);
        st_cluster4(dst, merged + 8 * j);
        st_cluster4(dst + 16u * kTileM, merged + 8 * j + 4);
        if (++owner == cs) { owner = 0; ++slot; }
      }
    }
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 13);
    __syncwarp();
    cluster_arrive_release();
    cluster_wait();
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 8);
    const ulonglong2* mine = reinterpret_cast<const ulonglong2*>(&sm->k[0][0][0]) + r;
    if (row_valid)
      for (int slot = chain; slot * cs + split < 16; slot += 2) {  // the two warp groups share this CTA's slots
        const ulonglong2* src = mine + slot * 2 * kTileM;
        ulonglong2 x = src[0], y = src[kTileM];
        for (int q = 1; q < cs; ++q) {
          src += slots * 2 * kTileM;
          const ulonglong2 u = src[0], v = src[kTileM];
          x.x = add2(x.x, u.x); x.y = add2(x.y, u.y); y.x = add2(y.x, v.x); y.y = add2(y.y, v.y);
        }
        float o[8];
        unpair(x.x, o[0], o[1]); unpair(x.y, o[2], o[3]); unpair(y.x, o[4], o[5]); unpair(y.y, o[6], o[7]);
        uint4 val;
        val.x = pack2<kBf16>(o[0], o[1]);
        val.y = pack2<kBf16>(o[2], o[3]);
        val.z = pack2<kBf16>(o[4], o[5]);
        val.w = pack2<kBf16>(o[6], o[7]);
        *reinterpret_cast<uint4*>(out_row + 2 * (8 * (slot * cs + split))) = val;
      }
    if (split == 0 && chain == 0 && row_valid && a.lse != nullptr) a.lse[(size_t)h * a.n + i] = (Mg + log2f(Ls)) * kLn2;
  }
  if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 9);
  pos = sg.next;
  ++seg_n; base_n += n_mine;
  if (stop_here) break;
  }  // segments
#ifdef SEQ_TRACE
  if (threadIdx.x == 128 && cta_lin < 1024) g_cta_times[cta_lin][1] = gtimer();
#endif
  // no remote access happens after the last cluster barrier, so CTAs may leave independently
  tc_fence_before();
  __syncthreads();  // pairs with warp group 0, whose MMA warp then frees the tensor memory
}

__global__ void zero_words_kernel(int32_t* words, int n) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) words[i] = 0;
}

// ---------------------------------------------------------------- host side ---------------------
bool umma_supported(const seq_tree_attention_params& p) {
  if (p.dtype != SEQ_F16 && p.dtype != SEQ_BF16) return false;
  return p.num_q_heads / p.num_kv_heads <= kTileM;  // a tile holds at least one node's group of heads
}

// How the tiles are spread over the SMs.  Grid schedule: one CTA (or a cluster of `splits` CTAs along the key
// range) per (tile, kv head), in as many waves as that takes.  Stream schedule: one CTA per SM, each with an equal range of the
// flattened block space and share the tiles that a range boundary cuts.  p.kernel = 3 / 4 force one of them.
struct UmmaPlan { int splits; bool stream; };
constexpr size_t kUmmaSmemBytes = sizeof(UmmaSmem) + 1024;
// Clusters of cs CTAs that the device runs at a time (one CTA fills an SM).  Asked once per device and size; without a
// device, or where the question fails, what the SMs would hold.
static int clusters_side_by_side(int cs) {
  const int sms = device_sm_count();
  if (cs == 1) return sms;
  static int known[kMaxClusterSplit + 1][64];  // + 1; 0 = not asked yet
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return sms / cs; }
  n = __atomic_load_n(&known[cs][dev], __ATOMIC_ACQUIRE);
  if (n == 0) {
    auto kernel = tree_attention_umma_kernel<true, kCluster, false>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1, 1, cs);
    cfg.blockDim = dim3(kUmmaThreads);
    cfg.dynamicSmemBytes = kUmmaSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = cs;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kUmmaSmemBytes) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = sms / cs;
    }
    ++n;
    __atomic_store_n(&known[cs][dev], n, __ATOMIC_RELEASE);
  }
  return n - 1;
}
static UmmaPlan umma_plan(const seq_tree_attention_params& p) {
  const int G = p.num_q_heads / p.num_kv_heads;
  const int nodes_per_tile = kTileM / G;
  const int tiles = (p.n_tree + nodes_per_tile - 1) / nodes_per_tile;
  const long units = (long)tiles * p.num_kv_heads;
  const int nblk = (p.prefix_len + p.n_tree + kBlockN - 1) / kBlockN;
  // (a range of the stream schedule crosses kv heads: one length; positions are 32-bit)
  const bool can_stream = tiles <= kMaxStreamTiles && p.prefix_len_dev_count <= 1 && (double)units * (nblk + kStreamTileCost) < 2147483648.0;
  const int kNumSMs = device_sm_count();
#ifdef SEQ_TRACE
  if (const char* e = getenv("SEQ_DEBUG_SPLITS")) return {atoi(e), false};  // debug builds only
#endif
  if (p.kernel == 3 && can_stream) return {1, true};
  // More units than SMs.  Measured over batches of the paper's shapes (5 to 32 requests stacked as heads): plain
  // waves of one CTA per unit win by 5-50 % when tiles are short (a tile cut by a range boundary costs a trip
  // through the workspace, and every CTA starts and finishes two tiles more), the stream schedule wins by 5-15 %
  // when tiles are long (72 blocks and more) or when the last wave would be at most 60 % full.
  if (p.kernel != 4 && can_stream && units > kNumSMs) {
    const long waves = (units + kNumSMs - 1) / kNumSMs;
    const bool last_wave_thin = units * 10 <= waves * kNumSMs * 6;
    if (nblk >= 32 && (last_wave_thin || nblk >= 72)) return {1, true};
  }
  // Otherwise the split with the lowest estimate.  Microseconds per wave, fitted to launches of 72 shapes (8 to 768 nodes,
  // prefixes of 100 to 8000 keys, 8 to 384 units) with every split forced: 0.45 per block of a CTA's key range, 4.7 fixed,
  // and the merge across the cluster, which grows with the pieces that an owner's threads add up one after the other
  // (ceil(ceil(16 / cs) / 2) * cs, hence 4 below 3).  What a wave holds is asked of the device: a cluster lies in one
  // GPC, so the SMs left over in each are lost to it (74, 44, 36, 28, 21, 14 and 14 clusters of 2 to 8 CTAs were seen, where
  // 148 / cs had been assumed; 24 units of 17 blocks 17.3 -> 10.1 us, 16 of 48 21.8 -> 12.5, 48 of 66 34.7 -> 23.3).
  static const double kMerge[kMaxClusterSplit + 1] = {0.0, 0.0, 2.25, 3.2, 2.8, 3.5, 3.8, 4.2, 4.2};
  int best = 1;
  double best_cost = -1.0;
  for (int cs = 1; cs <= kMaxClusterSplit && cs <= nblk; ++cs) {
    const int room = clusters_side_by_side(cs);
    if (room == 0) continue;
    const long waves = (units + room - 1) / room;
    const double cost = (double)waves * (0.45 * ((nblk + cs - 1) / cs) + 4.7 + kMerge[cs]);
    if (best_cost < 0 || cost < best_cost - 1e-9) { best = cs; best_cost = cost; }
  }
  return {best, false};
}

int umma_default_splits(const seq_tree_attention_params& p) { return umma_plan(p).splits; }

static bool umma_stream_mode(const seq_tree_attention_params& p, int splits) {
  (void)splits;
  return umma_plan(p).stream;
}

// Workspace of the stream mode: one arrival counter per (kv head, tile), then two slots per CTA for the
// pieces of tiles that its range cuts: (m, l) per row and the 128 x 128 fp32 accumulator.
static size_t stream_count_bytes(const seq_tree_attention_params& p) {
  const int G = p.num_q_heads / p.num_kv_heads;
  const int nodes_per_tile = kTileM / G;
  const int tiles = (p.n_tree + nodes_per_tile - 1) / nodes_per_tile;
  return ((size_t)tiles * p.num_kv_heads * sizeof(int32_t) + 255) & ~(size_t)255;
}
static size_t stream_ml_bytes() { return (size_t)2 * device_sm_count() * kTileM * sizeof(float2); }
static size_t stream_o_bytes() { return (size_t)2 * device_sm_count() * 2 * 16 * kTileM * sizeof(float4); }

size_t umma_workspace_bytes(const seq_tree_attention_params& p) {
  if (!umma_stream_mode(p, umma_default_splits(p))) return 0;
  return stream_count_bytes(p) + stream_ml_bytes() + stream_o_bytes();
}

int launch_attention_umma(const seq_tree_attention_params& p, int splits, cudaStream_t stream) {
  const int G = p.num_q_heads / p.num_kv_heads;
  const int nodes_per_tile = kTileM / G;
  const int tiles = (p.n_tree + nodes_per_tile - 1) / nodes_per_tile;
  const CUtensorMapDataType dt = p.dtype == SEQ_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;

  CUtensorMap q_map, k_map, v_map;
  {
    // q viewed as [kv head][node][head in group][head_dim]
    // head_dim is split into its two 64-element halves (a dimension of its own, 128 bytes apart) so that one copy
    // brings the tile as [half][row][64 elements], the layout of two 128-byte-swizzled sub-tiles
    cuuint64_t dims[5] = {64, (cuuint64_t)G, (cuuint64_t)p.n_tree, 2, (cuuint64_t)p.num_kv_heads};
    cuuint64_t strides[4] = {(cuuint64_t)p.q_stride_head * 2, (cuuint64_t)p.q_stride_tok * 2, 128,
                             (cuuint64_t)p.q_stride_head * 2 * G};
    cuuint32_t box[5] = {64, (cuuint32_t)G, (cuuint32_t)nodes_per_tile, kTileM % G == 0 ? 2u : 1u, 1};  // (see load_q)
    if (!tensor_map(&q_map, dt, 5, p.q, dims, strides, box)) return SEQ_ERR_CUDA;
  }
  for (int which = 0; which < 2; ++which) {
    // only the live rows [0, prefix_len + n_tree) are mapped: anything past them reads as zero.  (With the prefix
    // length in device memory the map cannot end there: it covers the cache, and the kernel clears the tail rows.)
    cuuint64_t dims[4] = {64, (cuuint64_t)(p.prefix_len_dev != nullptr ? p.kv_capacity : p.prefix_len + p.n_tree), 2, (cuuint64_t)p.num_kv_heads};
    cuuint64_t strides[3] = {(cuuint64_t)p.kv_stride_tok * 2, 128, (cuuint64_t)p.kv_stride_head * 2};
    cuuint32_t box[4] = {64, (cuuint32_t)kBlockN, 2, 1};
    if (!tensor_map(which == 0 ? &k_map : &v_map, dt, 4, which == 0 ? p.k_cache : p.v_cache, dims, strides, box)) return SEQ_ERR_CUDA;
  }

  UmmaArgs a;
  a.n = p.n_tree; a.L_host = p.prefix_len; a.Hq = p.num_q_heads; a.Hkv = p.num_kv_heads; a.group = G;
  a.mask_wpr = p.mask_words_per_row; a.splits = splits; a.nodes_per_tile = nodes_per_tile; a.tiles = tiles;
  a.rows = nodes_per_tile * G;
  const float scale = p.softmax_scale > 0.f ? p.softmax_scale : 0.08838834764831845f;
  a.scale_log2 = scale * kLog2e;
  const uint32_t fmt = p.dtype == SEQ_BF16 ? 1u : 0u;
  // instruction descriptor: D fp32 (bit 4), A/B format (bits 7, 10), B major (bit 16), N>>3 (bit 17), M>>4 (bit 24)
  const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(kTileM >> 4) << 24);
  a.idesc_qk = idesc | ((uint32_t)(kBlockN >> 3) << 17);                 // S: N = 64 keys
  a.idesc_pv = idesc | ((uint32_t)(kHeadDim >> 3) << 17) | (1u << 16);   // O: N = 128, V is MN-major
  a.mask_bits = p.mask_bits;
  a.parent = p.parent;
  a.out = p.out; a.o_stride_tok = p.o_stride_tok; a.o_stride_head = p.o_stride_head;
  a.lse = p.lse;
  a.dev_status = p.dev_status;
  a.stream = umma_stream_mode(p, splits) ? 1 : 0;
  a.blocks_per_head_host = 0; a.total_blocks_host = 0;
  a.L_dev = p.prefix_len_dev; a.L_count = p.prefix_len_dev_count; a.zero_tail = p.prefix_len_dev != nullptr ? 1 : 0;
  a.ws_count = nullptr; a.ws_ml = nullptr; a.ws_o = nullptr;
  const bool lent = p.workspace != nullptr && p.workspace_bytes >= stream_count_bytes(p) + stream_ml_bytes() + stream_o_bytes();
  // (groups that do not divide 128 used to run on the CUDA cores, which ask for nothing at these sizes: without a workspace
  // they take the grid schedule instead, 500 nodes on 4600 keys of 40/8 heads 99 us against 67)
  if (!lent && p.kernel == 0 && kTileM % G != 0) a.stream = 0;
  if (a.stream) {
    const size_t cnt_bytes = stream_count_bytes(p);
    if (!lent) return SEQ_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(p.workspace) % 256 != 0) return SEQ_ERR_INVALID_ARG;
    for (int t = 0; t < tiles; ++t) {
      const int i1 = (t + 1) * nodes_per_tile < p.n_tree ? (t + 1) * nodes_per_tile : p.n_tree;
      a.blocks_per_head_host += kStreamTileCost + (p.prefix_len + i1 + kBlockN - 1) / kBlockN;
    }
    a.total_blocks_host = a.blocks_per_head_host * p.num_kv_heads;
    uint8_t* ws = static_cast<uint8_t*>(p.workspace);
    a.ws_count = reinterpret_cast<int32_t*>(ws);
    a.ws_ml = reinterpret_cast<float2*>(ws + cnt_bytes);
    a.ws_o = reinterpret_cast<float4*>(ws + cnt_bytes + stream_ml_bytes());
    // The counters start at zero.  A kernel of one's own, not a memset: it is scheduled under the tail of the launch before
    // and lets the attention's set-up run under itself (768 nodes on 4096 keys of 64/8 heads 123.1 -> 120.8 us, 384 on 2048
    // of 52 heads 43.1 -> 40.9).
    cudaLaunchConfig_t zero = {};
    const int words = (int)(cnt_bytes / sizeof(int32_t));
    zero.gridDim = dim3((words + 255) / 256);
    zero.blockDim = dim3(256);
    zero.stream = stream;
    cudaLaunchAttribute early[1];
    early[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early[0].val.programmaticStreamSerializationAllowed = 1;
    zero.attrs = early;
    zero.numAttrs = 1;
    SEQ_CUDA_OK(cudaLaunchKernelEx(&zero, zero_words_kernel, a.ws_count, words));
  }

  const size_t smem = kUmmaSmemBytes;
  cudaLaunchConfig_t cfg = {};
  // Stream schedule: one CTA per SM, but never more CTAs than positions in the layout: a range must not be empty
  // (the CTAs that share a cut tile are counted from the ranges, and each of them has to arrive).
  const int sms = device_sm_count();
  const int stream_ctas = a.total_blocks_host < sms ? a.total_blocks_host : sms;
  cfg.gridDim = a.stream ? dim3(stream_ctas, 1, 1) : dim3(tiles, p.num_kv_heads, splits);
  cfg.blockDim = dim3(kUmmaThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = splits;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // start under the previous kernel's tail (see the kernel)
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  // An instantiation per element type, schedule and form of P.  None carries another's code: half of a short call's
  // instructions run once, at the rate at which they are fetched.
  auto launch = [&](auto kernel, int which) -> int {
    static int attr_done[12][64];  // the opt-in shared-memory size is set once per kernel and device
    const int rc = once_per_device(attr_done[which], [&]() -> int {
      SEQ_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      return SEQ_OK;
    });
    if (rc != SEQ_OK) return rc;
    SEQ_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, q_map, k_map, v_map, a));
    return SEQ_OK;
  };
  const int mode = a.stream ? kStreamed : splits > 1 ? kCluster : kGrid;
  auto launch_type = [&](auto bf16, auto fine, int first) -> int {
    constexpr bool kB = decltype(bf16)::value, kF = decltype(fine)::value;
    return mode == kStreamed ? launch(tree_attention_umma_kernel<kB, kStreamed, kF>, first)
           : mode == kCluster ? launch(tree_attention_umma_kernel<kB, kCluster, kF>, first + 1)
                              : launch(tree_attention_umma_kernel<kB, kGrid, kF>, first + 2);
  };
  const bool fine = kTileM % G != 0;
  if (p.dtype == SEQ_BF16) return fine ? launch_type(std::true_type(), std::true_type(), 6) : launch_type(std::true_type(), std::false_type(), 0);
  return fine ? launch_type(std::false_type(), std::true_type(), 9) : launch_type(std::false_type(), std::false_type(), 3);
}

}  // namespace seqtree
