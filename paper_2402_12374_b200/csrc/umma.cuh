// What the tensor-core attention kernels share: wrappers of the PTX they are made of, the tiles' layouts in shared memory and
// their descriptors, the packed arithmetic of the softmax, the windows of the ancestor mask.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace seqtree {

constexpr int kTileM = 128;         // query rows per CTA
constexpr int kBlockN = 64;         // keys per block
constexpr int kUmmaThreads = 384;   // warp group 0: TMA and MMA warps; warp groups 1, 2: one thread per query row each
constexpr int kRegsLight = 40, kRegsRows = 232;  // after setmaxnreg: 128*40 + 256*232 = 384*168
constexpr uint32_t kTileBytes = 128 * 128 * 2;   // the Q tile: 128 rows x 128 elements of 16 bits
constexpr uint32_t kHalfBytes = kTileBytes / 2;  // one 128-row x 64-element sub-tile of Q (128 B rows)
constexpr float kRescaleThreshold = 8.f;         // log2 units
constexpr float kRescaleLimit = 256.f;           // 2^kRescaleThreshold: no term of a row sum at or below it came from a score above the threshold
constexpr uint32_t kSpinLimit = 1u << 22;

// The stream schedule (tree_attention_stream.cu): the 64-key blocks of all (tile, kv head) units laid end to end, each tile
// preceded by kStreamTileCost positions for its fixed cost, and cut into a range for each SM.
constexpr int kMaxStreamTiles = 128;  // tiles per kv head the layout can index
constexpr int kStreamTileCost = 8;
size_t stream_workspace_bytes(const seq_tree_attention_params& p);
int launch_attention_stream(const seq_tree_attention_params& p, cudaStream_t stream);
// The tensor maps of a call: q as rows (node, head in group) of a kv head in two 64-element halves, K and V with `kv_halves`
// (1 or 2) of the two halves in a copy.
bool attention_maps(const seq_tree_attention_params& p, int kv_halves, CUtensorMap* q_map, CUtensorMap* k_map, CUtensorMap* v_map);

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

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
template <typename Smem>
__device__ __forceinline__ bool mbar_wait(Smem* sm, uint64_t* bar, uint32_t parity, int32_t* dev_status) {
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

}  // namespace seqtree
