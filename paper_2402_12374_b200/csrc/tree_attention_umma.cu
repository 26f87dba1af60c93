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
// Work distribution.  One CTA per (tile, kv head), in as many waves as that takes, or (up to one wave) a cluster of 2 to 8
// CTAs that split its key range; the thread that arms the barriers requests the Q tile and the first K tiles itself, before
// the CTA-wide barrier.  Many units of long tiles go to the kernel of tree_attention_stream.cu.
//
// Merge.  The CTAs that share (tile, kv head) form a thread-block cluster along the key range (cs = 1 .. 8).  Each sends
// its rows' (m, l) into every CTA as soon as its two chains are done, puts its piece into its V stages, slice by slice of 8
// output columns, and copies each owner its run of slices in one go (into the K stages: an MMA commit of
// every chain of the cluster says that no S is to come).  While the pieces travel each owner works out the rows' common
// maximum, sum and the pieces' shares; then it adds its slices up.  Both transfers count their bytes into an mbarrier of the
// receiver; the only cluster barriers are at the start and, off the path, at the end.  No workspace, no second kernel.  (With
// scaled pieces stored one by one and three cluster barriers, whose release waits for all of a warp's stores: 64 nodes on 1024
// keys of 32 heads 9.1 us instead of 8.5, 128 on 2048 of 40 13.8 / 13.3.)
//
// Most of the code around the loop over blocks runs once per launch, at the rate at which its instructions are fetched, so it
// is kept short: quotients as products, loops that are not unrolled (merge with shares in registers and the loop over
// contributors unrolled: 8.7 us).
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
#include <stdlib.h>

#include <type_traits>

#include "common.cuh"
#include "tensor_map.cuh"
#include "trace_attention.cuh"
#include "umma.cuh"

namespace cg = cooperative_groups;

namespace seqtree {

constexpr int kMaxClusterSplit = 8;
constexpr uint32_t kKvBytes = kBlockN * 128 * 2; // a K or V tile: 64 keys x 128 elements
constexpr uint32_t kKvHalf = kKvBytes / 2;       // one 64-row x 64-element sub-tile of K or V

// Tiles of up to so many rows store their output a row per thread, 16 bytes at a time; beyond, where every such store of a
// warp touches 32 lines, the way through shared memory is the shorter one.  (16 rows 5.3 us against 5.85, 64 rows 5.85 / 6.1, 80
// rows 4.85 / 5.05; 100 rows 6.85 / 6.7, 256 nodes on 2048 keys of 52 heads 23.2 / 22.35.)
constexpr uint32_t kDirectRows = 80;

struct UmmaSmem {
  // all tiles 1024-byte aligned (128-byte swizzle atoms are 8 rows x 128 B)
  uint8_t q[kTileBytes];
  uint8_t receive[20480];     // with the K stages behind it, once their S are done: the other CTAs' pieces (cluster merge)
  uint8_t k[2][2][kKvBytes];  // [chain][stage]
  uint8_t v[2][2][kKvBytes];  // [chain][stage]; after the last block: this CTA's piece (cluster merge)
  float2 ml_chain[2][kTileM];                // [chain]: (m, l) of every row of the two chains of this CTA
  float2 ml_cta[kMaxClusterSplit][kTileM];   // (m, l) of every row of every CTA of the cluster, after its chains are merged
  uint64_t q_full;
  uint64_t k_full[2][2], k_empty[2][2], v_full[2][2], v_empty[2][2], s_full[2][2], p_full[2][2];  // [chain][stage]
  uint64_t pv_done[2];                       // [chain]: one phase per block of the chain
  uint64_t all_done[2];                      // [chain]: every MMA of the chain has completed
  uint64_t k_free;                           // cluster merge: no chain of any CTA has an S to come, the K stages may be written
  uint64_t ml_full, data_full;               // ... and this CTA's ml_cta and pieces are here
  uint32_t tmem_base;
  volatile int abort_flag;
  // mask from the parent array: the tree, and the ancestor rows of the current tile's nodes (row stride 33 words)
  int32_t parent[SEQ_MAX_TREE];
  uint32_t tile_mask[kTileM][SEQ_MAX_TREE / 32 + 1];
};

static_assert(offsetof(UmmaSmem, k) == offsetof(UmmaSmem, receive) + sizeof(UmmaSmem::receive) && sizeof(UmmaSmem::receive) + sizeof(UmmaSmem::k) >= 7 * 3 * 4096,
              "the cluster merge receives cs * ceil(16 / cs) slices of 4 KB in one buffer");

struct UmmaArgs {
  int32_t n, L_host, Hq, Hkv, group, mask_wpr, splits, nodes_per_tile, tiles;
  int32_t rows;           // query rows of a full tile: nodes_per_tile * group, 128 when the group divides it
  const int32_t* L_dev;   // nullable: the prefix length in device memory (<= L_host)
  int32_t L_count;       // > 1: one length per request, requests stacked as heads (a CTA has one kv head)
  int32_t zero_tail;      // the K/V maps cover the whole cache: rows past the tree are cleared in shared memory
  // Quotients by the group and by the cluster's size as products: a division is 30 instructions and three trips through the
  // unit that also takes the exponentials.  (Together with the tree's way into shared memory, see below: 64 nodes on 1024 keys
  // of 32 heads 9.4 -> 9.1 us, 16 on 128 5.8 -> 5.4, 256 on 2048 of 52 23.2 -> 22.8.)
  uint32_t group_magic;   // x / group = x * group_magic >> 16 for x < 128
  uint32_t split_magic;   // x / splits = high word of x * split_magic for x < 2^29 (splits > 1)
  int32_t slots, slices_each, slices_more;  // ceil(16 / splits), 16 / splits, 16 % splits
  float scale_log2;
  uint32_t idesc_qk, idesc_pv;
  const uint32_t* mask_bits;
  const int32_t* parent;  // used when mask_bits is null
  void* out; int64_t o_stride_tok, o_stride_head;
  float* lse;
  int32_t* dev_status;
};

__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// The address of a shared-memory word of CTA `rank` of the cluster, and stores to it.
__device__ __forceinline__ uint32_t remote_smem(uint32_t addr, int rank) {
  uint32_t d;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
  return d;
}
// An asynchronous store of 8 bytes, and a copy of shared memory, to another CTA of the cluster; both count their bytes into an
// mbarrier there.
__device__ __forceinline__ void st_async2(uint32_t addr, float x, float y, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];"
               ::"r"(addr), "r"(__float_as_uint(x)), "r"(__float_as_uint(y)), "r"(bar) : "memory");
}
__device__ __forceinline__ void copy_to_cta(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
// Arrives on the mbarrier at the same place of every CTA in `mask` when the MMAs issued so far have completed.
__device__ __forceinline__ void tc_commit_cluster(uint64_t* bar, uint32_t mask) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)), "h"((uint16_t)mask) : "memory");
}
// Of the 16 slices of 8 output columns each CTA owns a run.
__device__ __forceinline__ int slices_of(int cta, const UmmaArgs& a) { return a.slices_each + (cta < a.slices_more); }
__device__ __forceinline__ int slices_before(int cta, const UmmaArgs& a) { return cta * a.slices_each + min(cta, a.slices_more); }
enum { kGrid, kCluster };  // the schedule: a CTA per unit, a cluster of CTAs per unit
// kFineP: P enters its product as two 16-bit pieces, the rounded value and the rest, each in a run of MMAs of its own.  For
// the groups of heads that do not divide 128, whose probabilities are held to single precision (the other groups round P
// to the input type).  Relative error of the output against fp64, 100 nodes on 1501 keys of 40/8 heads: 1.658e-3 in
// bfloat16 and 2.071e-4 in half, which is what rounding the exact output gives; with P rounded once 2.26e-3 and 2.82e-4.
// The second run costs that call 11.6 -> 12.7 us.
template <bool kBf16, int kMode, bool kFineP>
__global__ void __launch_bounds__(kUmmaThreads, 1)
tree_attention_umma_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                           const __grid_constant__ CUtensorMap v_map, const UmmaArgs a) {
  extern __shared__ uint8_t smem_raw[];
  // (An offset, not a rounded pointer: the compiler keeps seeing shared memory.  With generic accesses to barriers, mask
  // rows and the merge's pieces 64 nodes on 1024 keys of 32 heads take 9.8 us instead of 9.45, 256 on 2048 of 52 24.0 / 23.5,
  // 100 on 1501 of 40/8 12.0 / 11.65.)
  UmmaSmem* sm = reinterpret_cast<UmmaSmem*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
  const int warp = uniform((int)threadIdx.x >> 5), lane = threadIdx.x & 31;
#ifdef SEQ_TRACE
  int utrace_i = 0;
#endif
  const int split = kMode == kCluster ? blockIdx.z : 0;  // the cluster spans blockIdx.z
  if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 10);
#ifdef SEQ_TRACE
  const unsigned cta_lin = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  if (threadIdx.x == 128 && cta_lin < 1024) g_cta_times[cta_lin][0] = gtimer();
#endif

  // The prefix length: the host's, or - for a step replayed from one CUDA graph while the prefix grows - read from
  // device memory below (the host's value is then the largest it can be, which the launch was planned for).
  int L = a.L_host;
  const int g = blockIdx.y, i0 = blockIdx.x * a.nodes_per_tile, i1 = min(i0 + a.nodes_per_tile, a.n);  // kv head, the tile's nodes
  // The 64-key blocks of this CTA: all that the tile can see - its keys end at L + i1, a node sees no later node - or its share.
  int blk_lo, nblk;
  auto take_blocks = [&]() {
    const int all = (L + i1 + kBlockN - 1) / kBlockN;
    // (rounded up: the CTA of the last keys, which are masked, is not the one with a block more)
    blk_lo = kMode == kGrid ? 0 : (int)__umulhi((uint32_t)(split * all + a.splits - 1), a.split_magic);
    nblk = kMode == kGrid ? all : (int)__umulhi((uint32_t)((split + 1) * all + a.splits - 1), a.split_magic) - blk_lo;
  };
  take_blocks();
  // A stage barrier counts the blocks its chain has processed so far; q_full and all_done[] have one phase.
  const uint32_t live_rows = (uint32_t)((i1 - i0) * a.group);
  const uint32_t plane = ((live_rows + 31u) & ~31u) * 16u;  // cluster merge: bytes of four columns of all rows
  if (threadIdx.x == 0) {  // the barriers of the first loads, which this thread requests below
    mbar_init(&sm->q_full, 1);
    mbar_init(&sm->k_full[0][0], 1);
    mbar_init(&sm->k_full[1][0], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // programmatic dependent launch: the next kernel in the stream may be scheduled onto free SMs from now on (it
    // waits, as this one does below, before it touches memory); without the launch attribute this does nothing
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  if (threadIdx.x == 64) {  // all others
    for (int c = 0; c < 2; ++c) {
      mbar_init(&sm->k_full[c][1], 1);
      for (int b = 0; b < 2; ++b) {
        mbar_init(&sm->k_empty[c][b], 1);
        mbar_init(&sm->v_full[c][b], 1); mbar_init(&sm->v_empty[c][b], 1);
        mbar_init(&sm->s_full[c][b], 1); mbar_init(&sm->p_full[c][b], 4);
      }
      mbar_init(&sm->pv_done[c], 1);
      mbar_init(&sm->all_done[c], 1);  // one arriver: the chain's MMA warp
    }
    if (kMode == kCluster) { mbar_init(&sm->k_free, 2 * a.splits); mbar_init(&sm->ml_full, 1); mbar_init(&sm->data_full, 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (kMode == kCluster) {
      mbar_expect_tx(&sm->ml_full, (uint32_t)a.splits * live_rows * 8u);
      mbar_expect_tx(&sm->data_full, (uint32_t)(a.splits - 1) * (uint32_t)slices_of(split, a) * 2u * plane);
    }
    sm->abort_flag = 0;
  }
  if (kMode == kCluster) {  // "this CTA runs and its barriers count": waited for before anything is sent
    __syncwarp();
    cluster_arrive_relaxed();
  }
  // ... and everything above ran while the previous kernel in the stream was still finishing.  Nothing before this
  // line reads or writes global memory.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (a.L_dev != nullptr) {
    const int v = a.L_dev[a.L_count > 1 ? (g * a.L_count) / a.Hkv : 0];
    if (v < 0 || v > a.L_host) { if (threadIdx.x == 0) dev_flag(a.dev_status, SEQ_DEV_BAD_LENGTH); }
    L = uniform(min(max(v, 0), a.L_host));
    take_blocks();
  }
  // The thread that armed the barriers requests the Q tile and the first K tile of each chain right away, before the
  // CTA-wide barrier below and the hand-over to the producer warps (which skip what has been requested here).
  if (threadIdx.x == 0 && nblk > 0) {
    load_q(sm->q, &q_map, &sm->q_full, a.rows, i0, g);
    for (int jj = 0; jj < 2 && jj < nblk; ++jj) {
      mbar_expect_tx(&sm->k_full[jj][0], kKvBytes);
      tma_load_4d(sm->k[jj][0], &k_map, &sm->k_full[jj][0], 0, (blk_lo + jj) * kBlockN, 0, g);
    }
  }
  // The tree on its way to the row threads, which derive the ancestor rows from it (if the CTA's keys reach the tree's); they
  // put it into shared memory behind the CTA-wide barrier, which would otherwise wait for it.
  const bool derive = a.mask_bits == nullptr && (blk_lo + nblk) * kBlockN > L;
  int32_t tree[SEQ_MAX_TREE / 256];
  if (derive && warp >= 4) {
#pragma unroll
    for (int k = 0; k < SEQ_MAX_TREE / 256; ++k) {
      const int t = (int)threadIdx.x - 128 + 256 * k;
      tree[k] = t < a.n ? a.parent[t] : -1;
    }
  }
  if (a.rows < kTileM) {  // rows no copy writes (the group does not divide 128): zeros, so that their scores are finite
    for (int t = a.rows * 8 + (int)threadIdx.x; t < kTileM * 8; t += kUmmaThreads) {
      reinterpret_cast<uint4*>(sm->q)[t] = make_uint4(0u, 0u, 0u, 0u);
      reinterpret_cast<uint4*>(sm->q + kHalfBytes)[t] = make_uint4(0u, 0u, 0u, 0u);
    }
    fence_async_smem();
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
    uint32_t issued = 0, issued_parity = 0;   // producers: stages (bit 2*chain + stage) this warp has requested a tile for, and the phase of the last request
    if (warp == 0 || warp == 3) {
      // ---------------------------------------------------------- TMA producers -----------------
      // Warp 0 loads Q and the K tiles, warp 3 the V tiles.  A K stage is free as soon as its S has been
      // computed, a V stage only after the block's softmax and P.V; in one queue the K loads would wait
      // behind the V stages and arrive just in time instead of a block ahead.
      // The whole warp runs the loop; one elected lane issues the copies (coordinates stay warp-uniform).
      if (nblk > 0) {
        const bool is_v = warp == 3;
        const CUtensorMap* map = is_v ? &v_map : &k_map;
        for (int jj = is_v ? 0 : min(2, nblk); jj < nblk; ++jj) {
          const int c = jj & 1, b = (jj >> 1) & 1, w = jj >> 2;  // chain, stage, use count of the stage
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
      const bool q_here = nblk > 0 && mbar_wait(sm, &sm->q_full, 0, a.dev_status);
      if (kMode == kCluster) {
        __syncwarp();
        cluster_wait();
      }
      const uint32_t everyone = (1u << a.splits) - 1u;
      if (n_c > 0) {
        bool go = q_here;
        const uint32_t q_lo = desc_lo(smem_u32(sm->q), 16);
        const uint32_t tmem_o = tmem + 256u + 128u * c;
        // S of block u of the chain: buffer u & 1
        auto issue_qk = [&](int u) -> bool {
          const int b = u & 1, w = u >> 1;
          if (!mbar_wait(sm, &sm->k_full[c][b], w & 1, a.dev_status)) return false;
          tc_fence_after();
          const uint32_t d = tmem + 128u * c + 64u * b;
          if (elect_one()) {
            mma_qk<kHalfBytes, kKvHalf>(d, q_lo, desc_lo(smem_u32(sm->k[c][b]), 16), a.idesc_qk);
            tc_commit(&sm->s_full[c][b]);  // the row threads wait for this one
            tc_commit(&sm->k_empty[c][b]);
            if (kMode == kCluster && u + 1 == n_c) tc_commit_cluster(&sm->k_free, everyone);
          }
          __syncwarp();
          if (lane == 0) UTRACE(c == 0 ? 1 : 3, 2);
          return true;
        };
        // two S in flight before the first P is needed
        if (go) go = issue_qk(0);
        if (go && n_c > 1) go = issue_qk(1);
        for (int u = 0; u < n_c && go; ++u) {
          const int b = u & 1, w = u >> 1;
          if (!mbar_wait(sm, &sm->v_full[c][b], w & 1, a.dev_status)) break;
          if (!mbar_wait(sm, &sm->p_full[c][b], w & 1, a.dev_status)) break;
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
      } else if (lane == 0) {  // a chain without blocks
        if (nblk > 0) mbar_arrive(&sm->all_done[c]);
        if (kMode == kCluster)
          for (int q = 0; q < a.splits; ++q)
            asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(remote_smem(smem_u32(&sm->k_free), q)) : "memory");
      }
      __syncwarp();
    }
    if (kMode == kCluster) {  // (nobody leaves before every piece has arrived, see the row threads)
      __syncwarp();
      if (warp == 0 || warp == 3) cluster_wait();
      cluster_arrive_relaxed();
      cluster_wait();
    }
    if (threadIdx.x == 32) UTRACE(1, 9);
    // A CTA that gives up must not leave while a tile it has requested is still on its way into its shared memory
    // (the next CTA on this SM could get that memory): the producers wait, with a bound of their own, for the last
    // tile requested into each stage.  (Whether its consumer has taken that phase or not, the parity test answers
    // when the bytes have landed.  Tiles requested earlier into the same stage landed before the stage was reused.)
    if (sm->abort_flag && (warp == 0 || warp == 3)) {
      for (int st = 0; st < 4; ++st) {
        if (!((issued >> st) & 1u)) continue;
        uint64_t* full = warp == 3 ? &sm->v_full[st >> 1][st & 1] : &sm->k_full[st >> 1][st & 1];
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
  const int r_node = (int)((uint32_t)r * a.group_magic >> 16);
  const int i = i0 + r_node;                  // node of this row
  const int h = g * a.group + r - r_node * a.group;
  const bool row_valid = i < i1;           // (a row past the tile's nodes may be one of the next tile's)
  // The row's ancestor bits: the caller's mask, or rows derived from the parent array by the first thread of each node
  // (0 <= parent[j] < j, so a walk ends; anything else is flagged and read as "no parent"); the row threads are idle at
  // this point, waiting for the first tiles.
  if (derive) {  // (prefix keys alone need none)
#pragma unroll
    for (int k = 0; k < SEQ_MAX_TREE / 256; ++k) {
      const int t = (int)threadIdx.x - 128 + 256 * k;
      if (t < a.n) sm->parent[t] = tree[k];
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (chain == 0 && r == r_node * a.group) {
      uint32_t* row = sm->tile_mask[r_node];
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
  const uint32_t* mrow = a.mask_bits + (size_t)min(i, a.n - 1) * a.mask_wpr;  // (the caller's mask, if there is one)
  const int mask_wpr = a.mask_bits != nullptr ? a.mask_wpr : (a.n + 31) >> 5;
  const float sc = a.scale_log2;

  float m_used = -INFINITY, l = 0.f;
  bool ok = true;
  const int n_mine = nblk > chain ? (nblk - chain + 1) >> 1 : 0;  // blocks of this chain
  // A warp whose 32 rows all lie past the tile's last node (small trees fill only part of a 128-row tile) leaves
  // the special-function unit and the issue slots to the warps with real rows; its P rows stay whatever they are
  // (rows of the product are independent).
  const bool warp_live = (uint32_t)(quad * 32) < live_rows;
  for (int u = 0; u < n_mine && ok; ++u) {
    const int jj = 2 * u + chain, b = u & 1, w = u >> 1;
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
      // 64 bits of the row from tree index kb - L on; negative indices are prefix keys (visible)
      const int t = kb - L, w0 = t >> 5;  // (floor)
      uint32_t word[3];
#pragma unroll
      for (int x = 0; x < 3; ++x) word[x] = w0 + x < 0 ? 0xFFFFFFFFu : 0u;
      if (a.mask_bits != nullptr) {
#pragma unroll
        for (int x = 0; x < 3; ++x)
          if ((uint32_t)(w0 + x) < (uint32_t)mask_wpr) word[x] = mrow[w0 + x];
      } else {
#pragma unroll
        for (int x = 0; x < 3; ++x)
          if ((uint32_t)(w0 + x) < (uint32_t)mask_wpr) word[x] = sm->tile_mask[r_node][w0 + x];
      }
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int live = a.n - t - 32 * x;  // tree indices >= n do not exist, whatever the mask words hold there
        vis[x] = __funnelshift_r(word[x], word[x + 1], t & 31) & (live >= 32 ? 0xFFFFFFFFu : live <= 0 ? 0u : (1u << live) - 1u);
      }
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
            if (!mbar_wait(sm, &sm->pv_done[chain], (u - 1) & 1, a.dev_status)) { ok = false; break; }
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
      tc_wait_st();  // (for the hand-over below, and because a repeated pass stores other values to the same columns: stores to
                     // tensor memory are not ordered among themselves.  A wait of its own there: 2 us more for 32 layers)
      if (settle) break;
      settle = __any_sync(0xffffffffu, !(sum <= kRescaleLimit));
      if (!settle) break;
    }
    if (!ok) break;
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 3);
    l = l * alpha + sum;
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 4);
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 12);
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm->p_full[chain][b]);  // one arrival per warp
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 5);
  }
  // Both chains must be done with the tensor pipe before O is read and the K stages are reused.  (A
  // parity wait on pv_done could be fooled here: the other chain may be several phases behind.)
  if (nblk > 0 && ok) ok = mbar_wait(sm, &sm->all_done[0], 0, a.dev_status) && mbar_wait(sm, &sm->all_done[1], 0, a.dev_status);
  tc_fence_after();

  // ---------------------------------------------------------------- merge ------------------------
  // Step 1, inside the CTA: both accumulators live in this CTA's tensor memory and a warp may read
  // any column of its 32 lanes, so the thread of chain c and row r merges columns [64c, 64c+64) of
  // O_A and O_B itself; only (m, l) goes through shared memory.
  if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 6);
  sm->ml_chain[chain][r] = (ok && n_mine > 0) ? make_float2(m_used, l) : make_float2(-INFINITY, 0.f);
  asm volatile("bar.sync 1, 256;" ::: "memory");  // the 256 row threads only
  float M, Lc;           // reference maximum and denominator of the CTA's merged partial
  float merged[64];      // its columns [64*chain, 64*chain + 64), unnormalised
  {
    const float2 mlA = sm->ml_chain[0][r], mlB = sm->ml_chain[1][r];
    M = fmaxf(mlA.x, mlB.x);
    const float fA = mlA.x == -INFINITY ? 0.f : ex2(mlA.x - M), fB = mlB.x == -INFINITY ? 0.f : ex2(mlB.x - M);
    Lc = mlA.y * fA + mlB.y * fB;
    if (kMode == kCluster) {
      __syncwarp();
      cluster_wait();  // every CTA of the cluster runs
      if (chain == 0 && row_valid) {
        const uint32_t to = smem_u32(&sm->ml_cta[split][r]), bar = smem_u32(&sm->ml_full);
        for (int q = 0; q < a.splits; ++q) st_async2(remote_smem(to, q), M, Lc, remote_smem(bar, q));
      }
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
    if (nblk > 1 && ok) {  // (one block has left O_B alone)
      uint32_t o[64];
      tmem_ld32(oB, o, 0);
      tmem_ld32(oB + 32u, o, 32);
      tc_wait_ld();
      const uint64_t f2 = pair_of(fB, fB);
#pragma unroll
      for (int e = 0; e < 32; ++e) m2[e] = fma2(pair_of(__uint_as_float(o[2 * e]), __uint_as_float(o[2 * e + 1])), f2, m2[e]);
    }
  }
  uint8_t* out_row = reinterpret_cast<uint8_t*>(a.out) + 2 * ((int64_t)i * a.o_stride_tok + (int64_t)h * a.o_stride_head);
  if (kMode != kCluster) {
    const float inv = 1.f / Lc;  // the row saw at least its own key, so Lc > 0
    auto words = [&](int j) -> uint4 {  // columns 8j .. 8j+7 of the thread's 64
      const float* x = merged + 8 * j;
      return make_uint4(pack2<kBf16>(x[0] * inv, x[1] * inv), pack2<kBf16>(x[2] * inv, x[3] * inv), pack2<kBf16>(x[4] * inv, x[5] * inv), pack2<kBf16>(x[6] * inv, x[7] * inv));
    };
    if (live_rows <= kDirectRows) {
      if (row_valid) {
#pragma unroll
        for (int j = 0; j < 8; ++j) *reinterpret_cast<uint4*>(out_row + 128 * chain + 16 * j) = words(j);
      }
    } else {
      // Out through this warp's 32 rows of the Q tile, where 16 bytes of 32 rows turn into 128 bytes of four.
      uint8_t* stage = sm->q + (uint32_t)chain * kHalfBytes + (uint32_t)quad * 4096u;
      if (row_valid) {
#pragma unroll
        for (int j = 0; j < 8; ++j) *reinterpret_cast<uint4*>(stage + lane * 128 + ((j ^ (lane & 7)) << 4)) = words(j);
      }
      __syncwarp();
      const int64_t mine = row_valid ? out_row - reinterpret_cast<uint8_t*>(a.out) : -1;  // (strides are positive)
      uint8_t* const column = reinterpret_cast<uint8_t*>(a.out) + 128 * chain + 16 * (lane & 7);
#pragma unroll 1
      for (int row = lane >> 3; row < 32; row += 4) {
        const int64_t at = __shfl_sync(0xffffffffu, mine, row);
        if (at >= 0) *reinterpret_cast<uint4*>(column + at) = *reinterpret_cast<const uint4*>(stage + row * 128 + (((lane & 7) ^ (row & 7)) << 4));
      }
    }
    if (chain == 0 && row_valid && a.lse != nullptr) a.lse[(size_t)h * a.n + i] = (M + log2f(Lc)) * kLn2;
  } else {
    // Step 2, across the cluster (cs = 2 .. 8 CTAs along the key range).  The piece goes into the V stages, slice by slice, as
    // float4 planes [half][row]; one copy takes an owner its slices, into its receive buffer
    // [contributor][slot][half][row].
    const int cs = a.splits, slots = a.slots;  // (the last slot of some CTAs may be empty)
    const uint32_t piece = smem_u32(&sm->v[0][0][0]), receive = smem_u32(&sm->receive[0]);
    if (row_valid) {  // (rows past the tile's last node are padding: nothing of theirs is written, reduced or stored)
      float4* to = reinterpret_cast<float4*>(&sm->v[0][0][0] + (uint32_t)chain * 16u * plane) + r;
#pragma unroll
      for (int j = 0; j < 16; ++j) to[(uint32_t)j * (plane / 16u)] = make_float4(merged[4 * j], merged[4 * j + 1], merged[4 * j + 2], merged[4 * j + 3]);
    }
    fence_async_smem();
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (warp == 4) {
      mbar_wait(sm, &sm->k_free, 0, a.dev_status);  // (on a timeout the copies go out all the same: the others count on them)
      if (lane < cs && lane != split)
        copy_to_cta(remote_smem(receive + (uint32_t)(split * slots) * 2u * plane, lane), piece + (uint32_t)slices_before(lane, a) * 2u * plane,
                    (uint32_t)slices_of(lane, a) * 2u * plane, remote_smem(smem_u32(&sm->data_full), lane));
      __syncwarp();
    }
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 13);
    // The rows' common maximum and sum, and each piece's share of the output, while the pieces travel.
    mbar_wait(sm, &sm->ml_full, 0, a.dev_status);
    float Mg = -INFINITY, Ls = 0.f;
#pragma unroll 1
    for (int q = 0; q < cs; ++q) {  // (one pass: the sum so far follows the maximum)
      const float2 ml = sm->ml_cta[q][r];
      const float m = fmaxf(Mg, ml.x);
      if (m != -INFINITY) Ls = Ls * ex2(Mg - m) + ml.y * ex2(ml.x - m);
      Mg = m;
    }
    const float inv = 1.f / Ls;  // some CTA saw the row's own key, so Ls > 0
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 7);
    // the two warp groups share this CTA's slices
    const int owned = slices_of(split, a), before = slices_before(split, a);
    const int first_slot = chain ? (owned + 1) >> 1 : 0, end_slot = chain ? owned : (owned + 1) >> 1;
    mbar_wait(sm, &sm->data_full, 0, a.dev_status);
    __syncwarp();
    cluster_arrive_relaxed();  // every piece for this CTA is here: its senders may leave
    if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 8);
    if (row_valid)
      for (int slot = first_slot; slot < end_slot; ++slot) {
        uint64_t x[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 2
        for (int q = 0; q < cs; ++q) {
          const uint8_t* at = q == split ? &sm->v[0][0][0] + (uint32_t)(before + slot) * 2u * plane
                                         : &sm->receive[0] + (uint32_t)(q * slots + slot) * 2u * plane;
          const ulonglong2 u = *(reinterpret_cast<const ulonglong2*>(at) + r), w = *(reinterpret_cast<const ulonglong2*>(at + plane) + r);
          const float f = ex2(sm->ml_cta[q][r].x - Mg) * inv;
          const uint64_t f2 = pair_of(f, f);
          x[0] = fma2(u.x, f2, x[0]); x[1] = fma2(u.y, f2, x[1]); x[2] = fma2(w.x, f2, x[2]); x[3] = fma2(w.y, f2, x[3]);
        }
        float o[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) unpair(x[e], o[2 * e], o[2 * e + 1]);
        uint4 val;
        val.x = pack2<kBf16>(o[0], o[1]);
        val.y = pack2<kBf16>(o[2], o[3]);
        val.z = pack2<kBf16>(o[4], o[5]);
        val.w = pack2<kBf16>(o[6], o[7]);
        *reinterpret_cast<uint4*>(out_row + 2 * (8 * (before + slot))) = val;
      }
    if (split == 0 && chain == 0 && row_valid && a.lse != nullptr) a.lse[(size_t)h * a.n + i] = (Mg + log2f(Ls)) * kLn2;
    __syncwarp();
    cluster_wait();
  }
  if (threadIdx.x == SEQ_TRACE_ROW) UTRACE(2, 9);
#ifdef SEQ_TRACE
  if (threadIdx.x == 128 && cta_lin < 1024) g_cta_times[cta_lin][1] = gtimer();
#endif
  tc_fence_before();
  __syncthreads();  // pairs with warp group 0, whose MMA warp then frees the tensor memory
}

// ---------------------------------------------------------------- host side ---------------------
bool umma_supported(const seq_tree_attention_params& p) {
  if (p.dtype != SEQ_F16 && p.dtype != SEQ_BF16) return false;
  return p.num_q_heads / p.num_kv_heads <= kTileM;  // a tile holds at least one node's group of heads
}

// How the tiles are spread over the SMs.  Grid schedule: one CTA (or a cluster of `splits` CTAs along the key
// range) per (tile, kv head), in as many waves as that takes.  Stream schedule: one CTA per SM, each with an equal range of the
// flattened block space and share the tiles that a range boundary cuts.  p.kernel = 3 / 4 force one of them.
struct UmmaPlan { int splits; bool stream, optional; };  // optional: without a workspace, the grid schedule
constexpr long kOptionalStreamUnits = 48;  // (see umma_plan)
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
  if (const char* e = getenv("SEQ_DEBUG_SPLITS")) return {atoi(e), false, false};  // debug builds only
#endif
  if (p.kernel == 3 && can_stream) return {1, true, false};
  // More units than SMs.  Measured over batches of the paper's shapes (5 to 32 requests stacked as heads): plain
  // waves of one CTA per unit win by 5-50 % when tiles are short (a tile cut by a range boundary costs a trip
  // through the workspace, and every CTA starts and finishes two tiles more), the stream schedule wins by 5-15 %
  // when tiles are long (72 blocks and more) or when the last wave would be at most 60 % full.
  if (p.kernel != 4 && can_stream && units > kNumSMs) {
    const long waves = (units + kNumSMs - 1) / kNumSMs;
    const bool last_wave_thin = units * 10 <= waves * kNumSMs * 6;
    if (nblk >= 32 && (last_wave_thin || nblk >= 72)) return {1, true, false};
  }
  // Otherwise the split with the lowest estimate.  Microseconds per wave, fitted to launches of 110 shapes (1 to 256 nodes,
  // prefixes of 32 to 8192 keys, 8 to 148 units) with every split forced: 0.45 per block of a CTA's key range, 5 fixed, and
  // the merge across the cluster.  (Picks within 0.25 % of the best split on the average and 4 % at worst; with the figures of
  // the merge that stored its pieces one by one, 2.3 to 4.2, 2 % and 34 %: 4 nodes on 350 keys of 64/8 heads 6.05 -> 5.6 us,
  // 8 on 1024 7.25 -> 6.6.)  What a wave holds is asked of the device: a cluster lies in one
  // GPC, so the SMs left over in each are lost to it (74, 44, 36, 28, 21, 14 and 14 clusters of 2 to 8 CTAs were seen, where
  // 148 / cs had been assumed; 24 units of 17 blocks 17.3 -> 10.1 us, 16 of 48 21.8 -> 12.5, 48 of 66 34.7 -> 23.3).
  // A merge of tiles of more than 64 rows takes 0.75 to 1.1 us longer (32 units of 6 blocks, 128 rows: 7.8 us in one CTA, 8.4 in
  // four; 64 rows: 7.45 and 6.9), which decides between one CTA and a cluster up to 8 blocks: 32 units of 6 to 7 blocks 8.45 -> 7.8
  // and 9.05 -> 8.5.
  static const double kMerge[kMaxClusterSplit + 1] = {0.0, 0.0, 1.45, 2.0, 1.7, 2.3, 2.05, 1.8, 1.8};
  const double wide = (p.n_tree < nodes_per_tile ? p.n_tree : nodes_per_tile) * G > 64 ? 0.9 : 0.0;
  int best = 1;
  double best_cost = -1.0, grid_cost = 0.0;  // grid_cost: as the rule for the stream below was fitted, whatever the tiles' rows
  for (int cs = 1; cs <= kMaxClusterSplit && cs <= nblk; ++cs) {
    const int room = clusters_side_by_side(cs);
    if (room == 0) continue;
    const long waves = (units + room - 1) / room;
    const double plain = (double)waves * (0.45 * ((nblk + cs - 1) / cs) + 5.0 + kMerge[cs]), cost = plain + (cs > 1 ? waves * wide : 0.0);
    if (best_cost < 0 || cost < best_cost - 1e-9) { best = cs; best_cost = cost; grid_cost = plain; }
  }
  // ... against that of the stream schedule: 0.4 per block of an SM's range, 7 per tile it starts or finishes, 7 fixed (3 to 8
  // % off over 20 shapes of 96 to 384 units).  320 units of 67 blocks 99 -> 82 us, 104 of 200 95 -> 79; taken where it is an
  // eighth lower, because a caller has 19 MB of workspace to find for it (the first time 0.2 ms).  These calls were served
  // without a workspace before there was this rule, and without one they still are.  It holds
  // - from 48 units on (48 of 200 blocks 52 -> 49 us, 52 of 300 92 -> 64, 80 of 200 73 -> 65): with fewer a tile has more than
  //   three pieces and one CTA adds them all up, which the estimate knows nothing of (1 unit of 200 blocks 19 us in a cluster,
  //   237 as a stream; 8 of 300 26 / 53; 16 of 500 46 / 53; 32 of 500 64 / 67);
  // - for a length given by the host: one in device memory is planned for at its largest, and the stream is the slower one of
  //   the two well below that (96 units planned for 128 blocks: 64 / 54 us there, 37 / 39 at half of it, 12 / 23 at 500 keys);
  // - where L2 holds K and V: the tiles of a head, in step when they start together, each fetch them anew from memory (80 units
  //   of 450 blocks, 118 MB: 149 us in one wave, 155 as a stream; 104 of 132, 220 MB: 66 / 84; 312 of 67, 114 MB: 99 / 90).
  // Over 537 shapes of 48 to 400 units and 24 to 450 blocks no pick of the stream by this rule is more than 3 % slower than the
  // grid schedule.
  const double kv_bytes = 4.0 * ((double)p.prefix_len + p.n_tree) * kHeadDim * p.num_kv_heads;
  const double stream_cost = 0.4 * units * nblk / kNumSMs + 7.0 * ((double)units / kNumSMs + 1.0) + 7.0;
  if (p.kernel != 4 && can_stream && units >= kOptionalStreamUnits && p.prefix_len_dev == nullptr && nblk >= 24 && kv_bytes < 115e6 &&
      stream_cost < 0.88 * grid_cost)
    return {best, true, true};
  return {best, false, false};
}

int umma_default_splits(const seq_tree_attention_params& p) { return umma_plan(p).splits; }

size_t umma_workspace_bytes(const seq_tree_attention_params& p) { return umma_plan(p).stream ? stream_workspace_bytes(p) : 0; }

bool attention_maps(const seq_tree_attention_params& p, int kv_halves, CUtensorMap* q_map, CUtensorMap* k_map, CUtensorMap* v_map) {
  const int G = p.num_q_heads / p.num_kv_heads;
  const int nodes_per_tile = kTileM / G;
  const CUtensorMapDataType dt = p.dtype == SEQ_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  {
    // q viewed as [kv head][node][head in group][head_dim]
    // head_dim is split into its two 64-element halves (a dimension of its own, 128 bytes apart) so that one copy
    // brings the tile as [half][row][64 elements], the layout of two 128-byte-swizzled sub-tiles
    cuuint64_t dims[5] = {64, (cuuint64_t)G, (cuuint64_t)p.n_tree, 2, (cuuint64_t)p.num_kv_heads};
    cuuint64_t strides[4] = {(cuuint64_t)p.q_stride_head * 2, (cuuint64_t)p.q_stride_tok * 2, 128,
                             (cuuint64_t)p.q_stride_head * 2 * G};
    cuuint32_t box[5] = {64, (cuuint32_t)G, (cuuint32_t)nodes_per_tile, kTileM % G == 0 ? 2u : 1u, 1};  // (see load_q)
    if (!tensor_map(q_map, dt, 5, p.q, dims, strides, box)) return false;
  }
  for (int which = 0; which < 2; ++which) {
    // only the live rows [0, prefix_len + n_tree) are mapped: anything past them reads as zero.  (With the prefix
    // length in device memory the map cannot end there: it covers the cache, and the kernel clears the tail rows.)
    cuuint64_t dims[4] = {64, (cuuint64_t)(p.prefix_len_dev != nullptr ? p.kv_capacity : p.prefix_len + p.n_tree), 2, (cuuint64_t)p.num_kv_heads};
    cuuint64_t strides[3] = {(cuuint64_t)p.kv_stride_tok * 2, 128, (cuuint64_t)p.kv_stride_head * 2};
    cuuint32_t box[4] = {64, (cuuint32_t)kBlockN, (cuuint32_t)kv_halves, 1};
    if (!tensor_map(which == 0 ? k_map : v_map, dt, 4, which == 0 ? p.k_cache : p.v_cache, dims, strides, box)) return false;
  }
  return true;
}

int launch_attention_umma(const seq_tree_attention_params& p, int splits, cudaStream_t stream) {
  const int G = p.num_q_heads / p.num_kv_heads;
  const int nodes_per_tile = kTileM / G;
  const int tiles = (p.n_tree + nodes_per_tile - 1) / nodes_per_tile;
  // (groups that do not divide 128 used to run on the CUDA cores, which ask for nothing at these sizes: without a workspace
  // they take the grid schedule instead, 500 nodes on 4600 keys of 40/8 heads 99 us against 67)
  const bool lent = p.workspace != nullptr && p.workspace_bytes >= stream_workspace_bytes(p);
  const bool aligned = reinterpret_cast<uintptr_t>(p.workspace) % 256 == 0;
  const UmmaPlan plan = umma_plan(p);
  if (plan.stream && (plan.optional ? lent && aligned : lent || p.kernel != 0 || kTileM % G == 0)) return launch_attention_stream(p, stream);

  CUtensorMap q_map, k_map, v_map;
  if (!attention_maps(p, 2, &q_map, &k_map, &v_map)) return SEQ_ERR_CUDA;
  UmmaArgs a;
  a.n = p.n_tree; a.L_host = p.prefix_len; a.Hq = p.num_q_heads; a.Hkv = p.num_kv_heads; a.group = G;
  a.mask_wpr = p.mask_words_per_row; a.splits = splits; a.nodes_per_tile = nodes_per_tile; a.tiles = tiles;
  a.rows = nodes_per_tile * G;
  a.group_magic = (uint32_t)((65536 + G - 1) / G);
  a.split_magic = (uint32_t)((((uint64_t)1 << 32) / (uint64_t)splits) + 1);
  a.slots = (15 + splits) / splits; a.slices_each = 16 / splits; a.slices_more = 16 % splits;
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
  a.L_dev = p.prefix_len_dev; a.L_count = p.prefix_len_dev_count; a.zero_tail = p.prefix_len_dev != nullptr ? 1 : 0;
  const size_t smem = kUmmaSmemBytes;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tiles, p.num_kv_heads, splits);
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
    static int attr_done[8][64];  // the opt-in shared-memory size is set once per kernel and device
    const int rc = once_per_device(attr_done[which], [&]() -> int {
      SEQ_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      return SEQ_OK;
    });
    if (rc != SEQ_OK) return rc;
    SEQ_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, q_map, k_map, v_map, a));
    return SEQ_OK;
  };
  auto launch_type = [&](auto bf16, auto fine, int first) -> int {
    constexpr bool kB = decltype(bf16)::value, kF = decltype(fine)::value;
    return splits > 1 ? launch(tree_attention_umma_kernel<kB, kCluster, kF>, first) : launch(tree_attention_umma_kernel<kB, kGrid, kF>, first + 1);
  };
  const bool fine = kTileM % G != 0;
  if (p.dtype == SEQ_BF16) return fine ? launch_type(std::true_type(), std::true_type(), 4) : launch_type(std::true_type(), std::false_type(), 0);
  return fine ? launch_type(std::false_type(), std::true_type(), 6) : launch_type(std::false_type(), std::false_type(), 2);
}

}  // namespace seqtree
