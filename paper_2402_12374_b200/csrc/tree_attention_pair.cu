// Tree-masked attention on the 5th-generation tensor cores for trees of more than 128 query rows per kv head: two tiles of
// 128 query rows share every K/V tile and take turns on the tensor pipe.  (A query row is a (node, head-in-group) pair;
// up to 128 rows per kv head run on tree_attention_umma.cu, whose two chains share one query tile.)
//
// Work unit: (kv head, pair of query tiles A and B, range of the pair's keys).  Per block of 128 keys and tile:
//     S = Q K^T      128x128x128  tcgen05.mma, Q and K K-major in 128-byte-swizzled shared memory
//     P = 2^(scale*S - m) masked  one thread per row: S read from tensor memory, P written back over it as packed 16-bit
//     O += P V       128x128x128  tcgen05.mma, A = P from tensor memory, V MN-major in shared memory
// Tensor memory: S_A, S_B, O_A, O_B of 128 columns each.  One warp issues all MMAs in the order P.V of A, S of A's next
// block, P.V of B, S of B's next block: while the tensor pipe works for one tile (1024 cycles), the other tile's 128 row
// threads take their 128 exponentials (1024 cycles of the special-function units).  S of a tile's next block goes over the
// P just consumed, which the issue order makes safe.  With N = 128 both products run at 64 cycles per instruction, the full
// rate; the 64-key blocks of the one-tile kernel pay 51 instead of 32 for S, and each K/V tile is read from shared memory
// for one query tile only.
//
// Work distribution: as in tree_attention_umma.cu - grid mode, one CTA or a cluster of 2 to 8 CTAs along the key range per
// (pair, kv head), merged over distributed shared memory; stream mode, one CTA per SM with equal ranges of the flattened
// block space, tiles cut by a range boundary completed through the workspace.  The two row groups of a CTA work for
// different tiles and never wait for one another.
//
// Every mbarrier wait is bounded; a wait that runs out raises SEQ_DEV_TIMEOUT and the CTA drains.
#include <cooperative_groups.h>

#include "common.cuh"
#include "tensor_map.cuh"
#include "umma.cuh"

namespace cg = cooperative_groups;

namespace seqtree {
namespace pair {

constexpr int kTileM = 128;         // query rows per tile
constexpr int kBlockN = 128;        // keys per block
constexpr int kThreads = 384;       // warp group 0: TMA warp, MMA warp, two spare; warp groups 1, 2: rows of tiles A, B
constexpr int kRegsLight = 56, kRegsRows = 224;  // after setmaxnreg: 128*56 + 256*224 = 384*168
constexpr int kMaxClusterSplit = 8;
constexpr int kMaxStreamPairs = 128;
constexpr int kStreamPairCost = 4;  // positions in front of a pair's blocks that stand for what starting and finishing it costs

constexpr uint32_t kTileBytes = 128 * 128 * 2;   // a Q, K or V tile: 128 rows x 128 elements of 16 bits
constexpr uint32_t kHalfBytes = kTileBytes / 2;  // one 128-row x 64-element sub-tile (128 B rows)
constexpr float kRescaleThreshold = 8.f;         // log2 units
constexpr float kRescaleLimit = 256.f;           // 2^kRescaleThreshold: no term of a row sum at or below it came from a score above the threshold

struct Smem {
  // tiles 1024-byte aligned (128-byte swizzle atoms are 8 rows x 128 B); after the last block their 192 KB receive the
  // cluster merge
  uint8_t q[2][kTileBytes];
  uint8_t k[2][kTileBytes];
  uint8_t v[2][kTileBytes];
  // mask from the parent array: the tree, and the ancestor rows of the pair's nodes, word by word
  uint32_t mask[SEQ_MAX_TREE / 32][2 * kTileM];
  int16_t parent[SEQ_MAX_TREE];
  int32_t pair_prefix[kMaxStreamPairs + 1];  // stream mode: positions of a kv head's layout before its t-th pair
  uint64_t q_full[2], q_empty, k_full[2], k_empty[2], v_full[2], v_empty[2];
  uint64_t s_full[2], p_full[2], o_full[2], o_free[2];  // [tile]: one phase per block, per block, per segment, per segment
  uint32_t tmem_base;
  volatile int abort_flag;
  int32_t abort_seen[2][2];  // [tile][segment parity]: abort_flag as one row thread saw it, so that a row group leaves together
  int32_t last_part[2];      // [tile] stream mode: this CTA completed the tile
};
constexpr size_t kMergeMlOffset = 176 << 10;  // the merge's (m, l) behind its planes (cs * ceil(16 / cs) * 8 KB <= 168 KB)
static_assert(sizeof(Smem) <= 227 * 1024, "one CTA's shared memory");

struct Args {
  int32_t n, L_host, Hkv, group, mask_wpr, splits, nodes_per_tile, tiles, pairs;
  int32_t rows;           // query rows of a full tile: nodes_per_tile * group, 128 when the group divides it
  const int32_t* L_dev;   // nullable: the prefix length in device memory (<= L_host)
  int32_t L_count;        // > 1: one length per request, requests stacked as heads (grid schedule only)
  int32_t zero_tail;      // the K/V maps cover the whole cache: rows past the tree are cleared in shared memory
  int32_t blocks_per_head_host;
  int64_t total_blocks_host;
  int32_t* ws_count;      // [Hkv * tiles] arrivals per tile, zero on entry and on exit
  float2* ws_ml;          // [2 * gridDim.x][tile][128] (m, l) of a partial result
  float4* ws_o;           // [2 * gridDim.x][tile][32][128] its unnormalised accumulator, thread-major
  float scale_log2;
  uint32_t idesc_qk, idesc_pv;
  const uint32_t* mask_bits;
  const int32_t* parent;  // used when mask_bits is null
  void* out; int64_t o_stride_tok, o_stride_head;
  float* lse;
  int32_t* dev_status;
};

// blocks of a pair whose last node is i1 - 1: a node sees no later node
__host__ __device__ __forceinline__ int pair_blocks(int L, int i1) { return (L + i1 + kBlockN - 1) / kBlockN; }

// The Q tile of nodes [i0, i0 + nodes_per_tile) of kv head g: one copy for both 64-element halves when the tile has 128
// rows, else (the second half would land off the swizzle's 1024-byte boundary) a copy each.
__device__ __forceinline__ void load_q(uint8_t* dst, const CUtensorMap* map, uint64_t* bar, int rows, int i0, int g) {
  mbar_expect_tx(bar, (uint32_t)rows * 256u);
  tma_load_5d(dst, map, bar, 0, 0, i0, 0, g);
  if (rows < kTileM) tma_load_5d(dst + kHalfBytes, map, bar, 0, 0, i0, 1, g);
}
__device__ __forceinline__ void load_kv(uint8_t* dst, const CUtensorMap* map, uint64_t* bar, int row, int g) {
  mbar_expect_tx(bar, kTileBytes);
  tma_load_4d(dst, map, bar, 0, row, 0, g);  // both 64-element halves by one copy
}
__device__ __forceinline__ void group_sync(int tile) {
  if (tile == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
  else asm volatile("bar.sync 2, 128;" ::: "memory");
}

template <bool kBf16, bool kStream>
__global__ void __launch_bounds__(kThreads, 1)
tree_attention_pair_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                           const __grid_constant__ CUtensorMap v_map, const __grid_constant__ Args a) {
  extern __shared__ __align__(1024) uint8_t pair_smem[];
  Smem* sm = reinterpret_cast<Smem*>(pair_smem);
  cg::cluster_group cluster = cg::this_cluster();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int split = blockIdx.z;  // the cluster spans blockIdx.z

  // A CTA works through segments: (kv head, pair, range of the pair's blocks).  Grid mode: the one segment (blockIdx.y,
  // blockIdx.x, this CTA's share of the cluster's key range).  Stream mode: the pieces of the units that its range
  // [range_lo, range_hi) of the flattened block space overlaps.
  int L = a.L_host;
  int blocks_per_head = a.blocks_per_head_host;
  int64_t total_blocks = a.total_blocks_host;
  int64_t range_lo = 0, range_hi = 1;
  struct Seg { int g, pair, slot_in_head, i0, i1, blk_lo, nblk, nblk_pair; bool has_b; int64_t next; };
  // Stream mode lays the pairs of a kv head out alternating from both ends (0, P-1, 1, P-2, ...): late pairs have more
  // masked blocks, which cost more, and this way every range gets its share of them.
  auto pair_at = [&](int k) { return (k & 1) ? a.pairs - 1 - (k >> 1) : (k >> 1); };
  auto pair_end = [&](int p) { return min((2 * p + 2) * a.nodes_per_tile, a.n); };
  auto seg_at = [&](int64_t pos) -> Seg {
    Seg x;
    if (!kStream) {
      x.pair = blockIdx.x; x.g = blockIdx.y; x.slot_in_head = x.pair;
    } else {
      x.g = (int)(pos / blocks_per_head);
      const int rem = (int)(pos % blocks_per_head);
      int lo = 0, hi = a.pairs - 1;  // the last place in the head's layout whose first position is at or before rem
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sm->pair_prefix[mid] <= rem) lo = mid; else hi = mid - 1;
      }
      x.slot_in_head = lo;
      x.pair = pair_at(lo);
    }
    x.i0 = x.pair * 2 * a.nodes_per_tile;
    x.i1 = pair_end(x.pair);
    x.has_b = x.i0 + a.nodes_per_tile < a.n;
    if (!kStream) {
      x.nblk_pair = pair_blocks(L, x.i1);
      x.blk_lo = (int)(((long)split * x.nblk_pair) / a.splits);
      x.nblk = (int)(((long)(split + 1) * x.nblk_pair) / a.splits) - x.blk_lo;
      x.next = 1;
    } else {
      // the pair's positions are [vs, ve): kStreamPairCost positions of overhead, then its blocks
      const int rem = (int)(pos % blocks_per_head);
      const int vs = sm->pair_prefix[x.slot_in_head], ve = sm->pair_prefix[x.slot_in_head + 1];
      const int end = (int)min((int64_t)ve, (int64_t)rem + (range_hi - pos));  // where this CTA leaves the pair
      const int from = max(rem, vs + kStreamPairCost);
      x.blk_lo = from - (vs + kStreamPairCost);
      x.nblk_pair = ve - vs - kStreamPairCost;
      x.nblk = max(end - from, 0);  // 0: the range ends in the overhead positions, the pair is the next CTA's
      x.next = pos + (end - rem);
    }
    return x;
  };
  // The barriers are armed once; their phases run on from segment to segment.
  if (threadIdx.x == 0) {
    for (int c = 0; c < 2; ++c) {
      mbar_init(&sm->q_full[c], 1);
      mbar_init(&sm->k_full[c], 1); mbar_init(&sm->k_empty[c], 1);
      mbar_init(&sm->v_full[c], 1); mbar_init(&sm->v_empty[c], 1);
      mbar_init(&sm->s_full[c], 1); mbar_init(&sm->p_full[c], 4);
      mbar_init(&sm->o_full[c], 1); mbar_init(&sm->o_free[c], 4);
    }
    mbar_init(&sm->q_empty, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sm->abort_flag = 0;
    // programmatic dependent launch: the next kernel in the stream may be scheduled onto free SMs from now on (it
    // waits, as this one does below, before it touches memory)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  // Nothing before this line reads or writes global memory.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (a.L_dev != nullptr) {
    const int v = a.L_dev[(!kStream && a.L_count > 1) ? ((int)blockIdx.y * a.L_count) / a.Hkv : 0];
    if (v < 0 || v > a.L_host) { if (threadIdx.x == 0) dev_flag(a.dev_status, SEQ_DEV_BAD_LENGTH); }
    L = min(max(v, 0), a.L_host);
    if (kStream) {  // the flattened block space of this prefix length (every warp for itself)
      int sum = 0;
      for (int t = lane; t < a.pairs; t += 32) sum += kStreamPairCost + pair_blocks(L, pair_end(t));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      blocks_per_head = sum;
      total_blocks = (int64_t)sum * a.Hkv;
    }
  }
  if (kStream) {
    range_lo = (total_blocks * (int64_t)blockIdx.x) / (int64_t)gridDim.x;
    range_hi = (total_blocks * (int64_t)(blockIdx.x + 1)) / (int64_t)gridDim.x;
  }
  // Grid schedule: the thread that armed the barriers requests the Q tiles and the first K and V tile right away, before
  // the CTA-wide barrier below and the hand-over to the producer warp (which skips what has been requested here).
  if (!kStream && threadIdx.x == 0) {
    const Seg s0 = seg_at(range_lo);
    if (s0.nblk > 0) {
      load_q(sm->q[0], &q_map, &sm->q_full[0], a.rows, s0.i0, s0.g);
      load_kv(sm->k[0], &k_map, &sm->k_full[0], s0.blk_lo * kBlockN, s0.g);
      if (s0.has_b) load_q(sm->q[1], &q_map, &sm->q_full[1], a.rows, s0.i0 + a.nodes_per_tile, s0.g);
      load_kv(sm->v[0], &v_map, &sm->v_full[0], s0.blk_lo * kBlockN, s0.g);
    }
  }
  if (a.mask_bits == nullptr)  // an entry that is no earlier node is flagged and read as "no parent"
    for (int t = threadIdx.x; t < a.n; t += kThreads) {
      int pj = a.parent[t];
      if (pj < -1 || pj >= t) { if (pj != -1) dev_flag(a.dev_status, SEQ_DEV_BAD_PARENT); pj = -1; }
      sm->parent[t] = (int16_t)pj;
    }
  if (a.rows < kTileM) {  // rows no copy writes (the group does not divide 128): zeros, so that their scores are finite
    for (int t = a.rows * 8 + (int)threadIdx.x; t < kTileM * 8; t += kThreads)
      for (int c = 0; c < 2; ++c) {
        reinterpret_cast<uint4*>(sm->q[c])[t] = make_uint4(0u, 0u, 0u, 0u);
        reinterpret_cast<uint4*>(sm->q[c] + kHalfBytes)[t] = make_uint4(0u, 0u, 0u, 0u);
      }
    fence_async_smem();
  }
  if (kStream && warp == 2) {  // positions of a kv head before each place of its layout: four places per lane, then a warp scan
    constexpr int kPer = kMaxStreamPairs / 32;
    int local[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int t = lane * kPer + k;
      local[k] = t < a.pairs ? kStreamPairCost + pair_blocks(L, pair_end(pair_at(t))) : 0;
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
    for (int k = 0; k < kPer; ++k) {
      const int t = lane * kPer + k;
      if (t < a.pairs) sm->pair_prefix[t] = run;
      run += local[k];
    }
    if (lane == 31) sm->pair_prefix[a.pairs] = incl;
  }
  if (warp == 1) {  // all 512 tensor-memory columns: S_A, S_B (P over them), O_A, O_B
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&sm->tmem_base)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm->tmem_base;
  const uint32_t q_addr = smem_u32(pair_smem);  // the Q, K and V tiles, two each, one behind the other

  if (warp < 4) {
    // ============================ warp group 0: data movement and MMA issue, few registers =========
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLight));
    int seg = 0, seg_b = 0, base = 0, base_b = 0;  // segments done (with a tile B), blocks done in them
    uint32_t issued = 0, issued_parity = 0;        // producer: stages (bits 0, 1: K; 2, 3: V; 4, 5: Q) requested, phase of the last request
    auto note = [&](int bit, int phase) { issued |= 1u << bit; issued_parity = (issued_parity & ~(1u << bit)) | ((uint32_t)(phase & 1) << bit); };
    for (int64_t pos = range_lo; pos < range_hi;) {
      const Seg sg = seg_at(pos);
      if (kStream && sg.nblk == 0) { pos = sg.next; continue; }
      const int nblk = sg.nblk, g = sg.g;
      if (warp == 0 && nblk > 0) {
        // ------------------------------------------------------------ TMA producer ----------------
        // Fixed order Q_A, K(0), Q_B, V(0), K(1), V(1), ...: a K stage is free once both tiles' S have used it, a V stage
        // after both tiles' P.V, in the same order.  The whole warp runs the loop; one elected lane issues the copies.
        if (!kStream) {
          note(4, 0); note(0, 0); note(2, 0);
          if (sg.has_b) note(5, 0);
        } else {
          if (seg > 0 && !mbar_wait(&sm->abort_flag, &sm->q_empty, (seg - 1) & 1, a.dev_status)) break;
          if (elect_one()) load_q(sm->q[0], &q_map, &sm->q_full[0], a.rows, sg.i0, g);
          __syncwarp();
          note(4, seg);
        }
        for (int j = kStream ? 0 : 1; j < nblk; ++j) {
          const int b = (base + j) & 1, w = (base + j) >> 1, row = (sg.blk_lo + j) * kBlockN;
          if (w > 0 && !mbar_wait(&sm->abort_flag, &sm->k_empty[b], (w - 1) & 1, a.dev_status)) break;
          if (elect_one()) {
            load_kv(sm->k[b], &k_map, &sm->k_full[b], row, g);
            if (kStream && j == 0 && sg.has_b) load_q(sm->q[1], &q_map, &sm->q_full[1], a.rows, sg.i0 + a.nodes_per_tile, g);
          }
          __syncwarp();
          note(b, w);
          if (kStream && j == 0 && sg.has_b) note(5, seg_b);
          if (w > 0 && !mbar_wait(&sm->abort_flag, &sm->v_empty[b], (w - 1) & 1, a.dev_status)) break;
          if (elect_one()) load_kv(sm->v[b], &v_map, &sm->v_full[b], row, g);
          __syncwarp();
          note(2 + b, w);
        }
      } else if (warp == 1 && nblk > 0) {
        // ------------------------------------------------------------ MMA issuer ------------------
        // The whole warp runs this code; only the MMAs and commits are issued by one elected lane, so descriptors and
        // addresses stay warp-uniform.  Waits on another role's barrier come once per phase, so none can be missed.
        const int last_tile = sg.has_b ? 1 : 0;
        auto wait = [&](uint64_t* bar, int phase) { return mbar_wait(&sm->abort_flag, bar, phase & 1, a.dev_status); };
        auto issue_s = [&](int c, int j) {  // S of block j of tile c (the K tile is in place)
          const int b = (base + j) & 1;
          if (elect_one()) {
            mma_qk<kHalfBytes, kHalfBytes>(tmem + 128u * c, desc_lo(q_addr + c * kTileBytes, 16), desc_lo(q_addr + (2 + b) * kTileBytes, 16), a.idesc_qk);
            tc_commit(&sm->s_full[c]);
            if (c == last_tile) {
              tc_commit(&sm->k_empty[b]);
              if (j == nblk - 1) tc_commit(&sm->q_empty);
            }
          }
          __syncwarp();
        };
        auto issue_pv = [&](int c, int j) {
          const int b = (base + j) & 1;
          if (elect_one()) {
            mma_pv<8>(tmem + 256u + 128u * c, tmem + 128u * c, desc_lo(q_addr + (4 + b) * kTileBytes, kHalfBytes), a.idesc_pv, j > 0);
            if (c == last_tile) tc_commit(&sm->v_empty[b]);
            if (j == nblk - 1) tc_commit(&sm->o_full[c]);
          }
          __syncwarp();
        };
        bool go = wait(&sm->q_full[0], seg) && wait(&sm->k_full[base & 1], base >> 1);
        if (go) {
          tc_fence_after();
          issue_s(0, 0);
          if (sg.has_b) {
            go = wait(&sm->q_full[1], seg_b);
            if (go) issue_s(1, 0);
          }
        }
#pragma unroll 1
        for (int j = 0; j < nblk && go; ++j) {
          const int b = (base + j) & 1, w = (base + j) >> 1;
#pragma unroll 1
          for (int c = 0; c <= last_tile && go; ++c) {
            const int cseg = c ? seg_b : seg, cbase = c ? base_b : base;
            go = wait(&sm->p_full[c], cbase + j);
            // the first P.V of a segment overwrites O: the row threads must have read the tile's previous one
            if (go && j == 0 && cseg > 0) go = wait(&sm->o_free[c], cseg - 1);
            if (go && c == 0) {
              go = wait(&sm->v_full[b], w);
              // (zero_tail: the maps cover the whole cache, so a block that reaches past the last tree row has fetched rows
              // that may hold anything; their probabilities are exactly 0, but 0 * NaN is not: the rows are cleared here,
              // whole 128-byte rows of both halves, and that is made visible to the tensor core's reads)
              const int live = L + a.n - (sg.blk_lo + j) * kBlockN;
              if (go && a.zero_tail && live < kBlockN) {
                uint4* vt = reinterpret_cast<uint4*>(sm->v[b]);
                for (int i = max(live, 0) * 8 + lane; i < kBlockN * 8; i += 32) {
                  vt[i] = make_uint4(0u, 0u, 0u, 0u);
                  vt[kHalfBytes / 16 + i] = make_uint4(0u, 0u, 0u, 0u);
                }
                fence_async_smem();
                __syncwarp();
              }
            }
            if (!go) break;
            tc_fence_after();
            issue_pv(c, j);
            // S of the next block goes where P of this one lives.  tcgen05.mma operations issued by one thread execute
            // in issue order, so this QK^T cannot overtake the P.V just issued.
            if (j + 1 < nblk) {
              if (c == 0) go = wait(&sm->k_full[(base + j + 1) & 1], (base + j + 1) >> 1);
              if (go) { tc_fence_after(); issue_s(c, j + 1); }
            }
          }
        }
      }
      __syncwarp();
      if (a.splits > 1) {  // the two cluster barriers of the merge (see the row threads)
        cluster.sync();
        cluster.sync();
      }
      pos = sg.next;
      ++seg; base += nblk;
      if (sg.has_b) { ++seg_b; base_b += nblk; }
      if (kStream && sm->abort_flag) break;
    }  // segments
    // A CTA that gives up must not leave while a tile it has requested is still on its way into its shared memory: the
    // producer waits, with a bound of its own, for the last tile requested into each stage.
    if (sm->abort_flag && warp == 0) {
      for (int st = 0; st < 6; ++st) {
        if (!((issued >> st) & 1u)) continue;
        uint64_t* full = st < 2 ? &sm->k_full[st] : st < 4 ? &sm->v_full[st - 2] : &sm->q_full[st - 4];
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

  // ============================== warp groups 1, 2: one thread per query row of tile A, B ============
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsRows));
  const int c = (warp >> 2) - 1;              // the tile
  const int quad = warp & 3;                  // tensor-memory lane quarter this warp may access
  const int r = quad * 32 + lane;             // row of the tile = tensor-memory lane
  const bool first_thread = r == 0;
  const uint32_t lane_sel = (uint32_t)(quad * 32) << 16;
  const uint32_t tmem_s = tmem + 128u * c + lane_sel, tmem_o = tmem + 256u + 128u * c + lane_sel;
  const float sc = a.scale_log2;
  int seg = 0, base = 0;  // segments done, blocks done in them (of this tile)
  for (int64_t pos = range_lo; pos < range_hi;) {
    const Seg sg = seg_at(pos);
    if (kStream && (sg.nblk == 0 || (c == 1 && !sg.has_b))) { pos = sg.next; continue; }
    const int g = sg.g, nblk = (c == 0 || sg.has_b) ? sg.nblk : 0;
    const int i0 = sg.i0 + c * a.nodes_per_tile, i_end = min(i0 + a.nodes_per_tile, a.n);
    const int i = i0 + r / a.group;             // node of this row
    const int h = g * a.group + r % a.group;
    const bool row_valid = i < i_end;
    // The row's ancestor bits: the caller's mask, or rows derived from the parent array by the first thread of each node,
    // while the first tiles are on their way.  (The previous segment's rows are out of use: this group's last reads of
    // them are behind it, and nobody else reads them.)
    const int slot = c * kTileM + r / a.group;
    if (a.mask_bits == nullptr) {
      group_sync(c);
      if (r % a.group == 0 && row_valid) {
        const int wpr = (a.n + 31) >> 5;
        for (int w = 0; w < wpr; ++w) sm->mask[w][slot] = 0u;
        for (int j = i; j >= 0; j = sm->parent[j]) sm->mask[j >> 5][slot] |= 1u << (j & 31);
      }
      group_sync(c);
    }
    const uint32_t* mrow = a.mask_bits != nullptr ? a.mask_bits + (size_t)min(i, a.n - 1) * a.mask_wpr : &sm->mask[0][slot];
    const int mask_stride = a.mask_bits != nullptr ? 1 : 2 * kTileM, mask_wpr = a.mask_bits != nullptr ? a.mask_wpr : (a.n + 31) >> 5;

    float m_used = -INFINITY, l = 0.f;
    bool ok = true;
    // A warp whose 32 rows all lie past the tile's last node leaves the special-function unit and the issue slots to the
    // warps with real rows; its P rows stay whatever they are (rows of the product are independent).
    const bool warp_live = i0 + (quad * 32) / a.group < i_end;
    for (int u = 0; u < nblk; ++u) {
      if (!mbar_wait(&sm->abort_flag, &sm->s_full[c], (base + u) & 1, a.dev_status)) { ok = false; break; }
      if (!warp_live) {  // 32 padding rows: nothing to compute, only keep in step with the barriers
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm->p_full[c]);
        continue;
      }
      tc_fence_after();
      const int kb = (sg.blk_lo + u) * kBlockN;
      if (kb + kBlockN > L) {
        // The block reaches into the tree keys (or past the end): masked scores become -inf where they lie, so that their
        // probability is exactly 0 and they cannot raise the maximum.
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          const uint32_t vis = row_valid ? mask_window(mrow, mask_stride, mask_wpr, a.n, kb - L + 32 * q) : 0u;
          uint32_t x[32];
          tmem_ld32(tmem_s + 32u * q, x, 0);
          tc_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; ++e)
            if (!(vis & (1u << e))) x[e] = __float_as_uint(-INFINITY);
          tmem_st32(tmem_s + 32u * q, x, 0);
        }
        tc_wait_st();
      }
      uint32_t sreg[kBlockN];
#pragma unroll
      for (int e = 0; e < kBlockN; e += 32) tmem_ld32(tmem_s + e, sreg, e);
      tc_wait_ld();
      // P = 2^(scale*s - m) written over S as packed 16-bit values (64 columns, four stores of 16); returns the row sum.
      // (A row without a reference sees nothing in this block: its scores are all -inf and its P are 0.)
      auto exponentials = [&]() -> float {
        const float neg_m = m_used == -INFINITY ? 0.f : -m_used;
        const uint64_t sc2 = pair_of(sc, sc), neg_m2 = pair_of(neg_m, neg_m);
        uint64_t sm2[2] = {pair_of(0.f, 0.f), pair_of(0.f, 0.f)};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t packed[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) {  // two scores at a time: one packed multiply-add, two exponentials, one packed add
            float x0, x1;
            unpair(fma2(pair_of(__uint_as_float(sreg[32 * q + 2 * e]), __uint_as_float(sreg[32 * q + 2 * e + 1])), sc2, neg_m2), x0, x1);
            const float p0 = ex2(x0), p1 = ex2(x1);
            sm2[e & 1] = add2(sm2[e & 1], pair_of(p0, p1));
            packed[e] = pack2<kBf16>(p0, p1);
          }
          tmem_st16(tmem_s + 16u * q, packed);
        }
        float s0, s1, s2, s3;
        unpair(sm2[0], s0, s1);
        unpair(sm2[1], s2, s3);
        return (s0 + s1) + (s2 + s3);
      };
      // The exponentials are taken against the reference maximum as it stands, and their sum tells whether that was right:
      // a score more than the threshold above the reference gives a term, hence a sum, above 2^threshold.  Only then (or
      // without a reference) is the block maximum taken, the reference moved, O rescaled, and the pass repeated (the
      // scores are still in registers).
      float alpha = 1.f, sum;
      bool settle = __any_sync(0xffffffffu, m_used == -INFINITY);
#pragma unroll 1
      for (int pass = 0;; ++pass) {  // (a loop, so that the exponentials' code exists once)
        if (settle) {
          float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int e = 0; e < kBlockN; e += 2)  // three-input maximum: two scores per instruction
            mx[(e >> 1) & 3] = max3(mx[(e >> 1) & 3], __uint_as_float(sreg[e]), __uint_as_float(sreg[e + 1]));
          const float m_blk = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sc;  // scale > 0
          const bool move = m_blk > m_used + kRescaleThreshold || (m_used == -INFINITY && m_blk != -INFINITY);
          if (__any_sync(0xffffffffu, move)) {
            if (move) {
              alpha = m_used == -INFINITY ? 0.f : ex2(m_used - m_blk);
              m_used = m_blk;
            }
            if (u > 0) {  // (S of this block was issued behind the P.V of the one before, so O is complete)
#pragma unroll 1
              for (int q = 0; q < 8; ++q) {
                float o[16];
                tmem_ld8(tmem_o + 16u * q, o);
                tmem_ld8(tmem_o + 16u * q + 8u, o + 8);
                tc_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) o[e] *= alpha;
                tmem_st16(tmem_o + 16u * q, reinterpret_cast<uint32_t*>(o));
              }
            }
          }
        }
        sum = exponentials();
        if (settle) break;
        settle = __any_sync(0xffffffffu, !(sum <= kRescaleLimit));
        if (!settle) break;
      }
      l = l * alpha + sum;
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm->p_full[c]);  // one arrival per warp
    }
    if (nblk > 0 && ok) ok = mbar_wait(&sm->abort_flag, &sm->o_full[c], seg & 1, a.dev_status);
    tc_fence_after();

    // ---------------------------------------------------------------- merge ------------------------
    // Whether to stop after this segment is decided once for the row group: a flag raised between two threads' own reads
    // would send some to the closing barrier and the rest into the next segment's group_sync, which has no bound.
    bool stop_here = false;
    if (kStream) {
      if (first_thread) sm->abort_seen[c][seg & 1] = sm->abort_flag;
      group_sync(c);
      stop_here = sm->abort_seen[c][seg & 1] != 0;
    }
    const bool have = nblk > 0 && ok;
    float M = have ? m_used : -INFINITY, Lc = have ? l : 0.f;
    // The accumulator stays in tensor memory and is taken 32 or 8 columns at a time by loops that are not unrolled: code
    // that runs once per tile is fetched as it runs, about 80 cycles for eight instructions.  (The next segment's first P.V
    // waits for this row group's P, hence for the end of this.)
    auto own32 = [&](int q, float* x) {
      if (have) {
        tmem_ld32(tmem_o + 32u * q, reinterpret_cast<uint32_t*>(x), 0);
        tc_wait_ld();
      } else {
#pragma unroll
        for (int e = 0; e < 32; ++e) x[e] = 0.f;
      }
    };
    uint8_t* out_row = reinterpret_cast<uint8_t*>(a.out) + 2 * ((int64_t)i * a.o_stride_tok + (int64_t)h * a.o_stride_head);
    auto store8 = [&](int col, const float* x, float inv) {
      uint4 val;
      val.x = pack2<kBf16>(x[0] * inv, x[1] * inv);
      val.y = pack2<kBf16>(x[2] * inv, x[3] * inv);
      val.z = pack2<kBf16>(x[4] * inv, x[5] * inv);
      val.w = pack2<kBf16>(x[6] * inv, x[7] * inv);
      *reinterpret_cast<uint4*>(out_row + 2 * col) = val;
    };
    if (a.splits == 1) {
      bool write = true;
      int c_first = 0, c_last = -1;
      int64_t t0 = 0;
      auto cta_lo = [&](int x) { return (total_blocks * (int64_t)x) / (int64_t)gridDim.x; };
      auto slot_of = [&](int x) { return (2 * x + (max(t0, cta_lo(x)) == cta_lo(x) ? 0 : 1)) * 2 + c; };
      if (kStream && nblk < sg.nblk_pair) {
        // A piece of a tile.  Every piece is written to this CTA's slot of the workspace (slot 0 if the piece opens the
        // CTA's range, else 1), then counted; the CTA whose count completes the tile adds the other pieces to its own and
        // writes the output.  Nobody waits for anybody.
        t0 = (int64_t)g * blocks_per_head + sm->pair_prefix[sg.slot_in_head] + kStreamPairCost;
        const int64_t t1 = t0 + sg.nblk_pair;
        c_first = (int)((t0 * (int64_t)gridDim.x) / total_blocks);  // the CTA whose range holds block t0 ...
        while (cta_lo(c_first + 1) <= t0) ++c_first;                 // ... exactly
        while (cta_lo(c_first) > t0) --c_first;
        c_last = c_first;
        while (cta_lo(c_last + 1) < t1) ++c_last;
        const int my_slot = 2 * (int)blockIdx.x + (max(t0, range_lo) == range_lo ? 0 : 1);
        int* cnt = a.ws_count + (size_t)g * a.tiles + 2 * sg.pair + c;
        const int parts = c_last - c_first + 1;
        // If every other piece has been counted already (the usual case for the piece that closes a range), this CTA
        // completes the tile without writing its own piece.
        if (first_thread) {
          const int done = *reinterpret_cast<volatile int*>(cnt) == parts - 1;
          if (done) *cnt = 0;  // leave the counter as it was found
          sm->last_part[c] = done;
        }
        group_sync(c);
        if (!sm->last_part[c]) {
          a.ws_ml[(size_t)(my_slot * 2 + c) * kTileM + r] = make_float2(M, Lc);
          float4* my_o = a.ws_o + (size_t)(my_slot * 2 + c) * 32 * kTileM + r;
#pragma unroll 1
          for (int q = 0; q < 4; ++q) {
            float x[32];
            own32(q, x);
#pragma unroll
            for (int j = 0; j < 8; ++j) my_o[(size_t)(8 * q + j) * kTileM] = make_float4(x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]);
          }
          __threadfence();
          group_sync(c);
          if (first_thread) {
            const int last = atomicAdd(cnt, 1) == parts - 1;
            if (last) *cnt = 0;  // every piece has been counted
            sm->last_part[c] = last;
          }
          group_sync(c);
        }
        write = sm->last_part[c] != 0;
        if (write) __threadfence();
      }
      if (write) {
        // The pieces (one, usually) are added in the order of their CTAs, this CTA's own at its place, with one common
        // reference maximum: the result does not depend on which CTA happened to finish last.
        float Mg = M, Ls = 0.f;
#pragma unroll 1
        for (int x = c_first; x <= c_last; ++x)
          if (x != (int)blockIdx.x) Mg = fmaxf(Mg, __ldcg(a.ws_ml + (size_t)slot_of(x) * kTileM + r).x);
        const float f_own = M == -INFINITY ? 0.f : ex2(M - Mg);
#pragma unroll 1
        for (int x = c_first; x <= c_last; ++x) {
          if (x == (int)blockIdx.x) { Ls = fmaf(Lc, f_own, Ls); continue; }
          const float2 ml = __ldcg(a.ws_ml + (size_t)slot_of(x) * kTileM + r);
          if (ml.x != -INFINITY) Ls = fmaf(ml.y, ex2(ml.x - Mg), Ls);
        }
        if (c_last < c_first) Ls = Lc;
        const float inv = 1.f / Ls;  // the row saw at least its own key, so Ls > 0
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          float acc[32];
          if (c_last < c_first) {
            own32(q, acc);
          } else {
#pragma unroll
            for (int e = 0; e < 32; ++e) acc[e] = 0.f;
#pragma unroll 1
            for (int x = c_first; x <= c_last; ++x) {
              float y[32], f = f_own;
              if (x == (int)blockIdx.x) {
                own32(q, y);
              } else {
                const int slot_x = slot_of(x);
                const float mx = __ldcg(a.ws_ml + (size_t)slot_x * kTileM + r).x;
                f = mx == -INFINITY ? 0.f : ex2(mx - Mg);
                const float4* its = a.ws_o + ((size_t)slot_x * 32 + 8 * q) * kTileM + r;
#pragma unroll
                for (int j = 0; j < 8; ++j) *reinterpret_cast<float4*>(y + 4 * j) = __ldcg(its + (size_t)j * kTileM);
              }
#pragma unroll
              for (int e = 0; e < 32; ++e) acc[e] = fmaf(y[e], f, acc[e]);
            }
          }
          if (row_valid) {
#pragma unroll
            for (int e = 0; e < 32; e += 8) store8(32 * q + e, acc + e, inv);
          }
        }
        if (row_valid && a.lse != nullptr) a.lse[(size_t)h * a.n + i] = (Mg + log2f(Ls)) * kLn2;
      }
    } else {
      // Across the cluster (cs = 2 .. 8 CTAs along the key range).  The 16 slices of 8 output columns are owned
      // round-robin: slice s by CTA s % cs, as its slot s / cs.  Every CTA pushes each 8-column piece of its partial that
      // another CTA owns into the owner's receive buffer (the Q, K and V tiles, dead by then), laid out as float4 planes
      // [contributor][slot][half][tile row], and its (m, l) into every CTA, with plain remote stores; after a cluster
      // barrier each owner adds what it received to its own pieces.
      const int cs = a.splits, slots = (16 + cs - 1) / cs;  // (the last slots of some CTAs may be empty)
      const int row2 = c * kTileM + r;
      tc_fence_before();
      cluster.sync();  // every CTA of the cluster is done with its tiles before anyone writes into them
      float2* ml_here = reinterpret_cast<float2*>(pair_smem + kMergeMlOffset);
      // (rows past the tile's last node are padding: nothing of theirs is pushed, reduced or stored)
      if (row_valid)
        for (int q = 0; q < cs; ++q) cluster.map_shared_rank(ml_here, q)[split * 2 * kTileM + row2] = make_float2(M, Lc);
      {
        int owner = 0, slot_i = 0;
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          float x[32];
          own32(q, x);
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            if (owner != split && row_valid) {
              float4* dst = cluster.map_shared_rank(reinterpret_cast<float4*>(pair_smem), owner) + ((split * slots + slot_i) * 2) * (2 * kTileM) + row2;
              dst[0] = make_float4(x[8 * s], x[8 * s + 1], x[8 * s + 2], x[8 * s + 3]);
              dst[2 * kTileM] = make_float4(x[8 * s + 4], x[8 * s + 5], x[8 * s + 6], x[8 * s + 7]);
            }
            if (++owner == cs) { owner = 0; ++slot_i; }
          }
        }
      }
      cluster.sync();
      float Mg = -INFINITY, Ls = 0.f;
#pragma unroll 1
      for (int q = 0; q < cs; ++q) Mg = fmaxf(Mg, row_valid ? ml_here[q * 2 * kTileM + row2].x : 0.f);
#pragma unroll 1
      for (int q = 0; q < cs; ++q) {
        const float2 mlq = row_valid ? ml_here[q * 2 * kTileM + row2] : make_float2(0.f, 1.f);
        if (mlq.x != -INFINITY) Ls = fmaf(mlq.y, ex2(mlq.x - Mg), Ls);
      }
      const float inv = 1.f / Ls;  // some CTA saw the row's own key, so Ls > 0
      const float f_own = M == -INFINITY ? 0.f : ex2(M - Mg);
#pragma unroll 1
      for (int slot_i = 0; slot_i * cs + split < 16; ++slot_i) {
        const int s = slot_i * cs + split;
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (have) {
          tmem_ld8(tmem_o + 8u * s, acc);
          tc_wait_ld();
        }
        if (row_valid) {
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[e] *= f_own;
#pragma unroll 1
          for (int q = 0; q < cs; ++q) {
            if (q == split) continue;
            const float mq = ml_here[q * 2 * kTileM + row2].x;
            const float f = mq == -INFINITY ? 0.f : ex2(mq - Mg);
            const float4* src = reinterpret_cast<const float4*>(pair_smem) + ((q * slots + slot_i) * 2) * (2 * kTileM) + row2;
            const float4 x = src[0], y = src[2 * kTileM];
            acc[0] = fmaf(x.x, f, acc[0]); acc[1] = fmaf(x.y, f, acc[1]); acc[2] = fmaf(x.z, f, acc[2]); acc[3] = fmaf(x.w, f, acc[3]);
            acc[4] = fmaf(y.x, f, acc[4]); acc[5] = fmaf(y.y, f, acc[5]); acc[6] = fmaf(y.z, f, acc[6]); acc[7] = fmaf(y.w, f, acc[7]);
          }
          store8(8 * s, acc, inv);
        }
      }
      if (split == 0 && row_valid && a.lse != nullptr) a.lse[(size_t)h * a.n + i] = (Mg + log2f(Ls)) * kLn2;
    }
    if (kStream) {  // the accumulator has been read: the next segment's first P.V may overwrite it
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm->o_free[c]);
    }
    pos = sg.next;
    ++seg; base += nblk;
    if (stop_here) break;
  }  // segments
  // no remote access happens after the second cluster barrier, so CTAs may leave independently
  tc_fence_before();
  __syncthreads();  // pairs with warp group 0, whose MMA warp then frees the tensor memory
}

}  // namespace pair

// ---------------------------------------------------------------- host side ---------------------
namespace {
struct Shape { int group, nodes_per_tile, tiles, pairs; long units; };
Shape shape_of(const seq_tree_attention_params& p) {
  Shape s;
  s.group = p.num_q_heads / p.num_kv_heads;
  s.nodes_per_tile = pair::kTileM / s.group;
  s.tiles = (p.n_tree + s.nodes_per_tile - 1) / s.nodes_per_tile;
  s.pairs = (s.tiles + 1) / 2;
  s.units = (long)s.pairs * p.num_kv_heads;
  return s;
}
size_t count_bytes(const seq_tree_attention_params& p, const Shape& s) {
  return ((size_t)s.tiles * p.num_kv_heads * sizeof(int32_t) + 255) & ~(size_t)255;
}
size_t ml_bytes() { return (size_t)2 * device_sm_count() * 2 * pair::kTileM * sizeof(float2); }
size_t o_bytes() { return (size_t)2 * device_sm_count() * 2 * 32 * pair::kTileM * sizeof(float4); }
}  // namespace

struct PairPlan { int splits; bool stream; double cost; };  // as tree_attention_api.cu declares it
PairPlan pair_plan(const seq_tree_attention_params& p) {
  const Shape s = shape_of(p);
  PairPlan plan = {1, false, -1.0};
  if (s.tiles < 2) return plan;  // one tile: tree_attention_umma.cu
  const int nblk = pair::pair_blocks(p.prefix_len, p.n_tree), sms = device_sm_count();
  const bool can_stream = s.pairs <= pair::kMaxStreamPairs && p.prefix_len_dev_count <= 1;  // (a range crosses kv heads: one length)
  const double per_block = 1.45, fixed = 5.0;
  for (int cs = 1; cs <= pair::kMaxClusterSplit && p.kernel != 3; ++cs) {
    if (cs > 1 && cs > nblk) break;
    const long waves = (s.units * cs + sms - 1) / sms;
    const double merge = cs == 1 ? 0.0 : 1.6 + 0.5 * (cs - 2);
    const double cost = (double)waves * (per_block * ((nblk + cs - 1) / cs) + fixed + merge);
    if (plan.cost < 0 || cost < plan.cost - 1e-9) plan = {cs, false, cost};
  }
  if (can_stream && p.kernel != 4) {
    const double cost = per_block * ((double)s.units * (nblk + pair::kStreamPairCost) / sms) + fixed + 4.0;
    if (plan.cost < 0 || cost < plan.cost) plan = {1, true, cost};
  }
  return plan;
}

size_t pair_workspace_bytes(const seq_tree_attention_params& p, const PairPlan& plan) {
  return plan.stream ? count_bytes(p, shape_of(p)) + ml_bytes() + o_bytes() : 0;
}

int launch_attention_pair(const seq_tree_attention_params& p, const PairPlan& plan, cudaStream_t stream) {
  const Shape s = shape_of(p);
  const CUtensorMapDataType dt = p.dtype == SEQ_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  CUtensorMap q_map, k_map, v_map;
  {
    // q viewed as [kv head][half][node][head in group][64 elements], see tree_attention_umma.cu
    const cuuint64_t dims[5] = {64, (cuuint64_t)s.group, (cuuint64_t)p.n_tree, 2, (cuuint64_t)p.num_kv_heads};
    const cuuint64_t strides[4] = {(cuuint64_t)p.q_stride_head * 2, (cuuint64_t)p.q_stride_tok * 2, 128, (cuuint64_t)p.q_stride_head * 2 * s.group};
    const cuuint32_t box[5] = {64, (cuuint32_t)s.group, (cuuint32_t)s.nodes_per_tile, pair::kTileM % s.group == 0 ? 2u : 1u, 1};  // (see load_q)
    if (!tensor_map(&q_map, dt, 5, p.q, dims, strides, box)) return SEQ_ERR_CUDA;
  }
  for (int which = 0; which < 2; ++which) {
    // the live rows only (what lies behind them reads as zero); with the length in device memory, the whole cache
    const cuuint64_t dims[4] = {64, (cuuint64_t)(p.prefix_len_dev != nullptr ? p.kv_capacity : p.prefix_len + p.n_tree), 2, (cuuint64_t)p.num_kv_heads};
    const cuuint64_t strides[3] = {(cuuint64_t)p.kv_stride_tok * 2, 128, (cuuint64_t)p.kv_stride_head * 2};
    const cuuint32_t box[4] = {64, (cuuint32_t)pair::kBlockN, 2, 1};
    if (!tensor_map(which == 0 ? &k_map : &v_map, dt, 4, which == 0 ? p.k_cache : p.v_cache, dims, strides, box)) return SEQ_ERR_CUDA;
  }
  pair::Args a;
  a.n = p.n_tree; a.L_host = p.prefix_len; a.Hkv = p.num_kv_heads; a.group = s.group;
  a.mask_wpr = p.mask_words_per_row; a.splits = plan.splits; a.nodes_per_tile = s.nodes_per_tile; a.tiles = s.tiles; a.pairs = s.pairs;
  a.rows = s.nodes_per_tile * s.group;
  a.scale_log2 = (p.softmax_scale > 0.f ? p.softmax_scale : 0.08838834764831845f) * kLog2e;
  const uint32_t fmt = p.dtype == SEQ_BF16 ? 1u : 0u;
  // instruction descriptor: D fp32 (bit 4), A/B format (bits 7, 10), B major (bit 16), N>>3 (bit 17), M>>4 (bit 24)
  const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(pair::kTileM >> 4) << 24);
  a.idesc_qk = idesc | ((uint32_t)(pair::kBlockN >> 3) << 17);           // S: N = 128 keys
  a.idesc_pv = idesc | ((uint32_t)(kHeadDim >> 3) << 17) | (1u << 16);   // O: N = 128, V is MN-major
  a.mask_bits = p.mask_bits; a.parent = p.parent;
  a.out = p.out; a.o_stride_tok = p.o_stride_tok; a.o_stride_head = p.o_stride_head;
  a.lse = p.lse; a.dev_status = p.dev_status;
  a.L_dev = p.prefix_len_dev; a.L_count = p.prefix_len_dev_count; a.zero_tail = p.prefix_len_dev != nullptr ? 1 : 0;
  a.blocks_per_head_host = 0; a.total_blocks_host = 0;
  a.ws_count = nullptr; a.ws_ml = nullptr; a.ws_o = nullptr;
  if (plan.stream) {
    const size_t cnt = count_bytes(p, s);
    if (p.workspace == nullptr || p.workspace_bytes < pair_workspace_bytes(p, plan)) return SEQ_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(p.workspace) % 256 != 0) return SEQ_ERR_INVALID_ARG;
    for (int t = 0; t < s.pairs; ++t) {
      const int i1 = (2 * t + 2) * s.nodes_per_tile < p.n_tree ? (2 * t + 2) * s.nodes_per_tile : p.n_tree;
      a.blocks_per_head_host += pair::kStreamPairCost + pair::pair_blocks(p.prefix_len, i1);
    }
    a.total_blocks_host = (int64_t)a.blocks_per_head_host * p.num_kv_heads;
    uint8_t* ws = static_cast<uint8_t*>(p.workspace);
    a.ws_count = reinterpret_cast<int32_t*>(ws);
    a.ws_ml = reinterpret_cast<float2*>(ws + cnt);
    a.ws_o = reinterpret_cast<float4*>(ws + cnt + ml_bytes());
    SEQ_CUDA_OK(cudaMemsetAsync(a.ws_count, 0, cnt, stream));  // the counters start at zero (the kernel leaves them at zero)
  }
  // Stream schedule: one CTA per SM, but never more CTAs than positions in the layout (a range must not be empty).
  const int sms = device_sm_count();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = plan.stream ? dim3(a.total_blocks_host < sms ? (int)a.total_blocks_host : sms) : dim3(s.pairs, p.num_kv_heads, plan.splits);
  cfg.blockDim = dim3(pair::kThreads);
  cfg.dynamicSmemBytes = sizeof(pair::Smem);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = plan.splits;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // start under the previous kernel's tail (see the kernel)
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  auto launch = [&](auto kernel, int which) -> int {
    static int attr_done[4][64];  // the opt-in shared-memory size is set once per kernel and device
    const int rc = once_per_device(attr_done[which], [&]() -> int {
      SEQ_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(pair::Smem)));
      return SEQ_OK;
    });
    if (rc != SEQ_OK) return rc;
    SEQ_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, q_map, k_map, v_map, a));
    return SEQ_OK;
  };
  if (p.dtype == SEQ_BF16) return plan.stream ? launch(pair::tree_attention_pair_kernel<true, true>, 0) : launch(pair::tree_attention_pair_kernel<true, false>, 1);
  return plan.stream ? launch(pair::tree_attention_pair_kernel<false, true>, 2) : launch(pair::tree_attention_pair_kernel<false, false>, 3);
}

}  // namespace seqtree
