// Tree-masked attention on the 5th-generation tensor cores for many units of long tiles: the stream schedule.
//
// Work unit, tiles and masking are those of tree_attention_umma.cu (a query row is a (node, head-in-group) pair, a tile has
// 128 of them).  One CTA per SM; the 64-key blocks of all units are laid end to end (each tile preceded by a few positions
// that stand for its fixed cost, tiles of a head taken alternately from both ends) and cut into equal ranges.  A CTA works
// through the segments of its range with barrier phases that run on from segment to segment; Q has two buffers, so the next
// segment's loads and first scores are under way while the rows still merge and store.  A tile cut by a range boundary is
// completed by whichever of its CTAs finishes last: the others leave their piece (m, l, unnormalised accumulator) in the
// workspace and count themselves on the tile's counter; the pieces are added in CTA order, so the result does not depend on
// who finishes last.
//
// Keys go in pairs of blocks, 128 keys at a time:
//     S = Q K^T      128x128x128  into one of three S/P buffers of 128 tensor-memory columns
//     P = 2^(scale*S - m) masked  one thread per row of the warp group whose turn the pair is: even pairs chain A, odd pairs B
//     O += P V       128x128x128  one accumulator for both chains, the remaining 128 columns
// With chains of 64-key blocks and an accumulator each (the kernel for shorter ranges) a row thread spends a third of a
// block's time on what a block costs whatever its size - waiting for S, reading it, handing P over - and Q is read from shared
// memory twice as often: 48 cycles per 128x64x16 product where a 128x128x16 one takes 64.  One accumulator is what makes room
// for three S buffers of 128 columns; the price is that both chains have to exponentiate against the same reference maximum
// (see the row threads).
//
// What bounds it: shared memory.  A pair of blocks costs 512 cycles of writes by TMA, 512 of Q and K read by S, 256 of V read by
// P V, 1280 of about 1430; the exponentials take 1024 of them, the products as many.  Calls on several inputs in turn, against
// the kernel with chains of 64 keys: 768 nodes on 4096 keys of 64/8 heads 136.7 -> 124.6 us (bursts of 40, before the power cap
// sets in, 119 -> 104), on 8192 keys 243 -> 201, 384 nodes on 2048 keys of 52 heads 41.3 -> 40.0.  Of that, in bursts, the scores of a pair read in two halves, the second while the first is worked on: 107 -> 104; the
// output through shared memory and Q in two buffers: a tile's end 9000 -> 7000 cycles.  Without gain: a quarter of the
// exponentials as polynomials on the FMA pipe (120 -> 125), P rounded by integer arithmetic (124), the ancestor rows derived
// by the V producer (118 -> 121), the next pair's scores read ahead of this one's hand-over (104 -> 111).
//
// Every mbarrier wait is bounded; a wait that runs out raises SEQ_DEV_TIMEOUT and the CTA drains.
#include <cstddef>

#include <type_traits>

#include "tensor_map.cuh"
#include "umma.cuh"

namespace seqtree {

constexpr uint32_t kPairBytes = kTileBytes;      // a K or V stage: a pair of blocks, 128 keys x 128 elements
constexpr uint32_t kPairHalf = kPairBytes / 2;   // its 128-row x 64-element sub-tiles
constexpr uint32_t kPairBox = kBlockN * 64 * 2;  // what one copy brings: 64 keys x 64 elements
constexpr int kSBufs = 3;                        // S/P buffers
constexpr uint32_t kTmemS = 128;                 // tensor memory: O in columns 0..127, then the S/P buffers

struct StreamSmem {
  // all tiles 1024-byte aligned (128-byte swizzle atoms are 8 rows x 128 B)
  uint8_t q[2][kTileBytes];    // [segment parity]; once the segment's S are done, the rows' output on its way to memory
  uint8_t k[2][kPairBytes];    // [pair parity]
  uint8_t v[2][kPairBytes];
  float2 ml_chain[2][2][kTileM];  // [segment parity][chain]: (m, l) of every row
  float ref[kTileM];              // the rows' reference maximum, handed from chain to chain
  uint64_t q_full[2], q_empty[2];  // empty: the segment's last S has completed, and each warp of row threads has its output out
  uint64_t k_full[2], k_empty[2], v_full[2], v_empty[2];
  uint64_t s_full[kSBufs], p_full[kSBufs], pv_done[kSBufs];
  uint64_t settled[2][4];          // [chain][lane quarter]: the reference of the quarter's rows is settled for the chain's pair
  uint64_t all_done;               // every MMA of this segment has completed (one phase per segment)
  uint64_t o_free;                 // the row threads have read the accumulator (one phase per segment)
  uint32_t tmem_base;
  volatile int abort_flag;
  int32_t abort_seen[2];           // [segment parity]: abort_flag as one row thread saw it, so that all 256 leave together
  int32_t last_part[2];            // [segment parity]: this CTA completes the tile
  // mask from the parent array: the tree, and the ancestor rows of the current tile's nodes (row stride 33 words)
  int32_t parent[SEQ_MAX_TREE];
  uint32_t tile_mask[kTileM][SEQ_MAX_TREE / 32 + 1];
  int32_t tile_prefix[kMaxStreamTiles + 1];  // positions of a kv head's layout before its t-th tile
};
constexpr size_t kStreamSmemBytes = sizeof(StreamSmem) + 1024;
static_assert(kStreamSmemBytes <= 227 * 1024, "one CTA's shared memory");

struct StreamArgs {
  int32_t n, L_host, Hkv, group, mask_wpr, nodes_per_tile, tiles;
  int32_t rows;           // query rows of a full tile: nodes_per_tile * group, 128 when the group divides it
  const int32_t* L_dev;   // nullable: the prefix length in device memory (<= L_host)
  int32_t zero_tail;      // the K/V maps cover the whole cache: rows past the tree are cleared in shared memory
  int32_t blocks_per_head_host, total_blocks_host;  // (a layout of 2^31 positions and more is not streamed)
  int32_t* ws_count;   // [Hkv * tiles] arrivals per tile, zero on entry and on exit
  float2* ws_ml;       // [2 * gridDim.x][128] (m, l) of a partial result
  float4* ws_o;        // [2 * gridDim.x][2][16][128] its unnormalised accumulator, thread-major
  float scale_log2;
  uint32_t idesc_qk, idesc_qk_half, idesc_pv;
  const uint32_t* mask_bits;
  const int32_t* parent;  // used when mask_bits is null
  void* out; int64_t o_stride_tok, o_stride_head;
  float* lse;
  int32_t* dev_status;
};

// `blocks` (1 or 2) blocks of 64 keys from block `blk` on into a K or V stage: its sub-tiles hold 64 elements of all its keys.
__device__ __forceinline__ void load_pair(uint8_t* dst, const CUtensorMap* map, uint64_t* bar, int blk, int blocks, int g) {
  mbar_expect_tx(bar, (uint32_t)blocks * 2u * kPairBox);
  for (int x = 0; x < blocks; ++x) {
    tma_load_4d(dst + x * kPairBox, map, bar, 0, (blk + x) * kBlockN, 0, g);
    tma_load_4d(dst + x * kPairBox + kPairHalf, map, bar, 0, (blk + x) * kBlockN, 1, g);
  }
}

// kFineP: P enters its product as two 16-bit pieces (see tree_attention_umma.cu).
template <bool kBf16, bool kFineP>
__global__ void __launch_bounds__(kUmmaThreads, 1)
tree_attention_stream_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                             const __grid_constant__ CUtensorMap v_map, const StreamArgs a) {
  extern __shared__ uint8_t smem_raw[];
  // (an offset, not a rounded pointer: the compiler keeps seeing shared memory)
  StreamSmem* sm = reinterpret_cast<StreamSmem*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
  const int warp = uniform((int)threadIdx.x >> 5), lane = threadIdx.x & 31;
  // The prefix length: the host's, or - for a step replayed from one CUDA graph while the prefix grows - read from
  // device memory below (the host's value is then the largest it can be, which the launch was planned for).
  int L = a.L_host;
  int blocks_per_head = a.blocks_per_head_host;
  int total_blocks = a.total_blocks_host;
  int range_lo = 0, range_hi = 1;
  // A segment: (kv head, tile, range of the tile's 64-key blocks), a piece of the units that the CTA's range [range_lo,
  // range_hi) of the flattened block space overlaps.
  struct Seg { int g, tile, slot_in_head, i0, i1, blk_lo, nblk, nblk_tile, next; };
  // The tiles of a kv head are laid out alternating from both ends (0, T-1, 1, T-2, ...): late tiles
  // have more masked blocks, which cost more, and this way every range gets its share of them.
  auto tile_at = [&](int k) { return (k & 1) ? a.tiles - 1 - (k >> 1) : (k >> 1); };
  auto seg_at = [&](int pos) -> Seg {
    Seg x;
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
    return x;
  };
  // The barriers are armed once.  Their phases run on from segment to segment: a stage or buffer barrier counts the pairs
  // processed so far, q_full, q_empty, all_done and o_free count segments.
  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sm->q_full[b], 1); mbar_init(&sm->q_empty[b], 9);
      mbar_init(&sm->k_full[b], 1); mbar_init(&sm->k_empty[b], 1);
      mbar_init(&sm->v_full[b], 1); mbar_init(&sm->v_empty[b], 1);
      for (int q = 0; q < 4; ++q) mbar_init(&sm->settled[b][q], 1);
    }
    for (int b = 0; b < kSBufs; ++b) { mbar_init(&sm->s_full[b], 1); mbar_init(&sm->p_full[b], 4); mbar_init(&sm->pv_done[b], 1); }
    mbar_init(&sm->all_done, 1);
    mbar_init(&sm->o_free, 8);    // one arrival per warp of row threads
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sm->abort_flag = 0;
    // programmatic dependent launch: the next kernel in the stream may be scheduled onto free SMs from now on
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  // ... and everything above ran while the previous kernel in the stream was still finishing.  Nothing before this
  // line reads or writes global memory.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (a.L_dev != nullptr) {
    const int v = *a.L_dev;
    if (v < 0 || v > a.L_host) { if (threadIdx.x == 0) dev_flag(a.dev_status, SEQ_DEV_BAD_LENGTH); }
    L = uniform(min(max(v, 0), a.L_host));
    // the flattened block space of this prefix length (every warp for itself)
    int sum = 0;
    for (int t = lane; t < a.tiles; t += 32) sum += kStreamTileCost + (L + min((t + 1) * a.nodes_per_tile, a.n) + kBlockN - 1) / kBlockN;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    blocks_per_head = sum;
    total_blocks = sum * a.Hkv;
  }
  // where the range of CTA x starts: total_blocks * x / ctas.  The launch was planned for the longest prefix; a short one can
  // have fewer positions than the grid has CTAs.  The CTAs that share a cut tile are counted from the ranges and each of them
  // has to arrive, so none of those may be empty: the first `ctas` have one each, the others none.
  const int ctas = min((int)gridDim.x, total_blocks);
  const int per_cta = total_blocks / ctas, left_over = total_blocks - per_cta * ctas;
  auto cta_lo = [&](int x) { return per_cta * x + (left_over * x) / ctas; };
  range_lo = cta_lo(min((int)blockIdx.x, ctas));
  range_hi = cta_lo(min((int)blockIdx.x + 1, ctas));
  if (a.mask_bits == nullptr)
    for (int t = threadIdx.x; t < a.n; t += kUmmaThreads) sm->parent[t] = a.parent[t];
  if (a.rows < kTileM) {  // rows no copy writes (the group does not divide 128): zeros, so that their scores are finite
    for (int t = a.rows * 8 + (int)threadIdx.x; t < kTileM * 8; t += kUmmaThreads)
      for (int b = 0; b < 2; ++b) {
        reinterpret_cast<uint4*>(sm->q[b])[t] = make_uint4(0u, 0u, 0u, 0u);
        reinterpret_cast<uint4*>(sm->q[b] + kHalfBytes)[t] = make_uint4(0u, 0u, 0u, 0u);
      }
    fence_async_smem();
  }
  if (warp == 2) {  // blocks of a kv head before each place of its layout: four places per lane, then a warp scan
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
  if (warp == 1) {  // all 512 tensor-memory columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&sm->tmem_base)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = uniform(sm->tmem_base);

  if (warp < 4) {
    // ============================ warp group 0: data movement and MMA issue, few registers =========
    // The whole warp runs its role's code; copies, MMAs and commits are issued by one elected lane, so coordinates,
    // descriptors and addresses stay warp-uniform.
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLight));
    int seg = 0, base = 0;  // segments done, pairs of blocks in them
    uint32_t issued = 0, issued_parity = 0;   // producers: stages (bits 4, 5: Q) this warp has requested a tile for, and the phase of the last request
    for (int pos = range_lo; pos < range_hi;) {
      const Seg sg = seg_at(pos);
      if (sg.nblk == 0) { pos = sg.next; continue; }
      const int g = sg.g, blk_lo = sg.blk_lo, nblk = sg.nblk, pairs = (nblk + 1) >> 1;
      if (warp == 0 || warp == 3) {
        // TMA producers: warp 0 loads Q and the K tiles, warp 3 the V tiles.  A K stage is free as soon as its S has been
        // computed, a V stage only after the pair's softmax and P V; in one queue the K loads would wait behind the V stages.
        const bool is_v = warp == 3;
        if (!is_v) {
          const int qb = seg & 1, w = seg >> 1;
          if (w > 0 && !mbar_wait(sm, &sm->q_empty[qb], (w - 1) & 1, a.dev_status)) break;
          if (elect_one()) load_q(sm->q[qb], &q_map, &sm->q_full[qb], a.rows, sg.i0, g);
          __syncwarp();
          issued |= 16u << qb;
          issued_parity = (issued_parity & ~(16u << qb)) | ((uint32_t)(w & 1) << (4 + qb));
        }
        const CUtensorMap* map = is_v ? &v_map : &k_map;
        for (int u = 0; u < pairs; ++u) {
          const int b = (base + u) & 1, w = (base + u) >> 1;  // stage, use count of the stage
          uint64_t* full = is_v ? &sm->v_full[b] : &sm->k_full[b];
          uint64_t* empty = is_v ? &sm->v_empty[b] : &sm->k_empty[b];
          if (w > 0 && !mbar_wait(sm, empty, (w - 1) & 1, a.dev_status)) break;
          if (elect_one()) load_pair(is_v ? sm->v[b] : sm->k[b], map, full, blk_lo + 2 * u, min(2, nblk - 2 * u), g);
          __syncwarp();
          issued |= 1u << b;
          issued_parity = (issued_parity & ~(1u << b)) | ((uint32_t)(w & 1) << b);
        }
      } else if (warp == 1) {
        // S issuer: S of a pair goes where P of the pair three before lived
        if (mbar_wait(sm, &sm->q_full[seg & 1], (seg >> 1) & 1, a.dev_status)) {
          const uint32_t q_lo = desc_lo(smem_u32(sm->q[seg & 1]), 16);
          for (int u = 0; u < pairs; ++u) {
            const int x = base + u, w = x / kSBufs, b = x - w * kSBufs, kb = x & 1;
            if (!mbar_wait(sm, &sm->k_full[kb], (x >> 1) & 1, a.dev_status)) break;
            if (w > 0 && !mbar_wait(sm, &sm->pv_done[b], (w - 1) & 1, a.dev_status)) break;
            tc_fence_after();
            if (elect_one()) {  // 128 keys, 64 if the pair has one block
              mma_qk<kHalfBytes, kPairHalf>(tmem + kTmemS + 128u * b, q_lo, desc_lo(smem_u32(sm->k[kb]), 16), 2 * u + 1 < nblk ? a.idesc_qk : a.idesc_qk_half);
              tc_commit(&sm->s_full[b]);
              tc_commit(&sm->k_empty[kb]);
              if (u + 1 == pairs) tc_commit(&sm->q_empty[seg & 1]);
            }
            __syncwarp();
          }
        }
      } else {
        // P V issuer
        for (int u = 0; u < pairs; ++u) {
          const int x = base + u, w = x / kSBufs, b = x - w * kSBufs, vb = x & 1;
          if (!mbar_wait(sm, &sm->v_full[vb], (x >> 1) & 1, a.dev_status)) break;
          if (!mbar_wait(sm, &sm->p_full[b], w & 1, a.dev_status)) break;
          // the first P V of a segment overwrites O: the row threads must have read the previous segment's
          if (u == 0 && seg > 0 && !mbar_wait(sm, &sm->o_free, (seg - 1) & 1, a.dev_status)) break;
          if (a.zero_tail) {
            // The tensor maps of this mode cover the whole cache, so a pair that reaches past the last tree row has
            // fetched rows that may hold anything; their probabilities are exactly 0, but 0 * NaN is not: the rows are
            // cleared here (whole 128-byte rows of both halves: the swizzle stays inside a row), and the clearing is
            // made visible to the tensor core's reads.
            const int live = L + a.n - (blk_lo + 2 * u) * kBlockN;  // rows of this pair that exist
            if (live < 2 * kBlockN) {
              uint4* vt = reinterpret_cast<uint4*>(sm->v[vb]);
              for (int i = max(live, 0) * 8 + lane; i < 2 * kBlockN * 8; i += 32) {
                vt[i] = make_uint4(0u, 0u, 0u, 0u);
                vt[kPairHalf / 16 + i] = make_uint4(0u, 0u, 0u, 0u);
              }
              fence_async_smem();
              __syncwarp();
            }
          }
          tc_fence_after();
          const uint32_t pa = tmem + kTmemS + 128u * b, v_lo = desc_lo(smem_u32(sm->v[vb]), kPairHalf);
          if (elect_one()) {
            const bool both = 2 * u + 1 < nblk;  // (a block that is not there has no V, and its P is not used)
            mma_pv(tmem, pa, v_lo, a.idesc_pv, u > 0 ? 1u : 0u);
            if (both) mma_pv(tmem, pa + 32u, v_lo + (kPairBox >> 4), a.idesc_pv, 1u);
            if (kFineP) {
              mma_pv(tmem, pa + 64u, v_lo, a.idesc_pv, 1u);
              if (both) mma_pv(tmem, pa + 96u, v_lo + (kPairBox >> 4), a.idesc_pv, 1u);
            }
            tc_commit(&sm->pv_done[b]);
            tc_commit(&sm->v_empty[vb]);
          }
          __syncwarp();
        }
        if (elect_one()) tc_commit(&sm->all_done);  // arrives when every P V of this segment has completed (no S outlives its P V)
        __syncwarp();
      }
      __syncwarp();
      pos = sg.next;
      ++seg; base += pairs;
      if (sm->abort_flag) break;
    }
    // A CTA that gives up must not leave while a tile it has requested is still on its way into its shared memory
    // (the next CTA on this SM could get that memory): the producers wait, with a bound of their own, for the last
    // tile requested into each stage.  (Whether its consumer has taken that phase or not, the parity test answers
    // when the bytes have landed.  Tiles requested earlier into the same stage landed before the stage was reused.)
    if (sm->abort_flag && (warp == 0 || warp == 3)) {
      for (int st = 0; st < 6; ++st) {
        if (!((issued >> st) & 1u)) continue;
        uint64_t* full = st >= 4 ? &sm->q_full[st & 1] : (warp == 3 ? &sm->v_full[st] : &sm->k_full[st]);
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

  // ============================== warp groups 1, 2: one thread per query row ============
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsRows));
  const int chain = (warp >> 2) - 1;
  const int quad = warp & 3;                  // tensor-memory lane quarter this warp may access
  const int r = quad * 32 + lane;             // row of the tile = tensor-memory lane
  const uint32_t lane_sel = (uint32_t)(quad * 32) << 16;
  const uint32_t tmem_o = tmem + lane_sel;
  int seg = 0, base = 0, base_a = 0, base_b = 0;  // segments done, pairs in them, those of chains A and B
  for (int pos = range_lo; pos < range_hi;) {
  const Seg sg = seg_at(pos);
  if (sg.nblk == 0) { pos = sg.next; continue; }
  const int g = sg.g, i0 = sg.i0, blk_lo = sg.blk_lo, nblk = sg.nblk, pairs = (nblk + 1) >> 1;
  const int i = i0 + r / a.group;             // node of this row
  const int h = g * a.group + r % a.group;
  const bool row_valid = i < sg.i1;           // (a row past the tile's nodes may be one of the next tile's)
  // The row's ancestor bits: the caller's mask, or rows derived from the parent array at the start of the
  // segment by the first thread of each node (0 <= parent[j] < j, so a walk ends; anything else is flagged and
  // read as "no parent").
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
  // A warp whose 32 rows all lie past the tile's last node leaves the special-function unit and the issue slots to the
  // warps with real rows; its P rows stay whatever they are (rows of the product are independent).
  const bool warp_live = i0 + (quad * 32) / a.group < sg.i1;
  for (int u = chain; u < pairs && ok; u += 2) {
    const int w = (base + u) / kSBufs, b = (base + u) - w * kSBufs;
    const uint32_t tmem_s = tmem + kTmemS + 128u * b + lane_sel;
    if (!mbar_wait(sm, &sm->s_full[b], w & 1, a.dev_status)) { ok = false; break; }
    if (!warp_live) {  // 32 padding rows: nothing to compute, only keep in step with the barriers
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&sm->settled[chain][quad]);
        mbar_arrive(&sm->p_full[b]);
      }
      continue;
    }
    tc_fence_after();
    uint32_t sreg[128];
    // The second half of the scores is on its way while the first is worked on.
    tmem_ld32(tmem_s, sreg, 0);
    tmem_ld32(tmem_s + 32u, sreg, 32);
    auto second_half = [&]() {
      tc_wait_ld();
#pragma unroll
      for (int e = 64; e < 128; ++e) asm volatile("" : "+r"(sreg[e]));  // (nothing of it moves ahead of the wait)
    };
    const int kb = (blk_lo + 2 * u) * kBlockN;
    const bool masked = kb + 2 * kBlockN > L || 2 * u + 1 >= nblk;  // the pair reaches into the tree keys (or past the end)
    uint32_t vis[4] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu};
    if (masked) {
#pragma unroll
      for (int x = 0; x < 4; ++x) vis[x] = x < 2 || 2 * u + 1 < nblk ? mask_window(mrow, mask_wpr, a.n, kb - L + 32 * x) : 0u;
    }
    tc_wait_ld();
#pragma unroll
    for (int e = 0; e < 64; ++e) asm volatile("" : "+r"(sreg[e]));
    tmem_ld32(tmem_s + 64u, sreg, 64);
    tmem_ld32(tmem_s + 96u, sreg, 96);
    if (masked) {  // masked scores become -inf: probability exactly 0, and they cannot raise the maximum
      second_half();
#pragma unroll
      for (int e = 0; e < 128; ++e)
        if (!(vis[e >> 5] & (1u << (e & 31)))) sreg[e] = __float_as_uint(-INFINITY);
    }
    // P = 2^(scale*s - m) written over S as packed 16-bit values (64 columns, four stores of 16; with kFineP the rests in the
    // 64 columns behind); returns the row sum.
    // (A row without a reference sees nothing in this pair: its scores are all -inf and its P are 0.)
    auto exponentials = [&]() -> float {
      const float neg_m = m_used == -INFINITY ? 0.f : -m_used;
      const uint64_t sc2 = pair_of(sc, sc), neg_m2 = pair_of(neg_m, neg_m);
      uint64_t sm2[2] = {pair_of(0.f, 0.f), pair_of(0.f, 0.f)};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        // (with kFineP the first store already goes to columns that the second half is read from, and nothing but a wait orders
        // a store to tensor memory behind a load)
        if (c == (kFineP ? 0 : 2)) second_half();
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
        if (kFineP) tmem_st16(tmem_s + 64u + 16u * c, rest);
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
    // Both chains add to one accumulator, so they share the reference: it is settled pair by pair in key order, and a
    // pair's P goes out only when the pair before it (the other chain's) is settled.  If that one moved the reference,
    // this one follows and repeats its pass.  (The other chain being half a pair ahead, the wait is rarely one.)
    const bool opening = u == 0 && chain == 0;  // the segment's first pair
    bool mine = opening;                        // everything before this pair is settled: the reference is this warp's to move
    float ref = -INFINITY;                      // ... and what it is
    bool settle = __any_sync(0xffffffffu, m_used == -INFINITY);
    float sum;
#pragma unroll 1
    for (;;) {  // (a loop, so that the exponentials' code exists once)
      if (settle) {
        if (!mine) {
          if (!mbar_wait(sm, &sm->settled[chain ^ 1][quad], ((chain ? base_a : base_b) + ((u - 1) >> 1)) & 1, a.dev_status)) { ok = false; break; }
          mine = true;
          ref = sm->ref[r];
        }
        if (ref != m_used) {
          l *= m_used == -INFINITY ? 0.f : ex2(m_used - ref);
          m_used = ref;
        }
        second_half();
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int e = 0; e < 128; e += 2)  // three-input maximum: two scores per instruction
          mx[(e >> 1) & 3] = max3(mx[(e >> 1) & 3], __uint_as_float(sreg[e]), __uint_as_float(sreg[e + 1]));
        const float m_blk = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sc;  // scale > 0
        const bool move = m_blk > m_used + kRescaleThreshold || (m_used == -INFINITY && m_blk != -INFINITY);
        if (__any_sync(0xffffffffu, move)) {
          float alpha = 1.f;
          if (move) {
            alpha = m_used == -INFINITY ? 0.f : ex2(m_used - m_blk);
            l *= alpha;
            m_used = m_blk;
          }
          if (!opening) {
            // O may still be taking the pair before: wait for it, then rescale this warp's rows.  (The barrier's phase
            // before is over, as a parity wait needs: it counted the pair whose P lived there before that pair's S.)
            if (!mbar_wait(sm, &sm->pv_done[(base + u - 1) % kSBufs], ((base + u - 1) / kSBufs) & 1, a.dev_status)) { ok = false; break; }
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
      if (!settle && !mine) {
        if (!mbar_wait(sm, &sm->settled[chain ^ 1][quad], ((chain ? base_a : base_b) + ((u - 1) >> 1)) & 1, a.dev_status)) { ok = false; break; }
        mine = true;
        ref = sm->ref[r];
        settle = __any_sync(0xffffffffu, ref != m_used);
      }
      if (!settle) break;
      tc_wait_st();  // (a pass that is repeated stores to the same columns, and stores are not ordered among themselves)
    }
    if (!ok) break;
    if (opening || m_used != ref) sm->ref[r] = m_used;
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm->settled[chain][quad]);
    l += sum;
    tc_wait_st();
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm->p_full[b]);  // one arrival per warp
  }
  // The tile's other pieces (a range boundary cuts it): its positions in the layout, and the CTAs whose ranges hold some.
  const bool piece = nblk < sg.nblk_tile;
  int t0 = 0, c_first = 0, c_last = 0;
  int* const cnt = a.ws_count + (size_t)g * a.tiles + sg.tile;
  int counted = 0;  // one thread: the pieces counted by now, looked up while the last products finish
  if (piece) {
    t0 = g * blocks_per_head + sm->tile_prefix[sg.slot_in_head] + kStreamTileCost;
    const int t1 = t0 + sg.nblk_tile;
    c_first = min((int)((float)t0 / (float)total_blocks * (float)ctas), ctas - 1);  // the CTA whose range holds block t0 ...
    while (cta_lo(c_first + 1) <= t0) ++c_first;                      // ... exactly
    while (cta_lo(c_first) > t0) --c_first;
    c_last = c_first;
    while (cta_lo(c_last + 1) < t1) ++c_last;
    if (threadIdx.x == 128) counted = *reinterpret_cast<volatile int*>(cnt);
  }
  // Every MMA must have completed before O is read and Q is overwritten.
  if (ok) ok = mbar_wait(sm, &sm->all_done, seg & 1, a.dev_status);
  tc_fence_after();

  // ---------------------------------------------------------------- merge ------------------------
  // A warp may read any column of its 32 lanes, so the thread of chain c and row r takes columns [64c, 64c+64) of O.  The
  // two chains' sums meet in shared memory; the later reference of the two is the one O is in.
  sm->ml_chain[seg & 1][chain][r] = (ok && pairs > chain) ? make_float2(m_used, l) : make_float2(-INFINITY, 0.f);
  // Whether to stop after this segment is decided once for all row threads: a flag raised between two threads' own
  // reads would send some to the closing barrier and the rest into the next segment's bar.sync, which has no bound.
  // If every other piece has been counted already (the usual case for the piece that closes a range: the others were
  // finished long ago), this CTA completes the tile without writing its own piece.
  if (threadIdx.x == 128) {
    sm->abort_seen[seg & 1] = sm->abort_flag;
    const bool done = piece && counted == c_last - c_first;
    if (done) *cnt = 0;  // leave the counter as it was found
    sm->last_part[seg & 1] = done;
  }
  asm volatile("bar.sync 1, 256;" ::: "memory");  // the 256 row threads only
  const bool stop_here = sm->abort_seen[seg & 1] != 0;
  const float2 mlA = sm->ml_chain[seg & 1][0][r], mlB = sm->ml_chain[seg & 1][1][r];
  float M = fmaxf(mlA.x, mlB.x);  // reference maximum and denominator of what this CTA holds of the row
  float Lc = (mlA.x == -INFINITY ? 0.f : mlA.y * ex2(mlA.x - M)) + (mlB.x == -INFINITY ? 0.f : mlB.y * ex2(mlB.x - M));
  float merged[64];               // its columns [64*chain, 64*chain + 64), unnormalised
  if (ok) {
    tmem_ld32(tmem_o + 64u * chain, reinterpret_cast<uint32_t*>(merged), 0);
    tmem_ld32(tmem_o + 64u * chain + 32u, reinterpret_cast<uint32_t*>(merged), 32);
    tc_wait_ld();
  } else {
#pragma unroll
    for (int e = 0; e < 64; ++e) merged[e] = 0.f;
  }
  // the accumulator is in registers: the next segment's first P V may overwrite it
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(&sm->o_free);
  bool complete = true;  // this CTA writes the tile's output
  if (piece) {
    // Every piece is written to this CTA's slot of the workspace (slot 0 if the piece opens the CTA's range, else 1), then
    // counted; the CTA whose count completes the tile adds the other pieces to its own and writes the output.  Nobody waits
    // for anybody.
    auto slot_of = [&](int c) { return 2 * c + (max(t0, cta_lo(c)) == cta_lo(c) ? 0 : 1); };
    complete = sm->last_part[seg & 1] != 0;
    if (!complete) {
      const int my_slot = slot_of((int)blockIdx.x);
      if (chain == 0) a.ws_ml[(size_t)my_slot * kTileM + r] = make_float2(M, Lc);
      float4* my_o = a.ws_o + ((size_t)(my_slot * 2 + chain) * 16) * kTileM + r;
#pragma unroll
      for (int j = 0; j < 16; ++j) my_o[(size_t)j * kTileM] = make_float4(merged[4 * j], merged[4 * j + 1], merged[4 * j + 2], merged[4 * j + 3]);
      __threadfence();
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (threadIdx.x == 128) {
        const int last = atomicAdd(cnt, 1) == c_last - c_first;
        if (last) *cnt = 0;  // every piece has been counted
        sm->last_part[seg & 1] = last;
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      complete = sm->last_part[seg & 1] != 0;
    }
    if (complete) {
      // The pieces are added in the order of their CTAs, this CTA's own (from registers) at its place, with one
      // common reference maximum: the result does not depend on which CTA happened to finish last.
      __threadfence();
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
            const float4* its = a.ws_o + ((size_t)(slot * 2 + chain) * 16 + 8 * half) * kTileM + r;
            float4 x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = __ldcg(its + (size_t)j * kTileM);
            const float2 ml = __ldcg(a.ws_ml + (size_t)slot * kTileM + r);
            const float f = ml.x == -INFINITY ? 0.f : ex2(ml.x - Mg);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              acc[4 * j] = fmaf(x[j].x, f, acc[4 * j]);
              acc[4 * j + 1] = fmaf(x[j].y, f, acc[4 * j + 1]);
              acc[4 * j + 2] = fmaf(x[j].z, f, acc[4 * j + 2]);
              acc[4 * j + 3] = fmaf(x[j].w, f, acc[4 * j + 3]);
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
  if (complete) {
    // Out through this warp's 32 rows of the Q tile, where 16 bytes of 32 rows turn into 128 bytes of four: a store of one
    // 16-byte word per row touches 32 lines.  (Rows past the tile's nodes stay as they are: zeros where no copy of Q writes.)
    uint8_t* stage = sm->q[seg & 1] + (uint32_t)chain * kHalfBytes + (uint32_t)quad * 4096u;
    const float inv = 1.f / Lc;  // the row saw at least its own key, so Lc > 0
    if (row_valid) {
#pragma unroll
      for (int e = 0; e < 64; e += 8) {
        uint4 val;
        val.x = pack2<kBf16>(merged[e] * inv, merged[e + 1] * inv);
        val.y = pack2<kBf16>(merged[e + 2] * inv, merged[e + 3] * inv);
        val.z = pack2<kBf16>(merged[e + 4] * inv, merged[e + 5] * inv);
        val.w = pack2<kBf16>(merged[e + 6] * inv, merged[e + 7] * inv);
        *reinterpret_cast<uint4*>(stage + lane * 128 + (((e >> 3) ^ (lane & 7)) << 4)) = val;
      }
      if (chain == 0 && a.lse != nullptr) a.lse[(size_t)h * a.n + i] = (M + log2f(Lc)) * kLn2;
    }
    __syncwarp();
    const int64_t mine = row_valid ? 2 * ((int64_t)i * a.o_stride_tok + (int64_t)h * a.o_stride_head) : -1;  // (strides are positive)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int row = 4 * j + (lane >> 3);
      const int64_t at = __shfl_sync(0xffffffffu, mine, row);
      const uint4 val = *reinterpret_cast<const uint4*>(stage + row * 128 + (((lane & 7) ^ (row & 7)) << 4));
      if (at >= 0) *reinterpret_cast<uint4*>(static_cast<uint8_t*>(a.out) + at + 128 * chain + 16 * (lane & 7)) = val;
    }
    fence_async_smem();  // (the next Q tile arrives by the asynchronous proxy)
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(&sm->q_empty[seg & 1]);
  pos = sg.next;
  ++seg; base += pairs; base_a += (pairs + 1) >> 1; base_b += pairs >> 1;
  if (stop_here) break;
  }  // segments
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
// Workspace: one arrival counter per (kv head, tile), then two slots per CTA for the pieces of tiles that its range cuts:
// (m, l) per row and the 128 x 128 fp32 accumulator.
static int tiles_of(const seq_tree_attention_params& p) {
  const int nodes_per_tile = kTileM / (p.num_q_heads / p.num_kv_heads);
  return (p.n_tree + nodes_per_tile - 1) / nodes_per_tile;
}
static size_t stream_count_bytes(const seq_tree_attention_params& p) {
  return ((size_t)tiles_of(p) * p.num_kv_heads * sizeof(int32_t) + 255) & ~(size_t)255;
}
static size_t stream_ml_bytes() { return (size_t)2 * device_sm_count() * kTileM * sizeof(float2); }
static size_t stream_o_bytes() { return (size_t)2 * device_sm_count() * 2 * 16 * kTileM * sizeof(float4); }
size_t stream_workspace_bytes(const seq_tree_attention_params& p) { return stream_count_bytes(p) + stream_ml_bytes() + stream_o_bytes(); }

int launch_attention_stream(const seq_tree_attention_params& p, cudaStream_t stream) {
  const int G = p.num_q_heads / p.num_kv_heads;
  const int tiles = tiles_of(p);
  CUtensorMap q_map, k_map, v_map;
  if (!attention_maps(p, 1, &q_map, &k_map, &v_map)) return SEQ_ERR_CUDA;
  if (p.workspace == nullptr || p.workspace_bytes < stream_workspace_bytes(p)) return SEQ_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(p.workspace) % 256 != 0) return SEQ_ERR_INVALID_ARG;

  StreamArgs a;
  a.n = p.n_tree; a.L_host = p.prefix_len; a.Hkv = p.num_kv_heads; a.group = G;
  a.mask_wpr = p.mask_words_per_row; a.nodes_per_tile = kTileM / G; a.tiles = tiles;
  a.rows = a.nodes_per_tile * G;
  a.L_dev = p.prefix_len_dev; a.zero_tail = p.prefix_len_dev != nullptr ? 1 : 0;
  a.blocks_per_head_host = 0;
  for (int t = 0; t < tiles; ++t) {
    const int i1 = (t + 1) * a.nodes_per_tile < p.n_tree ? (t + 1) * a.nodes_per_tile : p.n_tree;
    a.blocks_per_head_host += kStreamTileCost + (p.prefix_len + i1 + kBlockN - 1) / kBlockN;
  }
  a.total_blocks_host = a.blocks_per_head_host * p.num_kv_heads;
  uint8_t* ws = static_cast<uint8_t*>(p.workspace);
  const size_t cnt_bytes = stream_count_bytes(p);
  a.ws_count = reinterpret_cast<int32_t*>(ws);
  a.ws_ml = reinterpret_cast<float2*>(ws + cnt_bytes);
  a.ws_o = reinterpret_cast<float4*>(ws + cnt_bytes + stream_ml_bytes());
  const float scale = p.softmax_scale > 0.f ? p.softmax_scale : 0.08838834764831845f;
  a.scale_log2 = scale * kLog2e;
  const uint32_t fmt = p.dtype == SEQ_BF16 ? 1u : 0u;
  // instruction descriptor: D fp32 (bit 4), A/B format (bits 7, 10), B major (bit 16), N>>3 (bit 17), M>>4 (bit 24)
  const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(kTileM >> 4) << 24);
  a.idesc_qk = idesc | ((uint32_t)(2 * kBlockN >> 3) << 17);             // S: N = 128 keys
  a.idesc_qk_half = idesc | ((uint32_t)(kBlockN >> 3) << 17);            // ... of a pair with one block: 64
  a.idesc_pv = idesc | ((uint32_t)(kHeadDim >> 3) << 17) | (1u << 16);   // O: N = 128, V is MN-major
  a.mask_bits = p.mask_bits;
  a.parent = p.parent;
  a.out = p.out; a.o_stride_tok = p.o_stride_tok; a.o_stride_head = p.o_stride_head;
  a.lse = p.lse;
  a.dev_status = p.dev_status;

  cudaLaunchAttribute early[1];  // start under the previous kernel's tail (see the kernels)
  early[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early[0].val.programmaticStreamSerializationAllowed = 1;
  // The counters start at zero.  A kernel of one's own, not a memset: it is scheduled under the tail of the launch before
  // and lets the attention's set-up run under itself (768 nodes on 4096 keys of 64/8 heads 123.1 -> 120.8 us, 384 on 2048
  // of 52 heads 43.1 -> 40.9).
  cudaLaunchConfig_t zero = {};
  const int words = (int)(cnt_bytes / sizeof(int32_t));
  zero.gridDim = dim3((words + 255) / 256);
  zero.blockDim = dim3(256);
  zero.stream = stream;
  zero.attrs = early;
  zero.numAttrs = 1;
  SEQ_CUDA_OK(cudaLaunchKernelEx(&zero, zero_words_kernel, a.ws_count, words));

  cudaLaunchConfig_t cfg = {};
  // One CTA per SM, but no more than positions in the layout (of the longest prefix: see the kernel).
  const int sms = device_sm_count();
  cfg.gridDim = dim3(a.total_blocks_host < sms ? a.total_blocks_host : sms);
  cfg.blockDim = dim3(kUmmaThreads);
  cfg.dynamicSmemBytes = kStreamSmemBytes;
  cfg.stream = stream;
  cfg.attrs = early;
  cfg.numAttrs = 1;
  auto launch = [&](auto kernel, int which) -> int {
    static int attr_done[4][64];  // the opt-in shared-memory size is set once per kernel and device
    const int rc = once_per_device(attr_done[which], [&]() -> int {
      SEQ_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStreamSmemBytes));
      return SEQ_OK;
    });
    if (rc != SEQ_OK) return rc;
    SEQ_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, q_map, k_map, v_map, a));
    return SEQ_OK;
  };
  const bool fine = kTileM % G != 0;
  if (p.dtype == SEQ_BF16) return fine ? launch(tree_attention_stream_kernel<true, true>, 0) : launch(tree_attention_stream_kernel<true, false>, 1);
  return fine ? launch(tree_attention_stream_kernel<false, true>, 2) : launch(tree_attention_stream_kernel<false, false>, 3);
}

}  // namespace seqtree
