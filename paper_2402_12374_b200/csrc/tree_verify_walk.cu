// seq_tree_verify, the walk with rows in registers: Algorithm 2 of the Sequoia paper applied from the root down the
// tree (Section 2.2) by ONE cluster of 16 CTAs, the next node's rows already on their way while the current node's
// children are being tested.
//
// The vocabulary is cut into one contiguous slice per CTA and one contiguous segment per warp; a thread keeps its
// 4 * NCH elements of the target row and of the draft row in registers (8 elements per row at 32000 tokens, 32 at
// 128256), so every vocabulary-wide pass (exponentials, the residual's normaliser after a rejection) is a few
// instructions per thread, followed by one warp reduction and one table of per-warp partials, sent into every CTA's shared
// memory and counted in there by an mbarrier.  What the walk will need next is known one step ahead: while child i of
// the current node is being tested, child i's own rows are loaded into a second set of registers (they are needed
// exactly if child i is accepted); on a rejection the loads for child i + 1 are issued before the residual pass, so
// they land behind that pass and its exchange.  A visited node therefore costs its arithmetic and one exchange, not
// a trip to HBM, unless the accepted child was decided within a microsecond.
//
// Arithmetic: R and D of Algorithm 2 are never materialised.  With p, q the two softmaxes and S the rejected set,
//     R[t] = max(p[t] - C q[t] - U, 0) / Z ,     D[t] = q[t] / ZD   (or 1/(V-|S|) once the uniform fallback has fired)
// for scalars C, U, Z, ZD: the residual update R <- norm(max(R - D, 0)) is C += Z/ZD (or U += Z/(V-|S|)) and one sum
// for the new Z; sum(D) is the direct sum of the surviving q.  A rejected token needs no clearing in R: the rejection
// says R[s] < D[s], which makes max(p[s] - C q[s] - U, 0) zero from the new C (or U) on; the final draw applies the
// marks all the same.  The per-warp partial sums of the last pass are the coarse level of the final inverse CDF,
// which the one warp that holds the crossing finishes on its own.
//
// Serves the default mode and the variant without the draft update at T > 0, and - with kernels of their own at the end of
// this file - greedy decoding (T = 0, every mode) and sampling from the target (T > 0, fp32 logits); the every-node hook and
// what does not fit the registers run on the kernels of tree_verify.cu.
#include <cooperative_groups.h>
#include <float.h>
#include <limits.h>
#include <math.h>

#include "common.cuh"
#include "trace.cuh"
#include "tree_verify_nodes.cuh"

namespace cg = cooperative_groups;

namespace seqtree {
namespace vwk {

constexpr int kCl = 16;               // CTAs in the cluster of one request (not a portable size: asked for, and checked, at launch)
constexpr int kClBatch = 8;           // ... of each request of a batch too large for clusters of 16 side by side
constexpr int kTh = 256;              // threads per CTA
constexpr int kWarps = kTh / 32;
// (rank, warp) segments, in vocabulary order: CL * kWarps of them; table entries per lane: CL / 4

struct Shared {
  int32_t parent[SEQ_MAX_TREE];
  int32_t tokens[SEQ_MAX_TREE];
  float uniforms[SEQ_MAX_TREE + 1];
  uint32_t has_child[SEQ_MAX_TREE / 32];
  // The current node's children in ascending order (the order they were drawn in): (node, token).  Two copies, used in
  // turn: a warp may still be reading the previous node's.  After the last test: scratch of the final draw's fine level.
  int2 kid[2][SEQ_MAX_TREE];
  int32_t chunk_cnt[32];              // children among nodes [32 j, 32 j + 32)
  float4 xbuf[2][kCl * kWarps];             // cluster exchange: one entry per (rank, warp), double-buffered
  uint64_t xbar[2];                   // ... and the mbarrier that counts each buffer's bytes in
  float4 drawn[2];                    // sampling walk: the drawn token, from the warp that found it; used in turn
  uint64_t dbar[2];
  int32_t node_flags;
  int32_t pick[2][4];                 // greedy walk, by hop parity: the matching child, the first child with a bad token, the first child
};

__device__ __forceinline__ float fast_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rel_exp(float m, float M, float c2) { return m == -INFINITY ? 0.f : fast_ex2((m - M) * c2); }
__device__ __forceinline__ float resid(float pn, float qn, float Cf, float Uf) { return fmaxf(fmaf(-Cf, qn, pn) - Uf, 0.f); }
__device__ __forceinline__ float max_lanes(float v) {
  float m;
  asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(v));
  return m;
}
__device__ __forceinline__ double sum_lanes(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// 1 / x for a positive double to nearly full precision without the division routine
__device__ __forceinline__ double fast_rcp(double x) {
  double r = (double)__frcp_rn((float)x);
  r = r * (2.0 - x * r);
  return r * (2.0 - x * r);
}
// A logit as the kernels read it: NaN counts as -inf, +inf as the largest finite value (both are flagged).
__device__ __forceinline__ float clean_logit(float x) { return x == x ? fminf(x, FLT_MAX) : -INFINITY; }

struct Ctx {
  Shared* sh;
  int rank, lo, cnt;     // CTA in cluster, its vocabulary slice
  int tid, warp, lane;
  uint32_t local, remote;  // shared-window addresses of this CTA's Shared and of CTA `lane`'s
  uint32_t xn;             // exchanges done
};

// One row slice into registers: NCH independent 16-byte loads per thread, the ragged end element by element;
// positions past the slice read as -inf (probability 0).  A warp holds 128 * NCH consecutive elements, in chunks of
// 128; within a chunk a lane holds four consecutive ones.
__device__ __forceinline__ float bf16_bits_to_float(uint32_t b) { return __uint_as_float(b << 16); }  // exact
template <bool kBf16>
__device__ __forceinline__ float load_logit(const void* row, int64_t i) {
  if (kBf16) return bf16_bits_to_float(__ldg(static_cast<const unsigned short*>(row) + i));
  return __ldg(static_cast<const float*>(row) + i);
}
// One row slice into registers, as it lies in memory: NCH independent loads per thread (16 bytes each for fp32 logits,
// 8 for 16-bit ones), the ragged end element by element; positions past the slice read as -inf (probability 0).  A
// warp holds 128 * NCH consecutive elements, in chunks of 128; within a chunk a lane holds four consecutive ones.
// Nothing here touches the loaded values, so the loads stay in flight until widen() is called on them: that is what
// lets the next node's rows travel while the current node is worked on.
template <int NCH, bool kBf16>
struct RawRow { uint32_t w[kBf16 ? 2 * NCH : 4 * NCH]; };
template <int NCH, bool kBf16>
__device__ __forceinline__ void load_row(const Ctx& c, const void* row_v, RawRow<NCH, kBf16>& r) {
  const int first = c.warp * (128 * NCH) + c.lane * 4;
  const int room = c.cnt - first;
  if (kBf16) {
    const unsigned short* base = static_cast<const unsigned short*>(row_v) + c.lo + first;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      uint2 v;
      if (room - 128 * j >= 4) {
        v = __ldcs(reinterpret_cast<const uint2*>(base + 128 * j));
      } else {
        const uint32_t h0 = room - 128 * j > 0 ? __ldcs(base + 128 * j) : 0xFF80u, h1 = room - 128 * j > 1 ? __ldcs(base + 128 * j + 1) : 0xFF80u;
        const uint32_t h2 = room - 128 * j > 2 ? __ldcs(base + 128 * j + 2) : 0xFF80u;  // (0xFF80: -inf)
        v = make_uint2(h0 | (h1 << 16), h2 | (0xFF80u << 16));
      }
      r.w[2 * j] = v.x; r.w[2 * j + 1] = v.y;
    }
  } else {
    const float* base = static_cast<const float*>(row_v) + c.lo + first;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      float4 v;
      if (room - 128 * j >= 4) {
        v = __ldcs(reinterpret_cast<const float4*>(base + 128 * j));
      } else {
        v.x = room - 128 * j > 0 ? __ldcs(base + 128 * j) : -INFINITY;
        v.y = room - 128 * j > 1 ? __ldcs(base + 128 * j + 1) : -INFINITY;
        v.z = room - 128 * j > 2 ? __ldcs(base + 128 * j + 2) : -INFINITY;
        v.w = -INFINITY;
      }
      r.w[4 * j] = __float_as_uint(v.x); r.w[4 * j + 1] = __float_as_uint(v.y);
      r.w[4 * j + 2] = __float_as_uint(v.z); r.w[4 * j + 3] = __float_as_uint(v.w);
    }
  }
}
// The lines that load_row will read, asked for before the previous kernel has ended: the tree's arrays, node 0's rows and the
// target row of node 1, the root's first child (which the walk requests before it knows whether it needs it).  Not node 1's
// draft row: it need not exist if node 1 is a leaf, and the tree is not known yet.  In calls on several sets of inputs in turn
// 768 nodes x 128256 tokens 18.6 -> 18.4 us, 16 requests of 64 x 32000 21.5 -> 21.15, greedy 128 x 32000 5.23 -> 5.18; with
// node 1's draft row the same.
template <int NCH, bool kBf16>
__device__ __forceinline__ void prefetch_row(const Ctx& c, const void* row) {
  constexpr int kEsz = kBf16 ? 2 : 4, kLine = 128 / kEsz;  // elements of a line
#pragma unroll
  for (int x = 0; x < 128 * NCH; x += 32 * kLine) {
    const int at = x + c.lane * kLine;
    if (at < 128 * NCH && c.warp * (128 * NCH) + at < c.cnt) prefetch_l2(static_cast<const char*>(row) + (int64_t)(c.lo + c.warp * (128 * NCH) + at) * kEsz);
  }
}
template <bool kUniforms>
__device__ __forceinline__ void prefetch_tree(const Ctx& c, const VerifyArgs& a) {
  const int i = 32 * c.tid;  // a line of 32 words
  if (i < a.n) {
    prefetch_l2(a.parent + i);
    prefetch_l2(a.tokens + i);
    if (kUniforms) prefetch_l2(a.uniforms + i);
  }
}
// ... and widened to fp32 (exact)
template <int NCH, bool kBf16>
__device__ __forceinline__ void widen(const RawRow<NCH, kBf16>& r, float* x) {
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    if (kBf16) {
      x[4 * j] = __uint_as_float(r.w[2 * j] << 16); x[4 * j + 1] = __uint_as_float(r.w[2 * j] & 0xFFFF0000u);
      x[4 * j + 2] = __uint_as_float(r.w[2 * j + 1] << 16); x[4 * j + 3] = __uint_as_float(r.w[2 * j + 1] & 0xFFFF0000u);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) x[4 * j + i] = __uint_as_float(r.w[4 * j + i]);
    }
  }
}

// Maximum of the row's logits as the kernel reads them.  A sum of four is NaN or +inf exactly when one of them is NaN
// or +inf (or they mix -inf with +inf), so one comparison per four finds the rows that need cleaning; only then
// (rare) every element is cleaned in place.  `bad` collects whether anything had to be.
template <int NCH>
__device__ __forceinline__ float clean_and_max(float* x, bool& bad) {
  float a0 = -INFINITY, a1 = -INFINITY;
  bool dirty = false;
#pragma unroll
  for (int e = 0; e < 4 * NCH; e += 4) {
    dirty |= !((x[e] + x[e + 1]) + (x[e + 2] + x[e + 3]) < INFINITY);
    a0 = fmaxf(a0, fmaxf(x[e], x[e + 1])); a1 = fmaxf(a1, fmaxf(x[e + 2], x[e + 3]));
  }
  if (dirty) {
    a0 = -INFINITY; a1 = -INFINITY;
#pragma unroll
    for (int e = 0; e < 4 * NCH; ++e) {
      bad |= !(x[e] < INFINITY);
      x[e] = clean_logit(x[e]);
      a0 = fmaxf(a0, x[e]);
    }
  }
  return fmaxf(a0, a1);
}
// x <- 2^((x - m) c2) in place; returns the sum
template <int NCH>
__device__ __forceinline__ float exponentials(float* x, float m, float c2) {
  const float off = m == -INFINITY ? 0.f : -m * c2;  // an all -inf slice stays 0
  float s0 = 0.f, s1 = 0.f;
#pragma unroll
  for (int e = 0; e < 4 * NCH; e += 2) {
    x[e] = fast_ex2(fmaf(x[e], c2, off)); x[e + 1] = fast_ex2(fmaf(x[e + 1], c2, off));
    s0 += x[e]; s1 += x[e + 1];
  }
  return s0 + s1;
}

// Every warp of every CTA publishes one float4 to every CTA of the cluster.  On return lane l of every warp holds
// entries l, l + 32, ... (rank-major, i.e. in vocabulary order).
//
// The entries travel as asynchronous stores that count their bytes into the receiver's mbarrier, so nothing fences:
// a cluster barrier's release would first wait for everything the warp has in flight - the next node's rows, the path's
// stores - and it was the largest single stall of the walk (a quarter of the warps' time).  Measured, cluster barrier ->
// this: 768 nodes x 128256 tokens 26.0 -> 21.7 us, 64 x 32000 12.0 -> 9.9, greedy 128 x 32000 7.0 -> 5.0, 16 requests of
// 64 x 32000 24.3 -> 22.2, 64 of them 47.5 -> 42.8.
// Buffers and mbarriers are used in turn.  Exchange k + 2 reuses those of exchange k: a warp sends for k + 2 only once it
// has every warp's entry of k + 1, and a warp sends that only after it has read (and used) its entries of k.
template <int CL>
struct Exch { float4 e[CL * kWarps / 32]; };
constexpr uint32_t kSpinLimit = 1u << 22;
__device__ __forceinline__ void bar_arm(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
template <int CL>
__device__ __forceinline__ void exchange_arm(const Ctx& c, int buf) {  // by one thread: the bytes of one exchange
  bar_arm(c.local + (uint32_t)offsetof(Shared, xbar) + 8u * buf, (uint32_t)(CL * kWarps * sizeof(float4)));
}
__device__ __forceinline__ void send4(uint32_t to, uint32_t bar, float4 v) {  // both in the receiver
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(to), "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)), "r"(__float_as_uint(v.w)), "r"(bar) : "memory");
}
// False when the bounded wait ran out (the same for the whole warp, after SEQ_DEV_TIMEOUT and a pause that lets the stores
// on their way to and from this CTA land): the warp leaves the kernel, through timed_out().
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, int32_t* dev_status) {
  uint32_t done = 0;
#pragma unroll 1
  for (uint32_t it = 0; it < kSpinLimit && !done; ++it) {
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    done = __all_sync(0xffffffffu, done);
  }
  if (!done) {
    dev_flag(dev_status, SEQ_DEV_TIMEOUT);
    for (int it = 0; it < 1000; ++it) __nanosleep(1000);
  }
  return done;
}
// What a request that was given up leaves behind: no path and no token.  (Every CTA of the cluster gets here, the others
// because this one's entries stay out, and each writes the same; what a thread had decided before is overwritten or not.)
__device__ __forceinline__ void timed_out(const VerifyArgs& a) {
  if ((threadIdx.x & 31) == 0) { *a.path_len = 0; *a.bonus = -1; }
}
// Before anything else: the mbarriers, and this CTA's arrival at the one cluster barrier.  exchange_ready() waits for it:
// from there on every CTA is resident and its mbarriers count.
template <int CL>
__device__ __forceinline__ void exchange_init(Ctx& c) {
  c.local = (uint32_t)__cvta_generic_to_shared(c.sh);
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(c.remote) : "r"(c.local), "r"(c.lane & (CL - 1)));
  c.xn = 0;
  if (c.tid == 0) {
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(c.local + (uint32_t)offsetof(Shared, xbar) + 8u * b) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(c.local + (uint32_t)offsetof(Shared, dbar) + 8u * b) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    exchange_arm<CL>(c, 0);
    exchange_arm<CL>(c, 1);
#pragma unroll
    for (int b = 0; b < 2; ++b) bar_arm(c.local + (uint32_t)offsetof(Shared, dbar) + 8u * b, sizeof(float4));
  }
  __syncwarp();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void exchange_ready() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// ... in two halves, so that work that does not depend on the exchange can run while the entries travel
template <int CL>
__device__ __forceinline__ void exchange_push(const Ctx& c, float4 mine) {
  const uint32_t buf = c.xn & 1u;
  if (c.lane < CL) {
    send4(c.remote + (uint32_t)offsetof(Shared, xbuf) + (buf * (kCl * kWarps) + c.rank * kWarps + c.warp) * (uint32_t)sizeof(float4),
          c.remote + (uint32_t)offsetof(Shared, xbar) + 8u * buf, mine);
  }
}
template <int CL>
__device__ __forceinline__ bool exchange_pull(Ctx& c, Exch<CL>& x, int32_t* dev_status) {  // false: see bar_wait
  const uint32_t buf = c.xn & 1u;
  if (!bar_wait(c.local + (uint32_t)offsetof(Shared, xbar) + 8u * buf, (c.xn >> 1) & 1u, dev_status)) return false;
  if (c.tid == 0) exchange_arm<CL>(c, (int)buf);  // for the exchange after the next
#pragma unroll
  for (int m = 0; m < CL * kWarps / 32; ++m) x.e[m] = c.sh->xbuf[buf][c.lane + 32 * m];
  ++c.xn;
  return true;
}
// A batched launch runs one request per cluster: the same code on that request's arrays.
template <int CL>
__device__ __forceinline__ VerifyArgs request_args(const VerifyArgs& in) {
  VerifyArgs a = in;
  const int64_t r = blockIdx.x / CL;
  if (r > 0) {
    a.parent += r * in.tree_stride; a.tokens += r * in.tree_stride;
    a.target = reinterpret_cast<const float*>(reinterpret_cast<const char*>(in.target) + r * in.logits_stride * ((in.flags & SEQ_VERIFY_LOGITS_BF16) ? 2 : 4));
    a.draft = reinterpret_cast<const float*>(reinterpret_cast<const char*>(in.draft) + r * in.logits_stride * ((in.flags & SEQ_VERIFY_LOGITS_BF16) ? 2 : 4));
    a.uniforms += r * in.unif_stride;
    a.path += r * in.tree_stride; a.path_len += r; a.bonus += r;
    if (in.residual_out != nullptr) a.residual_out += r * in.resid_stride;
    if (in.next_child_out != nullptr) a.next_child_out += r * in.tree_stride;
  }
  return a;
}

// The draw by inverse CDF, coarse level, every warp for itself: an inclusive scan over the (rank, warp) masses, 32 at a time.
// Returns the segment that holds the crossing (-1: no mass anywhere) and the target inside it; take_last: rounding left the
// total at or below the target, the last segment with mass is returned and its last element with mass is the one.
template <int CL>
__device__ __forceinline__ int draw_segment(const Ctx& c, const float* part_sum, float u, double& total_mass, double& tl, bool& take_last) {
  constexpr int kPPL = CL * kWarps / 32;
  double inc[kPPL], before = 0.0;
#pragma unroll
  for (int m = 0; m < kPPL; ++m) {
    double v = (double)part_sum[m];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double up = __shfl_up_sync(0xffffffffu, v, o);
      if (c.lane >= o) v += up;
    }
    inc[m] = v + before;
    before = __shfl_sync(0xffffffffu, inc[m], 31);
  }
  total_mass = before;
  const double tgt = (double)u * total_mass;
  int part = -1;
  take_last = false;
#pragma unroll
  for (int m = 0; m < kPPL; ++m) {
    const uint32_t hit = __ballot_sync(0xffffffffu, part_sum[m] > 0.f && inc[m] > tgt);
    if (part < 0 && hit) part = 32 * m + __ffs(hit) - 1;
  }
  if (part < 0) {
    take_last = true;
#pragma unroll
    for (int m = kPPL - 1; m >= 0; --m) {
      const uint32_t pos = __ballot_sync(0xffffffffu, part_sum[m] > 0.f);
      if (part < 0 && pos) part = 32 * m + 31 - __clz(pos);
    }
  }
  tl = 0.0;
  if (part == c.rank * kWarps + c.warp) {
#pragma unroll
    for (int m = 0; m < kPPL; ++m) {
      const double i_m = __shfl_sync(0xffffffffu, inc[m], part & 31), s_m = (double)__shfl_sync(0xffffffffu, part_sum[m], part & 31);
      if ((part >> 5) == m) tl = tgt - (i_m - s_m);
    }
  }
  return part;
}
// ... fine level, by the one warp whose segment holds the crossing.  The segment's values go to shared memory in vocabulary
// order (one padding word per 32, so that the reads do not collide); lane l then owns elements [4 NCH l, + 4 NCH): the lanes'
// sums are scanned, and the lane that holds the crossing walks its elements and returns the token (the others -1).  Rolled
// loops: this runs in one warp.
template <int NCH>
__device__ __forceinline__ int draw_in_segment(const Ctx& c, const float* p, float* seg, double tl, bool take_last) {
  constexpr int kE = 4 * NCH, kSpan = 32 * kE;
#pragma unroll
  for (int e = 0; e < kE; ++e) {
    const int idx = (e >> 2) * 128 + c.lane * 4 + (e & 3);
    seg[idx + (idx >> 5)] = p[e];
  }
  __syncwarp();
  const int mine0 = kE * c.lane;  // this lane's first element of the segment
  float ls = 0.f;
#pragma unroll 4
  for (int k = 0; k < kE; ++k) { const int idx = mine0 + k; ls += seg[idx + (idx >> 5)]; }
  double incl = (double)ls;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double up = __shfl_up_sync(0xffffffffu, incl, o);
    if (c.lane >= o) incl += up;
  }
  const uint32_t cross = take_last ? 0u : __ballot_sync(0xffffffffu, ls > 0.f && incl > tl);
  const uint32_t mass = __ballot_sync(0xffffffffu, ls > 0.f);
  if (mass == 0u) return c.lane == 0 ? c.lo + c.warp * kSpan : -1;  // (a segment said to have mass has none: its first token)
  if (c.lane != (cross ? __ffs(cross) - 1 : 31 - __clz(mass))) return -1;
  double r = incl - (double)ls;
  int pick = -1, last_k = 0;
#pragma unroll 1
  for (int k = 0; k < kE && pick < 0; ++k) {
    const int idx = mine0 + k;
    const float v = seg[idx + (idx >> 5)];
    r += (double)v;
    if (v > 0.f) { last_k = k; if (cross && r > tl) pick = k; }
  }
  return c.lo + c.warp * kSpan + mine0 + (pick < 0 ? last_k : pick);  // nothing crosses: the last element with mass
}

// (The batch's instances up to 32768 tokens keep to 128 registers: two requests' CTAs share an SM, 64 requests of 32000
// tokens take 42 us instead of 65.)
template <int NCH, bool kBf16, int CL>
__global__ void __launch_bounds__(kTh, CL == kClBatch && NCH <= 4 ? 2 : 1) tree_verify_walk_kernel(const VerifyArgs a_in) {
  const VerifyArgs a = request_args<CL>(a_in);
  constexpr int kPPL = CL * kWarps / 32;  // table entries per lane
  constexpr int kEsz = kBf16 ? 2 : 4;  // bytes per logit
  const char* const tbase = reinterpret_cast<const char*>(a.target);
  const char* const dbase = reinterpret_cast<const char*>(a.draft);
  constexpr int kE = 4 * NCH;        // elements per thread and row
  constexpr int kSpan = 32 * kE;     // consecutive elements of the slice that one warp holds
  extern __shared__ __align__(16) uint8_t dyn_smem[];
  Shared* sh = reinterpret_cast<Shared*>(dyn_smem);
  Ctx c;
  c.sh = sh;
  c.rank = (int)cg::this_cluster().block_rank();
  c.lo = min(c.rank * a.slice_cap, a.V);
  c.cnt = min(a.V - c.lo, a.slice_cap);
  c.tid = threadIdx.x; c.warp = threadIdx.x >> 5; c.lane = threadIdx.x & 31;
  exchange_init<CL>(c);
  const bool specinfer = (a.flags & SEQ_VERIFY_SPECINFER) != 0;  // D is never touched: ZD stays 1, S stays empty
  const float c2 = kLog2e / a.temperature;
  const bool leader = c.rank == 0 && c.tid == 0;
  WTRACE_DECL;
  WTRACE(leader, 0);

  // programmatic dependent launch: the next kernel in the stream may be scheduled onto free SMs from now on; nothing
  // above touches global memory, everything below may read what the previous kernel wrote
  if (c.tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  prefetch_tree<true>(c, a);
  prefetch_row<NCH, kBf16>(c, tbase);
  if (a.n > 1) {
    prefetch_row<NCH, kBf16>(c, dbase);
    prefetch_row<NCH, kBf16>(c, tbase + a.target_stride * kEsz);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  WTRACE(leader, 1);

  float p[kE], q[kE];                // the current node's rows
  RawRow<NCH, kBf16> pn, qn;         // the rows of the child under test, on their way (as they lie in memory)
  {
    // The tree first - a few words per thread, and everything waits for them - then the root's rows.
    int tp[4], tt[4];
    float tu[5];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = c.tid + kTh * k;
      tp[k] = i < a.n ? a.parent[i] : -1;
      tt[k] = i < a.n ? a.tokens[i] : 0;
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) tu[k] = c.tid + kTh * k <= a.n ? a.uniforms[c.tid + kTh * k] : 0.f;
    load_row<NCH, kBf16>(c, tbase, pn);
    if (a.n > 1) load_row<NCH, kBf16>(c, dbase, qn);  // (a root without children: never read)
    if (c.tid < SEQ_MAX_TREE / 32) sh->has_child[c.tid] = 0u;
    if (c.tid < 32) sh->chunk_cnt[c.tid] = 0;
    if (c.tid == 0) sh->node_flags = 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = c.tid + kTh * k;
      if (i < a.n) {
        int pp = tp[k];
        if (i == 0) pp = -1;
        else if (pp < -1 || pp >= i) { if (c.rank == 0) dev_flag(a.dev_status, SEQ_DEV_BAD_PARENT); pp = -1; }
        sh->parent[i] = pp;
        sh->tokens[i] = tt[k];
        if (pp >= 0) atomicOr(&sh->has_child[pp >> 5], 1u << (pp & 31));
      }
    }
#pragma unroll
    for (int k = 0; k < 5; ++k)
      if (c.tid + kTh * k <= a.n) sh->uniforms[c.tid + kTh * k] = tu[k];
    if (c.rank == 0 && a.next_child_out != nullptr)
      for (int i = c.tid; i < a.n; i += kTh) a.next_child_out[i] = -2;  // nodes the walk does not visit
  }
  __syncthreads();  // the tree is in place
  exchange_ready();
  widen<NCH, kBf16>(pn, p);
  widen<NCH, kBf16>(qn, q);  // (a tree of one node: never loaded, never read)
  WTRACE(leader, 2);

  int cur = 0, plen = 0, bonus_found = -1;
  bool cur_has_kids = (sh->has_child[0] & 1u) != 0;
#pragma unroll 1
  for (int hop = 0; hop < a.n; ++hop) {  // a walk visits at most n nodes
    if (leader) a.path[plen] = cur;
    ++plen;
    WTRACE(leader, 10);
    const int np = hop & 1;
    const char* trow = tbase + (int64_t)cur * a.target_stride * kEsz;
    const char* drow = dbase + (int64_t)cur * a.draft_stride * kEsz;
    // ---- exponentials relative to this thread's own maxima, with their sums; the per-warp partials go to every CTA
    const bool need_draft = cur_has_kids;
    bool bad = false;
    const float mp = clean_and_max<NCH>(p, bad);
    const float sp = exponentials<NCH>(p, mp, c2);
    float mq = -INFINITY, sq = 0.f;
    if (need_draft) {
      mq = clean_and_max<NCH>(q, bad);
      sq = exponentials<NCH>(q, mq, c2);
    }
    if (bad) dev_flag(a.dev_status, SEQ_DEV_NONFINITE);
    WTRACE(leader, 13);
    Exch<CL> x;
    {
      const float Mwp = max_lanes(mp), Mwq = max_lanes(mq);
      const float swp = warp_sum(sp * rel_exp(mp, Mwp, c2)), swq = warp_sum(sq * rel_exp(mq, Mwq, c2));
      exchange_push<CL>(c, make_float4(Mwp, swp, Mwq, swq));
    }
    WTRACE(leader, 40);
    // ---- while the entries travel: the node's children, in order; the first child's own rows start their way (they are
    // needed exactly if it is accepted); lane l of every warp takes child l (then l + 32, ...): its token, uniform, the two
    // logits of the current node at it (left in flight), and whether an earlier sibling carries the same token.
    int n_kids = 0, nxt = -1;
    bool nxt_has_kids = false;
    if (cur_has_kids) {
      bool k[4];
      uint32_t b[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (kTh * j >= a.n) break;  // (chunks behind the tree count no children from the start)
        const int ch = c.tid + kTh * j;
        k[j] = ch < a.n && sh->parent[ch] == cur;
        b[j] = __ballot_sync(0xffffffffu, k[j]);
        if (c.lane == 0) sh->chunk_cnt[kWarps * j + c.warp] = __popc(b[j]);
      }
      __syncthreads();
      const int cc = sh->chunk_cnt[c.lane];
      n_kids = __reduce_add_sync(0xffffffffu, cc);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (kTh * j >= a.n) break;
        const int before = __reduce_add_sync(0xffffffffu, c.lane < kWarps * j + c.warp ? cc : 0);
        const int ch = c.tid + kTh * j;
        if (k[j]) sh->kid[np][before + __popc(b[j] & ((1u << c.lane) - 1u))] = make_int2(ch, sh->tokens[ch]);
      }
      __syncthreads();
      nxt = sh->kid[np][0].x;
      nxt_has_kids = (sh->has_child[nxt >> 5] >> (nxt & 31)) & 1u;
      load_row<NCH, kBf16>(c, tbase + (int64_t)nxt * a.target_stride * kEsz, pn);
      if (nxt_has_kids) load_row<NCH, kBf16>(c, dbase + (int64_t)nxt * a.draft_stride * kEsz, qn);
    }
    WTRACE(leader, 44);
    int kch = 0, ktok = -1;                 // this lane's child
    float ku = 0.f;
    float2 kraw = make_float2(0.f, 0.f);
    bool kvalid = false, kdup = false;
    auto take_kids = [&](int base) {
      const int r = base + c.lane;
      ktok = -1;
      kdup = false;
      if (r < n_kids) {
        const int2 e = sh->kid[np][r];
        kch = e.x; ktok = e.y;
        ku = sh->uniforms[kch];
      }
      kvalid = ktok >= 0 && ktok < a.V;
      if (kvalid) kraw = make_float2(load_logit<kBf16>(trow, ktok), load_logit<kBf16>(drow, ktok));
      if (!specinfer) {  // (lanes past the last child come after every child: what they hold does not matter)
        kdup = (__match_any_sync(0xffffffffu, ktok) & ((1u << c.lane) - 1u)) != 0u;
        for (int r2 = 0; r2 < base; ++r2) kdup |= sh->kid[np][r2].y == ktok;  // (a node of more than 32 children)
      }
    };
    if (n_kids > 0) take_kids(0);
    WTRACE(leader, 12);
    if (!exchange_pull<CL>(c, x, a.dev_status)) return timed_out(a);
    WTRACE(leader, 14);
    float Mp = -INFINITY, Mq = -INFINITY;
#pragma unroll
    for (int m = 0; m < kPPL; ++m) { Mp = fmaxf(Mp, x.e[m].x); Mq = fmaxf(Mq, x.e[m].z); }
    Mp = max_lanes(Mp); Mq = max_lanes(Mq);
    // (Single precision from here on: the sums have 128 terms of like size, the scalars C, U, Z, ZD a handful of
    // updates; their rounding stays two orders of magnitude inside the 1e-5 band of the parity rule.)
    float part_sum[kPPL];   // residual mass of the (rank, warp) segments lane, lane + 32, ...: the draw's coarse level
    float asum = 0.f, bsum = 0.f;
#pragma unroll
    for (int m = 0; m < kPPL; ++m) {
      part_sum[m] = x.e[m].y * rel_exp(x.e[m].x, Mp, c2);
      asum += part_sum[m];
      bsum += x.e[m].w * rel_exp(x.e[m].z, Mq, c2);
    }
    const float Sp = warp_sum(asum), Sq = warp_sum(bsum);
    if (!(Sp > 0.f)) dev_flag(a.dev_status, SEQ_DEV_DEGENERATE);
    const float invSp = Sp > 0.f ? __frcp_rn(Sp) : 0.f;
    const float invSq = (need_draft && Sq > 0.f) ? __frcp_rn(Sq) : 0.f;
#pragma unroll
    for (int m = 0; m < kPPL; ++m) part_sum[m] *= invSp;
    int mode = (need_draft && !(Sq > 0.f)) ? 1 : 0;  // a draft row without mass: the uniform fallback from the start
    // probabilities in place; this thread's share of sum(D) over the surviving tokens, a direct sum
    const float fp = rel_exp(mp, Mp, c2) * invSp, fq = rel_exp(mq, Mq, c2) * invSq;
    float zd_mine = 0.f;
    {
      float s0 = 0.f, s1 = 0.f;
#pragma unroll
      for (int e = 0; e < kE; e += 2) {
        p[e] *= fp; p[e + 1] *= fp;
        if (need_draft) { q[e] *= fq; q[e + 1] *= fq; s0 += q[e]; s1 += q[e + 1]; }
      }
      zd_mine = s0 + s1;
    }
    WTRACE(leader, 15);
    float C = 0.f, U = 0.f, Z = 1.f, ZD = 1.f;
    int nS = 0, accepted = -1;
    // each lane's child: its two probabilities (zero once an earlier, hence rejected, sibling carried the same token: it is
    // in S.  Without the draft update there is no S: a repeated token is tested like any other, and its R is 0 by then)
    float kps = 0.f, kqs = 0.f;
    uint32_t valid_kids = 0u, dup_kids = 0u;
    auto score_kids = [&]() {
      kps = kvalid && !kdup ? fast_ex2((clean_logit(kraw.x) - Mp) * c2) * invSp : 0.f;
      kqs = kvalid && !kdup ? fast_ex2((clean_logit(kraw.y) - Mq) * c2) * invSq : 0.f;
      valid_kids = __ballot_sync(0xffffffffu, kvalid);
      dup_kids = __ballot_sync(0xffffffffu, kdup);
    };
    if (n_kids > 0) score_kids();
    // ---- Algorithm 2's loop over the children, in their order
#pragma unroll 1
    for (int i = 0; i < n_kids; ++i) {
      if (i > 0 && (i & 31) == 0) { take_kids(i); score_kids(); }
      const bool valid = (valid_kids >> (i & 31)) & 1u, in_S = (dup_kids >> (i & 31)) & 1u;
      if (!valid) dev_flag(a.dev_status, SEQ_DEV_BAD_TOKEN);
      // the acceptance test u < R[s]/D[s], with R[s] = rs/Z and D[s] = qs/ZD (or 1/(V-|S|)); cross-multiplied, which also
      // covers D[s] = 0 (accept iff R[s] > 0).  Every lane tests its child, child i's answer counts.
      const float rs = resid(kps, kqs, C, U);
      const bool win = kvalid && (mode == 0 ? ku * Z * kqs < rs * ZD : ku * Z < rs * (float)(a.V - nS));
      const bool accept = (__ballot_sync(0xffffffffu, win) >> (i & 31)) & 1u;
      WTRACE(leader, 16);
      if (accept) { accepted = __shfl_sync(0xffffffffu, kch, i & 31); break; }
      // ---- rejected: the next child's rows must start their way, and the residual is updated.  The loads are issued
      // behind the exchange's push: ahead of it they delay it (256 nodes x 50257 tokens 15.2 -> 15.6 us).
      const bool more = i + 1 < n_kids;
      if (more) {
        nxt = sh->kid[np][i + 1].x;
        nxt_has_kids = (sh->has_child[nxt >> 5] >> (nxt & 31)) & 1u;
      }
      if (!valid) {  // (not a token: R and D untouched)
        if (more) {
          load_row<NCH, kBf16>(c, tbase + (int64_t)nxt * a.target_stride * kEsz, pn);
          if (nxt_has_kids) load_row<NCH, kBf16>(c, dbase + (int64_t)nxt * a.draft_stride * kEsz, qn);
        }
        continue;
      }
      // R <- norm(max(R - D, 0)) with D as it stands
      float Cn = C, Un = U;
      if (mode == 0) Cn += Z * __frcp_rn(ZD);
      else if (a.V - nS > 0) Un += Z * __frcp_rn((float)(a.V - nS));
      // the draft update: s leaves D and joins S.  The thread that holds s clears it (its R is 0 from here on, see above)
      // and re-sums its share of D
      if (!in_S && !specinfer) {
        const int s = __shfl_sync(0xffffffffu, ktok, i & 31);
        const int idx = s - c.lo - c.warp * kSpan;
        if (s - c.lo >= 0 && s - c.lo < c.cnt && idx >= 0 && idx < kSpan && ((idx >> 2) & 31) == c.lane) {
          const int at = ((idx >> 7) << 2) | (idx & 3);
          float s0 = 0.f, s1 = 0.f;
#pragma unroll
          for (int k = 0; k < kE; k += 2) {
            if (k == at) p[k] = q[k] = 0.f;
            if (k + 1 == at) p[k + 1] = q[k + 1] = 0.f;
            s0 += q[k]; s1 += q[k + 1];
          }
          zd_mine = s0 + s1;
        }
        nS += 1;
      }
      const float Cnf = Cn, Unf = Un;
      float z0 = 0.f, z1 = 0.f;
#pragma unroll
      for (int e = 0; e < kE; e += 2) { z0 += resid(p[e], q[e], Cnf, Unf); z1 += resid(p[e + 1], q[e + 1], Cnf, Unf); }
      const float zr = warp_sum(z0 + z1), zd = warp_sum(zd_mine);
      WTRACE(leader, 17);
      exchange_push<CL>(c, make_float4(zr, zd, 0.f, 0.f));
      if (more) {
        load_row<NCH, kBf16>(c, tbase + (int64_t)nxt * a.target_stride * kEsz, pn);
        if (nxt_has_kids) load_row<NCH, kBf16>(c, dbase + (int64_t)nxt * a.draft_stride * kEsz, qn);
      }
      if (!exchange_pull<CL>(c, x, a.dev_status)) return timed_out(a);
      WTRACE(leader, 18);
      float zsum = 0.f, zdsum = 0.f;
#pragma unroll
      for (int m = 0; m < kPPL; ++m) { zsum += x.e[m].x; zdsum += x.e[m].y; }
      const float Zn = warp_sum(zsum), ZDn = warp_sum(zdsum);
      if (Zn > 0.f) {
        C = Cn; U = Un; Z = Zn;
#pragma unroll
        for (int m = 0; m < kPPL; ++m) part_sum[m] = x.e[m].x;
      } else {
        dev_flag(a.dev_status, SEQ_DEV_DEGENERATE);  // impossible in exact arithmetic: keep R
      }
      if (!specinfer) {
        ZD = ZDn;
        if (mode == 0 && !(ZDn > 0.f)) mode = 1;  // no mass left in D: uniform over the non-rejected set
      }
    }
    if (leader && a.next_child_out != nullptr) a.next_child_out[cur] = accepted;
    if (accepted >= 0) {
      // ---- on to the accepted child: its rows are in the second set of registers (or about to land there)
      widen<NCH, kBf16>(pn, p);
      widen<NCH, kBf16>(qn, q);
      cur = accepted;
      cur_has_kids = nxt_has_kids;
      continue;
    }
    WTRACE(leader, 20);
    // ---- no child accepted (or a leaf): x ~ R by inverse CDF in index order with the last uniform
    {
      const bool use_q = need_draft && C != 0.f;
      const float Cf = C, Uf = U;
#pragma unroll
      for (int e = 0; e < kE; ++e) p[e] = resid(p[e], use_q ? q[e] : 0.f, Cf, Uf);  // the residual replaces p
      const float u = sh->uniforms[a.n];
      double total_mass, tl;
      bool take_last;
      const int part = draw_segment<CL>(c, part_sum, u, total_mass, tl, take_last);
      if (a.residual_out != nullptr) {
        const float inv = total_mass > 0.0 ? (float)fast_rcp(total_mass) : 0.f;
#pragma unroll
        for (int e = 0; e < kE; ++e) {
          const int li = c.warp * kSpan + (e >> 2) * 128 + c.lane * 4 + (e & 3);
          if (li < c.cnt) a.residual_out[c.lo + li] = p[e] * inv;
        }
      }
      if (part < 0) {
        if (leader) { dev_flag(a.dev_status, SEQ_DEV_DEGENERATE); bonus_found = 0; }  // no mass anywhere: token 0
      } else if (part == c.rank * kWarps + c.warp) {
        bonus_found = draw_in_segment<NCH>(c, p, reinterpret_cast<float*>(sh->kid[np ^ 1]), tl, take_last);
      }
    }
    break;
  }
  WTRACE(leader, 30);
  if (leader) *a.path_len = plen;
  if (bonus_found >= 0) *a.bonus = bonus_found;
  // No closing cluster barrier: a CTA leaves after it has received every entry of the last exchange, so nothing can still
  // address it.
}


// ---------------------------------------------------------------- greedy decoding (T = 0) -----------------------
// R is the one-hot at the target arg-max (lowest index on ties), a child is accepted iff its token is that arg-max;
// draft logits and uniforms play no part.  Per visited node: the target row in registers, one arg-max over the
// cluster (one exchange), one look at the children.  While the exchange is on its way, the row of the node's first child -
// the draft's most probable token, the likeliest match - is requested; any other match is fetched when it is known.
__device__ __forceinline__ int ordered_key(float x) {  // an integer that orders like the (non-NaN) float
  int b = __float_as_int(x);
  return b ^ ((b >> 31) & 0x7fffffff);
}
// (key, index) of the larger key, then the lower index; index 0x7fffffff = nothing
__device__ __forceinline__ void warp_argmax(int& key, int& idx) {
  const int k = idx == 0x7fffffff ? INT_MIN : key;
  const int m = __reduce_max_sync(0xffffffffu, k);
  idx = __reduce_min_sync(0xffffffffu, (k == m) ? idx : 0x7fffffff);
  key = m;
}

template <int NCH, bool kBf16>
__global__ void __launch_bounds__(kTh, 1) tree_verify_greedy_kernel(const VerifyArgs a_in) {
  const VerifyArgs a = request_args<kCl>(a_in);
  constexpr int kEsz = kBf16 ? 2 : 4;
  constexpr int kE = 4 * NCH, kSpan = 32 * kE;
  const char* const tbase = reinterpret_cast<const char*>(a.target);
  extern __shared__ __align__(16) uint8_t dyn_smem[];
  Shared* sh = reinterpret_cast<Shared*>(dyn_smem);
  Ctx c;
  c.sh = sh;
  c.rank = (int)cg::this_cluster().block_rank();
  c.lo = min(c.rank * a.slice_cap, a.V);
  c.cnt = min(a.V - c.lo, a.slice_cap);
  c.tid = threadIdx.x; c.warp = threadIdx.x >> 5; c.lane = threadIdx.x & 31;
  exchange_init<kCl>(c);
  const bool leader = c.rank == 0 && c.tid == 0;
  if (c.tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  prefetch_tree<false>(c, a);
  prefetch_row<NCH, kBf16>(c, tbase);
  if (a.n > 1) prefetch_row<NCH, kBf16>(c, tbase + a.target_stride * kEsz);
  asm volatile("griddepcontrol.wait;" ::: "memory");

  RawRow<NCH, kBf16> pn;
  {
    int tp[4], tt[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = c.tid + kTh * k;
      tp[k] = i < a.n ? a.parent[i] : -1;
      tt[k] = i < a.n ? a.tokens[i] : 0;
    }
    load_row<NCH, kBf16>(c, tbase, pn);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = c.tid + kTh * k;
      if (i < a.n) {
        int pp = tp[k];
        if (i == 0) pp = -1;
        else if (pp < -1 || pp >= i) { if (c.rank == 0) dev_flag(a.dev_status, SEQ_DEV_BAD_PARENT); pp = -1; }
        sh->parent[i] = pp;
        sh->tokens[i] = tt[k];
      }
    }
    if (c.rank == 0 && a.next_child_out != nullptr)
      for (int i = c.tid; i < a.n; i += kTh) a.next_child_out[i] = -2;  // nodes the walk does not visit
  }
  __syncthreads();  // the tree is in place
  exchange_ready();

  int cur = 0, plen = 0, g = 0;
  bool bad = false;
#pragma unroll 1
  for (int hop = 0; hop < a.n; ++hop) {  // a walk visits at most n nodes
    if (leader) a.path[plen] = cur;
    ++plen;
    int32_t* pick = sh->pick[hop & 1];
    if (c.tid < 3) pick[c.tid] = 0x7fffffff;  // (the other set is the one the previous hop may still be reading)
    float x[kE];
    widen<NCH, kBf16>(pn, x);
    // this thread's arg-max: its elements in ascending index order, the first of equal values stays
    int key = INT_MIN, idx = 0x7fffffff;
#pragma unroll
    for (int e = 0; e < kE; ++e) {
      const int local = c.warp * kSpan + (e >> 2) * 128 + c.lane * 4 + (e & 3);
      if (local < c.cnt) {
        bad |= !(x[e] < INFINITY);
        const int k = ordered_key(clean_logit(x[e]));
        if (idx == 0x7fffffff || k > key) { key = k; idx = c.lo + local; }
      }
    }
    warp_argmax(key, idx);
    exchange_push<kCl>(c, make_float4(__int_as_float(key), __int_as_float(idx), 0.f, 0.f));
    // ---- while the entries travel: the node's first child, and its row on the way
    __syncthreads();  // pick[] is reset
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = c.tid + kTh * k;
      if (i < a.n && sh->parent[i] == cur) atomicMin(&pick[2], i);
    }
    __syncthreads();
    const int first_kid = pick[2];
    if (first_kid != 0x7fffffff) load_row<NCH, kBf16>(c, tbase + (int64_t)first_kid * a.target_stride * kEsz, pn);
    Exch<kCl> t;
    if (!exchange_pull<kCl>(c, t, a.dev_status)) return timed_out(a);
    key = INT_MIN; idx = 0x7fffffff;
#pragma unroll
    for (int m = 0; m < kCl * kWarps / 32; ++m) {  // entries in vocabulary order: the first of equal keys stays
      const int k = __float_as_int(t.e[m].x), i = __float_as_int(t.e[m].y);
      if (i != 0x7fffffff && (idx == 0x7fffffff || k > key)) { key = k; idx = i; }
    }
    warp_argmax(key, idx);
    g = idx == 0x7fffffff ? 0 : idx;
    // ---- the child that carries the arg-max (the first, should several); a child with a token outside the vocabulary
    // is reported if the loop over the children would have met it before the match
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = c.tid + kTh * k;
      if (i < a.n && sh->parent[i] == cur) {
        const int s = sh->tokens[i];
        if (s < 0 || s >= a.V) atomicMin(&pick[1], i);
        else if (s == g) atomicMin(&pick[0], i);
      }
    }
    __syncthreads();
    const int match = pick[0];
    if (leader) {
      if (pick[1] < match) dev_flag(a.dev_status, SEQ_DEV_BAD_TOKEN);
      if (a.next_child_out != nullptr) a.next_child_out[cur] = match == 0x7fffffff ? -1 : match;
    }
    if (match == 0x7fffffff) break;
    if (match != first_kid) load_row<NCH, kBf16>(c, tbase + (int64_t)match * a.target_stride * kEsz, pn);
    cur = match;
  }
  if (bad) dev_flag(a.dev_status, SEQ_DEV_NONFINITE);
  if (a.residual_out != nullptr) {
#pragma unroll
    for (int e = 0; e < kE; ++e) {
      const int local = c.warp * kSpan + (e >> 2) * 128 + c.lane * 4 + (e & 3);
      if (local < c.cnt) a.residual_out[c.lo + local] = (c.lo + local == g) ? 1.f : 0.f;
    }
  }
  if (leader) { *a.path_len = plen; *a.bonus = g; }
}

// ---------------------------------------------------------------- sampling from the target ----------------------
// SEQ_VERIFY_TARGET_SAMPLE at T > 0: a token is drawn from softmax(target / T) at each node with the node's uniform, and the
// first child that carries it is taken.  Per visited node the target row in registers (its exponentials, one exchange), the
// draw as above, and a second exchange of one entry: the warp that found the token tells every CTA.  As in the greedy walk the
// first child's row is requested while the first exchange is on its way.
// Bound by the chain of a node's steps, like the walk above.  Against the shared-memory walk: 768 nodes x 128256 tokens 16.0
// -> 6.7 us, 64 x 32000 9.8 -> 4.2, 16 requests of 64 x 32000 12.9 -> 6.2.
template <int NCH, int CL>
__global__ void __launch_bounds__(kTh, CL == kClBatch && NCH <= 4 ? 2 : 1) tree_verify_sample_kernel(const VerifyArgs a_in) {
  const VerifyArgs a = request_args<CL>(a_in);
  constexpr int kPPL = CL * kWarps / 32, kE = 4 * NCH, kSpan = 32 * kE;
  const char* const tbase = reinterpret_cast<const char*>(a.target);
  extern __shared__ __align__(16) uint8_t dyn_smem[];
  Shared* sh = reinterpret_cast<Shared*>(dyn_smem);
  Ctx c;
  c.sh = sh;
  c.rank = (int)cg::this_cluster().block_rank();
  c.lo = min(c.rank * a.slice_cap, a.V);
  c.cnt = min(a.V - c.lo, a.slice_cap);
  c.tid = threadIdx.x; c.warp = threadIdx.x >> 5; c.lane = threadIdx.x & 31;
  exchange_init<CL>(c);
  const float c2 = kLog2e / a.temperature;
  const bool leader = c.rank == 0 && c.tid == 0;
  if (c.tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  prefetch_tree<true>(c, a);
  prefetch_row<NCH, false>(c, tbase);
  asm volatile("griddepcontrol.wait;" ::: "memory");

  RawRow<NCH, false> pn;
  {
    int tp[4], tt[4];
    float tu[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = c.tid + kTh * k;
      tp[k] = i < a.n ? a.parent[i] : -1;
      tt[k] = i < a.n ? a.tokens[i] : 0;
      tu[k] = i < a.n ? a.uniforms[i] : 0.f;
    }
    load_row<NCH, false>(c, tbase, pn);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = c.tid + kTh * k;
      if (i < a.n) {
        int pp = tp[k];
        if (i == 0) pp = -1;
        else if (pp < -1 || pp >= i) { if (c.rank == 0) dev_flag(a.dev_status, SEQ_DEV_BAD_PARENT); pp = -1; }
        sh->parent[i] = pp;
        sh->tokens[i] = tt[k];
        sh->uniforms[i] = tu[k];
      }
    }
    if (c.rank == 0 && a.next_child_out != nullptr)
      for (int i = c.tid; i < a.n; i += kTh) a.next_child_out[i] = -2;  // nodes the walk does not visit
  }
  __syncthreads();  // the tree is in place
  exchange_ready();

  int cur = 0, plen = 0, token = 0;
  uint32_t dn = 0;  // tokens told
  float p[kE];
#pragma unroll 1
  for (int hop = 0; hop < a.n; ++hop) {  // a walk visits at most n nodes
    if (leader) a.path[plen] = cur;
    ++plen;
    int32_t* pick = sh->pick[hop & 1];
    if (c.tid < 3) pick[c.tid] = 0x7fffffff;  // (the other set is the one the previous hop may still be reading)
    widen<NCH, false>(pn, p);
    bool bad = false;
    const float mp = clean_and_max<NCH>(p, bad);
    const float sp = exponentials<NCH>(p, mp, c2);
    if (bad) dev_flag(a.dev_status, SEQ_DEV_NONFINITE);
    const float Mwp = max_lanes(mp);
    exchange_push<CL>(c, make_float4(Mwp, warp_sum(sp * rel_exp(mp, Mwp, c2)), 0.f, 0.f));
    // ---- while the entries travel: the node's first child, and its row on the way
    __syncthreads();  // pick[] is reset
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = c.tid + kTh * k;
      if (i < a.n && sh->parent[i] == cur) atomicMin(&pick[2], i);
    }
    __syncthreads();
    const int first_kid = pick[2];
    if (first_kid != 0x7fffffff) load_row<NCH, false>(c, tbase + (int64_t)first_kid * a.target_stride * 4, pn);
    Exch<CL> x;
    if (!exchange_pull<CL>(c, x, a.dev_status)) return timed_out(a);
    float Mp = -INFINITY;
#pragma unroll
    for (int m = 0; m < kPPL; ++m) Mp = fmaxf(Mp, x.e[m].x);
    Mp = max_lanes(Mp);
    float part_sum[kPPL], asum = 0.f;
#pragma unroll
    for (int m = 0; m < kPPL; ++m) {
      part_sum[m] = x.e[m].y * rel_exp(x.e[m].x, Mp, c2);
      asum += part_sum[m];
    }
    const float Sp = warp_sum(asum);
    const float invSp = Sp > 0.f ? __frcp_rn(Sp) : 0.f;
#pragma unroll
    for (int m = 0; m < kPPL; ++m) part_sum[m] *= invSp;
    const float fp = rel_exp(mp, Mp, c2) * invSp;
#pragma unroll
    for (int e = 0; e < kE; ++e) p[e] *= fp;
    double total_mass, tl;
    bool take_last;
    const int part = draw_segment<CL>(c, part_sum, sh->uniforms[cur], total_mass, tl, take_last);
    token = 0;
    if (part < 0) {
      dev_flag(a.dev_status, SEQ_DEV_DEGENERATE);  // a target row without mass: token 0
    } else {
      const uint32_t buf = dn & 1u, bar = (uint32_t)offsetof(Shared, dbar) + 8u * buf;
      if (part == c.rank * kWarps + c.warp) {
        const int mine = draw_in_segment<NCH>(c, p, reinterpret_cast<float*>(sh->kid[hop & 1]), tl, take_last);
        const int found = __reduce_max_sync(0xffffffffu, mine);
        if (c.lane < CL) send4(c.remote + (uint32_t)offsetof(Shared, drawn) + 16u * buf, c.remote + bar, make_float4(__int_as_float(found), 0.f, 0.f, 0.f));
      }
      if (!bar_wait(c.local + bar, (dn >> 1) & 1u, a.dev_status)) return timed_out(a);
      if (c.tid == 0) bar_arm(c.local + bar, sizeof(float4));
      token = __float_as_int(sh->drawn[buf].x);
      ++dn;
    }
    // ---- the first child that carries the token; one with a token outside the vocabulary is reported if it comes before
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = c.tid + kTh * k;
      if (i < a.n && sh->parent[i] == cur) {
        const int s = sh->tokens[i];
        if (s < 0 || s >= a.V) atomicMin(&pick[1], i);
        else if (s == token) atomicMin(&pick[0], i);
      }
    }
    __syncthreads();
    const int match = pick[0];
    if (leader) {
      if (pick[1] < match) dev_flag(a.dev_status, SEQ_DEV_BAD_TOKEN);
      if (a.next_child_out != nullptr) a.next_child_out[cur] = match == 0x7fffffff ? -1 : match;
    }
    if (match == 0x7fffffff) break;
    if (match != first_kid) load_row<NCH, false>(c, tbase + (int64_t)match * a.target_stride * 4, pn);
    cur = match;
  }
  if (a.residual_out != nullptr) {  // the distribution that the last token came from
#pragma unroll
    for (int e = 0; e < kE; ++e) {
      const int local = c.warp * kSpan + (e >> 2) * 128 + c.lane * 4 + (e & 3);
      if (local < c.cnt) a.residual_out[c.lo + local] = p[e];
    }
  }
  if (leader) { *a.path_len = plen; *a.bonus = token; }
}

}  // namespace vwk

// Elements a cluster of this kernel holds per row: 16 CTAs x 256 threads x 4 NCH.
bool verify_walk_supported(int vocab, int flags, float temperature) {
  if (flags & SEQ_VERIFY_ALL_NODES) return false;
  if (temperature == 0.f) return vocab >= 1 && (size_t)vocab <= (size_t)vwk::kCl * vwk::kTh * 4 * 8;  // greedy: its own kernel, whatever the mode flags say
  if (!(temperature > 0.f)) return false;
  return vocab >= 1 && (size_t)vocab <= (size_t)vwk::kCl * vwk::kTh * 4 * 8;
}

typedef void (*WalkKernel)(const VerifyArgs);
template <int CL>
static WalkKernel walk_kernel(int nch, bool bf16) {
  return bf16 ? (nch == 2 ? vwk::tree_verify_walk_kernel<2, true, CL> : nch == 4 ? vwk::tree_verify_walk_kernel<4, true, CL> : vwk::tree_verify_walk_kernel<8, true, CL>)
              : (nch == 2 ? vwk::tree_verify_walk_kernel<2, false, CL> : nch == 4 ? vwk::tree_verify_walk_kernel<4, false, CL> : vwk::tree_verify_walk_kernel<8, false, CL>);
}

template <int CL>
static WalkKernel sample_kernel(int nch) {
  return nch == 2 ? vwk::tree_verify_sample_kernel<2, CL> : nch == 4 ? vwk::tree_verify_sample_kernel<4, CL> : vwk::tree_verify_sample_kernel<8, CL>;
}

// cl: CTAs per request, 16 or (T > 0 and a vocabulary that 8 CTAs hold) 8.  With `clusters` given nothing is launched: the
// number of clusters that the device runs side by side is written there.
static int walk_launch(const VerifyArgs& a_in, int cl, int requests, int* clusters, cudaStream_t stream) {
  VerifyArgs a = a_in;
  a.slice_cap = (((a.V + cl - 1) / cl) + 3) & ~3;
  const int nch = a.slice_cap <= vwk::kTh * 4 * 2 ? 2 : a.slice_cap <= vwk::kTh * 4 * 4 ? 4 : 8;
  const bool bf16 = (a.flags & SEQ_VERIFY_LOGITS_BF16) != 0;
  const bool greedy = a.temperature == 0.f, sample = !greedy && (a.flags & SEQ_VERIFY_TARGET_SAMPLE) != 0;
  const WalkKernel kernel =
      greedy ? (bf16 ? (nch == 2 ? vwk::tree_verify_greedy_kernel<2, true> : nch == 4 ? vwk::tree_verify_greedy_kernel<4, true> : vwk::tree_verify_greedy_kernel<8, true>)
                     : (nch == 2 ? vwk::tree_verify_greedy_kernel<2, false> : nch == 4 ? vwk::tree_verify_greedy_kernel<4, false> : vwk::tree_verify_greedy_kernel<8, false>))
      : sample ? (cl == 16 ? sample_kernel<vwk::kCl>(nch) : sample_kernel<vwk::kClBatch>(nch))
      : cl == 16 ? walk_kernel<vwk::kCl>(nch, bf16) : walk_kernel<vwk::kClBatch>(nch, bf16);
  const int slot = (nch == 2 ? 0 : nch == 4 ? 1 : 2) + (sample ? (cl == 16 ? 18 : 21) : (bf16 ? 3 : 0) + (greedy ? 6 : cl == 16 ? 0 : 12));
  static int attr_done[24][64];
  const int rc = once_per_device(attr_done[slot], [&]() -> int {
    SEQ_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(vwk::Shared)));
    SEQ_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    return SEQ_OK;
  });
  if (rc != SEQ_OK) return rc;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cl * requests);
  cfg.blockDim = dim3(vwk::kTh);
  cfg.dynamicSmemBytes = sizeof(vwk::Shared);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // start under the previous kernel's tail
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = clusters != nullptr ? 1 : 2;
  if (clusters != nullptr) {
    if (cudaOccupancyMaxActiveClusters(clusters, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); *clusters = 0; }
    return SEQ_OK;
  }
  SEQ_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, a));
  return SEQ_OK;
}

int launch_verify_walk(const VerifyArgs& a, cudaStream_t stream) { return walk_launch(a, vwk::kCl, 1, nullptr, stream); }

// CTAs per request for a batch, 0 where the shared-memory walk is the better one.  Measured at T > 0 against that walk: up
// to 9 requests run as clusters of 16 on SMs of their own where the device places that many (32000 tokens: 18.2 us against
// 26); more of them, as clusters of 8 with rows of up to 65536 tokens in registers, win at any size (10 / 16 / 32 / 64
// requests of 32000 tokens: 22 / 21 / 22 / 42 us against 31 / 29 / 28 / 57; of 50257: 24 / 30 / 46 / 72 against 43 / 51 / 54
// / 86).  Larger vocabularies need 16 CTAs and are served in turns: 10 / 32 requests of 128256 tokens 29 / 68 us against 41
// / 71, 48 requests 99 against 92.  Greedy walks keep 16 CTAs (64 requests of 32000 tokens: 27 us against 33).  Sampling
// from the target, with half the bytes per node, is the better one at every size (87 requests of 128256 tokens 68 us
// against 104, 64 of 50257 27 against 37).  16-bit logits always stay here: the shared-memory walk does not read them.
static int walk_batch_cluster(const VerifyArgs& a, int requests) {
  if (a.temperature == 0.f) return vwk::kCl;
  const bool sample = (a.flags & SEQ_VERIFY_TARGET_SAMPLE) != 0;
  const bool bf16 = (a.flags & SEQ_VERIFY_LOGITS_BF16) != 0;
  if (a.V > vwk::kClBatch * vwk::kTh * 32) return sample || bf16 || requests * vwk::kCl <= 4 * device_sm_count() ? vwk::kCl : 0;
  if (requests * vwk::kCl > device_sm_count()) return vwk::kClBatch;
  static int side_by_side[9][64];  // per kernel shape and device: clusters of 16, + 1; 0 = not asked yet
  const int slice = (((a.V + vwk::kCl - 1) / vwk::kCl) + 3) & ~3;
  const int shape = (slice <= vwk::kTh * 8 ? 0 : slice <= vwk::kTh * 16 ? 1 : 2) + (sample ? 6 : bf16 ? 3 : 0);
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return vwk::kCl;
  if (dev >= 0 && dev < 64) n = __atomic_load_n(&side_by_side[shape][dev], __ATOMIC_ACQUIRE);
  if (n == 0) {
    if (walk_launch(a, vwk::kCl, 1, &n, nullptr) != SEQ_OK) n = 0;
    ++n;
    if (dev >= 0 && dev < 64) __atomic_store_n(&side_by_side[shape][dev], n, __ATOMIC_RELEASE);
  }
  return requests <= n - 1 ? vwk::kCl : vwk::kClBatch;
}

// SEQ_ERR_UNSUPPORTED: not a batch for this schedule.
int launch_verify_walk_batch(const VerifyArgs& a, int requests, cudaStream_t stream) {
  const int cl = walk_batch_cluster(a, requests);
  return cl == 0 ? SEQ_ERR_UNSUPPORTED : walk_launch(a, cl, requests, nullptr, stream);
}

}  // namespace seqtree

#ifdef SEQ_TRACE
// debug builds only: copy out and reset the timeline recorded by WTRACE()
extern "C" int seq_debug_walk_trace(unsigned long long* host_out) {
  int n = 0;
  cudaDeviceSynchronize();
  cudaMemcpyFromSymbol(&n, seqtree::g_wtrace_n, sizeof(int));
  if (n > 255) n = 255;
  cudaMemcpyFromSymbol(host_out, seqtree::g_wtrace, sizeof(unsigned long long) * 2 * n);
  int zero = 0;
  cudaMemcpyToSymbol(seqtree::g_wtrace_n, &zero, sizeof(int));
  return n;
}
#endif
