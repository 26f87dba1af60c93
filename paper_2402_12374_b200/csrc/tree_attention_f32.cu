// Tree-masked attention in single precision (fp32 inputs, fp32 FMAs on the CUDA cores).
//
// Work unit: (kv head, tile of 8 * RPT query rows, share of the key range).  A query row is a (node, head-in-group)
// pair, row = node * group + head, so the heads of a group share the K/V tiles; one CTA of 8 warps per SM.  Keys go in
// tiles of up to 128, fetched in groups of 32 by TMA (one thread, no issue slots of the warps that compute):
//     S   warp w scores its RPT rows against the tile, lane l the keys l, l+32, l+64, l+96: per step of 4 dimensions the
//         rows' q values are one broadcast load each and the K values one conflict-free 16-byte load per group, for
//         RPT * 4 * 4 multiply-adds taken two at a time (even and odd dimensions in one packed accumulator)
//     P   the row maximum and sum stay inside the warp (the rows of a warp are its own in both products), the
//         probabilities pass through shared memory to become broadcast operands: a warp barrier, no CTA barrier
//     O   lane l accumulates output dimensions 4l .. 4l+3 of the warp's rows, 32 keys in an accumulator of their own: one
//         chain over all keys of a long prefix rounds more than the short sums it stands for
// K of tile j+1 travels while P.V of tile j runs, V of tile j+1 while S of tile j+1 runs: one buffer each.
//
// What bounds it: multiply-adds and shared-memory reads side by side (12 16-byte loads per 128 FMA slots at RPT = 8) for
// 32 rows and more, the K/V stream below.  32 heads, 64 nodes, a prefix of 1024: one CTA per (node, head), which re-read
// K and V for each, took 331 us; this one 46 (the FMAs alone would take 16).  Rows fetched by cp.async from the computing
// warps: 58; by row-sized bulk copies: 71 (about 70 cycles for each 512 bytes).
#include <type_traits>

#include "common.cuh"
#include "tensor_map.cuh"

namespace seqtree {

constexpr int kF32Warps = 8;
constexpr int kF32Threads = 32 * kF32Warps;
constexpr int kF32Keys = 128;               // keys per tile
constexpr int kF32GroupBytes = 32 * kHeadDim * 4;  // 32 keys: [4 quarters of head_dim][32 keys][128 bytes], 128-byte swizzle

struct F32Args {
  const float* q; float* out;
  const uint32_t* mask_bits;
  float* lse;
  float* o_part; float2* ml;
  int64_t q_stride_tok, q_stride_head, o_stride_tok, o_stride_head;
  int32_t n, L_host, Hq, Hkv, group, mask_wpr, splits;
  int32_t L_count;       // > 1: one prefix length per request, requests stacked as heads
  const int32_t* L_dev;  // nullable: the prefix length in device memory (<= L_host)
  int32_t* dev_status;
  float scale_log2;      // softmax_scale * log2(e)
};

template <int RPT>
struct F32Smem {
  uint8_t k[4 * kF32GroupBytes];
  uint8_t v[4 * kF32GroupBytes];
  float q[kF32Warps * RPT][kHeadDim];
  float p[kF32Warps * RPT][kF32Keys];
  uint64_t k_full, v_full;  // one phase per tile
  uint32_t seen[kF32Warps][4];  // by group of the tile: the keys that some row of the warp sees (groups of tree keys)
};

__device__ __forceinline__ uint32_t f32_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// Waits for a phase of an mbarrier, with a bound; raises the device status when it runs out.
__device__ __forceinline__ void f32_wait(uint64_t* bar, uint32_t parity, int32_t* dev_status) {
  for (uint32_t it = 0; it < (1u << 22); ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(f32_smem(bar)), "r"(parity) : "memory");
    if (ok) return;
  }
  dev_flag(dev_status, SEQ_DEV_TIMEOUT);
}
__device__ __forceinline__ uint64_t f32_fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t f32_mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t f32_add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t f32_pair(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ float f32_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Scores of the warp's RPT rows against NJ groups of 32 keys.
template <int RPT, int NJ>
__device__ __forceinline__ void f32_scores(const F32Smem<RPT>& sm, int row0, int lane, float (&s)[RPT][NJ]) {
  uint64_t acc[RPT][NJ];
#pragma unroll
  for (int i = 0; i < RPT; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[i][j] = 0ull;
  const uint8_t* krow = sm.k + lane * 128;
#pragma unroll 2
  for (int w = 0; w < 32; ++w) {  // 16-byte words of head_dim: 8 to a quarter, the swizzle puts word x of key l at x ^ (l & 7)
    const int at = (w >> 3) * 4096 + (((w ^ lane) & 7) << 4);
    ulonglong2 kv[NJ], qv[RPT];
#pragma unroll
    for (int j = 0; j < NJ; ++j) kv[j] = *reinterpret_cast<const ulonglong2*>(krow + j * kF32GroupBytes + at);
#pragma unroll
    for (int i = 0; i < RPT; ++i) qv[i] = *reinterpret_cast<const ulonglong2*>(&sm.q[row0 + i][w * 4]);
    // (all accumulators once, then once more: a packed multiply-add never waits for the one before it)
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) acc[i][j] = f32_fma2(qv[i].x, kv[j].x, acc[i][j]);
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) acc[i][j] = f32_fma2(qv[i].y, kv[j].y, acc[i][j]);
  }
#pragma unroll
  for (int i = 0; i < RPT; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      float lo, hi;
      asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[i][j]));
      s[i][j] = lo + hi;
    }
}

// 32 visibility bits of tree indices [t, t + 32) of a mask row; negative indices are prefix keys (visible)
__device__ __forceinline__ uint32_t f32_window(const uint32_t* row, int wpr, int n, int t) {
  const int w = t >> 5;  // floor
  const uint32_t lo = w < 0 ? 0xFFFFFFFFu : (w < wpr ? row[w] : 0u);
  const uint32_t hi = (w + 1) < 0 ? 0xFFFFFFFFu : ((w + 1) < wpr ? row[w + 1] : 0u);
  uint32_t bits = __funnelshift_r(lo, hi, t & 31);
  const int nvis = n - t;
  if (nvis < 32) bits &= nvis <= 0 ? 0u : ((1u << nvis) - 1u);
  return bits;
}

// One tile of NJ groups of 32 keys for one warp: scores, softmax step, and (when the caller has made sure that V is in
// place) the product with V.
template <int RPT>
struct F32Row { float m[RPT], l[RPT]; ulonglong2 o[RPT]; };  // running maximum (the whole row's), this lane's share of the sum, output (two packed pairs)

template <int RPT, int NJ>
__device__ __forceinline__ void f32_softmax(F32Smem<RPT>& sm, F32Row<RPT>& st, int row0, int lane, float (&s)[RPT][NJ]) {
  float mx[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    mx[i] = s[i][0];
#pragma unroll
    for (int j = 1; j < NJ; ++j) mx[i] = fmaxf(mx[i], s[i][j]);
  }
#pragma unroll
  for (int i = 0; i < RPT; ++i) mx[i] = fmaxf(st.m[i], warp_max(mx[i]));
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const float ref = mx[i] == -INFINITY ? 0.f : mx[i];  // (a row that sees nothing so far: its terms are all 0)
    const float alpha = f32_ex2(st.m[i] - ref);
    float sum = 0.f;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const float p = f32_ex2(s[i][j] - ref);
      sum += p;
      sm.p[row0 + i][lane + 32 * j] = p;
    }
    st.l[i] = fmaf(st.l[i], alpha, sum);
    st.m[i] = mx[i];
    const uint64_t alpha2 = f32_pair(alpha, alpha);
    st.o[i].x = f32_mul2(st.o[i].x, alpha2);
    st.o[i].y = f32_mul2(st.o[i].y, alpha2);
  }
  __syncwarp();
}

// O += P V over group `grp` of 32 keys of the tile, summed by themselves and then added: relative error of the output against
// fp64, 64 nodes on 1024 keys: 4.8e-7 with one chain over all of a CTA's keys, 2.8e-7 so (a CTA per node and head, four
// chains: 3.9e-7), for 43.4 -> 45.4 us.
//
// kTree: the group reaches into the tree's keys, of which a row sees few.  A product is left out where p is 0, so that what
// another branch's row of V holds - infinities and NaN too - never reaches a row, and four keys that no row of the warp sees
// (`seen`, a bit for each key) are passed over: 64 nodes on 1024 keys 45.4 -> 46.4 us, 128 on 128 40.2 -> 36.8, 768 on none
// 84 -> 73 (branches in place of the predicates: 51.6, 44 and 100).
template <int RPT, bool kTree>
__device__ __forceinline__ void f32_pv(const F32Smem<RPT>& sm, F32Row<RPT>& st, int row0, int lane, int grp, uint32_t seen) {
  const uint8_t* vcol = sm.v + (lane >> 3) * 4096 + grp * kF32GroupBytes;  // this lane's quarter of head_dim
  ulonglong2 t[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) t[i] = make_ulonglong2(0ull, 0ull);
#pragma unroll (RPT < 8 ? 2 : 1)  // (the next four keys' operands on their way.  64 nodes on 1024 keys of 32 heads, RPT 4, 46.9 -> 44.8 us, one
  // node on 2000, RPT 1, 20.5 -> 18.8; with 8 rows a step has loads enough of its own: 85 nodes on 104 keys of 64/8 31.6 -> 32.9)
  for (int c = 0; c < 32; c += 4) {
    if (kTree && !((seen >> c) & 15u)) continue;
    const uint8_t* at = vcol + c * 128;
    const int word = (lane ^ c) & 7;  // (c is a multiple of 4: key c + e has swizzle (c & 7) + e)
    ulonglong2 vv[4];
    float4 p[RPT];
#pragma unroll
    for (int e = 0; e < 4; ++e) vv[e] = *reinterpret_cast<const ulonglong2*>(at + e * 128 + ((word ^ e) << 4));
#pragma unroll
    for (int i = 0; i < RPT; ++i) p[i] = *reinterpret_cast<const float4*>(&sm.p[row0 + i][32 * grp + c]);
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const float pe = e == 0 ? p[i].x : e == 1 ? p[i].y : e == 2 ? p[i].z : p[i].w;
        const uint64_t pp = f32_pair(pe, pe);
        if (kTree) {
          asm("{\n\t.reg .pred s;\n\tsetp.neu.f32 s, %4, 0f00000000;\n\t"
              "@s fma.rn.f32x2 %0, %5, %2, %0;\n\t@s fma.rn.f32x2 %1, %5, %3, %1;\n\t}"
              : "+l"(t[i].x), "+l"(t[i].y) : "l"(vv[e].x), "l"(vv[e].y), "f"(pe), "l"(pp));
        } else {
          t[i].x = f32_fma2(pp, vv[e].x, t[i].x);
          t[i].y = f32_fma2(pp, vv[e].y, t[i].y);
        }
      }
  }
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    st.o[i].x = f32_add2(st.o[i].x, t[i].x);
    st.o[i].y = f32_add2(st.o[i].y, t[i].y);
  }
}

template <int RPT>
__global__ void __launch_bounds__(kF32Threads, 1)
tree_attention_f32_kernel(const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap v_map, const F32Args a) {
  extern __shared__ uint8_t f32_raw[];
  // (an offset, not a rounded pointer: the compiler keeps seeing shared memory and the loads stay LDS)
  F32Smem<RPT>& sm = *reinterpret_cast<F32Smem<RPT>*>(f32_raw + ((1024u - (f32_smem(f32_raw) & 1023u)) & 1023u));
  constexpr int kRows = kF32Warps * RPT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, row0 = warp * RPT;
  const int g = blockIdx.y, split = blockIdx.z, R0 = blockIdx.x * kRows;
  const int rows_all = a.n * a.group;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(f32_smem(&sm.k_full)) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(f32_smem(&sm.v_full)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the kernel that merges the splits may be scheduled from now on (it waits before it reads)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  int L = a.L_host;
  if (a.L_dev != nullptr) {
    const int len = a.L_dev[a.L_count > 1 ? (g * a.L_count) / a.Hkv : 0];
    if ((len < 0 || len > a.L_host) && threadIdx.x == 0) dev_flag(a.dev_status, SEQ_DEV_BAD_LENGTH);
    L = min(max(len, 0), a.L_host);
  }
  // a node sees no later node: the tile's keys end behind its last node's own; the splits share them by groups of 32
  const int n_keys = L + (min(R0 + kRows, rows_all) - 1) / a.group + 1;
  const int groups = (n_keys + 31) >> 5;
  const int grp_lo = (int)(((int64_t)split * groups) / a.splits), grp_hi = (int)(((int64_t)(split + 1) * groups) / a.splits);

  // thread 0 requests the groups of a tile; a group's copy brings the four quarters of its keys' rows
  auto request = [&](const CUtensorMap* map, uint8_t* dst, uint64_t* full, int grp) {
    const int cnt = min(4, grp_hi - grp);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(f32_smem(full)), "r"(cnt * kF32GroupBytes) : "memory");
    for (int j = 0; j < cnt; ++j)
      asm volatile(
          "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
          ::"r"(f32_smem(dst + j * kF32GroupBytes)), "l"(map), "r"(f32_smem(full)), "r"(0), "r"((grp + j) * 32), "r"(0), "r"(g) : "memory");
  };
  if (threadIdx.x == 0 && grp_lo < grp_hi) {
    request(&k_map, sm.k, &sm.k_full, grp_lo);
    request(&v_map, sm.v, &sm.v_full, grp_lo);
  }
  // this warp's query rows, scaled into the log2 domain
  {
    float4 x[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int R = R0 + row0 + i;
      x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (R < rows_all) {
        const int node = R / a.group, h = g * a.group + R - node * a.group;
        x[i] = *reinterpret_cast<const float4*>(a.q + (int64_t)node * a.q_stride_tok + (int64_t)h * a.q_stride_head + lane * 4);
      }
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i)
      *reinterpret_cast<float4*>(&sm.q[row0 + i][lane * 4]) =
          make_float4(x[i].x * a.scale_log2, x[i].y * a.scale_log2, x[i].z * a.scale_log2, x[i].w * a.scale_log2);
  }
  F32Row<RPT> st;
#pragma unroll
  for (int i = 0; i < RPT; ++i) { st.m[i] = -INFINITY; st.l[i] = 0.f; st.o[i] = make_ulonglong2(0ull, 0ull); }
  const bool warp_live = R0 + row0 < rows_all;
  __syncthreads();  // the barriers are armed

  uint32_t phase = 0;
  for (int grp = grp_lo; grp < grp_hi; grp += 4, phase ^= 1u) {
    const int nj = min(4, grp_hi - grp);
    const bool more = grp + 4 < grp_hi;
    f32_wait(&sm.k_full, phase, a.dev_status);
    auto tile = [&](auto nj_const) {
      constexpr int NJ = decltype(nj_const)::value;
      float s[RPT][NJ];
      if (warp_live) f32_scores<RPT, NJ>(sm, row0, lane, s);
      __syncthreads();  // everyone has read K
      if (more && threadIdx.x == 0) request(&k_map, sm.k, &sm.k_full, grp + 4);
      if (warp_live) {
        if ((grp + NJ) * 32 > L) {  // the tile reaches into the tree's keys (or past the end)
          uint32_t seen[NJ] = {};
#pragma unroll
          for (int i = 0; i < RPT; ++i) {
            const int node = min((R0 + row0 + i) / a.group, a.n - 1);
            const uint32_t* mrow = a.mask_bits + (size_t)node * a.mask_wpr;
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
              const uint32_t bits = f32_window(mrow, a.mask_wpr, node + 1, (grp + j) * 32 - L);
              if (!((bits >> lane) & 1u)) s[i][j] = -INFINITY;
              seen[j] |= bits;
            }
          }
#pragma unroll
          for (int j = 0; j < NJ; ++j)
            if (lane == j) sm.seen[warp][j] = seen[j];
        }
        f32_softmax<RPT, NJ>(sm, st, row0, lane, s);
      }
    };
    if (nj == 4) tile(std::integral_constant<int, 4>());
    else if (nj == 3) tile(std::integral_constant<int, 3>());
    else if (nj == 2) tile(std::integral_constant<int, 2>());
    else tile(std::integral_constant<int, 1>());
    f32_wait(&sm.v_full, phase, a.dev_status);
    if (warp_live) {
#pragma unroll 1
      for (int j = 0; j < nj; ++j) {
        if ((grp + j + 1) * 32 <= L) f32_pv<RPT, false>(sm, st, row0, lane, j, 0u);
        else f32_pv<RPT, true>(sm, st, row0, lane, j, sm.seen[warp][j]);
      }
    }
    __syncthreads();  // everyone has read V
    if (more && threadIdx.x == 0) request(&v_map, sm.v, &sm.v_full, grp + 4);
  }

#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int R = R0 + row0 + i;
    if (R >= rows_all) break;
    const int node = R / a.group, h = g * a.group + R - node * a.group;
    const float sum = warp_sum(st.l[i]);
    if (a.splits == 1) {
      const float inv = 1.f / sum;  // the row sees itself, so sum > 0
      const ulonglong2 o = make_ulonglong2(f32_mul2(st.o[i].x, f32_pair(inv, inv)), f32_mul2(st.o[i].y, f32_pair(inv, inv)));
      *reinterpret_cast<float4*>(a.out + (int64_t)node * a.o_stride_tok + (int64_t)h * a.o_stride_head + lane * 4) =
          *reinterpret_cast<const float4*>(&o);
      if (a.lse != nullptr && lane == 0) a.lse[(size_t)h * a.n + node] = (st.m[i] + log2f(sum)) * kLn2;
    } else {
      const size_t row = ((size_t)split * a.Hq + h) * a.n + node;
      *reinterpret_cast<float4*>(a.o_part + row * kHeadDim + lane * 4) = *reinterpret_cast<const float4*>(&st.o[i]);
      if (lane == 0) a.ml[row] = make_float2(st.m[i], sum);
    }
  }
}

// Rows per tile and key-range splits: the pair with the least estimated time.  Measured per CTA and group of 32 keys:
// 4.1 / 2.1 us for 64 / 32 rows (both products at about 60 % of the FMA pipe, where the shared-memory port is as busy);
// fewer rows end at the 32 KB of K and V that an SM streams in 0.8 us.  About 4.5 us per CTA for launch, first tiles and
// epilogue, 3 for the merge launch.  (Figures of the kernel with one step of P V in flight; with two, for up to 32 rows, a
// group takes 3 to 8 % less.  Over 44 shapes the picks were 2 % above the best of all pairs on the average and 35 % at worst, 37
// nodes on 586 keys of 52 heads.)
struct F32Plan { int rpt, splits; };
static F32Plan f32_plan(const seq_tree_attention_params& p, size_t max_workspace) {
  const int G = p.num_q_heads / p.num_kv_heads, rows = p.n_tree * G, sms = device_sm_count();
  const int groups = (p.prefix_len + p.n_tree + 31) / 32;
  F32Plan best = {8, 1};
  double best_cost = -1.0;
  for (int rpt = 1; rpt <= 8; rpt *= 2) {
    const long units = (long)((rows + kF32Warps * rpt - 1) / (kF32Warps * rpt)) * p.num_kv_heads;
    const double per_group = rpt == 8 ? 4.1 : rpt == 4 ? 2.1 : rpt == 2 ? 1.25 : 0.85;
    for (int splits = 1; splits <= 32 && splits <= groups; ++splits) {
      if (splits > 1 && split_workspace_bytes(splits, p.num_q_heads, p.n_tree) > max_workspace) break;
      const long waves = (units * splits + sms - 1) / sms;
      const double cost = (double)waves * (per_group * ((groups + splits - 1) / splits) + 4.5) + (splits > 1 ? 3.0 + 0.1 * splits : 0.0);
      if (best_cost < 0 || cost < best_cost - 1e-9) { best = {rpt, splits}; best_cost = cost; }
    }
  }
  return best;
}

int f32_splits(const seq_tree_attention_params& p) { return f32_plan(p, ~(size_t)0).splits; }

// max_workspace: what the caller can lend for the partial results of the splits
int launch_attention_f32(const seq_tree_attention_params& p, size_t max_workspace, cudaStream_t stream) {
  const F32Plan plan = f32_plan(p, max_workspace);
  F32Args a;
  a.q = static_cast<const float*>(p.q);
  a.out = static_cast<float*>(p.out);
  a.mask_bits = p.mask_bits; a.lse = p.lse;
  const SplitLayout sl = split_layout(p.workspace, plan.splits, p.num_q_heads, p.n_tree);
  a.o_part = sl.o_part; a.ml = sl.ml;
  a.q_stride_tok = p.q_stride_tok; a.q_stride_head = p.q_stride_head;
  a.o_stride_tok = p.o_stride_tok; a.o_stride_head = p.o_stride_head;
  a.n = p.n_tree; a.L_host = p.prefix_len; a.Hq = p.num_q_heads; a.Hkv = p.num_kv_heads;
  a.group = p.num_q_heads / p.num_kv_heads;
  a.mask_wpr = p.mask_words_per_row; a.splits = plan.splits;
  a.L_count = p.prefix_len_dev_count; a.L_dev = p.prefix_len_dev; a.dev_status = p.dev_status;
  a.scale_log2 = (p.softmax_scale > 0.f ? p.softmax_scale : 0.08838834764831845f) * kLog2e;
  CUtensorMap k_map, v_map;
  for (int which = 0; which < 2; ++which) {
    // the live rows only (what lies behind them reads as zero); with the length in device memory, the whole cache.
    // head_dim in four quarters of 128 bytes, the swizzle's width
    const cuuint64_t dims[4] = {32, (cuuint64_t)(p.prefix_len_dev != nullptr ? p.kv_capacity : p.prefix_len + p.n_tree), 4, (cuuint64_t)p.num_kv_heads};
    const cuuint64_t strides[3] = {(cuuint64_t)p.kv_stride_tok * 4, 128, (cuuint64_t)p.kv_stride_head * 4};
    const cuuint32_t box[4] = {32, 32, 4, 1};
    if (!tensor_map(which == 0 ? &k_map : &v_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, which == 0 ? p.k_cache : p.v_cache, dims, strides, box))
      return SEQ_ERR_CUDA;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kF32Threads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // set-up under the previous kernel's tail
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto launch = [&](auto kernel, size_t smem, int rpt, int which) -> int {
    static int attr_done[4][64];
    const int rc = once_per_device(attr_done[which], [&]() -> int {
      SEQ_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      return SEQ_OK;
    });
    if (rc != SEQ_OK) return rc;
    cfg.gridDim = dim3((p.n_tree * a.group + kF32Warps * rpt - 1) / (kF32Warps * rpt), p.num_kv_heads, plan.splits);
    cfg.dynamicSmemBytes = smem;
    SEQ_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, k_map, v_map, a));
    return SEQ_OK;
  };
  int rc = SEQ_ERR_UNSUPPORTED;
  switch (plan.rpt) {
    case 1: rc = launch(tree_attention_f32_kernel<1>, sizeof(F32Smem<1>) + 1024, 1, 0); break;
    case 2: rc = launch(tree_attention_f32_kernel<2>, sizeof(F32Smem<2>) + 1024, 2, 1); break;
    case 4: rc = launch(tree_attention_f32_kernel<4>, sizeof(F32Smem<4>) + 1024, 4, 2); break;
    case 8: rc = launch(tree_attention_f32_kernel<8>, sizeof(F32Smem<8>) + 1024, 8, 3); break;
  }
  if (rc != SEQ_OK || plan.splits == 1) return rc;
  return launch_combine_splits(p, plan.splits, stream);
}

}  // namespace seqtree
