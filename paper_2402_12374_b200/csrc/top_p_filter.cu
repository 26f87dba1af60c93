// seq_tree_top_p_filter: nucleus truncation of softmax(logits / T), row by row (the top-p hyperparameter of the
// robustness study, Section 4.2).  A histogram of the probability MASS over equal steps of the exponent argument finds the
// bin in which the cut falls; the tokens of that bin (a few dozen on the paper's shapes) are ordered exactly in shared
// memory by (logit bits, token id).  Masses are 2^-40 fixed point in 64-bit integers: sums are exact and independent of
// their order, so the kept set is reproducible bit for bit.
//
// One row is one cluster of up to 8 CTAs (vocabularies up to 131072) and is read once: each CTA's slice stays in shared
// memory through all passes.  (In registers it would take loops unrolled over all of a thread's tokens, and the passes would
// wait for their own instructions: 24 us for 64 rows of 32000.)  Exchanges over distributed shared memory: the row maximum,
// the histograms with the masses' sums, the tokens of the cut's bin; every CTA then finds the cut by itself and writes its
// slice.  The histogram covers the exponent arguments below 15 first - tokens below 2^-15 of the most probable one, most of
// the vocabulary, only enter the sum - and the rest, in two more rounds, in the rare case that the cut is not among them.
// Where more than 512 tokens share the cut's bin (flat rows, long runs of equal logits) the bin is cut up by the logit bits,
// 9 at a time, until few tokens are left or all are equal (tp_refine).  Larger vocabularies: one CTA takes the row through
// global memory, in four passes, or with more than 1024 tokens in the cut's bin in seven with a radix select on the logit
// bits (11 + 11 + 10).
//
// What bounds it: the chain of exchanges for a few rows, instruction issue for many (75 instructions for each token, 58 % of
// the issue slots, at 512 rows of 32000).  64 rows of 32000 tokens: 29.7 us with one CTA of 1024 threads per row reading it
// four times and adding every token to the histogram, 13.6 with a cluster per row that worked out every token's bin in two
// passes and queued the histogram's tokens by votes, 12.5 so: estimates to a margin tell most tokens off, their mass is taken
// without a branch, the histogram's tokens wait in lists of the threads' own.  127 rows of 128256 71 -> 61 us, 378 192 -> 168,
// 300 of 50257 68 -> 61; at temperature 1, where a third of the tokens are in the histogram, 127 rows 79.4 -> 76.0, 512 of 32000
// 64.6 -> 63.5, but 3 of 32000 9.14 -> 9.3; at 1.5, 512 rows of 128256 346 -> 344.  (Exact limits found by a search over the
// floats: 15.0; a warp's queue instead of lists: 13.4; lists of 16: 378 rows 180.)
#include <climits>
#include <cstddef>

#include <type_traits>

#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace seqtree {

constexpr int kTpThreads = 512;      // per CTA of a cluster
constexpr int kTpWarps = kTpThreads / 32;
constexpr int kTpRowThreads = 1024;  // of the one CTA that takes a row of a larger vocabulary
constexpr float kTpScale = 1099511627776.f;  // 2^40
constexpr int kTpCand = 1024;  // tokens of the cut's bin that are ordered in shared memory (more: radix select)

struct TopPArgs {
  const float* logits; int64_t in_stride;
  float* out; int64_t out_stride;
  int32_t V;
  float c2;       // log2(e) / T
  float bin_width;  // of a first-level bin, in logits (rounded: for estimates)
  double top_p;
  int32_t* kept_out; int32_t* dev_status;
};

struct TpShared {
  __align__(16) unsigned long long hist[2048];
  // first-level histogram as three 32-bit limbs per bin (native 32-bit shared-memory adds; a 64-bit add is a
  // compare-and-swap loop): mass = lo + hi * 2^21 + top * 2^53, carries moved up when an add wraps
  uint32_t lo[2048], hi[2048], top[2048];
  uint32_t count[1024];
  __align__(16) unsigned long long warp_tot[kTpRowThreads / 32];
  float warp_max[kTpRowThreads / 32];
  // results of a level's search
  uint32_t sel_bin; unsigned long long sel_above; unsigned long long sel_mass; uint32_t sel_count;
  int32_t tie_limit;
  int32_t bad, kept, ncand;
  unsigned long long tau_comp;
};

// order-preserving map float -> uint32 (ascending)
__device__ __forceinline__ uint32_t tp_key(float x) {
  const uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
// NaN and +inf count as -inf (never kept)
__device__ __forceinline__ float tp_clean(float x, int& bad) {
  if (!(x < INFINITY)) { bad = 1; return -INFINITY; }
  return x;
}
__device__ __forceinline__ float tp_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ unsigned long long tp_mass(float x, float M, float c2) {
  return __float2ull_rn(tp_ex2((x - M) * c2) * kTpScale);  // (-inf - M) * c2 = -inf -> 0
}

// calls f(index, value) for every element of the row: float4 body with four independent loads in flight per
// thread (the passes are latency-bound otherwise), scalar tail
template <typename F>
__device__ __forceinline__ void tp_for_each(const float* row, int V, F f) {
  const int V4 = V & ~3;
  constexpr int kStride = kTpRowThreads * 4;
  int i = threadIdx.x * 4;
  for (; i + 3 * kStride < V4; i += 4 * kStride) {
    float4 x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = *reinterpret_cast<const float4*>(row + i + k * kStride);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int j = i + k * kStride;
      f(j, x[k].x); f(j + 1, x[k].y); f(j + 2, x[k].z); f(j + 3, x[k].w);
    }
  }
  {  // up to three more, again loaded together
    float4 x[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (i + k * kStride < V4) x[k] = *reinterpret_cast<const float4*>(row + i + k * kStride);
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (i + k * kStride < V4) {
        const int j = i + k * kStride;
        f(j, x[k].x); f(j + 1, x[k].y); f(j + 2, x[k].z); f(j + 3, x[k].w);
      }
  }
  for (int t = V4 + threadIdx.x; t < V; t += kTpRowThreads) f(t, row[t]);
}

// Exclusive prefix sum over the block's threads in thread order; every thread also gets the total.
template <int kThreads>
__device__ __forceinline__ unsigned long long tp_block_scan(unsigned long long v, unsigned long long* warp_tot, unsigned long long& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long up = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += up;
  }
  __syncthreads();  // warp_tot free for reuse
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  unsigned long long before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; w += 2) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(&warp_tot[w]);
    if (w < warp) before += t.x;
    if (w + 1 < warp) before += t.y;
    all += t.x + t.y;
  }
  total = all;
  return before + inc - v;
}

// Among `bins` bins of sh.hist taken from the highest index down, finds the one in which the running mass reaches
// `target` (> 0, <= the bins' total); leaves its index, the mass above it, its own mass (and token count when
// `with_count`) in sh.sel_*.  bins is 2048 or 1024: two or one per thread.
__device__ __forceinline__ void tp_find_crossing(TpShared& sh, int bins, unsigned long long target, bool with_count) {
  const int per = bins / kTpRowThreads;
  const int hi = bins - 1 - (int)threadIdx.x * per;  // this thread's highest bin
  unsigned long long mine = 0, total;
  for (int b = 0; b < per; ++b) mine += sh.hist[hi - b];
  unsigned long long above = tp_block_scan<kTpRowThreads>(mine, sh.warp_tot, total);
  if (above < target && target <= above + mine) {
    for (int b = 0; b < per; ++b) {
      const unsigned long long m = sh.hist[hi - b];
      if (above < target && target <= above + m) {
        sh.sel_bin = hi - b; sh.sel_above = above; sh.sel_mass = m; sh.sel_count = with_count ? sh.count[hi - b] : 0u;
      }
      above += m;
    }
  }
  __syncthreads();
}

// First-level bin of a (cleaned) logit: 2048 equal steps of the exponent argument d = (M - x) * log2(e) / T over
// [0, 40), most probable tokens in the highest bin; -1 beyond (mass below one unit of the fixed point: never kept).
// Sub, multiply by a positive constant and truncation are monotone, so a higher bin never holds a smaller logit.
__device__ __forceinline__ int tp_lbin(float x, float M, float c2) {
  const float d = (M - x) * c2;
  return d < 40.f ? 2047 - (int)(d * 51.2f) : -1;
}

// Among n tokens of the cut's bin, (key and index, mass) each, finds the last kept one: the first, in descending order, at
// which the running mass reaches `rest`.  No sort: a token's running mass is the sum over those before it.
template <int kThreads>
__device__ __forceinline__ void tp_cut(const ulonglong2* tokens, int n, unsigned long long rest, unsigned long long* tau_comp) {
  for (int i = threadIdx.x; i < n; i += kThreads) {
    const ulonglong2 mine = tokens[i];
    unsigned long long before = 0;
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      const ulonglong2 t = tokens[j];
      before += t.x > mine.x ? t.y : 0ull;
    }
    if (before < rest && rest <= before + mine.y) *tau_comp = mine.x;
  }
  __syncthreads();
}

// One row by one CTA through global memory.  (64 rows of 151936 tokens: 85 us; with 512 threads,
// and half the loads in flight, 132.)
__global__ void __launch_bounds__(kTpRowThreads, 1) top_p_row_kernel(const TopPArgs a) {
  extern __shared__ __align__(16) uint8_t tp_smem[];
  TpShared& sh = *reinterpret_cast<TpShared*>(tp_smem);
  const int row_index = blockIdx.x;
  const float* row = a.logits + (int64_t)row_index * a.in_stride;
  float* orow = a.out + (int64_t)row_index * a.out_stride;
  const int V = a.V, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  // ---- the row maximum (NaN / +inf flagged and read as -inf), histogram cleared meanwhile
  for (int i = threadIdx.x; i < 2048; i += kTpRowThreads) { sh.lo[i] = 0u; sh.hi[i] = 0u; sh.top[i] = 0u; }
  if (threadIdx.x == 0) { sh.bad = 0; sh.kept = 0; sh.tie_limit = INT_MAX; sh.ncand = 0; sh.tau_comp = 0ull; }
  int bad = 0;
  float m = -INFINITY;
  tp_for_each(row, V, [&](int, float x) { m = fmaxf(m, tp_clean(x, bad)); });
  m = warp_max(m);
  if (lane == 0) sh.warp_max[warp] = m;
  __syncthreads();
  float M = -INFINITY;
#pragma unroll 1
  for (int w = 0; w < kTpRowThreads / 32; ++w) M = fmaxf(M, sh.warp_max[w]);
  if (bad) sh.bad = 1;
  if (M == -INFINITY) {  // no token with any mass: nothing to keep
    tp_for_each(row, V, [&](int i, float) { orow[i] = -INFINITY; });
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
      dev_flag(a.dev_status, SEQ_DEV_DEGENERATE | (bad ? SEQ_DEV_NONFINITE : 0));
      if (a.kept_out != nullptr) a.kept_out[row_index] = 0;
    }
    return;
  }

  // ---- first level: every token with mass, equal steps of the exponent argument (tokens spread over many bins:
  // few collisions between the atomic adds, and the bin of the cut holds few tokens)
  tp_for_each(row, V, [&](int, float x) {
    int b2 = 0;
    x = tp_clean(x, b2);
    const int lb = tp_lbin(x, M, a.c2);
    if (lb >= 0) {
      const unsigned long long w = tp_mass(x, M, a.c2);
      const uint32_t l = (uint32_t)w & 0x1fffffu, h = (uint32_t)(w >> 21);
      uint32_t carry = h;
      if (l) {
        const uint32_t old = atomicAdd(&sh.lo[lb], l);
        carry += (old + l < old) ? 2048u : 0u;  // a wrap of lo is 2^32 = 2048 units of hi
      }
      if (carry) {
        const uint32_t old = atomicAdd(&sh.hi[lb], carry);
        if (old + carry < old) atomicAdd(&sh.top[lb], 1u);
      }
    }
  });
  __syncthreads();
  for (int i = threadIdx.x; i < 2048; i += kTpRowThreads)
    sh.hist[i] = (unsigned long long)sh.lo[i] + ((unsigned long long)sh.hi[i] << 21) + ((unsigned long long)sh.top[i] << 53);
  __syncthreads();
  unsigned long long target;
  {
    // the whole mass, then the mass the nucleus has to reach (rounded up, at least one unit)
    unsigned long long mine = 0, S;
    for (int i = threadIdx.x; i < 2048; i += kTpRowThreads) mine += sh.hist[i];
    tp_block_scan<kTpRowThreads>(mine, sh.warp_tot, S);
    const double want = ceil(a.top_p * (double)S);
    target = want < 1.0 ? 1ull : (want >= (double)S ? S : (unsigned long long)want);
  }
  tp_find_crossing(sh, 2048, target, false);
  const int B0 = (int)sh.sel_bin;                    // the bin in which the cut falls
  const unsigned long long rest0 = target - sh.sel_above;  // mass still to find inside it
  __syncthreads();

  // ---- the tokens of that bin, as (key, ~index) so that a larger value means "earlier in the order"
  ulonglong2* cand = reinterpret_cast<ulonglong2*>(sh.hist);  // [kTpCand]   (the histogram is no longer needed)
  tp_for_each(row, V, [&](int i, float x) {
    int b2 = 0;
    x = tp_clean(x, b2);
    if (tp_lbin(x, M, a.c2) == B0) {
      const int pos = atomicAdd(&sh.ncand, 1);
      if (pos < kTpCand) {
        cand[pos] = make_ulonglong2(((unsigned long long)tp_key(x) << 32) | (uint32_t)~(uint32_t)i, tp_mass(x, M, a.c2));
      }
    }
  });
  __syncthreads();
  const int ncand = sh.ncand;
  uint32_t tau = 0;          // fallback only: key of the least probable kept token
  bool exact = ncand <= kTpCand;
  if (exact) {
    tp_cut<kTpRowThreads>(cand, ncand, rest0, &sh.tau_comp);
  } else {
    // ---- many tokens in one bin (a flat row, runs of equal logits): radix select on the key bits inside the bin
    __syncthreads();
    for (int i = threadIdx.x; i < 2048; i += kTpRowThreads) sh.hist[i] = 0ull;
    __syncthreads();
    tp_for_each(row, V, [&](int, float x) {
      int b2 = 0;
      x = tp_clean(x, b2);
      if (tp_lbin(x, M, a.c2) == B0) atomicAdd(&sh.hist[tp_key(x) >> 21], tp_mass(x, M, a.c2));
    });
    __syncthreads();
    tp_find_crossing(sh, 2048, rest0, false);
    const uint32_t p0 = sh.sel_bin;
    const unsigned long long above0 = sh.sel_above;
    __syncthreads();
    for (int i = threadIdx.x; i < 2048; i += kTpRowThreads) sh.hist[i] = 0ull;
    __syncthreads();
    tp_for_each(row, V, [&](int, float x) {
      int b2 = 0;
      x = tp_clean(x, b2);
      const uint32_t k = tp_key(x);
      if ((k >> 21) == p0 && tp_lbin(x, M, a.c2) == B0) atomicAdd(&sh.hist[(k >> 10) & 0x7ffu], tp_mass(x, M, a.c2));
    });
    __syncthreads();
    tp_find_crossing(sh, 2048, rest0 - above0, false);
    const uint32_t p1 = (p0 << 11) | sh.sel_bin;
    const unsigned long long above1 = above0 + sh.sel_above;
    __syncthreads();
    for (int i = threadIdx.x; i < 1024; i += kTpRowThreads) { sh.hist[i] = 0ull; sh.count[i] = 0u; }
    __syncthreads();
    tp_for_each(row, V, [&](int, float x) {
      int b2 = 0;
      x = tp_clean(x, b2);
      const uint32_t k = tp_key(x);
      if ((k >> 10) == p1 && tp_lbin(x, M, a.c2) == B0) {
        atomicAdd(&sh.hist[k & 0x3ffu], tp_mass(x, M, a.c2));
        atomicAdd(&sh.count[k & 0x3ffu], 1u);
      }
    });
    __syncthreads();
    tp_find_crossing(sh, 1024, rest0 - above1, true);
    tau = (p1 << 10) | sh.sel_bin;
    // tokens with exactly that logit share one mass: the first `need` of them in token order are kept
    const uint32_t ties = sh.sel_count;
    const unsigned long long each = sh.sel_mass / (ties ? ties : 1u);
    const unsigned long long rest = rest0 - above1 - sh.sel_above;
    uint32_t need = each ? (uint32_t)((rest + each - 1) / each) : ties;
    need = need < 1u ? 1u : (need > ties ? ties : need);
    __syncthreads();
    if (need < ties) {
      // the cut falls inside a run of equal logits: contiguous chunks per thread, a scan of the tie counts, and the
      // thread whose chunk holds the need-th tie finds its index
      const int len = (V + kTpRowThreads - 1) / kTpRowThreads;
      const int lo = min((int)threadIdx.x * len, V), hi = min(lo + len, V);
      unsigned long long cnt = 0;
      for (int i = lo; i < hi; ++i) {
        int b2 = 0;
        cnt += tp_key(tp_clean(row[i], b2)) == tau;
      }
      unsigned long long total;
      const unsigned long long before = tp_block_scan<kTpRowThreads>(cnt, sh.warp_tot, total);
      if (before < need && need <= before + cnt) {
        unsigned long long seen = before;
        for (int i = lo; i < hi; ++i) {
          int b2 = 0;
          if (tp_key(tp_clean(row[i], b2)) == tau && ++seen == need) { sh.tie_limit = i; break; }
        }
      }
      __syncthreads();
    }
  }
  const unsigned long long tau_comp = exact ? sh.tau_comp : (((unsigned long long)tau << 32) | (uint32_t)~(uint32_t)min(sh.tie_limit, V - 1));

  // ---- write: the logit itself inside the nucleus, -inf outside.  Inside: a more probable bin, or the cut's bin
  // and not behind the last kept token in the order (key descending, index ascending).
  int kept = 0;
  tp_for_each(row, V, [&](int i, float x) {
    int b2 = 0;
    const float c = tp_clean(x, b2);
    const int lb = tp_lbin(c, M, a.c2);
    const unsigned long long comp = ((unsigned long long)tp_key(c) << 32) | (uint32_t)~(uint32_t)i;
    const bool keep = lb > B0 || (lb == B0 && comp >= tau_comp);
    orow[i] = keep ? x : -INFINITY;
    kept += keep;
  });
  kept = __reduce_add_sync(0xffffffffu, kept);
  if (lane == 0) atomicAdd(&sh.kept, kept);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (a.kept_out != nullptr) a.kept_out[row_index] = sh.kept;
    if (sh.bad) dev_flag(a.dev_status, SEQ_DEV_NONFINITE);
  }
}

// One row by one cluster, the CTA's slice in shared memory.
constexpr int kTpBins = 768;           // bins of one round of the histogram, 24 groups of 32
constexpr int kTpRounds = 3;           // 2048 bins in rounds, most probable first (the last one is shorter)
constexpr int kTpMaxCluster = 8, kTpMaxSlice = 16384;
// Tokens of the cut's bin that are ordered by their running masses (more: tp_refine; with 1024, rows of deviation 0.5 below
// take 408 us instead of 452, ordinary ones 208 instead of 193, for the room), and from how many on each CTA of the cluster
// looks at its own ones only.
constexpr int kTpFastCand = 512, kTpAlone = 128;
constexpr int kTpList = 8;             // per thread: tokens of the round's bins waiting to be added
struct TpFast {
  // Two limbs of 20 and 21 bits per bin, added without a return value; from 4096 tokens in one bin on they could wrap, and
  // then the bins' total is not the exact sum of the round's masses any more.
  uint32_t limb[2][kTpBins];
  unsigned long long coarse[32];       // masses of the groups of bins; [24] all tokens' mass, [25] the round's tokens' (both exact)
  unsigned long long stage[kTpMaxCluster][32];  // what was read from the cluster's CTAs
  __align__(16) unsigned long long part[2][kTpWarps];
  __align__(16) ulonglong2 cand[kTpFastCand];  // this CTA's tokens of the cut's bin (read by the other CTAs); before that the threads' lists
  __align__(16) ulonglong2 all[kTpFastCand];   // the cluster's
  unsigned long long tau_comp;
  int32_t max;                         // the row's maximum as an ordered integer (every CTA of the cluster adds its warps')
  int32_t ncand;
  uint32_t kmin, kmax;                 // tp_refine: range of the keys in question (every CTA of the cluster adds its warps')
  uint32_t klo, khi;                   // ... and what is left of it
  __align__(16) float x[4];            // the slice (as long as it is)
};

static_assert(offsetof(TpFast, all) == offsetof(TpFast, cand) + sizeof(TpFast::cand) && sizeof(TpFast::cand) + sizeof(TpFast::all) >= kTpList * kTpThreads * 4,
              "the threads' lists take the place of both token lists");

// float <-> int of the same order
__device__ __forceinline__ int tp_ordered(float x) { const int b = __float_as_int(x); return b ^ ((b >> 31) & 0x7fffffff); }
__device__ __forceinline__ float tp_unordered(int b) { return __int_as_float(b ^ ((b >> 31) & 0x7fffffff)); }

// Warp-wide: inclusive prefix sum over the lanes.
__device__ __forceinline__ unsigned long long tp_warp_scan(unsigned long long v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long up = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += up;
  }
  return v;
}
__device__ __forceinline__ unsigned long long tp_warp_sum(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// tp_cut for many tokens: each CTA looks among its own ones, up to 32 threads share one's running mass, and whoever holds the
// last kept token tells the others, for one barrier more on the way.  (378 rows of 128256 logits of deviation 1, 400 tokens
// in the bin: 440 us when every CTA looked at all of them, so 284.  64 rows of 32000 of deviation 3, where few are in the
// bin, would take 13.4 us instead of 12.8.)
__device__ __forceinline__ void tp_cut_own(TpFast& me, int n, unsigned long long rest, int ranks) {
  cg::cluster_group cluster = cg::this_cluster();
  const int count = me.ncand;
  int log_share = 0;
  while (log_share < 5 && (count << (log_share + 1)) <= kTpThreads) ++log_share;
  const int sub = threadIdx.x & ((1 << log_share) - 1);
  for (int i0 = 0; i0 < count; i0 += kTpThreads >> log_share) {  // (whole warps)
    const int i = i0 + ((int)threadIdx.x >> log_share);
    const ulonglong2 mine = i < count ? me.cand[i] : make_ulonglong2(~0ull, 0ull);
    unsigned long long before = 0;
#pragma unroll 4
    for (int j = sub; j < n; j += 1 << log_share) {
      const ulonglong2 t = me.all[j];
      before += t.x > mine.x ? t.y : 0ull;
    }
    for (int d = 0; d < log_share; ++d) before += __shfl_xor_sync(0xffffffffu, before, 1 << d);
    if (sub == 0 && before < rest && rest <= before + mine.y)
      for (int r = 0; r < ranks; ++r) cluster.map_shared_rank(&me, r)->tau_comp = mine.x;
  }
}

// The tokens of the cluster's lists (me.cand, me.ncand of them, which may be more than were stored): their number, and when
// they are few a copy of all of them in me.all.  `before`: those of lower ranks.  A cluster barrier precedes the reads.
__device__ __forceinline__ int tp_gather(TpFast& me, int ranks, int rank, int& before) {
  cg::cluster_group cluster = cg::this_cluster();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  cluster.sync();
  const int c = lane < ranks ? cluster.map_shared_rank(&me, lane)->ncand : 0;
  int incl = c;
#pragma unroll
  for (int o = 1; o < kTpMaxCluster; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  const int n = __shfl_sync(0xffffffffu, incl, kTpMaxCluster - 1);
  const int theirs = __shfl_sync(0xffffffffu, c, warp % kTpMaxCluster);
  const int at = __shfl_sync(0xffffffffu, incl, warp % kTpMaxCluster) - theirs;
  if (warp < ranks && n <= kTpFastCand) {  // warp r copies CTA r's list
    const TpFast* other = cluster.map_shared_rank(&me, warp);
    for (int i = lane; i < theirs; i += 32) me.all[at + i] = other->cand[i];
  }
  before = __shfl_sync(0xffffffffu, incl - c, rank);
  return n;
}

// Where more than kTpFastCand tokens are in question - a flat row, runs of equal logits, a bin of the histogram that
// wrapped: the tokens with cut_lo <= bin < cut_hi, in which mass `rest` is still to be found.  Their keys are cut into 512
// equal steps, the step with the cut is found by the masses (three limbs of 14 bits, which cannot wrap), and so on inside
// it until few tokens are left or they are all equal; equal ones are kept in token order.  Leaves the range of keys in
// which the cut lies in me.klo, me.khi.  True: the tokens to be ordered are in me.all (n of them), the mass to find among
// them in `rest`.  False: they are equal, and the last kept one, as far as this CTA is concerned, is in me.tau_comp.
// (When one CTA took such a row through global memory instead: 64 rows of 128256 equal logits 8.8 ms, so 0.19; of
// deviation 0.05 440 us, so 95; 378 rows of deviation 0.5 1001, so 452.  With fewer tokens in the cut's bin nothing of this
// runs.)
__device__ __noinline__ bool tp_refine(TpFast& me, int rank, int ranks, int lo, int cnt, float M, float c2, float cut_lo, float cut_hi,
                                       unsigned long long& rest, int& n) {
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cnt_all = (cnt + 31) & ~31;
  uint32_t lowest = 0xffffffffu, highest = 0u;
  for (int i = tid; i < cnt; i += kTpThreads) {
    const float x = me.x[i], d = (M - x) * c2, p = d * 51.2f;
    if (p >= cut_lo && p < cut_hi && d < 40.f) { lowest = min(lowest, tp_key(x)); highest = max(highest, tp_key(x)); }
  }
  lowest = __reduce_min_sync(0xffffffffu, lowest);
  highest = __reduce_max_sync(0xffffffffu, highest);
  if (lane < ranks && highest != 0u) {
    atomicMin(&cluster.map_shared_rank(&me, lane)->kmin, lowest);
    atomicMax(&cluster.map_shared_rank(&me, lane)->kmax, highest);
  }
  cluster.sync();  // (also: the lists and bins have been read)
  uint32_t klo = me.kmin, khi = me.kmax;
  uint32_t* limb = me.limb[0];  // [3][512]
  static_assert(2 * kTpBins >= 3 * 512, "the three limbs take the place of the two");
  for (;;) {
    if (tid == 0) me.ncand = 0;
    if (klo != khi) {
      const int shift = max(0, 32 - __clz(khi - klo) - 9);
      for (int i = tid; i < 3 * 512; i += kTpThreads) limb[i] = 0u;
      __syncthreads();
#pragma unroll 1
      for (int i = tid; i < cnt_all; i += kTpThreads) {  // (whole warps)
        const float x = i < cnt ? me.x[i] : -INFINITY;
        const uint32_t key = tp_key(x);
        const bool in = i < cnt && key >= klo && key <= khi;
        const uint32_t who = __ballot_sync(0xffffffffu, in);
        if (who == 0u) continue;
        const int b = in ? (int)((khi - key) >> shift) : 0;
        const unsigned long long w = in ? tp_mass(x, M, c2) : 0ull;
        const uint32_t w0 = (uint32_t)w & 0x3fffu, w1 = (uint32_t)(w >> 14) & 0x3fffu, w2 = (uint32_t)(w >> 28);
        const int first = __shfl_sync(0xffffffffu, b, __ffs(who) - 1);
        if (__all_sync(0xffffffffu, !in || b == first)) {  // one bin: equal logits, or steps wider than the warp's tokens
          const uint32_t s0 = __reduce_add_sync(0xffffffffu, w0), s1 = __reduce_add_sync(0xffffffffu, w1), s2 = __reduce_add_sync(0xffffffffu, w2);
          if (lane < 3) atomicAdd(&limb[512 * lane + first], lane == 0 ? s0 : lane == 1 ? s1 : s2);
        } else if (in) {
          atomicAdd(&limb[b], w0);
          atomicAdd(&limb[512 + b], w1);
          atomicAdd(&limb[1024 + b], w2);
        }
      }
      __syncthreads();
      auto mass_of = [](const TpFast& of, int b) -> unsigned long long {
        const uint32_t* l = of.limb[0];
        return l[b] + ((unsigned long long)l[512 + b] << 14) + ((unsigned long long)l[1024 + b] << 28);
      };
      {
        static_assert(kTpWarps == 16, "one warp for each group of 32 bins");
        const unsigned long long v = tp_warp_sum(mass_of(me, 32 * warp + lane));
        if (lane == 0) me.coarse[warp] = v;
      }
      cluster.sync();
      // the cluster's groups, then the bins of the one that holds the cut (every warp for itself)
      int at = 0;
#pragma unroll 1
      for (int level = 0; level < 2; ++level) {
        if (warp < ranks) {
          const TpFast* other = cluster.map_shared_rank(&me, warp);
          me.stage[warp][lane] = level ? mass_of(*other, 32 * at + lane) : lane < 16 ? other->coarse[lane] : 0ull;
        }
        __syncthreads();
        unsigned long long v = 0;
        for (int r = 0; r < ranks; ++r) v += me.stage[r][lane];
        const unsigned long long incl = tp_warp_scan(v);
        const int hit = max(__ffs(__ballot_sync(0xffffffffu, incl - v < rest && rest <= incl)) - 1, 0);  // (there is one: the masses are exact)
        rest -= __shfl_sync(0xffffffffu, incl - v, hit);
        at = level ? 32 * at + hit : hit;
        __syncthreads();
      }
      khi -= (uint32_t)at << shift;
      klo = max(klo, khi - min(khi, (1u << shift) - 1u));
    } else {
      __syncthreads();
    }
    for (int i = tid; i < cnt; i += kTpThreads) {
      const float x = me.x[i];
      const uint32_t key = tp_key(x);
      if (key < klo || key > khi) continue;
      const int pos = atomicAdd(&me.ncand, 1);
      if (pos < kTpFastCand) me.cand[pos] = make_ulonglong2(((unsigned long long)key << 32) | (uint32_t)~(uint32_t)(lo + i), tp_mass(x, M, c2));
    }
    int before;
    n = tp_gather(me, ranks, rank, before);
    if (tid == 0) { me.klo = klo; me.khi = khi; }
    if (n <= kTpFastCand) return true;
    if (klo == khi) {
      // equal logits share one mass: the first `need` of them in token order are kept, `mine` of them this CTA's
      const float x = __uint_as_float((khi & 0x80000000u) ? khi & 0x7fffffffu : ~khi);
      const unsigned long long each = tp_mass(x, M, c2);
      const unsigned long long need = each ? (rest + each - 1) / each : (unsigned long long)n;
      const int have = me.ncand;
      const int mine = need <= (unsigned long long)before ? 0 : need >= (unsigned long long)before + have ? have : (int)(need - before);
      if (mine > 0 && mine < have) {  // the last of them: runs of an odd length per thread (no bank conflicts), counted and scanned
        const int len = ((cnt + kTpThreads - 1) / kTpThreads) | 1;
        const int i0 = min(tid * len, cnt), i1 = min(i0 + len, cnt);
        unsigned long long own = 0, total;
        for (int i = i0; i < i1; ++i) own += tp_key(me.x[i]) == khi;
        unsigned long long seen = tp_block_scan<kTpThreads>(own, me.part[0], total);
        if (seen < (unsigned long long)mine && (unsigned long long)mine <= seen + own)
          for (int i = i0; i < i1; ++i)
            if (tp_key(me.x[i]) == khi && ++seen == (unsigned long long)mine) {
              me.tau_comp = ((unsigned long long)khi << 32) | (uint32_t)~(uint32_t)(lo + i);
              break;
            }
      } else if (tid == 0) {
        me.tau_comp = mine == have ? (unsigned long long)khi << 32 : ~0ull;
      }
      return false;
    }
    cluster.sync();  // everyone has read the lists and the bins
  }
}

__global__ void __launch_bounds__(kTpThreads, 2) top_p_cluster_kernel(const TopPArgs a, const int slice) {
  extern __shared__ __align__(16) uint8_t tp_smem[];
  TpFast& me = *reinterpret_cast<TpFast*>(tp_smem);
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = blockIdx.x, ranks = gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lo = rank * slice, cnt = max(min(slice, a.V - lo), 0), cnt4 = (cnt + 3) & ~3;
  const float* row = a.logits + (int64_t)blockIdx.y * a.in_stride + lo;
  float* orow = a.out + (int64_t)blockIdx.y * a.out_stride + lo;

  if (tid == 0) { me.ncand = 0; me.tau_comp = 0ull; me.max = tp_ordered(-INFINITY); me.kmin = 0xffffffffu; me.kmax = 0u; }
  __syncthreads();
  cluster.barrier_arrive();  // waited for before the first remote access
  for (int i = tid; i < 2 * kTpBins; i += kTpThreads) me.limb[0][i] = 0u;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int i = 32 * tid; i < cnt; i += 32 * kTpThreads) prefetch_l2(row + i);  // the slice, while the previous kernel ends (64 rows of 32000: 14.4 -> 13.7 us)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (a.kept_out != nullptr && rank == 0 && tid == 0) a.kept_out[blockIdx.y] = 0;  // (the cluster's barriers order it before the counts)

  // ---- the slice (NaN / +inf flagged and read as -inf, padded to groups of four with -inf) and the row maximum
  int bad = 0;
  float m = -INFINITY;
  auto take = [&](int i, float4 v) {
    if (!((v.x + v.y) + (v.z + v.w) < INFINITY)) {  // a NaN or +inf among them (or a sum beyond the largest number)
      v.x = tp_clean(v.x, bad); v.y = tp_clean(v.y, bad); v.z = tp_clean(v.z, bad); v.w = tp_clean(v.w, bad);
    }
    m = fmaxf(fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)), m);
    *reinterpret_cast<float4*>(&me.x[i]) = v;
  };
  constexpr int kDeep = 8, kPass = 4 * kTpThreads;  // eight loads in flight per thread
  const int full = cnt & ~3;
  for (int i0 = 4 * tid; i0 < full; i0 += kDeep * kPass) {
    float4 v[kDeep];
#pragma unroll
    for (int k = 0; k < kDeep; ++k)
      if (i0 + k * kPass < full) v[k] = *reinterpret_cast<const float4*>(row + i0 + k * kPass);
#pragma unroll
    for (int k = 0; k < kDeep; ++k)
      if (i0 + k * kPass < full) take(i0 + k * kPass, v[k]);
  }
  if (full < cnt && tid == 0)  // the row's last tokens
    take(full, make_float4(row[full], full + 1 < cnt ? row[full + 1] : -INFINITY, full + 2 < cnt ? row[full + 2] : -INFINITY, -INFINITY));
  m = warp_max(m);
  if (bad) dev_flag(a.dev_status, SEQ_DEV_NONFINITE);
  cluster.barrier_wait();
  if (lane < ranks) atomicMax(&cluster.map_shared_rank(&me, lane)->max, tp_ordered(m));
  cluster.sync();
  const float M = tp_unordered(me.max);
  if (M == -INFINITY) {  // no token with any mass: nothing to keep
    for (int i = tid; i < cnt; i += kTpThreads) orow[i] = -INFINITY;
    if (rank == 0 && tid == 0) dev_flag(a.dev_status, SEQ_DEV_DEGENERATE);
    return;
  }

  // ---- masses: the sum of all of them (first round), the histogram of the round's bins
  // With d = (M - x) * c2 the exponent argument, a token's bin counted from the most probable is (int)(d * 51.2).
  unsigned long long target = 0, above_round = 0, rest0 = 0;
  int B0 = -1;            // the bin in which the cut falls, and the mass still to find inside it
  bool wrapped = false;
  // Where a bin begins among the logits, to a margin of 4e-6, eight times what the rounding of a bin's number can be off: one
  // comparison tells most tokens off, and only for the others is the bin itself worked out.  (The margin is never 0.)
  auto margin = [&](float x) { return fmaf(4e-6f, fabsf(M) + fabsf(x), 1e-30f); };
  for (int round = 0, bin0 = 0; round < kTpRounds; ++round, bin0 += kTpBins) {
    const float first = (float)bin0, last = fminf(first + (float)kTpBins, 2048.f);
    const float x_last = M - last * a.bin_width, x_first = M - first * a.bin_width;
    const float t_low = x_last - margin(x_last), t_high = x_first + margin(x_first);
    unsigned long long sum = 0;
    uint32_t small = 0;  // tokens behind the first round's bins: below 2^25 each, 32 of them at most
    auto add = [&](float x) {  // a token that may be one of the round's bins
      const float d = (M - x) * a.c2, p = d * 51.2f;
      const unsigned long long w = __float2ull_rn(tp_ex2(-d) * kTpScale);
      if (p >= first && p < last && d < 40.f) {
        const int b = (int)p - bin0;
        sum += w;
        atomicAdd(&me.limb[0][b], (uint32_t)w & 0xfffffu);
        const uint32_t high = (uint32_t)(w >> 20);
        if (high) atomicAdd(&me.limb[1][b], high);
      } else if (round == 0 && d < 40.f) {
        small += (uint32_t)w;
      }
    };
    // The round's tokens wait in a list of the thread's own, so that the lanes of a warp add theirs side by side.
    float* const list = reinterpret_cast<float*>(me.cand) + tid;
    float* end = list;
    // (Two at a time, both loads ahead of the first one's atomics.  512 rows of 128256 at temperature 1.5: 354 us one at a time,
    // 344 so, 341 four at a time, which at 1 is 281 against 277; 3 rows at 1.5 16.9, 16.3 and 16.1, at 1 14.2, 14.0 and 14.2.)
    auto flush = [&]() {
      for (float* t = list; __any_sync(0xffffffffu, t < end); t += 2 * kTpThreads) {
        float x[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) x[k] = t + k * kTpThreads < end ? t[k * kTpThreads] : -INFINITY;
#pragma unroll
        for (int k = 0; k < 2; ++k) add(x[k]);
      }
      end = list;
    };
    auto pass = [&](auto opening) {
#pragma unroll 1
      for (int i0 = 0; i0 < cnt4; i0 += 4 * kTpThreads) {  // (whole warps take part)
        const int i = i0 + 4 * tid;
        const float4 v = i < cnt4 ? *reinterpret_cast<const float4*>(&me.x[i]) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        if (__any_sync(0xffffffffu, end > list + (kTpList - 4) * kTpThreads)) flush();
        const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const bool listed = x[e] >= t_low && (decltype(opening)::value || x[e] < t_high);
          if (decltype(opening)::value) {  // (no branch: the sum is taken of all of them, 0 for those that do not count)
            const float d = (M - x[e]) * a.c2;
            const uint32_t w = __float2uint_rn(tp_ex2(-d) * kTpScale);
            small += !listed && d < 40.f ? w : 0u;
          }
          if (listed) {
            *end = x[e];
            end += kTpThreads;
          }
        }
      }
    };
    if (round == 0) pass(std::true_type()); else pass(std::false_type());
    flush();
    const unsigned long long sum_all = tp_warp_sum(sum + small), sum_round = tp_warp_sum(sum);
    if (lane == 0) { me.part[0][warp] = sum_all; me.part[1][warp] = sum_round; }
    __syncthreads();
    for (int grp = warp; grp < 26; grp += kTpWarps) {
      unsigned long long v;
      if (grp < 24) v = me.limb[0][32 * grp + lane] + ((unsigned long long)me.limb[1][32 * grp + lane] << 20);
      else v = lane < kTpWarps ? me.part[grp - 24][lane] : 0ull;
      v = tp_warp_sum(v);
      if (lane == 0) me.coarse[grp] = v;
    }
    cluster.sync();
    // the cluster's groups: one remote load per thread, then every warp finds the cut's group for itself
    if (warp < ranks && lane < 26) me.stage[warp][lane] = cluster.map_shared_rank(&me, warp)->coarse[lane];
    __syncthreads();
    unsigned long long v = 0;
    if (lane < 26)
      for (int r = 0; r < ranks; ++r) v += me.stage[r][lane];
    const unsigned long long all_mass = __shfl_sync(0xffffffffu, v, 24), exact = __shfl_sync(0xffffffffu, v, 25);
    if (round == 0) {  // the mass the nucleus has to reach (rounded up, at least one unit)
      const double want = ceil(a.top_p * (double)all_mass);
      target = want < 1.0 ? 1ull : (want >= (double)all_mass ? all_mass : (unsigned long long)want);
    }
    if (lane >= 24) v = 0;
    unsigned long long incl = tp_warp_scan(v);
    wrapped = __shfl_sync(0xffffffffu, incl, 31) != exact;
    if (wrapped) break;  // (every warp of every CTA of the cluster sees the same)
    uint32_t hit = __ballot_sync(0xffffffffu, above_round + incl - v < target && target <= above_round + incl);
    __syncthreads();     // the staged groups have been read
    if (hit) {
      const int grp = __ffs(hit) - 1;
      const unsigned long long above = above_round + __shfl_sync(0xffffffffu, incl - v, grp);
      if (warp < ranks) {
        const TpFast* other = cluster.map_shared_rank(&me, warp);
        me.stage[warp][lane] = other->limb[0][32 * grp + lane] + ((unsigned long long)other->limb[1][32 * grp + lane] << 20);
      }
      __syncthreads();
      v = 0;
      for (int r = 0; r < ranks; ++r) v += me.stage[r][lane];
      incl = tp_warp_scan(v);
      hit = __ballot_sync(0xffffffffu, above + incl - v < target && target <= above + incl);
      const int b = __ffs(hit) - 1;
      B0 = bin0 + 32 * grp + b;
      rest0 = target - (above + __shfl_sync(0xffffffffu, incl - v, b));
      break;
    }
    above_round += __shfl_sync(0xffffffffu, incl, 31);
    cluster.sync();  // everyone has read the groups before the bins are cleared
    for (int i = tid; i < 2 * kTpBins; i += kTpThreads) me.limb[0][i] = 0u;
    __syncthreads();
  }
  const bool whole_row = wrapped || B0 < 0;
  const float cut_lo = whole_row ? 4096.f : (float)B0, cut_hi = cut_lo + 1.f;  // (whole row: no token is collected)

  // ---- the tokens of that bin, as (key, ~index) so that a larger value means "earlier in the order".  Every other token
  // is decided by its bin: the logit itself in a more probable one, -inf in a less probable one.  It is written at once,
  // unless the call works in place: the row may still be needed as it was.
  const bool early = row != orow && !whole_row;
  int kept = 0;
  auto decide = [&](float x, int i) -> float {
    const float d = (M - x) * a.c2, p = d * 51.2f;
    if (p >= cut_lo && p < cut_hi && d < 40.f) {
      const int pos = atomicAdd(&me.ncand, 1);
      if (pos < kTpFastCand)
        me.cand[pos] = make_ulonglong2(((unsigned long long)tp_key(x) << 32) | (uint32_t)~(uint32_t)(lo + i), __float2ull_rn(tp_ex2(-d) * kTpScale));
    }
    const bool keep = p < cut_lo;
    kept += keep;
    return keep ? x : -INFINITY;
  };
  auto store = [&](int i, float4 v) {
    if (i + 3 < cnt) {
      *reinterpret_cast<float4*>(orow + i) = v;
    } else {
      orow[i] = v.x;
      if (i + 1 < cnt) orow[i + 1] = v.y;
      if (i + 2 < cnt) orow[i + 2] = v.z;
    }
  };
  // from t_keep on a more probable bin, below t_drop a less probable one
  const float x_lo = M - cut_lo * a.bin_width, x_hi = M - cut_hi * a.bin_width, t_keep = x_lo + margin(x_lo), t_drop = x_hi - margin(x_hi);
#pragma unroll 1
  for (int i = 4 * tid; i < (whole_row ? 0 : cnt4); i += 4 * kTpThreads) {
    float4 v = *reinterpret_cast<const float4*>(&me.x[i]);
    const bool k0 = v.x >= t_keep, k1 = v.y >= t_keep, k2 = v.z >= t_keep, k3 = v.w >= t_keep;
    const float near = fmaxf(fmaxf(k0 ? -INFINITY : v.x, k1 ? -INFINITY : v.y), fmaxf(k2 ? -INFINITY : v.z, k3 ? -INFINITY : v.w));
    if (near >= t_drop) {  // one of the four is in the bin, or so close to it that its own bin has to tell
      v.x = decide(v.x, i); v.y = decide(v.y, i + 1); v.z = decide(v.z, i + 2); v.w = decide(v.w, i + 3);
    } else {
      kept += k0 + k1 + k2 + k3;
      v = make_float4(k0 ? v.x : -INFINITY, k1 ? v.y : -INFINITY, k2 ? v.z : -INFINITY, k3 ? v.w : -INFINITY);
    }
    if (early) store(i, v);
  }
  int before, n = tp_gather(me, ranks, rank, before);  // tokens of the whole cluster
  const bool refine = whole_row || n > kTpFastCand;    // (the same for every CTA)
  unsigned long long rest = whole_row ? target : rest0;
  bool order = true;
  if (refine) order = tp_refine(me, rank, ranks, lo, cnt, M, a.c2, whole_row ? 0.f : cut_lo, whole_row ? INFINITY : cut_hi, rest, n);
  const bool alone = order && n > kTpAlone && ranks > 1;
  if (alone) {
    __syncthreads();
    tp_cut_own(me, n, rest, ranks);
    cluster.sync();
  } else {
    cluster.barrier_arrive();  // waited for at the end: nobody leaves while its list is being read
    __syncthreads();
    if (order) tp_cut<kTpThreads>(me.all, n, rest, &me.tau_comp);
  }
  const unsigned long long tau_comp = me.tau_comp;

  // ---- the tokens of the cut's bin: kept if not behind the last kept one in the order (key descending, index ascending)
  if (refine) {  // ... of the range of keys that is left; all is written (again)
    const uint32_t klo = me.klo, khi = me.khi;
    kept = 0;
    auto inside = [&](float x, int i) -> float {
      const uint32_t key = tp_key(x);
      const unsigned long long comp = ((unsigned long long)key << 32) | (uint32_t)~(uint32_t)(lo + i);
      const bool keep = key > khi || (key >= klo && comp >= tau_comp);
      kept += keep;
      return keep ? x : -INFINITY;
    };
#pragma unroll 1
    for (int i = 4 * tid; i < cnt4; i += 4 * kTpThreads) {
      const float4 v = *reinterpret_cast<const float4*>(&me.x[i]);
      store(i, make_float4(inside(v.x, i), inside(v.y, i + 1), inside(v.z, i + 2), inside(v.w, i + 3)));
    }
  } else if (!early) {
#pragma unroll 1
    for (int i = 4 * tid; i < cnt4; i += 4 * kTpThreads) {
      float4 v = *reinterpret_cast<const float4*>(&me.x[i]);
      auto inside = [&](float x) { return (M - x) * a.c2 * 51.2f < cut_lo ? x : -INFINITY; };
      store(i, make_float4(inside(v.x), inside(v.y), inside(v.z), inside(v.w)));
    }
    __syncthreads();
  }
  for (int j = tid; j < (refine ? 0 : me.ncand); j += kTpThreads)
    if (me.cand[j].x >= tau_comp) {
      const int i = (int)~(uint32_t)me.cand[j].x - lo;
      orow[i] = me.x[i];
      ++kept;
    }
  if (a.kept_out != nullptr) {
    kept = __reduce_add_sync(0xffffffffu, kept);
    if (lane == 0) atomicAdd(a.kept_out + blockIdx.y, kept);
  }
  if (!alone) cluster.barrier_wait();
}

// top_p >= 1: every token stays (rows copied when the call is not in place)
__global__ void top_p_copy_kernel(const TopPArgs a) {
  const float* row = a.logits + (int64_t)blockIdx.x * a.in_stride;
  float* orow = a.out + (int64_t)blockIdx.x * a.out_stride;
  if (row != orow)
    for (int i = threadIdx.x; i < a.V; i += blockDim.x) orow[i] = row[i];
  if (threadIdx.x == 0 && a.kept_out != nullptr) a.kept_out[blockIdx.x] = a.V;
}

// Clusters of `ranks` CTAs, with the largest slice's shared memory, that the device runs at a time.  Asked once per device and
// size; without a device, or where the question fails, what the SMs would hold at two CTAs each.
static int tp_clusters_side_by_side(int ranks) {
  const int all = 2 * device_sm_count() / ranks;
  static int known[kTpMaxCluster + 1][64];  // + 1; 0 = not asked yet
  int dev = 0;
  if (ranks == 1 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return all; }
  int n = __atomic_load_n(&known[ranks][dev], __ATOMIC_ACQUIRE);
  if (n == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ranks);
    cfg.blockDim = dim3(kTpThreads);
    cfg.dynamicSmemBytes = offsetof(TpFast, x) + kTpMaxSlice * 4;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ranks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, top_p_cluster_kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = all;
    }
    ++n;
    __atomic_store_n(&known[ranks][dev], n, __ATOMIC_RELEASE);
  }
  return n - 1;
}

// CTAs per row: as many as let the rows' clusters run side by side (two CTAs per SM), of at least 4096 tokens each and 8 at
// most; at least what keeps a slice within 16384 tokens.  A row of more than 8 x 16384 tokens goes to one CTA.
// What runs side by side is asked of the device, as a cluster lies in one GPC (33, 37, 45, 56, 71 and 93 clusters of 8 to 3 CTAs
// were seen, 2 * 148 / ranks had been assumed), and three places are left free: in a row of calls the next one's clusters
// come in as these leave, and where all places are needed they get between (45 rows of 32000 in clusters of 6: 13.4 us or 17.5
// from one build to the next; in clusters of 5 12.1).  One place where a step down makes the slices a third longer and more
// (70 rows at temperature 1 in clusters of 4 15.1, of 3 16.9).  36 rows of 32000 19.2 -> 11.6 us, 58 20.0 -> 12.3, 98 22.7 -> 16.1, 48 of
// 50257 21.8 -> 13.8; no room for a tenth of the rows: 66 rows at temperature 1 16.9 instead of 14.7.
static int launch_top_p(int rows, const TopPArgs& a, cudaStream_t stream) {
  const int least = (a.V + kTpMaxSlice - 1) / kTpMaxSlice, most = (a.V + 4095) / 4096;
  const bool cluster = least <= kTpMaxCluster;
  int64_t ranks = 2 * (int64_t)device_sm_count() / rows;
  ranks = ranks > most ? most : ranks;
  ranks = ranks > kTpMaxCluster ? kTpMaxCluster : ranks < least ? least : ranks;
  // (the attributes first: the question below asks for the shared memory of the largest slice)
  static int attr_done[64];
  const int rc = once_per_device(attr_done, [&]() -> int {  // above the 48 KB a kernel gets without asking
    SEQ_CUDA_OK(cudaFuncSetAttribute(top_p_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(offsetof(TpFast, x) + kTpMaxSlice * 4)));
    SEQ_CUDA_OK(cudaFuncSetAttribute(top_p_row_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TpShared)));
    return SEQ_OK;
  });
  if (rc != SEQ_OK) return rc;
  while (cluster && ranks > least && tp_clusters_side_by_side((int)ranks) < (int64_t)rows + (ranks > 4 ? 3 : 1)) --ranks;
  const int slice = (int)(((a.V + ranks - 1) / ranks + 3) & ~(int64_t)3);
  const size_t smem = offsetof(TpFast, x) + (size_t)slice * 4;
  if (!cluster) {
    top_p_row_kernel<<<rows, kTpRowThreads, sizeof(TpShared), stream>>>(a);
    SEQ_CUDA_OK(cudaGetLastError());
    return SEQ_OK;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kTpThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)ranks;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // set-up under the previous kernel's tail
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  TopPArgs part = a;
  for (int first = 0; first < rows; first += 65535) {  // (a grid's y extent)
    cfg.gridDim = dim3((unsigned)ranks, rows - first < 65535 ? rows - first : 65535);
    part.logits = a.logits + (int64_t)first * a.in_stride;
    part.out = a.out + (int64_t)first * a.out_stride;
    part.kept_out = a.kept_out != nullptr ? a.kept_out + first : nullptr;
    SEQ_CUDA_OK(cudaLaunchKernelEx(&cfg, top_p_cluster_kernel, part, slice));
  }
  return SEQ_OK;
}

}  // namespace seqtree

using namespace seqtree;

extern "C" int seq_tree_top_p_filter(const seq_tree_top_p_params* p, void* stream) {
  if (p == nullptr || p->logits == nullptr || p->out == nullptr) return SEQ_ERR_INVALID_ARG;
  if (p->n_rows < 1 || p->vocab < 1 || p->vocab > (1 << 22)) return SEQ_ERR_INVALID_ARG;
  if (!(p->temperature > 0.f) || isinf(p->temperature) || !(p->top_p > 0.f)) return SEQ_ERR_INVALID_ARG;
  if (p->logits_row_stride < p->vocab || p->out_row_stride < p->vocab || p->logits_row_stride % 4 != 0 ||
      p->out_row_stride % 4 != 0 || reinterpret_cast<uintptr_t>(p->logits) % 16 != 0 ||
      reinterpret_cast<uintptr_t>(p->out) % 16 != 0)
    return SEQ_ERR_INVALID_ARG;
  TopPArgs a;
  a.logits = p->logits; a.in_stride = p->logits_row_stride;
  a.out = p->out; a.out_stride = p->out_row_stride;
  a.V = p->vocab;
  a.c2 = kLog2e / p->temperature;
  a.bin_width = 1.f / (51.2f * a.c2);
  a.top_p = (double)p->top_p;
  a.kept_out = p->kept_out; a.dev_status = p->dev_status;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (p->top_p >= 1.f)
    top_p_copy_kernel<<<p->n_rows, 256, 0, s>>>(a);
  else
    return launch_top_p(p->n_rows, a, s);
  SEQ_CUDA_OK(cudaGetLastError());
  return SEQ_OK;
}
