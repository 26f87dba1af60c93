// seq_tree_draft_sample: the draft side's draw of a node's children, k tokens without replacement from
// softmax(logits / T), by exponential sort (Section 5, "Implementation Details": the exponential-sort
// algorithm; the draw s_i ~ D of Algorithm 2's loop, for all children of a node at once).
//
// Token t gets the key E_t / q_t with E_t = -log(u_t); ascending keys are the draw order.  The kernels work
// with the logarithm of the inverse key, logit_t / T - log(-log u_t) (the softmax normaliser is the same for
// every token of a row and drops out), and take the k largest in descending order, ties to the lower
// token.  No pass for a maximum or a sum is needed: a row is read once.
//
// One CTA takes a part of a row - all of it when there are enough rows - in steps of 4096 tokens, the next step's loads in
// flight while one is worked on.  Almost every token only has to be shown to be out of the running, and for that an upper
// bound of its score will do: -log u >= 1 - u, so score <= logit/T - log(1 - u), one logarithm and a handful of
// instructions, tight where the winners are (u near 1).  The first step finds a threshold that k tokens are known to reach
// (each thread scores the token with its best bound; the k-th largest of the bests of 64 or 128 groups of threads); after
// that only tokens whose bound passes the threshold are listed.  Whenever the steps done have doubled (about k tokens pass
// in that time), and at the end, the listed tokens are scored and ranked against each other, the k best stay and the
// threshold becomes the k-th score itself.  A list that overflows (long runs of equal scores, rows in ascending order) leaves
// the rest of the part to k block-wide arg-max rounds per step.  The parts of a row are a thread-block cluster (up to 8): each pushes its k best into
// the first CTA's shared memory, which ranks them in the same way.  No workspace, one launch.
//
// What bounds it: the two streams of logits and uniforms from HBM.  378 rows of 128256 tokens, k = 9: k block-wide arg-max
// rounds per 4096 tokens and two logarithms and a series per token took 213 us; this takes 62 (95 % of the copy
// bandwidth of 6.55 TB/s; k = 32: 72).  A few short rows are bound by the chain of steps, rankings and the cluster: 5 us.
#include <cooperative_groups.h>
#include <float.h>
#include <limits.h>
#include <math.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace seqtree {

constexpr int kDsThreads = 256;
constexpr int kDsWarps = kDsThreads / 32;
constexpr int kDsMaxK = 64;
constexpr int kDsStep = 4096;            // tokens per step of a CTA
constexpr int kDsE = kDsStep / kDsThreads;  // 16 per thread
constexpr int kDsList = 1024;            // tokens in the running
constexpr int kDsMaxParts = 8;           // CTAs per row: a portable cluster

struct DraftSampleArgs {
  int32_t n_rows, V, k, parts, part_tokens;  // part_tokens: a multiple of the step
  int32_t early;                             // the next kernel is let in at the start (see ds_early), not behind the last step
  const float* logits; int64_t logits_stride;
  const float* uniforms; int64_t uniforms_stride;
  float inv_T;
  int32_t* out;
  int32_t* dev_status;
};

// -log(u) for u in (0, 1) with a relative error of a few 1e-7 everywhere.  The winners of a draw are the
// tokens with SMALL -log u, where the fast logarithm's absolute error (2^-21 near 1) would be a large relative
// one: there -log u = 2 atanh((1 - u) / (1 + u)) is summed as a series (z <= 1/3, seven terms); below 0.5 the
// fast logarithm is good to 3 ulp.
__device__ __forceinline__ float ds_neg_log(float u) {
  if (u < 0.5f) return -__logf(u);
  const float z = __fdividef(1.f - u, 1.f + u), z2 = z * z;
  float p = fmaf(z2, 1.f / 13.f, 1.f / 11.f);
  p = fmaf(p, z2, 1.f / 9.f);
  p = fmaf(p, z2, 1.f / 7.f);
  p = fmaf(p, z2, 1.f / 5.f);
  p = fmaf(p, z2, 1.f / 3.f);
  p = fmaf(p, z2, 1.f);
  return 2.f * z * p;
}
// log of the inverse key, up to the row's constant; -inf = no chance (probability 0, or a uniform outside (0,1))
__device__ __forceinline__ float ds_score(float logit, float u, float inv_T, bool& bad) {
  if (!(logit < INFINITY)) { bad = true; return -INFINITY; }  // NaN or +inf logit: flagged, never drawn
  if (!(u > 0.f && u < 1.f)) return -INFINITY;
  return logit * inv_T - __logf(ds_neg_log(u));
}

// float -> int of the same order
__device__ __forceinline__ int ds_ordered(float x) { const int b = __float_as_int(x); return b ^ ((b >> 31) & 0x7fffffff); }

struct DsShared {
  float2 list[kDsList];  // (score, token bits); behind the ranked ones, tokens not scored yet
  __align__(16) float top[128];  // the first step's group maxima
  float2 cand[kDsMaxParts * kDsMaxK];  // the first CTA of a cluster: every part's k best, in order
  float tau;             // a score that k tokens reach, -inf before there are k
  int count;
};

// Ranks the first `count` entries of the list against each other - larger score first, then lower token -, leaves the k
// best in order at its front, their number in sh.count and, once there are k, the last one's score in sh.tau.  Entries
// without a chance (-inf) drop out.  All threads call it after a barrier behind the last write to the list.  The number is
// also returned: a thread that read sh.count afterwards could find what a warp ahead of it has listed since.
__device__ __forceinline__ int ds_compact(DsShared& sh, int count, int k) {
  const int tid = threadIdx.x;
  if (count <= kDsThreads / 2) {
    // a short list: two, four or eight threads share an entry's comparisons
    const int share = count <= kDsThreads / 8 ? 8 : count <= kDsThreads / 4 ? 4 : 2;
    const int j = tid / share;
    float2 mine = make_float2(-INFINITY, 0.f);
    int rank = 0;
    if (j < count) mine = sh.list[j];
    const bool live = mine.x > -INFINITY;
    const int mi = __float_as_int(mine.y);
    for (int o = tid % share; o < count; o += share) {
      const float2 x = sh.list[o];
      rank += x.x > mine.x || (x.x == mine.x && __float_as_int(x.y) < mi);
    }
    for (int d = 1; d < share; d <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, d);
    const int total = __syncthreads_count(live && tid % share == 0);  // (also: everyone has read the list)
    if (live && tid % share == 0 && rank < k) {
      sh.list[rank] = mine;
      if (rank == k - 1) sh.tau = mine.x;
    }
    if (tid == 0) sh.count = min(total, k);
    __syncthreads();
    return min(total, k);
  }
  float2 mine[kDsList / kDsThreads];
  int rank[kDsList / kDsThreads];
  int live = 0;
#pragma unroll
  for (int q = 0; q < kDsList / kDsThreads; ++q) {
    const int j = tid + q * kDsThreads;
    rank[q] = k;
    if (j >= count) continue;
    mine[q] = sh.list[j];
    if (!(mine[q].x > -INFINITY)) continue;
    ++live;
    const int mi = __float_as_int(mine[q].y);
    int r = 0;
#pragma unroll 4
    for (int o = 0; o < count; ++o) {
      const float2 x = sh.list[o];
      r += x.x > mine[q].x || (x.x == mine[q].x && __float_as_int(x.y) < mi);
    }
    rank[q] = r;
  }
  int total = __syncthreads_count(live > 0);  // (also: everyone has read the list)
  if (count > kDsThreads)
    for (int extra = 2; extra <= kDsList / kDsThreads; ++extra) total += __syncthreads_count(live >= extra);
#pragma unroll
  for (int q = 0; q < kDsList / kDsThreads; ++q)
    if (rank[q] < k) {
      sh.list[rank[q]] = mine[q];
      if (rank[q] == k - 1) sh.tau = mine[q].x;
    }
  if (tid == 0) sh.count = min(total, k);
  __syncthreads();
  return min(total, k);
}

// The bound a token has to pass: the threshold less what the bounds' rounding may cost (31 ulp of place in the first step,
// a few ulp of the approximations: below 4e-6 of it at every magnitude).
__device__ __forceinline__ float ds_cut(float tau) { return fminf(tau - 1e-3f - 1e-5f * fminf(fabsf(tau), 3e38f), 3e38f); }

template <bool kVec>
__global__ void __launch_bounds__(kDsThreads) draft_sample_kernel(const DraftSampleArgs a) {
  __shared__ DsShared sh;
  const int part = blockIdx.x, row = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (a.parts > 1) cg::this_cluster().barrier_arrive();  // waited for before the first remote store
  const int lo = part * a.part_tokens, cnt = min(a.part_tokens, a.V - lo);
  const float* lrow = a.logits + (int64_t)row * a.logits_stride + lo;
  const float* urow = a.uniforms + (int64_t)row * a.uniforms_stride + lo;
  // While the previous kernel ends this one asks for its first two steps, a line of 32 tokens a thread: call after call, 378 rows x
  // 50257 31.9 -> 31.9 us, 37 x 128256 15.5 -> 13.8, 23 x 50257 9.2 -> 8.1, 1 x 32000 5.97 -> 5.87 (k = 9).
  if (a.early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (32 * tid < cnt) {
    prefetch_l2(lrow + 32 * tid);
    prefetch_l2(urow + 32 * tid);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // a thread's tokens of a step: groups of four consecutive ones (kVec), else every 256th
  auto token_of = [&](int t0, int e) { return t0 + (kVec ? 4 * (tid + kDsThreads * (e >> 2)) + (e & 3) : tid + kDsThreads * e); };
  float x[kDsE], u[kDsE];
  auto fetch = [&](int t0) {  // tokens past the part: no chance
    if (kVec) {
#pragma unroll
      for (int j = 0; j < kDsE / 4; ++j) {
        const int t = token_of(t0, 4 * j);
        const bool in = t < cnt;  // (cnt is a multiple of 4 here)
        const float4 xv = in ? __ldg(reinterpret_cast<const float4*>(lrow + t)) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        const float4 uv = in ? __ldg(reinterpret_cast<const float4*>(urow + t)) : make_float4(0.5f, 0.5f, 0.5f, 0.5f);
        x[4 * j] = xv.x; x[4 * j + 1] = xv.y; x[4 * j + 2] = xv.z; x[4 * j + 3] = xv.w;
        u[4 * j] = uv.x; u[4 * j + 1] = uv.y; u[4 * j + 2] = uv.z; u[4 * j + 3] = uv.w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < kDsE; ++e) {
        const int t = token_of(t0, e);
        x[e] = t < cnt ? __ldg(lrow + t) : -INFINITY;
        u[e] = t < cnt ? __ldg(urow + t) : 0.5f;
      }
    }
  };
  bool bad = false, unused = false;
  // The bounds of the fetched tokens into ub, their largest returned.  A bound that is not a number stands for "look at the score".
  float ub[kDsE];
  auto bounds = [&](bool place) -> float {
    float best = -INFINITY;
#pragma unroll
    for (int e = 0; e < kDsE; ++e) {
      bad |= !(x[e] < INFINITY);  // NaN or +inf logit: flagged, never drawn
      float b = fminf(fmaf(__log2f(1.f - u[e]), -kLn2, x[e] * a.inv_T), FLT_MAX);
      if (place && b > -INFINITY) b = __uint_as_float((__float_as_uint(b) & ~31u) | (uint32_t)e);  // the token's place in the lowest bits
      ub[e] = b;
      best = fmaxf(best, b);
    }
    return best;
  };
  auto list_passing = [&](int t0, float cut) {
#pragma unroll
    for (int e = 0; e < kDsE; ++e)
      if (ub[e] > cut) {
        const int pos = atomicAdd(&sh.count, 1);
        if (pos < kDsList) sh.list[pos].y = __int_as_float(token_of(t0, e));
      }
  };

  // ---- first step: the threshold
  fetch(0);
  {
    const float best = bounds(true);
    fetch(kDsStep);
    float top = -INFINITY;
    if (best > -INFINITY) {
      const int t = token_of(0, (int)(__float_as_uint(best) & 31u) % kDsE);
      if (t < cnt) top = ds_score(lrow[t], urow[t], a.inv_T, unused);
    }
    const int share = a.k > 16 ? 2 : 4, groups = kDsThreads / share;
    top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 1));
    if (share == 4) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 2));
    if (tid % share == 0) sh.top[tid / share] = top;
    if (tid == 0) { sh.tau = -INFINITY; sh.count = 0; }
    __syncthreads();
    if (tid < groups) {
      const float mine = sh.top[tid];
      int above = 0, reach = 0;
#pragma unroll 8
      for (int o = 0; o < groups; o += 4) {
        const float4 v = *reinterpret_cast<const float4*>(&sh.top[o]);
        above += (v.x > mine) + (v.y > mine) + (v.z > mine) + (v.w > mine);
        reach += (v.x >= mine) + (v.y >= mine) + (v.z >= mine) + (v.w >= mine);
      }
      if (above < a.k && a.k <= reach) sh.tau = mine;  // (equal ones write the same value)
    }
    __syncthreads();
  }
  float cut = ds_cut(sh.tau);
  list_passing(0, cut);

  // ---- the other steps: bounds against the threshold, a ranking every few of them
  int ranked = 0;  // entries at the list's front that carry their score: the best of the tokens before `next`
  int next = 0;
  bool overflow = false;
  auto rank_list = [&](int seen) {
    __syncthreads();
    const int count = sh.count;
    overflow |= count > kDsList;
    if (overflow) return;
    for (int j = ranked + tid; j < count; j += kDsThreads) {
      const int t = __float_as_int(sh.list[j].y);
      sh.list[j].x = ds_score(lrow[t], urow[t], a.inv_T, unused);
    }
    __syncthreads();
    ranked = ds_compact(sh, count, a.k);
    next = seen;
    cut = ds_cut(sh.tau);
  };
  for (int t0 = kDsStep, step = 1; t0 < cnt; t0 += kDsStep, ++step) {
    const float best = bounds(false);
    if (t0 + kDsStep < cnt) fetch(t0 + kDsStep);
    if (best > cut) list_passing(t0, cut);
    if ((step & (step + 1)) == 0) {
      rank_list(t0 + kDsStep);
      if (overflow) break;
    }
  }
  if (!overflow) rank_list(cnt);
  if (overflow) {
    // Too many tokens in the running.  From the first step that is not ranked on, the step's k best are found by k arg-max
    // rounds - each thread keeps its scores and its best, whoever loses the best looks for the next one - and ranked
    // with those of the steps before.  A token has to beat the k-th of those: an equal one comes later in the order.  (378
    // rows of 128256 equal or ascending tokens, k = 9: 130 and 241 us; ranking 256 tokens at a time took 10 ms.)
    int2* w_best = reinterpret_cast<int2*>(sh.top);  // [2][kDsWarps], used in turn
    int turn = 0;
    if (ranked < a.k && tid == 0) sh.tau = -INFINITY;
    __syncthreads();
    fetch(next);
    for (int t0 = next; t0 < cnt; t0 += kDsStep) {
      const float tau = sh.tau;
      float best = -INFINITY;
      int at = 0;
#pragma unroll
      for (int e = 0; e < kDsE; ++e) {
        const float s = ds_score(x[e], u[e], a.inv_T, bad);
        ub[e] = s > tau ? s : -INFINITY;
        if (ub[e] > best) { best = ub[e]; at = e; }
      }
      if (t0 + kDsStep < cnt) fetch(t0 + kDsStep);
      int found = 0;
      for (; found < a.k; ++found, ++turn) {
        const bool any = best > -INFINITY;
        const int mine = token_of(t0, at);
        auto argmax = [](int key, int token) {  // over the warp: the larger key, then the lower token
          const int m = __reduce_max_sync(0xffffffffu, key);
          return make_int2(m, __reduce_min_sync(0xffffffffu, key == m ? token : INT_MAX));
        };
        int2 w = argmax(any ? ds_ordered(best) : INT_MIN, any ? mine : INT_MAX);
        if (lane == 0) w_best[(turn & 1) * kDsWarps + warp] = w;
        __syncthreads();
        w = w_best[(turn & 1) * kDsWarps + lane % kDsWarps];
        w = argmax(w.x, w.y);
        if (w.y == INT_MAX) break;
        if (any && mine == w.y) {
          sh.list[ranked + found] = make_float2(best, __int_as_float(mine));
          best = -INFINITY;
          const int gone = at;
#pragma unroll
          for (int e = 0; e < kDsE; ++e) {
            if (e == gone) ub[e] = -INFINITY;
            if (ub[e] > best) { best = ub[e]; at = e; }
          }
        }
      }
      ++turn;  // (the round that ended the step read one of the two as well)
      if (found > 0) {
        __syncthreads();
        ranked = ds_compact(sh, ranked + found, a.k);
      }
    }
  }
  if (bad) dev_flag(a.dev_status, SEQ_DEV_NONFINITE);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (nothing to it if the next kernel has been let in)
  int have = ranked;
  if (a.parts > 1) {
    cg::this_cluster().barrier_wait();  // the first CTA runs: its shared memory may be written
    float2* to = cg::this_cluster().map_shared_rank(sh.cand, 0) + part * a.k;
    for (int j = tid; j < a.k; j += kDsThreads) {
      const float2 e = j < have ? sh.list[j] : make_float2(-INFINITY, 0.f);
      to[j] = make_float2(e.x, __int_as_float(lo + __float_as_int(e.y)));
    }
    cg::this_cluster().sync();
    if (part != 0) return;
    // Threshold: warp w looks at the d-th candidate of every part, d = 2^w and k at last; the ceil(k / d)-th largest of
    // them is reached by d candidates of each of ceil(k / d) parts, hence by k.  The largest such bound lets few more than
    // k pass, however the row's best spread over the parts.
    float kth = -INFINITY;
    if (warp < 7) {
      const int d = min(1 << warp, a.k), need = (a.k + d - 1) / d;
      const float mine = lane < a.parts ? sh.cand[lane * a.k + d - 1].x : -INFINITY;
      int above = 0, reach = 0;
#pragma unroll
      for (int o = 0; o < kDsMaxParts; ++o) {
        const float v = __shfl_sync(0xffffffffu, mine, o);
        above += v > mine;
        reach += v >= mine;
      }
      kth = warp_max(lane < a.parts && above < need && need <= reach ? mine : -INFINITY);
    }
    if (tid == 0) sh.count = 0;
    if (lane == 0) sh.top[warp] = kth;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kDsWarps; ++w) kth = fmaxf(kth, sh.top[w]);
    for (int j = tid; j < a.parts * a.k; j += kDsThreads) {
      const float2 c = sh.cand[j];
      if (c.x > -INFINITY && c.x >= kth) sh.list[atomicAdd(&sh.count, 1)] = c;
    }
    __syncthreads();
    const int count = sh.count;
    __syncthreads();
    have = ds_compact(sh, count, a.k);
  }
  for (int j = tid; j < a.k; j += kDsThreads) a.out[(int64_t)row * a.k + j] = j < have ? __float_as_int(sh.list[j].y) : -1;
}

}  // namespace seqtree

using namespace seqtree;

// Parts per row: as many as give every SM three CTAs (about what its memory pipeline needs in flight), of at least one
// step each, eight at most (the CTAs of a row are a portable cluster).
static int ds_part_tokens(const seq_tree_draft_sample_params* p) {
  const int steps = (p->vocab + kDsStep - 1) / kDsStep;
  const int want = (int)(((int64_t)device_sm_count() * 3 + p->n_rows / 2) / p->n_rows);
  const int most = steps < kDsMaxParts ? steps : kDsMaxParts;
  const int parts = want < 1 ? 1 : want > most ? most : want;
  return (steps + parts - 1) / parts * kDsStep;
}
static int ds_parts(const seq_tree_draft_sample_params* p) { return (p->vocab + ds_part_tokens(p) - 1) / ds_part_tokens(p); }

// Whether the next kernel in the stream (which waits before it reads) may be scheduled as soon as every CTA of this one runs,
// its own first steps then asked for while these CTAs still work: 378 rows x 128256 64.9 -> 63.0 us, 378 x 50257 31.9 -> 30.3,
// 200 x 32000 16.0 -> 14.8, 84 x 32000 10.4 -> 9.4 (k = 9).  Its CTAs take what places are free, so that they start unevenly over
// the SMs; what that costs shows
// - where the SMs are far from full, below 1.75 CTAs each (17 rows x 128256, k = 24: 16.9 us, let in early 19.7);
// - where a launch in clusters of 3, 5, 6 or 7 just fits at three CTAs an SM, 2.63 to 2.9 each (80 rows x 50257, 5 CTAs each:
//   15.7 and 18.1; 136 x 128256, 3 each: 34.5 and 39.2; 69 x 128256, 6 each: 21.4 and 23.1).
// Against the kernel that neither let in early nor asked ahead, over 2 to 420 rows of 32000, 50257 and 128256 tokens at k = 2, 9
// and 24, calls are 8 % faster on the average and 3 % slower at worst (241 rows x 50257, where a second wave begins).
static bool ds_early(int ctas, int parts) {
  const int sms = device_sm_count();
  const bool just_fits = 100 * ctas > 263 * sms && 10 * ctas <= 29 * sms;
  return 4 * ctas >= 7 * sms && !(just_fits && (parts & (parts - 1)) != 0);
}

static int ds_validate(const seq_tree_draft_sample_params* p) {
  if (p == nullptr || p->draft_logits == nullptr || p->uniforms == nullptr || p->tokens_out == nullptr)
    return SEQ_ERR_INVALID_ARG;
  if (p->n_rows < 1 || p->n_rows > 65535 || p->vocab < 1 || p->k < 1 || p->k > kDsMaxK) return SEQ_ERR_INVALID_ARG;
  if (p->logits_row_stride < p->vocab || p->uniforms_row_stride < p->vocab) return SEQ_ERR_INVALID_ARG;
  if (!(p->temperature > 0.f) || isinf(p->temperature)) return SEQ_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(p->draft_logits) % 4 != 0 || reinterpret_cast<uintptr_t>(p->uniforms) % 4 != 0)
    return SEQ_ERR_INVALID_ARG;
  return SEQ_OK;
}

extern "C" size_t seq_tree_draft_sample_workspace_bytes(const seq_tree_draft_sample_params* p) {
  (void)p;
  return 0;  // the candidates of a row's parts meet in shared memory
}

extern "C" int seq_tree_draft_sample(const seq_tree_draft_sample_params* p, void* stream) {
  const int rc = ds_validate(p);
  if (rc != SEQ_OK) return rc;
  if ((int64_t)(p->vocab + kDsStep - 1) / kDsStep * p->k > 25600) return SEQ_ERR_UNSUPPORTED;  // vocabularies beyond 1.6 M tokens at k = 64
  const int parts = ds_parts(p);
  DraftSampleArgs a;
  a.n_rows = p->n_rows; a.V = p->vocab; a.k = p->k; a.parts = parts; a.part_tokens = ds_part_tokens(p);
  a.early = ds_early((int)(parts * (p->n_rows < 4096 ? p->n_rows : 4096)), parts);  // (more rows: beyond either line)
  a.logits = p->draft_logits; a.logits_stride = p->logits_row_stride;
  a.uniforms = p->uniforms; a.uniforms_stride = p->uniforms_row_stride;
  a.inv_T = 1.f / p->temperature;
  a.out = p->tokens_out;
  a.dev_status = p->dev_status;
  // a part starts at a multiple of 4096 tokens, so 16-byte alignment of the rows carries over to the parts
  const bool vec = reinterpret_cast<uintptr_t>(p->draft_logits) % 16 == 0 && reinterpret_cast<uintptr_t>(p->uniforms) % 16 == 0 &&
             p->logits_row_stride % 4 == 0 && p->uniforms_row_stride % 4 == 0 && p->vocab % 4 == 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(parts, p->n_rows);
  cfg.blockDim = dim3(kDsThreads);
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = parts;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // scheduled under the tail of the launch before
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  SEQ_CUDA_OK(vec ? cudaLaunchKernelEx(&cfg, draft_sample_kernel<true>, a) : cudaLaunchKernelEx(&cfg, draft_sample_kernel<false>, a));
  return SEQ_OK;
}
