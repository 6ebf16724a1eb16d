// GRPO objective of Sec. 3.1 without the KL term (the paper drops it), fused over the tokens of a batch:
//   J = mean_q (1/G_q) sum_{i in q} (1/|o_i|) sum_t min( r_{i,t} A_i , clip(r_{i,t}, 1-eps, 1+eps) A_i ),
//   r_{i,t} = exp(logp_{i,t} - logp_old_{i,t}),
// together with dJ/dlogp per token (what the backward of the vocabulary pass takes as g_logp) and the
// fraction of response tokens whose clipped term is the active one.  The data is a few bytes per token
// (nothing of vocabulary size), so the kernels are latency-bound; they are written for determinism:
// all arithmetic in fp64 (the clip decision compares two products and must not depend on fp32 rounding),
// fixed-order reductions, one CTA per response and a single block for the final sum.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "e3.h"

namespace cg = cooperative_groups;

namespace {

constexpr int kThreads = 256;

struct SeqPartial {
  double J;        // this response's share of the objective, already divided by |o_i| and G_q
  double tokens;   // |o_i|
  double clipped;  // tokens whose clipped term is active
};

// Sums of N values over the block, in a fixed order; every thread gets them.
template <int N>
__device__ __forceinline__ void block_sums(double (&v)[N], double (*sh)[N]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < N; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < N; ++k) sh[warp][k] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < N; ++k) {
    v[k] = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) v[k] += sh[w][k];
  }
}

// What a thread or a warp of a batch adds up: terms of the objective, tokens, clipped tokens (an eighth of a response at most: 32 bits hold
// what fits the device's memory).
struct Sums {
  double terms;
  uint32_t on, clipped;
};
// ... and a block.
struct Totals {
  double terms;
  int64_t on, clipped;
};
__device__ __forceinline__ Sums warp_sums(Sums v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v.terms += __shfl_xor_sync(0xffffffffu, v.terms, o);
  v.on = __reduce_add_sync(0xffffffffu, v.on);
  v.clipped = __reduce_add_sync(0xffffffffu, v.clipped);
  return v;
}
// ... over the block, in a fixed order; every thread gets them.
__device__ __forceinline__ Totals block_sums(const Sums &mine, Sums *sh) {
  const Sums warp = warp_sums(mine);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = warp;
  __syncthreads();
  Totals v = {0.0, 0, 0};
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) {
    v.terms += sh[w].terms;
    v.on += sh[w].on;
    v.clipped += sh[w].clipped;
  }
  return v;
}

struct Token {
  bool clip_active;
  double s1, term;  // r A; the token's term of the objective
};
__device__ __forceinline__ Token token_term(float lp, float lp_old, double A, double clip_lo, double clip_hi) {
  Token k;
  const double r = exp((double)lp - (double)lp_old);
  const double rc = r < clip_lo ? clip_lo : (r > clip_hi ? clip_hi : r);
  const double s2 = rc * A;
  k.s1 = r * A;
  k.clip_active = s2 < k.s1;  // the clipped term is the strictly smaller one: no gradient
  k.term = k.clip_active ? s2 : k.s1;
  return k;
}

// Bound by latency: one round of loads (the first kKeep tokens of every thread at once, the group offsets by all
// threads), one reduction, of which only the objective's terms are fp64 (the counts are exact as integers), one round of stores.  512
// responses of 2,048 tokens: 10.2 us with a binary search by one thread, a pass that counted the mask before the pass over the tokens and
// three reductions one after the other, 8.5 with four fp64 sums in one, now 8.1.
constexpr int kKeep = 8;                       // tokens whose terms a thread keeps in registers: responses of up to 2,048
constexpr int64_t kScanGroups = 8 * kThreads;  // group offsets that the block reads in eight rounds of loads; a search (eleven
                                               // dependent loads and more) beyond

__global__ void __launch_bounds__(kThreads) grpo_seq_kernel(const float *__restrict__ logp,
                                                            const float *__restrict__ logp_old,
                                                            const uint8_t *__restrict__ mask, int64_t seq_len,
                                                            const float *__restrict__ adv,
                                                            const int64_t *__restrict__ off, int64_t n_groups,
                                                            double clip_lo, double clip_hi,
                                                            float *__restrict__ g_out, SeqPartial *__restrict__ part) {
  __shared__ Sums sh[kThreads / 32];
  __shared__ double sh_group;
  if (threadIdx.x == 0) sh_group = 0.0;
  // programmatic dependent launch: the final kernel may be set up while this one runs
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int64_t i = blockIdx.x;
  const int64_t base = i * seq_len;
  Sums sum = {0.0, 0, 0};
  const double A = (double)adv[i];
  float lp[kKeep], lpo[kKeep];
  bool on[kKeep];
#pragma unroll
  for (int k = 0; k < kKeep; ++k) {
    const int64_t t = (int64_t)threadIdx.x + k * kThreads, j = base + t;
    on[k] = t < seq_len && (!mask || mask[j]);
    lp[k] = t < seq_len ? logp[j] : 0.f;
    lpo[k] = t < seq_len ? logp_old[j] : 0.f;
  }
  __syncthreads();
  // group of this response: the q with off[q] <= i < off[q+1]
  if (n_groups <= kScanGroups) {
    for (int64_t q = threadIdx.x; q < n_groups; q += kThreads) {
      const int64_t a = off[q], b = off[q + 1];
      if (a <= i && i < b) sh_group = (double)(b - a);
    }
  } else if (threadIdx.x == 0 && off[0] <= i && i < off[n_groups]) {
    int64_t lo = 0, hi = n_groups;  // invariant: off[lo] <= i, answer in [lo, hi)
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) >> 1;
      if (off[mid] <= i) lo = mid; else hi = mid;
    }
    sh_group = (double)(off[lo + 1] - off[lo]);
  }
  double g[kKeep];  // gradient before the weight
#pragma unroll
  for (int k = 0; k < kKeep; ++k) {
    g[k] = 0.0;
    if (!on[k]) continue;
    const Token x = token_term(lp[k], lpo[k], A, clip_lo, clip_hi);
    sum.on += 1;
    sum.terms += x.term;
    sum.clipped += x.clip_active ? 1 : 0;
    g[k] = x.clip_active ? 0.0 : x.s1;
  }
  // the tokens of a longer response are counted now and evaluated when the weight is known
  const bool longer = seq_len > kKeep * kThreads;
  const int64_t t_rest = (int64_t)threadIdx.x + kKeep * kThreads;
  Sums rest = sum;
  for (int64_t t = t_rest; t < seq_len; t += kThreads) sum.on += (!mask || mask[base + t]) ? 1 : 0;
  Totals total = block_sums(sum, sh);
  const double len = (double)total.on, gq = sh_group;
  const bool counts = len > 0.0 && gq > 0.0;
  const double w = counts ? 1.0 / (len * gq * (double)n_groups) : 0.0;
  if (g_out) {
#pragma unroll
    for (int k = 0; k < kKeep; ++k) {
      const int64_t t = (int64_t)threadIdx.x + k * kThreads;
      if (t < seq_len) g_out[base + t] = on[k] && counts ? (float)(g[k] * w) : 0.f;
    }
  }
  if (longer) {
    __shared__ Sums sh_rest[kThreads / 32];
    for (int64_t t = t_rest; t < seq_len; t += kThreads) {
      const int64_t j = base + t;
      float v = 0.f;
      if (counts && (!mask || mask[j])) {
        const Token x = token_term(logp[j], logp_old[j], A, clip_lo, clip_hi);
        rest.terms += x.term;
        rest.clipped += x.clip_active ? 1 : 0;
        if (!x.clip_active) v = (float)(x.s1 * w);
      }
      if (g_out) g_out[j] = v;
    }
    total = block_sums(rest, sh_rest);
  }
  if (threadIdx.x == 0) {
    part[i].J = counts ? total.terms / (len * gq) : 0.0;
    part[i].tokens = gq > 0.0 ? len : 0.0;
    part[i].clipped = counts ? (double)total.clipped : 0.0;
  }
}

// A short batch in one launch: a warp per response, the blocks of one cluster, whose sums meet in shared memory.  Two launches, the second
// behind the first, take the host 6.4 us whatever there is to do, this one 4.3 (1 x 16 tokens; 100 x 100 4.9).  Longer responses and several
// of them one after the other cost a warp more than that (64 x 512 tokens 10.1 us, 512 x 100 11.3; 128 x 256 6.1, but 5.4 instead of 4.2 in
// a captured graph, where the host has no part in it).
constexpr int kShortThreads = 512;
constexpr int kShortWarps = kShortThreads / 32;
constexpr int kShortCtas = 8;
constexpr int kShortKeep = 4;                    // tokens whose terms a lane keeps in registers: responses of up to 128
constexpr int64_t kShortSeqs = kShortCtas * kShortWarps, kShortLength = 32 * kShortKeep, kShortGroups = 1024;

__global__ void __launch_bounds__(kShortThreads) grpo_short_kernel(const float *__restrict__ logp, const float *__restrict__ logp_old,
                                                                   const uint8_t *__restrict__ mask, int n_seq, int seq_len,
                                                                   const float *__restrict__ adv, const int64_t *__restrict__ off,
                                                                   int n_groups, double clip_lo, double clip_hi,
                                                                   float *__restrict__ g_out, double *__restrict__ out_J,
                                                                   double *__restrict__ out_clip_frac) {
  __shared__ SeqPartial sh[kShortWarps];
  __shared__ SeqPartial part;
  cg::cluster_group cluster = cg::this_cluster();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  SeqPartial total = {0.0, 0.0, 0.0};
  const int i = (int)blockIdx.x * kShortWarps + warp;
  if (i < n_seq) {
    const int base = i * seq_len;
    const double A = (double)adv[i];
    float lp[kShortKeep], lpo[kShortKeep];
    uint32_t on = 0u;
#pragma unroll
    for (int k = 0; k < kShortKeep; ++k) {
      const int t = lane + 32 * k;
      lp[k] = lpo[k] = 0.f;
      if (t < seq_len) {
        on |= (!mask || mask[base + t] ? 1u : 0u) << k;
        lp[k] = logp[base + t];
        lpo[k] = logp_old[base + t];
      }
    }
    int group = 0;
    for (int q = lane; q < n_groups; q += 32) {
      const int64_t a = off[q], b = off[q + 1];
      if (a <= i && i < b) group = (int)(b - a);
    }
    group = __reduce_max_sync(kAll, group);
    Sums sum = {0.0, (uint32_t)__popc(on), 0};
    double g[kShortKeep];  // gradient before the weight
#pragma unroll
    for (int k = 0; k < kShortKeep; ++k) {
      g[k] = 0.0;
      if (!__any_sync(kAll, on >> k & 1u)) continue;
      const Token x = token_term(lp[k], lpo[k], A, clip_lo, clip_hi);
      const bool live = (on >> k & 1u) != 0u;
      sum.terms += live ? x.term : 0.0;
      sum.clipped += live && x.clip_active ? 1 : 0;
      g[k] = x.clip_active ? 0.0 : x.s1;
    }
    sum = warp_sums(sum);
    const double len = (double)sum.on, gq = (double)group;
    const bool counts = sum.on > 0 && group > 0;
    const double w = counts ? 1.0 / (len * gq * (double)n_groups) : 0.0;
    if (g_out) {
#pragma unroll
      for (int k = 0; k < kShortKeep; ++k) {
        const int t = lane + 32 * k;
        if (t < seq_len) g_out[base + t] = counts && (on >> k & 1u) ? (float)(g[k] * w) : 0.f;
      }
    }
    total.J = counts ? sum.terms / (len * gq) : 0.0;
    total.tokens = group > 0 ? len : 0.0;
    total.clipped = counts ? (double)sum.clipped : 0.0;
  }
  if (lane == 0) sh[warp] = total;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int v = 1; v < kShortWarps; ++v) {
      total.J += sh[v].J;
      total.tokens += sh[v].tokens;
      total.clipped += sh[v].clipped;
    }
    part = total;
  }
  if (gridDim.x > 1) cluster.sync();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    for (unsigned r = 1; r < cluster.num_blocks(); ++r) {
      const SeqPartial *q = cluster.map_shared_rank(&part, r);
      total.J += q->J;
      total.tokens += q->tokens;
      total.clipped += q->clipped;
    }
    *out_J = n_groups > 0 ? total.J / (double)n_groups : 0.0;
    if (out_clip_frac) *out_clip_frac = total.tokens > 0.0 ? total.clipped / total.tokens : 0.0;
  }
  if (gridDim.x > 1) cluster.sync();  // the other blocks' shared memory stays until it has been read
}

__global__ void __launch_bounds__(kThreads) grpo_final_kernel(const SeqPartial *__restrict__ part, int64_t n_seq,
                                                              int64_t n_groups, double *__restrict__ out_J,
                                                              double *__restrict__ out_clip_frac) {
  __shared__ double sh[kThreads / 32][3];
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the per-response partials are complete and visible
  double sum[3] = {0.0, 0.0, 0.0};  // shares of the objective, tokens, clipped
  for (int64_t i = threadIdx.x; i < n_seq; i += kThreads) {
    sum[0] += part[i].J;
    sum[1] += part[i].tokens;
    sum[2] += part[i].clipped;
  }
  block_sums(sum, sh);
  if (threadIdx.x == 0) {
    *out_J = n_groups > 0 ? sum[0] / (double)n_groups : 0.0;
    if (out_clip_frac) *out_clip_frac = sum[1] > 0.0 ? sum[2] / sum[1] : 0.0;
  }
}

inline bool misaligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) != 0; }

}  // namespace

namespace e3 {
size_t grpo_workspace_bytes(int64_t n_seq) { return (size_t)(n_seq > 0 ? n_seq : 1) * sizeof(SeqPartial); }
}  // namespace e3

extern "C" e3_status e3_grpo_objective(const float *logp, const float *logp_old, const uint8_t *mask, int64_t n_seq,
                                       int64_t seq_len, const float *adv, const int64_t *group_offsets,
                                       int64_t n_groups, float clip_eps, float *out_g_logp, double *out_objective,
                                       double *out_clip_frac, void *workspace, size_t workspace_bytes, void *stream) {
  if (n_seq < 0 || seq_len < 0 || n_groups < 0 || !(clip_eps >= 0.f) || !out_objective) return E3_ERR_INVALID_ARG;
  if (n_seq > 0 && (!adv || (seq_len > 0 && (!logp || !logp_old)))) return E3_ERR_INVALID_ARG;
  if (n_groups > 0 && !group_offsets) return E3_ERR_INVALID_ARG;
  if (n_seq >= (int64_t(1) << 31)) return E3_ERR_INVALID_ARG;
  if (misaligned(logp, 4) || misaligned(logp_old, 4) || misaligned(adv, 4) || misaligned(group_offsets, 8) ||
      misaligned(out_g_logp, 4) || misaligned(out_objective, 8) || misaligned(out_clip_frac, 8) || misaligned(workspace, 8))
    return E3_ERR_ALIGNMENT;
  if (!workspace || workspace_bytes < e3::grpo_workspace_bytes(n_seq)) return E3_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  SeqPartial *part = static_cast<SeqPartial *>(workspace);
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (n_seq <= kShortSeqs && n_groups <= kShortGroups && seq_len <= kShortLength) {
    const int64_t ctas = n_seq <= kShortWarps ? 1 : (n_seq + kShortWarps - 1) / kShortWarps;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)ctas;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kShortThreads);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, grpo_short_kernel, logp, logp_old, mask, (int)n_seq, (int)seq_len, adv, group_offsets,
                                             (int)n_groups, 1.0 - (double)clip_eps, 1.0 + (double)clip_eps, out_g_logp, out_objective, out_clip_frac);
    return e == cudaSuccess ? E3_OK : E3_ERR_CUDA;
  }
  cfg.blockDim = dim3(kThreads);
  if (n_seq > 0) {
    cfg.gridDim = dim3((unsigned)n_seq);
    if (cudaLaunchKernelEx(&cfg, grpo_seq_kernel, logp, logp_old, mask, seq_len, adv, group_offsets, n_groups,
                           1.0 - (double)clip_eps, 1.0 + (double)clip_eps, out_g_logp, part) != cudaSuccess)
      return E3_ERR_CUDA;
  }
  cfg.gridDim = dim3(1);
  if (cudaLaunchKernelEx(&cfg, grpo_final_kernel, (const SeqPartial *)part, n_seq, n_groups, out_objective,
                         out_clip_frac) != cudaSuccess)
    return E3_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? E3_OK : E3_ERR_CUDA;
}
