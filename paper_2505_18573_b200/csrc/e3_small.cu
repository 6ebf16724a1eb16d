// The small device steps: masked mean entropy (Sec. 4.2, H_t), its per-sequence reading and the group-relative
// advantage (Eq. "adv").  They are bound by launches and memory latency, not by bandwidth, and written for determinism
// (fixed summation order, fp64 accumulation).
#include "e3_small.cuh"

#include <cooperative_groups.h>
#include <math_constants.h>

#include "e3_internal.h"

namespace cg = cooperative_groups;

namespace e3 {
namespace {

constexpr int kMeanThreads = 256;
// Up to 8 x 32,768 tokens the mean is one launch: a cluster of up to eight CTAs whose partial sums meet in shared memory
// (131,072 tokens: the two launches cost the host 2 us more and the GPU a second launch latency).  Larger inputs
// want more SMs than a portable cluster has: there many blocks write partials and a second kernel adds them.
constexpr int kClusterThreads = 1024;
constexpr int kClusterMost = 8;
constexpr int64_t kClusterTokens = 32768;  // most tokens of a CTA

struct MeanPartial {
  double sum;
  double cnt;
};

__device__ __forceinline__ void block_reduce_2(double &a, double &b, double *sh /* [2*warps] */) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (lane == 0) { sh[2 * warp] = a; sh[2 * warp + 1] = b; }
  __syncthreads();
  if (warp == 0) {
    a = lane < nw ? sh[2 * lane] : 0.0;
    b = lane < nw ? sh[2 * lane + 1] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
  }
}

// Sum and count over the block, in a fixed order; the first warp gets them.
__device__ __forceinline__ void block_sum_count(double &a, int &n, MeanPartial *sh /* [warps] */) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  n = __reduce_add_sync(0xffffffffu, n);
  if (lane == 0) { sh[warp].sum = a; sh[warp].cnt = (double)n; }
  __syncthreads();
  if (warp == 0) {
    a = lane < nw ? sh[lane].sum : 0.0;
    n = lane < nw ? (int)sh[lane].cnt : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    n = __reduce_add_sync(0xffffffffu, n);
  }
}

// Both stages may be launched with programmatic stream serialization behind the kernel that writes `ent`:
// they wait for it (and for its writes) before they touch memory.  Without that launch attribute the wait
// returns at once.
__device__ __forceinline__ void wait_for_stream_predecessor() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Adds the unmasked tokens of [lo, hi) into the thread's sums; lo is a multiple of 4 and thread t takes tokens 4 (t + k T) ... + 3,
// so that the order of the sums does not depend on the alignment of the arrays.  Four 16-byte loads are in flight at a time.
template <int T>
__device__ __forceinline__ void add_tokens(const float *__restrict__ ent, const uint8_t *__restrict__ mask, int64_t lo, int64_t hi,
                                           double &s, int &count) {
  const bool vec = (reinterpret_cast<uintptr_t>(ent) & 15u) == 0 && (reinterpret_cast<uintptr_t>(mask) & 3u) == 0;
  for (int64_t v0 = lo / 4 + threadIdx.x; 4 * v0 < hi; v0 += 4 * T) {
    float e[4][4];
    uint32_t m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t j = 4 * (v0 + k * T);
      m[k] = 0u;
      if (vec && j + 4 <= hi) {
        const float4 q = __ldg(reinterpret_cast<const float4 *>(ent + j));
        e[k][0] = q.x; e[k][1] = q.y; e[k][2] = q.z; e[k][3] = q.w;
        m[k] = mask ? __ldg(reinterpret_cast<const uint32_t *>(mask + j)) : 0x01010101u;
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (j + i < hi) {
            e[k][i] = __ldg(ent + j + i);
            m[k] |= (mask ? (uint32_t)__ldg(mask + j + i) : 1u) << (8 * i);
          }
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if ((m[k] >> (8 * i)) & 0xFFu) {
          s += (double)e[k][i];
          ++count;
        }
  }
}

// Counts are integers (one instruction per warp where a shuffled fp64 sum takes ten), and one CTA alone meets nobody: a call for 64 tokens
// 2.6 us before and 1.8 now, 4,096 tokens 3.6 and 2.7, 131,072 tokens 3.8 and 3.5.
// The whole mean in one launch: CTA r of the cluster adds its tokens, the first one adds the CTAs' sums in rank order.
__global__ void __launch_bounds__(kClusterThreads) mean_cluster_kernel(const float *__restrict__ ent,
                                                                       const uint8_t *__restrict__ mask, int64_t n, int64_t chunk,
                                                                       double *__restrict__ out_mean, double *__restrict__ out_count,
                                                                       int want_sum) {
  __shared__ MeanPartial sh[kClusterThreads / 32];
  __shared__ MeanPartial part;
  cg::cluster_group cluster = cg::this_cluster();
  wait_for_stream_predecessor();
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = lo + chunk < n ? lo + chunk : n;
  double s = 0.0;
  int count = 0;
  add_tokens<kClusterThreads>(ent, mask, lo, hi, s, count);
  block_sum_count(s, count, sh);
  double c = (double)count;
  if (gridDim.x > 1) {
    if (threadIdx.x == 0) { part.sum = s; part.cnt = c; }
    cluster.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      s = c = 0.0;
      for (unsigned r = 0; r < cluster.num_blocks(); ++r) {
        const MeanPartial *q = cluster.map_shared_rank(&part, r);
        s += q->sum;
        c += q->cnt;
      }
    }
    cluster.sync();  // the other CTAs' shared memory stays until it has been read
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *out_mean = want_sum ? s : (c > 0.0 ? s / c : CUDART_NAN);
    *out_count = c;
  }
}

// Larger inputs, stage 1: block b sums tokens [b*chunk, (b+1)*chunk) in a fixed order and stores one partial.
__global__ void __launch_bounds__(kMeanThreads) mean_partial_kernel(const float *__restrict__ ent,
                                                                    const uint8_t *__restrict__ mask, int64_t n,
                                                                    int64_t chunk, MeanPartial *__restrict__ part) {
  __shared__ MeanPartial sh[kMeanThreads / 32];
  wait_for_stream_predecessor();
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = lo + chunk < n ? lo + chunk : n;
  double s = 0.0;
  int count = 0;
  add_tokens<kMeanThreads>(ent, mask, lo, hi, s, count);
  block_sum_count(s, count, sh);
  if (threadIdx.x == 0) { part[blockIdx.x].sum = s; part[blockIdx.x].cnt = (double)count; }
}

// Stage 2: one block adds the partials in index order and writes mean (or, with want_sum, the sum) and count.
__global__ void __launch_bounds__(kMeanThreads) mean_final_kernel(const MeanPartial *__restrict__ part, int nparts,
                                                                  double *__restrict__ out_mean,
                                                                  double *__restrict__ out_count, int want_sum) {
  __shared__ double sh[2 * kMeanThreads / 32];
  wait_for_stream_predecessor();
  double s = 0.0, c = 0.0;
  for (int j = threadIdx.x; j < nparts; j += kMeanThreads) { s += part[j].sum; c += part[j].cnt; }
  block_reduce_2(s, c, sh);
  if (threadIdx.x == 0) {
    *out_mean = want_sum ? s : (c > 0.0 ? s / c : CUDART_NAN);
    *out_count = c;
  }
}

// Mean of per-sequence means: block s adds the unmasked tokens of sequence s in a fixed order ...
__global__ void __launch_bounds__(kMeanThreads) seq_partial_kernel(const float *__restrict__ ent,
                                                                   const uint8_t *__restrict__ mask, int64_t seq_len,
                                                                   MeanPartial *__restrict__ part) {
  __shared__ double sh[2 * kMeanThreads / 32];
  wait_for_stream_predecessor();
  const int64_t lo = (int64_t)blockIdx.x * seq_len;
  double s = 0.0, c = 0.0;
  for (int64_t j = threadIdx.x; j < seq_len; j += kMeanThreads) {
    const bool on = mask ? mask[lo + j] != 0 : true;
    if (on) { s += (double)ent[lo + j]; c += 1.0; }
  }
  block_reduce_2(s, c, sh);
  if (threadIdx.x == 0) { part[blockIdx.x].sum = s; part[blockIdx.x].cnt = c; }
}

// ... and one block averages the sequences' means in index order (sequences without tokens take no part).
__global__ void __launch_bounds__(kMeanThreads) seq_final_kernel(const MeanPartial *__restrict__ part, int64_t n_seq,
                                                                 double *__restrict__ out_mean,
                                                                 double *__restrict__ out_count) {
  __shared__ double sh[2 * kMeanThreads / 32];
  wait_for_stream_predecessor();
  double m = 0.0, c = 0.0;
  for (int64_t j = threadIdx.x; j < n_seq; j += kMeanThreads)
    if (part[j].cnt > 0.0) { m += part[j].sum / part[j].cnt; c += 1.0; }
  block_reduce_2(m, c, sh);
  if (threadIdx.x == 0) {
    *out_mean = c > 0.0 ? m / c : CUDART_NAN;
    *out_count = c;
  }
}

// One warp per group; a group of any size is walked in strides of 32 (what a lane takes first stays in its registers: groups of
// up to 32 rollouts, the usual ones, are read once).  n_fill >= 0: the entries of adv outside every group (n_fill in all) become 0.
__global__ void __launch_bounds__(128) group_advantage_kernel(const float *__restrict__ rewards,
                                                              const int64_t *__restrict__ off, int64_t n_groups,
                                                              float eps, int unbiased, float *__restrict__ adv,
                                                              uint8_t *__restrict__ flags, int64_t n_fill) {
  wait_for_stream_predecessor();
  const int lane = threadIdx.x & 31;
  if (n_fill >= 0) {
    const int64_t first = off[0], last = off[n_groups], step = (int64_t)gridDim.x * blockDim.x;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = t; i < first && i < n_fill; i += step) adv[i] = 0.f;
    for (int64_t i = last + t; i < n_fill; i += step) adv[i] = 0.f;
  }
  const int64_t g = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (g >= n_groups) return;
  const int64_t lo = off[g], hi = off[g + 1], n = hi - lo;
  if (n <= 0) {
    if (flags && lane == 0) flags[g] = 0;
    return;
  }
  const float mine = lo + lane < hi ? rewards[lo + lane] : 0.f;
  const float r0 = __shfl_sync(0xffffffffu, mine, 0);
  double s = (double)mine;
  int differs = lo + lane < hi && mine != r0, nonzero = mine != 0.f;
  for (int64_t i = lo + 32 + lane; i < hi; i += 32) {
    const float r = rewards[i];
    s += (double)r;
    differs |= (r != r0);
    nonzero |= (r != 0.f);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  differs = __any_sync(0xffffffffu, differs);
  nonzero = __any_sync(0xffffffffu, nonzero);
  const double mean = s / (double)n;
  double d = lo + lane < hi ? (double)mine - mean : 0.0;
  double ss = d * d;
  for (int64_t i = lo + 32 + lane; i < hi; i += 32) {
    d = (double)rewards[i] - mean;
    ss += d * d;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  const double denom = unbiased ? (double)(n - 1) : (double)n;
  const double sd = n == 1 ? 0.0 : sqrt(ss / denom);
  // std + eps == 0 (eps == 0 and identical rewards): every r_i - mean is 0 and the advantage is 0, not 0/0
  const double inv = sd + (double)eps > 0.0 ? 1.0 / (sd + (double)eps) : 0.0;
  if (lo + lane < hi) adv[lo + lane] = n == 1 ? 0.f : (float)(((double)mine - mean) * inv);
  for (int64_t i = lo + 32 + lane; i < hi; i += 32)
    adv[i] = n == 1 ? 0.f : (float)(((double)rewards[i] - mean) * inv);
  if (flags && lane == 0) flags[g] = (uint8_t)((differs ? 0 : 1) | (nonzero ? 0 : 2));
}

}  // namespace

int mean_blocks(int64_t n) {
  int64_t b = (n + 4095) / 4096;
  if (b < 1) b = 1;
  if (b > kMeanBlocksMost) b = kMeanBlocksMost;
  return (int)b;
}

size_t mean_workspace_bytes(int64_t n) { return (size_t)mean_blocks(n) * sizeof(MeanPartial); }

cudaError_t launch_masked_mean(const float *ent, const uint8_t *mask, int64_t n, double *out_mean,
                               double *out_count, void *workspace, bool want_sum, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (n <= kClusterMost * kClusterTokens) {
    // a CTA takes 4,096 tokens (one round of its threads) before another one joins
    int64_t ctas = (n + 4 * kClusterThreads - 1) / (4 * kClusterThreads);
    ctas = ctas < 1 ? 1 : (ctas > kClusterMost ? kClusterMost : ctas);
    const int64_t chunk = (((n + ctas - 1) / ctas) + 3) / 4 * 4;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)ctas;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
    cfg.blockDim = dim3(kClusterThreads);
    cfg.gridDim = dim3((unsigned)ctas);
    return cudaLaunchKernelEx(&cfg, mean_cluster_kernel, ent, mask, n, chunk, out_mean, out_count, want_sum ? 1 : 0);
  }
  const int blocks = mean_blocks(n);
  const int64_t chunk = (((n + blocks - 1) / blocks) + 3) / 4 * 4;
  MeanPartial *part = static_cast<MeanPartial *>(workspace);
  cfg.blockDim = dim3(kMeanThreads);
  cfg.gridDim = dim3((unsigned)blocks);
  cudaError_t e = cudaLaunchKernelEx(&cfg, mean_partial_kernel, ent, mask, n, chunk, part);
  if (e != cudaSuccess) return e;
  cfg.gridDim = dim3(1);
  return cudaLaunchKernelEx(&cfg, mean_final_kernel, (const MeanPartial *)part, blocks, out_mean, out_count,
                            want_sum ? 1 : 0);
}

size_t seq_mean_workspace_bytes(int64_t n_seq) { return (size_t)(n_seq < 1 ? 1 : n_seq) * sizeof(MeanPartial); }

cudaError_t launch_sequence_mean(const float *ent, const uint8_t *mask, int64_t n_seq, int64_t seq_len,
                                 double *out_mean, double *out_count, void *workspace, cudaStream_t stream) {
  MeanPartial *part = static_cast<MeanPartial *>(workspace);
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kMeanThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (n_seq > 0) {
    cfg.gridDim = dim3((unsigned)n_seq);
    cudaError_t e = cudaLaunchKernelEx(&cfg, seq_partial_kernel, ent, mask, seq_len, part);
    if (e != cudaSuccess) return e;
  }
  cfg.gridDim = dim3(1);
  return cudaLaunchKernelEx(&cfg, seq_final_kernel, (const MeanPartial *)part, n_seq, out_mean, out_count);
}

cudaError_t launch_group_advantage(const float *rewards, const int64_t *off, int64_t n_groups, float eps,
                                   int unbiased, float *adv, uint8_t *flags, int64_t n_fill, cudaStream_t stream) {
  constexpr int kWarpsPerBlock = 4;
  const int64_t blocks = n_groups > 0 ? (n_groups + kWarpsPerBlock - 1) / kWarpsPerBlock : 1;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kWarpsPerBlock * 32);
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, group_advantage_kernel, rewards, off, n_groups, eps, unbiased, adv, flags, n_fill);
}

}  // namespace e3
