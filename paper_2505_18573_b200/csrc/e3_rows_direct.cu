// Row kernel of short calls: what rows_kernel (e3_rows.cu) gives, for calls whose logits the SMs' shared memory holds (nearly) at once.
// Such a call is bound by the length of its chain of dependent steps and not by bandwidth: the streaming kernel's start (rings, barriers,
// the first strips), its records and the exchange of cut rows through global memory took 8 to 12 us for a call of a few KB.
//
// A row is cut into 1 to 16 parts of equal length, one CTA each, which form a cluster.  Every warp copies what its own lanes are going to
// look at (`cp.async`, one commit group per step) and waits for nothing but that; a step is 16 entries (one group of sampler 0's
// coarse stream) per lane, so that 32 lanes hold two of sampler 1's blocks.  Meanwhile it makes its random numbers, which do not depend on
// the logits: sampler 0's coarse bytes and the Gumbel variates of the entries whose byte is 255 (one in 256), sampler 1's Gumbel variates
// and the draw inside the block.  Sums refer to the warp's largest logit so far; clamped entries (-inf) cost one instruction a pair here.
// A warp whose 512 entries of a step are all a fill value such as -1e9 has that as its largest: its products are rounded down and,
// where they are too large for that, taken with a power of two in place of c (far_terms), at no cost to the sums of other rows.
// Sampler 0 scores its hits, takes the best of the CTA as bound, and scores the few entries above the gate that this leaves, whatever
// their coarse byte.  Sampler 1 draws inside the leading block of every part, of which the row's is one.
// The first warp merges the CTA's warps and hands the result to the first CTA of the row by `st.async` (data and signal in one); there the
// parts are merged in their order, near-ties settled in fp64 and the row finished.  Results depend on the size of the call alone.
//
// us per call, back to back, streaming kernel and this one: blocked sampler 1 x 8,000 bf16 8.1, 4.3; 64 x 32,000 fp32 11.8, 7.2; 64 x 151,936 bf16 16.0,
// 12.0; token sampler 1 x 8,000 12.4, 6.0; 8 x 151,936 26.7, 10.2; 45 x 45,000 23.9, 10.8; training pass (with the sum of the entropies) 16 x 20,000
// fp32 13.5, 6.2.
#include "e3_rows.cuh"
#include "e3_rows_device.cuh"

#include <atomic>
#include <mutex>
#include <type_traits>

namespace e3 {
namespace {

constexpr int kWords = 5;                       // sampler 0: words of hit bits, two steps each
constexpr int kChunkBytes = 104 * 1024;         // most bytes of a row that a CTA takes
constexpr int kSlackBytes = 32;                 // ... and reads around them: rows that begin anywhere
static_assert(70 * 1024 / 2 <= 2 * kWords * 256 * kGroup && kChunkBytes / 2 <= 2 * kWords * 512 * kGroup, "steps");
constexpr int kClusterMost = 16;
constexpr int kQueue = 64;                      // a push meets at most 31 entries and adds at most 32

// State of a part of a row: of a warp, of a CTA (handed to the row's first one).
struct __align__(16) Part {
  float M, Z, W;   // reference (log2 units), sum 2^t, sum 2^t t
  float zmax;      // largest logit (only where the mean logit gap is asked for)
  float ty[3];     // leading scores: sampler 0 entries, sampler 1 blocks; greedy rows: ty[0] = largest logit
  int err;
  int tb[3];       // ... and their vocabulary / block indices, -1 = none
  int tok;         // of a CTA, sampler 1: the token drawn in its leading block
  float zf;        // of a CTA: logit of entry tb[0], of that token
  int pad[3];
};
static_assert(sizeof(Part) == 64, "four 16-byte stores");

template <int kWarps>
struct Shared {
  Part hand[kClusterMost];  // first CTA of the row: of all its CTAs
  Part warp[kWarps];
  uint32_t queue[kWarps][kQueue];
  u64 handed;               // the other CTAs' parts have come
  int best;                 // sampler 0: encoded bound of the best score
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const char *src, u64 policy) {
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "l"(policy) : "memory");
}
// Waits until at most `later` of the thread's groups of copies are under way.
__device__ __forceinline__ void cp_async_wait(int later) {
  switch (later) {
    case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    case 3: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
    case 4: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
    case 5: asm volatile("cp.async.wait_group 5;" ::: "memory"); break;
    case 6: asm volatile("cp.async.wait_group 6;" ::: "memory"); break;
    case 7: asm volatile("cp.async.wait_group 7;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 8;" ::: "memory"); break;
  }
}
// One poll of a barrier that counts what other CTAs of the cluster send (their stores are visible once it says so).
__device__ __forceinline__ bool mbar_try_wait_cluster(u64 *b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// The 16-byte vectors of the group of 16 entries that begins `off` bytes into the chunk; v[i] is vector i xor sw.  a: bytes by which
// the chunk lies behind a 16-byte boundary (sw is 0 then, else spreads eight lanes over the banks).  Entries from `valid` on become -inf.
template <int DT>
__device__ __forceinline__ void load_vecs(uint32_t base, uint32_t a, uint32_t off, int sw, int valid, uint4 (&v)[Fmt<DT>::kVG]) {
  constexpr int N = Fmt<DT>::kVG;
  if (a == 0u) {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = lds128(base + off + (uint32_t)((i ^ sw) << 4));
  } else {
    uint4 x = lds128(base + off);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const uint4 y = lds128(base + off + (uint32_t)((i + 1) << 4));
      v[i] = shift_vec(x, y, a);
      x = y;
    }
  }
  if (valid < kGroup) {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = mask_vec<DT>(v[i], valid, i ^ sw);
  }
}

// The lane's entries that equal R: groups of 16, a step of `step_e` entries apart, of which `left` entries are valid from the first on.
template <int DT>
__device__ __noinline__ float far_entries(uint32_t addr, int step_e, int left, float R) {
  float n = 0.f;
#pragma unroll 1
  for (; left > 0; left -= step_e, addr += (uint32_t)(step_e * Fmt<DT>::kEsize)) n += far_count<DT>(addr, left, R);
  return n;
}

template <int DT, int SAMPLER, int kThreads>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads) rows_direct_kernel(const __grid_constant__ RowsParams p, int chunk, int ctas) {
  extern __shared__ __align__(128) unsigned char dyn[];
  constexpr int kWarps = kThreads / 32;
  constexpr int kStepE = kThreads * kGroup;       // entries that the CTA takes per step
  __shared__ Shared<kWarps> sh;
  using F = Fmt<DT>;
  constexpr int N = F::kVG;
  constexpr unsigned kAll = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(kAll, tid >> 5, 0);
  const uint32_t row = blockIdx.x / (uint32_t)ctas, rank = blockIdx.x - row * (uint32_t)ctas;
  const int e0 = (int)rank * chunk, n = p.V - e0 < chunk ? p.V - e0 : chunk;  // (n may be 0 or less)
  if (ctas > 1) {
    // the first CTA has started, and its barrier stands, when its memory is written to
    if (rank == 0 && tid == 0) {
      mbar_init(&sh.handed, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      // (test hook: 16 bytes that nobody sends)
      mbar_arrive_expect(&sh.handed, (uint32_t)(ctas * sizeof(Part)) + (row_ptr(p, row) == p.stall_src ? 16u : 0u));
    }
    __syncwarp();
    cluster_arrive();
  }
  if (SAMPLER == 0) {
    if (tid == 0) sh.best = enc_neg_inf();
    __syncthreads();
  }
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (SAMPLER < 0 && p.mask != nullptr && __ldg(p.mask + row) == 0) {
    if (rank == 0 && tid == 0) write_plain(p, row, 0.f);
    return;
  }

  // ---- every warp copies what it is going to look at: per step 32 groups
  const char *src = row_ptr(p, row) + (size_t)e0 * F::kEsize;
  const uint32_t a = (uint32_t)(reinterpret_cast<uintptr_t>(src) & 15u), base = smem_addr(dyn);
  const int steps = n > warp * 32 * kGroup ? (n - warp * 32 * kGroup + kStepE - 1) / kStepE : 0;  // of this warp
  {
    const u64 policy = l2_evict_first_policy();
    src -= a;
    const int units = n > 0 ? ((int)a + n * F::kEsize + 15) >> 4 : 0;
#pragma unroll 1
    for (int k = 0; k < steps; ++k) {
      const int u0 = (k * kThreads + warp * 32) * N;
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const int u = u0 + i * 32 + lane;
        if (u < units) cp_async16(base + (uint32_t)u * 16u, src + (size_t)u * 16u, policy);
      }
      if (a != 0u && lane == 0 && u0 + 32 * N < units)
        cp_async16(base + (uint32_t)(u0 + 32 * N) * 16u, src + (size_t)(u0 + 32 * N) * 16u, policy);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
  }
  const float tau = p.temps != nullptr ? __ldg(p.temps + row) : p.temp_scalar;
  const bool finisher = rank == 0 && warp == 0;  // finishes the row
  int target = -1;
  if (SAMPLER < 0 && finisher) target = __ldg(p.targets + row);

  // ---- random numbers, while the copies are under way
  EvalCtx ex;
  ex.rk = p.round_key; ex.row = row_ptr(p, row); ex.tau = 0.f; ex.slack_k = p.slack_scale;
  ex.grow = p.row_base + row;
  ex.ctr_lo = p.ctr_lo; ex.ctr_hi8 = p.ctr_hi8; ex.V = p.V;
  const int g0 = warp * 32 + lane;  // the lane's group of step 0
  uint32_t hw[kWords];              // sampler 0: coarse bytes that are 255: bit 8*byte + 4*(step mod 2) + word; hw[0]: the last steps
  int pair = -1, qn = 0;            // steps that hw[0] belongs to; entries in the queue
  int hit_i = -1;                   // the lane's hit: entry of the chunk,
  float hit_g = 0.f;                // its Gumbel variate
  uint32_t *const queue = sh.queue[warp];
  const PhiloxRow prow = SAMPLER == 0 ? philox_row(p.round_key, p.row_base + row, p.ctr_lo, p.ctr_hi8 | 0u) : PhiloxRow{};
  auto push = [&](bool f, uint32_t e) {
    const uint32_t ballot = __ballot_sync(kAll, f);
    if (f) queue[qn + __popc(ballot & ((1u << lane) - 1u))] = e;
    qn += __popc(ballot);
  };
  // Moves hits into the queue until 32 wait there or none is left, and gives each lane one of them.
  auto next_hits = [&]() {
#pragma unroll 1
    while (pair >= 0 && qn < 32) {
      const uint32_t w = hw[0];
      if (!__any_sync(kAll, w != 0u)) {
#pragma unroll
        for (int i = 0; i + 1 < kWords; ++i) hw[i] = hw[i + 1];
        --pair;
        continue;
      }
      const int bit = __ffs((int)w) - 1;
      const int e = ((2 * pair + ((bit >> 2) & 1)) * kThreads + g0) * kGroup + 4 * (bit & 3) + (bit >> 3);
      hw[0] = w & (w - 1u);
      push(w != 0u && e < n, (uint32_t)e);
    }
    __syncwarp();
    const int from = qn > 32 ? qn - 32 : 0;
    hit_i = from + lane < qn ? (int)queue[from + lane] : -1;
    qn = from;
    __syncwarp();
    if (hit_i >= 0) {
      const int i = e0 + hit_i;
      const uint4 fw = philox(p.round_key, (uint32_t)i >> 2, p.row_base + row, p.ctr_lo, p.ctr_hi8 | 1u);
      hit_g = gumbel_f32(255u, pick_word(fw, i & 3));
    }
  };
  float block_g = 0.f;     // sampler 1: Gumbel variate of block lane mod 2 of the warp's step lane / 2
  uint32_t in_block = 0u;  // ... the draw inside the block
  if (SAMPLER == 0) {
#pragma unroll
    for (int i = 0; i < kWords; ++i) hw[i] = 0u;
#pragma unroll 1
    for (int k = 0; k < steps; k += 2) {
#pragma unroll
      for (int i = kWords - 1; i > 0; --i) hw[i] = hw[i - 1];
      hw[0] = 0u;
      ++pair;
#pragma unroll 1
      for (int h = 0; h < 2 && k + h < steps; ++h) {
        const uint4 cb = philox_call(p.round_key, prow, (uint32_t)(e0 >> 4) + (uint32_t)((k + h) * kThreads + g0));
        hw[0] |= ((ff_bytes(cb.x) >> 7) | (ff_bytes(cb.y) >> 6) | (ff_bytes(cb.z) >> 5) | (ff_bytes(cb.w) >> 4)) << (4 * h);
      }
    }
    next_hits();
  }
  if (SAMPLER == 1) {
    // one call a lane: lane 31 of the first warp makes the draw inside the block, the others the blocks of their steps
    const int b = (e0 >> 8) + ((lane >> 1) * kThreads + warp * 32) / 16 + (lane & 1);
    const bool draw = warp == 0 && lane == 31;
    const uint4 x = philox(p.round_key, draw ? 0u : (uint32_t)b >> 2, p.row_base + row, p.ctr_lo, p.ctr_hi8 | (draw ? 3u : 2u));
    block_g = gumbel_from_word(pick_word(x, b & 3));
    in_block = __shfl_sync(kAll, x.x, 31);
  }
  float z_target = 0.f;
  if (SAMPLER < 0 && (uint32_t)target < (uint32_t)p.V) z_target = load_elem<DT>(ex.row, target);
  const bool greedy = SAMPLER >= 0 && tau == 0.f, usable = greedy || (tau > 0.f && tau < CUDART_INF_F);
  const float c = greedy || !usable ? 0.f : __fdiv_rn(kLog2e, tau);
  ex.tau = tau;
  const int sw = a != 0u ? 0 : (DT == 1 ? (lane >> 2) & 1 : (lane >> 1) & 3);
  Part pc;
  pc.M = pc.Z = pc.W = pc.zf = 0.f;
  pc.zmax = -CUDART_INF_F;
  pc.err = usable ? 0 : kErrValue;
  pc.tok = -1;
  Top3 top;  // the lane's leaders
  top3_reset(top);
  if (ctas > 1) cluster_wait();

  if (greedy) {
    // largest logit, lowest index
    cp_async_wait(0);
    __syncwarp();
    bool bad = false;
#pragma unroll 1
    for (int k = 0; k < steps; ++k) {
      const int g = k * kThreads + g0;
#pragma unroll 1
      for (int e = g * kGroup; e < n && e < (g + 1) * kGroup; ++e) {
        const float z = lds_elem<DT>(base + a + (uint32_t)(e * F::kEsize)) + 0.f;  // (-0 and +0 are the same logit)
        bad |= !(z < CUDART_INF_F);
        if (z > top.y[0]) {
          top.y[0] = z;
          top.b[0] = e0 + e;
        }
      }
    }
    if (__any_sync(kAll, bad)) pc.err = kErrValue;
  } else if (usable) {
    // ---- sums, relative to the largest logit of the warp so far
    f2 c2 = pack2f(c, c), nRc2 = pack2f(0.f, 0.f), Zt = nRc2, Wa = Zt, Wb = Zt;  // t = z c2 + nRc2
    float R = -CUDART_INF_F, nRc = 0.f;
#pragma unroll 1
    for (int k = 0; k < steps; ++k) {
      const int g = k * kThreads + g0, valid = n - g * kGroup;
      cp_async_wait(steps - 1 - k);
      __syncwarp();
      uint4 v[N];
      float m = -CUDART_INF_F;
      if (valid > 0) {
        load_vecs<DT>(base, a, (uint32_t)(g * kGroup * F::kEsize), sw, valid, v);
        m = vec_max<DT>(v);
      }
      m = warp_max(m);
      if (m > R) {
        const float up = reference(m, c);
        if (R > -CUDART_INF_F) {
          const float d = up - nRc, f = ex2f(d);
          Wa = fma2(pack2f(d, d), Zt, add2(Wa, Wb));
          Wb = pack2f(0.f, 0.f);
          Wa = fma2(pack2f(f, f), Wa, Wb);
          Zt = fma2(pack2f(f, f), Zt, Wb);
        }
        R = m;
        nRc = up;
        float ct = c, nt = up;
        if (fabsf(up) >= kFar) far_terms(m, ct, nt);
        c2 = pack2f(ct, ct);
        nRc2 = pack2f(nt, nt);
      }
      f2 Za = pack2f(0.f, 0.f), Zb = Za;
      if (valid > 0) {
#pragma unroll
        for (int i = 0; i < N; ++i) vec_sums<DT, true>(v[i], c2, nRc2, Za, Zb, Wa, Wb);
      }
      Za = add2(Za, Zb);
      Zt = add2(Zt, Za);
      if (SAMPLER == 1) {  // 16 lanes hold a block
        float S = sum2(Za);
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) S += __shfl_xor_sync(kAll, S, o);
        const float gum = __shfl_sync(kAll, block_g, 2 * k + (lane >> 4));
        if (S > 0.f && (lane & 15) == 0) top3_insert(top, (lg2f(S) - nRc) * kLn2f + gum, (e0 >> 8) + (k * kThreads + g0) / 16);
      }
    }
    pc.Z = sum2(Zt);
    pc.W = sum2(add2(Wa, Wb));
    if (R < kClampAt && R > -CUDART_INF_F)  // (entries of -inf are not to count)
      pc.Z = fabsf(nRc) >= kFar ? far_entries<DT>(base + a + (uint32_t)(g0 * kGroup * F::kEsize), kStepE, n - g0 * kGroup, R) : CUDART_NAN_F;
    bool bad = !(pc.Z <= 1e6f) || !(fabsf(pc.W) <= kSoundW) || !(c < CUDART_INF_F);
    if (R == -CUDART_INF_F) bad |= pc.Z != 0.f;
    if (__any_sync(kAll, bad)) {
      pc.err = kErrValue;
      pc.Z = pc.W = 0.f;
    } else {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        pc.Z += __shfl_xor_sync(kAll, pc.Z, o);
        pc.W += __shfl_xor_sync(kAll, pc.W, o);
      }
      pc.M = -nRc;
      pc.zmax = R;
    }

    if (SAMPLER == 0) {
      const float inv_tau = __frcp_rn(tau);
      // Score of entry i (not one with coarse byte 255: those are in the list of hits).
      auto enter = [&](bool valid, int i, float z) {
        const uint4 cw = philox_call(p.round_key, prow, (uint32_t)i >> 4);
        const uint4 fw = philox(p.round_key, (uint32_t)i >> 2, p.row_base + row, p.ctr_lo, p.ctr_hi8 | 1u);
        const uint32_t cbyte = (pick_word(cw, (i & 15) >> 2) >> (8 * (i & 3))) & 0xFFu;
        if (valid && cbyte != 255u) top3_insert(top, score_f32(z, inv_tau, cbyte, pick_word(fw, i & 3)), i);
      };
      // ---- entries with coarse byte 255
#pragma unroll 1
      for (;;) {
        if (hit_i >= 0) {
          const float z = lds_elem<DT>(base + a + (uint32_t)(hit_i * F::kEsize));
          if (z > -CUDART_INF_F && z < CUDART_INF_F) top3_insert(top, score_of(z, inv_tau, hit_g), e0 + hit_i);
        }
        if (pair < 0 && qn == 0) break;
        next_hits();
      }
      // lower bound of the row's best score: four slacks below the best of the CTA so far
      auto bound = [&]() {
        const int e = __reduce_max_sync(kAll, top.b[0] >= 0 ? enc_float(top.y[0]) : enc_neg_inf());
        if (e == enc_neg_inf()) return e;
        const float y = dec_float(e);
        return enc_float(y - 4.f * score_slack(y, p.slack_scale) - 2e-7f * fabsf(y));
      };
      {
        const int mine = bound();
        if (lane == 0) atomicMax(&sh.best, mine);
      }
      __syncthreads();
      // ---- the other entries above the gate, whatever their coarse byte
      float gate = logit_gate(sh.best, tau, kGumbelCapCoarse);
      auto drain = [&]() {
        __syncwarp();
        const int from = qn > 32 ? qn - 32 : 0;
        const bool valid = from + lane < qn;
        const int e = valid ? (int)queue[from + lane] : 0;
        const float z = lds_elem<DT>(base + a + (uint32_t)(e * F::kEsize));
        enter(valid && z < CUDART_INF_F, e0 + e, z);
        qn = from;
        gate = fmaxf(gate, logit_gate(bound(), tau, kGumbelCapCoarse));
        __syncwarp();
      };
      if (R > gate) {
#pragma unroll 1
        for (int k = 0; k < steps; ++k) {
          const int g = k * kThreads + g0, valid = n - g * kGroup;
          uint32_t above = 0u;  // bit e: entry e of the group
          if (valid > 0) {
            uint4 v[N];
            load_vecs<DT>(base, a, (uint32_t)(g * kGroup * F::kEsize), sw, valid, v);
#pragma unroll
            for (int i = 0; i < N; ++i) above |= entries_above<DT>(v[i], gate) << ((i ^ sw) * (16 / F::kEsize));
          }
#pragma unroll 1
          for (;;) {
            const uint32_t ballot = __ballot_sync(kAll, above != 0u);
            if (ballot == 0u) break;
            if (above != 0u) queue[qn + __popc(ballot & ((1u << lane) - 1u))] = (uint32_t)(g * kGroup + __ffs((int)above) - 1);
            qn += __popc(ballot);
            above &= above - 1u;
            if (qn >= 32) drain();
          }
        }
        if (qn > 0) drain();
      }
    }
  } else {
    cp_async_wait(0);  // (a temperature that cannot be used: the copies still land before the CTA's memory goes to another)
  }

  // ---- the CTA's result
  auto merge_leaders = [&]() {
    if (SAMPLER == 0) warp_merge_near(top, 4.f * p.slack_scale * 1.7e-4f, 4.f * p.slack_scale * 1e-6f);
    if (SAMPLER == 1) merge_near_blocks(top);
#pragma unroll
    for (int i = 0; i < 3; ++i) { pc.ty[i] = top.y[i]; pc.tb[i] = top.b[i]; }
  };
  // Merges the parts held by lanes below `lanes`, a power of two.
  auto merge_parts = [&](int lanes) {
    const bool has = pc.Z > 0.f;
    const int em = __reduce_max_sync(kAll, has ? enc_float(pc.M) : enc_neg_inf());
    if (em != enc_neg_inf()) {
      const float Mw = dec_float(em), d = pc.M - Mw, f = ex2f(d);
      pc.W = has ? f * fmaf(d, pc.Z, pc.W) : 0.f;
      pc.Z = has ? f * pc.Z : 0.f;
      pc.M = Mw;
#pragma unroll 1
      for (int o = lanes >> 1; o > 0; o >>= 1) {
        pc.Z += __shfl_xor_sync(kAll, pc.Z, o);
        pc.W += __shfl_xor_sync(kAll, pc.W, o);
      }
    }
    pc.Z = __shfl_sync(kAll, pc.Z, 0);
    pc.W = __shfl_sync(kAll, pc.W, 0);
    pc.err = __any_sync(kAll, pc.err != 0) ? kErrValue : 0;
    if (p.out_gap != nullptr) pc.zmax = dec_float(__reduce_max_sync(kAll, enc_float(pc.zmax)));
    if (SAMPLER >= 0) {
#pragma unroll
      for (int i = 0; i < 3; ++i) { top.y[i] = pc.ty[i]; top.b[i] = pc.tb[i]; }
      merge_leaders();
    }
  };
  auto no_part = [&]() {
    pc.M = pc.Z = pc.W = 0.f;
    pc.zmax = -CUDART_INF_F;
    pc.err = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) { pc.ty[i] = -CUDART_INF_F; pc.tb[i] = -1; }
  };
  if (SAMPLER >= 0) merge_leaders();
  if (lane == 0) sh.warp[warp] = pc;
  __syncthreads();
  if (warp != 0) return;
  if (lane < kWarps) pc = sh.warp[lane];
  else no_part();
  merge_parts(kWarps);
  if (SAMPLER == 1 && !greedy && pc.tb[0] >= 0) {
    // draws inside the CTA's leading block: if that block leads the row (and no other comes close) the draw stands
    float z[8];
    const int e = pc.tb[0] * 256 - e0 + lane * 8;
#pragma unroll
    for (int k = 0; k < 8; ++k) z[k] = e + k < n ? lds_elem<DT>(base + a + (uint32_t)((e + k) * F::kEsize)) : -CUDART_INF_F;
    pc.tok = draw_among<DT>(ex, pc.tb[0], lane, z, in_block, pc.zf);
  }
  if (SAMPLER == 0 && pc.tb[0] >= 0) pc.zf = lds_elem<DT>(base + a + (uint32_t)((pc.tb[0] - e0) * F::kEsize));
  if (ctas > 1) {
    if (lane < 4) {
      const float x0 = lane == 0 ? pc.M : (lane == 1 ? pc.ty[0] : (lane == 2 ? __int_as_float(pc.tb[0]) : pc.zf));
      const float x1 = lane == 0 ? pc.Z : (lane == 1 ? pc.ty[1] : (lane == 2 ? __int_as_float(pc.tb[1]) : 0.f));
      const float x2 = lane == 0 ? pc.W : (lane == 1 ? pc.ty[2] : (lane == 2 ? __int_as_float(pc.tb[2]) : 0.f));
      const float x3 = lane == 0 ? pc.zmax : (lane == 1 ? __int_as_float(pc.err) : (lane == 2 ? __int_as_float(pc.tok) : 0.f));
      uint32_t to, bar;
      asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(to) : "r"(smem_addr(&sh.hand[rank]) + 16u * lane));
      asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(bar) : "r"(smem_addr(&sh.handed)));
      asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(to),
                   "r"(__float_as_uint(x0)), "r"(__float_as_uint(x1)), "r"(__float_as_uint(x2)), "r"(__float_as_uint(x3)), "r"(bar)
                   : "memory");
    }
    if (rank != 0) return;
    __syncwarp();
    bool came = mbar_try_wait_cluster(&sh.handed, 0);
    if (!__all_sync(kAll, came)) {
      const u64 t0 = global_ns();
      for (uint32_t it = 1; !came; ++it) {
        came = mbar_try_wait_cluster(&sh.handed, 0);
        if ((it & 63u) == 0u && global_ns() - t0 > p.wait_ns) break;
      }
      if (!__all_sync(kAll, came)) {
        // given up: the row has no result; what may still come must find this CTA's memory
        if (lane == 0) {
          write_plain(p, row, CUDART_NAN_F);
          if (p.status != nullptr) atomicOr(p.status, kStatusTimeout);
        }
        cluster_arrive();
        cluster_wait();
        return;
      }
    }
    no_part();
    if (lane < ctas) pc = sh.hand[lane];
    const int own = pc.tb[0];
    merge_parts(kClusterMost);
    if (SAMPLER >= 0) {
      const uint32_t from = __ballot_sync(kAll, own >= 0 && own == pc.tb[0]);
      const int l = from != 0u ? __ffs((int)from) - 1 : 0;
      pc.tok = __shfl_sync(kAll, pc.tok, l);
      pc.zf = __shfl_sync(kAll, pc.zf, l);
    }
  }
  // ---- the row's result
  int id = SAMPLER < 0 ? ((uint32_t)target < (uint32_t)p.V ? target : -1) : pc.tb[0];
  float zt = SAMPLER < 0 ? z_target : pc.zf;
  if (SAMPLER >= 0 && !greedy && id >= 0) {
    if (SAMPLER == 1) {
      id = pc.tok;
      if (top.b[1] >= 0 && blocks_too_close(top)) id = pc.err == 0 ? sample_in_blocks<DT>(ex, top, lane, zt) : -1;
    } else {
      const float slack2 = 2.f * fmaxf(score_slack(top.y[0], p.slack_scale), score_slack(top.y[1], p.slack_scale));
      if (top.b[1] >= 0 && !(top.y[0] - top.y[1] > slack2)) id = settle_exact<DT>(ex, top, slack2, lane, zt);
    }
  }
  RowInfo ri;
  ri.greedy = greedy;
  ri.c = c;
  if (lane == 0) finish_row(p, row, ri, pc.M, pc.Z, pc.W, pc.zmax, id, pc.err, id >= 0, zt);
}

int64_t chunk_of(int64_t V, int64_t ctas) { return ((V + ctas - 1) / ctas + 255) / 256 * 256; }

// The most CTAs of a cluster that the device can hold, each with the shared memory a CTA takes at most.  A whole B200 holds kClusterMost;
// a partition of one (or of its SMs) may hold fewer.
template <class K>
int largest_cluster(K kern, int threads) {
  for (int n = kClusterMost; n > 1; --n) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)n;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = kChunkBytes + kSlackBytes;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) == cudaSuccess && clusters > 0) return n;
    cudaGetLastError();  // (no such cluster here: nobody's error)
  }
  return 1;
}

template <int DT, int SAMPLER, int kThreads>
cudaError_t launch(const RowsParams &p, int64_t rows, int ctas, int dev, const RowStall &stall, cudaStream_t stream, bool &taken) {
  static std::mutex lock;
  static int most[64];  // CTAs of a cluster; 0: not asked yet
  auto kern = rows_direct_kernel<DT, SAMPLER, kThreads>;
  {
    std::lock_guard<std::mutex> hold(lock);
    if (most[dev] == 0) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kChunkBytes + kSlackBytes);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
      most[dev] = largest_cluster(kern, kThreads);
    }
    if (ctas > most[dev]) return cudaSuccess;  // (the streaming kernel needs no cluster)
  }
  taken = true;
  RowsParams q = p;
  const int chunk = (int)chunk_of(p.V, ctas);
  q.wait_ns = kDefaultWaitNs;
  q.stall_src = nullptr;
  if (stall.row >= 0) {
    q.wait_ns = stall.wait_ns;
    q.stall_src = p.logits + stall.row * p.row_bytes;
  }
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)ctas;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(rows * ctas));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (size_t)(chunk * Fmt<DT>::kEsize + kSlackBytes);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = ctas > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, q, chunk, ctas);
}

// Threads of a CTA and CTAs of a row for a call of this size; no threads: the call is for the streaming kernel.
//
// Up to two CTAs per SM the call lives on latency: 256 threads with a step or two each, or 512 where a CTA's part is longer (us with
// 256 and 512: 45 x 45,000 bf16 in 6 parts 7.8, 8.2; 64 x 32,000 fp32 in 4 parts 7.8, 7.2).  Clusters of more than eight are worth their slower
// launch for a few rows alone (1 x 151,936: 8 parts 7.0, 16 parts 5.5; 16 x 100,000, token sampler: 10.8, 12.4).
// Beyond, three or four CTAs of 256 threads per SM hold more of the call at once, as long as one wave of them holds (nearly) all of it: 100 x
// 64,000 fp32 15.1 (streaming 17.1), 600 x 20,000 bf16 15.2 (16.1), but 1,000 x 20,000 21.2 (20.0).  A second wave that holds a few blocks is
// borne by rows of one block (blocked sampler 645 x 24,384 bf16, 109 % of a wave, 18.4 (21.4)); of two blocks with the statistics, and not with the
// blocked sampler, which has more to do behind its sums (226 x 55,552 bf16, 102 %, 20.6 (18.5); 223 x 28,416 fp32, 100 %, 15.2 (16.7)); of three
// and more, which do not fill the SMs to the last place, with the statistics of fp32 (119 x 57,434, 107 %, 13.2 (14.7)) and where an SM holds four
// blocks (104 x 150,592 bf16, 105 %, 13.4 (14.9)), else up to a full wave (87 x 160,036, 98 %, 15.7 (16.1); 155 x 91,282 in three
// parts, 105 %, 17.1 (16.4), in four, four to an SM, 13.9); with the blocked sampler well below one (171 x 74,368, 87 %, 16.8 (17.5); 78 x 169,646,
// 88 %, 20.2 (19.3); 82 x 177,472, 92 %, 23.9 (17.9); 160 x 100,000, 108 %, 26.0 (18.6)).
// Sampler 0 gains more here than a second wave costs: 1,000 x 20,000 31.6 (48.6), 128 x 151,936 35.9 (41.7), 256 x 151,936 62.2 (57.5).
// Of the CTAs of a call with a response mask many have nothing to do, and which is not known here: the lines lie where the kernels are even
// with seven or eight rows of ten unmasked (us with six, eight and all ten).  Two parts a row 1,010 x 43,712 bf16 (3.4 waves) 19.6 (21.7), 23.5
// (24.9), 27.0 (25.2), 862 x 67,984 (3.9) 25.1 (24.2), 31.2 (27.2), 35.5 (30.2); three 386 x 94,683 (2.6) 21.8 (24.9), 26.1 (27.0), 29.8 (29.5),
// 404 x 103,568 (2.7) 20.7 (21.6), 25.2 (23.9), 28.3 (25.9); fp32 four parts 379 x 54,976 (3.4) 17.0 (18.8), 20.2 (21.6), 22.9 (23.9).
// Where one block takes a whole row of 32 KB or more, more waves still pay: five with a mask (1,250 x 40,000 bf16 20.4 (23.7), all rows
// 28.3 (30.6); 2,400 x 35,000, 5.4 waves, 30.8 (29.7), 44.7 (42.2); 1,500 x 50,000, 5.1, 27.9 (29.3), 39.8 (37.7)), and seven of rows up to 64
// KB (4,096 x 20,000 bf16, 6.9, 29.2 (30.6), 41.7 (43.3), 3,255 x 19,520, 5.5, with 57 rows of a hundred 24.9 (28.0); 3,500 x 17,000, 5.9, 24.4
// (24.4), but all rows 34.4 (32.4)), not 8,192 x 32,000 87.1 (71.3).  Sampler 0: four, 1,500 x 32,000
// 63.5 (72.1), but 3,000 x 32,000 116 (113).  Without a mask the streaming kernel has no mask to count.
struct Plan {
  int threads, ctas;
};
Plan plan(int64_t rows, int64_t V, int64_t esize, int sampler, bool mask, int64_t sms) {
  const int64_t most = rows <= 4 ? kClusterMost : 8, two = 2 * sms / rows;
  auto fits = [&](int64_t ctas, int64_t bytes) { return ctas >= 1 && chunk_of(V, ctas) * esize <= bytes; };
  auto least_of = [](int64_t a, int64_t b, int64_t c) { return a < b ? (a < c ? a : c) : (b < c ? b : c); };
  int64_t ctas = least_of(most, (V + 4095) / 4096, two);
  if (fits(ctas, 12 * 1024)) return Plan{256, (int)ctas};
  ctas = least_of(most, (V + 8191) / 8192, two);
  if (fits(ctas, kChunkBytes)) return Plan{512, (int)ctas};
  auto waves_percent = [&](int64_t parts, int64_t per_sm) {
    if (sampler == 0) return 200;
    if (mask) return parts == 1 || esize == 4 ? 400 : (parts == 2 ? 350 : 270);
    if (sampler == 1) return parts == 1 ? 110 : (parts == 2 ? 101 : 87);
    return parts >= 3 && esize == 2 && per_sm < 4 ? 100 : 110;
  };
  for (ctas = 1; ctas <= 8; ++ctas) {
    if (!fits(ctas, 70 * 1024)) continue;
    const int64_t smem = chunk_of(V, ctas) * esize + 6 * 1024, per_sm = 227 * 1024 / smem < 4 ? 227 * 1024 / smem : 4;
    if (rows * ctas * 100 <= per_sm * sms * waves_percent(ctas, per_sm)) return Plan{256, (int)ctas};
  }
  // one block a row
  const int64_t row = chunk_of(V, 1) * esize;
  if ((mask || sampler == 0) && row >= 32 * 1024 && row <= kChunkBytes) {
    const int64_t threads = row <= 70 * 1024 ? 256 : 512, fit = 227 * 1024 / (row + 6 * 1024);
    const int64_t per_sm = fit < 1024 / threads ? fit : 1024 / threads;
    const int64_t waves = sampler == 0 ? 4 : (row <= 64 * 1024 ? 7 : 5);
    if (rows <= waves * per_sm * sms) return Plan{(int)threads, 1};
  }
  return Plan{0, 0};
}

}  // namespace

int direct_ctas(int64_t rows, int64_t V, int dtype, int sampler, bool mask, int sms, int largest) {
  const Plan w = plan(rows, V, dtype == 0 ? 4 : 2, sampler, mask, sms);
  return w.ctas <= largest ? w.ctas : 0;
}

cudaError_t launch_rows_direct(const RowsParams &p, int64_t rows, int dtype, int sampler, const RowStall &stall, cudaStream_t stream, bool &taken) {
  static std::atomic<int> sms[64];
  taken = false;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  int count = sms[dev].load();
  if (count == 0) {
    e = cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    sms[dev].store(count);
  }
  const Plan w = plan(rows, p.V, dtype == 0 ? 4 : 2, sampler, p.mask != nullptr, count);
  if (w.threads == 0) return cudaSuccess;
  auto go = [&](auto threads) {
    constexpr int T = decltype(threads)::value;
    if (dtype == 0) {
      if (sampler < 0) return launch<0, -1, T>(p, rows, w.ctas, dev, stall, stream, taken);
      return sampler == 0 ? launch<0, 0, T>(p, rows, w.ctas, dev, stall, stream, taken) : launch<0, 1, T>(p, rows, w.ctas, dev, stall, stream, taken);
    }
    if (sampler < 0) return launch<1, -1, T>(p, rows, w.ctas, dev, stall, stream, taken);
    return sampler == 0 ? launch<1, 0, T>(p, rows, w.ctas, dev, stall, stream, taken) : launch<1, 1, T>(p, rows, w.ctas, dev, stall, stream, taken);
  };
  return w.threads == 256 ? go(std::integral_constant<int, 256>()) : go(std::integral_constant<int, 512>());
}

}  // namespace e3
