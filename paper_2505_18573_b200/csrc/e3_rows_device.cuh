// Device helpers of the row kernel: shared-memory barriers and copies, Philox, the packed sums of a tile and their
// careful form, the fp32 scores of both samplers, the merging of partial row states and the exact (fp64) paths.
#pragma once
#include "e3_rows.cuh"

#include <cuda_bf16.h>
#include <limits.h>
#include <math_constants.h>
#include <string.h>

namespace e3 {
namespace {

using u64 = unsigned long long;
using f2 = float2;  // two fp32 values in a register pair

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2f = 0.6931471805599453f;
constexpr double kLn2 = 0.6931471805599453094;
// Largest Gumbel value an entry whose coarse byte is below 255 can reach is -ln(-ln(255/256)) = 5.54322...;
// with all 40 bits set the largest value is -ln(-ln(1 - 2^-41)) = 28.41903...  Both rounded up.
constexpr float kGumbelCapCoarse = 5.5433f;
constexpr float kGumbelCapAll = 28.4192f;
// A tile's sums refer to a reference logit R: t = (z - R) c.  R comes from a sample of the strip, the margin (log2 units) puts it
// above most of what the sample may have missed.  A lane's sum of 2^t above the limit (or NaN) means that it has missed an
// entry with t near 7 or more: the tile is then taken again with its largest logit as R.  So |W/Z| stays
// small and the entropy ln Z - ln2 W/Z is free of cancellation at the 1e-5 level.
constexpr float kMargin = 5.f;
constexpr float kSoundZ = 128.f;
constexpr float kSoundW = 1e30f;  // |sum 2^t t| of a sound tile stays far below (a -inf logit makes it NaN)
// From this size of R c on (a fill value such as -1e9 with nothing else beside it) the reference is "far": fp32 logits that differ lie 64
// or more apart in log2 units and the rounding of R c is as large, so the sum is the number of entries that equal R.
constexpr float kFar = 0x1p30f;
constexpr float kFarMost = 0x1p103f;  // references are kept below this: their distance times a sum is finite
constexpr float kClampAt = -0x1p60f;  // smaller logits enter the clamped sums as this: its product with c is finite from tau = 1e-20 on
constexpr float kFloatMost = 3.402823466e38f;

enum : int { kErrValue = 1 };
// What a warp of the streaming kernel knows of the rows' strips in hand.  kClamped: full tiles do not take the plain sums (an entry of -inf
// was seen, or the reference is far).
enum : uint32_t { kGreedy = 1u, kUnusable = 2u, kClamped = 4u };

template <int DT>
struct Fmt {
  static constexpr int kEsize = DT == 0 ? 4 : 2;
  static constexpr int kLaneE = kLaneBytes / kEsize;  // entries per thread and tile: 32 fp32 / 64 bf16
  static constexpr int kTileE = 32 * kLaneE;          // entries per tile: 1,024 / 2,048
  static constexpr int kVG = kEsize;                  // 16-byte vectors per group of 16 entries: 4 / 2
  static constexpr int kG = 8 / kVG;                  // groups per thread and tile: 2 / 4
  static constexpr int kLB = 256 / kLaneE;            // lanes that hold one block of sampler 1: 8 / 4
  static constexpr int kBT = kTileE / 256;            // blocks per tile: 4 / 8
};

// One partial row state.  In the workspace it is kPieceWords 64-bit words, each (tag << 32 | payload):
// the tag depends on the call and on the word, so a reader knows word by word whether what it sees was
// written by this call (64-bit accesses are single-copy atomic); stale or half-written pieces fail the check.
struct Piece {
  float M, Z, W;   // reference (log2 units), sum 2^t, sum 2^t t
  float zf;        // logit of entry tb[0] (sampler 0; training side: of the target)
  int err;
  float zmax;      // largest logit (only where the mean logit gap is asked for)
  float ty[3];     // the three best scores (fp32): sampler 0 entries, sampler 1 blocks; greedy rows: ty[0] = largest logit
  int tb[3];       // ... and their vocabulary / block indices, -1 = none
};
constexpr int kPieceWords = 12;
static_assert(sizeof(Piece) == kPieceWords * 4, "piece payload");
static_assert(kPieceWords * 8 <= kPieceBytes, "piece size");

// Bound on |fp32 score - exact score|: rounding of 1/tau, of the fused product-sum, of the integer
// conversions and of the two approximate logarithms (worst for coarse byte 254: 1.1e-4).
// k = 1 in normal operation; the audit sampler passes a large k, which sends most rows to the exact path.
__device__ __forceinline__ float score_slack(float y, float k) { return k * (1.7e-4f + 1e-6f * fabsf(y)); }

// ---------------------------------------------------------------------------------------------
// small helpers
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2f(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Packed fp32 arithmetic: both halves of a register pair in one instruction.
__device__ __forceinline__ f2 pack2f(float lo, float hi) { return make_float2(lo, hi); }
__device__ __forceinline__ float sum2(f2 v) { return v.x + v.y; }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
template <int DT>
__device__ __forceinline__ float lds_elem(uint32_t addr) {
  if (DT == 0) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
  }
  unsigned short h;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(h) : "r"(addr));
  return __uint_as_float((uint32_t)h << 16);
}

__device__ __forceinline__ void mbar_init(u64 *b, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
// Arrives on `b` and announces the bytes of the bulk copies that complete on it.
__device__ __forceinline__ void mbar_arrive_expect(u64 *b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(b)), "r"(bytes) : "memory");
}
// One poll (the hardware may park the thread for a short, implementation-defined time; a loop of these
// needs no sleep of its own, and a warp that has slept with nanosleep runs slowly for a while afterwards).
__device__ __forceinline__ bool mbar_try_wait(u64 *b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bulk asynchronous copy global -> this CTA's shared memory; completion is counted in bytes on `bar`.
// The logits are read once: their lines are marked evict-first in L2, so that the stream does not push out what
// is used again and again (the kernel's instructions, the workspace, temperatures) -- an L2 miss of any of
// those waits behind the whole queue of the stream.
__device__ __forceinline__ u64 l2_evict_first_policy() {
  u64 pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst, const void *src, uint32_t bytes, u64 *bar, u64 policy) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(policy)
               : "memory");
}
// Orders the thread's earlier shared-memory writes before later reads of the asynchronous proxy (bulk copies).
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---------------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11) with precomputed round keys.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox(const uint32_t *rk, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint64_t a = (uint64_t)c0 * 0xD2511F53u;
    const uint64_t b = (uint64_t)c2 * 0xCD9E8D57u;
    const uint32_t y0 = (uint32_t)(b >> 32) ^ c1 ^ rk[2 * r];
    const uint32_t y2 = (uint32_t)(a >> 32) ^ c3 ^ rk[2 * r + 1];
    c1 = (uint32_t)b;
    c3 = (uint32_t)a;
    c0 = y0;
    c2 = y2;
  }
  return make_uint4(c0, c1, c2, c3);
}

// Calls whose counter words 1..3 are the same for a whole row: the two multiplications of the first two rounds that
// see only those words are taken out of the loop over the calls.
struct PhiloxRow {
  uint32_t x1, y0, x2, y2;
};
__device__ __forceinline__ PhiloxRow philox_row(const uint32_t *rk, uint32_t c1, uint32_t c2, uint32_t c3) {
  const uint64_t b = (uint64_t)c2 * 0xCD9E8D57u;
  const uint64_t a2 = (uint64_t)((uint32_t)(b >> 32) ^ c1 ^ rk[0]) * 0xD2511F53u;
  PhiloxRow r;
  r.x1 = c3 ^ rk[1];
  r.y0 = (uint32_t)b ^ rk[2];
  r.x2 = (uint32_t)(a2 >> 32) ^ rk[3];
  r.y2 = (uint32_t)a2;
  return r;
}
// philox(rk, call, c1, c2, c3) for the words philox_row was given.
__device__ __forceinline__ uint4 philox_call(const uint32_t *rk, const PhiloxRow &row, uint32_t call) {
  const uint64_t a1 = (uint64_t)call * 0xD2511F53u;
  const uint64_t b2 = (uint64_t)((uint32_t)(a1 >> 32) ^ row.x1) * 0xCD9E8D57u;
  uint32_t c0 = (uint32_t)(b2 >> 32) ^ row.y0, c1 = (uint32_t)b2;
  uint32_t c2 = row.x2 ^ (uint32_t)a1, c3 = row.y2;
#pragma unroll
  for (int r = 2; r < 10; ++r) {
    const uint64_t a = (uint64_t)c0 * 0xD2511F53u;
    const uint64_t b = (uint64_t)c2 * 0xCD9E8D57u;
    const uint32_t y0 = (uint32_t)(b >> 32) ^ c1 ^ rk[2 * r];
    const uint32_t y2 = (uint32_t)(a >> 32) ^ c3 ^ rk[2 * r + 1];
    c1 = (uint32_t)b;
    c3 = (uint32_t)a;
    c0 = y0;
    c2 = y2;
  }
  return make_uint4(c0, c1, c2, c3);
}

__device__ __forceinline__ uint32_t pick_word(const uint4 &w, int k) {
  return k == 0 ? w.x : (k == 1 ? w.y : (k == 2 ? w.z : w.w));
}
// Bit 7 of every byte that equals 0xFF (exact).
__device__ __forceinline__ uint32_t ff_bytes(uint32_t w) { return w & 0x80808080u & ((w & 0x7F7F7F7Fu) + 0x01010101u); }

__device__ __forceinline__ int enc_float(float f) {
  int b = __float_as_int(f);
  return b >= 0 ? b : (b ^ 0x7FFFFFFF);
}
__device__ __forceinline__ float dec_float(int e) { return __int_as_float(e >= 0 ? e : (e ^ 0x7FFFFFFF)); }
__device__ __forceinline__ int enc_neg_inf() { return enc_float(-CUDART_INF_F); }

// ---------------------------------------------------------------------------------------------
// Loads
// ---------------------------------------------------------------------------------------------
template <int DT>
__device__ __forceinline__ float load_elem(const char *row, int64_t i) {
  if (DT == 0) return __ldg(reinterpret_cast<const float *>(row) + i);
  return __uint_as_float((uint32_t)__ldg(reinterpret_cast<const unsigned short *>(row) + i) << 16);
}

// 16 consecutive logits of a tile in shared memory (plain order).
template <int DT>
__device__ __forceinline__ void load_group_smem(uint32_t addr, float (&z)[16]) {
  if (DT == 0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 v = lds128(addr + 16 * q);
      z[4 * q] = __uint_as_float(v.x); z[4 * q + 1] = __uint_as_float(v.y);
      z[4 * q + 2] = __uint_as_float(v.z); z[4 * q + 3] = __uint_as_float(v.w);
    }
  } else {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const uint4 v = lds128(addr + 16 * q);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        z[8 * q + 2 * j] = __uint_as_float(w[j] << 16);
        z[8 * q + 2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Sums of a tile
// ---------------------------------------------------------------------------------------------
// A thread's 128 bytes of a tile (its slice): B = shared-memory address of the slice with (lane mod 8) << 4 or-ed in;
// the vector at B xor (i << 4) is 16-byte vector number i xor (lane mod 8) of the slice (eight neighbouring lanes
// then read from distinct banks).

// Largest of the logits of some 16-byte vectors (NaN entries are passed over).
template <int DT, int N>
__device__ __forceinline__ float vec_max(const uint4 (&v)[N]) {
  if (DT == 1) {
    uint32_t m0 = v[0].x, m1 = v[0].y;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (i > 0) {
        asm("max.bf16x2 %0, %1, %2;" : "=r"(m0) : "r"(m0), "r"(v[i].x));
        asm("max.bf16x2 %0, %1, %2;" : "=r"(m1) : "r"(m1), "r"(v[i].y));
      }
      asm("max.bf16x2 %0, %1, %2;" : "=r"(m0) : "r"(m0), "r"(v[i].z));
      asm("max.bf16x2 %0, %1, %2;" : "=r"(m1) : "r"(m1), "r"(v[i].w));
    }
    asm("max.bf16x2 %0, %1, %2;" : "=r"(m0) : "r"(m0), "r"(m1));
    return fmaxf(__uint_as_float(m0 << 16), __uint_as_float(m0 & 0xFFFF0000u));
  } else {
    float m = -CUDART_INF_F;
#pragma unroll
    for (int i = 0; i < N; ++i)
      m = fmaxf(fmaxf(m, fmaxf(__uint_as_float(v[i].x), __uint_as_float(v[i].y))),
                fmaxf(__uint_as_float(v[i].z), __uint_as_float(v[i].w)));
    return m;
  }
}
// Largest finite logit over the lanes (-inf when there is none; a lane whose largest is +inf is passed over, the sums flag it).
__device__ __forceinline__ float warp_max(float lane_max) {
  if (!(lane_max < CUDART_INF_F)) lane_max = -CUDART_INF_F;
  return dec_float(__reduce_max_sync(0xffffffffu, enc_float(lane_max)));
}

// Adds the packed sums of 2^t and of 2^t t over the entries of one 16-byte vector, t = z c + nRc.  CLAMP: logits below -2^60
// (also -inf) enter as -2^60, which gives them weight 0 and keeps 2^t t finite; NaN stays NaN.
template <int DT, bool CLAMP>
__device__ __forceinline__ void vec_sums(const uint4 &v, f2 c2, f2 nRc2, f2 &Za, f2 &Zb, f2 &Wa, f2 &Wb) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < (DT == 1 ? 4 : 2); ++j) {
    f2 z2;
    if (DT == 1) {
      uint32_t x = w[j];
      if (CLAMP) asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(x) : "r"(x), "r"(0xDD80DD80u));
      z2 = pack2f(__uint_as_float(x << 16), __uint_as_float(x & 0xFFFF0000u));
    } else {
      float a = __uint_as_float(w[2 * j]), b = __uint_as_float(w[2 * j + 1]);
      if (CLAMP) {
        asm("max.NaN.f32 %0, %1, %2;" : "=f"(a) : "f"(a), "f"(kClampAt));
        asm("max.NaN.f32 %0, %1, %2;" : "=f"(b) : "f"(b), "f"(kClampAt));
      }
      z2 = pack2f(a, b);
    }
    const f2 t2 = fma2(z2, c2, nRc2);
    const f2 e2 = pack2f(ex2f(t2.x), ex2f(t2.y));
    if (j & 1) { Zb = add2(Zb, e2); Wb = fma2(e2, t2, Wb); } else { Za = add2(Za, e2); Wa = fma2(e2, t2, Wa); }
  }
}

// Sums of a whole slice: Z = sum 2^t, W = sum 2^t t.  A loop over the two halves of the slice: a body short enough for the
// instruction cache.
template <int DT, bool CLAMP = false>
__device__ __forceinline__ void slice_sums(uint32_t B, float c, float nRc, float &Z, float &W) {
  const f2 c2 = pack2f(c, c), nRc2 = pack2f(nRc, nRc);
  f2 Za = pack2f(0.f, 0.f), Zb = Za, Wa = Za, Wb = Za;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    uint4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = lds128((B ^ (uint32_t)(h * 64)) ^ (uint32_t)(i << 4));
#pragma unroll
    for (int i = 0; i < 4; ++i) vec_sums<DT, CLAMP>(v[i], c2, nRc2, Za, Zb, Wa, Wb);
  }
  Z = sum2(add2(Za, Zb));
  W = sum2(add2(Wa, Wb));
}
// The same with the sum of 2^t of every group of 16 entries: Zg[j] belongs to group j xor ((lane mod 8) / vectors per group).
template <int DT, bool CLAMP = false>
__device__ __forceinline__ void slice_sums_groups(uint32_t B, float c, float nRc, float &Z, float &W, float (&Zg)[Fmt<DT>::kG]) {
  const f2 c2 = pack2f(c, c), nRc2 = pack2f(nRc, nRc);
  f2 Wa = pack2f(0.f, 0.f), Wb = Wa, Zt = Wa;
#pragma unroll
  for (int j = 0; j < Fmt<DT>::kG; ++j) {
    f2 Za = pack2f(0.f, 0.f), Zb = Za;
#pragma unroll
    for (int i = j * Fmt<DT>::kVG; i < (j + 1) * Fmt<DT>::kVG; ++i)
      vec_sums<DT, CLAMP>(lds128(B ^ (uint32_t)(i << 4)), c2, nRc2, Za, Zb, Wa, Wb);
    Za = add2(Za, Zb);
    Zg[j] = sum2(Za);
    Zt = add2(Zt, Za);
  }
  Z = sum2(Zt);
  W = sum2(add2(Wa, Wb));
}
// Largest logit of a slice.
template <int DT>
__device__ __forceinline__ float slice_max(uint32_t B) {
  float m = -CUDART_INF_F;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    uint4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = lds128((B ^ (uint32_t)(h * 64)) ^ (uint32_t)(i << 4));
    m = fmaxf(m, vec_max<DT>(v));
  }
  return m;
}

// -R c, rounded down: no entry up to R has t above 0, however large R c is (rounded to nearest, a group of entries of -1e9 had t up to
// +32, and sums beyond any limit).
__device__ __forceinline__ float reference(float R, float c) {
  return fminf(fmaxf(__fmul_rd(-R, c), -kFarMost), kFarMost);
}
// t = z c + n for entries beside a largest logit R whose R c is far: 0 for R, -64 and less for the others (both products are exact,
// and those of clamped entries finite).  An R below the clamp becomes the clamp, as its entries do.
__device__ __forceinline__ void far_terms(float R, float &c, float &n) {
  R = fmaxf(R, kClampAt);
  const int k = 31 + 127 - (int)((__float_as_uint(R) >> 23) & 255u);
  c = __uint_as_float((uint32_t)((k < 66 ? k : 66) + 127) << 23);
  n = -R * c;
}
// Entries that equal R among the `valid` first ones from `addr` on (at most 16); NaN where there is a NaN or a +inf.
template <int DT>
__device__ __forceinline__ float far_count(uint32_t addr, int valid, float R) {
  float n = 0.f;
#pragma unroll 1
  for (int e = 0; e < kGroup && e < valid; ++e) {
    const float z = lds_elem<DT>(addr + (uint32_t)(e * Fmt<DT>::kEsize));
    n += z == R ? 1.f : 0.f;
    if (!(z < CUDART_INF_F)) n = CUDART_NAN_F;
  }
  return n;
}

// -R c for a strip's reference R from a sample, the lanes' first vectors; +inf: none (no finite entry there, or one that is far).
template <int DT>
__device__ __forceinline__ float sample_reference(uint32_t B, float c) {
  const uint4 v[1] = {lds128(B)};
  const float up = __fmaf_rd(-warp_max(vec_max<DT>(v)), c, -kMargin);
  return fabsf(up) < kFar ? up : CUDART_INF_F;
}
// Moves a strip's reference down to `up`, if it lies above, and rescales its sums.
__device__ __forceinline__ void lower_reference(float up, float &nRc, float &Zs, float &Ws) {
  if (up < nRc) {
    const float d = up - nRc, f = nRc == CUDART_INF_F ? 0.f : ex2f(d);
    Ws = f == 0.f ? 0.f : f * fmaf(d, Zs, Ws);
    Zs = f == 0.f ? 0.f : f * Zs;
    nRc = up;
  }
}
__device__ __forceinline__ bool is_far(float nRc) { return fabsf(nRc) >= kFar && nRc < CUDART_INF_F; }
// The same for the logit R; false (nothing done) when there is none or R c is far.
__device__ __forceinline__ bool move_reference(float R, float c, float &nRc, float &Zs, float &Ws) {
  const float up = __fmul_rd(-R, c);
  if (!(fabsf(up) < kFar)) return false;
  lower_reference(up, nRc, Zs, Ws);
  return true;
}

// Bit k: entry k of the vector is above the gate (bf16: above the gate rounded down to bf16, which is the same).
template <int DT>
__device__ __forceinline__ uint32_t entries_above(const uint4 &v, float gate) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  uint32_t bits = 0u;
  if (DT == 1) {
    const __nv_bfloat162 g = __bfloat162bfloat162(__float2bfloat16_rd(gate));
#pragma unroll
    for (int j = 0; j < 4; ++j)
      bits |= __hgt2_mask(*reinterpret_cast<const __nv_bfloat162 *>(&w[j]), g) & ((1u << (2 * j)) | (0x20000u << (2 * j)));
    bits = (bits | bits >> 16) & 0xFFu;
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) bits |= (__uint_as_float(w[j]) > gate ? 1u : 0u) << j;
  }
  return bits;
}

// The vector number i (counted from 0 to 7 in vocabulary order) of a slice of which the first nlane entries are valid:
// the others become -inf.
template <int DT>
__device__ __forceinline__ uint4 mask_vec(const uint4 &v, int nlane, int i) {
  uint32_t w[4] = {v.x, v.y, v.z, v.w};
  const int rem = nlane - (DT == 1 ? 8 : 4) * i;  // entries of this vector that are valid
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (DT == 1) {
      w[j] = (2 * j < rem ? (w[j] & 0xFFFFu) : 0xFF80u) | (2 * j + 1 < rem ? (w[j] & 0xFFFF0000u) : 0xFF800000u);
    } else {
      w[j] = j < rem ? w[j] : 0xFF800000u;
    }
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// The careful form, for a tile that lies only partly inside the row, for one whose sums stay out of range clamped and with its
// largest logit as reference (a NaN, a +inf), and for one whose reference is far: entries are masked and clamped.  One vector per
// step, so that the code that few tiles run stays short.
template <int DT>
__device__ __forceinline__ float slice_max_careful(uint32_t B, int nlane, int r8) {
  float m = -CUDART_INF_F;
#pragma unroll 1
  for (int i = 0; i < 8; ++i) {
    const uint4 v[1] = {mask_vec<DT>(lds128(B ^ (uint32_t)(i << 4)), nlane, i ^ r8)};
    m = fmaxf(m, vec_max<DT>(v));
  }
  return m;
}
template <int DT>
__device__ __forceinline__ void slice_sums_careful(uint32_t B, int nlane, int r8, float c, float nRc, float &Z, float &W,
                                                   float (&Zg)[Fmt<DT>::kG]) {
  const f2 c2 = pack2f(c, c), nRc2 = pack2f(nRc, nRc);
  f2 Wa = pack2f(0.f, 0.f), Wb = Wa;
  Z = 0.f;
#pragma unroll
  for (int j = 0; j < Fmt<DT>::kG; ++j) Zg[j] = 0.f;
#pragma unroll 1
  for (int i = 0; i < 8; ++i) {
    f2 Za = pack2f(0.f, 0.f), Zb = Za;
    vec_sums<DT, true>(mask_vec<DT>(lds128(B ^ (uint32_t)(i << 4)), nlane, i ^ r8), c2, nRc2, Za, Zb, Wa, Wb);
    const float z = sum2(add2(Za, Zb));
    Z += z;
#pragma unroll
    for (int j = 0; j < Fmt<DT>::kG; ++j) Zg[j] += i / Fmt<DT>::kVG == j ? z : 0.f;
  }
  W = sum2(add2(Wa, Wb));
}

// The lane's groups of a tile whose reference is far: how many of their entries equal R.
template <int DT>
struct FarTile {
  float Zg[Fmt<DT>::kG];
};
template <int DT>
__device__ __noinline__ FarTile<DT> far_tile(uint32_t B, int nlane, float R) {
  FarTile<DT> f;
#pragma unroll
  for (int j = 0; j < Fmt<DT>::kG; ++j) {
    const int g = j ^ ((int)(threadIdx.x & 7) / Fmt<DT>::kVG);
    f.Zg[j] = far_count<DT>((B & ~(uint32_t)(kLaneBytes - 1)) + (uint32_t)(g * kGroup * Fmt<DT>::kEsize), nlane - g * kGroup, R);
  }
  return f;
}

// Sums of a tile in the careful form; the strip's reference moves up to the tile's largest logit first (zmax takes it in).  True: a
// NaN, a +inf, or numbers outside the fp32 range (the sums are 0 then).
template <int DT>
__device__ __forceinline__ bool careful_tile(uint32_t B, int n, float c, float &nRc, float &Zs, float &Ws, float &Z, float &W,
                                             float (&Zg)[Fmt<DT>::kG], float &zmax) {
  const int lane = threadIdx.x & 31, nlane = n - lane * Fmt<DT>::kLaneE;  // entries from the lane's first on (may be < 0)
  const float R = warp_max(slice_max_careful<DT>(B, nlane, lane & 7));
  zmax = fmaxf(zmax, R);
  const float up = reference(R, c);
  bool bad = !(c < CUDART_INF_F);
  if (R > -CUDART_INF_F && !bad) lower_reference(up, nRc, Zs, Ws);
  // without any reference (nothing finite so far) the sums must come out as zero
  const bool none = nRc == CUDART_INF_F;
  if (is_far(nRc)) {  // (a tile below the reference counts nothing)
    const FarTile<DT> f = far_tile<DT>(B, nlane, up == nRc ? R : CUDART_INF_F);
    Z = W = 0.f;
#pragma unroll
    for (int j = 0; j < Fmt<DT>::kG; ++j) {
      Zg[j] = f.Zg[j];
      Z += Zg[j];
    }
  } else {
    slice_sums_careful<DT>(B, nlane, lane & 7, c, none ? 0.f : nRc, Z, W, Zg);
  }
  bad |= !(Z <= kSoundZ) || !(fabsf(W) <= kSoundW) || (none && Z != 0.f);
  bad = __any_sync(0xffffffffu, bad);
  if (bad) {
    Z = W = 0.f;
#pragma unroll
    for (int j = 0; j < Fmt<DT>::kG; ++j) Zg[j] = 0.f;
  }
  return bad;
}

// Sums of a tile that the streaming loop's plain form does not give: with a -inf, a NaN or a +inf, and with CAREFUL one that lies
// only partly inside the row or has an entry far above the strip's reference (`over`: the reference moves first).  A full tile is
// summed with clamped entries in the plain form's order, its reference following the same steps: the same bits where no
// entry is that low.
// Out of line: the streaming loop stays short (bound by issue and instruction fetch).  us with it inside the loop, with the clamped
// sums alone out of line, and with all of it: statistics 4,096 x 151,936 bf16 211, 208, 204, token sampler 512 rows 88.5, 88.5,
// 85.5; the blocked sampler 4,096 rows 230 with the clamped sums alone, 250 with all of it.  A tenth of the logits -inf, 2,048 rows, one
// vector at a time and now: statistics 222 and 126, blocked 248 and 145, token sampler 421 and 298.
template <int DT>
struct SlowTile {
  float Zs, Ws, nRc;  // the strip's sums and reference, moved
  float Z, W, zmax;
  float Zg[Fmt<DT>::kG];
  int flags;          // kErrValue: not summed (a NaN, a +inf, or numbers outside the fp32 range); kClamped: see there
};
template <int DT, bool GROUPS, bool CAREFUL>
__device__ __noinline__ SlowTile<DT> tile_slow(uint32_t B, int n, bool over, bool want_max, float c, float nRc, float Zs, float Ws) {
  SlowTile<DT> s;
  s.zmax = -CUDART_INF_F;
  bool bad = true;
  if ((!CAREFUL || n == Fmt<DT>::kTileE) && !is_far(nRc)) {
    if (nRc == CUDART_INF_F && !over) nRc = sample_reference<DT>(B, c);
    bool moved = over || nRc == CUDART_INF_F;
#pragma unroll 1
    for (;;) {
      bool none = false;  // no finite entry so far: the sums must come out as 0
      if (moved) {
        const float R = warp_max(slice_max<DT>(B));
        none = R == -CUDART_INF_F && nRc == CUDART_INF_F;
        if (!none && !move_reference(R, c, nRc, Zs, Ws)) break;
      }
      if (GROUPS) slice_sums_groups<DT, true>(B, c, none ? 0.f : nRc, s.Z, s.W, s.Zg);
      else slice_sums<DT, true>(B, c, none ? 0.f : nRc, s.Z, s.W);
      bad = __any_sync(0xffffffffu, !(s.Z <= (none ? 0.f : kSoundZ)) || !(fabsf(s.W) <= kSoundW));
      if (!bad || moved) break;
      moved = true;
    }
    if (!bad && want_max) s.zmax = warp_max(slice_max<DT>(B));
  }
  if (CAREFUL && bad) bad = careful_tile<DT>(B, n, c, nRc, Zs, Ws, s.Z, s.W, s.Zg, s.zmax);
  s.Zs = Zs; s.Ws = Ws; s.nRc = nRc;
  s.flags = (bad ? kErrValue : 0) | (is_far(nRc) ? (int)kClamped : 0);
  return s;
}

// The 16 bytes that begin `a` bytes (1..15) into the 32 bytes x, y.
__device__ __forceinline__ uint4 shift_vec(const uint4 &x, const uint4 &y, uint32_t a) {
  const uint32_t q = a >> 2, sh = (a & 3u) * 8u;
  uint32_t w[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
  if (q & 2u) {
#pragma unroll
    for (int k = 0; k < 6; ++k) w[k] = w[k + 2];
  }
  if (q & 1u) {
#pragma unroll
    for (int k = 0; k < 5; ++k) w[k] = w[k + 1];
  }
  return make_uint4(__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh), __funnelshift_r(w[2], w[3], sh),
                    __funnelshift_r(w[3], w[4], sh));
}

// A tile that begins `a` bytes (1..15) behind a 16-byte boundary was copied from that boundary on: moves it down by a
// bytes within its slot (the 16 bytes behind the slot are in `spill`), 16 bytes per lane and step (the reads of a step lie at or
// above its writes and below those of the next).
__device__ __noinline__ void realign_tile(uint32_t base, uint32_t spill, uint32_t a) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int i = 0; i < 8; ++i) {
    const uint32_t addr = base + (uint32_t)(i * 512 + lane * 16);
    const uint4 o = shift_vec(lds128(addr), lds128(i == 7 && lane == 31 ? spill : addr + 16), a);
    __syncwarp();
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(o.x), "r"(o.y), "r"(o.z), "r"(o.w) : "memory");
    __syncwarp();
  }
  fence_async_smem();  // the next bulk copy into the slot comes after these stores
}

// Greedy rows (tau = 0): largest logit of the warp's tile, lowest index (-1: nothing finite, -2: a NaN or a +inf).
struct Greedy {
  float y;
  int i;
};
template <int DT>
__device__ __noinline__ Greedy tile_greedy(uint32_t B, int e_lane, int nlane, int r8) {
  float ybest = -CUDART_INF_F;
  int ibest = INT_MAX;
  bool bad = false;
#pragma unroll 1
  for (int i = 0; i < 8; ++i) {
    const uint4 v = mask_vec<DT>(lds128(B ^ (uint32_t)(i << 4)), nlane, i ^ r8);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    const int e0 = e_lane + (i ^ r8) * (DT == 1 ? 8 : 4);
#pragma unroll
    for (int k = 0; k < (DT == 1 ? 8 : 4); ++k) {
      const float z = DT == 1 ? __uint_as_float((k & 1) ? (w[k >> 1] & 0xFFFF0000u) : (w[k >> 1] << 16)) : __uint_as_float(w[k]);
      bad |= !(z < CUDART_INF_F);
      if (z > ybest || (z == ybest && z > -CUDART_INF_F && e0 + k < ibest)) {
        ybest = z;
        ibest = e0 + k;
      }
    }
  }
  ybest += 0.f;  // -0 and +0 are the same logit
  const int e = ibest == INT_MAX ? INT_MIN : enc_float(ybest), emax = __reduce_max_sync(0xffffffffu, e);
  const int imin = __reduce_min_sync(0xffffffffu, e == emax ? ibest : INT_MAX);
  const bool any_bad = __any_sync(0xffffffffu, bad);
  return Greedy{dec_float(emax), any_bad ? -2 : (emax == INT_MIN ? -1 : imin)};
}

// ---------------------------------------------------------------------------------------------
// Scores
// ---------------------------------------------------------------------------------------------
// enc: encoded value that is below the row's best score by at least four slacks.  An entry whose largest possible
// Gumbel is `cap` can only win with a logit above the result.
__device__ __forceinline__ float logit_gate(int enc, float tau, float cap) {
  if (enc == enc_neg_inf()) return -CUDART_INF_F;
  const float t = (dec_float(enc) - cap) * tau;
  return t - fabsf(t) * 1e-6f - 1e-30f;  // two fp32 roundings (<= 1.2e-7 relative) are covered by the 1e-6 relative slack
}

// The gate of the streaming loop: an entry whose coarse byte is below 255 can only win if
// 2^t_i > 2^((B - 5.5433) log2 e - R c); the group sum of 2^t bounds every term from above.  The slack
// covers the fp32 roundings of t_i, of the threshold and of the approximate 2^x.
__device__ __forceinline__ float gate_threshold(int enc, float nRc) {
  if (enc == enc_neg_inf()) return 0.f;
  const float B = dec_float(enc);
  const float a = (B - kGumbelCapCoarse) * kLog2e;
  const float t = a + nRc - (1e-3f + (fabsf(a) + fabsf(nRc)) * 4e-7f);
  return ex2f(t);  // 0 when far below the range (every group with weight passes), +inf when far above
}

struct EvalCtx {
  const uint32_t *rk;
  const char *row;
  float tau, slack_k;
  uint32_t grow, ctr_lo, ctr_hi8;
  int V;
};

// y_i = z_i/tau + g_i of the definition, in fp64 and in its expression order:
// u = (c + (x + 1/2) 2^-32) / 256 (exact), g = -ln(-ln u).
__device__ __noinline__ double exact_score(float zf, float tau, uint32_t cbyte, uint32_t xw) {
  const double u = ((double)cbyte + ((double)xw + 0.5) * 0x1p-32) / 256.0;
  const double s = (double)zf / (double)tau;
  return s + (-log(-log(u)));
}

// fp32 Gumbel variate for coarse byte cbyte, fine word xw.
__device__ __forceinline__ float gumbel_f32(uint32_t cbyte, uint32_t xw) {
  float w;  // -ln u
  if (cbyte == 255u) {
    // 1 - u = (2^32 - x - 1/2) 2^-40 < 2^-8 and -ln u = d + d^2/2 + d^3/3 + ...
    const float d = ((float)(~xw) + 0.5f) * 0x1p-40f;
    w = d * fmaf(d, fmaf(d, 0.33333334f, 0.5f), 1.0f);
  } else {
    const float u = ((float)cbyte + ((float)xw + 0.5f) * 0x1p-32f) * 0.00390625f;
    w = -lg2f(u) * kLn2f;
  }
  return -lg2f(w) * kLn2f;
}
// fp32 value of y_i (within score_slack of the exact value; finite for every finite logit).
__device__ __forceinline__ float score_of(float zf, float inv_tau, float gumbel) {
  return fminf(fmaxf(fmaf(zf, inv_tau, gumbel), -kFloatMost), kFloatMost);
}
__device__ __forceinline__ float score_f32(float zf, float inv_tau, uint32_t cbyte, uint32_t xw) {
  return score_of(zf, inv_tau, gumbel_f32(cbyte, xw));
}

__device__ __forceinline__ bool best_before(float y, int i, float y2, int i2) {
  return i2 < 0 || y > y2 || (y == y2 && i < i2);
}

// ---------------------------------------------------------------------------------------------
// Leaders (entries of sampler 0, blocks of sampler 1)
// ---------------------------------------------------------------------------------------------
struct Top3 {
  float y[3];
  int b[3];
};
__device__ __forceinline__ void top3_reset(Top3 &t) {
  t.y[0] = t.y[1] = t.y[2] = -CUDART_INF_F;
  t.b[0] = t.b[1] = t.b[2] = -1;
}
// order: larger score first, equal scores by lower block index; NaN scores never enter
__device__ __forceinline__ bool top3_before(float y, int b, float y2, int b2) {
  return b2 < 0 || y > y2 || (y == y2 && b < b2);
}
__device__ __forceinline__ void top3_insert(Top3 &t, float y, int b) {
  if (b < 0 || !(y == y)) return;
  if (top3_before(y, b, t.y[0], t.b[0])) {
    t.y[2] = t.y[1]; t.b[2] = t.b[1]; t.y[1] = t.y[0]; t.b[1] = t.b[0]; t.y[0] = y; t.b[0] = b;
  } else if (top3_before(y, b, t.y[1], t.b[1])) {
    t.y[2] = t.y[1]; t.b[2] = t.b[1]; t.y[1] = y; t.b[1] = b;
  } else if (top3_before(y, b, t.y[2], t.b[2])) {
    t.y[2] = y; t.b[2] = b;
  }
}

// fp32 Gumbel variate from a 32-bit word: u = (x + 1/2) 2^-32, g = -ln(-ln u)
__device__ __forceinline__ float gumbel_from_word(uint32_t xw) {
  float a;  // -ln u
  if (xw >= 0xFE000000u) {
    const float d = ((float)(~xw) + 0.5f) * 0x1p-32f;  // 1 - u < 2^-7: series of -ln(1 - d)
    a = d * fmaf(d, fmaf(d, 0.33333334f, 0.5f), 1.0f);
  } else {
    a = -lg2f(((float)xw + 0.5f) * 0x1p-32f) * kLn2f;
  }
  return -lg2f(a) * kLn2f;
}

// ---------------------------------------------------------------------------------------------
// Merging partial states
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void merge_stats_f(float &M, float &Z, float &W, float M2, float Z2, float W2) {
  if (Z2 == 0.f) return;
  if (Z == 0.f) {
    M = M2; Z = Z2; W = W2;
    return;
  }
  const float Mn = fmaxf(M, M2);
  const float d1 = M - Mn, d2 = M2 - Mn;
  const float a = ex2f(d1), b = ex2f(d2);
  W = a * fmaf(d1, Z, W) + b * fmaf(d2, Z2, W2);
  Z = a * Z + b * Z2;
  M = Mn;
}

__device__ __forceinline__ uint32_t piece_tag(u64 call_id, int j) {
  return (uint32_t)((((call_id << 4) | (u64)j) * 0x9E3779B97F4A7C15ull) >> 32);
}

__device__ __forceinline__ void piece_store(u64 *dst, u64 call_id, const Piece &pc) {
  uint32_t w[kPieceWords];
  memcpy(w, &pc, sizeof(Piece));
#pragma unroll
  for (int j = 0; j < kPieceWords; ++j) {
    const u64 v = ((u64)piece_tag(call_id, j) << 32) | w[j];
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(dst + j), "l"(v) : "memory");
  }
}

// False when some word does not carry this call's tag.
__device__ __forceinline__ bool piece_load(const u64 *src, u64 call_id, Piece &pc) {
  u64 v[kPieceWords];
#pragma unroll
  for (int j = 0; j < kPieceWords; ++j)
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v[j]) : "l"(src + j) : "memory");
  uint32_t w[kPieceWords];
  bool ok = true;
#pragma unroll
  for (int j = 0; j < kPieceWords; ++j) {
    ok &= (uint32_t)(v[j] >> 32) == piece_tag(call_id, j);
    w[j] = (uint32_t)v[j];
  }
  memcpy(&pc, w, sizeof(Piece));
  return ok;
}

// Makes a piece unreadable for every call id: word j gets the complement of this call's tag.
__device__ __forceinline__ void piece_wipe(u64 *dst, u64 call_id) {
#pragma unroll
  for (int j = 0; j < kPieceWords; ++j) {
    const u64 v = (u64)(~piece_tag(call_id, j)) << 32;
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(dst + j), "l"(v) : "memory");
  }
}

// Merges the lists of leaders held by the 32 lanes of a warp (sampler 0 entries, sampler 1 blocks, greedy
// maxima); every lane ends with the result, zf follows top.b[0].  Three rounds of "take the best head":
// larger score first, equal scores by lower index.
__device__ __forceinline__ void warp_merge_top(Top3 &top, float &zf) {
  constexpr unsigned kAll = 0xffffffffu;
  Top3 out;
  top3_reset(out);
  int pos = 0;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const float hy = pos == 0 ? top.y[0] : (pos == 1 ? top.y[1] : top.y[2]);
    const int hb = pos >= 3 ? -1 : (pos == 0 ? top.b[0] : (pos == 1 ? top.b[1] : top.b[2]));
    const int e = hb >= 0 ? enc_float(hy) : INT_MIN;
    const int emax = __reduce_max_sync(kAll, e);
    if (emax != INT_MIN) {
      const bool c2 = hb >= 0 && e == emax;
      const int bmin = __reduce_min_sync(kAll, c2 ? hb : INT_MAX);
      out.y[r] = dec_float(emax);
      out.b[r] = bmin;
      const bool mine = c2 && hb == bmin;
      if (r == 0) zf = __shfl_sync(kAll, zf, __ffs(__ballot_sync(kAll, mine)) - 1);
      if (mine) ++pos;
    }
  }
  top = out;
}

// The same, but what lies further than `near` below the largest score is left out (none of it: index -1), which takes one round
// where no two scores are that close.
__device__ __forceinline__ void warp_merge_near(Top3 &top, float near_scale, float near_rel) {
  constexpr unsigned kAll = 0xffffffffu;
  Top3 out;
  top3_reset(out);
  float hy = top.y[0];
  int hb = top.b[0];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int e = hb >= 0 ? enc_float(hy) : INT_MIN, emax = __reduce_max_sync(kAll, e);
    if (emax == INT_MIN) break;
    const float y = dec_float(emax);
    if (r > 0 && !(out.y[0] - y <= near_scale + near_rel * fabsf(out.y[0]))) break;
    const int bmin = __reduce_min_sync(kAll, e == emax ? hb : INT_MAX);
    out.y[r] = y;
    out.b[r] = bmin;
    if (e == emax && hb == bmin) {
      hy = top.y[1]; hb = top.b[1];
      top.y[1] = top.y[2]; top.b[1] = top.b[2];
      top.b[2] = -1;
    }
  }
  top = out;
}

// The leaders of sampler 1: those within twice the margin below which scores are settled in fp64.
__device__ __forceinline__ float near_blocks(float y) { return 2e-4f + 4e-5f * fabsf(y); }
__device__ __forceinline__ void merge_near_blocks(Top3 &top) { warp_merge_near(top, 2e-4f, 4e-5f); }

// Merges the sums and largest logits held by the 32 lanes of a warp; every lane ends with the result.  A lane
// without weight (Z = 0) takes no part.  The order of all sums is fixed by lane numbers.
__device__ __forceinline__ void warp_merge(Piece &pc) {
  constexpr unsigned kAll = 0xffffffffu;
  // softmax sums: move every lane to the largest reference, then add
  const bool has = pc.Z > 0.f;
  const int em = __reduce_max_sync(kAll, has ? enc_float(pc.M) : enc_neg_inf());
  float Mw = 0.f, Zs = 0.f, Ws = 0.f;
  if (em != enc_neg_inf()) {
    Mw = dec_float(em);
    if (has) {
      const float d = pc.M - Mw, a = ex2f(d);
      Zs = a * pc.Z;
      Ws = a * fmaf(d, pc.Z, pc.W);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      Zs += __shfl_xor_sync(kAll, Zs, o);
      Ws += __shfl_xor_sync(kAll, Ws, o);
    }
  }
  pc.M = Mw; pc.Z = Zs; pc.W = Ws;
  pc.zmax = dec_float(__reduce_max_sync(kAll, enc_float(pc.zmax)));
}

// Largest y over the lanes, then lowest index (lanes with idx < 0 take no part); all lanes get the winner.
__device__ __forceinline__ void warp_argmax_double(double &y, int &idx, float &zf) {
  constexpr unsigned kAll = 0xffffffffu;
  const long long bits = __double_as_longlong(y);
  const long long code = bits >= 0 ? bits : (bits ^ 0x7FFFFFFFFFFFFFFFll);  // order-preserving
  bool cand = idx >= 0 && y == y;
  const int hi = cand ? (int)(code >> 32) : INT_MIN;
  const int hmax = __reduce_max_sync(kAll, hi);
  if (hmax == INT_MIN) {
    idx = -1;
    return;
  }
  cand = cand && hi == hmax;
  const unsigned lo = cand ? (unsigned)code : 0u;
  const unsigned lmax = __reduce_max_sync(kAll, lo);
  cand = cand && lo == lmax;
  const int imin = __reduce_min_sync(kAll, cand ? idx : INT_MAX);
  const int src = __ffs(__ballot_sync(kAll, cand && idx == imin)) - 1;
  y = __shfl_sync(kAll, y, src);
  zf = __shfl_sync(kAll, zf, src);
  idx = imin;
}

// ---------------------------------------------------------------------------------------------
// Exact paths
// ---------------------------------------------------------------------------------------------
struct BlockView {
  double s[8];  // z/tau of the lane's entries (-inf beyond the row)
  double m;     // block maximum
};

template <int DT>
__device__ __forceinline__ void load_block(const char *row, int b, int V, double tau, int lane, BlockView &v) {
  double m = -CUDART_INF;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = b * 256 + lane * 8 + k;
    const float z = i < V ? load_elem<DT>(row, i) : -CUDART_INF_F;
    v.s[k] = (double)z / tau;
    m = fmax(m, v.s[k]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  v.m = m;
}

// Y_b = m_b + ln sum exp(s_i - m_b) + g_b in fp64; -inf for a block without mass.
template <int DT>
__device__ __noinline__ double exact_block_score(const EvalCtx &x, int b, int lane) {
  BlockView v;
  load_block<DT>(x.row, b, x.V, (double)x.tau, lane, v);
  if (v.m == -CUDART_INF) return -CUDART_INF;
  double sum = 0.0;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (v.s[k] != -CUDART_INF) sum += exp(v.s[k] - v.m);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const uint4 w = philox(x.rk, (uint32_t)b >> 2, x.grow, x.ctr_lo, x.ctr_hi8 | 2u);
  const double u = ((double)pick_word(w, b & 3) + 0.5) * 0x1p-32;
  return v.m + log(sum) + (-log(-log(u)));
}

// Token inside block b: first entry whose inclusive prefix sum of exp(s_i - m_b) exceeds v * total.
// Exact form (fp64, the definition's expression order).
template <int DT>
__device__ __noinline__ int draw_in_block_exact(const EvalCtx &x, int b, int lane) {
  BlockView v;
  load_block<DT>(x.row, b, x.V, (double)x.tau, lane, v);
  double pre[8];
  double run = 0.0;
  int last_nonzero = -1;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const double w = (v.s[k] != -CUDART_INF) ? exp(v.s[k] - v.m) : 0.0;
    if (w > 0.0) last_nonzero = k;
    run += w;
    pre[k] = run;
  }
  double incl = run;  // inclusive scan of the lane totals
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  const double total = __shfl_sync(0xffffffffu, incl, 31);
  const double before = incl - run;
  const uint4 w3 = philox(x.rk, 0u, x.grow, x.ctr_lo, x.ctr_hi8 | 3u);
  const double t = (((double)w3.x + 0.5) * 0x1p-32) * total;
  int hit = -1;
#pragma unroll
  for (int k = 7; k >= 0; --k)
    if (before + pre[k] > t) hit = k;
  const uint32_t found = __ballot_sync(0xffffffffu, hit >= 0);
  int tok;
  if (found != 0u) {
    const int src = __ffs(found) - 1;
    tok = b * 256 + src * 8 + __shfl_sync(0xffffffffu, hit, src);
  } else {  // rounding left t at or above the total: last entry that carries mass
    const uint32_t any = __ballot_sync(0xffffffffu, last_nonzero >= 0);
    if (any == 0u) return -1;
    const int src = 31 - __clz(any);
    tok = b * 256 + src * 8 + __shfl_sync(0xffffffffu, last_nonzero, src);
  }
  return tok;
}

// The same draw in fp32.  The prefix sums are good to about 3e-6 of the block sum (entries that matter
// have |t| < 25, so the rounding of t costs 2e-6 relative, `ex2` 2e-7, the 13 additions 8e-7); when the
// threshold comes closer than ten times that to a prefix boundary the exact form decides.
// z: the lane's eight logits of the block (-inf beyond the row); word: draw_word(x); z_tok: logit of the token.
__device__ __forceinline__ uint32_t draw_word(const EvalCtx &x) { return philox(x.rk, 0u, x.grow, x.ctr_lo, x.ctr_hi8 | 3u).x; }
template <int DT>
__device__ __forceinline__ int draw_among(const EvalCtx &x, int b, int lane, const float (&z)[8], uint32_t word, float &z_tok) {
  float m = -CUDART_INF_F;
#pragma unroll
  for (int k = 0; k < 8; ++k) m = fmaxf(m, z[k]);
  m = dec_float(__reduce_max_sync(0xffffffffu, enc_float(m)));
  int tok = -1;
  bool exact = !(m > -CUDART_INF_F && m < CUDART_INF_F);
  if (!exact) {
    const float c = __fdiv_rn(kLog2e, x.tau);
    float pre[8];
    float run = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      run += z[k] > -CUDART_INF_F ? ex2f((z[k] - m) * c) : 0.f;
      pre[k] = run;
    }
    float incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    const float total = __shfl_sync(0xffffffffu, incl, 31);
    const float before = incl - run;
    const float t = (float)((((double)word + 0.5) * 0x1p-32) * (double)total);
    int hit = -1;
    float gap = CUDART_INF_F;
#pragma unroll
    for (int k = 7; k >= 0; --k) {
      const float pk = before + pre[k];
      if (pk > t) hit = k;
      gap = fminf(gap, fabsf(pk - t));
    }
    gap = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(gap)));  // (not negative: ordered like its bits)
    const uint32_t found = __ballot_sync(0xffffffffu, hit >= 0);
    exact = !(gap > 3e-5f * total) || found == 0u || !(total > 0.f) || !(total < CUDART_INF_F);
    if (!exact) {
      const int src = __ffs(found) - 1;
      const int k = __shfl_sync(0xffffffffu, hit, src);
      tok = b * 256 + src * 8 + k;
      float zk = z[0];
#pragma unroll
      for (int j = 1; j < 8; ++j) zk = k == j ? z[j] : zk;
      z_tok = __shfl_sync(0xffffffffu, zk, src);
    }
  }
  if (exact) {
    tok = draw_in_block_exact<DT>(x, b, lane);
    z_tok = tok >= 0 ? load_elem<DT>(x.row, tok) : 0.f;
  }
  return tok;
}

template <int DT>
__device__ __noinline__ int draw_in_block(const EvalCtx &x, int b, int lane, float &z_tok) {
  float z[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = b * 256 + lane * 8 + k;
    z[k] = i < x.V ? load_elem<DT>(x.row, i) : -CUDART_INF_F;
  }
  return draw_among<DT>(x, b, lane, z, draw_word(x), z_tok);
}

// Whether the runner-up's score is too close to the leader's for fp32 to decide.
__device__ __forceinline__ float block_margin(const Top3 &top) { return 1e-4f + 2e-5f * fabsf(top.y[0]); }
__device__ __forceinline__ bool blocks_too_close(const Top3 &top) { return top.y[0] - top.y[1] <= block_margin(top); }

// Picks the winning block from the three fp32 leaders (exact scores where they are too close) and
// draws the token.  Returns -1 when the row has no block with mass.
template <int DT>
__device__ __noinline__ int sample_in_blocks(const EvalCtx &x, const Top3 &top, int lane, float &z_tok) {
  if (top.b[0] < 0) return -1;
  int bstar = top.b[0];
  const float margin = block_margin(top);
  if (top.b[1] >= 0 && blocks_too_close(top)) {
    double ybest = -CUDART_INF;
    int bbest = -1;
    if (top.b[2] >= 0 && top.y[0] - top.y[2] <= margin) {
      const int nb = (x.V + 255) / 256;  // more than two contenders: settle all blocks exactly
      for (int b = 0; b < nb; ++b) {
        const double y = exact_block_score<DT>(x, b, lane);
        if (y > ybest) { ybest = y; bbest = b; }
      }
    } else {
      const int lo = top.b[0] < top.b[1] ? top.b[0] : top.b[1], hi = top.b[0] < top.b[1] ? top.b[1] : top.b[0];
      const double y0 = exact_block_score<DT>(x, lo, lane), y1 = exact_block_score<DT>(x, hi, lane);
      bbest = y1 > y0 ? hi : lo;
    }
    if (bbest >= 0) bstar = bbest;
  }
  return draw_in_block<DT>(x, bstar, lane, z_tok);
}

template <int DT>
__device__ __noinline__ int settle_exact(const EvalCtx &x, const Top3 &top, float slack2, int lane, float &z_tok) {
  double ybest = -CUDART_INF;
  int ibest = -1;
  float zbest = 0.f;
  const bool rescan = top.b[2] >= 0 && !(top.y[0] - top.y[2] > slack2);
  if (!rescan) {
    const int i = lane == 0 ? top.b[0] : (lane == 1 ? top.b[1] : -1);
    if (i >= 0) {
      const float z = load_elem<DT>(x.row, i);
      const uint4 cw = philox(x.rk, (uint32_t)i >> 4, x.grow, x.ctr_lo, x.ctr_hi8 | 0u);
      const uint32_t cbyte = (pick_word(cw, (i & 15) >> 2) >> (8 * (i & 3))) & 0xFFu;
      const uint4 fw = philox(x.rk, (uint32_t)i >> 2, x.grow, x.ctr_lo, x.ctr_hi8 | 1u);
      ybest = exact_score(z, x.tau, cbyte, pick_word(fw, i & 3));
      ibest = i;
      zbest = z;
    }
  } else {
    const float inv_tau = __frcp_rn(x.tau);
    const float floor_y = top.y[0] - slack2;
#pragma unroll 1
    for (int q0 = lane * 4; q0 < x.V; q0 += 128) {  // four entries (one fine call) per lane and round
      const uint4 cw = philox(x.rk, (uint32_t)q0 >> 4, x.grow, x.ctr_lo, x.ctr_hi8 | 0u);
      const uint32_t cword = pick_word(cw, (q0 & 15) >> 2);
      const uint4 fw = philox(x.rk, (uint32_t)q0 >> 2, x.grow, x.ctr_lo, x.ctr_hi8 | 1u);
#pragma unroll 1
      for (int k = 0; k < 4 && q0 + k < x.V; ++k) {
        const float z = load_elem<DT>(x.row, q0 + k);
        if (!(z > -CUDART_INF_F && z < CUDART_INF_F)) continue;
        const uint32_t cbyte = (cword >> (8 * k)) & 0xFFu, xw = pick_word(fw, k);
        if (!(score_f32(z, inv_tau, cbyte, xw) >= floor_y)) continue;
        const double y = exact_score(z, x.tau, cbyte, xw);
        if (ibest < 0 || y > ybest) {  // indices ascend within a lane
          ybest = y;
          ibest = q0 + k;
          zbest = z;
        }
      }
    }
  }
  warp_argmax_double(ybest, ibest, zbest);
  z_tok = zbest;
  return ibest;
}

__device__ __forceinline__ const char *row_ptr(const RowsParams &p, uint32_t row) { return p.logits + (size_t)row * (size_t)p.row_bytes; }

// ---------------------------------------------------------------------------------------------
// Row states and results
// ---------------------------------------------------------------------------------------------
struct RowInfo {
  float c;
  bool greedy;
};

// One thread, fp64.  zt: logit of the token whose log-probability is wanted.
__device__ __forceinline__ void finish_row(const RowsParams &p, uint32_t row, const RowInfo &ri, float Mf, float Zf,
                                           float Wf, float zmax, int idx, int err, bool have_zt, float zt) {
  const double M = Mf, Z = Zf, W = Wf;
  // z c - M; where the reference is far the product is rounded like it, so that the largest logit gives 0 (in line: a call, which only far
  // rows would make, cost 20,000 x 11,124 bf16 128 -> 131 us)
  const bool far = fabsf(Mf) >= kFar;
  auto above = [&](float z) { return (far ? -(double)reference(z, ri.c) : (double)z * (double)ri.c) - M; };
  const bool sample = p.mode == kModeSample;
  int tok = -1;
  float logp = CUDART_NAN_F, ent = CUDART_NAN_F, gap = CUDART_NAN_F;
  if (ri.greedy) {
    if (err == 0 && idx >= 0) { tok = idx; logp = 0.f; ent = 0.f; gap = 0.f; }
  } else if (err == 0 && Z > 0.0) {
    const double lnZ = log(Z), mean = W / Z;
    ent = (float)(lnZ - kLn2 * mean);
    // sum p_i (s_max - s_i) with s = z/tau: the mean of s is (M + W/Z) ln2
    gap = (float)((above(zmax) - mean) * kLn2);
    if (sample) tok = idx;
    if (have_zt) logp = (float)(above(zt) * kLn2 - lnZ);
  }
  if (p.out_ent) p.out_ent[row] = ent;
  if (p.out_gap) p.out_gap[row] = gap;
  if (sample) p.out_tok[row] = tok;
  if (p.out_logp) p.out_logp[row] = logp;
}

// A row without a result: masked out (v = 0) or given up on because a wait ran out (v = NaN).
__device__ __forceinline__ void write_plain(const RowsParams &p, uint32_t row, float v) {
  if (p.mode == kModeSample) p.out_tok[row] = -1;
  if (p.out_logp) p.out_logp[row] = v;
  if (p.out_ent) p.out_ent[row] = v;
  if (p.out_gap) p.out_gap[row] = v;
}

}  // namespace
}  // namespace e3
