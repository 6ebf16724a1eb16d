// Row kernel: one pass over the logits of a row gives the softmax statistics
// (App. A: Z(beta), Eq. "entropy" in its shifted form H = ln Z + beta sum p_i Delta_i), the
// log-probability of one token and, for rollouts, a Gumbel-max sample.
//
// Work split.  A row is cut into strips of a few tiles of 4 KiB and every CTA of a persistent grid (one per SM) takes an equal,
// contiguous run of strips, so all CTAs stream the same number of bytes whatever the number of rows.  With a response
// mask the run is taken from the rows that the mask lets through: every CTA counts the mask first (a few bytes per
// row), so that masked rows cost nothing and unbalance nothing.  A run covers the tail of one row, some whole rows and
// the head of another; when its last row is cut that piece comes first, so that the end of a CTA's life is the cheap
// finish of a row it holds alone.  A CTA publishes its piece of a cut row in the caller's workspace (64-bit words tagged with
// a per-call id), issues a sequentially consistent fence and looks for the row's other pieces: of all CTAs that hold a
// piece, the one whose fence comes last finds them all, merges them in piece order and finishes the row.  It wipes the
// tags of the pieces, so that a replay of the same launch (a captured graph) never meets a piece of an earlier run.
// Nobody waits for anybody.
//
// Inside a CTA.  There are no roles: each of the 24 warps takes the next strip of the run from a counter in shared memory,
// copies its tiles into a ring of its own (two slots of 4 KiB, one bulk asynchronous copy per tile, 192 KiB in flight
// per SM), sums them and takes the next strip, through all rows of the run, without meeting the other warps.  What a strip
// gives depends on the strip alone (its reference logit is taken from a sample of its own entries) and is left as a record
// in shared memory; the warp that completes a segment (the strips of a row in this run, at most half a ring of records at a
// time) merges its records in their order.  So results do not depend on which warp took which strip, and the hand-out may
// follow the speed of the warps: with tiles dealt in advance (tile i to warp i mod 24) the slowest warp of an SM was done
// after 31 us when the average was done after 23 (512 x 151,936 bf16).  A design with one warp feeding all rings, one finishing
// rows and eight consuming, twice per SM, had too few warps per scheduler to hide the exponentials (60 % of the
// special-function unit's time).
//
// A thread takes 128 contiguous bytes of a slot, read as 16-byte vectors in the order i xor (lane mod 8),
// which keeps the eight lanes of a quarter warp on distinct banks.  A bulk copy starts and ends on 16-byte boundaries:
// a tile of a row that does not is copied from the boundary below to the boundary above it (every 16-byte unit
// that is touched holds a byte of the row) and moved into place in shared memory.
//
// Every wait is bounded in time: when one runs out the CTA stops waiting altogether, marks the rows it has not finished
// as invalid (token -1, NaN), sets the timeout bit of the caller's status word, sees its copies in flight land (bounded
// again) and returns.  The kernel is launched with programmatic stream serialization: its set-up overlaps the tail of
// the kernel before it in the stream, and it touches global memory only after griddepcontrol.wait.
//
// Numerics.  A strip's sums are Z = sum 2^t, W = sum 2^t * t with t = z*c - R*c and c = log2(e)/tau, two entries per
// instruction (packed fp32).  R is the largest of a sample of 256 (bf16) or 128 (fp32) of the first tile's entries plus a
// margin; one vote per tile checks its sums, and when an entry is far above R (or there is a NaN or a +inf) R moves up to
// the tile's largest logit and the tile is summed again; where there is a -inf it is summed with clamped entries, and if neither
// helps in a careful form that flags NaN and +inf.  R c is rounded down, so that t <= 0 up to R however large it is (a strip may begin
// with a fill value such as -1e9); from |R c| = 2^30 on the careful form counts the entries that equal R.  R therefore stays
// close to the largest logit of the strip, which keeps W/Z small and the entropy free of cancellation.  Records merge associatively; the per-row result is formed in fp64:
// H = ln Z - ln2 * W / Z,  ln p_tok = (z_tok*c - M) ln2 - ln Z, and, where the caller asks for it, the mean logit gap
// beta sum p_i Delta_i = (z_max*c - M - W/Z) ln2 of App. A.
//
// Sampler 0 (one Gumbel per vocabulary entry).  u_i has 8 coarse + 32 fine bits.  An entry can
// only win if its coarse byte is 255 (g_i >= 5.5432) or if z_i/tau exceeds the best score so
// far minus 5.5432; the second condition is tested on the sum of 2^t over the entry's group of 16,
// which bounds every term from above.  Per tile a thread makes its groups' coarse bytes (one Philox call per group)
// and notes which are 255.  Those entries (one in 256) whose logit is not hopeless, and the entries above the gate, go
// into a small per-warp queue with ballot-compacted positions, and the warp scores 32 of them at a time, one per lane, in
// fp32 with a proven error bound, and keeps three leaders.  Whoever finishes the row takes the fp32 leader when
// it is ahead by more than two error bounds; otherwise it evaluates the contenders in fp64 with the expression order of
// the definition (or looks at the whole row again when there are three or more).  The token never depends on the
// gating or on fp32.
//
// Sampler 1 (one Gumbel per block of 256 entries).  4 or 8 neighbouring lanes hold a block of the tile: two or three
// shuffles add their sums up.  The Gumbel variates do not depend on the logits: a warp makes those of its strip (four per Philox
// call, one call per lane) while the strip's first tile is under way, adds the blocks' log-sum-exps to them, and leaves the strip's
// leading blocks beside its record (one, and two more only where they come close).  The segment's finisher merges those; the row's
// finisher settles near-ties of block scores in fp64 and draws inside the winning block by inverse CDF (fp32, fp64 near a prefix
// boundary).  With the scores of all blocks in a ring of shared memory instead (512 tiles of them, the variates of a segment made by the warp
// that took its first strip, added up by atomics, looked through by the segment's finisher) strips could be four tiles long at most in
// a long run: 4,096 x 151,936 bf16 240-252 us, now 223-238 (two GPUs), 512 rows 41.3, now
// 38.4, 256 x 256,000 fp32 64.5, now 49.9.
#include "e3_rows.cuh"
#include "e3_rows_device.cuh"
#include "e3_rows_split.cuh"

#include <atomic>
#include <chrono>
#include <mutex>

namespace e3 {
namespace {

constexpr int kThreads = kWarps * 32;
constexpr int kStages = 2;       // ring slots per warp
constexpr int kMaxLive = 1024;   // rows of a CTA's run with a response mask (their numbers are kept in shared memory)
constexpr int kQueueCap = 64;    // sampler 0: a push meets at most 31 entries and adds at most 32
constexpr int kStripBlocks = longest_strip(1, true) * Fmt<1>::kBT;  // sampler 1: most blocks of a strip
static_assert(longest_strip(1, false) * Fmt<0>::kBT <= kStripBlocks && kLongRunStrip <= longest_strip(1, true) && kLongRunStrip <= longest_strip(1, false),
              "room for the blocks of every strip");

// An entry of sampler 0 that may win: vocabulary index (with kAnyByte: its coarse byte has not been looked at, else it is
// 255) and logit.
struct Candidate {
  uint32_t i;
  float z;
};
constexpr uint32_t kAnyByte = 0x80000000u;

// A strip that a warp has taken.
struct __align__(8) StripMeta {
  int q;         // strip of the run
  int tile;      // first tile within the row
  int seg;       // strip number (in the run) of the segment's first strip
  uint32_t row;
  int end;       // behind its last tile
  int need;      // strips of the segment
};

// What a warp keeps about the segment in hand.
struct WarpState {
  uint32_t row;
  float tau;
  float ty[3];     // leaders: entries of sampler 0, the largest logit of a greedy row
  int tb[3];
  float zf;        // logit of entry tb[0]
  PhiloxRow prow;  // sampler 0: coarse stream
};

// A segment: what its warps have handed in.  At the ring place of its first strip.
struct Segment {
  int arrived;     // strips summed
  int lock, err;
  float ty[3], zf;
  int tb[3];       // (training side: tb[0] = the target, once its logit has come by)
};

// State of a row piece of several segments, merged in their order.
struct LongPiece {
  int q0, turn;    // first strip; segments merged
  Piece state;
};

// Sampler 1: the leading blocks of a strip (further ones than the first only where they come close to it; index -1: none).
struct BlockLeaders {
  float y[3];
  int b[3];
};

struct Smem {
  u64 full[kWarps][kStages];     // per warp and ring slot: the slot's tile has landed
  StripMeta meta[kWarps][2];     // the warp's even and odd strips
  float4 record[kRing];          // per strip: reference (log2 units), sum 2^t, sum 2^t t, largest logit
  int freed[kRing];              // 1 + number of the last strip at this place whose record has been merged
  Segment seg[kRing];
  WarpState warp[kWarps];
  uint4 spill[kWarps][kStages];  // last 16 bytes of a tile that spans one 16-byte unit more
  LongPiece piece[kLong];
  Run run;
  int next;                      // strips handed out
  int timeout;                   // set when a bounded wait ran out
  int exited;                    // warps that have left the streaming loop
  RowsParams p;                  // the launch parameters, for the code that is not inlined
};
// Shared state of the CTA.  At namespace scope, so that functions that are not inlined reach it without a pointer (every
// value the streaming loop keeps for them costs it a register).
__shared__ Smem sm;

__device__ __forceinline__ int volatile_int(const int &x) { return *reinterpret_cast<const volatile int *>(&x); }
__device__ __forceinline__ bool timed_out() { return volatile_int(sm.timeout) != 0; }
// A wait has run out: from now on no wait of the CTA blocks, and the caller's status word says so.
__device__ __noinline__ void raise_timeout() {
  *reinterpret_cast<volatile int *>(&sm.timeout) = 1;
  if (sm.p.status != nullptr) atomicOr(sm.p.status, kStatusTimeout);
}
// Polls until `ready` says so; false when the wait was given up (it took longer than the launch's limit, or another wait of
// the CTA has run out before: then no wait blocks any more).
template <class F>
__device__ __forceinline__ bool bounded_wait(F ready) {
  const u64 t0 = global_ns();
  for (uint32_t it = 1;; ++it) {
    if (ready()) return true;
    if (timed_out()) return false;
    if ((it & 63u) == 0u && global_ns() - t0 > sm.p.wait_ns) break;
  }
  raise_timeout();
  return false;
}
__device__ __noinline__ bool mbar_wait_slow(int warp, int slot, uint32_t parity) {
  return bounded_wait([&] { return mbar_try_wait(&sm.full[warp][slot], parity); });
}
__device__ __forceinline__ bool mbar_wait(int warp, int slot, uint32_t parity) {
  return mbar_try_wait(&sm.full[warp][slot], parity) ? true : mbar_wait_slow(warp, slot, parity);
}

// Sampler 0: best score of a segment, as far as the CTA's warps have posted it: 64-bit word (first strip, order-preserving
// code) at the segment's place in the array `bests`.
__device__ __forceinline__ void post_best(u64 *bests, int seg, int enc) {
  atomicMax(bests + (seg & (sm.p.ring - 1)), ((u64)(seg + 1) << 32) | (uint32_t)(enc ^ 0x80000000));
}
__device__ __forceinline__ int read_best(const u64 *bests, int seg) {
  const u64 v = *reinterpret_cast<const volatile u64 *>(bests + (seg & (sm.p.ring - 1)));
  return (uint32_t)(v >> 32) == (uint32_t)(seg + 1) ? (int)((uint32_t)v ^ 0x80000000u) : enc_neg_inf();
}

// ---------------------------------------------------------------------------------------------
// Row results
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void piece_reset(Piece &pc) {
  pc.M = pc.Z = pc.W = pc.zf = 0.f;
  pc.err = 0;
  pc.zmax = -CUDART_INF_F;
#pragma unroll
  for (int i = 0; i < 3; ++i) { pc.ty[i] = -CUDART_INF_F; pc.tb[i] = -1; }
}
// Merges q into pc.
__device__ __forceinline__ void piece_merge(Piece &pc, const Piece &q) {
  pc.err |= q.err;
  pc.zmax = fmaxf(pc.zmax, q.zmax);
  merge_stats_f(pc.M, pc.Z, pc.W, q.M, q.Z, q.W);
  Top3 top;
#pragma unroll
  for (int i = 0; i < 3; ++i) { top.y[i] = pc.ty[i]; top.b[i] = pc.tb[i]; }
  if (q.tb[0] >= 0 && best_before(q.ty[0], q.tb[0], top.y[0], top.b[0])) pc.zf = q.zf;
#pragma unroll
  for (int i = 0; i < 3; ++i) top3_insert(top, q.ty[i], q.tb[i]);
#pragma unroll
  for (int i = 0; i < 3; ++i) { pc.ty[i] = top.y[i]; pc.tb[i] = top.b[i]; }
}

// A row piece of this CTA is complete (all lanes hold the same pc): finishes the row, or, when the row is cut, publishes
// the piece and finishes the row if the other pieces are all there.
template <int DT, int SAMPLER>
__device__ __noinline__ void finish_piece(const Piece &pc_in, int j, bool whole, uint32_t row, float tau) {
  const RowsParams &p = sm.p;
  const Run &run = sm.run;
  const int lane = threadIdx.x & 31;
  RowInfo ri;
  ri.greedy = p.mode == kModeSample && tau == 0.f;
  ri.c = ri.greedy || !(tau > 0.f && tau < CUDART_INF_F) ? 0.f : __fdiv_rn(kLog2e, tau);
  Piece pc = pc_in;
  if (!whole) {
    const uint32_t rank = run.r0 + (uint32_t)j, spr = (uint32_t)p.spr;
    const int k0 = cta_of_strip(p, run, rank * spr), k1 = cta_of_strip(p, run, rank * spr + spr - 1u);
    u64 *const pieces = reinterpret_cast<u64 *>(p.ws_pieces);
    // CTA k keeps this row's piece in its workspace slot 0 when its run begins in the row, else in slot 1
    auto piece_of = [&](int k) {
      const bool first = first_strip_of(p, run, (uint32_t)k) >= rank * spr;
      return pieces + ((size_t)k * 2 + (first ? 0 : 1)) * (kPieceBytes / 8);
    };
    // Store the piece, then, after a sequentially consistent fence, look for the others: of all CTAs that hold a piece, the
    // one whose fence comes last is sure to find them all.  Two CTAs may both find all pieces; they then write the same
    // values.
    if (lane == 0) {
      piece_store(piece_of((int)blockIdx.x), p.call_id, pc);
      asm volatile("fence.sc.gpu;" ::: "memory");
    }
    __syncwarp();
    const Piece own = pc;
    piece_reset(pc);
    bool ok = true;
    for (int k = k0 + lane; k <= k1; k += 32) {
      Piece q;
      if (k == (int)blockIdx.x) {
        q = own;
      } else if (!piece_load(piece_of(k), p.call_id, q)) {
        ok = false;
        break;
      }
      piece_merge(pc, q);
    }
    if (!__all_sync(0xffffffffu, ok)) return;
    warp_merge(pc);
    pc.err = __reduce_or_sync(0xffffffffu, pc.err);
    Top3 top;
#pragma unroll
    for (int i = 0; i < 3; ++i) { top.y[i] = pc.ty[i]; top.b[i] = pc.tb[i]; }
    warp_merge_top(top, pc.zf);
#pragma unroll
    for (int i = 0; i < 3; ++i) { pc.ty[i] = top.y[i]; pc.tb[i] = top.b[i]; }
    // the row is done: nobody needs its pieces any more (a later run of this very launch must not find them)
    for (int k = k0 + lane; k <= k1; k += 32) piece_wipe(piece_of(k), p.call_id);
  }
  // training side: the leader is the target itself, with its logit in zf (no leader: target outside the vocabulary)
  int id = pc.tb[0];
  float zt = pc.zf;
  if (SAMPLER >= 0 && !ri.greedy && id >= 0) {
    EvalCtx ex;
    ex.rk = p.round_key; ex.row = row_ptr(p, row); ex.tau = tau; ex.slack_k = p.slack_scale;
    ex.grow = p.row_base + row;
    ex.ctr_lo = p.ctr_lo; ex.ctr_hi8 = p.ctr_hi8; ex.V = p.V;
    Top3 top;
#pragma unroll
    for (int i = 0; i < 3; ++i) { top.y[i] = pc.ty[i]; top.b[i] = pc.tb[i]; }
    if (SAMPLER == 1) {
      id = pc.err == 0 ? sample_in_blocks<DT>(ex, top, lane, zt) : -1;
    } else {
      // fp32 scores decide unless the runner-up is within two slacks of the leader
      const float slack2 = 2.f * fmaxf(score_slack(top.y[0], p.slack_scale), score_slack(top.y[1], p.slack_scale));
      if (top.b[1] >= 0 && !(top.y[0] - top.y[1] > slack2)) id = settle_exact<DT>(ex, top, slack2, lane, zt);
    }
  }
  if (lane == 0) finish_row(p, row, ri, pc.M, pc.Z, pc.W, pc.zmax, id, pc.err, id >= 0, zt);
}

// The warp that completes the segment whose first strip is number q merges its records, in their order, and gives their
// places free.  With the row piece's last segment the piece is complete.  False when a wait was given up.
template <int DT, int SAMPLER>
__device__ __noinline__ bool finish_segment(int q, uint32_t row, float tau, const BlockLeaders *blocks) {
  const RowsParams &p = sm.p;
  const int lane = threadIdx.x & 31;
  const Place w = place_of(p, sm.run, q);
  const int n = segment_strips(p, w), mask = p.ring - 1, half = p.ring / 2;
  Segment &sg = sm.seg[q & mask];
  Piece pc;
  pc.M = pc.Z = pc.W = 0.f;
  pc.zmax = -CUDART_INF_F;
  for (int i = lane; i < n; i += 32) {
    const float4 r = sm.record[(q + i) & mask];
    merge_stats_f(pc.M, pc.Z, pc.W, r.x, r.y, r.z);
    pc.zmax = fmaxf(pc.zmax, r.w);
  }
  warp_merge(pc);
  pc.err = sg.err;
  pc.zf = sg.zf;
#pragma unroll
  for (int i = 0; i < 3; ++i) { pc.ty[i] = sg.ty[i]; pc.tb[i] = sg.tb[i]; }
  if (SAMPLER == 1) {
    Top3 top;
    top3_reset(top);
    for (int i = lane; i < n; i += 32) {
      const BlockLeaders &l = blocks[(q + i) & mask];
#pragma unroll
      for (int k = 0; k < 3; ++k) top3_insert(top, l.y[k], l.b[k]);
    }
    if (tau > 0.f && tau < CUDART_INF_F) {  // (the others have none)
      merge_near_blocks(top);
#pragma unroll
      for (int i = 0; i < 3; ++i) { pc.ty[i] = top.y[i]; pc.tb[i] = top.b[i]; }
    }
  }
  __syncwarp();
  if (lane == 0) {
    sg.arrived = sg.lock = sg.err = 0;
    sg.zf = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) { sg.ty[i] = -CUDART_INF_F; sg.tb[i] = -1; }
    __threadfence_block();
  }
  __syncwarp();
  const bool single = w.hi - w.lo <= half, last = w.strip + n == w.hi;
  if (!single) {  // in the order of the segments (they are handed out in that order: the ones before are under way)
    LongPiece &lp = sm.piece[long_piece_place(w)];
    const int turn = (w.strip - w.lo) / half;
    if (turn > 0) {
      const bool ok = bounded_wait([&] { return volatile_int(lp.q0) == w.q0 && volatile_int(lp.turn) == turn; });
      if (!__all_sync(0xffffffffu, ok)) return false;
      __threadfence_block();
      Piece sum = lp.state;
      piece_merge(sum, pc);
      pc = sum;
    }
    __syncwarp();
    if (lane == 0) {
      lp.state = pc;
      __threadfence_block();
      *reinterpret_cast<volatile int *>(&lp.turn) = turn + 1;
      *reinterpret_cast<volatile int *>(&lp.q0) = w.q0;
    }
    __syncwarp();
  }
  if (last) finish_piece<DT, SAMPLER>(pc, w.j, w.hi - w.lo == p.spr, row, tau);
  __threadfence_block();
  __syncwarp();
  for (int i = lane; i < n; i += 32) *reinterpret_cast<volatile int *>(&sm.freed[(q + i) & mask]) = q + i + 1;
  return true;
}

// After a timeout, when all warps have left: the rows of pieces that were never completed are marked (nobody else can finish
// them: a cut row needs this CTA's piece, which was not published).  One warp.
__device__ __noinline__ void mark_unfinished(const uint32_t *live_rows) {
  const RowsParams &p = sm.p;
  const Run &run = sm.run;
  __threadfence_block();
  for (int j = threadIdx.x & 31; j < run.n; j += 32) {
    const int lo = j == 0 ? run.lo0 : 0, hi = j == run.n - 1 ? run.hin : p.spr;
    const int q0 = run.head && j == run.n - 1 ? 0 : run.head + (j == 0 ? 0 : j * p.spr - run.lo0);
    const int half = p.ring / 2, last = q0 + (hi - lo - 1) / half * half;  // first strip of the piece's last segment
    if (volatile_int(sm.freed[last & (p.ring - 1)]) < last + 1)
      write_plain(p, live_rows ? live_rows[j] : run.r0 + (uint32_t)j, CUDART_NAN_F);
  }
}

// ---------------------------------------------------------------------------------------------
// Samplers
// ---------------------------------------------------------------------------------------------
// Enters (y, b) in a list of three leaders (a warp's or a segment's); zf follows the first.  One lane.
template <class L>
__device__ __forceinline__ void lead_insert(L &ws, float y, int b, float z) {
  if (top3_before(y, b, ws.ty[0], ws.tb[0])) {
    ws.ty[2] = ws.ty[1]; ws.tb[2] = ws.tb[1]; ws.ty[1] = ws.ty[0]; ws.tb[1] = ws.tb[0]; ws.ty[0] = y; ws.tb[0] = b;
    ws.zf = z;
  } else if (top3_before(y, b, ws.ty[1], ws.tb[1])) {
    ws.ty[2] = ws.ty[1]; ws.tb[2] = ws.tb[1]; ws.ty[1] = y; ws.tb[1] = b;
  } else if (top3_before(y, b, ws.ty[2], ws.tb[2])) {
    ws.ty[2] = y; ws.tb[2] = b;
  }
}

// Enters the lanes' scored candidates (y, i; logit z) that may win in a list of leaders.  best: encoded lower bound of the best score
// (the same in all lanes); returns it, raised.
template <class L>
__device__ __forceinline__ int enter_leaders(L &ws, bool valid, float y, int i, float z, int best, float slack_scale) {
  constexpr unsigned kAll = 0xffffffffu;
#pragma unroll 1
  for (;;) {
    valid = valid && y >= dec_float(best);  // else more than two slacks below a score already seen (or NaN)
    if (!__any_sync(kAll, valid)) break;
    const int e = valid ? enc_float(y) : INT_MIN, emax = __reduce_max_sync(kAll, e);
    const int imin = __reduce_min_sync(kAll, valid && e == emax ? i : INT_MAX);
    if (valid && e == emax && i == imin) {
      lead_insert(ws, y, i, z);
      valid = false;
    }
    __syncwarp();
    const float ym = dec_float(emax);
    const int enc = enc_float(ym - 4.f * score_slack(ym, slack_scale) - 2e-7f * fabsf(ym));
    best = enc > best ? enc : best;
  }
  return best;
}

// Enters a warp's leaders in its segment's list.  One lane; the list is locked for the few instructions this takes.  False
// when the wait for the lock ran out.
__device__ __noinline__ bool hand_in_leaders(int seg) {
  const WarpState &ws = sm.warp[threadIdx.x >> 5];
  Segment &sg = sm.seg[seg & (sm.p.ring - 1)];
  if (!bounded_wait([&] { return atomicCAS(&sg.lock, 0, 1) == 0; })) return false;
  __threadfence_block();
#pragma unroll
  for (int i = 0; i < 3; ++i)
    if (ws.tb[i] >= 0) lead_insert(sg, ws.ty[i], ws.tb[i], ws.zf);  // (zf matters for the first alone)
  __threadfence_block();
  atomicExch(&sg.lock, 0);
  return true;
}

// Sampler 0: scores one candidate per lane (lanes below `count`) in fp32 and enters those that may win in the warp's list.
// best: encoded lower bound of the row's best score (the same in all lanes); returns it, raised.
__device__ __noinline__ int score_candidates(const Candidate *queue, int count, int best) {
  const int lane = threadIdx.x & 31;
  const RowsParams &p = sm.p;
  WarpState &ws = sm.warp[threadIdx.x >> 5];
  const float tau = ws.tau;
  float y = 0.f, z = 0.f;
  int i = 0;
  bool valid = lane < count;
  __syncwarp();
  if (valid) {
    const Candidate c = queue[lane];
    z = c.z;
    i = (int)(c.i & ~kAnyByte);
    uint32_t cbyte = 255u;
    if (c.i & kAnyByte) {  // entries with byte 255 are in the queue on their own
      const uint4 cw = philox_call(p.round_key, ws.prow, (uint32_t)i >> 4);
      cbyte = (pick_word(cw, (i & 15) >> 2) >> (8 * (i & 3))) & 0xFFu;
      valid = cbyte != 255u;
    }
    // what cannot win even with the largest Gumbel of its coarse byte is passed over (a +inf has flagged the row)
    valid = valid && z > logit_gate(best, tau, cbyte == 255u ? kGumbelCapAll : kGumbelCapCoarse) && z < CUDART_INF_F;
    const uint4 fw = philox(p.round_key, (uint32_t)i >> 2, p.row_base + ws.row, p.ctr_lo, p.ctr_hi8 | 1u);
    y = score_f32(z, __frcp_rn(tau), cbyte, pick_word(fw, i & 3));
  }
  best = enter_leaders(ws, valid, y, i, z, best, p.slack_scale);
  __syncwarp();
  return best;
}

// Sampler 1: the Gumbel variates of the blocks of a strip (n tiles from tile `first` of the row on), four per Philox call and lane.
template <int DT>
__device__ __noinline__ void make_gumbels(uint32_t row, int first, int n, float *score) {
  constexpr int kCalls = Fmt<DT>::kBT / 4;  // per tile
  static_assert(kStripBlocks / 4 <= 32, "one call per lane");
  const int lane = threadIdx.x & 31;
  const RowsParams &p = sm.p;
  if (lane < n * kCalls) {
    const uint4 x = philox(p.round_key, (uint32_t)(first * kCalls + lane), p.row_base + row, p.ctr_lo, p.ctr_hi8 | 2u);
    *reinterpret_cast<float4 *>(score + 4 * lane) =
        make_float4(gumbel_from_word(x.x), gumbel_from_word(x.y), gumbel_from_word(x.z), gumbel_from_word(x.w));
  }
  __syncwarp();
}
// ... the leaders of the strip's n blocks, whose scores stand in `score`; b0: number of the first.
__device__ __noinline__ void hand_in_blocks(const float *score, int n, int b0, BlockLeaders *out) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int kMine = (kStripBlocks + 31) / 32;
  const int lane = threadIdx.x & 31;
  __syncwarp();
  float y[kMine], m = -CUDART_INF_F;  // (-inf: a block without mass, or beyond the row)
#pragma unroll
  for (int k = 0; k < kMine; ++k) {
    y[k] = lane + 32 * k < n ? score[lane + 32 * k] : -CUDART_INF_F;
    m = fmaxf(m, y[k]);
  }
  const float best = dec_float(__reduce_max_sync(kAll, enc_float(m)));
  const float near = best - near_blocks(best);
  int close = 0, at = INT_MAX;
#pragma unroll
  for (int k = kMine - 1; k >= 0; --k) {
    close += y[k] >= near ? 1 : 0;
    if (y[k] == best) at = b0 + lane + 32 * k;
  }
  Top3 top;
  top3_reset(top);
  if (best == -CUDART_INF_F) {
  } else if (__reduce_add_sync(kAll, close) == 1) {
    top.y[0] = best;
    top.b[0] = __reduce_min_sync(kAll, at);
  } else {
#pragma unroll 1
    for (int i = lane; i < n; i += 32)
      if (score[i] > -CUDART_INF_F) top3_insert(top, score[i], b0 + i);
    merge_near_blocks(top);
  }
  if (lane < 3) {
    out->y[lane] = lane == 0 ? top.y[0] : (lane == 1 ? top.y[1] : top.y[2]);
    out->b[lane] = lane == 0 ? top.b[0] : (lane == 1 ? top.b[1] : top.b[2]);
  }
  __syncwarp();
}

// ---------------------------------------------------------------------------------------------
// Response mask: numbers of the rows of the CTA's run.  Every CTA counts the whole mask (16 rows per load) and then
// lists the rows whose rank falls into its run.  Returns with sm.run set; ends with a barrier of the CTA.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t w) {  // bit 7 of every byte that is not zero
  return (((w & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w) & 0x80808080u;
}
struct MaskWord {
  uint32_t w[4];
};
// 16 mask bytes number v (counted from the 16-byte boundary at or below the mask), as bits 7 of non-zero bytes inside it.
__device__ __forceinline__ MaskWord mask_word(const RowsParams &p, uint32_t shift, uint32_t v) {
  const uint4 q = __ldg(reinterpret_cast<const uint4 *>(p.mask - shift) + v);
  MaskWord m = {{nonzero_bytes(q.x), nonzero_bytes(q.y), nonzero_bytes(q.z), nonzero_bytes(q.w)}};
  const uint32_t first = v * 16u, lo = shift, hi = shift + p.rows;
  if (first < lo || first + 16u > hi) {
#pragma unroll
    for (uint32_t b = 0; b < 16; ++b)
      if (first + b < lo || first + b >= hi) m.w[b >> 2] &= ~(0x80u << (8u * (b & 3u)));
  }
  return m;
}
__device__ __noinline__ void scan_mask(uint32_t *live_rows) {
  const RowsParams &p = sm.p;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint32_t *const live_warp = live_rows + kMaxLive;  // counts of the warps
  const uint32_t shift = (uint32_t)(reinterpret_cast<uintptr_t>(p.mask) & 15u);
  const uint32_t words = (shift + p.rows + 15u) / 16u, per = (words + kThreads - 1u) / kThreads;
  const uint32_t v0 = (uint32_t)tid * per < words ? (uint32_t)tid * per : words, v1 = v0 + per < words ? v0 + per : words;
  uint32_t count = 0;
  for (uint32_t v = v0; v < v1; ++v) {
    const MaskWord m = mask_word(p, shift, v);
    count += __popc(m.w[0]) + __popc(m.w[1]) + __popc(m.w[2]) + __popc(m.w[3]);
  }
  uint32_t incl = count;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  if (lane == 31) live_warp[warp] = incl;
  __syncthreads();
  uint32_t before = incl - count, total = 0;
  for (int w = 0; w < kWarps; ++w) {
    before += w < warp ? live_warp[w] : 0u;
    total += live_warp[w];
  }
  if (tid == 0) set_run(p, sm.run, total, blockIdx.x, gridDim.x);
  __syncthreads();
  const uint32_t r0 = sm.run.r0, n = (uint32_t)sm.run.n;
  if (count > 0 && before < r0 + n && before + count > r0) {
    uint32_t rank = before;
    for (uint32_t v = v0; v < v1; ++v) {
      const MaskWord m = mask_word(p, shift, v);
#pragma unroll
      for (uint32_t q = 0; q < 4; ++q)
        for (uint32_t f = m.w[q]; f != 0u; f &= f - 1u, ++rank)
          if (rank - r0 < n) live_rows[rank - r0] = v * 16u + q * 4u + (uint32_t)(__ffs((int)f) - 1) / 8u - shift;
    }
  }
  // masked rows read zero; every CTA writes those of its share of the rows
  const uint32_t share = (p.rows + gridDim.x - 1u) / gridDim.x, lo = blockIdx.x * share;
  for (uint32_t i = tid; i < share; i += kThreads)
    if (lo + i < p.rows && __ldg(p.mask + lo + i) == 0) write_plain(p, lo + i, 0.f);
  __syncthreads();
}

// ---------------------------------------------------------------------------------------------
// The kernel
// ---------------------------------------------------------------------------------------------
// Dynamic shared memory: the warps' rings, then sampler 0's queues and best scores, or sampler 1's block scores, or the rows
// of the run with a response mask.
template <int SAMPLER>
constexpr size_t dyn_smem_bytes(bool mask) {
  return (size_t)kWarps * kStages * kTileBytes + (SAMPLER == 0 ? kWarps * kQueueCap * sizeof(Candidate) + kRing * sizeof(u64) : 0) +
         (SAMPLER == 1 ? kWarps * kStripBlocks * sizeof(float) + kRing * sizeof(BlockLeaders) : 0) + (mask ? (kMaxLive + kWarps) * sizeof(uint32_t) : 0);
}

constexpr size_t kSmemMost = 232448;  // 227 KiB
static_assert(dyn_smem_bytes<-1>(true) + sizeof(Smem) <= kSmemMost && dyn_smem_bytes<0>(false) + sizeof(Smem) <= kSmemMost &&
                  dyn_smem_bytes<1>(false) + sizeof(Smem) <= kSmemMost, "shared memory of a CTA");

template <int DT, int SAMPLER>
__global__ void __launch_bounds__(kThreads, 1) rows_kernel(const __grid_constant__ RowsParams p) {
  extern __shared__ __align__(128) unsigned char dyn[];
  using F = Fmt<DT>;
  constexpr int kG = F::kG;
  constexpr unsigned kAll = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(kAll, tid >> 5, 0);  // (known to be the same in all lanes)
  unsigned char *const extra = dyn + kWarps * kStages * kTileBytes;
  u64 *const bests = reinterpret_cast<u64 *>(extra + kWarps * kQueueCap * sizeof(Candidate));  // sampler 0
  float *const score = reinterpret_cast<float *>(extra) + warp * kStripBlocks;                 // sampler 1: the warp's
  BlockLeaders *const blocks = reinterpret_cast<BlockLeaders *>(extra + kWarps * kStripBlocks * sizeof(float));

  if (tid < kWarps * kStages) mbar_init(&sm.full[0][0] + tid, 1);
  if (tid < kRing) {
    Segment &sg = sm.seg[tid];
    sg.arrived = sg.lock = sg.err = 0;
    sg.zf = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) { sg.ty[k] = -CUDART_INF_F; sg.tb[k] = -1; }
    if (SAMPLER == 0) bests[tid] = 0ull;
    sm.freed[tid] = tid - p.ring + 1;
  }
  if (tid < kLong) sm.piece[tid].q0 = -1;
  if (tid < (int)(sizeof(RowsParams) / 4)) reinterpret_cast<uint32_t *>(&sm.p)[tid] = reinterpret_cast<const uint32_t *>(&p)[tid];
  if (tid == kThreads - 32) {
    sm.timeout = sm.exited = 0;
    sm.next = kWarps;  // (the first strips go to the warps by their numbers: a short run then loads the schedulers evenly)
    if (p.mask == nullptr) set_run(p, sm.run, p.rows, blockIdx.x, gridDim.x);
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncthreads();
  // Programmatic dependent launch: this grid may have been started while the kernel before it in the
  // stream was still finishing (launch latency, block start-up and the set-up above then overlap with that
  // kernel's tail).  Nothing in global memory may be touched before griddepcontrol.wait, which returns once the
  // earlier kernel has completed and its writes are visible; the grid behind this one may start likewise.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t *const live_rows = SAMPLER < 0 && p.mask != nullptr ? reinterpret_cast<const uint32_t *>(extra) : nullptr;
  if (SAMPLER < 0 && p.mask != nullptr) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    scan_mask(reinterpret_cast<uint32_t *>(extra));
  }
  const int len = sm.run.len;

  const uint32_t ring = smem_addr(dyn) + (uint32_t)warp * (kStages * kTileBytes);
  const uint32_t lane_off = (uint32_t)(lane * kLaneBytes) | (uint32_t)((lane & 7) << 4);  // the lane's vector 0 in a slot
  WarpState &ws = sm.warp[warp];
  // Lane t of `aux` holds the temperature, lane t + 16 the target of the row of the warp's even or odd strip t.
  int aux = __float_as_int(p.temp_scalar);
  int fetched = 0, done = 0;   // tiles copied; tiles summed
  int strips = 0;              // strips taken
  const char *src = nullptr;   // the 16-byte boundary at or below the next tile of the strip that was taken last,
  int left = 0;                // how many of its tiles are left to copy,
  uint32_t bytes = 0, last_bytes = 0;  // the bytes from boundary to boundary of its tiles, and of its last one
  int skip = -1;               // (test hook: the tile that is never copied, by the number that are left behind it)
  int waiting = warp;          // a strip that has been taken and whose record has no place yet (or the warp's first)
  bool dry = false;            // no strip is left (or a wait was given up)
  const u64 policy = l2_evict_first_policy();

  // Loads what the warp's strip number t needs to know of its row.
  auto load_aux = [&](uint32_t row, int t) {
    if (p.temps != nullptr && lane == (t & 1)) aux = __float_as_int(__ldg(p.temps + row));
    if (SAMPLER < 0 && lane == (t & 1) + 16) aux = __ldg(p.targets + row);
  };
  // Takes the next strip of the run.  block: wait for a place for its record (only when the warp holds no other strip, which
  // others might wait for).
  auto take = [&](bool block) {
    int q = waiting;
    if (q < 0) {
      if (lane == 0) q = atomicAdd(&sm.next, 1);
      q = __shfl_sync(kAll, q, 0);
    }
    waiting = -1;
    if (q >= len) {
      dry = true;
      return;
    }
    const Place w = place_of(p, sm.run, q);
    const int seg = segment_start(p, w);
    auto free_places = [&] { return may_take(p, q, seg, [](int at) { return volatile_int(sm.freed[at]); }); };
    if (!__all_sync(kAll, free_places())) {
      bool ok = false;
      if (block) ok = bounded_wait(free_places);
      if (!__all_sync(kAll, ok)) {
        if (block) dry = true; else waiting = q;
        return;
      }
    }
    const uint32_t row = live_rows ? live_rows[w.j] : sm.run.r0 + (uint32_t)w.j;
    const int tile = w.strip * p.strip_tiles;
    const char *const at = row_ptr(p, row) + (size_t)tile * kTileBytes;
    const uint32_t a = (uint32_t)(reinterpret_cast<uintptr_t>(at) & 15u);
    src = at - a;
    left = p.strip_tiles;
    bytes = last_bytes = a != 0u ? kTileBytes + 16u : kTileBytes;
    if (w.strip == p.spr - 1) {
      left = p.tpr - tile;
      last_bytes = (a + (uint32_t)(p.V - (p.tpr - 1) * F::kTileE) * F::kEsize + 15u) & ~15u;
    }
    skip = -1;
    if (p.stall_src != nullptr && p.stall_src >= at && p.stall_src < at + left * kTileBytes)
      skip = left - 1 - (int)((p.stall_src - at) / kTileBytes);
    if (strips > 0) load_aux(row, strips);  // (the first strip is taken before global memory may be read)
    if (lane == 0) {
      const int half = p.ring / 2, behind = w.q0 + w.hi - w.lo - seg;  // strips of the piece from the segment's first on
      StripMeta m;
      m.q = q; m.tile = tile; m.row = row; m.seg = seg;
      m.end = tile + left;
      m.need = behind < half ? behind : half;
      sm.meta[warp][strips & 1] = m;
    }
    ++strips;
  };
  // Copies the next tile into the ring slot that is free (every lane has read it), if there is one.
  auto feed = [&](bool block) {
    if (left == 0 && !dry) take(block);
    if (left > 0) {
      --left;
      const uint32_t slot = (uint32_t)(fetched % kStages), n = left == 0 ? last_bytes : bytes;
      const uint32_t bar = smem_addr(&sm.full[warp][0]) + slot * 8u, dst = ring + slot * kTileBytes;
      if (n <= (uint32_t)kTileBytes) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %0, 0;\n\t"
            "@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%1], %2;\n\t"
            "@p cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%3], [%4], %2, [%1], %5;\n\t}"
            ::"r"(lane == 0 && left != skip ? 1 : 0), "r"(bar), "r"(n), "r"(dst), "l"(src), "l"(policy)
            : "memory");
      } else if (lane == 0 && left != skip) {  // one 16-byte unit more than a slot holds
        u64 *const b = &sm.full[warp][slot];
        mbar_arrive_expect(b, n);
        bulk_copy_g2s(dst, src, kTileBytes, b, policy);
        bulk_copy_g2s(smem_addr(&sm.spill[warp][slot]), src + kTileBytes, n - kTileBytes, b, policy);
      }
      src += kTileBytes;
      ++fetched;
    }
  };

  bool given_up = false;
  int strip = 0;  // strips summed
  // The warp's first strip is found before the kernel waits for the one before it in the stream (8 x 32,000 bf16: 9.0 us a
  // launch with all of it behind the wait, now 7.9).
  take(true);
  __syncwarp();
  if (live_rows == nullptr) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (strips > 0) load_aux(sm.meta[warp][0].row, 0);
  feed(false);
  for (;;) {
    if (done == fetched) feed(true);
    __syncwarp();
    if (done == fetched) break;
    if (fetched < done + kStages) feed(false);
    __syncwarp();
    // ------------------------------------------------------------------ strips of one segment, one after the other
    uint32_t mode;
    float c;
    uint32_t shift;             // bytes by which the row's tiles lie behind a 16-byte boundary
    int target = -1;            // training side
    int best = enc_neg_inf();   // sampler 0: bound of the row's best score
    int qn = 0;                 // ... candidates in the queue
    int count = 0, err = 0;     // strips summed
    int seg, need;
    {
      const StripMeta &m = sm.meta[warp][strip & 1];
      const uint32_t row = m.row;
      seg = m.seg;
      need = m.need;
      const float tau = __int_as_float(__shfl_sync(kAll, aux, strip & 1));
      mode = SAMPLER >= 0 && tau == 0.f ? kGreedy : (tau > 0.f && tau < CUDART_INF_F ? 0u : kUnusable);
      c = mode != 0u ? 0.f : __fdiv_rn(kLog2e, tau);
      shift = (uint32_t)(reinterpret_cast<uintptr_t>(row_ptr(p, row)) & 15u);
      if (SAMPLER < 0) target = __shfl_sync(kAll, aux, (strip & 1) + 16);
      if (lane == 0) {
        ws.row = row; ws.tau = tau;
        if (SAMPLER >= 0) {
          ws.zf = 0.f;
#pragma unroll
          for (int i = 0; i < 3; ++i) { ws.ty[i] = -CUDART_INF_F; ws.tb[i] = -1; }
        }
        if (SAMPLER == 0) ws.prow = philox_row(p.round_key, p.row_base + row, p.ctr_lo, p.ctr_hi8 | 0u);
      }
      if (mode & kUnusable) err = kErrValue;
      __syncwarp();
    }
    bool more;
    do {
      float Zs = 0.f, Ws = 0.f, nRc = CUDART_INF_F, zmax = -CUDART_INF_F;  // the strip's sums; no reference yet
      const StripMeta &meta = sm.meta[warp][strip & 1];
      const int q = meta.q, first = meta.tile, end = meta.end;
      if (SAMPLER == 1) make_gumbels<DT>(ws.row, first, end - first, score);
      for (int tile = first; tile < end; ++tile) {
        const int slot = done % kStages;
        // a wait that was given up ends the warp's work
        if (__any_sync(kAll, !mbar_wait(warp, slot, (uint32_t)(done / kStages) & 1u))) { given_up = true; break; }
        if (!(mode & kUnusable)) {
          const uint32_t base = ring + (uint32_t)slot * kTileBytes, B = base + lane_off;
          const int e_tile = tile * F::kTileE;
          const int n = p.V - e_tile < F::kTileE ? p.V - e_tile : F::kTileE;  // entries of the tile
          if (shift != 0u) realign_tile(base, smem_addr(&sm.spill[warp][slot]), shift);
          if (SAMPLER < 0 && (uint32_t)(target - e_tile) < (uint32_t)n && lane == 0) {
            Segment &sg = sm.seg[seg & (p.ring - 1)];
            sg.zf = lds_elem<DT>(base + (uint32_t)(target - e_tile) * F::kEsize);
            sg.tb[0] = target;
          }
          if (SAMPLER >= 0 && (mode & kGreedy)) {
            const Greedy g = tile_greedy<DT>(B, e_tile + lane * F::kLaneE, n - lane * F::kLaneE, lane & 7);
            if (g.i == -2) err = kErrValue;
            if (lane == 0 && g.i >= 0) lead_insert(ws, g.y, g.i, g.y);
          } else {
            float Z, W;
            float Zg[kG];
            bool summed = false;
            // Out of line: what only few tiles need (see tile_slow).  The blocked sampler keeps all but the clamped sums in the loop (us
            // with the careful form out of line and in the loop: 4,096 x 151,936 bf16 250, 230, 512 rows 40.1, 39.9).
            constexpr bool kLean = SAMPLER != 1;
            bool over = false;  // kLean: an entry far above the reference, or no reference yet
            if (n == F::kTileE && !(mode & kClamped)) {
              if (nRc == CUDART_INF_F) nRc = sample_reference<DT>(B, c);
              // kClamped: a -inf (a NaN, a +inf).  The clamp changes no other sum, so that the warp may keep it through the segment and
              // results still do not depend on which strips it takes.
              if (kLean) {
                over = nRc == CUDART_INF_F;
                if (!over) {
                  if (SAMPLER == 0) slice_sums_groups<DT>(B, c, nRc, Z, W, Zg);
                  else slice_sums<DT>(B, c, nRc, Z, W);
                  summed = !__any_sync(kAll, !(Z <= kSoundZ) || !(fabsf(W) <= kSoundW));
                  if (!summed) {
                    over = __any_sync(kAll, !(Z <= kSoundZ));
                    if (!over) mode |= kClamped;
                  } else if (p.out_gap) {
                    zmax = fmaxf(zmax, warp_max(slice_max<DT>(B)));
                  }
                }
              } else {
                bool moved = nRc == CUDART_INF_F;
#pragma unroll 1
                for (;;) {
                  if (moved) {
                    const float R = warp_max(slice_max<DT>(B));
                    if (R == -CUDART_INF_F || !move_reference(R, c, nRc, Zs, Ws)) break;
                  }
                  slice_sums<DT>(B, c, nRc, Z, W);
                  summed = !__any_sync(kAll, !(Z <= kSoundZ) || !(fabsf(W) <= kSoundW));
                  if (summed || moved || !__any_sync(kAll, !(Z <= kSoundZ))) break;
                  moved = true;
                }
                if (!summed) mode |= kClamped;
                else if (p.out_gap) zmax = fmaxf(zmax, warp_max(slice_max<DT>(B)));
              }
            }
            if (!summed && (kLean || n == F::kTileE)) {
              const SlowTile<DT> s = tile_slow<DT, SAMPLER == 0, kLean>(B, n, over, p.out_gap != nullptr, c, nRc, Zs, Ws);
              Zs = s.Zs; Ws = s.Ws; nRc = s.nRc;
              Z = s.Z; W = s.W;
              zmax = fmaxf(zmax, s.zmax);
              if (kLean) {
                err |= s.flags & kErrValue;
                mode |= (uint32_t)s.flags & kClamped;
              }
              if (!kLean) summed = s.flags == 0;
              if (SAMPLER == 0) {
#pragma unroll
                for (int j = 0; j < kG; ++j) Zg[j] = s.Zg[j];
              }
            }
            if (!kLean && !summed && careful_tile<DT>(B, n, c, nRc, Zs, Ws, Z, W, Zg, zmax)) err = kErrValue;
            Zs += Z;
            Ws += W;
            if (SAMPLER == 0) {
              Candidate *const queue = reinterpret_cast<Candidate *>(extra) + warp * kQueueCap;
              const int shared = read_best(bests, seg);
              best = shared > best ? shared : best;
              const int before = best;
              const int ga = (lane & 7) / F::kVG;  // order in which the lane has taken its groups
              const int e_lane = lane * F::kLaneE;
              // Scores up to 32 candidates of the queue, one per lane.
              auto drain = [&]() {
                const int from = qn > 32 ? qn - 32 : 0;
                best = score_candidates(queue + from, qn - from, best);
                qn = from;
              };
              auto push = [&](bool f, uint32_t i, float z) {
                const uint32_t ballot = __ballot_sync(kAll, f);
                if (f) queue[qn + __popc(ballot & ((1u << lane) - 1u))] = Candidate{i, z};
                qn += __popc(ballot);
                if (qn >= 32) drain();
              };
              // coarse bytes: bit 8*byte + 4*(j mod 2) + word of hit[j/2] = the byte is 255
              uint32_t hit[kG / 2] = {};
              {
                const PhiloxRow prow = ws.prow;
#pragma unroll
                for (int j = 0; j < kG; ++j) {
                  const uint4 cb = philox_call(p.round_key, prow, (uint32_t)(e_tile + e_lane + ((j ^ ga) << 4)) >> 4);
                  hit[j >> 1] |= ((ff_bytes(cb.x) >> 7) | (ff_bytes(cb.y) >> 6) | (ff_bytes(cb.z) >> 5) | (ff_bytes(cb.w) >> 4)) << (4 * (j & 1));
                }
              }
              // Entries with coarse byte 255 whose logit is not hopeless, one per lane and round.
              const float gate_all = logit_gate(best, ws.tau, kGumbelCapAll);
#pragma unroll 1
              for (;;) {
                const bool second = kG == 4 && hit[0] == 0u;
                uint32_t word = second ? hit[kG / 2 - 1] : hit[0];
                if (!__any_sync(kAll, word != 0u)) break;
                const int bit = __ffs((int)word) - 1;
                const int j = (second ? 2 : 0) + ((bit >> 2) & 1), k = 4 * (bit & 3) + (bit >> 3);
                const int e = e_lane + ((j ^ ga) << 4) + k;
                const bool f = word != 0u && e < n;
                word &= word - 1u;
                if (second) hit[kG / 2 - 1] = word; else hit[0] = word;
                float z = -CUDART_INF_F;
                if (f) z = lds_elem<DT>(base + (uint32_t)(e * F::kEsize));
                push(f && z > gate_all, (uint32_t)(e_tile + e), z);  // (passes over NaN and -inf too)
              }
              // Groups whose sum passed the gate: their entries above it, whatever the coarse byte.  While nothing is known
              // of the row's scores the gate is set just below the largest logit first, and again when those entries and the
              // ones with byte 255 have been scored.  Where many logits lie close to the largest (a high temperature, a flat
              // row: three lanes of four have one in their first vector) the latter alone give as good a bound: scoring a
              // tile's every entry cost as much as ten tiles' sums.
              constexpr int kCrowd = 24;
              constexpr float kFirstGate = 0.00422f;  // e^-2 2^-5: two units of score below the sample's largest
              float gate_hi = CUDART_INF_F, first_thr = CUDART_INF_F;
#pragma unroll 1
              for (int look = best == enc_neg_inf() ? 0 : 1; look < 2; ++look) {
                float gate, ethr;
                if (look == 0) {
                  gate = (-nRc - kMargin - 2.0f * kLog2e) / c;
                  ethr = kFirstGate;
                } else {
                  gate = logit_gate(best, ws.tau, kGumbelCapCoarse);
                  ethr = gate_threshold(best, nRc);
                }
                uint32_t over = 0u;  // bit j: the lane's group j passes
#pragma unroll
                for (int j = 0; j < kG; ++j) over |= (Zg[j] > ethr ? 1u : 0u) << j;
                if (look == 0) {
                  const uint4 v[1] = {lds128(B)};
                  if (__popc(__ballot_sync(kAll, vec_max<DT>(v) > gate)) > kCrowd) {
                    over = 0u;
                    gate = ethr = CUDART_INF_F;  // (none has been looked at)
                  }
                }
#pragma unroll 1
                while (__any_sync(kAll, over != 0u)) {  // one group per lane and round
                  const int j = over != 0u ? __ffs((int)over) - 1 : 0;
                  const int g = e_lane + ((j ^ ga) << 4);
                  uint32_t above = 0u;  // bit k: entry k of the group
                  // bf16: compared in pairs as they are (us with the 16 entries taken apart and now: 512 x 151,936 84.3, 81.7, 4,096 x 9,000
                  // 88.6, 85.1; fp32 gains nothing, 256 x 256,000 81.0, 82.0)
                  if (DT == 1) {
                    if (over != 0u) {
                      float zg = Zg[0];
#pragma unroll
                      for (int i = 1; i < kG; ++i) zg = j == i ? Zg[i] : zg;
                      const float top = zg > first_thr ? gate_hi : CUDART_INF_F;  // (entries above it have been looked at)
#pragma unroll
                      for (int i = 0; i < F::kVG; ++i) {
                        const uint4 v = lds128(base + (uint32_t)(g * F::kEsize + 16 * i));
                        above |= (entries_above<DT>(v, gate) & ~entries_above<DT>(v, top)) << (8 * i);
                      }
                      if (g + 16 > n) above &= g < n ? (1u << (n - g)) - 1u : 0u;
                    }
                  } else {
                    float z[16], zg = Zg[0];
#pragma unroll
                    for (int i = 1; i < kG; ++i) zg = j == i ? Zg[i] : zg;
                    load_group_smem<DT>(base + (uint32_t)(g * F::kEsize), z);
                    const float top = zg > first_thr ? gate_hi : CUDART_INF_F;
#pragma unroll
                    for (int k = 0; k < 16; ++k) above |= (z[k] > gate && z[k] <= top ? 1u : 0u) << k;
                    if (over == 0u) above = 0u;
                    if (g + 16 > n) above &= g < n ? (1u << (n - g)) - 1u : 0u;
                  }
                  over &= over - 1u;
#pragma unroll 1
                  while (__any_sync(kAll, above != 0u)) {
                    const int e = g + __ffs((int)above) - 1;
                    const bool f = above != 0u;
                    above &= above - 1u;
                    float z = 0.f;
                    if (f) z = lds_elem<DT>(base + (uint32_t)(e * F::kEsize));
                    push(f, (uint32_t)(e_tile + e) | kAnyByte, z);
                  }
                }
                if (look == 0) {
                  while (qn > 0) drain();
                  gate_hi = gate;
                  first_thr = ethr;
                }
              }
              if (best > before && lane == 0) post_best(bests, seg, best);
            }
            if (SAMPLER == 1) {
              float S = Z;
#pragma unroll
              for (int o = 1; o < F::kLB; o <<= 1) S += __shfl_xor_sync(kAll, S, o);
              if (lane % F::kLB == 0) {  // + ln of the block's sum of exp(z/tau); -inf for a block without mass
                float &y = score[(tile - first) * F::kBT + lane / F::kLB];
                y = S > 0.f ? y + (lg2f(S) - nRc) * kLn2f : -CUDART_INF_F;
              }
            }
          }
        }
        ++done;
        __syncwarp();  // every lane has read the slot
        feed(false);
      }
      if (given_up) break;
      // The strip's record.  Lanes 0..15 add up Z, lanes 16..31 W.
      {
        const bool low = lane < 16;
        float x = low ? Zs : Ws;
        x += __shfl_xor_sync(kAll, low ? Ws : Zs, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(kAll, x, o);
        float *const rec = reinterpret_cast<float *>(&sm.record[q & (p.ring - 1)]);
        if ((lane & 15) == 0) *reinterpret_cast<float2 *>(rec + (low ? 0 : 2)) = low ? make_float2(-nRc, x) : make_float2(x, zmax);
        if (SAMPLER == 1 && !(mode & (kGreedy | kUnusable))) hand_in_blocks(score, (end - first) * F::kBT, first * F::kBT, blocks + (q & (p.ring - 1)));
      }
      ++count;
      ++strip;
      __syncwarp();
      // the warp's next strip has been taken already (or there is none): is it of the same segment?
      more = strip < strips && sm.meta[warp][strip & 1].seg == seg;
    } while (more);
    if (given_up) break;
    if (SAMPLER == 0) {
      const Candidate *const queue = reinterpret_cast<const Candidate *>(extra) + warp * kQueueCap;
      if (qn > 0) score_candidates(queue, qn, best);  // (fewer than 32)
    }
    // ------------------------------------------------------------------ the warp hands in what it has of the segment
    int state = 0;  // 1: the segment is complete, 2: a wait was given up
    if (lane == 0) {
      Segment &sg = sm.seg[seg & (p.ring - 1)];
      if (err) atomicOr(&sg.err, err);
      if (SAMPLER >= 0 && ws.tb[0] >= 0 && !hand_in_leaders(seg)) state = 2;
      if (state == 0) {
        __threadfence_block();
        state = atomicAdd(&sg.arrived, count) + count == need;
      }
    }
    state = __shfl_sync(kAll, state, 0);
    if (state == 2) break;
    if (state == 1) {
      __threadfence_block();
      if (!finish_segment<DT, SAMPLER>(seg, ws.row, ws.tau, blocks)) break;
    }
    __syncwarp();
  }
  if (timed_out()) {
    // Given up: see the copies still in flight land (bounded) before the CTA's shared memory goes away.
    const u64 t0 = global_ns();
    for (int i = done; i < fetched; ++i) {
      const int st = i % kStages;
      for (uint32_t it = 1; !mbar_try_wait(&sm.full[warp][st], (uint32_t)(i / kStages) & 1u); ++it)
        if ((it & 63u) == 0u && global_ns() - t0 > sm.p.wait_ns) break;
    }
  }
  int gone = 0;
  if (lane == 0) {
    __threadfence_block();
    gone = atomicAdd(&sm.exited, 1) + 1;
  }
  if (__shfl_sync(kAll, gone, 0) == kWarps && timed_out()) mark_unfinished(live_rows);
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
// Per device and kernel variant, once: opt in to the dynamic shared memory and ask how many SMs there are.
template <int DT, int SAMPLER>
cudaError_t resident_ctas(int64_t &out) {
  static std::mutex lock;
  static int64_t cache[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> hold(lock);
  if (cache[dev] == 0) {
    auto kern = rows_kernel<DT, SAMPLER>;
    const size_t dyn = dyn_smem_bytes<SAMPLER>(SAMPLER < 0);
    int sms = 0, per_sm = 0;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, dyn);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorLaunchOutOfResources;
    cache[dev] = sms < kMaxGrid ? sms : kMaxGrid;
  }
  out = cache[dev];
  return cudaSuccess;
}

unsigned long long next_call_id() {
  static std::atomic<unsigned long long> counter{
      (unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count() & ((1ull << 40) - 1)};
  return (counter.fetch_add(1) + 1) & ((1ull << 48) - 1);
}

// Test hook state (see arm_stall).
std::atomic<long long> g_stall_tile{-1};
std::atomic<unsigned long long> g_stall_wait_ns{0};

size_t pieces_bytes() { return (size_t)kMaxGrid * 2 * kPieceBytes; }

// A launch that cannot give every SM as many tiles as it has warps spreads out until a CTA has this many: one tile for each of
// the SM's four schedulers.
constexpr int64_t kStripsPerCta = 4;

template <int DT, int SAMPLER>
cudaError_t launch_one(RowsParams p, int64_t rows, void *workspace, size_t workspace_bytes, cudaStream_t stream) {
  int64_t ctas = 0;
  cudaError_t e = resident_ctas<DT, SAMPLER>(ctas);
  if (e != cudaSuccess) return e;
  const int64_t tpr = ((int64_t)p.V + Fmt<DT>::kTileE - 1) / Fmt<DT>::kTileE;
  const int64_t strip = strip_tiles(rows, tpr, ctas, SAMPLER, Fmt<DT>::kTileE), spr = (tpr + strip - 1) / strip;
  const bool can_cut = workspace != nullptr && workspace_bytes >= pieces_bytes();
  p.tpr = (int)tpr;
  p.strip_tiles = (int)strip;
  p.spr = (int)spr;
  p.inv_spr = 1.0f / (float)spr;
  p.unit = can_cut ? 1 : (int)spr;
  p.ring = kRing;
  p.ws_pieces = can_cut ? static_cast<unsigned char *>(workspace) : nullptr;
  p.wait_ns = kDefaultWaitNs;
  const long long stall = g_stall_tile.exchange(-1);  // (row * tpr + tile within the row)
  p.stall_src = nullptr;
  if (stall >= 0) {
    p.stall_src = p.logits + stall / tpr * p.row_bytes + stall % tpr * kTileBytes;
    p.wait_ns = g_stall_wait_ns.load();
  }
  // Strip numbers of a launch stay within 31 bits and those of a CTA within what place_of counts exactly, the rows of a CTA's
  // run within its list when there is a mask.
  int64_t most = ((int64_t(1) << 30) - 1) / spr;
  const int64_t per_cta = ((int64_t(1) << 22) - 1) / spr;  // whole rows, where rows are not cut
  const int64_t exact = can_cut ? ctas * (int64_t(1) << 22) / spr : ctas * (per_cta > 0 ? per_cta : 1);
  if (most > exact) most = exact;
  if (p.mask != nullptr && most > ctas * (kMaxLive - 2)) most = ctas * (kMaxLive - 2);
  if (most < 1) most = 1;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = dyn_smem_bytes<SAMPLER>(p.mask != nullptr);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  for (int64_t done = 0; done < rows; done += most) {
    const int64_t now = rows - done < most ? rows - done : most;
    p.rows = (uint32_t)now;
    int64_t grid = can_cut ? (now * spr + kStripsPerCta - 1) / kStripsPerCta : now;
    if (grid > ctas) grid = ctas;
    p.call_id = next_call_id();
    cfg.gridDim = dim3((unsigned)grid);
    e = cudaLaunchKernelEx(&cfg, rows_kernel<DT, SAMPLER>, p);
    if (e != cudaSuccess) return e;
    p.logits += now * p.row_bytes;
    p.row_base += (uint32_t)now;
    if (p.temps) p.temps += now;
    if (p.targets) p.targets += now;
    if (p.mask) p.mask += now;
    if (p.out_tok) p.out_tok += now;
    if (p.out_logp) p.out_logp += now;
    if (p.out_ent) p.out_ent += now;
    if (p.out_gap) p.out_gap += now;
  }
  return cudaSuccess;
}

}  // namespace

size_t rows_workspace_bytes() { return pieces_bytes(); }
// 144 bytes per 4 KiB of logits and 16 per row beyond the pieces of cut rows are part of the call's contract (callers
// size their scratch once and for all); this implementation does not touch them.
size_t sample_workspace_bytes(int dtype, int64_t rows, int64_t V) {
  if (rows < 0 || V < 1) return pieces_bytes();
  const int64_t tile = dtype == 0 ? Fmt<0>::kTileE : Fmt<1>::kTileE;
  return pieces_bytes() + (size_t)rows * (16 + (size_t)((V + tile - 1) / tile) * 144);
}

void arm_stall(int64_t stall_tile, unsigned long long wait_ns) {
  g_stall_wait_ns.store(wait_ns);
  g_stall_tile.store(stall_tile);
}

cudaError_t launch_rows(const RowsParams &p, int64_t rows, int dtype, int sampler, void *workspace, size_t workspace_bytes,
                        cudaStream_t stream) {
  if ((dtype != 0 && dtype != 1) || sampler < -1 || sampler > 1) return cudaErrorInvalidValue;
  long long stall = g_stall_tile.load();
  if (stall < 0) {  // (else the hook stalls a tile of the streaming kernel)
    if (stall < -1) stall = g_stall_tile.exchange(-1);
    bool taken = false;
    const cudaError_t e = launch_rows_direct(p, rows, dtype, sampler, RowStall{-2 - stall, g_stall_wait_ns.load()}, stream, taken);
    if (taken || e != cudaSuccess) return e;
  }
  if (dtype == 0) {
    if (sampler < 0) return launch_one<0, -1>(p, rows, workspace, workspace_bytes, stream);
    if (sampler == 0) return launch_one<0, 0>(p, rows, workspace, workspace_bytes, stream);
    if (sampler == 1) return launch_one<0, 1>(p, rows, workspace, workspace_bytes, stream);
  } else if (dtype == 1) {
    if (sampler < 0) return launch_one<1, -1>(p, rows, workspace, workspace_bytes, stream);
    if (sampler == 0) return launch_one<1, 0>(p, rows, workspace, workspace_bytes, stream);
    if (sampler == 1) return launch_one<1, 1>(p, rows, workspace, workspace_bytes, stream);
  }
  return cudaErrorInvalidValue;
}

}  // namespace e3
