// Shared declarations of the row kernel (host side of the launch and device parameters).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace e3 {

constexpr int kGroup = 16;                   // vocabulary entries per coarse Philox call
constexpr int kLaneBytes = 128;              // bytes a thread takes from one tile
constexpr int kTileBytes = 32 * kLaneBytes;  // 4 KiB: what a warp sums at a time
constexpr int kMaxGrid = 1024;               // CTAs the piece workspace is sized for
constexpr unsigned long long kDefaultWaitNs = 2000000000ull;  // limit of a wait inside a kernel: two seconds
constexpr size_t kPieceBytes = 128;          // one partial row state in the workspace

enum RowsMode : int { kModeSample = 0, kModeTargets = 1 };

// Bits of the optional device status word.
enum : int { kStatusTimeout = 1 };

struct RowsParams {
  const char *logits;
  int64_t row_bytes;        // bytes from one row to the next
  uint32_t rows;            // rows of this launch
  int V;
  const float *temps;       // per-row temperature, or nullptr -> temp_scalar
  float temp_scalar;
  const int32_t *targets;   // kModeTargets
  const uint8_t *mask;      // kModeTargets, may be nullptr
  int32_t *out_tok;         // kModeSample
  float *out_logp;
  float *out_ent;
  float *out_gap;           // may be nullptr
  int32_t *status;          // may be nullptr: kStatusTimeout is OR-ed in when a bounded wait ran out
  uint32_t round_key[20];   // Philox round keys: key_lo + r*W0, key_hi + r*W1, r = 0..9
  uint32_t ctr_lo;          // low word of the step counter
  uint32_t ctr_hi8;         // (high bits of the step counter) << 8; the stream tag is OR-ed in
  uint32_t row_base;
  int mode;
  float slack_scale;        // 1; the audit sampler widens the fp32 score slack so that rows are settled in fp64
  // work split: a row has spr strips of strip_tiles tiles (the last one may be shorter); CTA b of the grid takes an equal,
  // contiguous share of all strips (of the rows the mask lets through), in units of `unit` strips (1, or spr when rows are not
  // to be cut)
  int tpr, spr, strip_tiles, unit;
  float inv_spr;                 // 1 / spr
  int ring;                      // strips whose records a CTA keeps (a power of two); a segment is half of it
  unsigned char *ws_pieces;      // [grid][2] partial states of cut rows, kPieceBytes each, every word tagged with the call id
  unsigned long long call_id;    // unique per call within the process (48 bits)
  unsigned long long wait_ns;    // time after which a wait inside the kernel gives up
  const char *stall_src;         // test hook: the copy of the tile that begins here is never issued (short calls: the row that begins here
                                 // waits for more than is handed over); nullptr = none
};

size_t rows_workspace_bytes();                                      // cut rows
size_t sample_workspace_bytes(int dtype, int64_t rows, int64_t V);  // e3_sample: what the call's contract asks for

// Test hook: the next launch_rows of this process gives up waiting after wait_ns and never issues the copy of
// tile stall_tile; below -1: if it is a short call, row -2 - stall_tile waits for a hand-over that never comes.  One shot.
void arm_stall(int64_t stall_tile, unsigned long long wait_ns);

// Launches the row kernel over `rows` rows (any number: more than one launch takes at a time are split).
// sampler: -1 = none (targets given), 0 = per-token Gumbel-max, 1 = blocked Gumbel-max (the caller sets slack_scale).
// workspace may be nullptr: rows are then never cut (whole rows per CTA).
cudaError_t launch_rows(const RowsParams &p, int64_t rows, int dtype, int sampler, void *workspace, size_t workspace_bytes,
                        cudaStream_t stream);

// The kernel of short calls; taken: whether the call is one (if not, nothing has been launched).
// Blocks per row that it gives such a call on a device of that many SMs whose largest cluster has `largest` blocks (0: not a short call).
int direct_ctas(int64_t rows, int64_t V, int dtype, int sampler, bool mask, int sms, int largest);
struct RowStall {  // test hook: the row whose first block waits for more than the others hand over (< 0: none), and the limit of that wait
  long long row;
  unsigned long long wait_ns;
};
cudaError_t launch_rows_direct(const RowsParams &p, int64_t rows, int dtype, int sampler, const RowStall &stall, cudaStream_t stream, bool &taken);

}  // namespace e3
