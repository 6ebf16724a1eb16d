// Work split of the row kernel: which strips a CTA takes, in which order they are handed out, and which places of
// its rings they use.  Plain arithmetic without device state, so that the hand-out can be played through on the host
// as well; P is RowsParams or anything with its fields spr, unit, ring and inv_spr.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define E3_SPLIT __host__ __device__ __forceinline__
#else
#define E3_SPLIT inline
#endif

namespace e3 {
namespace {

constexpr int kWarps = 24;           // one CTA per SM: 80 registers a thread
constexpr int kRing = 256;           // strips whose records the CTA keeps (RowsParams::ring)
// Most tiles of a strip: of the statistics (sampler -1), of sampler 0, of sampler 1.
constexpr int longest_strip(int sampler, bool bf16) { return sampler == 0 ? 25 : (bf16 ? (sampler == 1 ? 13 : 14) : 24); }
constexpr int kLongRunStrip = 8;  // ... of runs of many strips per warp (but for sampler 0)

// The CTA's run of strips, numbered q = 0..len-1 in hand-out order: vocabulary order, except that the strips of the last row
// come first when that row is cut.
struct Run {
  uint32_t q, r;        // all units = grid * q + r: CTA b starts at unit b*q + min(b, r)
  int len;              // strips
  uint32_t r0;          // row of the first strip (with a mask: its rank among the rows let through)
  int n;                // rows touched
  int lo0, hin;         // first strip within the first row; end strip within the last row (1..spr)
  int head;             // strips of the last row that come first (0: none)
};
// Strip q of the run.
struct Place {
  int j;                // row: position in vocabulary order
  int strip, lo, hi;    // strip within the row; strips of the row in this run
  int q0;               // number of the row's first strip within the run
};

template <class P>
E3_SPLIT uint32_t first_strip_of(const P &p, const Run &run, uint32_t b) {
  return (b * run.q + (b < run.r ? b : run.r)) * (uint32_t)p.unit;
}
template <class P>
E3_SPLIT int cta_of_strip(const P &p, const Run &run, uint32_t t) {
  const uint32_t u = t / (uint32_t)p.unit, big = run.r * (run.q + 1);
  return (int)(u < big ? u / (run.q + 1) : run.r + (u - big) / run.q);
}
// The run of CTA b of `ctas`.  live: rows that are streamed (all, or those the mask lets through).
template <class P>
E3_SPLIT void set_run(const P &p, Run &run, uint32_t live, uint32_t b, uint32_t ctas) {
  const uint32_t spr = (uint32_t)p.spr, unit = (uint32_t)p.unit, units = live * (spr / unit);
  run.q = units / ctas;
  run.r = units - run.q * ctas;
  const uint32_t t0 = first_strip_of(p, run, b), len = (run.q + (b < run.r ? 1u : 0u)) * unit;
  run.len = (int)len;
  run.r0 = t0 / spr;
  run.lo0 = (int)(t0 - run.r0 * spr);
  const uint32_t end = t0 + len, row_last = len ? (end - 1u) / spr : run.r0;
  run.hin = (int)(end - row_last * spr);
  run.n = len ? (int)(row_last - run.r0) + 1 : 0;
  run.head = run.n > 1 && run.hin < (int)spr ? run.hin : 0;
}
template <class P>
E3_SPLIT Place place_of(const P &p, const Run &run, int q) {
  Place w;
  const bool head = q < run.head;
  const int u = head ? q : q - run.head + run.lo0;  // strips from the start of the run's first row on (head: of its last)
  int k = (int)((float)u * p.inv_spr);              // rows passed; off by one at most (u < 2^23)
  int strip = u - k * p.spr;
  if (strip >= p.spr) { strip -= p.spr; ++k; }
  if (strip < 0) { strip += p.spr; --k; }
  w.j = head ? run.n - 1 : k;
  w.strip = strip;
  w.lo = w.j == 0 ? run.lo0 : 0;
  w.hi = w.j == run.n - 1 ? run.hin : p.spr;
  w.q0 = q - (strip - w.lo);
  return w;
}
// Strips of the segment that begins at w.
template <class P>
E3_SPLIT int segment_strips(const P &p, const Place &w) {
  return w.hi - w.strip < p.ring / 2 ? w.hi - w.strip : p.ring / 2;
}
// Number (in the run) of the first strip of the segment that strip w belongs to.
template <class P>
E3_SPLIT int segment_start(const P &p, const Place &w) {
  return w.q0 + ((w.strip - w.lo) & ~(p.ring / 2 - 1));
}

// Whether strip q of the segment that begins with strip number seg may be taken.  freed(place): 1 + number of the last strip
// at this ring place whose record has been merged.  The segment's own state lies at the place of its first strip: while a short
// segment one ring length before waits for a slow warp, that place is still in use although the strip's own may be free.
// Segments are handed out in their order, so the oldest one that is not finished always finds its places free.
template <class P, class F>
E3_SPLIT bool may_take(const P &p, int q, int seg, F freed) {
  return freed(q & (p.ring - 1)) == q - p.ring + 1 && freed(seg & (p.ring - 1)) == seg - p.ring + 1;
}

// A row piece of several segments (longer than half a ring) keeps a state in which they are merged in their order: one place for
// the piece that the run begins with, three for the others in turn.  The places of rows j and j + 3 cannot meet: two whole rows,
// so more than a ring of strips, lie between them.  While the last strip e of row j is not finished, strip e + ring cannot
// be taken; it belongs to a full segment, whose records therefore stay, and so the strips one ring behind that segment cannot be
// taken either.  These are more than there are warps (half a ring is at least 32 where a run is longer than a ring), and row
// j + 3 has no full segment before them.
constexpr int kLong = 4;
E3_SPLIT int long_piece_place(const Place &w) {
  return w.q0 == 0 && w.j > 0 ? kLong - 1 : w.j % (kLong - 1);
}

// ---- host: lengths of the strips
// Tiles per strip.  Strips of one length keep the warps of an SM in step, so that a run of a few strips per warp takes
// whole waves: in a short run one strip per warp is all, the shortest that does it (151,936 bf16 entries a row, us for the lengths
// below it, at it and behind it: sampler 1 300 rows 32.0, 28.0, 28.4; sampler 0 512 rows 6, 12, 13, 15 tiles 95, 87, 86, 94).  For the
// statistics and sampler 1 that pays up to 14 and 13 tiles of bf16 and 24 of fp32, which hold half as many entries (against 8 tiles:
// statistics 256 x 256,000 19 tiles 46.5 and 50.6, 300 x 256,000 23 tiles 51.4 and 54.7, 512 x 100,000 17 tiles 37.7 and 39.6, but 768 x 100,000 25
// tiles 52.0 and 50.7, 400 x 256,000 32 tiles 70.7 and 68.5; sampler 1 256 x 256,000 49.8 and 56.9, 512 x 100,000 40.5 and 48.0), and a
// few blocks may hold a strip more than they have warps where the last strip of a row is short (statistics 448 rows 10 tiles 28.2, 11
// tiles 29.7; 512 rows 12 tiles 32.6, 13 tiles 32.8; 593 rows 14 tiles 34.3, 8 tiles 36.9; 1,200 x 50,257 10 tiles 38.2, 8 tiles 40.4; sampler 1 512
// rows 12 tiles 39.0, 13 tiles 40.5) but not where it is long (256 x 256,000 fp32 18 tiles 51.3) or where strips are short anyway
// (512 x 32,000 fp32 5 tiles 18.1, 6 tiles 17.3).
// In a long run the waves dissolve: there a strip is as long as makes its own cost small (taking it and handing in its record
// cost a warp about as many instructions as a tile's sums; for sampler 0 the first bound and the last look at the queue cost twice
// that: 4,096 rows 12 tiles 537, 25 tiles 494; sampler 1, 4,096 rows 4, 6, 8, 12 tiles 245, 230, 221, 230, 1,024 rows 72, 69, 67, 67).
inline int strip_tiles(int64_t rows, int64_t tpr, int64_t ctas, int sampler, int tile_entries) {
  const int64_t warps = ctas * kWarps, per_warp = rows * tpr / warps;
  const int64_t longest = longest_strip(sampler, tile_entries > 1024);
  for (int64_t n = per_warp < 1 ? 1 : per_warp; n <= longest; ++n) {
    const int64_t spr = (tpr + n - 1) / n, last = tpr - (spr - 1) * n, more = rows * spr - warps;
    if (more <= 0 || (sampler != 0 && n >= 8 && 2 * last <= n && more <= warps / 64)) return (int)n;
  }
  return sampler == 0 ? (int)longest : kLongRunStrip;
}

}  // namespace
}  // namespace e3
