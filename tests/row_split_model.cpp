// Plays the hand-out of strips of the row kernel through on the host, with the kernel's own split arithmetic: the warps of a CTA
// take strips ahead, sum them, hand in what they have of a segment and merge segments, one strip of the run taking `slow` times as
// long as the others.  Finds: state of a segment or of a long row piece that is used while an earlier one still lives in its
// place, a record that is overwritten before it has been merged, and warps that wait for each other.
//
// arguments: rows tiles_per_row sampler ctas slow, then the CTA (-1: every one) and how far apart the strips are that are slow in
// turn
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "e3_rows_split.cuh"

using namespace e3;

struct Split {
  int spr, unit, ring;
  float inv_spr;
};

struct Warp {
  int taken[2], n = 0;      // strips in hand, in their order
  int waiting;              // handed out, without a place yet (-1: none)
  bool dry = false;
  enum { kIdle, kStart, kSumming, kMerge, kGone } at = kIdle;
  double until = 0;         // end of the strip's sums
  int count = 0;            // strips of the segment summed
  int seg = -1;
};

struct Cta {
  Split p;
  Run run;
  int next = kWarps, slow_strip, slow;
  std::vector<int> freed, owner, arrived, record;
  int piece_owner[8], piece_turn[8];
  bool piece_live[8];
  Warp w[kWarps];
  const char *fault = nullptr;
  int fault_at = 0;

  Place place(int q) const { return place_of(p, run, q); }
  int mask() const { return p.ring - 1; }
  void fail(const char *what, int q) {
    if (!fault) { fault = what; fault_at = q; }
  }
  // the state of segment seg is written
  void touch(int seg) {
    int &o = owner[seg & mask()];
    if (o < 0) o = seg;
    else if (o != seg) fail("segment state", seg);
  }
  bool take(Warp &x) {
    int q = x.waiting;
    x.waiting = -1;
    if (q < 0) q = next++;
    if (q >= run.len) {
      x.dry = true;
      return false;
    }
    if (!may_take(p, q, segment_start(p, place(q)), [&](int at) { return freed[at]; })) {
      x.waiting = q;
      return false;
    }
    if (record[q & mask()] >= 0) fail("record", q);
    record[q & mask()] = q;
    x.taken[x.n++] = q;
    return true;
  }
  // One step of a warp at time t, if it can make one.
  bool step(Warp &x, double t) {
    switch (x.at) {
      case Warp::kIdle:
        if (x.n == 0 && !x.dry && !take(x) && !x.dry) return false;
        if (x.n == 0) {
          x.at = Warp::kGone;
          return true;
        }
        x.at = Warp::kStart;
        return true;
      case Warp::kStart: {
        const int q = x.taken[0], seg = segment_start(p, place(q));
        if (x.seg < 0) {
          x.seg = seg;
          x.count = 0;
        }
        if (x.n < 2 && !x.dry) take(x);
        x.until = t + (q == slow_strip ? slow : 1.0 + 0.01 * (q % 7));
        x.at = Warp::kSumming;
        return true;
      }
      case Warp::kSumming: {
        if (t < x.until) return false;
        touch(x.seg);  // the target's logit
        ++x.count;
        if (x.n < 2 && !x.dry) take(x);
        x.taken[0] = x.taken[1];
        --x.n;
        if (x.n > 0 && segment_start(p, place(x.taken[0])) == x.seg) {
          x.at = Warp::kStart;
          return true;
        }
        int &a = arrived[x.seg & mask()];
        a += x.count;
        const int need = segment_strips(p, place(x.seg));
        if (a > need) fail("count", x.seg);
        x.at = a == need ? Warp::kMerge : Warp::kIdle;
        if (a == need) {
          a = 0;
          owner[x.seg & mask()] = -1;
        } else {
          x.seg = -1;
        }
        return true;
      }
      case Warp::kMerge: {
        const int q = x.seg, half = p.ring / 2;
        const Place w = place(q);
        const int n = segment_strips(p, w), turn = (w.strip - w.lo) / half;
        const bool last = w.strip + n == w.hi;
        if (w.hi - w.lo > half) {
          const int at = long_piece_place(w);
          if (at < 0 || at >= kLong) { fail("long piece number", q); return false; }
          if (turn > 0 && !(piece_owner[at] == w.q0 && piece_turn[at] == turn)) return false;
          if (turn == 0 && piece_live[at]) fail("long piece", q);
          piece_owner[at] = w.q0;
          piece_turn[at] = turn + 1;
          piece_live[at] = !last;
        }
        for (int i = 0; i < n; ++i) {
          if (record[(q + i) & mask()] != q + i) fail("record", q + i);
          record[(q + i) & mask()] = -1;
          freed[(q + i) & mask()] = q + i + 1;
        }
        x.seg = -1;
        x.at = Warp::kIdle;
        return true;
      }
      case Warp::kGone: return false;
    }
    return false;
  }
  void play() {
    freed.resize(p.ring);
    for (int i = 0; i < p.ring; ++i) freed[i] = i - p.ring + 1;
    owner.assign(p.ring, -1);
    record.assign(p.ring, -1);
    arrived.assign(p.ring, 0);
    for (int i = 0; i < 8; ++i) { piece_owner[i] = -1; piece_turn[i] = 0; piece_live[i] = false; }
    for (int i = 0; i < kWarps; ++i) w[i].waiting = i;
    for (double t = 0; !fault;) {
      bool any = false;
      for (Warp &x : w) any |= step(x, t);
      if (any) continue;
      double then = 1e300;
      bool left = false;
      for (const Warp &x : w) {
        left |= x.at != Warp::kGone;
        if (x.at == Warp::kSumming && x.until > t && x.until < then) then = x.until;
      }
      if (!left) break;
      if (then == 1e300) fail("no progress", next);
      t = then;
    }
    for (int q = 0; q < run.len && !fault; ++q)
      if (freed[q & mask()] < q + 1) fail("unfinished", q);
  }
};

int main(int argc, char **argv) {
  if (argc != 8) return 2;
  const long rows = atol(argv[1]), tpr = atol(argv[2]);
  const int sampler = atoi(argv[3]), ctas = atoi(argv[4]), slow = atoi(argv[5]), cta = atoi(argv[6]), apart = atoi(argv[7]);
  const int strip = strip_tiles(rows, tpr, ctas, sampler, 2048);
  Split p;
  p.spr = (int)((tpr + strip - 1) / strip);
  p.unit = 1;
  p.ring = kRing;
  p.inv_spr = 1.0f / (float)p.spr;
  long faults = 0, plays = 0;
  int longest = 0;
  for (int b = cta < 0 ? 0 : cta; b < (cta < 0 ? ctas : cta + 1); ++b) {
    Cta c;
    c.p = p;
    set_run(p, c.run, (uint32_t)rows, (uint32_t)b, (uint32_t)ctas);
    if (c.run.len > longest) longest = c.run.len;
    for (int s = b % apart; s < c.run.len; s += apart, ++plays) {
      Cta d = c;
      d.slow_strip = s;
      d.slow = slow;
      d.play();
      if (d.fault && faults++ == 0) printf("CTA %d, slow strip %d: %s, strip %d\n", b, s, d.fault, d.fault_at);
    }
  }
  printf("%ld plays, %ld faults; %d tiles a strip, %d strips a row, run of %d, ring %d\n", plays, faults, strip, p.spr, longest, p.ring);
  return faults ? 1 : 0;
}
