// How the query stage's work is dealt out to CTAs: plain arithmetic, of the host but for the last function, which the CTAs evaluate for themselves.  Apart
// from CUDA so that it can be compiled and tested alone.
#pragma once

#include <algorithm>

#ifdef __CUDACC__
#define AS_HD __host__ __device__ __forceinline__
#else
#define AS_HD inline
#endif

struct AsUnits {
  int nx = 0, n_pairs = 0;       // two-tile units per (batch, head); over all (batch, head) pairs
  int n_single = 0;              // units of a (batch, head)'s last tile alone: one per (batch, head) or none
  int n_rounds = 0;              // rounds in which every CTA has a two-tile unit
  int split_last = 0;            // 1: the two-tile units left over after those rounds are cut in two, one tile per CTA
  int share = 0;                 // key tiles of a CTA in the last round; 0: units are whole
};

// What the plan has to know of a layer: key tiles, whether there is a linear branch, chunks of 128 features, slices of the hidden width (0: one layer), whether the
// general kernel runs it (biases, powers beyond 2).
struct AsLoop { int d, nkv, lin, fc, slices, gen; };

// How the 128-row tiles of a launch are dealt out to the CTAs: full rounds of two-tile units, then one last round.  A head
// with an odd number of tiles either has its last tile in a unit of its own, or in a two-tile unit whose other half is
// past the end; which is better depends on what the last round comes to (N = 7800, 61 tiles in each of 12 heads, 148 SMs:
// 360 units and 12 single tiles are two rounds and 140 tiles alone, 372 units are two rounds and 76 units: layer 92.8 -> 88.6
// us; N = 1024 with 2 heads on 16 CTAs instead of 8: 22.5 -> 21.4).  Returns the
// number of CTAs.
inline int as_plan_units(AsUnits& p, int N, int BH, int sms) {
  const int tiles = (N + 127) / 128;
  double best = 0.;
  int grid = 0;
  for (int alone = 0; alone <= (tiles & 1); ++alone) {
    const int nx = (tiles + 1 - alone) / 2, pairs = nx * BH, single = alone * BH;
    const int rounds = pairs / sms, left = pairs - rounds * sms;
    const bool cut = 2 * left + single <= sms;
    const int last = (cut ? 2 * left : left) + single;
    if (last > sms) continue;                        // one last round only
    const double t = rounds + (last == 0 ? 0. : (cut || left == 0) ? 0.7 : 1.);
    if (grid != 0 && t > best) continue;             // (no worse: without empty tiles)
    best = t;
    p.nx = nx; p.n_pairs = pairs; p.n_single = single; p.n_rounds = rounds; p.split_last = cut ? 1 : 0;
    grid = rounds > 0 ? sms : last;
  }
  return grid;
}
// no CTA has more than one tile: one group works, the other one has nothing to do
inline bool as_one_tile_each(const AsUnits& p) { return p.n_rounds == 0 && p.split_last; }
// Threads per row of the kernel with a key loop (after as_plan_units and as_plan_parts).  Two (sixteen compute warps) hide more of the latencies; one draws less power per
// exponential and has 168 registers where two have 96.  At d = 64 always two.  At d = 128 the gain of two over one in the query stage, on layers that differ
// in the number of key tiles only (12 heads, N = 32760, 16384, 7800, 1560; 2 - 46 heads of 20140 - 442 rows; in bursts of 3 ms / in runs of 0.06 - 0.12 s,
// which the power cap slows down where a CTA has several units):
//   a CTA has one tile at most (2 heads, N = 4096), so that one group has the SM to itself: 4 - 10 % at any length with one layer, 0 - 5 % with two;
//   one layer without biases: 4 tiles 0 - 8 % / 0 - 8 %, 16 0 - 3 / -1 - +3, 31 0 - 2 / -2 - +3, 40 -1 - +2 / -2 - +3, 96 -1 - +1 / -3 - -1; F = 256 alike;
//   one layer with biases or powers beyond 2: 8 tiles 4 - 12 / 2 - 13, 16 2 - 7 / 2 - 6, 31 2 - 5 / -3 - +3, 48 1 - 4 / 0 - 2, 64 0 - 4 / -1 - +2;
//   two layers with one feature chunk: 0 tiles -14 - 0 / -11 - 0, 4 and more -7 - 0 / -8 - 0, biased or not; with two, which one thread has
//   to keep in its registers: 0 tiles -5 - 0 / -6 - 0, else -3 - +1 / -4 - +3, with biases or powers beyond 2 4 - 30 at few tiles, 16 4 - 16 / 2 - 12, 48 1 - 10 / -1 - +5.
// That is the query stage over and over.  In a whole layer its instructions arrive cold, which costs one thread's longer code more: of two-layer
// maps of few rounds 256 / 256 are 2 - 7 % faster with two (N = 1560 ... 9360, 0 to 10 tiles), 128 / 128 0 - 3 %.
inline int as_threads_per_row(const AsUnits& p, const AsLoop& l) {
  if (l.d == 64 || as_one_tile_each(p)) return 2;
  if (p.share > 0) return 1;                         // (with parts the key loop does not stay in 96 registers: full softmax, 4 heads of N = 5600 61 -> 67 us)
  if (l.slices == 0) return l.nkv <= (l.gen ? 48 : 31) ? 2 : 1;
  if (l.gen && l.fc > 1) return l.nkv <= 48 ? 2 : 1;
  if (l.fc == 1 && l.nkv == 0) return 1;
  return l.nkv <= 16 && p.n_rounds < 4 ? 2 : 1;
}

// The last round with the key loops of its units cut across CTAs: the key tiles of what is left after the full rounds, unit after unit, are dealt out in equal
// shares, so that a CTA finishes one unit and leaves the beginning of the next one to the CTA after it (as_deal_parts).  Whole units, or lone tiles, leave
// much of the GPU idle where a little more than half of a round is left, or little work in long loops.  What it costs: O of a part through L2, the wait for it, a
// unit's fixed work twice, 5 - 8 us in all (the 10000 or 14000 and 2500 clk below).  Taken where the rounds that as_plan_units deals out take longer by more than
// that, in the clocks that a key tile of a unit, one of a lone tile and a unit's tail were measured at.  Whole calls, units whole -> in parts (us): full softmax,
// d = 128, 2 heads of N = 10000 135 -> 86, 1 of 15000 126 -> 96, 1 of 8000 72 -> 49, 4 of 5600 79 -> 61, 7 of 3999 59 -> 57; d = 64, 1 of 8000 70 -> 38, 4 of
// 5600 76 -> 57; one key in two, 2 of 12288 102 -> 87, d = 64 94 -> 80; one rank of four of the 81-frame layer (two rounds and 88 units) 205 -> 202.  `gain` below: the
// most that they may take of what whole units take by this rule.  Measured there, in parts against whole units:
//   0.96 at d = 64, and at d = 128 where whole units have one thread per row as well: with full rounds in front 0.84 - 0.95 by the rule are 0.84 - 0.99 at d = 64
//     (28 layers: 5 heads of N = 9467 194 -> 167 us, 24 of 6582 370 -> 367; 23 layers without: 0.87 - 0.96 are 0.79 - 0.95), 0.83 - 0.96 are 0.84 - 0.99 at d = 128.
//     (The kernels for parts at d = 64 reload 110 - 180 bytes a key tile where the others reload 20 - 80; these figures have that in them);
//   0.90 at d = 128 where whole units have two threads per row (in parts there is one: see as_threads_per_row), 2 - 6 % more than the rule knows: 0.81 - 0.90 are
//     0.88 - 0.99, 0.92 - 0.96 are 0.97 - 1.06 (1 head of N = 6803, one key in two, 49 -> 52 us; 7 of 8689, one in three, 112 -> 118; with biases 7 of 8319 115 -> 122);
//   0.95 for two layers, whose tails cost more than the rule's: 0.76 - 0.94 are 0.85 - 0.96, 0.957 is 1.02 (7 of 8319, one in three, 127 -> 130).
// Called behind as_plan_units.  Returns the number of CTAs, 0: units stay whole.
inline int as_plan_parts(AsUnits& p, const AsLoop& l, int N, int BH, int sms) {
  if (l.nkv < 2) return 0;
  const double gain = l.d == 128 && as_threads_per_row(p, l) == 2 ? 0.90 : l.slices ? 0.95 : 0.96;
  const int nx = ((N + 127) / 128 + 1) / 2, pairs = nx * BH, rounds = pairs / sms, left = pairs - rounds * sms;
  if (left == 0) return 0;
  const int all = left * l.nkv, share = std::max(2, (all + sms - 1) / sms);
  if (share >= l.nkv) return 0;
  const int merges = (l.nkv - 1) / share + 1;                 // the most that a CTA adds up
  if (merges > 8) return 0;
  const double tail = l.lin ? 9000. + 4500. * ((l.fc - 1) + (l.slices ? l.slices * (1 + l.fc) : 0)) : 4000.;
  const double unit = l.nkv * 2900. + tail, lone = l.nkv * 1800. + 0.7 * tail;
  const int last = p.split_last ? (p.n_pairs > p.n_rounds * sms || p.n_single > 0) : 2 * (p.n_pairs > p.n_rounds * sms);   // 0: none, 1: lone tiles, 2: units
  const double now = p.n_rounds * unit + (last == 2 ? unit : last == 1 ? lone : 0.);
  const double then = rounds * unit + share * 2900. + tail + (l.lin ? 14000. : 10000.) + 2500. * merges;
  if (then > gain * now) return 0;
  p.nx = nx; p.n_pairs = pairs; p.n_single = 0; p.n_rounds = rounds; p.split_last = 0; p.share = share;
  return rounds > 0 ? sms : (all + share - 1) / share;
}

// The parts of CTA c of a launch of n CTAs in the last round: at most two, the one that it leaves to the next CTA first.  With each, the ring items, phases and tails that
// the CTA has had before it (cf. the query stage's ring).
struct AsPart {
  int unit, k0, k1;              // of the units left over, and its key tiles
  int leaves, merges;            // 1: leaves what it has to another CTA; number of CTAs right before this one that have left it theirs
  int at_items, at_s, at_p, at_pf, at_tail;
};
AS_HD int as_deal_parts(int n_pairs, int n_rounds, int share, int nkv, int lin, int fc_, int slices_, int n, int c, AsPart* to) {
  const int left = n_pairs - n_rounds * n, all = left * nkv;
  const int r0 = c * share, r1 = all < r0 + share ? all : r0 + share;
  if (r0 >= r1) return 0;
  const int fc = lin ? fc_ : 0, slices = lin ? slices_ : 0, tail_items = slices ? slices + fc * slices + fc : 2 * fc;
  int at_items = n_rounds * (2 * nkv + tail_items), at_s = n_rounds * (nkv + slices + fc), at_p = n_rounds * (nkv + fc);
  int at_pf = n_rounds * (nkv + (slices ? 1 : fc)), np = 0;
  auto add = [&](int unit, int k0, int k1) {
    const int leaves = k1 < nkv ? 1 : 0, tiles = k1 - k0;
    to[np++] = AsPart{unit, k0, k1, leaves, leaves || k0 == 0 ? 0 : c - unit * nkv / share, at_items, at_s, at_p, at_pf, n_rounds};
    at_items += 2 * tiles; at_s += tiles; at_p += tiles; at_pf += tiles;       // (of one that is left; nothing comes behind another)
  };
  const int unit = r0 / nkv, k0 = r0 - unit * nkv, over = r1 - (unit + 1) * nkv;
  if (over > 0) add(unit + 1, 0, over);
  add(unit, k0, over > 0 ? nkv : r1 - unit * nkv);
  return np;
}
