// grass_project_grad: host side (argument checks, tiling plan, TMA descriptors,
// launches).  The kernels are in project_tc.cuh (bf16, tcgen05) and
// project_simt.cuh (fp32).
#include <cudaTypedefs.h>
#include <math.h>
#include <string.h>

#include <deque>
#include <unordered_map>

#include "common.cuh"
#include "project_simt.cuh"
#include "project_tc.cuh"
#include "update_common.cuh"

namespace grass {
namespace {

constexpr int kSmCount = 148;

// How the selected dY columns reach the GEMM (values of grass_project_opts_t::gather; 0 in a
// plan means the operand is dY itself, i.e. the dense gradient).
constexpr int kOptAuto = 0, kOptPrepass = 1, kOptCta = 2, kOptCoop = 3;

struct PlanOpts {
  int gather = kOptAuto;   // kOpt*
  int mb = 0;              // n-blocks of 128 columns per CTA: 0 = cost model, else 1, 2 or 4 if it fits
  int pair = 0;            // 0 = cost model, 1 = single CTAs only, 2 = CTA pairs wherever the shape allows
  int split = 0;           // token slices: 0 = cost model
  int gather_warps = 0;    // cooperative gather: warps per CTA that gather (0 = default)
  // not options of the ABI:
  bool wide = false;       // layer-steps and row norms: free row blocks and gather (choose_wide, choose_dense)
  int unit_of = 0;         // slices will be set to units of this many tokens (dense, split > 0)
};

PlanOpts to_plan_opts(const grass_project_opts_t* o) {
  PlanOpts po;
  if (o != nullptr) {
    po.gather = o->gather;
    po.mb = o->n_blocks_per_cta;
    po.pair = o->cta_pair;
    po.split = o->token_slices;
    po.gather_warps = o->gather_warps;
  }
  return po;
}
bool opts_ok(const grass_project_opts_t* o) {
  return o == nullptr ||
         (o->gather >= kOptAuto && o->gather <= kOptCoop &&
          (o->n_blocks_per_cta == 0 || o->n_blocks_per_cta == 1 || o->n_blocks_per_cta == 2 ||
           o->n_blocks_per_cta == 4) &&
          o->cta_pair >= 0 && o->cta_pair <= 2 && o->token_slices >= 0 &&
          o->gather_warps >= 0 && o->gather_warps <= 8);
}

struct TcPlan {
  int gather;     // 0: operand read from dY as it is; else kOptPrepass / kOptCta / kOptCoop
  int kb_unit;    // token slices start on multiples of this many token blocks
  size_t ctrl_bytes;   // cooperative gather: queue head and per-chunk counters
  int r_pad;      // r_blocks * r_cta: width of the gathered operand
  int r_cta, r_blocks;
  int MB, n_blocks;   // n_blocks = CTAs along n (an even number when pair)
  bool pair;          // two CTAs share each MMA (cta_group::2)
  int k_blocks, stages, bk;   // bk: tokens per pipeline stage
  int split_k, s_long;        // token slices; the first s_long are long, the rest short
  int unit_begin[kTcMaxSlices + 1];   // slice z = units [unit_begin[z], unit_begin[z + 1])
  size_t smem_bytes;
  long long ld_part;        // pitch of a split-K partial, elements
  size_t ag_bytes, part_bytes;
  double us;                // projection_us with its slices taken as equal
};

// Whether the gathers fetch 64-byte halves of dY's lines instead of whole ones.  A line holds 64
// columns: with r/m = 1/10 a half already holds a pick in 97 of 100 cases and there is nothing
// left to save; below that the bytes follow 1 - (1 - r/m)^32 instead of 1 - (1 - r/m)^64.  Measured:
// 1B gate,up r = 64 (1/85) 223.9 -> 187.1 us, 7B gate,up r = 256 (1/43) 315.7 -> 276.1 us a
// layer-group step; where all is fetched anyway (1/4: 60M q,k,v,o, 350M down) it costs 1 %.
bool sparse_pick(int64_t m, int r) { return static_cast<int64_t>(r) * 10 < m; }

// Output tile, gather mode and token slices of one call, as the search below tries them.
struct TileChoice {
  int gather, r_cta, r_blocks, mb;
  bool pair;
  int s_long, s_short;
  int x_units;               // units per long slice where there are short ones
};

// Tokens in a unit of a slice.
int unit_tokens(const TileChoice& t) {
  return t.gather == kOptCoop ? kCoopChunk : tc_bk(t.mb, t.pair ? t.r_cta / 128 : t.r_cta / 64);
}
int tiles_along_n(const TileChoice& t, int64_t n) {
  const int cols = t.mb * 128 * (t.pair ? 2 : 1);
  return static_cast<int>((n + cols - 1) / cols);
}

// A gather mode's and a tile's limit on the tokens of a call: the separate gather's grid.y, and the units of
// the kernel's 16-bit slice table.
bool tokens_fit(int gather, int unit, int64_t T) {
  return (gather != kOptPrepass || T <= 65535LL * kGatherTokens) && (T + unit - 1) / unit <= 65535;
}

// Slice lengths for s_long equal slices and ss extra SHORT ones.  With N = tiles-per-slice x slices tiles
// on W workers equal slices leave the last wave partly empty whenever W does not divide N; the
// R = N_long mod W workers that receive one long tile more than the rest are then finished, and the
// other W - R workers share the short tiles.  The lengths (x units long, y units short) are set so that
// both kinds of worker finish together:
//     x c + f = ns (y c + f),  s_long x + s_short y = U,  ns = ceil(N_short / (W - R)),
// c = time per unit, f = per tile.  Returns the busiest worker's time, 1e300 where it does not go.
double short_slices(TileChoice& t, int64_t n_out, int W, int U, double c, double f) {
  const int sl = t.s_long, ss = t.s_short;
  const int64_t n_long = n_out * sl, F = n_long / W, R = n_long % W;
  const int64_t ns = (n_out * ss + (W - R) - 1) / (W - R);
  const double x = (U + ss * (f / c) * (1.0 - 1.0 / ns)) / (sl + static_cast<double>(ss) / ns);
  double span = 1e300;
  for (int cand = static_cast<int>(x); cand <= static_cast<int>(x) + 1; ++cand) {
    const int y_total = U - sl * cand;
    if (cand < 1 || y_total < ss) continue;
    const int y_max = (y_total + ss - 1) / ss;
    const double a = (F + 1) * (cand * c + f);
    const double b = F * (cand * c + f) + ns * (y_max * c + f);
    const double sp = a > b ? a : b;
    if (sp < span) { span = sp; t.x_units = cand; }
  }
  return span;
}

// Estimated microseconds of projecting `groups` layers with this choice, beyond what every choice
// costs; 1e299 for more tokens than the choice takes.  The form is what the parts wait for; the constants are fitted to 25 000 timed layer-steps (80
// shapes of the LLaMA range, T = 600 .. 65536, r = 16 .. 1024, every tile, mode and slice count that
// exists) and predict the good choices to 7 %.  The choice made is 2 % slower than the best one on
// average; the rules that this replaces (tiles as wide as TMEM allows, a separate gather only for
// tiles of at most 128 rows) were 10 % slower on average and 48 % at worst.
//   a tile    per 32 tokens: its operands through the load path, or its MMAs; then what it costs to start
//             and to drain its accumulators
//   a launch  waves of tiles (a part-filled wave costs less than a full one: its tiles run faster)
//             against HBM, in the 2.5-norm, since they overlap only in part; a gather inside the
//             kernel against both, in the 3-norm: the cooperative one needs 15 us where the separate one needs
//             1 (eight warps an SM against a full one), and is the better choice only when the rest hides it
//   around    the separate gather, or the start of the cooperative one; the partials
//
// A search tries thousands of choices, most of them slice counts of the same tile, so what the slices do not
// change is computed once per tile (TileCost), and choices that cannot beat one already priced are left
// out (least_span, most_span): 113 us a search without, 9 with, the mean of 6000 shapes of the LLaMA range.
struct Problem {
  int64_t T, m, n;
  int r, groups;
  double picks, lines;       // selected share of dY's columns; share of its lines that are touched
};
Problem make_problem(int64_t T, int64_t m, int64_t n, int r, int groups) {
  Problem q = {T, m, n, r, groups, static_cast<double>(r) / m, 0};
  q.lines = 1.0 - pow(1.0 - q.picks, sparse_pick(m, r) ? 32 : 64);
  return q;
}
struct TileCost {
  int W, U;
  int64_t n_out;             // tiles per slice
  double c, f, drain;        // us per unit, per tile; drain > 0: hidden behind the next tile's MMAs
  double hbm, hbm_p, gather, gather_p;     // and their powers in the norms
  double l2, around, per_slice;
  bool fits;
};

double pow_2_5(double x) { return x * x * sqrt(x); }

TileCost tile_cost(const Problem& q, const TileChoice& t) {
  const double MBYTE = 1e-6;
  const int64_t T = q.T, m = q.m, n = q.n;
  const int r = q.r, groups = q.groups;
  TileCost k;
  k.W = t.pair ? kSmCount / 2 : kSmCount;
  const int tiles_x = tiles_along_n(t, n);
  k.n_out = static_cast<int64_t>(tiles_x) * t.r_blocks * groups;
  const int unit = unit_tokens(t);
  k.fits = tokens_fit(t.gather, unit, T);
  k.U = static_cast<int>((T + unit - 1) / unit);
  const double cols = t.mb * 128.0, rows = t.pair ? t.r_cta / 2 : t.r_cta;
  k.c = (cols + rows) * (1.092 / 1700);                                          // us per 32 tokens
  const double mma = t.mb * t.r_cta * (t.pair ? 0.22 : 0.17) / 1700;
  if (mma > k.c) k.c = mma;
  k.c *= unit / 32.0;
  k.f = 0.42 + (t.pair ? 2.0 : 0.0) + 4.5 * t.mb * t.r_cta / 512;
  // row-norm epilogue, few tokens: with two accumulator sets the drain of one tile hides behind the
  // MMAs of the next (stores do not: they meet the next tile's loads in L2).  Not where a pair's tile has
  // 128 columns: its MMAs are too short to hide a pair's start as well (70 shapes: 8 % slower than tiles as
  // large as TMEM allows, where the model had them 20 % faster)
  const int columns = t.mb * t.r_cta;
  k.drain = t.gather == 0 && T <= 1536 && columns <= 256 && !(t.pair && columns <= 128) ? 4.5 * columns / 512 : 0;
  const double dy_mb = groups * 2.0 * T * m * q.lines * MBYTE, x_mb = groups * 2.0 * T * n * MBYTE;
  const double ag_mb = groups * 2.0 * T * t.r_cta * t.r_blocks * MBYTE, out_mb = groups * 4.0 * r * n * MBYTE;
  // load-unit time of one pass over the picks, and how many lines a load instruction of 32 spans
  const double lsu = groups * static_cast<double>(T) * t.r_cta * t.r_blocks / kSmCount / 32e3;
  double per_load = (m < 32 / q.picks ? m : 32 / q.picks) / 64;
  per_load = per_load < 1 ? 1 : per_load > 32 ? 32 : per_load;
  k.hbm = x_mb / 6.0;
  k.gather = k.around = 0;
  if (t.gather == kOptPrepass) {
    // (fitted to a gather with fewer loads in flight: too dear by 1.3 to 1.6 at 512 x 512, r = 128)
    k.hbm += 1.1 * ag_mb / 6.0;
    k.around = 0.5 + pow(pow_2_5(lsu * (0.87 + 0.033 * per_load)) + pow_2_5((dy_mb + ag_mb) / 6.6), 0.4);
  } else if (t.gather == kOptCoop) {
    k.hbm += dy_mb / 5.8;
    k.gather = lsu * (15.3 + 0.1 * per_load);
    k.around = 5.9;
  } else if (t.gather == kOptCta) {
    k.hbm += dy_mb / 4.1;
    k.gather = 2.7 * tiles_x * lsu;
  } else {
    k.hbm += dy_mb / 6.0;            // the dense gradient: dY is the operand
  }
  k.hbm_p = pow_2_5(k.hbm);
  k.gather_p = k.gather * k.gather * k.gather;
  const double l2_mb = static_cast<double>(k.n_out) * (t.pair ? 2 : 1) * T * (cols + rows) * 2 * MBYTE;
  k.l2 = 0.0018 * l2_mb;
  k.per_slice = out_mb / 11.2 + 0.056;
  return k;
}

int next_slices(int s) { return s + 1 + s / 16; }      // the counts that a search tries
int max_slices(const TileCost& k) { return k.U < kTcMaxSlices ? k.U : kTcMaxSlices; }

double around_us(const TileCost& k, int slices) {
  double around = k.around;
  if (slices > 1) around += 1.0 + slices * k.per_slice;
  return around;
}

double projection_us(const TileCost& k, TileChoice& t) {
  if (!k.fits) return 1e299;                       // the call would refuse it
  double span;
  if (t.s_short == 0) {
    const double per_worker = static_cast<double>(k.n_out) * t.s_long / k.W;
    const double waves = static_cast<double>((k.n_out * t.s_long + k.W - 1) / k.W);
    double tile = (k.U + t.s_long - 1) / t.s_long * k.c + k.f;
    if (k.drain > 0 && t.s_long == 1 && per_worker > 2)
      tile = 0.4 + (tile - k.f > k.drain ? tile - k.f : k.drain);
    span = tile * (0.83 * waves + 0.17 * (per_worker > 1 ? per_worker : 1));
  } else {
    span = short_slices(t, k.n_out, k.W, k.U, k.c, k.f);
    if (span >= 1e300) return span;
  }
  const double stream = pow(pow_2_5(span) + k.hbm_p, 0.4);
  return cbrt(stream * stream * stream + k.gather_p) + k.l2 + around_us(k, t.s_long + t.s_short);
}

// The workers' time of a choice of this tile is at least this: what it is if they all finish together
// (without the per-tile part where that may hide).
double least_span(const TileCost& k, int slices) {
  return static_cast<double>(k.n_out) / k.W * (k.U * k.c + (k.drain > 0 ? 0 : slices * k.f));
}
// And beyond this a choice of so many slices, or more, costs more than cap: projection_us solved for the
// span.  (One part in 10^9 is for the rounding of the powers.)
double most_span(const TileCost& k, int slices, double cap) {
  const double stream = cap * (1 + 1e-9) - k.l2 - around_us(k, slices);
  const double cube = stream * stream * stream - k.gather_p;
  if (stream <= 0 || cube <= 0) return -1;
  const double p = pow(cube, 2.5 / 3) * (1 + 1e-9) - k.hbm_p;
  return p <= 0 ? -1 : pow(p, 0.4) * (1 + 1e-9);
}

// The cheapest choice for a layer-step: any gather, and the rows cut into more blocks than TMEM requires
// where that pays (1 x 4096 x 2048 x 1024, r = 512: 31 us with 512-row tiles, 26 with 128).
TileChoice choose_wide(int64_t T, int64_t m, int64_t n, int r, int groups) {
  struct Tile { TileChoice t; TileCost k; };
  const Problem q = make_problem(T, m, n, r, groups);
  const int r64 = static_cast<int>(round_up(static_cast<size_t>(r), 64)) / 64;   // in slabs of 64 rows
  const int rb_min = (r64 + 7) / 8;
  int rb_max = rb_min < 8 ? 8 : rb_min + 4;
  if (rb_max > r64) rb_max = r64;
  Tile tiles[8 * 3 * 3 * 2];          // row blocks, gathers, n-blocks, pairs
  int count = 0, tried_slabs = 0;
  double cap = 1e301;                 // what some choice costs
  for (int rb = rb_min; rb <= rb_max; ++rb) {
    const int slabs = (r64 + rb - 1) / rb;
    if (slabs == tried_slabs) continue;            // the same tile with an empty block more
    tried_slabs = slabs;
    TileChoice t = {};
    t.r_blocks = rb;
    t.r_cta = slabs * 64;
    int mb_max = 512 / t.r_cta;
    mb_max = mb_max >= 4 ? 4 : (mb_max >= 2 ? 2 : 1);
    while (mb_max > 1 && static_cast<int64_t>(mb_max / 2) * 128 >= n) mb_max /= 2;  // not past n
    for (int gather : {kOptPrepass, kOptCta, kOptCoop}) {
      t.gather = gather;
      for (t.mb = mb_max; t.mb >= 1; t.mb /= 2) {
        // four n-blocks a CTA save re-reads of the gathered operand that L2 serves anyway, and stream
        // 32-token stages: 5 to 12 % slower than one or two on every shape measured
        if (t.mb == 4 && gather != kOptCta) continue;
        for (int pair = slabs % 2 == 0 ? 1 : 0; pair >= 0; --pair) {
          if (pair && n <= static_cast<int64_t>(t.mb) * 128) continue;  // nothing for the second CTA
          t.pair = pair != 0;
          // In-CTA gather: every tile picks its own columns, so tiles of at most 128 rows (the load unit
          // keeps up), picks dense enough that a load of 32 spans at most 6 lines, and at most two
          // CTAs (pairs) that share a token slice.
          if (gather == kOptCta && (t.r_cta > 128 || tiles_along_n(t, n) * t.r_blocks > 2 ||
                                    static_cast<int64_t>(r) * 12 < m))
            continue;
          const TileCost k = tile_cost(q, t);
          tiles[count++] = {t, k};
          // one and two full waves of tiles: usually close to the best, so that little else is priced
          for (int wave = 1; wave <= 2; ++wave) {
            const int64_t fill = wave * k.W / k.n_out < max_slices(k) ? wave * k.W / k.n_out : max_slices(k);
            for (t.s_long = 1; next_slices(t.s_long) <= fill;) t.s_long = next_slices(t.s_long);
            const double us = projection_us(k, t);
            if (us < cap) cap = us;
          }
        }
      }
    }
  }
  TileChoice best = {};
  double best_us = 1e301;
  for (int i = 0; i < count; ++i) {
    TileChoice t = tiles[i].t;
    const TileCost& k = tiles[i].k;
    double most = 0;
    int most_at = 0;                                   // most_span of this many slices
    for (int sl = 1; sl <= max_slices(k); sl = next_slices(sl)) {
      if (most_at == 0 || sl == 2 || sl >= 2 * most_at) most = most_span(k, most_at = sl, cap);
      if (least_span(k, sl) > most) break;             // and more slices cost more
      t.s_long = sl;
      // short slices where they were measured to pay: launches of three or more waves (7B
      // down, r = 1024: 587 -> 539 us), and the in-CTA gather, where each worker is bound by its
      // own gather warps (60M q,k,v,o: 179 -> 155 us)
      const int64_t n_long = k.n_out * t.s_long;
      const int max_short = n_long % k.W == 0 || (n_long / k.W < 2 && t.gather != kOptCta) ? 0 : 3;
      for (t.s_short = 0; t.s_short <= max_short && t.s_long + t.s_short <= max_slices(k); ++t.s_short) {
        if (least_span(k, t.s_long + t.s_short) > most) break;
        const double us = projection_us(k, t);
        if (us < best_us) { best_us = us; best = t; }
        if (us < cap) cap = us;
      }
    }
  }
  return best;
}

// How the selected columns get to the GEMM for a given tile shape.  In-CTA gather: the GEMM's
// own warps pick the columns out of dY into shared memory.  It pays when a tile holds at most
// 128 rows (the load unit keeps up), at most two CTAs (pairs) share a token slice (each gathers
// for itself) and the picks are dense enough that a 32-lane load spans at most 6 cache lines
// (12 r >= m); measured on the 60M q,k,v,o group (m = 512, r = 128): step 253 -> 274 TFLOP/s,
// while at m = 2048, r = 128 the sparser pick made the in-kernel loads the bottleneck.
// Everything else: cooperative gather (all CTAs share one pass over dY, overlapped with the
// MMAs); the stand-alone pre-pass remains selectable.
int choose_gather(bool has_idx, const PlanOpts& opts, int r_cta, int tiles_x, int64_t m, int r) {
  if (!has_idx) return 0;
  const bool cta_ok = r_cta <= 128;
  if (opts.gather == kOptCta && cta_ok) return kOptCta;
  if (opts.gather == kOptPrepass) return kOptPrepass;
  if (opts.gather == kOptCoop) return kOptCoop;
  if (opts.gather == kOptAuto && cta_ok && tiles_x <= 2 && static_cast<int64_t>(r) * 12 >= m)
    return kOptCta;
  // Few selected rows (r <= 128): the GEMM is a pure HBM stream of X and the gather is as large
  // as the GEMM itself; as two kernels the gather of one layer overlaps the GEMM of another
  // stream's layer, which measured better than one kernel doing both (1B shapes, r = 64 / 128:
  // 98 / 116 us per layer-step against 107 / 128).
  if (opts.gather == kOptAuto && cta_ok) return kOptPrepass;
  return kOptCoop;
}

// The choice for the dense gradient, for the projection calls (whose plan grass_project_plan reports and
// whose options callers set against it), and for the projection of a refresh iteration.  Row blocks as
// large as TMEM allows.  The cost model in SM clocks is the busiest worker's time (MMAs, or for a single
// CTA the shared-memory ceiling; pipeline fill and accumulator drain per tile), half of the L2 -> SM
// operand traffic at about 8.6 TB/s (each CTA fetches its own tiles; it overlaps the MMAs only in
// part), and the partials' write and read.
TileChoice choose_by_clocks(int64_t T, int64_t m, int64_t n, int r, bool has_idx, const PlanOpts& opts,
                            bool single_split, int groups) {
  TileChoice t = {};
  const int r64 = static_cast<int>(round_up(static_cast<size_t>(r), 64));
  t.r_blocks = (r64 + 511) / 512;
  t.r_cta = static_cast<int>(round_up(static_cast<size_t>((r64 + t.r_blocks - 1) / t.r_blocks), 64));
  int mb_max = 512 / t.r_cta;
  mb_max = mb_max >= 4 ? 4 : (mb_max >= 2 ? 2 : 1);
  while (mb_max > 1 && static_cast<int64_t>(mb_max / 2) * 128 >= n) mb_max /= 2;  // not past n
  const double hbm_bytes_per_clk = 6.5e12 / 1.7e9;  // whole chip, per SM clock
  TileChoice best = t;
  best.mb = best.s_long = 1;
  best.gather = choose_gather(has_idx, opts, t.r_cta, tiles_along_n(best, n), m, r);
  double best_clk = 1e300;
  const bool can_pair = t.r_cta % 128 == 0 && opts.pair != 1;
  for (t.mb = mb_max; t.mb >= 1; t.mb /= 2) {
    if (opts.mb > 0 && opts.mb <= mb_max && t.mb != opts.mb) continue;
    for (int pair = can_pair ? 1 : 0; pair >= 0; --pair) {
      if (pair && n <= static_cast<int64_t>(t.mb) * 128) continue;  // nothing for the second CTA
      if (!pair && opts.pair == 2 && can_pair && n > static_cast<int64_t>(t.mb) * 128) continue;
      t.pair = pair != 0;
      const int tiles_x = tiles_along_n(t, n);
      const int64_t n_out = static_cast<int64_t>(tiles_x) * t.r_blocks * groups;   // tiles per slice
      const int W = pair ? kSmCount / 2 : kSmCount;
      t.gather = choose_gather(has_idx, opts, t.r_cta, tiles_x, m, r);
      const int unit = unit_tokens(t);
      const int U = static_cast<int>((T + unit - 1) / unit);
      double c = static_cast<double>(t.mb) * t.r_cta;               // clocks per 32 tokens
      if (!pair) c *= 1.4;
      if (c < 256.0) c = 256.0;
      c *= unit / 32.0;
      const double f = 3000.0 + t.mb * 128.0 * t.r_cta * 4.0 / 128.0;   // pipeline fill, accumulator drain
      const double cta_rows = pair ? t.r_cta / 2 : t.r_cta;
      const double l2_clk = static_cast<double>(tiles_x) * t.r_blocks * groups * (pair ? 2 : 1) *
                            static_cast<double>((T + 31) / 32) * (t.mb * 128.0 + cta_rows) * 64.0 / 4500.0;
      const int max_s = single_split ? 1 : (U < kTcMaxSlices ? U : kTcMaxSlices);
      for (int sl = 1; sl <= max_s; ++sl) {
        if (opts.split > 0 && !single_split && sl != (opts.split < max_s ? opts.split : max_s)) continue;
        t.s_long = sl;
        const int64_t n_long = n_out * sl;
        // short slices where they were measured to pay: launches of three or more waves (7B down,
        // r = 1024: 587 -> 539 us), and the in-CTA gather, where each worker is bound by its own
        // gather warps (60M q,k,v,o: 179 -> 155 us).  With fewer waves the kernel is bound by operand
        // traffic, and the extra partials cost more than the idle SMs.
        const int max_short = (single_split || opts.split > 0 || n_long % W == 0 ||
                               (n_long / W < 2 && t.gather != kOptCta)) ? 0 : 3;
        for (t.s_short = 0; t.s_short <= max_short && sl + t.s_short <= max_s; ++t.s_short) {
          t.x_units = 0;
          const double span = t.s_short == 0
                                  ? static_cast<double>((n_long + W - 1) / W) * (((U + sl - 1) / sl) * c + f)
                                  : short_slices(t, n_out, W, U, c, f);
          if (span >= 1e300) continue;
          double cost = span + 0.5 * l2_clk;
          if (sl + t.s_short > 1)
            cost += 8.0 * (sl + t.s_short) * groups * static_cast<double>(r) * n / hbm_bytes_per_clk;
          if (cost < best_clk) { best_clk = cost; best = t; }
        }
      }
    }
  }
  return best;
}

// The cheapest choice for a refresh's dense gradient (all m rows), in one slice (single_split: the row-norm
// epilogue) or several.  Tiles of fewer rows than TMEM allows pay where the tokens are few: a drained
// tile of 256 columns overlaps the next one's MMAs, and odd row counts pad less (628 x 13824 x 11008:
// 189 us with 512 rows, 166 with 256; 3584 x 13824 x 1024: 88, 74 with 384; 3328 x 1376 x 4096: 48, 41 with 192).
TileChoice choose_dense(int64_t T, int64_t m, int64_t n, const PlanOpts& opts, bool single_split) {
  const int r64 = static_cast<int>(round_up(static_cast<size_t>(m), 64)) / 64;
  const Problem q = make_problem(T, m, n, static_cast<int>(m), 1);
  TileChoice best = {};
  double best_us = 1e301;
  for (int want = r64 < 8 ? r64 : 8; want >= 1; --want) {
    TileChoice t = {};
    t.r_blocks = (r64 + want - 1) / want;
    const int slabs = (r64 + t.r_blocks - 1) / t.r_blocks;
    if (slabs != want) continue;
    t.r_cta = slabs * 64;
    for (t.mb = t.r_cta <= 256 && n > 128 ? 2 : 1; t.mb >= 1; --t.mb) {
      for (int pair = slabs % 2 == 0 ? 1 : 0; pair >= 0; --pair) {
        if (pair && n <= static_cast<int64_t>(t.mb) * 128) continue;  // nothing for the second CTA
        t.pair = pair != 0;
        if (opts.unit_of > 0 && opts.unit_of % unit_tokens(t) != 0) continue;
        const TileCost k = tile_cost(q, t);
        const int max_s = single_split ? 1 : max_slices(k);
        double most = 0;
        for (int sl = 1; sl <= max_s; sl = next_slices(sl)) {
          t.s_long = opts.split > 0 ? (opts.split < max_s ? opts.split : max_s) : sl;
          if (sl == 2) most = most_span(k, sl, best_us);
          if (sl >= 2 && least_span(k, sl) > most) break;
          const double us = projection_us(k, t);
          if (us < best_us) { best_us = us; best = t; }
          if (opts.split > 0) break;
        }
      }
    }
  }
  // the tile as large as TMEM allows stays unless another is better by more than the model is sure of
  TileChoice large = choose_by_clocks(T, m, n, static_cast<int>(m), false, opts, single_split, 1);
  if (opts.unit_of > 0 && opts.unit_of % unit_tokens(large) != 0) return best;
  return projection_us(tile_cost(q, large), large) < 1.06 * best_us ? large : best;
}

// The result depends only on the arguments.
TcPlan search_plan(int64_t T, int64_t m, int64_t n, int r, bool has_idx, const PlanOpts& opts,
                   bool single_split, int groups) {
  const TileChoice t = !opts.wide ? choose_by_clocks(T, m, n, r, has_idx, opts, single_split, groups)
                       : has_idx  ? choose_wide(T, m, n, r, groups)
                                  : choose_dense(T, m, n, opts, single_split);
  TcPlan p;
  p.gather = t.gather;
  p.r_blocks = t.r_blocks;
  if (t.r_blocks == 0) return p;
  p.r_cta = t.r_cta;
  p.r_pad = p.r_cta * p.r_blocks;
  p.MB = t.mb;
  p.pair = t.pair;
  p.s_long = t.s_long;
  p.split_k = t.s_long + t.s_short;
  p.n_blocks = tiles_along_n(t, n) * (p.pair ? 2 : 1);
  const int a_slabs = p.pair ? p.r_cta / 128 : p.r_cta / 64;
  p.bk = tc_bk(p.MB, a_slabs);
  p.k_blocks = static_cast<int>((T + p.bk - 1) / p.bk);
  p.kb_unit = p.gather == kOptCoop ? kCoopChunk / p.bk : 1;
  {
    // slice table: long slices of best_x units (or an equal cut), then the short ones
    const int U = (p.k_blocks + p.kb_unit - 1) / p.kb_unit;
    if (p.split_k > U) { p.split_k = U; if (p.s_long > U) p.s_long = U; }
    const int ss = p.split_k - p.s_long;
    int at = 0;
    for (int z = 0; z < p.split_k; ++z) {
      p.unit_begin[z] = at;
      if (ss == 0) at += U / p.split_k + (z < U % p.split_k ? 1 : 0);
      else if (z < p.s_long) at += t.x_units;
      else {
        const int y_total = U - p.s_long * t.x_units, zs = z - p.s_long;
        at += y_total / ss + (zs < y_total % ss ? 1 : 0);
      }
    }
    p.unit_begin[p.split_k] = U;
    for (int z = p.split_k + 1; z <= kTcMaxSlices; ++z) p.unit_begin[z] = U;
  }
  p.ctrl_bytes = p.gather == kOptCoop
                     ? round_up((kCoopCtrlInts + static_cast<size_t>(groups) *
                                                     ((T + kCoopChunk - 1) / kCoopChunk)) * sizeof(int), 256)
                     : 0;
  p.stages = tc_stages(p.MB, a_slabs);
  p.smem_bytes = static_cast<size_t>(p.stages) * tc_stage_bytes(p.MB, a_slabs) + 1024;
  p.ld_part = static_cast<long long>(round_up(static_cast<size_t>(n), 4));
  p.ag_bytes = p.gather == kOptPrepass || p.gather == kOptCoop
                   ? round_up(static_cast<size_t>(T) * p.r_pad * sizeof(__nv_bfloat16), 256)
                   : 0;
  p.part_bytes = p.split_k > 1
                     ? round_up(static_cast<size_t>(p.split_k) * r * p.ld_part * sizeof(float), 256)
                     : 0;
  TileChoice equal = {p.gather, p.r_cta, p.r_blocks, p.MB, p.pair, p.split_k, 0, 0};
  p.us = projection_us(tile_cost(make_problem(T, m, n, r, groups), equal), equal);
  return p;
}

// A search costs the host ten to a hundred microseconds and a training loop asks for the same few dozen
// plans over and over (a block of a model has three shapes; a step, a refresh's norms and its projection have
// plans of their own).  Each host thread keeps the last kPlans that it searched and forgets the oldest
// first, so no set of up to kPlans shapes in use loses one.  (A table with one plan per hash bucket lost
// two of the three shapes of a 350M block to one another: 0.76 ms of searching a block.)  A plan is a
// function of its key and of nothing else.
struct PlanKey {
  int64_t v[12];
  bool operator==(const PlanKey& o) const { return memcmp(v, o.v, sizeof(v)) == 0; }
};
struct PlanKeyHash {
  size_t operator()(const PlanKey& k) const {
    uint64_t h = 0;
    for (int64_t x : k.v) h = (h ^ static_cast<uint64_t>(x)) * 0x9E3779B97F4A7C15ull, h ^= h >> 32;
    return static_cast<size_t>(h);
  }
};
constexpr size_t kPlans = 256;
thread_local int64_t plan_searches = 0;

TcPlan make_plan(int64_t T, int64_t m, int64_t n, int r, bool has_idx, const PlanOpts& opts,
                 bool single_split = false, int groups = 1) {
  static thread_local std::unordered_map<PlanKey, TcPlan, PlanKeyHash> plans;
  static thread_local std::deque<PlanKey> order;
  const PlanKey key = {{T, m, n, r, has_idx, opts.gather, opts.mb, opts.pair, opts.split,
                        opts.unit_of * 2 + (opts.wide ? 1 : 0), single_split, groups}};
  const auto hit = plans.find(key);
  if (hit != plans.end()) return hit->second;
  ++plan_searches;
  const TcPlan plan = search_plan(T, m, n, r, has_idx, opts, single_split, groups);
  if (plans.size() >= kPlans) {
    plans.erase(order.front());
    order.pop_front();
  }
  plans.emplace(key, plan);
  order.push_back(key);
  return plan;
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (fn == nullptr) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// bf16 matrix [rows][cols] with row pitch ld (elements): box = {64 cols, bk rows}, 128B swizzle.
// Encoded on every call: a host-side cache keyed by (pointer, shape, pitch) was measured and
// saved nothing (40.8 us against 41.9 us of host time per batched call of four 60M layers).
bool make_map(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld, int bk) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (fn == nullptr) return false;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld) * 2};
  cuuint32_t box[2] = {64, static_cast<cuuint32_t>(bk)};
  cuuint32_t estr[2] = {1, 1};
  CUresult res = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                    box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (res != CUDA_SUCCESS) {
    fprintf(stderr, "grass: cuTensorMapEncodeTiled failed with %d\n", static_cast<int>(res));
    return false;
  }
  return true;
}

template <int MB, int NSLAB, bool PAIR, int GATHER>
int launch_tc_one(dim3 tile_grid, size_t smem, cudaStream_t s, const TcMaps& maps, TcParams p,
                  int kernel_id) {
  constexpr bool FUSED = GATHER != kGatherNone;   // the variants with eight extra warps
  static bool attr_set[64] = {false};
  static int max_workers[64] = {0};
  int dev = 0;
  GRASS_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return GRASS_ERR_INVALID_ARG;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(FUSED ? kTcThreads + kTcGatherThreads : kTcThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = PAIR ? 2 : 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (!attr_set[dev]) {
    GRASS_CUDA_TRY(cudaFuncSetAttribute(project_tc_kernel<MB, NSLAB, PAIR, GATHER>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        kTcSmemBudget));
    // how many workers (CTAs, or CTA pairs) the device holds at once: one per SM / SM pair
    int workers = 0;
    if (PAIR) {
      cfg.gridDim = dim3(2 * kSmCount);
      GRASS_CUDA_TRY(cudaOccupancyMaxActiveClusters(&workers, project_tc_kernel<MB, NSLAB, PAIR, GATHER>,
                                                    &cfg));
    } else {
      GRASS_CUDA_TRY(cudaDeviceGetAttribute(&workers, cudaDevAttrMultiProcessorCount, dev));
    }
    if (workers < 1) workers = 1;
    max_workers[dev] = workers;
    attr_set[dev] = true;
  }
  // persistent launch: never more workers than are resident at once, each loops over its tiles
  p.tiles_x = static_cast<int>(tile_grid.x);
  p.tiles_y = static_cast<int>(tile_grid.y);
  const long long n_tiles = static_cast<long long>(tile_grid.x) * tile_grid.y * tile_grid.z;
  // (cooperative gather: every SM takes part in the gather, also those without a tile)
  const int workers = n_tiles < max_workers[dev] && GATHER != kGatherCoop && p.s_long == p.split_k
                          ? static_cast<int>(n_tiles) : max_workers[dev];
  cfg.gridDim = dim3(static_cast<unsigned>(PAIR ? 2 * workers : workers));
  attr[1] = dependent_launch_attr();
  cfg.numAttrs = 2;
  {
    ProfileScope prof(kernel_id, s);
    GRASS_CUDA_TRY(cudaLaunchKernelEx(&cfg, project_tc_kernel<MB, NSLAB, PAIR, GATHER>, maps, p));
  }
  return GRASS_OK;
}

// (MB, NSLAB) with MB * 64 * NSLAB <= 512 TMEM columns; pairs need an even NSLAB.
// gather: kGatherNone / kGatherCta (tiles of at most 128 rows) / kGatherCoop.
int launch_tc(int MB, int nslab, bool pair, int gather, dim3 grid, size_t smem, cudaStream_t s,
              const TcMaps& maps, const TcParams& p, int kernel_id) {
#define GRASS_TC_CASE(mb, ns, pr, ga)                                                          \
  if (MB == mb && nslab == ns && pair == pr && gather == ga)                                   \
    return launch_tc_one<mb, ns, pr, ga>(grid, smem, s, maps, p, kernel_id)
#define GRASS_TC_BOTH(mb, ns, pr)                                                              \
  GRASS_TC_CASE(mb, ns, pr, kGatherNone);                                                      \
  GRASS_TC_CASE(mb, ns, pr, kGatherCoop)
  GRASS_TC_BOTH(1, 1, false); GRASS_TC_BOTH(1, 2, false); GRASS_TC_BOTH(1, 3, false);
  GRASS_TC_BOTH(1, 4, false); GRASS_TC_BOTH(1, 5, false); GRASS_TC_BOTH(1, 6, false);
  GRASS_TC_BOTH(1, 7, false); GRASS_TC_BOTH(1, 8, false);
  GRASS_TC_BOTH(2, 1, false); GRASS_TC_BOTH(2, 2, false); GRASS_TC_BOTH(2, 3, false);
  GRASS_TC_BOTH(2, 4, false);
  GRASS_TC_BOTH(4, 1, false); GRASS_TC_BOTH(4, 2, false);
  GRASS_TC_BOTH(1, 2, true); GRASS_TC_BOTH(1, 4, true); GRASS_TC_BOTH(1, 6, true);
  GRASS_TC_BOTH(1, 8, true);
  GRASS_TC_BOTH(2, 2, true); GRASS_TC_BOTH(2, 4, true); GRASS_TC_BOTH(4, 2, true);
  // in-CTA gather: at most 128 selected rows per tile
  GRASS_TC_CASE(1, 1, false, kGatherCta); GRASS_TC_CASE(2, 1, false, kGatherCta);
  GRASS_TC_CASE(4, 1, false, kGatherCta); GRASS_TC_CASE(1, 2, false, kGatherCta);
  GRASS_TC_CASE(2, 2, false, kGatherCta); GRASS_TC_CASE(4, 2, false, kGatherCta);
  GRASS_TC_CASE(1, 2, true, kGatherCta); GRASS_TC_CASE(2, 2, true, kGatherCta);
  GRASS_TC_CASE(4, 2, true, kGatherCta);
#undef GRASS_TC_BOTH
#undef GRASS_TC_CASE
  return GRASS_ERR_UNSUPPORTED;
}

size_t norm_part_bytes(int64_t m, int64_t n) {
  return round_up(static_cast<size_t>((n + 31) / 32) * round_up(static_cast<size_t>(m), 32) *
                      sizeof(float), 256);
}

// Most bytes of partials of a kept gradient, twice L2: a bound on the workspace more than on the time.  Of the
// timed refreshes 250 have partials of 128 to 256 MB and are kept by the rule below; kept they take 5 %
// less time than projected again, in the mean (350M gate, 202 MB: 14 %).  Beyond, nothing is gained.
constexpr double kKeepMostBytes = 256e6;

// fp32 path.  128 x 128 tiles where they can give every SM its two CTAs at 128 tokens or more a
// slice, else 64 x 64 tiles; tokens are split to fill the GPU.
// slices_of > 0: the token slices are those that 64 x 64 tiles of that many rows would get.  Refresh
// iterations use it with the selected rows, whichever way they form G_C: after a state reset its bits
// decide signs (make_keep_plan).
struct Fp32Plan {
  bool big;
  int split;
  int64_t tokens_per_split;
  long long ld_part;
  size_t part_bytes;
};
Fp32Plan make_fp32_plan(int64_t T, int64_t n, int r, int slices_of = 0) {
  Fp32Plan p;
  const int64_t big_tiles = ((n + 127) / 128) * ((r + 127) / 128);
  p.big = big_tiles * (T / 128) >= 2 * kSmCount;
  int64_t split;
  if (p.big && slices_of == 0) {
    split = 2 * kSmCount / big_tiles;      // as many slices as two CTAs an SM can take at once
  } else {
    const int64_t tiles = ((n + 63) / 64) * (((slices_of > 0 ? slices_of : r) + 63) / 64);
    split = (2 * kSmCount + tiles - 1) / tiles;
  }
  const int64_t max_split = (T + 2 * kSimtBT - 1) / (2 * kSimtBT);   // at least 32 tokens a slice
  if (split > max_split) split = max_split;
  if (split > 64) split = 64;
  if (split < 1) split = 1;
  int64_t per = (T + split - 1) / split;
  per = (per + kSimtBT - 1) / kSimtBT * kSimtBT;
  p.tokens_per_split = per;
  p.split = static_cast<int>((T + per - 1) / per);
  p.ld_part = static_cast<long long>(round_up(static_cast<size_t>(n), 4));
  p.part_bytes = p.split > 1
                     ? round_up(static_cast<size_t>(p.split) * r * p.ld_part * sizeof(float), 256)
                     : 0;
  return p;
}
// Whether a refresh keeps the fp32 gradient (formed anyway; what it costs is the slices' partials).
bool keep_fp32(int64_t T, int64_t m, int64_t n, int r) {
  return static_cast<double>(make_fp32_plan(T, n, static_cast<int>(m), r).part_bytes) <= kKeepMostBytes;
}

template <int TM>
int launch_simt(const Fp32Plan& fp, const float* dY, int64_t lddy, const float* X, int64_t ldx, int64_t T,
                int64_t m, int64_t n, const int32_t* idx, const float* rho, int r, float* out,
                int64_t ld_out, int* status, cudaStream_t s) {
  static bool attr_set[64] = {false};
  int dev = 0;
  GRASS_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return GRASS_ERR_INVALID_ARG;
  if (!attr_set[dev]) {
    GRASS_CUDA_TRY(cudaFuncSetAttribute(project_simt_kernel<TM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        simt_smem_bytes(TM)));
    attr_set[dev] = true;
  }
  constexpr int B = simt_tile(TM);
  dim3 grid(static_cast<unsigned>((n + B - 1) / B), static_cast<unsigned>((r + B - 1) / B),
            static_cast<unsigned>(fp.split));
  const bool avec = idx == nullptr && aligned_to(dY, 16) && lddy % 4 == 0;
  const bool xvec = aligned_to(X, 16) && ldx % 4 == 0;
  const bool ovec = aligned_to(out, 16) && ld_out % 4 == 0;
  ProfileScope prof(GRASS_K_PROJECT_FP32, s);
  GRASS_CUDA_TRY(launch_kernel(project_simt_kernel<TM>, grid, kSimtThreads, simt_smem_bytes(TM), s,
                               dY, lddy, X, ldx, T, m, n, idx, rho, r, out, ld_out, fp.tokens_per_split,
                               static_cast<int64_t>(r) * fp.ld_part, avec, xvec, ovec, status));
  return GRASS_OK;
}

// Row-norm mode.  The squares must be taken of complete dot products, so the fused epilogue
// needs an unsplit token sum; that is the plan whenever the dense m x n output has enough tiles
// to occupy the GPU (every LLaMA shape from 1B up).  A small gradient (few tiles) would leave
// most SMs idle, so it is computed with the usual token split into fp32 partials -- small by
// the same token -- and splitk_rownorms_kernel sums, squares and reduces them.
TcPlan make_norms_plan(int64_t T, int64_t m, int64_t n, bool* small = nullptr) {
  PlanOpts o;
  o.wide = true;
  const bool few_tiles = ((n + 127) / 128) * ((m + 511) / 512) < 120;
  if (small != nullptr) *small = few_tiles;
  return make_plan(T, m, n, static_cast<int>(m), false, o, !few_tiles);
}

// A refresh whose small dense gradient also serves as G_C: where the norms leave it, its partials summed.
struct GradParts {
  int r = 0;                       // in: rows that will be selected
  const float* grad = nullptr;     // out; NULL: not kept
  long long ld = 0;
};
size_t grad_parts_bytes(int split_k, int64_t m, long long ld) {
  return round_up(static_cast<size_t>(split_k) * m * ld * sizeof(float), 256);
}

// The plan of a dense gradient that is kept for r selected rows, or false.  Its token slices are those
// of the projection that it replaces, so that G_C has the same bits: after a state reset the update is the
// sign of the gradient, and another summation order would turn elements that are zero to rounding.  That makes
// more partials than the norms alone need, which has to cost less than projecting again.  The rule sets
// the two forms' estimates against one another; its factors (the norms' and the update's passes over the
// partials, their start per slice, the launches saved) are fitted to 13 500 refreshes timed both ways (m, n =
// 256 .. 5461, T = 256 .. 65536, r = 8 .. 1024).  Over these it costs 0.3 % more than the better form,
// always keeping 25 %, never 21 %; weighing the partials' bytes alone against the projection cost 0.8 %, and up to
// 50 % where few rows of a small layer make many slices (T = 13056, 384 x 5461, r = 43: kept 155 us, projected 113).
// (Since the norms leave the partials' sum for the update, keeping costs up to 10 % less than in that fit.)
bool make_keep_plan(int64_t T, int64_t m, int64_t n, int r, TcPlan* plan) {
  bool small = false;
  const double norms_us = make_norms_plan(T, m, n, &small).us;
  if (!small) return false;
  const TcPlan proj = make_plan(T, m, n, r, true, PlanOpts());
  const int unit = proj.kb_unit * proj.bk;
  PlanOpts o;
  o.wide = true;
  o.split = proj.split_k;
  o.unit_of = unit;
  *plan = make_plan(T, m, n, static_cast<int>(m), false, o, false);
  if (plan->r_blocks == 0) return false;          // no tile takes such slices
  plan->kb_unit = unit / plan->bk;
  plan->split_k = proj.split_k;
  plan->s_long = proj.s_long;
  for (int z = 0; z <= kTcMaxSlices; ++z) plan->unit_begin[z] = proj.unit_begin[z];
  return static_cast<double>(grad_parts_bytes(plan->split_k, m, plan->ld_part)) <= kKeepMostBytes &&
         1.7 * (plan->us - norms_us) + 0.2 * plan->split_k < proj.us + 9.0;
}

// The same where the workspace of the norms has room for the partials.
bool keeps(int64_t T, int64_t m, int64_t n, int r, size_t ws_bytes, TcPlan* plan) {
  return make_keep_plan(T, m, n, r, plan) && ws_bytes >= grad_parts_bytes(plan->split_k, m, plan->ld_part);
}
bool keeps_fp32(int64_t T, int64_t m, int64_t n, int r, size_t ws_bytes) {
  return keep_fp32(T, m, n, r) && ws_bytes >= make_fp32_plan(T, n, static_cast<int>(m), r).part_bytes;
}

// Bytes of workspace a plan needs for `count` layers: [control block][per layer: gathered operand,
// split-K partials].
size_t plan_ws_bytes(const TcPlan& plan, int count) {
  return plan.ctrl_bytes + (plan.ag_bytes + plan.part_bytes) * static_cast<size_t>(count);
}

// What a plan cannot be run with: more tokens than its gather or its slice table take, or a workspace of
// less than `need` bytes.
int plan_refused(const TcPlan& plan, int64_t T, size_t need, const void* ws, size_t ws_bytes) {
  if (!tokens_fit(plan.gather, plan.kb_unit * plan.bk, T)) return GRASS_ERR_UNSUPPORTED;
  if (need > 0 && (ws == nullptr || !aligned_to(ws, 256) || ws_bytes < need)) return GRASS_ERR_WORKSPACE;
  return GRASS_OK;
}

// Rows of up to 128, 256 and 512 columns (four a thread) share a CTA, as long as two CTAs an SM are left (256 rows
// of 256 columns in 16 splits, an fp32 refresh step: 21.6 us with a CTA each, 22.8 with four a CTA).
cudaError_t launch_row_norms(float* part, long long ld, long long stride, int split_k, int64_t m, int64_t n,
                             float* norms, bool keep, cudaStream_t s) {
  int threads = n <= 128 ? 32 : n <= 256 ? 64 : n <= 512 ? 128 : 256;
  while (threads < 256 && m * threads / 256 < 2 * kSmCount) threads *= 2;
  const int rows = 256 / threads;
  keep = keep && split_k > 1;               // (one partial is the sum)
  auto kernel = threads < 256 ? keep ? splitk_rownorms_kernel<true, true> : splitk_rownorms_kernel<true, false>
                              : keep ? splitk_rownorms_kernel<false, true> : splitk_rownorms_kernel<false, false>;
  return launch_kernel(kernel, static_cast<unsigned>((m + rows - 1) / rows), 256, 0, s, part, ld, stride,
                       split_k, static_cast<int>(m), static_cast<int>(n), threads, norms);
}

// Projection of `count` same-shaped layers in one set of launches (count = 1 for the plain
// call).  norms != NULL (count must be 1): row-norm mode (idx NULL, r == m): the GEMM's epilogue
// reduces squares instead of storing the gradient, then the partial sums are finalised.
// upd != NULL: the update that follows; its kernel takes the place of the split-K reduce.
int project_bf16(int count, const void* const* dY, int64_t lddy, const void* const* X, int64_t ldx,
                 int64_t T, int64_t m, int64_t n, const int32_t* const* idx,
                 const float* const* rho, int r, float* const* Gc, int64_t ldgc, float* norms,
                 void* ws, size_t ws_bytes, const PlanOpts& opts, cudaStream_t s,
                 UpdateCall* upd = nullptr, GradParts* keep = nullptr) {
  if (count < 1 || count > kTcMaxGroup || (norms != nullptr && count != 1))
    return GRASS_ERR_INVALID_ARG;
  const bool gather = idx != nullptr && idx[0] != nullptr;
  for (int g = 0; g < count; ++g) {
    if (dY[g] == nullptr || X[g] == nullptr || (norms == nullptr && Gc[g] == nullptr))
      return GRASS_ERR_INVALID_ARG;
    if (gather != (idx != nullptr && idx[g] != nullptr)) return GRASS_ERR_INVALID_ARG;
    if (!aligned_to(X[g], 16) || ldx % 8 != 0) return GRASS_ERR_ALIGNMENT;
    if (!gather && (!aligned_to(dY[g], 16) || lddy % 8 != 0)) return GRASS_ERR_ALIGNMENT;
  }
  TcPlan plan;
  // kept for G_C (stored even where the tokens are not split), if there is room for it
  const bool stored = keep != nullptr && keeps(T, m, n, keep->r, ws_bytes, &plan);
  if (!stored)
    plan = norms != nullptr ? make_norms_plan(T, m, n) : make_plan(T, m, n, r, gather, opts, false, count);
  // a workspace sized for more tokens may fall short of a step's own tiling for fewer (more slices): then
  // the tiling of the projection calls
  if (opts.wide && gather && plan_refused(plan, T, plan_ws_bytes(plan, count), ws, ws_bytes) == GRASS_ERR_WORKSPACE)
    plan = make_plan(T, m, n, r, true, PlanOpts(), false, count);
  const bool fused_norms = norms != nullptr && plan.split_k == 1 && !stored;
  const size_t per_layer = fused_norms ? norm_part_bytes(m, n)
                           : stored    ? grad_parts_bytes(plan.split_k, m, plan.ld_part)
                                       : plan.ag_bytes + plan.part_bytes;
  const int refused = plan_refused(plan, T, plan.ctrl_bytes + per_layer * count, ws, ws_bytes);
  if (refused != GRASS_OK) return refused;
  cudaError_t err;
  int* status = status_word(&err);
  if (status == nullptr) GRASS_CUDA_TRY(err);

  TcMaps maps;
  GatherGroup gg;
  float* part[kTcMaxGroup];
  char* const layers_ws = static_cast<char*>(ws) + plan.ctrl_bytes;
  for (int g = 0; g < count; ++g) {
    char* wsp = layers_ws + per_layer * g;
    if (!make_map(&maps.x[g], X[g], T, n, ldx, plan.bk)) return GRASS_ERR_CUDA;
    gg.dY[g] = static_cast<const __nv_bfloat16*>(dY[g]);
    gg.idx[g] = gather ? idx[g] : nullptr;
    gg.Ag[g] = nullptr;
    if (plan.gather == kOptCta) {
      maps.a[g] = maps.x[g];          // unused by the kernel
    } else if (plan.gather == kOptPrepass || plan.gather == kOptCoop) {
      gg.Ag[g] = reinterpret_cast<__nv_bfloat16*>(wsp);
      if (!make_map(&maps.a[g], gg.Ag[g], T, plan.r_pad, plan.r_pad, plan.bk)) return GRASS_ERR_CUDA;
      wsp += plan.ag_bytes;
    } else {
      if (!make_map(&maps.a[g], dY[g], T, m, lddy, plan.bk)) return GRASS_ERR_CUDA;
    }
    part[g] = reinterpret_cast<float*>(wsp);
  }
  for (int g = count; g < kTcMaxGroup; ++g) {
    maps.x[g] = maps.x[0];
    maps.a[g] = maps.a[0];
    gg.dY[g] = nullptr; gg.idx[g] = nullptr; gg.Ag[g] = nullptr;
  }
  if (plan.gather == kOptPrepass) {
    ProfileScope prof(GRASS_K_GATHER, s);
    const int ni = plan.r_pad > 128 ? 8 : plan.r_pad / 32;   // r_pad is a multiple of 64
    dim3 ggrid(static_cast<unsigned>((plan.r_pad + 32 * ni - 1) / (32 * ni)),
               static_cast<unsigned>((T + kGatherTokens - 1) / kGatherTokens),
               static_cast<unsigned>(count));
    const bool sparse = sparse_pick(m, r);
    auto kernel = ni == 8   ? sparse ? gather_cols_kernel<8, true> : gather_cols_kernel<8, false>
                  : ni == 4 ? sparse ? gather_cols_kernel<4, true> : gather_cols_kernel<4, false>
                            : sparse ? gather_cols_kernel<2, true> : gather_cols_kernel<2, false>;
    GRASS_CUDA_TRY(launch_kernel(kernel, ggrid, kGatherThreads, 0, s, gg, lddy,
                                 static_cast<int>(T), static_cast<int>(m), r, plan.r_pad, status));
  }

  TcParams p;
  p.T = static_cast<int>(T);
  p.n = static_cast<int>(n);
  p.r = r;
  p.k_blocks = plan.k_blocks;
  p.split_k = plan.split_k;
  p.s_long = plan.s_long;
  p.kb_unit = plan.kb_unit;
  p.groups = count;
  for (int z = 0; z <= kTcMaxSlices; ++z) p.unit_begin[z] = static_cast<unsigned short>(plan.unit_begin[z]);
  p.status = status;
  p.norm_part = fused_norms ? part[0] : nullptr;
  const bool in_kernel = plan.gather == kOptCta || plan.gather == kOptCoop;
  for (int g = 0; g < kTcMaxGroup; ++g) {
    const int gi = g < count ? g : 0;
    p.dY[g] = in_kernel ? gg.dY[gi] : nullptr;
    p.idx[g] = in_kernel ? gg.idx[gi] : nullptr;
    p.Ag[g] = plan.gather == kOptCoop ? gg.Ag[gi] : nullptr;
  }
  p.lddy = lddy;
  p.m = static_cast<int>(m);
  p.r_pad = plan.r_pad;
  p.coop_ctrl = nullptr;
  p.coop_warps = opts.gather_warps > 0 ? opts.gather_warps : 8;
  p.sparse_pick = sparse_pick(m, r) ? 1 : 0;
  p.coop_chunks = static_cast<int>((T + kCoopChunk - 1) / kCoopChunk);
  p.coop_cg = (plan.r_pad + kCoopCols - 1) / kCoopCols;
  p.coop_pmax_long = p.coop_pmax_short = 0;
  for (int z = 0; z < plan.split_k; ++z) {
    const int units = plan.unit_begin[z + 1] - plan.unit_begin[z];
    int& pm = z < plan.s_long ? p.coop_pmax_long : p.coop_pmax_short;
    if (units > pm) pm = units;
  }
  if (plan.gather == kOptCoop) {
    // queue head and per-chunk counters start at zero for every launch
    p.coop_ctrl = static_cast<int*>(ws);
    const int ints = static_cast<int>(plan.ctrl_bytes / sizeof(int));
    GRASS_CUDA_TRY(launch_kernel(zero_ctrl_kernel, (ints + 1023) / 1024, 1024, 0, s,
                                 p.coop_ctrl, ints));
  }
  p.ld_norm = static_cast<long long>(round_up(static_cast<size_t>(m), 32));
  for (int g = 0; g < kTcMaxGroup; ++g) {
    const int gi = g < count ? g : 0;
    if (plan.split_k == 1 && !stored) {
      p.out[g] = Gc != nullptr ? Gc[gi] : nullptr;   // unused in row-norm mode
      p.rho[g] = rho != nullptr ? rho[gi] : nullptr;
    } else {
      p.out[g] = part[gi];
      p.rho[g] = nullptr;
    }
  }
  p.ld_out = plan.split_k == 1 && !stored ? ldgc : plan.ld_part;
  p.split_stride = plan.split_k == 1 ? 0 : static_cast<long long>(r) * plan.ld_part;
  // tile space handed to the persistent kernel (x counts pairs of CTAs in pair mode)
  dim3 grid(static_cast<unsigned>(plan.pair ? plan.n_blocks / 2 : plan.n_blocks),
            static_cast<unsigned>(plan.r_blocks), static_cast<unsigned>(plan.split_k * count));

  const int kernel_gather = plan.gather == kOptCta ? kGatherCta
                            : plan.gather == kOptCoop ? kGatherCoop : kGatherNone;
  const int rc = launch_tc(plan.MB, plan.r_cta / 64, plan.pair, kernel_gather, grid, plan.smem_bytes,
                           s, maps, p, gather ? GRASS_K_PROJECT_TC : GRASS_K_PROJECT_TC_DENSE);
  if (rc != GRASS_OK) return rc;
  if (norms != nullptr) {
    ProfileScope prof(GRASS_K_ROW_NORMS, s);
    if (fused_norms)
      GRASS_CUDA_TRY(launch_kernel(norms_finalize_kernel, static_cast<unsigned>((m + 255) / 256), 256, 0, s,
                                   p.norm_part, p.ld_norm, static_cast<int>((n + 31) / 32),
                                   static_cast<int>(m), norms));
    else
      GRASS_CUDA_TRY(launch_row_norms(part[0], plan.ld_part, p.split_stride, plan.split_k, m, n, norms, stored, s));
    if (stored) *keep = {keep->r, part[0], plan.ld_part};
    return GRASS_OK;
  }
  if (upd != nullptr) {
    for (int g = 0; g < count; ++g) upd->grp.part[g] = part[g];
    upd->split_k = plan.split_k > 1 ? plan.split_k : 0;
    upd->ld_part = plan.ld_part;
    upd->split_stride = p.split_stride;
    return launch_update(*upd, s);
  }
  if (plan.split_k > 1) {
    ReduceGroup rg;
    int vec = (n % 4 == 0) && (ldgc % 4 == 0);
    for (int g = 0; g < kTcMaxGroup; ++g) {
      const int gi = g < count ? g : 0;
      rg.part[g] = part[gi];
      rg.rho[g] = rho != nullptr ? rho[gi] : nullptr;
      rg.Gc[g] = Gc[gi];
      vec = vec && aligned_to(Gc[gi], 16);
    }
    const long long work = static_cast<long long>(r) * (vec ? n / 4 : n);
    long long blocks = (work + 255) / 256;
    if (blocks > kSmCount * 32) blocks = kSmCount * 32;
    ProfileScope prof(GRASS_K_SPLITK_REDUCE, s);
    GRASS_CUDA_TRY(launch_kernel(splitk_reduce_kernel,
                                 dim3(static_cast<unsigned>(blocks), static_cast<unsigned>(count)), 256, 0, s,
                                 rg, plan.ld_part, p.split_stride, plan.split_k, r,
                                 static_cast<int>(n), ldgc, vec));
  }
  return GRASS_OK;
}

void describe_plan(const TcPlan& plan, int count, grass_project_plan_t* out) {
  out->gather = plan.gather;
  out->rows_per_tile = plan.r_cta;
  out->row_blocks = plan.r_blocks;
  out->n_blocks_per_cta = plan.MB;
  out->ctas_per_slice = plan.n_blocks * plan.r_blocks * count;
  out->cta_pair = plan.pair ? 1 : 0;
  out->token_slices = plan.split_k;
  out->short_slices = plan.split_k - plan.s_long;
  out->long_slice_tokens = (plan.unit_begin[1] - plan.unit_begin[0]) * plan.kb_unit * plan.bk;
  out->tokens_per_stage = plan.bk;
  out->stages = plan.stages;
  out->workspace_bytes = plan_ws_bytes(plan, count) + 256;
}

}  // namespace
}  // namespace grass

namespace grass {
namespace {
PlanOpts wide_opts() {
  PlanOpts o;
  o.wide = true;
  return o;
}
// Workspace of the projection calls and of the layer-step on `count` layers.
size_t selected_ws_bytes(int count, int64_t T, int64_t m, int64_t n, int r) {
  const size_t call = plan_ws_bytes(make_plan(T, m, n, r, true, PlanOpts(), false, count), count);
  const size_t step = plan_ws_bytes(make_plan(T, m, n, r, true, wide_opts(), false, count), count);
  return call > step ? call : step;
}
}  // namespace
}  // namespace grass

extern "C" size_t grass_project_workspace_bytes(int64_t T, int64_t m, int64_t n, int32_t r,
                                                int dt) {
  if (T < 1 || m < 1 || n < 1 || r < 1) return 0;
  if (dt != GRASS_BF16) {
    const size_t step = grass::make_fp32_plan(T, n, r).part_bytes;
    const size_t refresh = grass::make_fp32_plan(T, n, r, r).part_bytes;
    return (step > refresh ? step : refresh) + 256;
  }
  // covers the call with and without idx (the dense form needs no gathered operand)
  const size_t with_idx = grass::selected_ws_bytes(1, T, m, n, r);
  const size_t dense = grass::plan_ws_bytes(grass::make_plan(T, m, n, r, false, grass::PlanOpts()), 1);
  return (with_idx > dense ? with_idx : dense) + 256;
}

namespace grass {
namespace {
int project_fp32(const void* dY, int64_t lddy, const void* X, int64_t ldx, int64_t T, int64_t m,
                 int64_t n, const int32_t* idx, const float* rho, int32_t r, float* Gc,
                 int64_t ldgc, void* ws, size_t ws_bytes, cudaStream_t s, UpdateCall* upd = nullptr,
                 float* norms = nullptr, GradParts* keep = nullptr, int slices_of = 0) {
  cudaError_t err;
  int* status = status_word(&err);
  if (status == nullptr) GRASS_CUDA_TRY(err);
  const Fp32Plan fp = make_fp32_plan(T, n, r, slices_of);
  if (fp.split > 1 && (ws == nullptr || !aligned_to(ws, 256) || ws_bytes < fp.part_bytes))
    return GRASS_ERR_WORKSPACE;
  float* out = fp.split > 1 ? static_cast<float*>(ws) : Gc;
  const int64_t ld_out = fp.split > 1 ? fp.ld_part : ldgc;
  const int rc = (fp.big ? launch_simt<8> : launch_simt<4>)(
      fp, static_cast<const float*>(dY), lddy, static_cast<const float*>(X), ldx, T, m, n, idx, rho, r, out,
      ld_out, status, s);
  if (rc != GRASS_OK) return rc;
  if (norms != nullptr) {
    // row-norm mode (idx NULL, r == m): the norms straight from the partials
    ProfileScope prof(GRASS_K_ROW_NORMS, s);
    const long long stride = static_cast<long long>(r) * fp.ld_part;
    GRASS_CUDA_TRY(launch_row_norms(out, ld_out, stride, fp.split, m, n, norms, keep != nullptr, s));
    if (keep != nullptr) *keep = {keep->r, out, static_cast<long long>(ld_out)};
    return GRASS_OK;
  }
  if (upd != nullptr) {
    upd->grp.part[0] = out;
    upd->split_k = fp.split > 1 ? fp.split : 0;
    upd->ld_part = fp.ld_part;
    upd->split_stride = static_cast<long long>(r) * fp.ld_part;
    return launch_update(*upd, s);
  }
  if (fp.split > 1) {
    const int vec = (n % 4 == 0) && (ldgc % 4 == 0) && aligned_to(Gc, 16);
    const long long work = static_cast<long long>(r) * (vec ? n / 4 : n);
    long long blocks = (work + 255) / 256;
    if (blocks > kSmCount * 32) blocks = kSmCount * 32;
    ProfileScope prof(GRASS_K_SPLITK_REDUCE, s);
    ReduceGroup rg;
    for (int g = 0; g < kTcMaxGroup; ++g) { rg.part[g] = out; rg.rho[g] = rho; rg.Gc[g] = Gc; }
    GRASS_CUDA_TRY(launch_kernel(splitk_reduce_kernel, static_cast<unsigned>(blocks), 256, 0, s, rg,
                                 fp.ld_part, static_cast<long long>(r) * fp.ld_part, fp.split, r,
                                 static_cast<int>(n), ldgc, vec));
  }
  return GRASS_OK;
}
}  // namespace
}  // namespace grass

extern "C" int grass_project_grad(const void* dY, int64_t lddy, const void* X, int64_t ldx, int dt,
                                  int64_t T, int64_t m, int64_t n, const int32_t* idx,
                                  const float* rho, int32_t r, float* Gc, int64_t ldgc, void* ws,
                                  size_t ws_bytes, void* stream) {
  using namespace grass;
  if (dY == nullptr || X == nullptr || Gc == nullptr || T < 1 || m < 1 || n < 1 || r < 1 ||
      lddy < m || ldx < n || ldgc < n || T > 0x7fffffffLL || m > 0x7fffffffLL ||
      n > 0x7fffffffLL)
    return GRASS_ERR_INVALID_ARG;
  if (idx == nullptr && r != m) return GRASS_ERR_INVALID_ARG;
  if (r > m) return GRASS_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (dt == GRASS_BF16)
    return project_bf16(1, &dY, lddy, &X, ldx, T, m, n, idx != nullptr ? &idx : nullptr, &rho, r,
                        &Gc, ldgc, nullptr, ws, ws_bytes, PlanOpts(), s);
  if (dt != GRASS_F32) return GRASS_ERR_UNSUPPORTED;
  return project_fp32(dY, lddy, X, ldx, T, m, n, idx, rho, r, Gc, ldgc, ws, ws_bytes, s);
}

extern "C" size_t grass_project_batched_workspace_bytes(int32_t count, int64_t T, int64_t m,
                                                        int64_t n, int32_t r) {
  if (count < 1 || count > grass::kTcMaxGroup || T < 1 || m < 1 || n < 1 || r < 1) return 0;
  return grass::selected_ws_bytes(count, T, m, n, r) + 256;
}

extern "C" int grass_project_grad_batched(int32_t count, const void* const* dY, int64_t lddy,
                                          const void* const* X, int64_t ldx, int64_t T, int64_t m,
                                          int64_t n, const int32_t* const* idx,
                                          const float* const* rho, int32_t r, float* const* Gc,
                                          int64_t ldgc, void* ws, size_t ws_bytes, void* stream) {
  return grass_project_grad_ex(count, dY, lddy, X, ldx, T, m, n, idx, rho, r, Gc, ldgc, ws, ws_bytes,
                               nullptr, stream);
}

extern "C" int grass_project_plan(int32_t count, int64_t T, int64_t m, int64_t n, int32_t r,
                                  const grass_project_opts_t* opts, grass_project_plan_t* plan) {
  using namespace grass;
  if (plan == nullptr || count < 1 || count > kTcMaxGroup || T < 1 || m < 1 || n < 1 || r < 1 ||
      r > m || T > 0x7fffffffLL || m > 0x7fffffffLL || n > 0x7fffffffLL || !opts_ok(opts))
    return GRASS_ERR_INVALID_ARG;
  describe_plan(make_plan(T, m, n, r, true, to_plan_opts(opts), false, count), count, plan);
  return GRASS_OK;
}

extern "C" int grass_step_plan(int32_t count, int64_t T, int64_t m, int64_t n, int32_t r,
                               grass_project_plan_t* plan) {
  using namespace grass;
  if (plan == nullptr || count < 1 || count > kTcMaxGroup || T < 1 || m < 1 || n < 1 || r < 1 ||
      r > m || T > 0x7fffffffLL || m > 0x7fffffffLL || n > 0x7fffffffLL)
    return GRASS_ERR_INVALID_ARG;
  describe_plan(make_plan(T, m, n, r, true, wide_opts(), false, count), count, plan);
  return GRASS_OK;
}

extern "C" int64_t grass_plan_searches(void) { return grass::plan_searches; }

extern "C" int grass_project_grad_ex(int32_t count, const void* const* dY, int64_t lddy,
                                     const void* const* X, int64_t ldx, int64_t T, int64_t m,
                                     int64_t n, const int32_t* const* idx, const float* const* rho,
                                     int32_t r, float* const* Gc, int64_t ldgc, void* ws,
                                     size_t ws_bytes, const grass_project_opts_t* opts,
                                     void* stream) {
  using namespace grass;
  if (count < 1 || count > kTcMaxGroup || dY == nullptr || X == nullptr || idx == nullptr ||
      Gc == nullptr || T < 1 || m < 1 || n < 1 || r < 1 || r > m || lddy < m || ldx < n ||
      ldgc < n || T > 0x7fffffffLL || m > 0x7fffffffLL || n > 0x7fffffffLL || !opts_ok(opts))
    return GRASS_ERR_INVALID_ARG;
  for (int g = 0; g < count; ++g)
    if (idx[g] == nullptr) return GRASS_ERR_INVALID_ARG;
  return project_bf16(count, dY, lddy, X, ldx, T, m, n, idx, rho, r, Gc, ldgc, nullptr, ws, ws_bytes,
                      to_plan_opts(opts), static_cast<cudaStream_t>(stream));
}

namespace grass {
namespace {

// Argument checks of a layer-step, and its update half.
int check_step(const grass_step_t* a, UpdateCall& u) {
  if (a == nullptr || a->count < 1 || a->count > kTcMaxGroup || a->T < 1 || a->m < 1 || a->n < 1 ||
      a->r < 1 || a->r > a->m || a->lddy < a->m || a->ldx < a->n || a->T > 0x7fffffffLL ||
      a->m > 0x7fffffffLL || a->n > 0x7fffffffLL || (a->dt == GRASS_F32 && a->count != 1) ||
      (a->side != GRASS_SIDE_ROWS && a->side != GRASS_SIDE_COLS))
    return GRASS_ERR_INVALID_ARG;
  if (a->dt != GRASS_F32 && a->dt != GRASS_BF16) return GRASS_ERR_UNSUPPORTED;
  for (int g = 0; g < a->count; ++g) {
    if (a->dY[g] == nullptr || a->X[g] == nullptr) return GRASS_ERR_INVALID_ARG;
    u.grp.Gc[g] = a->Gc[g]; u.grp.M[g] = a->M[g]; u.grp.V[g] = a->V[g]; u.grp.U[g] = a->U[g];
    u.grp.W[g] = a->W[g]; u.grp.idx[g] = a->idx[g]; u.grp.rho[g] = a->rho[g];
  }
  u.count = a->count; u.wdt = a->wdt; u.r = a->r; u.cols = a->side == GRASS_SIDE_COLS;
  u.m = a->m; u.n = a->n; u.ldgc = a->ldgc; u.ldstate = a->ldstate; u.ldw = a->ldw;
  return check_update(u, a->lr, a->beta1, a->beta2, a->eps, a->step, a->alpha);
}

// refresh: the projection of a refresh iteration, with the token slices of the projection calls
// (make_keep_plan says why).
int project_and_update(const grass_step_t* a, UpdateCall& u, cudaStream_t s, bool refresh = false) {
  if (a->dt == GRASS_F32)
    return project_fp32(a->dY[0], a->lddy, a->X[0], a->ldx, a->T, a->m, a->n, a->idx[0], a->rho[0],
                        a->r, a->Gc[0], a->ldgc, a->ws, a->ws_bytes, s, &u, nullptr, nullptr,
                        refresh ? a->r : 0);
  return project_bf16(a->count, a->dY, a->lddy, a->X, a->ldx, a->T, a->m, a->n, a->idx, a->rho, a->r,
                      a->Gc, a->ldgc, nullptr, a->ws, a->ws_bytes, refresh ? PlanOpts() : wide_opts(), s, &u);
}

// What the projection of a refresh iteration will refuse, if it has one: asked before the selection
// replaces the layer's rows.
int refresh_projection_refused(const grass_step_t* a, size_t norm_ws_bytes) {
  TcPlan plan;
  if (a->dt == GRASS_F32) {
    const Fp32Plan fp = make_fp32_plan(a->T, a->n, a->r, a->r);
    return fp.split > 1 && (a->ws == nullptr || !aligned_to(a->ws, 256) || a->ws_bytes < fp.part_bytes) &&
                   !keeps_fp32(a->T, a->m, a->n, a->r, norm_ws_bytes)
               ? GRASS_ERR_WORKSPACE : GRASS_OK;
  }
  plan = make_plan(a->T, a->m, a->n, a->r, true, PlanOpts());
  const int refused = plan_refused(plan, a->T, plan_ws_bytes(plan, 1), a->ws, a->ws_bytes);
  return refused != GRASS_OK && keeps(a->T, a->m, a->n, a->r, norm_ws_bytes, &plan) ? GRASS_OK : refused;
}

// Row norms of dY^T X; keep (may be NULL) learns where the gradient was formed, if it was.
int grad_row_norms(const void* dY, int64_t lddy, const void* X, int64_t ldx, int dt, int64_t T, int64_t m,
                   int64_t n, float* norms, void* ws, size_t ws_bytes, cudaStream_t s, GradParts* keep) {
  if (dY == nullptr || X == nullptr || norms == nullptr || T < 1 || m < 1 || n < 1 || lddy < m ||
      ldx < n || T > 0x7fffffffLL || m > 0x7fffffffLL || n > 0x7fffffffLL)
    return GRASS_ERR_INVALID_ARG;
  if (dt == GRASS_BF16)
    return project_bf16(1, &dY, lddy, &X, ldx, T, m, n, nullptr, nullptr, static_cast<int>(m),
                        nullptr, 0, norms, ws, ws_bytes, PlanOpts(), s, nullptr, keep);
  if (dt != GRASS_F32) return GRASS_ERR_UNSUPPORTED;
  // fp32 path: the (small) gradient is formed in the workspace, whole or as partials
  if (ws == nullptr || !aligned_to(ws, 256) ||
      ws_bytes < grass_grad_row_norms_workspace_bytes(T, m, n, dt) - 256)
    return GRASS_ERR_WORKSPACE;
  if (keep != nullptr && !keeps_fp32(T, m, n, keep->r, ws_bytes)) keep = nullptr;
  const long long ld = static_cast<long long>(round_up(static_cast<size_t>(n), 4));
  return project_fp32(dY, lddy, X, ldx, T, m, n, nullptr, nullptr, static_cast<int32_t>(m),
                      static_cast<float*>(ws), ld, ws, ws_bytes, s, nullptr, norms, keep,
                      keep != nullptr ? keep->r : 0);
}

}  // namespace
}  // namespace grass

extern "C" int grass_layer_step(const grass_step_t* a, void* stream) {
  using namespace grass;
  UpdateCall u = {};
  const int rc = check_step(a, u);
  return rc != GRASS_OK ? rc : project_and_update(a, u, static_cast<cudaStream_t>(stream));
}

extern "C" size_t grass_refresh_workspace_bytes(int64_t T, int64_t m, int64_t n, int32_t r, int dt) {
  using namespace grass;
  const size_t norms = grass_grad_row_norms_workspace_bytes(T, m, n, dt);
  if (norms == 0 || r < 1 || r > m) return 0;
  size_t kept = 0;
  TcPlan plan;
  if (dt != GRASS_BF16) {
    if (keep_fp32(T, m, n, r)) kept = make_fp32_plan(T, n, static_cast<int>(m), r).part_bytes + 256;
  } else if (make_keep_plan(T, m, n, r, &plan)) {
    kept = grad_parts_bytes(plan.split_k, m, plan.ld_part) + 256;
  }
  return kept > norms ? kept : norms;
}

extern "C" int grass_refresh_keeps_gradient(int64_t T, int64_t m, int64_t n, int32_t r, int dt) {
  using namespace grass;
  if (T < 1 || m < 1 || n < 1 || r < 1 || r > m) return 0;
  TcPlan plan;
  return (dt == GRASS_BF16 ? make_keep_plan(T, m, n, r, &plan) : dt == GRASS_F32 && keep_fp32(T, m, n, r)) ? 1 : 0;
}

extern "C" int grass_refresh_step(const grass_step_t* a, const grass_refresh_t* f, void* stream) {
  using namespace grass;
  UpdateCall u = {};
  const int rc = check_step(a, u);
  if (rc != GRASS_OK) return rc;
  if (f == nullptr || a->count != 1 || f->norms == nullptr || a->rho[0] == nullptr)
    return GRASS_ERR_INVALID_ARG;
  if (f->method < GRASS_SEL_TOPR || f->method > GRASS_SEL_UNIFORM_NR) return GRASS_ERR_UNSUPPORTED;
  if (f->method != GRASS_SEL_TOPR &&
      (f->select_ws == nullptr || !aligned_to(f->select_ws, 256) ||
       f->select_ws_bytes < grass_select_workspace_bytes(a->m, a->r, f->method)))
    return GRASS_ERR_WORKSPACE;
  int rc2 = refresh_projection_refused(a, f->norm_ws_bytes);
  if (rc2 != GRASS_OK) return rc2;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  GradParts kept;
  kept.r = a->r;
  rc2 = grad_row_norms(a->dY[0], a->lddy, a->X[0], a->ldx, a->dt, a->T, a->m, a->n, f->norms,
                           f->norm_ws, f->norm_ws_bytes, s, &kept);
  if (rc2 != GRASS_OK) return rc2;
  rc2 = select_rows(f->norms, a->m, a->r, f->method, f->seed, f->layer_id, f->epoch,
                     const_cast<int32_t*>(a->idx[0]), const_cast<float*>(a->rho[0]), f->select_ws,
                     f->select_ws_bytes, s);
  if (rc2 != GRASS_OK) return rc2;
  u.reset = f->reset_state != 0;
  if (kept.grad == nullptr) return project_and_update(a, u, s, true);
  u.grp.part[0] = kept.grad;
  u.ld_part = kept.ld;
  u.split_k = 1;
  u.part_by_row = true;
  return launch_update(u, s);
}

extern "C" size_t grass_grad_row_norms_workspace_bytes(int64_t T, int64_t m, int64_t n, int dt) {
  if (m < 1 || n < 1 || T < 1) return 0;
  if (dt == GRASS_BF16) {
    const grass::TcPlan plan = grass::make_norms_plan(T, m, n);
    return (plan.split_k == 1 ? grass::norm_part_bytes(m, n) : plan.part_bytes) + 256;
  }
  // (the pitch of the formed gradient is n rounded up to 4)
  return grass::round_up(static_cast<size_t>(m) * grass::round_up(static_cast<size_t>(n), 4) * sizeof(float), 256) +
         grass::make_fp32_plan(T, n, static_cast<int>(m)).part_bytes + 256;
}

extern "C" int grass_grad_row_norms(const void* dY, int64_t lddy, const void* X, int64_t ldx, int dt,
                                    int64_t T, int64_t m, int64_t n, float* norms, void* ws,
                                    size_t ws_bytes, void* stream) {
  return grass::grad_row_norms(dY, lddy, X, ldx, dt, T, m, n, norms, ws, ws_bytes,
                               static_cast<cudaStream_t>(stream), nullptr);
}
