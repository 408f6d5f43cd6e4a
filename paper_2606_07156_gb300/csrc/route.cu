// Which search serves a batch (the automatic choice): the cheapest by estimates
// of the searches' device time, from the shape of the batch and the index alone.
//
// Two searches serve every batch, and one of them is the base: the grouped
// kernels where the policy can choose tables of at most 8 bits, else the
// query-major kernel with one block a query. Three others finish some batches
// sooner: the query-major kernel with several blocks a query (few queries: the
// base leaves most of the GPU idle), or with one where the base is grouped (128-
// entry lists cost the grouped kernels a merge per pair), and the filter (the
// look-ups of large batches become a GEMM, behind some 100 us of launches, 150 to
// 180 us with quantised tables).
//
// The estimates are non-negative least-squares fits, in relative error, to the
// times of each search on 968 batches drawn over 1 to 10000 queries, 1 to 64
// probes, 5 thousand to 1 million vectors, D 48 to 960, M 12 to 120, k 1 to 128,
// lists of 120 to 2500 vectors on average, even and very uneven, all table widths
// (the part all searches share, the coarse stage, left out). Their errors are a
// factor of 1.25 to 1.7 (one standard deviation; the filter's most: its time
// depends on how well its bounds fit the data). So another search is taken by a
// margin: several blocks a query always on wide tables (hardly ever slower, 0.93
// at worst) and where estimated 1.1 times as fast as the grouped kernels, one
// block a query 1.3 times; the filter where estimated faster than one block a
// query, and 1.5 times as fast as several or as the grouped kernels. On those
// batches 27 of 968 are then more than 3 % slower than the base (the worst 0.71 of
// its speed), and the geometric mean is 1.83 times the base's speed; 1.91 if the
// fastest search were always known. (Lines drawn by size alone, as they were
// before, left 92 slower, the worst 0.22.)
#include <algorithm>
#include <cmath>

#include "internal.h"

namespace anns {
namespace {

// Shape of a batch: queries, probes a query, padded sub-spaces, vectors a probed
// list (lists are probed about as often as they are long: sum n^2 / sum n) and
// in the longest, dimension, k, and k / 128 where 128-entry lists are used.
struct Shape {
  double nq, p, Mp, L, longest, D, k, big;
};

enum Widths { kPlain, kWide, kFixed8, kFixed6, kFixed4, kMixed };

Widths widths_of(const anns_precision_policy& P) {
  switch (P.lut_mode) {
    case ANNS_LUT_PLAIN_FP32: return kPlain;
    case ANNS_LUT_FIXED_BITS:
      return P.fixed_bits > 8 ? kWide : P.fixed_bits == 8 ? kFixed8 : P.fixed_bits > 4 ? kFixed6 : kFixed4;
    default: return kMixed;
  }
}

// Microseconds of the query-major kernel with `split` blocks a query: a block's
// chain of pairs, and all pairs and queries over the 304 blocks that run at once
// (table builds by Mp, scans by L Mp), the longest list, and 128-entry lists, whose
// filling grows with k.
double query_major_us(Widths w, const Shape& s, double split) {
  static const double c[3][9] = {{54, .0616, .0566, 29.5e-6, 68e-6, .289, 130, 5.79, 4.1},    // FP32 tables
                                 {62, .1160, .1110, 34.0e-6, 62e-6, .307, 147, 4.83, 2.7},    // both
                                 {64, .0916, .0884, 18.2e-6, 51e-6, .326, 230, 2.19, 7.3}};   // byte tables
  static const double merge[3] = {179, 224, 79};  // of a query's 128-entry lists
  const int f = w == kPlain ? 0 : w == kWide || w == kMixed ? 1 : 2;
  const double* a = c[f];
  const double chain = std::max(1.0, s.p / split), all = s.nq * s.p / 304.0, blocks = s.nq * split / 304.0;
  return a[0] + (a[1] * chain + (a[2] + a[3] * s.L) * all + a[4] * s.longest + a[5] * blocks) * s.Mp +
         s.big * (a[6] + a[7] * chain + a[8] * all + merge[f] * blocks);
}

// The grouped kernels: table entries and look-ups of all pairs, the longest list,
// one group's latency, the queries' rank-0 pairs, and the per-pair lists of k > 32.
double grouped_us(Widths w, const Shape& s) {
  static const double c[3][8] = {{129, 204e-6, .0513e-6, 84e-6, 34e-6, 1.95e-3, 307, .087},    // 5..8 bits
                                 {136, 281e-6, .0148e-6, 88e-6, 0, 1.09e-3, 389, .0127},       // 4 bits
                                 {147, 211e-6, .0779e-6, 62e-6, 123e-6, .97e-3, 337, .0086}};  // mixed
  static const double merge[3] = {.341, .800, .986};
  const int f = w == kMixed ? 2 : w == kFixed4 ? 1 : 0;
  const double* a = c[f];
  const double pairs = s.nq * s.p;
  return a[0] + (a[1] * pairs + a[2] * pairs * s.L + a[3] * s.longest + a[4] * (256.0 + s.L) + a[5] * s.nq) * s.Mp +
         s.big * (a[6] + a[7] * pairs + merge[f] * s.nq);
}

// The filter: per pair, the GEMM (L D), per query row statistics and candidates,
// the longest list's tiles, and the depth of the exact stage.
double filter_us(Widths w, const Shape& s) {
  static const double c[4][8] = {{96, .80e-3, .75e-9, .31e-3, .46e-3, 5.0e-6, .78, .61},        // FP32
                                 {108, 2.12e-3, 1.14e-9, 1.31e-3, .60e-3, 4.0e-6, .83, .19},    // 12, 16 bits
                                 {152, .39e-3, 6.05e-9, 2.18e-3, 1.75e-3, 12e-6, 1.06, .62},    // 8 bits
                                 {180, .49e-3, 10.9e-9, .49e-3, 1.72e-3, 11e-6, .95, 1.78}};    // mixed
  const double* a = c[w == kPlain ? 0 : w == kWide ? 1 : w == kMixed ? 3 : 2];
  const double pairs = s.nq * s.p;
  return a[0] + a[1] * pairs + a[2] * pairs * s.L * s.D + a[3] * s.nq * s.Mp + a[4] * s.nq * s.k +
         a[5] * s.longest * s.D + a[6] * s.Mp + a[7] * s.k;
}

}  // namespace

Route route_of(const Index& ix, const anns_precision_policy& P, int64_t nq, int nprobe, int k, double probes) {
  const Widths w = widths_of(P);
  const Shape s{(double)nq, probes, (double)ix.Mp, ix.list_seen, (double)ix.max_list, (double)ix.dim, (double)k,
                k > 32 ? k / 128.0 : 0.0};
  Route r;
  const bool filter = filter_possible(ix, P, nq, nprobe, k);
  // fixed 6 bits: the quantiser's bound, four times that of 8 bits, leaves most
  // vectors in (0.2 to 3.6 times the speed of the grouped kernels, mostly below 1)
  const bool filter_pays = filter && w != kFixed6;
  switch (ix.opt_kernel) {
    case ANNS_KERNEL_BASIC:
    case ANNS_KERNEL_LIST_MAJOR:
    case ANNS_KERNEL_SPLIT_SCAN: return r;
    case ANNS_KERNEL_GROUPED: r.grouped = grouped_supported(ix, k); return r;
    case ANNS_KERNEL_SPLIT: r.filter = filter_pays && filter_us(w, s) < query_major_us(w, s, 1.0); return r;
    default: break;
  }
  const bool narrow = w != kPlain && w != kWide && grouped_supported(ix, k);
  const double one = query_major_us(w, s, 1.0);
  double best = narrow ? grouped_us(w, s) : one, margin = narrow ? 1.5 : 1.0;
  r.grouped = narrow;
  // several blocks a query run all at once: there is no order to ask for
  const bool any_order = ix.opt_schedule == ANNS_SCHED_AUTO;
  const int split = any_order ? search_split(nq, nprobe, k) : 1;
  const double some = split > 1 ? query_major_us(w, s, split) : INFINITY;
  if (split > 1 && (!narrow || 1.1 * some < best)) {
    best = some;
    margin = 1.5;
    r.grouped = false;
    r.split = split;
  } else if (narrow && any_order && 1.3 * one < best) {
    best = one;
    margin = 1.0;
    r.grouped = false;
  }
  r.filter = ix.opt_kernel == ANNS_KERNEL_FILTERED ? filter : filter_pays && margin * filter_us(w, s) < best;
  return r;
}

}  // namespace anns
