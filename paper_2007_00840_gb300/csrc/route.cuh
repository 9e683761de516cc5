// Which patterns are eliminated on chip and which are traversed: the predicted times, in
// us, that the choice compares, and the lines that were measured directly.  Times of whole
// calls on a GB300.
//
// Elimination costs panels, whatever is in them; a traversal costs what a row reaches.  The
// reach of a few rows is therefore sampled (band_reach_kernel): levels and entries of a
// breadth-first search below the row, cut off once the row is known to cost more than the
// elimination would; a row cut off counts as reaching every row before it, so that patterns
// of unknown reach stay with the elimination.  Before the sample, a million rows with one
// entry each at a random distance of up to 2,000 took 294 ms as a band against 7.9 by
// traversal, and ten thousand with an entry in every second row within 300 1,000 us
// against 233.
#pragma once

#include "band.cuh"

namespace gsofa {

// Orders from which the blocks of a dissection are looked for: any pattern whose band does
// not fit, and one that looks like a dissection (entries near the diagonal, few far out).
// Dissections of square grids, traversal / blocks: order 2,025 414 / 455 us, 2,809 468 /
// 452, 4,900 628 / 469, 10,000 993 / 561, 16,256 1,351 / 631.
constexpr int32_t FRONT_MIN_ORDER = 16384;
constexpr int32_t FRONT_NEAR_ORDER = 2600;

constexpr int REACH_ROWS = 128;        // rows sampled of one matrix
constexpr int REACH_ROWS_MIN = 4;      // and at least of each matrix of a batch (about two per SM in all)

// The traversal has to be this much faster by the prediction.
constexpr float ROUTE_MARGIN = 1.1f;

// Rows sampled per matrix when `mats` matrices are.
inline int reach_rows(int mats) {
  const int r = mats > 0 ? 304 / mats : 0;
  return r > REACH_ROWS ? REACH_ROWS : (r < REACH_ROWS_MIN ? REACH_ROWS_MIN : r);
}

// ns that a level and an entry of a row's search cost the traversal with the chip full of
// rows (and every row by itself, row).  Calls: chains of 50 to 510 levels 0.2 ns a level,
// grids of 64 x 64 to 32^3 3 to 4 ps an entry.  Counts alone (a CTA per row, its labels
// cleared for every row): 3 ns a level while several rows fit an SM, then growing with
// the order (20,000 rows 12 ns, 65,000 39).
struct TraverseCost {
  float row, level, entry;
};
__host__ __device__ inline TraverseCost traverse_cost(int n, bool counts) {
  if (!counts) return TraverseCost{6.4f, 0.2f, 0.004f};
  const float level = n < 12288 ? 3.f : 0.6e-3f * (float)n;
  return TraverseCost{n < 12288 ? 8.5f : 30.f, level, level / 700.f};
}
// What a traversal takes whatever its rows reach.
__host__ __device__ inline float traverse_base_us(int n, bool counts) {
  return (counts ? 45.f : 165.f) + 1e-3f * traverse_cost(n, counts).row * (float)n;
}
// The longest row alone, where few rows are long: 1 us a level, 12 ns an entry.
__host__ __device__ inline float row_us(float levels, float entries) { return levels + 0.012f * entries; }

// us of a panel: 1.5 at 2 words left and right, 2.5 at 10, 4.4 at 32 (up to 6 where few rows
// of a panel have partners), 8.6 at 63; sizes alone, where a warp counts a row, about 1 more
// on narrow bands.
__host__ __device__ inline float panel_us(int LB, int UB, bool counts) {
  const float w = 0.5f * (float)(LB + UB);
  return counts ? 2.4f + 0.08f * w : 1.3f + 0.115f * w;
}
// Elimination as a band: `chain` panels one after the other.
__host__ __device__ inline float band_us(int n, int chain, int LB, int UB, bool counts) {
  return (counts ? 30.f : 135.f + 0.9e-3f * (float)n) + (float)chain * panel_us(LB, UB, counts);
}
// Elimination block by block of a dissection: 472 us at order 2,601, 586 at 10,000, 954 at
// 65,536, 5.2 ms at 1,048,576.
__host__ __device__ inline float fronts_us(int n) { return 300.f + 5e-3f * (float)n; }
// The search for blocks, 150 to 200 us where there are none, is worth it from traversals of this time on.
__host__ __device__ inline float fronts_limit_us(int n) { return ROUTE_MARGIN * fronts_us(n) + 1.5e-3f * (float)n; }

// us that the searches of all rows together have to stay below for a traversal to be chosen
// instead of a band that takes `band` us (0: it does not fit) or of the search for blocks;
// 0: not sampled.  A band is left alone where it takes less than 1.6 times what a traversal
// takes at least, and below 3 ms where its rows have 3.25 entries or more (grids have 3.4 to
// 6, chains 3): the search would take 30 us of 600 there, and 100 of 7,400 on a 317 x 293
// grid.
__host__ __device__ inline float reach_limit_us(int n, unsigned long long nnz, float band, bool counts) {
  const float base = traverse_base_us(n, counts);
  if (band == 0.f) return counts || n < FRONT_NEAR_ORDER ? 0.f : fronts_limit_us(n) - base;
  if (band < 3000.f && (float)nnz >= 3.25f * (float)n) return 0.f;
  return band < 1.6f * ROUTE_MARGIN * base ? 0.f : band / ROUTE_MARGIN - base;
}

// Orders whose search is launched with the scan.  Below, the scan is waited for first: 25 us more
// where there is a search, 10 less where there is none (3% of a band of order 5,000).
constexpr int REACH_AT_ONCE = 16384;

// A traversal, from the sums over `rows` sampled rows (r.levels is 0 where none were).
inline float traverse_us(int n, const BandReach& r, int rows, bool counts) {
  const TraverseCost t = traverse_cost(n, counts);
  const float levels = (float)r.levels / (float)rows, entries = (float)((double)r.entries / rows);
  const float all = 1e-3f * (float)n * (t.level * levels + t.entry * entries);
  return traverse_base_us(n, counts) + (all > (float)r.longest ? all : (float)r.longest);
}

// The longest chain of panels of one matrix alone on `parts` CTAs or clusters.
inline int chain_panels(int n, int stretch, int parts) {
  const int share = ((n + 31) / 32 + parts - 1) / parts;
  return stretch > share ? stretch : share;
}

// Up to this order a dissection is one wide band (order 900: 283 us by traversal, 219 as a
// band; 1,600: 370 / 357; 2,025: 414 / 483); between the two lines it is traversed.
constexpr int32_t NEAR_BAND_ORDER = 1600;
// A band of more words than this needs a cluster of eight, 4 us per panel whatever is in it;
// with fewer entries than this in all the traversal is as fast or faster (3D grids: 27 x 27
// x 9, 37k entries, 942 us by traversal, 1,177 as a band; 33 x 33 x 9, 52k: 1,688 / 1,834;
// 27 x 27 x 20, 82k: 2,408 / 2,212; 33 x 33 x 20, 119k: 4,702 / 3,788), except for small
// orders (band 1,000 of order 3,000: 1,025 / 651).
constexpr int32_t WIDE_BAND = 16;
constexpr unsigned long long WIDE_NNZ = 56000;
constexpr int32_t WIDE_MIN_ORDER = 4096;
// Counts alone, against their own traversal: a wide band, which takes a cluster, pays from
// order 4,096 on (18 x 18 x 18 grid 845 us by traversal, 726 as a band; 12 x 12 x 12 with
// far entries 220 / 292; 18 x 18 x 9 322 / 352), and where most entries lie close to the
// diagonal, as in a dissection, up to 1,600 (40 x 40 348 / 290, 47 x 47 435 / 465).
constexpr int32_t COUNTS_WIDE_BAND = 8;

// A dissection with an entry per row beside the diagonal has long rows: blocks are looked for
// without a sample.
__host__ __device__ inline bool surely_blocks(int n, const BandCounters& h, bool near) {
  return near && h.nnz >= 2ull * (unsigned long long)n;
}

// Most entries lie close to the diagonal and few far out, as in a dissection (mean distance
// 0.04 of the band or less; bands and natural grids have 0.2 or more, with one far entry
// per row 0.09).
__host__ __device__ inline bool near_diagonal(const BandCounters& h, const int32_t* band) {
  const int32_t width = band[0] > band[1] ? band[0] : band[1];
  return h.spread < h.nnz * (unsigned long long)width / 16;
}

}  // namespace gsofa
