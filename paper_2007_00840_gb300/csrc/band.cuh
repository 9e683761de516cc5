// Banded path (band.cu): descriptors and launchers.
#pragma once

#include "internal.cuh"

namespace gsofa {

constexpr int BAND_SMEM_MAX = 227 * 1024;
constexpr int BAND_STAGE = 512;       // column indices of one panel staged ahead (more: read in place)
constexpr int BAND_REACH_MAX = 8192;  // above the widest band that eight CTAs hold

// Counters of one call.
struct BandCounters {
  unsigned long long total_L, total_U;
  unsigned long long nnz, spread;  // one matrix: entries of A, and the sum of their distances from the diagonal
  int32_t err;          // ERR_* bits
  int32_t bad_row;      // INT_MAX - first offending row (0: none)
  int32_t n_super;
  int32_t groups_done;
  int32_t stretch;      // one matrix: panels of its longest stretch between uncrossed boundaries (band_reach_kernel)
};

// What the sampled rows of a matrix reach: sums of the entries and levels of their searches,
// and the longest of them by itself (row_us, rounded up).
struct BandReach {
  unsigned long long entries;
  uint32_t levels, longest;
};

// Words of columns that a band of `reach` columns takes left and right of a row's own word.
// Left at least one: the window is the panels P .. P + LB, and while step P reads panel P + 1
// the loader writes panel P + LB + 1.  With none a batch's chain read panel P + 1 before it
// was there (a single matrix without entries below the diagonal is one stretch per panel).
__host__ __device__ inline int band_words_left(int32_t reach) { return reach > 32 ? (reach + 31) / 32 : 1; }
__host__ __device__ inline int band_words_right(int32_t reach) { return (reach + 31) / 32; }

// One matrix.  LB, UB: band_words_left and band_words_right of its band.
struct BandMat {
  const int32_t* rowptr;
  const int32_t* colidx;
  int64_t row_base;    // first row in the concatenated per-row arrays
  int64_t group_base;  // first row group
  int64_t bits_base;   // first word of its bitmap rows (LB + UB + 1 words each)
  int32_t n, LB, UB, pad;
};

struct BandArgs {
  const BandMat* mats;  // null: one matrix, `one`
  BandMat one;
  int32_t nmats;
  int32_t first;        // elimination: first matrix of this launch
  int64_t rows;         // rows of all matrices
  int64_t groups;       // row groups of all matrices
  int32_t chunk;        // rows per supernode chunk
  int32_t group_rows;   // rows per group: a multiple of chunk
  BandCounters* ctr;
  int32_t* band;        // per matrix: largest i - j, largest j - i
  int32_t* entries;     // per matrix of a batch: entries of A (null: one matrix, in ctr)
  BandReach* reach;     // per matrix
  int32_t sampled;      // matrices whose rows are sampled: the first ones
  int32_t reach_rows;   // rows sampled of each
  int32_t most_rows;    // the largest order among them
  uint32_t* cross;      // one matrix: bit q set where an entry below the diagonal crosses row 32q (null: batch)
  uint32_t* bits;       // null (one matrix): per-row sizes and fill counts only
  int32_t *row_nL, *row_nU, *fill, *flags;
  long long* part;      // per group: [nnz(L), nnz(U), supernodes], then exclusive sums
  unsigned long long* mat_tot;  // per matrix [nnz(L), nnz(U)] (null: one matrix)
  int32_t* mat_nsuper;
  int64_t *L_rowptr, *U_rowptr;
  int32_t *L_colidx, *U_colidx, *super_start;
};

// A front: one block of a nested dissection (fronts.cu).
struct FrontMat {
  int64_t bits_base;     // first word of its rows: (sz rounded up to 32) + nr of them, W words each
  int32_t first_vertex;  // the block is vertices [first_vertex, first_vertex + sz) of its level
  int32_t sz, nr, nb;    // pivots, rows above the block, columns right of it
  int32_t br_base, bc_base;
  int32_t id, pad;       // the block's number on its level
};

struct FrontArgs {
  const FrontMat* fronts;
  int32_t first;
  const int32_t *beg, *end, *col;  // rows of the level: columns col[beg[i] .. end[i])
  const int32_t *br_b, *br_e;      // rows above the blocks: their entries in the block's columns
  const int32_t* bc;               // columns right of the blocks, increasing
  const uint2* right;              // their places (FrontLevel::right), or null: searched in bc
  int32_t right_words;             // words of a block in right
  uint32_t* bits;
  const int32_t* gid;              // vertices of the level: original numbers
  int32_t *row_nL, *row_nU;        // per original vertex: entries of its own row in the block, and from the diagonal on
  int32_t* piece_nL;               // per row above a block: its entries in the block
};

inline size_t front_smem_bytes(int sz, int nr, int nb, int C) {
  const int pivots = (sz + 31) / 32, panels = pivots + (nr + 31) / 32, W = pivots + (nb + 31) / 32;
  const size_t slots = (size_t)(panels + C - 1) / C;
  return 4 * (128 + 64 + 68 + 192 * (size_t)((W - 1) | 1) + slots * 32 * (size_t)((W | 1) + 1));
}
// Clusters of C CTAs for fronts [a.first, a.first + count).
cudaError_t launch_front_elim(const FrontArgs& a, int count, int C, int threads, size_t smem, cudaStream_t st);

__host__ __device__ inline size_t band_smem_bytes(int LB, int UB, int C) {
  const int wx = LB + UB + 1;
  const size_t slots = (size_t)(LB + 2 + C - 1) / C;
  return 4 * (128 + 64 + 68 + 192 * (size_t)(UB | 1) + 4 * BAND_STAGE + slots * 32 * (size_t)((wx | 1) + 1));
}

struct BandShape {
  int C = 0;  // CTAs per matrix (0: the band does not fit on chip)
  int threads = 0;
  size_t smem = 0;
};

// Launch shape for a band of LB words left and UB words right of a row's own.  One matrix
// (alone) is spread over a cluster once its window is wide enough for the split to pay for
// the cluster's barriers (us per 32 rows with 1 / 4 / 8 CTAs: LB 3: 1.6 / 2.3 / 2.4, LB 7:
// 2.3 / 2.2 / 2.4, LB 10: 3.1 / 2.5 / 2.7, LB 33: - / 5.0 / 4.4).  Batches have other
// matrices to fill the chip with and take the smallest cluster that holds the window.
// most: CTAs that one matrix may take (a caller's cap).
__host__ __device__ inline BandShape band_shape(int LB, int UB, bool alone, int most = 8) {
  BandShape s;
  int first = !alone || LB <= 8 ? 1 : (LB <= 16 ? 4 : 8);
  while (first > 1 && first > most) first /= 2;
  for (int C = first; C <= 8 && C <= most; C *= 2) {
    const size_t b = band_smem_bytes(LB, UB, C);
    if (b > BAND_SMEM_MAX - 1024) continue;
    s.C = C;
    s.smem = b;
    break;
  }
  if (!s.C) return s;
  // 14 worker warps: a batch's longest matrix sets its time (512 matrices: 1.28 ms; with 256
  // threads 1.90, with 128 3.99)
  s.threads = 512;
  return s;
}

cudaError_t launch_band_scan(const BandArgs& a, cudaStream_t st);
// After the scan: reach and stretch of the first a.sampled matrices.  counts: for sizes alone.
cudaError_t launch_band_reach(const BandArgs& a, bool counts, cudaStream_t st);
// `count` matrices from a.first on, or the parts one matrix's panels are dealt to: C CTAs (a cluster) each.
cudaError_t launch_band_elim(const BandArgs& a, int count, int C, int threads, size_t smem, cudaStream_t st);
cudaError_t launch_band_count(const BandArgs& a, cudaStream_t st);
cudaError_t launch_band_expand(const BandArgs& a, cudaStream_t st);

}  // namespace gsofa
