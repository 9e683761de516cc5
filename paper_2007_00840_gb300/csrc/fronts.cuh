// Nested-dissection path (fronts.cu): level data and launchers.
#pragma once

#include "band.cuh"

namespace gsofa {

constexpr int FRONT_BLOCK_MAX = 1024;  // vertices of a block at most
constexpr int FRONT_BLOCK_MIN = 64;    // smaller closed stretches are left to the next level
constexpr int FRONT_PIECES = 64;       // blocks below one vertex at most
constexpr int FRONT_BC_MAX = 4096;     // columns right of a block at most

struct FrontCounters {
  int32_t nblocks;    // blocks found
  int32_t overflow;   // a capacity ran out: the path is given up
  int32_t br_total;   // rows above blocks, over all blocks
  int32_t bc_total;   // columns right of blocks, over all blocks
  int32_t max_pieces; // most blocks below one vertex so far
  int32_t pad[3];
};

// One level: n vertices (gid: their original numbers, increasing; null: the same), rows
// col[beg[i] .. end[i]), increasing.
struct FrontLevel {
  int32_t n;
  int32_t block_max;   // vertices of a block at most on this level
  int32_t wide;        // rows are long: a warp each, and columns right of blocks by bitmaps
  const int32_t *beg, *end, *col, *gid;
  int32_t* low;        // smallest neighbour in either direction (set to a large value before)
  int32_t* best;       // per start: end of the largest closed stretch of at most block_max (-1: none)
  int32_t* blk;        // per vertex: its block or -1
  int32_t* rem;        // per vertex: 1 where it stays for the next level
  const int64_t* rank; // exclusive sums of rem
  int32_t* bound;      // per vertex: entries its reduced row may have
  const int64_t* room; // exclusive sums of bound
  FrontCounters* ctr;
  int32_t cap;         // capacity in blocks
  int32_t *b_first, *b_size, *b_nr, *b_nb, *b_fill, *b_br, *b_bc;  // per block
  int32_t *br_row, *br_b, *br_e;  // rows above blocks: vertex, entries in the block's columns
  int32_t* bc;         // columns right of blocks
  int32_t* bc_next;    // the same as vertices of the next level
  int32_t bc_cap;
  uint2* right;        // wide: per block and 32 vertices, the columns right of it: bits, number before
  // per original vertex
  int32_t* own;        // block it is eliminated in (over all levels)
  int32_t* own_row;
  int32_t* head;       // newest piece (row above a block), -1: none
  int32_t* npieces;
  int32_t* piece_next; // per piece
  int32_t* piece_blk;
  int32_t* piece_row;
  int32_t* piece_nL;   // entries in the block
  int32_t blocks_before;  // blocks of earlier levels
  int32_t pieces_before;
  int32_t piece_cap, br_cap;
};

// One eliminated block, over all levels.
struct FrontBlock {
  const uint32_t* bits;
  const int32_t* cols;  // original numbers of its vertices
  const int32_t* bcols; // and of the columns right of it
  int32_t level, sz, nb, pivots, W;
  int32_t first;        // its first vertex where they are consecutive, else -1
};

struct FrontEmit {
  int32_t n;
  const FrontBlock* blocks;
  const int32_t *own, *own_row, *head, *piece_next, *piece_blk, *piece_row, *piece_nL;
  int32_t *row_nL, *row_nU, *fill;  // row_nL: of the own row alone before launch_front_count
  const int64_t *L_rowptr, *U_rowptr;
  int32_t *L_colidx, *U_colidx;
  const int32_t* left_gid;          // vertices that the first level leaves, increasing
  int32_t left;
};

cudaError_t launch_front_blocks(const FrontLevel& l, cudaStream_t st);   // low .. rem
cudaError_t launch_front_above(const FrontLevel& l, cudaStream_t st);    // rows above, columns right of the blocks
// Rows of the next level: beg, end, col, gid of its n1 vertices.
cudaError_t launch_front_reduce(const FrontLevel& l, int32_t n1, const FrontMat* fronts, const uint32_t* bits,
                                int32_t* beg, int32_t* end, int32_t* col, int32_t* gid, cudaStream_t st);
cudaError_t launch_front_whole(const FrontLevel& l, cudaStream_t st);    // every vertex into block 0
cudaError_t launch_front_iota(int32_t* out, int32_t n, cudaStream_t st);
// The columns right of blocks as original vertices and as vertices of the next level.
cudaError_t launch_front_gids(const FrontLevel& l, int32_t count, int32_t* out, cudaStream_t st);
cudaError_t launch_front_count(const FrontEmit& e, cudaStream_t st);
cudaError_t launch_front_expand(const FrontEmit& e, cudaStream_t st);
// Vertices of a next level that launch_front_reduce can take.
constexpr int32_t FRONT_REDUCED_MAX = 400000;

}  // namespace gsofa
