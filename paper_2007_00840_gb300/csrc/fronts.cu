// Symbolic LU of patterns in nested-dissection order by elimination of blocks.
//
// A stretch of consecutive vertices that no entry, in either direction, connects to a
// lower vertex outside it is closed: its rows need nothing from outside, and all that the
// rows above take from it passes through the columns right of it that its rows reach.  In
// an ordering by nested dissection every subtree is such a stretch.  So, level by level:
//   1. the largest closed stretches of at most 1,024 vertices are taken as blocks;
//   2. each is eliminated as a dense front of bits on chip (front_elim_kernel): its own
//      vertices as pivots, the rows above that have entries in it, the columns right of
//      it.  L and U of its vertices are finished, and so are the entries of L that the
//      rows above have in it;
//   3. the remaining vertices form the next level, their rows joined with what they reach
//      through the blocks.  A 1M-vertex grid goes 1,048,576 -> 61k -> 14k -> 6k -> 2k,
//      and the rest is one front.
// The traversal walks a separator's whole subdomain for each of its rows (13.2e9 scanned
// entries on that grid); here a subdomain costs its boundary.
//
// A vertex's L row is collected from the blocks below it (its pieces) and its own block.
// Two pieces are never interleaved unless their levels differ, and then the lower one lies
// between two columns of the higher one, so every entry's place is a sum of piece sizes.
#include "fronts.cuh"

namespace gsofa {

namespace {

__device__ __forceinline__ uint32_t gt_bits(int k) { return k >= 31 ? 0u : 0xFFFFFFFEu << k; }
__device__ __forceinline__ uint32_t lt_bits(int k) { return (1u << k) - 1u; }

constexpr int TILE = 1024;

// smallest neighbour of every vertex, over its row and its column; LANES lanes per row
// (eight for rows of A, 32 for the rows of a reduced level, which have hundreds of
// entries: 167 -> 40 us on a level of 6,000 rows)
template <int LANES>
__global__ void front_low_kernel(FrontLevel l) {
  const int sub = threadIdx.x % LANES;
  const int step = (gridDim.x * blockDim.x) / LANES;
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) / LANES; i < l.n; i += step) {
    const int e = l.end[i];
    int lo = i;
#pragma unroll 4
    for (int k = l.beg[i] + sub; k < e; k += LANES) {
      const int c = l.col[k];
      lo = min(lo, c);
      if (c > i && *(volatile int32_t*)(l.low + c) > i) atomicMin(l.low + c, i);
    }
    if (lo < *(volatile int32_t*)(l.low + i)) atomicMin(l.low + i, lo);
  }
}

// Closed stretches: for every vertex i the start R(i) of the smallest closed stretch that
// ends at i, where it has at most block_max vertices: the least fixed point of
// R(i) = min of R over [R(i), i], from the smallest neighbours.  A CTA does a tile of
// vertices and looks at the FRONT_BLOCK_MAX before it (a start further left is too far
// anyway).  Each round answers all range minima from windows of 1, 2, 4, .. vertices, and
// since every vertex uses the others' current starts few rounds are needed (a pass with a
// stack of starts by one thread took 186 us per level, this about 15).
__global__ void __launch_bounds__(1024) front_stretch_kernel(FrontLevel l) {
  constexpr int LEN = TILE + FRONT_BLOCK_MAX;
  static_assert(LEN == 2048 && FRONT_BLOCK_MAX <= 1 << 10, "two vertices per thread, eleven windows");
  __shared__ int16_t win[11][LEN];  // win[k][x]: smallest start over the 2^k vertices that end at x
  const int t0 = blockIdx.x * TILE;
  const int left = max(0, t0 - FRONT_BLOCK_MAX), len = min(l.n, t0 + TILE) - left;
  int v[2];
  for (int q = 0; q < 2; q++) {
    const int x = threadIdx.x + 1024 * q;
    const int lo = x < len ? min(l.low[left + x], left + x) - left : 0;
    v[q] = lo < 0 || x - lo >= l.block_max ? -1 : lo;  // -1: too far left
  }
  for (;;) {
    for (int q = 0; q < 2; q++) win[0][threadIdx.x + 1024 * q] = (int16_t)v[q];
    __syncthreads();
    for (int k = 1; k < 11; k++) {
      for (int q = 0; q < 2; q++) {
        const int x = threadIdx.x + 1024 * q, y = x - (1 << (k - 1));
        const int16_t a = win[k - 1][x];
        win[k][x] = y >= 0 ? min(a, win[k - 1][y]) : a;
      }
      __syncthreads();
    }
    int changed = 0;
    for (int q = 0; q < 2; q++) {
      const int x = threadIdx.x + 1024 * q;
      if (x >= len || v[q] < 0 || v[q] == x) continue;
      const int k = 31 - __clz(x - v[q] + 1);
      int r = min((int)win[k][x], (int)win[k][v[q] + (1 << k) - 1]);
      if (r < 0 || x - r >= l.block_max) r = -1;
      if (r != v[q]) {
        v[q] = r;
        changed = 1;
      }
    }
    if (!__syncthreads_or(changed)) break;
  }
  for (int q = 0; q < 2; q++) {
    const int x = threadIdx.x + 1024 * q;
    if (x < len && left + x >= t0 && v[q] >= 0) atomicMax(l.best + left + v[q], left + x);
  }
}

// Blocks: stretches not inside another.  Every start looks at the ends of the starts
// before it (a running maximum over the tile and FRONT_BLOCK_MAX before it).
__global__ void front_pick_kernel(FrontLevel l) {
  __shared__ int32_t far[TILE + FRONT_BLOCK_MAX];
  __shared__ int32_t part[1024];
  const int t0 = blockIdx.x * TILE;
  const int left = max(0, t0 - FRONT_BLOCK_MAX), right = min(l.n, t0 + TILE);
  const int len = right - left;
  // two elements per thread, then a scan over the threads
  int v[2];
  for (int q = 0; q < 2; q++) {
    const int i = 2 * threadIdx.x + q;
    v[q] = i < len ? l.best[left + i] : -1;
  }
  v[1] = max(v[0], v[1]);
  part[threadIdx.x] = v[1];
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const int x = (int)threadIdx.x >= o ? part[threadIdx.x - o] : -1;
    __syncthreads();
    part[threadIdx.x] = max(part[threadIdx.x], x);
    __syncthreads();
  }
  const int before = threadIdx.x > 0 ? part[threadIdx.x - 1] : -1;
  for (int q = 0; q < 2; q++) {
    const int i = 2 * threadIdx.x + q;
    if (i < len) far[i] = max(before, v[q]);
  }
  __syncthreads();
  for (int i = t0 + threadIdx.x; i < right; i += blockDim.x) {
    const int e = l.best[i];
    if (e - i + 1 < FRONT_BLOCK_MIN) continue;
    if (i > left && far[i - left - 1] >= i) continue;  // inside an earlier one
    const int b = atomicAdd(&l.ctr->nblocks, 1);
    if (b >= l.cap) {
      l.ctr->overflow = 1;
      continue;
    }
    l.b_first[b] = i;
    l.b_size[b] = e - i + 1;
  }
}

__global__ void front_mark_kernel(FrontLevel l) {
  const int nb = min(l.ctr->nblocks, l.cap);
  for (int b = blockIdx.x; b < nb; b += gridDim.x) {
    const int first = l.b_first[b], size = l.b_size[b];
    for (int k = threadIdx.x; k < size; k += blockDim.x) {
      const int v = l.gid ? l.gid[first + k] : first + k;
      l.blk[first + k] = b;
      l.rem[first + k] = 0;
      l.own[v] = l.blocks_before + b;
      l.own_row[v] = k;
    }
  }
}

// First entry at or after k0 whose column is at least c.
__device__ __forceinline__ int lower_entry(const int32_t* col, int k0, int k1, int c) {
  while (k0 < k1) {
    const int mid = (k0 + k1) >> 1;
    if (col[mid] < c) k0 = mid + 1; else k1 = mid;
  }
  return k0;
}

// Rows of remaining vertices: their entries in one block are consecutive (blocks are
// stretches).  FILL false: blocks' row counts, and the entries outside blocks; true: the
// rows into their blocks' lists, and onto their vertices' piece lists.
template <bool FILL, int LANES>
__global__ void front_runs_kernel(FrontLevel l) {
  const int sub = threadIdx.x % LANES;
  const int step = (gridDim.x * blockDim.x) / LANES;
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) / LANES; i < l.n; i += step) {
    if (l.blk[i] >= 0) continue;
    const int b0 = l.beg[i], e0 = l.end[i];
    int outside = 0, runs = 0;
#pragma unroll 2
    for (int k = b0 + sub; k < e0; k += LANES) {
      const int c = l.col[k];
      const int b = l.blk[c];
      if (b < 0) {
        outside++;
        continue;
      }
      if (k > b0 && l.blk[l.col[k - 1]] == b) continue;  // not the first of its run
      runs++;
      if (!FILL) {
        atomicAdd(l.b_nr + b, 1);
      } else {
        const int at = l.b_br[b] + atomicAdd(l.b_fill + b, 1);
        const int row = at - l.b_br[b];
        const int v = l.gid ? l.gid[i] : i;
        const int piece = l.pieces_before + at;
        if (at >= l.br_cap || piece >= l.piece_cap) {
          l.ctr->overflow = 1;
          continue;
        }
        l.br_row[at] = i;
        l.br_b[at] = k;
        l.br_e[at] = lower_entry(l.col, k, e0, l.b_first[b] + l.b_size[b]);
        l.piece_blk[piece] = l.blocks_before + b;
        l.piece_row[piece] = (l.b_size[b] + 31) / 32 * 32 + row;
        l.piece_next[piece] = atomicExch(l.head + v, piece);
        const int np = atomicAdd(l.npieces + v, 1) + 1;
        if (np > *(volatile int32_t*)&l.ctr->max_pieces) atomicMax(&l.ctr->max_pieces, np);
      }
    }
    if (!FILL && outside) atomicAdd(l.bound + i, outside);
  }
}

// Offsets of the blocks' row lists (one CTA).
__global__ void front_offsets_kernel(FrontLevel l) {
  __shared__ int32_t sh[32];
  __shared__ int32_t s_carry;
  const int nb = min(l.ctr->nblocks, l.cap);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_carry = 0;
  __syncthreads();
  for (int b0 = 0; b0 < nb; b0 += blockDim.x) {
    const int b = b0 + threadIdx.x;
    const int v = b < nb ? l.b_nr[b] : 0;
    int s = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(FULL, s, o);
      if (lane >= o) s += x;
    }
    if (lane == 31) sh[warp] = s;
    __syncthreads();
    int before = s_carry, all = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); k++) {
      if (k < warp) before += sh[k];
      all += sh[k];
    }
    if (b < nb) l.b_br[b] = before + s - v;
    __syncthreads();
    if (threadIdx.x == 0) s_carry += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) l.ctr->br_total = s_carry;
}

// The distinct columns right of every block, increasing: a hash set, then a sort, in
// shared memory.
__global__ void front_right_kernel(FrontLevel l) {
  constexpr int H = 2 * FRONT_BC_MAX;
  __shared__ int32_t key[H];
  __shared__ int32_t s_count, s_at;
  const int nb = min(l.ctr->nblocks, l.cap);
  for (int b = blockIdx.x; b < nb; b += gridDim.x) {
    const int first = l.b_first[b], size = l.b_size[b];
    for (int i = threadIdx.x; i < H; i += blockDim.x) key[i] = -1;
    if (threadIdx.x == 0) s_count = 0;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int r = warp; r < size; r += nw) {
      // entries right of the block are the last of the row
      const int e = l.end[first + r];
      const int k0 = lower_entry(l.col, l.beg[first + r], e, first + size);
      for (int k = k0 + lane; k < e; k += 32) {
        const int c = l.col[k];
        uint32_t h = ((uint32_t)c * 0x9E3779B1u) >> 19;  // 13 bits
        while (*(volatile int32_t*)&s_count <= FRONT_BC_MAX) {  // a fuller set is given up
          const int old = atomicCAS(&key[h & (H - 1)], -1, c);
          if (old == -1) atomicAdd(&s_count, 1);
          if (old == -1 || old == c) break;
          h++;
        }
      }
    }
    __syncthreads();
    const int count = s_count;
    __syncthreads();
    if (count > FRONT_BC_MAX) {
      if (threadIdx.x == 0) {
        l.ctr->overflow = 1;
        l.b_nb[b] = 0;
        l.b_bc[b] = 0;
      }
      __syncthreads();
      continue;
    }
    // empty places last, then sort the next power of two that holds the set: places are
    // compacted first (set order is free)
    if (threadIdx.x == 0) s_at = 0;
    __syncthreads();
    int mine[H / 512];
    int n = 0;
    for (int i = threadIdx.x; i < H; i += blockDim.x)
      if (key[i] >= 0) mine[n++] = key[i];
    __syncthreads();
    for (int i = threadIdx.x; i < H; i += blockDim.x) key[i] = 0x7FFFFFFF;
    const int at = n ? atomicAdd(&s_at, n) : 0;
    __syncthreads();
    for (int q = 0; q < n; q++) key[at + q] = mine[q];
    int p2 = 1;
    while (p2 < count) p2 <<= 1;
    __syncthreads();
    for (int k = 2; k <= p2; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int i = threadIdx.x; i < p2; i += blockDim.x) {
          const int x = i ^ j;
          if (x > i) {
            const int a = key[i], c = key[x];
            if ((a > c) == ((i & k) == 0)) {
              key[i] = c;
              key[x] = a;
            }
          }
        }
        __syncthreads();
      }
    if (threadIdx.x == 0) {
      s_at = atomicAdd(&l.ctr->bc_total, count);
      if (s_at + count > l.bc_cap) l.ctr->overflow = 1;
      l.b_nb[b] = count;
      l.b_bc[b] = s_at;
    }
    __syncthreads();
    const int base = s_at;
    if (base + count <= l.bc_cap)
      for (int i = threadIdx.x; i < count; i += blockDim.x) l.bc[base + i] = key[i];
    __syncthreads();
  }
}

// The same on a level of long rows: every block's bitmap over the level's vertices, a warp
// per row of the block (one CTA per block hashing half a million entries took 1,356 us on
// a level of 16 blocks) ...
__global__ void front_right_set_kernel(FrontLevel l) {
  const int lane = threadIdx.x & 31;
  const int step = (gridDim.x * blockDim.x) >> 5;
  const int words = (l.n + 31) >> 5;
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < l.n; i += step) {
    const int b = l.blk[i];
    if (b < 0) continue;
    uint2* right = l.right + (size_t)b * words;
    const int e = l.end[i];
    const int k0 = lower_entry(l.col, l.beg[i], e, l.b_first[b] + l.b_size[b]);
#pragma unroll 4
    for (int k = k0 + lane; k < e; k += 32) {
      const int c = l.col[k];
      const uint32_t bit = 1u << (c & 31);
      if (!(*(volatile uint32_t*)&right[c >> 5].x & bit)) atomicOr(&right[c >> 5].x, bit);
    }
  }
}

// ... then the numbers before each word, and the columns.
__global__ void front_right_list_kernel(FrontLevel l) {
  __shared__ int32_t sh[32];
  __shared__ int32_t s_carry, s_at;
  const int nb = min(l.ctr->nblocks, l.cap);
  const int words = (l.n + 31) >> 5;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int b = blockIdx.x; b < nb; b += gridDim.x) {
    uint2* right = l.right + (size_t)b * words;
    __syncthreads();
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int w0 = 0; w0 < words; w0 += blockDim.x) {
      const int w = w0 + threadIdx.x;
      const int v = w < words ? __popc(right[w].x) : 0;
      int s = v;
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(FULL, s, o);
        if (lane >= o) s += x;
      }
      if (lane == 31) sh[warp] = s;
      __syncthreads();
      int before = s_carry, all = 0;
      for (int k = 0; k < nw; k++) {
        if (k < warp) before += sh[k];
        all += sh[k];
      }
      if (w < words) right[w].y = (uint32_t)(before + s - v);
      __syncthreads();
      if (threadIdx.x == 0) s_carry += all;
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      const int count = s_carry;
      s_at = atomicAdd(&l.ctr->bc_total, count);
      if (s_at + count > l.bc_cap) l.ctr->overflow = 1;
      l.b_nb[b] = count;
      l.b_bc[b] = s_at;
    }
    __syncthreads();
    if (s_at + s_carry <= l.bc_cap)
      for (int w = threadIdx.x; w < words; w += blockDim.x) {
        int at = s_at + (int)right[w].y;
        for (uint32_t m = right[w].x; m; m &= m - 1) l.bc[at++] = 32 * w + __ffs(m) - 1;
      }
  }
}

// Entries a reduced row may have: those outside blocks (counted) and all columns right of
// the blocks below it.
__global__ void front_bound_kernel(FrontLevel l) {
  if (l.ctr->overflow) return;
  for (int at = blockIdx.x * blockDim.x + threadIdx.x; at < l.ctr->br_total; at += gridDim.x * blockDim.x) {
    const int b = l.piece_blk[l.pieces_before + at] - l.blocks_before;
    atomicAdd(l.bound + l.br_row[at], l.b_nb[b]);
  }
}

// Rows of the next level, one warp each: a bitmap of its vertices in shared memory takes
// the entries outside blocks and what the row reaches through the blocks below it.
__global__ void front_reduce_kernel(FrontLevel l, int32_t n1, const FrontMat* fronts, const uint32_t* bits,
                                    int32_t* beg1, int32_t* end1, int32_t* col1, int32_t* gid1) {
  extern __shared__ uint32_t sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int words = (n1 + 31) >> 5, swords = (words + 31) >> 5;
  uint32_t* set = sm + (size_t)warp * (words + swords);
  uint32_t* sum = set + words;  // one bit per nonzero word
  for (int w = lane; w < words + swords; w += 32) set[w] = 0u;
  __syncwarp();
  auto put = [&](int x) {
    const uint32_t bit = 1u << (x & 31);
    const uint32_t old = atomicOr(set + (x >> 5), bit);
    if (old == 0u) atomicOr(sum + (x >> 10), 1u << ((x >> 5) & 31));
  };
  for (int i = blockIdx.x * nw + warp; i < l.n; i += gridDim.x * nw) {
    if (l.blk[i] >= 0) continue;
    const int v = l.gid ? l.gid[i] : i;
    const int e = l.end[i];
    for (int k = l.beg[i] + lane; k < e; k += 32) {
      const int c = l.col[k];
      if (l.blk[c] < 0) put((int)l.rank[c]);
    }
    // this level's pieces are the newest on the vertex's list
    for (int p = l.head[v]; p >= l.pieces_before; p = l.piece_next[p]) {
      const FrontMat f = fronts[l.piece_blk[p] - l.blocks_before];
      const int pivots = (f.sz + 31) >> 5, W = pivots + ((f.nb + 31) >> 5);
      const uint32_t* row = bits + f.bits_base + (size_t)l.piece_row[p] * W + pivots;
      for (int w = lane; w < W - pivots; w += 32) {
        for (uint32_t m = row[w]; m; m &= m - 1) {
          put((int)l.rank[l.bc[f.bc_base + 32 * w + __ffs(m) - 1]]);
        }
      }
    }
    __syncwarp();
    const int to = (int)l.rank[i];
    int at = (int)l.room[i];
    if (lane == 0) {
      beg1[to] = at;
      gid1[to] = v;
    }
    for (int sw = 0; sw < swords; sw++) {
      const uint32_t some = sum[sw];
      if (!some) continue;
      const int w = 32 * sw + lane;
      uint32_t m = (some >> lane) & 1u ? set[w] : 0u;
      if (m) set[w] = 0u;
      const int cnt = __popc(m);
      int s = cnt;
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(FULL, s, o);
        if (lane >= o) s += x;
      }
      int to_at = at + s - cnt;
      for (; m; m &= m - 1) col1[to_at++] = 32 * w + __ffs(m) - 1;
      at += __shfl_sync(FULL, s, 31);
    }
    if (lane == 0) end1[to] = at;
    __syncwarp();
    for (int sw = lane; sw < swords; sw += 32) sum[sw] = 0u;
    __syncwarp();
  }
}

__global__ void front_whole_kernel(FrontLevel l) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < l.n; i += gridDim.x * blockDim.x) {
    const int v = l.gid ? l.gid[i] : i;
    l.own[v] = l.blocks_before;
    l.own_row[v] = i;
  }
}

__global__ void front_iota_kernel(int32_t* out, int32_t n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = i;
}

__global__ void front_gids_kernel(const int32_t* gid, const int32_t* cols, int32_t count, int32_t* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
    out[i] = gid ? gid[cols[i]] : cols[i];
}

// ------------------------------------------------------------ rows of the result
// One warp per vertex: sizes.
__global__ void front_count_kernel(FrontEmit e) {
  const int lane = threadIdx.x & 31;
  const int step = (gridDim.x * blockDim.x) >> 5;
  for (int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < e.n; v += step) {
    const FrontBlock b = e.blocks[e.own[v]];
    const int r = e.own_row[v];
    const uint32_t* row = b.bits + (size_t)r * b.W;
    int nl = 0, nu = 0;
    for (int w = lane; w < b.W; w += 32) {
      const uint32_t m = row[w];
      if (w < r >> 5) nl += __popc(m);
      else if (w > r >> 5) nu += __popc(m);
      else {
        nl += __popc(m & lt_bits(r & 31));
        nu += __popc(m & gt_bits(r & 31));
      }
    }
    for (int p = e.head[v]; p >= 0; p = e.piece_next[p]) {
      const FrontBlock q = e.blocks[e.piece_blk[p]];
      const uint32_t* x = q.bits + (size_t)e.piece_row[p] * q.W;
      for (int w = lane; w < q.pivots; w += 32) nl += __popc(x[w]);
    }
    nl = __reduce_add_sync(FULL, nl);
    nu = __reduce_add_sync(FULL, nu) + 1;
    if (lane == 0) {
      e.row_nL[v] = nl;
      e.row_nU[v] = nu;
      e.fill[v] = nl + nu - e.fill[v];
    }
  }
}

// One warp per vertex: columns.  L(v,:) comes from the vertex's pieces and the lower part
// of its own row (the last piece).  An entry's place is its rank in its piece plus the
// sizes of the pieces before it: of pieces of its level or below, those that end before
// it; of pieces above, their entries before its block.
__global__ void __launch_bounds__(256) front_expand_kernel(FrontEmit e) {
  struct Piece {
    const uint32_t* row;
    const int32_t* cols;
    int words, size, level, first, last, count;
    uint32_t mask;  // of the last word
  };
  __shared__ Piece s_piece[8][FRONT_PIECES + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  Piece* pc = s_piece[warp];
  const int step = (gridDim.x * blockDim.x) >> 5;
  for (int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < e.n; v += step) {
    const FrontBlock b = e.blocks[e.own[v]];
    const int r = e.own_row[v];
    const uint32_t* row = b.bits + (size_t)r * b.W;
    // U: the diagonal, the block's columns above v, the columns right of the block
    int32_t* U = e.U_colidx + e.U_rowptr[v];
    if (lane == 0) U[0] = v;
    U++;
    for (int w0 = r >> 5; w0 < b.W; w0 += 32) {
      uint32_t mine = w0 + lane < b.W ? row[w0 + lane] : 0u;
      if (w0 + lane == r >> 5) mine &= gt_bits(r & 31);
      unsigned any = __ballot_sync(FULL, mine != 0u);
      while (any) {
        const int k = __ffs(any) - 1;
        any &= any - 1;
        const uint32_t m = __shfl_sync(FULL, mine, k);
        const int w = w0 + k;
        if ((m >> lane) & 1u)
          U[__popc(m & lt_bits(lane))] = w < b.pivots ? b.cols[32 * w + lane] : b.bcols[32 * (w - b.pivots) + lane];
        U += __popc(m);
      }
    }
    // the pieces of L
    int np = 0;
    for (int p = e.head[v]; p >= 0; p = e.piece_next[p]) {
      if (lane == 0) {
        const FrontBlock q = e.blocks[e.piece_blk[p]];
        pc[np] = Piece{q.bits + (size_t)e.piece_row[p] * q.W, q.cols, q.pivots, q.sz, q.level, q.cols[0], q.cols[q.sz - 1], 0, FULL};
      }
      np++;
    }
    if (lane == 0) pc[np] = Piece{row, b.cols, (r >> 5) + 1, r, b.level, b.cols[0], v - 1, 0, lt_bits(r & 31)};
    np++;
    __syncwarp();
    for (int p = 0; p < np; p++) {
      int c = 0;
      for (int w = lane; w < pc[p].words; w += 32) {
        uint32_t m = pc[p].row[w];
        if (w == pc[p].words - 1) m &= pc[p].mask;
        c += __popc(m);
      }
      c = __reduce_add_sync(FULL, c);
      if (lane == 0) pc[p].count = c;
    }
    __syncwarp();
    int32_t* L = e.L_colidx + e.L_rowptr[v];
    for (int p = 0; p < np; p++) {
      const Piece me = pc[p];
      if (me.count == 0) continue;
      // entries before this piece's block in pieces of its level or above
      int base = 0;
      bool lower = false;
      for (int q = 0; q < np; q++) {
        if (q == p || pc[q].count == 0) continue;
        if (pc[q].level < me.level) {
          lower = true;
        } else if (pc[q].level == me.level) {
          if (pc[q].last < me.first) base += pc[q].count;
        } else {
          // columns of q below me.first: its first `lo`
          int lo = 0, hi = pc[q].size;
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (pc[q].cols[mid] < me.first) lo = mid + 1; else hi = mid;
          }
          int c = 0;
          for (int w = lane; w < pc[q].words && 32 * w < lo; w += 32) {
            uint32_t m = pc[q].row[w];
            if (w == pc[q].words - 1) m &= pc[q].mask;
            if (lo - 32 * w < 32) m &= lt_bits(lo - 32 * w);
            c += __popc(m);
          }
          base += __reduce_add_sync(FULL, c);
        }
      }
      for (int w0 = 0; w0 < me.words; w0 += 32) {
        uint32_t mine = w0 + lane < me.words ? me.row[w0 + lane] : 0u;
        if (w0 + lane == me.words - 1) mine &= me.mask;
        unsigned any = __ballot_sync(FULL, mine != 0u);
        while (any) {
          const int k = __ffs(any) - 1;
          any &= any - 1;
          const uint32_t m = __shfl_sync(FULL, mine, k);
          if ((m >> lane) & 1u) {
            const int c = me.cols[32 * (w0 + k) + lane];
            int at = base + __popc(m & lt_bits(lane));
            if (lower)
              for (int q = 0; q < np; q++)
                if (pc[q].level < me.level && pc[q].last < c) at += pc[q].count;
            L[at] = c;
          }
          base += __popc(m);
        }
      }
    }
    __syncwarp();
  }
}

int grid_for(long long threads, int block, int most) {
  long long g = (threads + block - 1) / block;
  if (g > most) g = most;
  return g < 1 ? 1 : (int)g;
}

}  // namespace

cudaError_t launch_front_blocks(const FrontLevel& l, cudaStream_t st) {
  if (l.wide) front_low_kernel<32><<<grid_for(32LL * l.n, 256, 8192), 256, 0, st>>>(l);
  else front_low_kernel<8><<<grid_for(8LL * l.n, 256, 8192), 256, 0, st>>>(l);
  const int tiles = (l.n + TILE - 1) / TILE;
  front_stretch_kernel<<<tiles, 1024, 0, st>>>(l);
  front_pick_kernel<<<tiles, 1024, 0, st>>>(l);
  front_mark_kernel<<<grid_for(l.cap, 1, 4096), 256, 0, st>>>(l);
  return cudaGetLastError();
}

cudaError_t launch_front_above(const FrontLevel& l, cudaStream_t st) {
  const int g8 = grid_for(8LL * l.n, 256, 8192), g32 = grid_for(32LL * l.n, 256, 8192);
  if (l.wide) front_runs_kernel<false, 32><<<g32, 256, 0, st>>>(l);
  else front_runs_kernel<false, 8><<<g8, 256, 0, st>>>(l);
  front_offsets_kernel<<<1, 1024, 0, st>>>(l);
  if (l.wide) front_runs_kernel<true, 32><<<g32, 256, 0, st>>>(l);
  else front_runs_kernel<true, 8><<<g8, 256, 0, st>>>(l);
  if (l.wide) {
    front_right_set_kernel<<<g32, 256, 0, st>>>(l);
    front_right_list_kernel<<<grid_for(l.cap, 1, 2048), 512, 0, st>>>(l);
  } else {
    front_right_kernel<<<grid_for(l.cap, 1, 2048), 512, 0, st>>>(l);
  }
  front_bound_kernel<<<grid_for(l.n, 256, 1024), 256, 0, st>>>(l);
  return cudaGetLastError();
}

cudaError_t launch_front_reduce(const FrontLevel& l, int32_t n1, const FrontMat* fronts, const uint32_t* bits,
                                int32_t* beg, int32_t* end, int32_t* col, int32_t* gid, cudaStream_t st) {
  const size_t per = 4 * ((size_t)((n1 + 31) / 32) + (size_t)((n1 + 1023) / 1024));
  int nw = 16;
  while (nw > 1 && per * nw > 96 * 1024) nw >>= 1;
  const cudaError_t e =
      cudaFuncSetAttribute(front_reduce_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BAND_SMEM_MAX);
  if (e != cudaSuccess) return e;
  front_reduce_kernel<<<grid_for(l.n, nw, 4096), 32 * nw, per * nw, st>>>(l, n1, fronts, bits, beg, end, col, gid);
  return cudaGetLastError();
}

cudaError_t launch_front_whole(const FrontLevel& l, cudaStream_t st) {
  front_whole_kernel<<<grid_for(l.n, 256, 1024), 256, 0, st>>>(l);
  return cudaGetLastError();
}

cudaError_t launch_front_iota(int32_t* out, int32_t n, cudaStream_t st) {
  front_iota_kernel<<<grid_for(n, 256, 1024), 256, 0, st>>>(out, n);
  return cudaGetLastError();
}

cudaError_t launch_front_gids(const FrontLevel& l, const int32_t* cols, int32_t count, int32_t* out, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  front_gids_kernel<<<grid_for(count, 256, 1024), 256, 0, st>>>(l.gid, cols, count, out);
  return cudaGetLastError();
}

cudaError_t launch_front_count(const FrontEmit& e, cudaStream_t st) {
  front_count_kernel<<<grid_for(32LL * e.n, 256, 16384), 256, 0, st>>>(e);
  return cudaGetLastError();
}

cudaError_t launch_front_expand(const FrontEmit& e, cudaStream_t st) {
  front_expand_kernel<<<grid_for(32LL * e.n, 256, 16384), 256, 0, st>>>(e);
  return cudaGetLastError();
}

}  // namespace gsofa
