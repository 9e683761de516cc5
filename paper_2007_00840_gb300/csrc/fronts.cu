// Symbolic LU of patterns in nested-dissection order by elimination of blocks.
//
// A stretch of consecutive vertices that no entry, in either direction, connects to a
// lower vertex outside it is closed: its rows need nothing from outside, and all that the
// rows above take from it passes through the columns right of it that its rows reach.  In
// an ordering by nested dissection every subtree is such a stretch.  So, level by level:
//   1. the largest closed stretches of at most 512 vertices (1,024 on later levels) are
//      taken as blocks;
//   2. each is eliminated as a dense front of bits on chip (front_elim_kernel): its own
//      vertices as pivots, the rows above that have entries in it, the columns right of
//      it.  L and U of its vertices are finished, and so are the entries of L that the
//      rows above have in it;
//   3. the remaining vertices form the next level, their rows joined with what they reach
//      through the blocks.  A 1M-vertex grid goes 1,048,576 -> 94k -> 22k -> 6k, and the
//      last 2.9k at most are one front.
// The traversal walks a separator's whole subdomain for each of its rows (13.2e9 scanned
// entries on that grid); here a subdomain costs its boundary.  Whole call on 1024 x 1024
// (512 x 512) vertices: 79.6 -> 5.2 ms (20.9 -> 1.8).  Elimination takes 2.3 ms of it, bound
// by the chain of panels in each front; the rest are chains of dependent loads over the
// levels' rows, about 90 launches.
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

// Calls put(column, rank) for the bits of 32 words, lane's word w0 + lane, and returns
// their number: a lane per word and its bits in turn, or a lane per bit and the words in
// turn, whichever has fewer turns.  (Four turns together are slower: 103 against 80 us for
// the rows of a 512 x 512 grid, by the instructions for turns that are not there.)
// AUX: also passes the word's aux.
template <bool AUX = false, class F>
__device__ __forceinline__ int each_bit(uint32_t mine, int w0, F put, int aux = 0) {
  const int lane = threadIdx.x & 31;
  unsigned any = __ballot_sync(FULL, mine != 0u);
  if (!any) return 0;
  const int cnt = __popc(mine);
  if (__reduce_max_sync(FULL, cnt) < __popc(any)) {
    int s = cnt;
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(FULL, s, o);
      if (lane >= o) s += x;
    }
    int at = s - cnt;
    for (uint32_t m = mine; m; m &= m - 1) put(32 * (w0 + lane) + __ffs(m) - 1, at++, aux);
    return __shfl_sync(FULL, s, 31);
  }
  int before = 0;
  while (any) {
    const int k = __ffs(any) - 1;
    any &= any - 1;
    const uint32_t m = __shfl_sync(FULL, mine, k);
    const int of = AUX ? __shfl_sync(FULL, aux, k) : 0;
    if ((m >> lane) & 1u) put(32 * (w0 + k) + lane, before + __popc(m & lt_bits(lane)), of);
    before += __popc(m);
  }
  return before;
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
  const int step = gridDim.x * nw;
  unsigned todo = 0u;
  for (int i0 = blockIdx.x * nw + warp, base = i0;;) {
    if (!todo) {  // the next of this warp's vertices that remain
      if (i0 >= l.n) break;
      base = i0;
      const long long mine = (long long)i0 + (long long)lane * step;
      todo = __ballot_sync(FULL, mine < l.n && l.blk[mine] < 0);
      i0 = (int)min((long long)l.n, (long long)i0 + 32LL * step);
      continue;
    }
    const int i = base + (__ffs(todo) - 1) * step;
    todo &= todo - 1;
    const int v = l.gid ? l.gid[i] : i;
    const int e = l.end[i];
#pragma unroll 4
    for (int k = l.beg[i] + lane; k < e; k += 32) {
      const int c = l.col[k];
      if (l.blk[c] < 0) put((int)l.rank[c]);
    }
    // this level's pieces are the newest on the vertex's list: a lane looks up each, then
    // all lanes take its words.  A word's columns mostly follow one another on the next
    // level too and go over as two words; the others column by column, four words in flight
    // (all columns so, one after the other: 891 us on a level of 1M vertices, 47,000 left)
    int p = l.head[v];
    while (p >= l.pieces_before) {
      int np = 0, id = -1;
      for (; p >= l.pieces_before && np < 32; np++) {
        if (lane == np) id = p;
        p = l.piece_next[p];
      }
      const uint32_t* row = nullptr;
      int nw_right = 0, bc0 = 0;
      if (id >= 0) {
        const FrontMat f = fronts[l.piece_blk[id] - l.blocks_before];
        const int pivots = (f.sz + 31) >> 5;
        nw_right = (f.nb + 31) >> 5;
        row = bits + f.bits_base + (size_t)l.piece_row[id] * (pivots + nw_right) + pivots;
        bc0 = f.bc_base;
      }
      for (int q = 0; q < np; q++) {
        const uint32_t* x = (const uint32_t*)__shfl_sync(FULL, (unsigned long long)row, q);
        const int nx = __shfl_sync(FULL, nw_right, q);
        const int32_t* to = l.bc_next + __shfl_sync(FULL, bc0, q);
        for (int w0 = 0; w0 < nx; w0 += 32) {
          uint32_t mine = w0 + lane < nx ? x[w0 + lane] : 0u;
          if (mine) {
            const int32_t* t = to + 32 * (w0 + lane);
            const int lo = __ffs(mine) - 1, hi = 31 - __clz(mine);
            const int c = t[lo];
            if (t[hi] - c == hi - lo) {
              const uint32_t m = mine >> lo, m1 = (c & 31) ? m >> (32 - (c & 31)) : 0u;
              atomicOr(set + (c >> 5), m << (c & 31));
              atomicOr(sum + (c >> 10), 1u << ((c >> 5) & 31));
              if (m1) {
                atomicOr(set + (c >> 5) + 1, m1);
                atomicOr(sum + ((c >> 5) + 1 >> 5), 1u << (((c >> 5) + 1) & 31));
              }
              mine = 0u;
            }
          }
          unsigned any = __ballot_sync(FULL, mine != 0u);
          while (any) {
            int at[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
              at[j] = -1;
              if (any) {
                const int w = __ffs(any) - 1;
                any &= any - 1;
                if ((__shfl_sync(FULL, mine, w) >> lane) & 1u) at[j] = to[32 * (w0 + w) + lane];
              }
            }
#pragma unroll
            for (int j = 0; j < 4; j++)
              if (at[j] >= 0) put(at[j]);
          }
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
      at += each_bit(m, 32 * sw, [&](int c, int k, int) { col1[at + k] = c; });
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

__global__ void front_gids_kernel(FrontLevel l, int32_t count, int32_t* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const int c = l.bc[i];
    out[i] = l.gid ? l.gid[c] : c;
    l.bc_next[i] = (int)l.rank[c];
  }
}

// ------------------------------------------------------------ rows of the result
// Row sizes: the own row of a vertex and its pieces, counted where they were written.
__global__ void front_count_kernel(FrontEmit e) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < e.n; v += gridDim.x * blockDim.x) {
    int nl = e.row_nL[v];
    for (int p = e.head[v]; p >= 0; p = e.piece_next[p]) nl += e.piece_nL[p];
    e.row_nL[v] = nl;
    e.fill[v] = nl + e.row_nU[v] - e.fill[v];
  }
}

// Column c of a block's bitmap rows.  The blocks of the first level are consecutive vertices.
__device__ __forceinline__ int block_column(const FrontBlock& b, int c) {
  if (c >= 32 * b.pivots) return __ldg(b.bcols + c - 32 * b.pivots);
  return b.first >= 0 ? b.first + c : __ldg(b.cols + c);
}

// Columns of the rows without pieces, by far the most: one bitmap row holds L, the diagonal
// and U as they stand.  A warp looks EXPAND_ROWS of them up together.
constexpr int EXPAND_ROWS = 8;
__global__ void __launch_bounds__(256) front_expand_kernel(FrontEmit e) {
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int v0 = gw * EXPAND_ROWS; v0 < e.n; v0 += nwarps * EXPAND_ROWS) {
    const int many = min(EXPAND_ROWS, e.n - v0);
    int my_blk = 0, my_row = 0, my_nl = 0;
    long long my_L = 0, my_U = 0;
    bool mine_too = false;
    if (lane < many) {
      mine_too = e.head[v0 + lane] < 0;
      my_blk = e.own[v0 + lane];
      my_row = e.own_row[v0 + lane];
      my_nl = e.row_nL[v0 + lane];
      my_L = e.L_rowptr[v0 + lane];
      my_U = e.U_rowptr[v0 + lane];
    }
    for (unsigned todo = __ballot_sync(FULL, mine_too); todo; todo &= todo - 1) {
      const int j = __ffs(todo) - 1;
      const FrontBlock b = e.blocks[__shfl_sync(FULL, my_blk, j)];
      const int r = __shfl_sync(FULL, my_row, j), nl = __shfl_sync(FULL, my_nl, j);
      const uint32_t* row = b.bits + (size_t)r * b.W;
      int32_t* L = e.L_colidx + __shfl_sync(FULL, my_L, j);
      int32_t* U = e.U_colidx + __shfl_sync(FULL, my_U, j) + 1;
      if (lane == 0) U[-1] = v0 + j;
      int before = 0;
      for (int w0 = 0; w0 < b.W; w0 += 32) {
        uint32_t mine = w0 + lane < b.W ? row[w0 + lane] : 0u;
        if (w0 + lane == r >> 5) mine &= ~(1u << (r & 31));
        before += each_bit(mine, w0, [&](int c, int at, int) {
          const int x = block_column(b, c);
          at += before;
          if (at < nl) L[at] = x;
          else U[at - nl] = x;
        });
      }
    }
  }
}

// Columns of the rows with pieces, a CTA each.  L(v,:) comes from the vertex's pieces and
// the lower part of its own row (the last piece).  An entry's place is its rank in its piece
// plus the sizes of the pieces before it: of pieces of its level or below, those that end
// before it; of pieces above, their entries before its block.  Only vertices that the first
// level leaves have pieces; a CTA takes one, the last separators', which are longest, first.
// (One warp per vertex: 247 us on a 512 x 512 grid; CTAs that look for their vertices among
// all: 144 to 190.)
constexpr int MERGE_PAIRS = 512;
__global__ void __launch_bounds__(64) front_merge_kernel(FrontEmit e) {
  struct Piece {
    const uint32_t* row;
    const int32_t* cols;
    int words, size, level, first, last, count, base, order;
    uint32_t mask;  // of the last word
  };
  __shared__ Piece pc[FRONT_PIECES + 1];
  __shared__ int sorted[FRONT_PIECES + 1], s_sum[2][FRONT_PIECES + 2], s_np, s_pairs;
  __shared__ uint16_t pair[MERGE_PAIRS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* sum = s_sum[warp];
  for (int i = blockIdx.x; i < e.left; i += gridDim.x) {
    const int v = e.left_gid[e.left - 1 - i];
    if (e.head[v] < 0) continue;
    const FrontBlock b = e.blocks[e.own[v]];
    const int r = e.own_row[v], nl = e.row_nL[v];
    const uint32_t* row = b.bits + (size_t)r * b.W;
    int32_t* L = e.L_colidx + e.L_rowptr[v];
    int32_t* U = e.U_colidx + e.U_rowptr[v];
    if (warp == 0) {
      int np = 0, count = 0;
      for (int p = e.head[v]; p >= 0;) {  // a lane looks up each piece
        int id = -1, some = 0;
        for (; p >= 0 && some < 32; some++) {
          if (lane == some) id = p;
          p = e.piece_next[p];
        }
        if (id >= 0) {
          const FrontBlock q = e.blocks[e.piece_blk[id]];
          const int nq = e.piece_nL[id];
          pc[np + lane] = Piece{q.bits + (size_t)e.piece_row[id] * q.W, q.cols, q.pivots, q.sz, q.level, q.cols[0],
                                q.cols[q.sz - 1], nq, 0, 0, FULL};
          count += nq;
        }
        np += some;
      }
      const int own = nl - __reduce_add_sync(FULL, count);
      if (lane == 0) {
        pc[np] = Piece{row, b.cols, (r >> 5) + 1, r, b.level, b.cols[0], v - 1, own, 0, 0, lt_bits(r & 31)};
        s_np = np + 1;
        s_pairs = 0;
        U[0] = v;
      }
    }
    __syncthreads();
    const int np = s_np;
    // a pair of pieces per thread: their order by last column, and the entries before a piece's
    // block in pieces of its level or above.  Those that need a search are few and collected
    // first (with a search wherever a pair comes up, rows of 60 pieces took 100 us)
    auto before_block = [&](int p, int q) {
      const int first = pc[p].first;
      const int32_t* cols = pc[q].cols;
      int lo = 0, hi = pc[q].size;  // columns of q below first: its first lo
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(cols + mid) < first) lo = mid + 1; else hi = mid;
      }
      const uint32_t* words = pc[q].row;
      const int last = pc[q].words - 1;
      int c = 0;
#pragma unroll 8
      for (int w = 0; w < lo >> 5; w++) c += __popc(__ldg(words + w) & (w == last ? pc[q].mask : FULL));
      if (lo & 31) c += __popc(words[lo >> 5] & lt_bits(lo & 31) & (lo >> 5 == last ? pc[q].mask : FULL));
      if (c) atomicAdd(&pc[p].base, c);
    };
    for (int x = threadIdx.x; x < np * np; x += blockDim.x) {
      const int p = x / np, q = x - p * np;
      if (p == q) continue;
      if (pc[q].last < pc[p].last || (pc[q].last == pc[p].last && q < p)) atomicAdd(&pc[p].order, 1);
      if (pc[p].count == 0 || pc[q].count == 0 || pc[q].level < pc[p].level) continue;
      if (pc[q].last < pc[p].first) {
        atomicAdd(&pc[p].base, pc[q].count);
      } else if (pc[q].level > pc[p].level && pc[q].first < pc[p].first) {
        const int at = atomicAdd(&s_pairs, 1);
        if (at < MERGE_PAIRS) pair[at] = (uint16_t)(p << 8 | q);
        else before_block(p, q);
      }
    }
    __syncthreads();
    for (int x = threadIdx.x; x < min(s_pairs, MERGE_PAIRS); x += blockDim.x) before_block(pair[x] >> 8, pair[x] & 255);
    __syncthreads();
    for (int p = threadIdx.x; p < np; p += blockDim.x) sorted[pc[p].order] = pc[p].last;
    __syncthreads();
    int level = -1;
    for (int p = warp; p < np; p += blockDim.x >> 5) {
      const Piece me = pc[p];
      if (me.count == 0) continue;
      if (me.level != level) {
        // pieces of levels below lie between this one's columns: sum[k] is the number of
        // their entries among the first k by last column
        level = me.level;
        __syncwarp();
        for (int q = lane; q < np; q += 32) sum[pc[q].order + 1] = pc[q].level < level ? pc[q].count : 0;
        __syncwarp();
        int carry = 0;
        for (int q0 = 0; q0 < np; q0 += 32) {
          int s = q0 + lane < np ? sum[q0 + lane + 1] : 0;
          for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(FULL, s, o);
            if (lane >= o) s += x;
          }
          if (q0 + lane < np) sum[q0 + lane + 1] = carry + s;
          carry += __shfl_sync(FULL, s, 31);
        }
        if (lane == 0) sum[0] = 0;
        __syncwarp();
      }
      const bool below = sum[np] > 0;
      int base = me.base;
      for (int w0 = 0; w0 < me.words; w0 += 32) {
        uint32_t mine = w0 + lane < me.words ? me.row[w0 + lane] : 0u;
        if (w0 + lane == me.words - 1) mine &= me.mask;
        // entries of levels below before a word's columns: the same number for all where its
        // first and last column have no piece between them (-1: they do)
        auto pieces_before = [&](int x) {
          int lo = 0, hi = np;
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (sorted[mid] < x) lo = mid + 1; else hi = mid;
          }
          return lo;
        };
        int word_add = 0;
        if (below && mine) {
          const int32_t* cols = me.cols + 32 * (w0 + lane);
          const int lo = pieces_before(__ldg(cols + __ffs(mine) - 1)), hi = pieces_before(__ldg(cols + 31 - __clz(mine)));
          word_add = lo == hi ? sum[lo] : -1;
        }
        base += each_bit<true>(mine, w0, [&](int c, int at, int add) {
          const int x = __ldg(me.cols + c);
          L[base + at + (add >= 0 ? add : sum[pieces_before(x)])] = x;
        }, word_add);
      }
    }
    // U: the block's columns above v and the columns right of the block
    if (warp == np % (blockDim.x >> 5)) {
      int before = 1;
      for (int w0 = r >> 5; w0 < b.W; w0 += 32) {
        uint32_t mine = w0 + lane < b.W ? row[w0 + lane] : 0u;
        if (w0 + lane == r >> 5) mine &= gt_bits(r & 31);
        before += each_bit(mine, w0, [&](int c, int at, int) { U[at + before] = block_column(b, c); });
      }
    }
    __syncthreads();
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

cudaError_t launch_front_gids(const FrontLevel& l, int32_t count, int32_t* out, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  front_gids_kernel<<<grid_for(count, 256, 1024), 256, 0, st>>>(l, count, out);
  return cudaGetLastError();
}

cudaError_t launch_front_count(const FrontEmit& e, cudaStream_t st) {
  front_count_kernel<<<grid_for(e.n, 256, 16384), 256, 0, st>>>(e);
  return cudaGetLastError();
}

cudaError_t launch_front_expand(const FrontEmit& e, cudaStream_t st) {
  front_expand_kernel<<<grid_for(32LL * ((e.n + EXPAND_ROWS - 1) / EXPAND_ROWS), 256, 16384), 256, 0, st>>>(e);
  if (e.left > 0) front_merge_kernel<<<e.left, 64, 0, st>>>(e);
  return cudaGetLastError();
}

}  // namespace gsofa
