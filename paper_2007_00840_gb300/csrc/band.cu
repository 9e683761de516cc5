// Symbolic LU of banded patterns by boolean elimination in shared memory.
//
// When every entry of A lies within a band around the diagonal (natural orderings of
// grids, banded systems), so do L and U: eliminating pivot k gives row i of L(:, k) the
// entries of row k right of k (the definition that Theorem 1 restates in paths, Section
// 2.1).  A window of band rows then holds everything that is still needed, as bits on
// chip, and each row costs the band's width in word operations; the path traversal walks
// the whole graph below the row instead (32^3 grid: 86,700 scanned entries per row, here
// 1,000 rows of 33 words once per 32 pivots).
//
// Rows are taken in panels of 32 (one 32-bit word of columns).  Per panel P:
//   A  factor: the 32 x 32 bit block on the diagonal, one row per lane;
//   B  the panel's rows right of the block (every pivot of the block is known, so the
//      32 rows are independent), written out as finished bitmap rows;
//   C  update of the rows below that the band lets P reach: the row's word of columns P
//      is closed over the block (that is its word of L), and it takes the panel rows it
//      needs.  A panel row l with a symmetric partner q in the same block (l -> q in U,
//      q -> l in L) is left out: U(l,:) right of q is contained in U(q,:), and the closure
//      holds q.  The few rows left (one in a dense band, about eight on a 2D grid) are
//      combined in tables of 16 for every four of them, so that a word of a row costs one
//      load per four panel rows.
// The chain from one block to the next cannot be shortened by more warps: one finds the next panel's
// block (panel P applied to that one word of its rows) and factors it while the other
// warps do B and C of panel P for all words.
// One CTA takes one matrix; wide bands are split over a cluster of up to eight (row
// panels in turn), and the panel's result is written to every CTA's shared memory.
//
// The finished rows are bitmaps in global memory: (bl + bu) / 32 + 1 words per row.
// Counts, fill counts and supernodes come from them, and the column lists are expanded
// straight into the result.
#include <climits>
#include <cooperative_groups.h>

#include "band.cuh"
#include "route.cuh"

namespace gsofa {

namespace {

namespace cg = cooperative_groups;

__device__ __forceinline__ uint32_t gt_mask(int k) { return k >= 31 ? 0u : 0xFFFFFFFEu << k; }  // bits above k
__device__ __forceinline__ uint32_t lt_mask(int k) { return (1u << k) - 1u; }                   // bits below k
// all ones where bit k of x is set (two shifts: shorter than a predicate's way to the OR)
__device__ __forceinline__ uint32_t spread(uint32_t x, int k) { return (uint32_t)((int32_t)(x << (31 - k)) >> 31); }

__device__ __forceinline__ void copy_async4(void* dst, const void* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Barrier `id` among `threads` threads of the CTA.
__device__ __forceinline__ void group_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// The same without waiting.
__device__ __forceinline__ void group_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// descriptor of a global row / group: the last matrix that starts at or before it
__device__ __forceinline__ int mat_at(const BandArgs& a, long long x, bool group) {
  int lo = 0, hi = a.nmats - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    const long long b = group ? a.mats[mid].group_base : a.mats[mid].row_base;
    if (b <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

}  // namespace

// ------------------------------------------------------------ check and measure
// The checks of validate_kernel, the rows' distance from the diagonal on both sides
// (largest over each matrix in band[2m], band[2m+1]), and every row's entries of A with the
// diagonal counted as present.  One matrix: also the panel boundaries that an entry below
// the diagonal crosses; where none does, the rows after the boundary take nothing from the
// rows before it.  A warp takes 32 rows and reports once (per CTA for one matrix): a look
// at the two maxima per row, all at one address, took 198 us on 1M rows, this 42.
__global__ void __launch_bounds__(256) band_scan_kernel(BandArgs a) {
  __shared__ int s_l[8], s_u[8];
  __shared__ unsigned long long s_nnz[8], s_spread[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane & 7;
  const long long chunks = (a.rows + 31) >> 5, step = (long long)gridDim.x * 8;
  int max_l = 0, max_u = 0;
  unsigned long long nnz = 0, spread = 0;
  // (indices are unsigned: a row that starts at the largest index wraps out of its range)
  for (long long q = (long long)blockIdx.x * 8 + warp; q < chunks; q += step) {
    // a row per lane
    const long long r = 32 * q + lane;
    int m = 0, i = 0, n = 0, rb = 0, re = 0, bad = 0;
    const int32_t* col = nullptr;
    if (r < a.rows) {
      m = a.mats ? mat_at(a, r, false) : 0;
      const BandMat d = a.mats ? a.mats[m] : a.one;
      i = (int)(r - d.row_base);
      n = d.n;
      col = d.colidx;
      rb = d.rowptr[i];
      re = d.rowptr[i + 1];
      if (re < rb || rb < 0 || (i == 0 && rb != 0)) bad = ERR_ROWPTR;
    }
    const int stop = bad ? rb : re;
    const int m0 = __shfl_sync(FULL, m, 0);
    const bool one = __all_sync(FULL, m == m0 || r >= a.rows);
    // then eight lanes per row, four rows at a time; the first eight columns of all rows in flight
    int c8[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int row = 4 * k + (lane >> 3);
      const unsigned e = (unsigned)(__shfl_sync(FULL, rb, row) + sub);
      const int32_t* x = (const int32_t*)__shfl_sync(FULL, (unsigned long long)col, row);
      c8[k] = e < (unsigned)__shfl_sync(FULL, stop, row) ? x[e] : 0;
    }
    int bl = 0, bu = 0, low = INT_MAX;
    unsigned has = 0u;  // bit x: row x has its diagonal
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int row = 4 * k + (lane >> 3);
      const unsigned b = (unsigned)__shfl_sync(FULL, rb, row), e1 = (unsigned)__shfl_sync(FULL, stop, row);
      const int at = __shfl_sync(FULL, i, row), nr = __shfl_sync(FULL, n, row);
      const int32_t* x = (const int32_t*)__shfl_sync(FULL, (unsigned long long)col, row);
      int wrong = 0, dg = 0, l = 0, u = 0;
      for (unsigned e = b + sub; e < e1; e += 8) {
        const int c = e == b + sub ? c8[k] : x[e];
        if ((unsigned)c >= (unsigned)nr) {
          wrong |= ERR_COL_RANGE;
          continue;
        }
        if (e > b && x[e - 1] >= c) wrong |= ERR_UNSORTED;
        l = max(l, at - c);
        u = max(u, c - at);
        spread += (unsigned)abs(at - c);
        dg |= c == at;
        if (at - c < BAND_REACH_MAX) low = min(low, c);
      }
      const unsigned d = __ballot_sync(FULL, dg);
#pragma unroll
      for (int g = 0; g < 4; g++)
        if ((d >> (8 * g)) & 0xFFu) has |= 1u << (4 * k + g);
      if (__any_sync(FULL, wrong != 0)) {
        for (int o = 4; o >= 1; o >>= 1) wrong |= __shfl_xor_sync(FULL, wrong, o);
        const int mine = __shfl_sync(FULL, wrong, 8 * (lane & 3));
        if (lane >> 2 == k) bad |= mine;
      }
      bl = max(bl, l);
      bu = max(bu, u);
      if (!one) {  // rows of several matrices: each row its own
        int32_t* band = a.band + 2 * (size_t)__shfl_sync(FULL, m, row);
        if (l > *(volatile int32_t*)band) atomicMax(band, l);
        if (u > *(volatile int32_t*)(band + 1)) atomicMax(band + 1, u);
      }
    }
    if (r < a.rows) {
      if (a.entries && i == n - 1) a.entries[m] = re;
      a.fill[r] = (re - rb) + ((has >> lane) & 1u ? 0 : 1);
      nnz += (unsigned)(stop - rb);
      if (bad) {
        atomicOr(&a.ctr->err, bad);
        atomicMax(&a.ctr->bad_row, INT_MAX - (int)r);
      }
    }
    if (!one) continue;
    bl = __reduce_max_sync(FULL, bl);
    bu = __reduce_max_sync(FULL, bu);
    if (a.mats) {
      if (lane == 0) {
        int32_t* band = a.band + 2 * (size_t)m0;
        if (bl > *(volatile int32_t*)band) atomicMax(band, bl);
        if (bu > *(volatile int32_t*)(band + 1)) atomicMax(band + 1, bu);
      }
      continue;
    }
    max_l = max(max_l, bl);
    max_u = max(max_u, bu);
    if (a.cross) {
      // panel boundaries between these rows, one panel, and their leftmost entry (no wider
      // band fits on chip, and more marks than needed only keep stretches together)
      low = __reduce_min_sync(FULL, low);
      const int q1 = (int)q, q0 = low == INT_MAX ? q1 + 1 : (low >> 5) + 1;
      if (q0 <= q1)
        for (int w = (q0 >> 5) + lane; w <= q1 >> 5; w += 32) {
          const int lo = max(q0 - 32 * w, 0), hi = min(q1 - 32 * w, 31);
          const uint32_t bits = (0xFFFFFFFFu << lo) & (0xFFFFFFFFu >> (31 - hi));
          if ((*(volatile uint32_t*)(a.cross + w) & bits) != bits) atomicOr(a.cross + w, bits);
        }
    }
  }
  if (a.mats) return;
  for (int o = 16; o >= 1; o >>= 1) {
    nnz += __shfl_xor_sync(FULL, nnz, o);
    spread += __shfl_xor_sync(FULL, spread, o);
  }
  if (lane == 0) {
    s_l[warp] = max_l;
    s_u[warp] = max_u;
    s_nnz[warp] = nnz;
    s_spread[warp] = spread;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; w++) {
      max_l = max(max_l, s_l[w]);
      max_u = max(max_u, s_u[w]);
      nnz += s_nnz[w];
      spread += s_spread[w];
    }
    atomicAdd(&a.ctr->nnz, nnz);
    atomicAdd(&a.ctr->spread, spread);
    if (max_l > *(volatile int32_t*)a.band) atomicMax(a.band, max_l);
    if (max_u > *(volatile int32_t*)(a.band + 1)) atomicMax(a.band + 1, max_u);
  }
}

// ------------------------------------------------------------ reach of sampled rows
// A CTA per sampled row s (one in each of reach_rows equal parts of a matrix, at a place
// that does not repeat with its structure): breadth-first search from s over vertices below
// s, level by level, a thread (or eight) per vertex, vertices found marked in a bitmap.
// Cut off after what the choice of the route can still use.  Bound by the latency of a
// level: row pointers, columns, bitmap, a barrier, 1.3 us or more.  A call that stays with the
// elimination after a search takes 100 us more on 317 x 293 (7,360), 40 for sizes alone on 27 x 25
// x 29 (2,360); where there is none (route.cuh) nothing to be seen.  The last CTA finds the
// longest stretch of one matrix.
namespace {
constexpr int REACH_THREADS = 256;
constexpr int REACH_QUEUE = 256;    // vertices of a level: wider searches are long (a band of 211: 20 us against 45 with 1,024)
constexpr int REACH_WORDS = 49152;  // of the bitmap at most: a search that goes further back is cut off
// Words of the bitmap for orders up to n (a multiple of four; room for the stretches' sums).
int reach_words(int n) {
  const int w = ((n - 1) / 32 + 4) & ~3;
  return w > REACH_WORDS ? REACH_WORDS : w < 3 * REACH_THREADS ? 3 * REACH_THREADS : w;
}
}  // namespace
__global__ void __launch_bounds__(REACH_THREADS) band_reach_kernel(BandArgs a, bool counts, int words) {
  extern __shared__ __align__(16) uint32_t bsm[];
  uint32_t* seen = bsm;                      // vertices first .. first + 32 words - 1
  int32_t* queue = (int32_t*)(bsm + words);  // [2][REACH_QUEUE]
  __shared__ int s_stretches;
  __shared__ struct { int found, cut; uint32_t entries; } level[3];  // one barrier a level: read, written, cleared
  const int m = blockIdx.x / a.reach_rows, k = blockIdx.x % a.reach_rows;
  const int tid = threadIdx.x, lane = tid & 31;
  if (m >= a.sampled) {
    // panel q > 0 starts a stretch where bit q of cross is clear; a thread takes some words in
    // turn: first and last start in them, and the longest stretch between
    const int panels = (a.one.n + 31) >> 5, cw = (panels + 31) >> 5;
    const int some = (cw + REACH_THREADS - 1) / REACH_THREADS;
    int first = -1, last = -1, most = 0;
    for (int w = some * tid; w < min(cw, some * (tid + 1)); w++) {
      uint32_t open = ~a.cross[w];
      if (w == 0) open |= 1u;
      for (; open; open &= open - 1) {
        const int q = 32 * w + __ffs(open) - 1;
        if (q >= panels) break;
        if (first < 0) first = q;
        else most = max(most, q - last);
        last = q;
      }
    }
    int32_t* part = (int32_t*)bsm;
    part[tid] = first;
    part[REACH_THREADS + tid] = last;
    part[2 * REACH_THREADS + tid] = most;
    __syncthreads();
    if (tid == 0) {
      int at = 0;
      for (int t = 0; t < REACH_THREADS; t++) {
        if (part[t] < 0) continue;
        most = max(most, max(part[2 * REACH_THREADS + t], part[t] - at));
        at = part[REACH_THREADS + t];
      }
      a.ctr->stretch = max(most, panels - at);
    }
    return;
  }
  const BandMat d = a.mats ? a.mats[m] : a.one;
  const int n = d.n;
  const int err = a.ctr->err, LB = band_words_left(a.band[2 * m]), UB = band_words_right(a.band[2 * m + 1]);
  const int nnz = d.rowptr[n], panels = (n + 31) >> 5;
  if (tid == 0) s_stretches = 1;
  for (int i = tid; i < words / 4; i += REACH_THREADS) ((uint4*)seen)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (err) return;  // nothing is followed unchecked
  const bool fits = band_shape(LB, UB, false).C > 0;
  if (!fits) {
    if (a.mats || counts) return;
    const bool near = near_diagonal(*a.ctr, a.band);
    if (n < (near ? FRONT_NEAR_ORDER : FRONT_MIN_ORDER) || surely_blocks(n, *a.ctr, near)) return;
  }
  // the panels in a chain: where there are stretches, about four of the mean length
  int chain = panels;
  if (a.cross) {
    __syncthreads();
    int open = 0;
    for (int w = tid; 32 * w < panels; w += REACH_THREADS) {
      const uint32_t inside = panels - 32 * w < 32 ? (1u << (panels & 31)) - 1u : FULL;
      open += __popc(~a.cross[w] & inside & (w == 0 ? ~1u : FULL));
    }
    open = __reduce_add_sync(FULL, open);
    if (lane == 0 && open) atomicAdd(&s_stretches, open);
    __syncthreads();
    chain = min(panels, 4 * (panels / s_stretches + 1));
  }
  const float band = fits ? band_us(n, chain, LB, UB, counts) : 0.f;
  const float limit = reach_limit_us(n, (unsigned long long)nnz, band, counts);
  if (limit <= 0.f) return;
  const TraverseCost cost = traverse_cost(n, counts);
  const float row_ns = 1e3f * limit / (float)n;
  // a row is searched up to this cost: one and a half times its share, more where the elimination takes long
  // (20 ms a share more: of a million rows of degree 1.3 some are long, 99 ms against 24)
  const float most_ns = row_ns * (1.5f + 5e-5f * band);
  // as many levels as take 2% of the elimination, at 1 us each
  const int most_levels = max(6, (int)(0.02f * (fits ? band : fronts_us(n))));

  const uint32_t place = ((uint32_t)k * 2654435761u) >> 16;
  const int s = (int)((((long long)k << 16) + place) * n / ((long long)a.reach_rows << 16));
  const int first = max(0, s - 32 * words + 1);
  const int lanes = nnz / n > 16 ? 8 : 1;  // threads per vertex; rows of more than 64 entries each end the search
  const int sub = tid & (lanes - 1);
  if (tid == 0) {
    queue[0] = s;
    level[1] = {0, 0, 0u};
  }
  const unsigned long long decided = (unsigned long long)(1.2f * row_ns / cost.entry * (float)a.reach_rows);
  uint32_t all = 0u;
  int levels = 0, count = 1;
  bool cut = false;
  __syncthreads();
  while (count > 0) {
    const int32_t* in = queue + REACH_QUEUE * (levels & 1);
    int32_t* out = queue + REACH_QUEUE * ((levels & 1) ^ 1);
    auto& next = level[(levels + 1) % 3];
    if (tid == 0) {
      level[(levels + 2) % 3] = {0, 0, 0u};
      // the other rows may have decided already
      if ((levels & 3) == 3 && *(volatile unsigned long long*)&a.reach[m].entries > decided) next.cut = 1;
    }
    uint32_t entries = 0u;
    for (int i0 = 0; i0 < count; i0 += REACH_THREADS / lanes) {
      const int i = i0 + tid / lanes;
      uint32_t b = 0, e = 0;  // unsigned: x may pass the largest index
      if (i < count) {
        const int v = in[i];
        b = (uint32_t)d.rowptr[v];
        e = (uint32_t)d.rowptr[v + 1];
        if (sub == 0) entries += e - b;
        if (e - b > 64u * lanes) {
          next.cut = 1;
          e = b;
        }
      }
      for (uint32_t x = b + sub; __any_sync(FULL, x < e); x += 8 * lanes) {
        // eight columns at a time: loads, then marks, in flight together (no mark: no bit of word 0)
        int c[8];
        uint32_t bit[8], old[8];
#pragma unroll
        for (int j = 0; j < 8; j++) c[j] = x + j * lanes < e ? d.colidx[x + j * lanes] : s;
#pragma unroll
        for (int j = 0; j < 8; j++) {
          const bool in_range = c[j] < s && c[j] >= first;
          bit[j] = in_range ? 1u << ((c[j] - first) & 31) : 0u;
          old[j] = atomicOr(seen + (in_range ? (c[j] - first) >> 5 : 0), bit[j]);
        }
        unsigned fresh = 0u, far = 0u;
#pragma unroll
        for (int j = 0; j < 8; j++) {
          if (bit[j] & ~old[j]) fresh |= 1u << j;
          far |= c[j] < first;
        }
        if (far) next.cut = 1;
        int before = __popc(fresh);
        const int mine = before;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(FULL, before, o);
          if (lane >= o) before += y;
        }
        int at = 0;
        if (lane == 31 && before > 0) at = atomicAdd(&next.found, before);
        at = __shfl_sync(FULL, at, 31) + before - mine;
#pragma unroll
        for (int j = 0; j < 8; j++)
          if ((fresh >> j) & 1u) {
            if (at < REACH_QUEUE) out[at] = c[j];
            at++;
          }
      }
    }
    if (__any_sync(FULL, entries > 0u)) {
      entries = __reduce_add_sync(FULL, entries);
      if (lane == 0) atomicAdd(&next.entries, entries);
    }
    __syncthreads();
    levels++;
    count = next.found;
    all += next.entries;
    cut = next.cut || count > REACH_QUEUE || levels >= most_levels ||
          cost.level * (float)levels + cost.entry * (float)all > most_ns ||
          row_us((float)levels, (float)all) > 1.5f * limit;
    if (cut) {
      cut = next.cut || count > 0;
      break;
    }
  }
  if (tid == 0) {
    unsigned long long entries = all;
    // cut off: as if it reached every row before it, and never less than three times its share
    if (cut) entries = max(entries, (unsigned long long)s * (unsigned long long)nnz / (unsigned long long)n);
    atomicMax(&a.reach[m].longest, (uint32_t)fminf(row_us((float)levels, (float)entries), 4e9f) + 1u);
    if (cut) entries = max(entries, (unsigned long long)(3.f * row_ns / cost.entry));
    atomicAdd(&a.reach[m].entries, entries);
    atomicAdd(&a.reach[m].levels, (uint32_t)levels);
  }
}

// ------------------------------------------------------------ elimination
namespace {

// One CTA's view of its matrix.  Panel q (rows 32q .. 32q+31) lives in CTA q % C at slot
// (q / C) % slots.  Band: word c of a row of panel q is at index c - q + LB, and a panel
// reaches UB words right of its own.  Front (a dense block of W words per row, all of its
// rows on chip): word c is at index c.
struct Band {
  const int32_t* rowptr;
  const int32_t* colidx;
  int n, LB, UB, W;
  int xs;          // words per row in shared memory (odd: lane-per-row accesses spread over the banks)
  int us;          // words per panel row in the panel buffers (odd)
  int slots;
  uint32_t* x;
};

template <int C>
__device__ __forceinline__ uint32_t* panel_rows(const Band& B, int q) {
  return B.x + (size_t)((q / C) % B.slots) * 32 * B.xs;
}

// Word 0 of the columns in a row of panel q, and the words right of panel P's own.
template <bool FRONT>
__device__ __forceinline__ int word0(const Band& B, int q) { return FRONT ? 0 : B.LB - q; }
template <bool FRONT>
__device__ __forceinline__ int words_right(const Band& B, int P) { return FRONT ? B.W - 1 - P : B.UB; }

// The entries of rows 32q .. 32q+31 into their zeroed slot (one warp), from the staged
// copy of the panel's columns or in place.
template <int C>
__device__ void fill_panel(const Band& B, int q, int rb, int re, const int32_t* stage, int chunk0) {
  const int lane = threadIdx.x & 31;
  uint32_t* x = panel_rows<C>(B, q);
  if (stage) {
    uint32_t* row = x + lane * B.xs - q + B.LB;
#pragma unroll 1
    for (int e = rb; e < re; e += 4) {
      int c[4];
#pragma unroll
      for (int k = 0; k < 4; k++) c[k] = e + k < re ? stage[e + k - chunk0] : -1;
#pragma unroll
      for (int k = 0; k < 4; k++)
        if (c[k] >= 0) atomicOr(row + (c[k] >> 5), 1u << (c[k] & 31));
    }
  } else {
#pragma unroll 1
    for (int r = 0; r < 32; r++) {
      const int b = __shfl_sync(FULL, rb, r), n = __shfl_sync(FULL, re, r);
      uint32_t* row = x + r * B.xs - q + B.LB;
#pragma unroll 1
      for (int e = b + lane; e < n; e += 32) {
        const int c = B.colidx[e];
        atomicOr(row + (c >> 5), 1u << (c & 31));
      }
    }
  }
  __syncwarp();
}

// Row pointers of this lane's row of panel q (empty past the end).
__device__ __forceinline__ void panel_rowptr(const Band& B, int q, int& rb, int& re) {
  const int i = 32 * q + (threadIdx.x & 31);
  rb = re = 0;
  if (i < B.n) {
    rb = __ldg(B.rowptr + i);
    re = __ldg(B.rowptr + i + 1);
  }
}

// Elimination of the diagonal block: w is the lane's row.  dip: the rows of the block the
// lane's row takes in, those of its L entries and, through them, of theirs (a pivot k
// reached brings what k itself took from lower pivots, fills of this row or not).  Four
// pivots per round: their rows are fetched together and finished in every lane's
// registers, so the chain is eight shuffles long, not 32.
__device__ __forceinline__ uint32_t factor_block(uint32_t w, uint32_t& dip) {
  const int lane = threadIdx.x & 31;
  const uint32_t below = lt_mask(lane);
  uint32_t t = 0u;
#pragma unroll
  for (int k0 = 0; k0 < 32; k0 += 4) {
    uint32_t v[4], dv[4];
#pragma unroll
    for (int p = 0; p < 4; p++) v[p] = __shfl_sync(FULL, w, k0 + p);
#pragma unroll
    for (int p = 0; p < 4; p++) dv[p] = __shfl_sync(FULL, t, k0 + p);
#pragma unroll
    for (int p = 0; p < 4; p++) {
      const uint32_t u = v[p] & gt_mask(k0 + p);
      const uint32_t dp = dv[p] | (1u << (k0 + p));
#pragma unroll
      for (int c = p + 1; c < 4; c++) {
        const uint32_t on = spread(v[c], k0 + p);
        v[c] |= u & on;
        dv[c] |= dp & on;
      }
      const uint32_t on = spread(w & below, k0 + p);
      w |= u & on;
      t |= dp & on;
    }
  }
  dip = t;
  return w;
}

// Rows of the block without a symmetric partner above them in the block: the 32 x 32 bits
// are transposed in five exchanges.
__device__ __forceinline__ uint32_t block_tops(uint32_t w) {
  const int lane = threadIdx.x & 31;
  uint32_t col = w;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    const uint32_t mask = o == 16 ? 0x0000FFFFu : o == 8 ? 0x00FF00FFu : o == 4 ? 0x0F0F0F0Fu : o == 2 ? 0x33333333u
                                                                                                  : 0x55555555u;
    const uint32_t y = __shfl_xor_sync(FULL, col, o);
    col = (lane & o) ? ((col & ~mask) | ((y >> o) & mask)) : ((col & mask) | ((y << o) & ~mask));
  }
  return __ballot_sync(FULL, (w & col & gt_mask(lane)) == 0u);
}

}  // namespace

// Smallest panel boundary in [q, end) that no entry below the diagonal crosses, else end (warp-wide).
__device__ __forceinline__ int next_cut(const uint32_t* cross, int q, int end) {
  const int lane = threadIdx.x & 31;
  for (int w0 = q >> 5; 32 * w0 < end; w0 += 32) {
    const int w = w0 + lane;
    uint32_t open = 32 * w < end ? ~__ldg(cross + w) : 0u;
    if (w == q >> 5) open &= 0xFFFFFFFFu << (q & 31);
    const unsigned b = __ballot_sync(FULL, open != 0u);
    if (b) {
      const int l = __ffs(b) - 1;
      open = __shfl_sync(FULL, open, l);
      return min(end, 32 * (w0 + l) + __ffs(open) - 1);
    }
  }
  return end;
}

namespace {

// The panel step's shared state (per CTA; clusters write every CTA's copy).
struct PanelBufs {
  uint32_t* pw;   // [2][32] block rows (the panel's CTA)
  uint32_t* pg;   // [2][32] the same, bits above the diagonal only
  uint32_t* dip;  // [2][32] rows of the block each row takes in (the panel's CTA)
  uint32_t* top;  // [2][33] block rows without a partner: their number, then the rows
  uint32_t* pu;   // [2][32][us] panel rows right of the block
  uint32_t* cl;   // [slots][32] this step's rows below: closed words, then the partnerless rows in them
  uint32_t* tb;   // [8][16][us] combinations of four partnerless panel rows
};

// A: factor the block of panel P, w its rows (one warp of its CTA).
template <int C>
__device__ __forceinline__ void step_factor(const PanelBufs& S, int P, uint32_t w) {
  const int lane = threadIdx.x & 31, at = 32 * (P & 1) + lane;
  uint32_t dip;
  w = factor_block(w, dip);
  S.pw[at] = w;
  S.dip[at] = dip;
  if constexpr (C > 1) {
#pragma unroll 1
    for (int t = 0; t < C; t++) cg::this_cluster().map_shared_rank(S.pg, t)[at] = w & gt_mask(lane);
  } else {
    S.pg[at] = w & gt_mask(lane);
  }
}

// The word m of a row's entries in the block's columns, closed over the block (its word of
// L): g has the block rows above the diagonal.
__device__ __forceinline__ uint32_t close_word(uint32_t m, const uint32_t* g) {
#pragma unroll
  for (int k = 0; k < 32; k += 4) {
    const uint4 u = *(const uint4*)(g + k);
    m |= u.x & spread(m, k);
    m |= u.y & spread(m, k + 1);
    m |= u.z & spread(m, k + 2);
    m |= u.w & spread(m, k + 3);
  }
  return m;
}

// The chain: panel P applied to the block of panel P + 1, then its factor.  With one CTA
// the panel's rows right of the block are not ready yet (B runs beside this): their first
// word is found here too.  Barrier 1 tells the workers that this warp's inputs are read.
template <int C, bool FRONT>
__device__ __forceinline__ void step_chain(const Band& B, const PanelBufs& S, int P, int sync_threads) {
  const int lane = threadIdx.x & 31, at = 32 * (P & 1) + lane;
  const uint32_t* x1 = panel_rows<C>(B, P + 1) + lane * B.xs + word0<FRONT>(B, P + 1) + P;
  uint32_t m = x1[0], y = x1[1];
  uint32_t first = 0u;
  const bool right = words_right<FRONT>(B, P) > 0;
  if constexpr (C == 1) {
    const uint32_t v = right ? panel_rows<C>(B, P)[lane * B.xs + word0<FRONT>(B, P) + P + 1] : 0u;
    const uint32_t dip = S.dip[at];
    group_arrive(1, sync_threads);
    first = v;
#pragma unroll
    for (int k = 0; k < 31; k++) first |= __shfl_sync(FULL, v, k) & spread(dip, k);
  } else {
    if (right) first = S.pu[(size_t)32 * B.us * (P & 1) + lane * B.us];
    group_arrive(1, sync_threads);
  }
  if (__any_sync(FULL, m != 0u)) {
    const uint32_t* g = S.pg + 32 * (P & 1);
#pragma unroll
    for (int k = 0; k < 32; k += 4) {
      const uint4 u = *(const uint4*)(g + k);
      const uint32_t uk[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const uint32_t on = spread(m, k + i);
        y |= __shfl_sync(FULL, first, k + i) & on;
        m |= uk[i] & on;
      }
    }
  }
  step_factor<C>(S, P + 1, y);
}

// i / d for 0 <= i < 2^16, 0 < d < 2^12: the quotient of i + 1/2 is at least 1 / (2 d) from
// a whole number, far more than its rounding.  An integer division per panel took 6-10% of
// a banded 32^3 or 317x293.
__device__ __forceinline__ int quotient(int i, int d) { return (int)__fdividef((float)i + 0.5f, (float)d); }

// B: the rows of panel P right of the block; a row takes rows of the block as they came
// in.  Items [i0, i0 + 32) of 16 * ub (ub words right of the block), one lane each: one
// word of two rows (one load of a block row serves both).
template <int C, bool FRONT>
__device__ __forceinline__ void step_rows(const Band& B, const PanelBufs& S, int P, int i0) {
  const int i = i0 + (threadIdx.x & 31);
  const int ub = words_right<FRONT>(B, P);
  if (i >= 16 * ub) return;
  uint32_t* pu = S.pu + (size_t)32 * B.us * (P & 1);
  const uint32_t* dip = S.dip + 32 * (P & 1);
  const int r0 = quotient(i, ub) * 2, c = i - (r0 >> 1) * ub;
  const uint32_t* col = panel_rows<C>(B, P) + word0<FRONT>(B, P) + P + 1 + c;
  uint32_t m0 = dip[r0], m1 = dip[r0 + 1];
  uint32_t v0 = col[r0 * B.xs], v1 = col[(r0 + 1) * B.xs];
#pragma unroll 1
  for (int k0 = 0; k0 <= r0; k0 += 8, col += 8 * B.xs, m0 >>= 8, m1 >>= 8) {
    uint32_t xk[8];
#pragma unroll
    for (int k = 0; k < 8; k++) xk[k] = col[k * B.xs];
#pragma unroll
    for (int k = 0; k < 8; k++) {
      v0 |= xk[k] & spread(m0, k);
      v1 |= xk[k] & spread(m1, k);
    }
  }
  uint32_t* dst = pu + r0 * B.us + c;
  if constexpr (C > 1) {
#pragma unroll 1
    for (int t = 0; t < C; t++) {
      uint32_t* o = cg::this_cluster().map_shared_rank(dst, t);
      o[0] = v0;
      o[B.us] = v1;
    }
  } else {
    dst[0] = v0;
    dst[B.us] = v1;
  }
}

// The block rows of panel P without partners (one warp).
template <int C>
__device__ __forceinline__ void step_tops(const PanelBufs& S, int P) {
  const int lane = threadIdx.x & 31;
  const uint32_t top = block_tops(S.pw[32 * (P & 1) + lane]);
  uint32_t* dst = S.top + 33 * (P & 1);
  const int at = ((top >> lane) & 1u) ? 1 + __popc(top & lt_mask(lane)) : -1;
  if constexpr (C > 1) {
#pragma unroll 1
    for (int t = 0; t < C; t++) {
      uint32_t* o = cg::this_cluster().map_shared_rank(dst, t);
      if (at > 0) o[at] = (uint32_t)lane;
      if (lane == 0) o[0] = (uint32_t)__popc(top);
    }
  } else {
    if (at > 0) dst[at] = (uint32_t)lane;
    if (lane == 0) dst[0] = (uint32_t)__popc(top);
  }
}

// The workers' part of the step of panel P: B (one CTA), then C for this CTA's panels
// P + 1 .. hi.  nwk worker warps, warp 1 the first; `next`: the chain runs beside this.
template <int C, bool FRONT>
__device__ __forceinline__ void step_below(const Band& B, const PanelBufs& S, int P, int hi, bool next, int rank,
                                           int nwk) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wk = 32 * nwk, me = (int)threadIdx.x - 32;
  const int ub = words_right<FRONT>(B, P);
  // first: B, and the rows that the panel reaches, their words closed
  const int lo = P + 1 + (C > 1 ? (rank - (P + 1) % C + C) % C : 0);  // this CTA's first panel from P + 1 on
  const int cnt = hi >= lo ? (hi - lo) / C + 1 : 0;
  const int nb = C == 1 ? (16 * ub + 31) / 32 : 0;
  for (int u = warp - 1; u < nb + cnt; u += nwk) {
    if (u < nb) {
      step_rows<C, FRONT>(B, S, P, 32 * u);
    } else {
      const int q = lo + C * (u - nb);
      const uint32_t m = panel_rows<C>(B, q)[lane * B.xs + word0<FRONT>(B, q) + P];
      S.cl[32 * (u - nb) + lane] = __any_sync(FULL, m != 0u) ? close_word(m, S.pg + 32 * (P & 1)) : 0u;
    }
  }
  if (next) group_sync(1, 32 * (C == 1 ? nwk + 2 : nwk + 1));
  else group_sync(2, 32 * nwk);
  if (cnt == 0) return;
  const uint32_t* pu = S.pu + (size_t)32 * B.us * (P & 1);
  const int slot0 = (lo / C) % B.slots;  // this CTA's panels from lo on have the slots from here on
  // this thread's word of a row, and the stride of all workers
  const int r_at = ub > 0 ? quotient(me, ub) : 0, c_at = me - r_at * ub;
  const int dr = ub > 0 ? quotient(wk, ub) : 0, dc = wk - dr * ub;
  // the closed words into place, and which partnerless rows they hold, numbered; the
  // tables of those rows
  const uint32_t* top = S.top + 33 * (P & 1);
  const int nt = (int)top[0];
  for (int u = warp - 1; u < cnt; u += nwk) {
    int slot = slot0 + u;
    if (slot >= B.slots) slot -= B.slots;
    const uint32_t m = S.cl[32 * u + lane];
    if (m) B.x[(slot * 32 + lane) * B.xs + word0<FRONT>(B, lo + C * u) + P] = m;
    uint32_t has = 0u;
#pragma unroll 4
    for (int i = 0; i < nt; i++) has |= ((m >> top[1 + i]) & 1u) << i;
    S.cl[32 * u + lane] = has;
  }
  if (ub > 0) {
    const int ne = (nt + 3) / 4 * 16;
    for (int e = r_at, c = c_at; e < ne;) {
      uint32_t v = 0u;
      const int g0 = e >> 4 << 2;
#pragma unroll
      for (int i = 0; i < 4; i++)
        if (((e >> i) & 1) && g0 + i < nt) v |= pu[top[1 + g0 + i] * B.us + c];
      S.tb[e * B.us + c] = v;
      e += dr;
      c += dc;
      if (c >= ub) {
        c -= ub;
        e++;
      }
    }
  }
  group_sync(2, 32 * nwk);
  if (ub == 0) return;
  // then C, a word of a row per lane
  for (int r = r_at, c = c_at; r < 32 * cnt;) {
    uint32_t has = S.cl[r];
    if (has) {
      const int u = r >> 5;
      int slot = slot0 + u;
      if (slot >= B.slots) slot -= B.slots;
      uint32_t* x = B.x + (slot * 32 + (r & 31)) * B.xs + word0<FRONT>(B, lo + C * u) + P + 1 + c;
      uint32_t v = *x;
      const uint32_t* tb = S.tb + c;
      do {
        v |= tb[(has & 15u) * B.us];
        tb += 16 * B.us;
        has >>= 4;
      } while (has);
      *x = v;
    }
    r += dr;
    c += dc;
    if (c >= ub) {
      c -= ub;
      r++;
    }
  }
}

}  // namespace

// Bound by latency, one panel of 32 rows after the other: 1.5 us on a 64 x 64 grid, 2.2 at
// band 211, 2.4 at 317 (cluster of 4), 4.3 at 1,024 (of 8).  With one CTA a narrow panel is the
// chain (2,370 of about 3,200 cycles: closing the next rows, 31 dependent shuffles for their
// first word, the factor), a wider one the workers' phases (band 211: 4,300 of 4,650, of which
// C 1,330).  In a cluster the chain (2,320 to 2,630) is followed by B of the next panel and its
// partnerless rows, stored to every CTA in turn: 1,800 and 3,300 cycles with four CTAs, 5,900
// and 5,100 with eight, the larger part of the panel.  Elimination against the
// traversal: 32^3 grid 8.7 -> 4.3 ms, 317 x 293 63 -> 7.0, band 211 of order 15,013 4.9 -> 1.05.
// Warps of a CTA: 0 the chain, the last the loader (rows into the window), the others
// workers (B, C and finished rows out).
template <int C>
__global__ void __launch_bounds__(512, 1) band_elim_kernel(BandArgs a) {
  extern __shared__ __align__(16) uint32_t bsm[];
  const int rank = C > 1 ? (int)(blockIdx.x % C) : 0;
  const BandMat d = a.mats ? a.mats[a.first + blockIdx.x / C] : a.one;
  const int nw = blockDim.x >> 5, nwk = nw - 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool chain = warp == 0, loader = warp == nw - 1;
  Band B;
  B.rowptr = d.rowptr;
  B.colidx = d.colidx;
  B.n = d.n;
  B.LB = d.LB;
  B.UB = d.UB;
  const int wx = B.LB + B.UB + 1;
  B.xs = wx | 1;
  B.us = B.UB | 1;
  B.slots = (B.LB + 2 + C - 1) / C;
  // the workers' stride over the words of finished rows
  const int wk = 32 * nwk, me = (int)threadIdx.x - 32;
  const int wx_r = wk / wx, wx_c = wk % wx;
  PanelBufs S;
  S.pw = bsm;
  S.pg = S.pw + 64;
  S.dip = S.pg + 64;
  S.top = S.dip + 64;
  S.pu = S.top + 68;
  int32_t* stage = (int32_t*)(S.pu + 64 * B.us);  // [4][BAND_STAGE]
  S.cl = (uint32_t*)(stage + 4 * BAND_STAGE);
  S.tb = S.cl + 32 * B.slots;
  B.x = S.tb + 128 * B.us;
  uint32_t* out = a.bits + d.bits_base;

  // loader: the columns of panel q into its stage buffer
  auto stage_panel = [&](int q, int end, int rb, int re) {
    if (q < end && q % C == rank) {
      const int c0 = __shfl_sync(FULL, rb, 0), c1 = __reduce_max_sync(FULL, re);
      if (c1 - c0 <= BAND_STAGE)
#pragma unroll 1
        for (int e = c0 + lane; e < c1; e += 32) copy_async4(stage + (q & 3) * BAND_STAGE + (e - c0), B.colidx + e);
    }
    copy_async_commit();
  };
  auto sync_all = [&] {
    if constexpr (C > 1) cg::this_cluster().sync();
    else __syncthreads();
  };

  // A batch: the CTA (cluster) has the whole matrix.  One matrix: the stretches of panels
  // between uncrossed boundaries are independent, and each goes to the CTA in whose share
  // of the panels it starts (a connected matrix is one stretch).
  const int all = (B.n + 31) >> 5;
  const int part = a.mats ? 0 : (int)(blockIdx.x / C), parts_all = a.mats ? 1 : (int)(gridDim.x / C);
  const int first = (int)((long long)all * part / parts_all), last = (int)((long long)all * (part + 1) / parts_all);
  int q0 = first > 0 ? next_cut(a.cross, first, all) : 0;
  while (q0 < last) {
    const int panels = a.cross ? next_cut(a.cross, q0 + 1, all) : all;  // the stretch is [q0, panels)

    // the first window, and an empty slot for the panel after it
    for (int i = threadIdx.x; i < B.slots * 32 * B.xs; i += blockDim.x) B.x[i] = 0u;
    __syncthreads();
    for (int q = q0 + warp; q <= q0 + B.LB && q < panels; q += nw)
      if (q % C == rank) {
        int rb, re;
        panel_rowptr(B, q, rb, re);
        fill_panel<C>(B, q, rb, re, nullptr, 0);
      }
    // loader state: row pointers up to three panels ahead, columns of two of them in flight
    int rb1 = 0, re1 = 0, rb2 = 0, re2 = 0, rb3 = 0, re3 = 0;
    if (loader) {
      panel_rowptr(B, q0 + B.LB + 1, rb1, re1);
      panel_rowptr(B, q0 + B.LB + 2, rb2, re2);
      panel_rowptr(B, q0 + B.LB + 3, rb3, re3);
      stage_panel(q0 + B.LB + 1, panels, rb1, re1);
      stage_panel(q0 + B.LB + 2, panels, rb2, re2);
    }
    sync_all();
    if (q0 % C == rank) {
      if (chain) step_factor<C>(S, q0, panel_rows<C>(B, q0)[lane * B.xs + B.LB]);
      __syncthreads();
      if constexpr (C > 1) {
        if (loader) step_tops<C>(S, q0);
        else
          for (int i = 32 * warp; i < 16 * B.UB; i += 32 * (nw - 1)) step_rows<C, false>(B, S, q0, i);
      }
    }
    sync_all();

    for (int P = q0; P < panels; P++) {
      // One CTA: B and C of panel P beside the chain to panel P + 1.  Cluster: every CTA does
      // C for its rows, the CTA of panel P + 1 runs the chain beside it, then B of panel
      // P + 1 into every CTA's buffers.
      const bool next = P + 1 < panels && (P + 1) % C == rank;
      if (chain) {
        if (next) step_chain<C, false>(B, S, P, 32 * (C == 1 ? nwk + 2 : nwk + 1));
      } else if (loader) {
        if constexpr (C == 1) {
          step_tops<C>(S, P);
          __syncwarp();
          if (next) group_arrive(1, 32 * (nwk + 2));
        }
        // rows entering the window: their slot held panel P - 1 or an older one
        const int q = P + B.LB + 1;
        stage_panel(q + 2, panels, rb3, re3);
        int rb4, re4;
        panel_rowptr(B, q + 3, rb4, re4);
        copy_async_wait<2>();
        __syncwarp();
        if (q < panels && q % C == rank) {
          const int s0 = __shfl_sync(FULL, rb1, 0), s1 = __reduce_max_sync(FULL, re1);
          fill_panel<C>(B, q, rb1, re1, s1 - s0 <= BAND_STAGE ? stage + (q & 3) * BAND_STAGE : nullptr, s0);
        }
        rb1 = rb2; re1 = re2;
        rb2 = rb3; re2 = re3;
        rb3 = rb4; re3 = re4;
      } else {
        const int hi = min(P + B.LB, panels - 1);
        step_below<C, false>(B, S, P, hi, next, rank, nwk);
        const uint32_t* pu = S.pu + (size_t)32 * B.us * (P & 1);
        {
          // finished rows out; their slot is zeroed for the panel that takes it
          if (P % C == rank && a.bits) {
            const int rows = min(32, B.n - 32 * P);
            uint32_t* x = panel_rows<C>(B, P);
            uint32_t* o = out + (size_t)32 * P * wx;
            const uint32_t* pw = S.pw + 32 * (P & 1);
            int r2 = me / wx, c2 = me % wx;
            for (int i = me; i < 32 * wx; i += wk) {
              uint32_t* at = x + r2 * B.xs + c2;
              if (r2 < rows) o[i] = c2 < B.LB ? *at : (c2 == B.LB ? pw[r2] : pu[r2 * B.us + c2 - B.LB - 1]);
              *at = 0u;
              r2 += wx_r;
              c2 += wx_c;
              if (c2 >= wx) {
                c2 -= wx;
                r2++;
              }
            }
          } else if (P % C == rank) {  // sizes alone
            for (int r2 = warp - 1; r2 < 32; r2 += nwk) {
              uint32_t* row = panel_rows<C>(B, P) + r2 * B.xs;
              const int i = 32 * P + r2;
              int l = 0, u = 0;
              for (int c2 = lane; c2 < wx; c2 += 32) {
                if (c2 < B.LB) l += __popc(row[c2]);
                else if (c2 > B.LB) u += __popc(pu[r2 * B.us + c2 - B.LB - 1]);
                row[c2] = 0u;
              }
              const uint32_t w = S.pw[32 * (P & 1) + r2];
              l = __reduce_add_sync(FULL, l) + __popc(w & lt_mask(r2));
              u = __reduce_add_sync(FULL, u) + __popc(w & gt_mask(r2)) + 1;
              if (lane == 0 && i < B.n) {
                a.row_nL[i] = l;
                a.row_nU[i] = u;
                a.fill[i] = l + u - a.fill[i];
              }
            }
          }
        }
      }
      if constexpr (C > 1) {
        if (next) {
          __syncthreads();
          if (loader) step_tops<C>(S, P + 1);
          else
            for (int i = 32 * warp; i < 16 * B.UB; i += 32 * (nw - 1)) step_rows<C, false>(B, S, P + 1, i);
        }
      }
      sync_all();
    }
    if (loader) copy_async_wait<0>();
    __syncthreads();
    q0 = panels < last ? panels : last;
  }
}

// ------------------------------------------------------------ fronts
// Elimination of one block of a nested dissection (fronts.cu): rows 0 .. sz-1 are the
// block's vertices (the pivots), then nr rows above the block that have entries in its
// columns; columns are the block's, then the nb columns right of it that its rows reach.
// The whole front is on chip; all of its rows come out: L and U of the block's vertices,
// and for the rows above their L entries in the block and what they reach through it.
template <int C>
__global__ void __launch_bounds__(512, 1) front_elim_kernel(FrontArgs a) {
  extern __shared__ __align__(16) uint32_t bsm[];
  const int rank = C > 1 ? (int)(blockIdx.x % C) : 0;
  const FrontMat d = a.fronts[a.first + blockIdx.x / C];
  const int nw = blockDim.x >> 5, nwk = nw - 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool chain = warp == 0, loader = warp == nw - 1;
  const int pivots = (d.sz + 31) >> 5, panels = pivots + ((d.nr + 31) >> 5);
  Band B;
  B.rowptr = nullptr;
  B.colidx = a.col;
  B.n = d.sz;
  B.LB = 0;
  B.W = pivots + ((d.nb + 31) >> 5);
  B.UB = B.W - 1;
  B.xs = B.W | 1;
  B.us = B.UB | 1;
  B.slots = (panels + C - 1) / C;
  PanelBufs S;
  S.pw = bsm;
  S.pg = S.pw + 64;
  S.dip = S.pg + 64;
  S.top = S.dip + 64;
  S.pu = S.top + 68;
  S.cl = S.pu + 64 * B.us;
  S.tb = S.cl + 32 * B.slots;
  B.x = S.tb + 128 * B.us;
  uint32_t* out = a.bits + d.bits_base;
  const int32_t* bc = a.bc + d.bc_base;
  const uint2* right = a.right ? a.right + (size_t)d.id * a.right_words : nullptr;
  auto sync_all = [&] {
    if constexpr (C > 1) cg::this_cluster().sync();
    else __syncthreads();
  };

  for (int i = threadIdx.x; i < B.slots * 32 * B.xs; i += blockDim.x) B.x[i] = 0u;
  __syncthreads();
  // the rows, one warp each: columns of the block are their offset, the others their place in bc
  for (int i = warp; i < 32 * panels; i += nw) {
    const int q = i >> 5;
    if (q % C != rank) continue;
    int b = 0, e = 0;
    if (q < pivots) {
      if (i < d.sz) {
        b = a.beg[d.first_vertex + i];
        e = a.end[d.first_vertex + i];
      }
    } else if (i - 32 * pivots < d.nr) {
      b = a.br_b[d.br_base + i - 32 * pivots];
      e = a.br_e[d.br_base + i - 32 * pivots];
    }
    uint32_t* row = panel_rows<C>(B, q) + (i & 31) * B.xs;
#pragma unroll 4
    for (int k = b + lane; k < e; k += 32) {
      const int c = a.col[k] - d.first_vertex;
      int at = c;
      if (c >= d.sz && right) {
        const uint2 x = right[(c + d.first_vertex) >> 5];
        at = 32 * pivots + (int)x.y + __popc(x.x & lt_mask((c + d.first_vertex) & 31));
      } else if (c >= d.sz) {
        int lo = 0, hi = d.nb - 1;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (bc[mid] < c + d.first_vertex) lo = mid + 1; else hi = mid;
        }
        at = 32 * pivots + lo;
      }
      atomicOr(row + (at >> 5), 1u << (at & 31));
    }
  }
  sync_all();
  if (rank == 0) {
    if (chain) step_factor<C>(S, 0, panel_rows<C>(B, 0)[lane * B.xs]);
    __syncthreads();
    if constexpr (C > 1) {
      if (loader) step_tops<C>(S, 0);
      else
        for (int i = 32 * warp; i < 16 * B.UB; i += 32 * (nw - 1)) step_rows<C, true>(B, S, 0, i);
    }
  }
  sync_all();
  const int W = B.W;
  for (int P = 0; P < pivots; P++) {
    const bool next = P + 1 < pivots && (P + 1) % C == rank;
    if (chain) {
      if (next) step_chain<C, true>(B, S, P, 32 * (C == 1 ? nwk + 2 : nwk + 1));
    } else if (loader) {
      if constexpr (C == 1) {
        // (without a chain beside them the workers wait for the partnerless rows by barrier 3)
        step_tops<C>(S, P);
        __syncwarp();
        if (next) group_arrive(1, 32 * (nwk + 2));
        else group_arrive(3, 32 * (nwk + 1));
      }
    } else {
      if constexpr (C == 1) {
        if (!next) group_sync(3, 32 * (nwk + 1));
      }
      step_below<C, true>(B, S, P, panels - 1, next, rank, nwk);
      if (P % C == rank) {  // finished rows out
        const int rows = min(32, d.sz - 32 * P);
        const uint32_t* x = panel_rows<C>(B, P);
        const uint32_t* pu = S.pu + (size_t)32 * B.us * (P & 1);
        uint32_t* o = out + (size_t)32 * P * W;
        for (int r = warp - 1; r < rows; r += nwk) {
          uint32_t cnt = 0u;  // entries below the diagonal, and 2^16 times those above
          for (int c = lane; c < W; c += 32) {
            const uint32_t w =
                c < P ? x[r * B.xs + c] : (c == P ? S.pw[32 * (P & 1) + r] : pu[r * B.us + c - P - 1]);
            o[(size_t)r * W + c] = w;
            if (c < P) cnt += __popc(w);
            else if (c > P) cnt += __popc(w) << 16;
            else cnt += __popc(w & lt_mask(r)) + (__popc(w & gt_mask(r)) << 16);
          }
          cnt = __reduce_add_sync(FULL, cnt);
          if (lane == 0) {
            const int v = a.gid[d.first_vertex + 32 * P + r];
            a.row_nL[v] = (int)(cnt & 0xFFFFu);
            a.row_nU[v] = (int)(cnt >> 16) + 1;
          }
        }
      }
    }
    if constexpr (C > 1) {
      if (next) {
        __syncthreads();
        if (loader) step_tops<C>(S, P + 1);
        else
          for (int i = 32 * warp; i < 16 * words_right<true>(B, P + 1); i += 32 * (nw - 1))
            step_rows<C, true>(B, S, P + 1, i);
      }
    }
    sync_all();
  }
  // the rows above the block
  for (int i = warp; i < d.nr; i += nw) {
    const int q = pivots + (i >> 5);
    if (q % C != rank) continue;
    const uint32_t* row = panel_rows<C>(B, q) + (i & 31) * B.xs;
    uint32_t* o = out + (size_t)(32 * pivots + i) * W;
    int cnt = 0;
    for (int c = lane; c < W; c += 32) {
      const uint32_t w = row[c];
      o[c] = w;
      if (c < pivots) cnt += __popc(w);
    }
    cnt = __reduce_add_sync(FULL, cnt);
    if (lane == 0) a.piece_nL[d.br_base + i] = cnt;
  }
}

// ------------------------------------------------------------ counts and supernodes
// One CTA per group of rows (whole supernode chunks): nnz of every row of L and U, fill
// counts, T3 supernode flags (two phases per chunk, Section 5, Fig. 7: flag runs of rows
// with nnz(U(s,:)) = nnz(U(s-1,:)) - 1, then test L(s, r) != 0, here one bit), sums per
// group and per matrix.  The last CTA turns the group sums into offsets.
__global__ void band_count_kernel(BandArgs a) {
  extern __shared__ int32_t sm[];  // nnz(U) of the group's rows
  __shared__ unsigned long long s_tot[2];
  __shared__ int s_n, s_last;
  const long long g = blockIdx.x;
  const int m = a.mats ? mat_at(a, g, true) : 0;
  const BandMat d = a.mats ? a.mats[m] : a.one;
  const int wx = d.LB + d.UB + 1;
  const int i0 = (int)(g - d.group_base) * a.group_rows;
  const int rows = min(a.group_rows, d.n - i0);
  const uint32_t* bits = a.bits + d.bits_base + (size_t)i0 * wx;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (threadIdx.x == 0) {
    s_tot[0] = s_tot[1] = 0ull;
    s_n = 0;
  }
  __syncthreads();
  unsigned long long tl = 0ull, tu = 0ull;
  for (int r = warp; r < rows; r += nw) {
    const int i = i0 + r;
    int l = 0, u = 0;
    for (int c = lane; c < wx; c += 32) {
      const uint32_t w = bits[(size_t)r * wx + c];
      if (c < d.LB) l += __popc(w);
      else if (c > d.LB) u += __popc(w);
      else {
        l += __popc(w & lt_mask(i & 31));
        u += __popc(w & gt_mask(i & 31));
      }
    }
    l = __reduce_add_sync(FULL, l);
    u = __reduce_add_sync(FULL, u) + 1;
    if (lane == 0) {
      const long long row = d.row_base + i;
      sm[r] = u;
      a.row_nL[row] = l;
      a.row_nU[row] = u;
      a.fill[row] = l + u - a.fill[row];
      tl += l;
      tu += u;
    }
  }
  if (lane == 0) {
    atomicAdd(&s_tot[0], tl);
    atomicAdd(&s_tot[1], tu);
  }
  __syncthreads();
  int starts = 0;
  for (int r = threadIdx.x; r < rows; r += blockDim.x) {
    if (r % a.chunk != 0 && sm[r] == sm[r - 1] - 1) continue;  // not a leading row
    int lead = r;
    a.flags[d.row_base + i0 + r] = 1;
    starts++;
    for (int s = r + 1; s < rows && s % a.chunk != 0 && sm[s] == sm[s - 1] - 1; s++) {
      const int ri = i0 + lead, si = i0 + s;
      const int at = (ri >> 5) - (si >> 5) + d.LB;
      const bool has = at >= 0 && ((bits[(size_t)s * wx + at] >> (ri & 31)) & 1u);
      a.flags[d.row_base + si] = has ? 0 : 1;
      if (!has) {
        lead = s;
        starts++;
      }
    }
  }
  if (starts) atomicAdd(&s_n, starts);
  __syncthreads();
  if (threadIdx.x == 0) {
    a.part[3 * g] = (long long)s_tot[0];
    a.part[3 * g + 1] = (long long)s_tot[1];
    a.part[3 * g + 2] = s_n;
    if (a.mat_tot) {
      atomicAdd(&a.mat_tot[2 * m], s_tot[0]);
      atomicAdd(&a.mat_tot[2 * m + 1], s_tot[1]);
      atomicAdd(&a.mat_nsuper[m], s_n);
    }
    atomicAdd(&a.ctr->total_L, s_tot[0]);
    atomicAdd(&a.ctr->total_U, s_tot[1]);
    atomicAdd(&a.ctr->n_super, s_n);
    __threadfence();
    s_last = atomicAdd(&a.ctr->groups_done, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  // exclusive sums over the groups, a blockDim of groups at a time
  __threadfence();
  __shared__ long long sh[3][33];
  long long carry[3] = {0, 0, 0};
  for (long long g0 = 0; g0 < a.groups; g0 += blockDim.x) {
    const long long x = g0 + threadIdx.x;
#pragma unroll
    for (int f = 0; f < 3; f++) {
      const long long v = x < a.groups ? *(volatile long long*)&a.part[3 * x + f] : 0;
      long long s = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(FULL, s, o);
        if (lane >= o) s += y;
      }
      if (lane == 31) sh[f][warp] = s;
      __syncthreads();
      long long before = 0, all = 0;
      for (int k = 0; k < nw; k++) {
        if (k < warp) before += sh[f][k];
        all += sh[f][k];
      }
      if (x < a.groups) a.part[3 * x + f] = carry[f] + before + s - v;
      carry[f] += all;
      __syncthreads();
    }
  }
}

// ------------------------------------------------------------ column lists
// One CTA per group: row pointers, supernode starts, and the set bits of every row as
// columns, a word at a time (32 lanes, 32 bits: the writes of a word are consecutive).
__global__ void band_expand_kernel(BandArgs a) {
  extern __shared__ int32_t sm[];  // offsets of the group's rows in L, then in U
  __shared__ int s_w[3][33];
  const long long g = blockIdx.x;
  const int m = a.mats ? mat_at(a, g, true) : 0;
  const BandMat d = a.mats ? a.mats[m] : a.one;
  const int wx = d.LB + d.UB + 1;
  const int i0 = (int)(g - d.group_base) * a.group_rows;
  const int rows = min(a.group_rows, d.n - i0);
  const uint32_t* bits = a.bits + d.bits_base + (size_t)i0 * wx;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const long long L0 = a.part[3 * g], U0 = a.part[3 * g + 1], S0 = a.part[3 * g + 2];
  const long long Lm = a.part[3 * d.group_base], Um = a.part[3 * d.group_base + 1];
  int32_t* offL = sm;
  int32_t* offU = sm + a.group_rows;
  int64_t* lrp = a.L_rowptr + d.row_base + m;
  int64_t* urp = a.U_rowptr + d.row_base + m;
  int cl = 0, cu = 0, cs = 0;
  for (int r0 = 0; r0 < rows; r0 += blockDim.x) {
    const int r = r0 + threadIdx.x;
    const long long row = d.row_base + i0 + r;
    const int v[3] = {r < rows ? a.row_nL[row] : 0, r < rows ? a.row_nU[row] : 0, r < rows ? a.flags[row] : 0};
    int s[3];
#pragma unroll
    for (int f = 0; f < 3; f++) {
      s[f] = v[f];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, s[f], o);
        if (lane >= o) s[f] += y;
      }
      if (lane == 31) s_w[f][warp] = s[f];
    }
    __syncthreads();
    int all[3] = {0, 0, 0};
    for (int k = 0; k < nw; k++)
#pragma unroll
      for (int f = 0; f < 3; f++) {
        if (k < warp) s[f] += s_w[f][k];
        all[f] += s_w[f][k];
      }
    if (r < rows) {
      const int l = cl + s[0] - v[0], u = cu + s[1] - v[1];
      offL[r] = l;
      offU[r] = u;
      lrp[i0 + r] = L0 - Lm + l;
      urp[i0 + r] = U0 - Um + u;
      if (v[2]) a.super_start[S0 + m + cs + s[2] - 1] = i0 + r;
      if (i0 + r == d.n - 1) {
        lrp[d.n] = L0 - Lm + l + v[0];
        urp[d.n] = U0 - Um + u + v[1];
        a.super_start[S0 + m + cs + s[2]] = d.n;
      }
    }
    cl += all[0];
    cu += all[1];
    cs += all[2];
    __syncthreads();
  }
  const uint32_t lt = lt_mask(lane);
  for (int r = warp; r < rows; r += nw) {
    const int i = i0 + r;
    const int first = 32 * ((i >> 5) - d.LB);  // column of bit 0 of word 0
    int32_t* pl = a.L_colidx + L0 + offL[r];
    int32_t* pu = a.U_colidx + U0 + offU[r];
    const int own = d.LB;
    for (int c0 = 0; c0 < wx; c0 += 32) {
      const uint32_t mine = c0 + lane < wx ? bits[(size_t)r * wx + c0 + lane] : 0u;
      const int nc = min(32, wx - c0);
      unsigned any = __ballot_sync(FULL, mine != 0u);
      if (own >= c0 && own < c0 + nc) any |= 1u << (own - c0);
      while (any) {
        const int k = __ffs(any) - 1;
        any &= any - 1;
        const uint32_t w = __shfl_sync(FULL, mine, k);
        const int c = c0 + k;
        const int col = first + 32 * c + lane;
        uint32_t wl = c < own ? w : (c == own ? w & lt_mask(i & 31) : 0u);
        uint32_t wu = c > own ? w : (c == own ? (w & gt_mask(i & 31)) | (1u << (i & 31)) : 0u);
        if ((wl >> lane) & 1u) pl[__popc(wl & lt)] = col;
        pl += __popc(wl);
        if ((wu >> lane) & 1u) pu[__popc(wu & lt)] = col;
        pu += __popc(wu);
      }
    }
  }
}

// ------------------------------------------------------------ launchers
cudaError_t launch_band_scan(const BandArgs& a, cudaStream_t st) {
  long long grid = (a.rows + 255) / 256;
  if (grid > 4096) grid = 4096;
  band_scan_kernel<<<(int)grid, 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_band_reach(const BandArgs& a, bool counts, cudaStream_t st) {
  if (a.sampled <= 0) return cudaSuccess;
  const int words = reach_words(a.most_rows);
  const size_t smem = 4 * ((size_t)words + 2 * REACH_QUEUE);
  const cudaError_t e = cudaFuncSetAttribute(band_reach_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             4 * (REACH_WORDS + 2 * REACH_QUEUE));
  if (e != cudaSuccess) return e;
  band_reach_kernel<<<a.sampled * a.reach_rows + (a.cross ? 1 : 0), REACH_THREADS, smem, st>>>(a, counts, words);
  return cudaGetLastError();
}

namespace {
template <int C>
cudaError_t launch_elim(const BandArgs& a, int count, int threads, size_t smem, cudaStream_t st) {
  cudaError_t e =
      cudaFuncSetAttribute(band_elim_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, BAND_SMEM_MAX);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(count * C));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = C > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, band_elim_kernel<C>, a);
}
}  // namespace

cudaError_t launch_band_elim(const BandArgs& a, int count, int C, int threads, size_t smem, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  switch (C) {
    case 1: return launch_elim<1>(a, count, threads, smem, st);
    case 2: return launch_elim<2>(a, count, threads, smem, st);
    case 4: return launch_elim<4>(a, count, threads, smem, st);
    default: return launch_elim<8>(a, count, threads, smem, st);
  }
}

namespace {
template <int C>
cudaError_t launch_front(const FrontArgs& a, int count, int threads, size_t smem, cudaStream_t st) {
  cudaError_t e =
      cudaFuncSetAttribute(front_elim_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, BAND_SMEM_MAX);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(count * C));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = C > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, front_elim_kernel<C>, a);
}
}  // namespace

cudaError_t launch_front_elim(const FrontArgs& a, int count, int C, int threads, size_t smem, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  switch (C) {
    case 1: return launch_front<1>(a, count, threads, smem, st);
    case 2: return launch_front<2>(a, count, threads, smem, st);
    case 4: return launch_front<4>(a, count, threads, smem, st);
    default: return launch_front<8>(a, count, threads, smem, st);
  }
}

cudaError_t launch_band_count(const BandArgs& a, cudaStream_t st) {
  band_count_kernel<<<(unsigned)a.groups, 256, sizeof(int32_t) * (size_t)a.group_rows, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_band_expand(const BandArgs& a, cudaStream_t st) {
  band_expand_kernel<<<(unsigned)a.groups, 256, 2 * sizeof(int32_t) * (size_t)a.group_rows, st>>>(a);
  return cudaGetLastError();
}

}  // namespace gsofa
