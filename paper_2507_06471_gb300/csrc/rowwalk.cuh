// A warp's walk over a contiguous range of the arcs of a CSR, with the row of
// every arc: work split by arcs instead of by rows.
//
// A split by rows gives a hub row of 4e5 arcs to one warp, a serial chain that
// the whole launch then waits for, and leaves most lanes of a warp idle on rows
// of a few arcs. Here every warp takes the same number of arcs. It finds the
// row of its first arc by a 32-way search of the offsets (5 dependent loads for
// 2^23 rows, once per warp), then goes on in tiles of 128 arcs (4 per lane, one
// 16-byte column load): the rows that start inside the tile are marked in
// shared memory and a running maximum turns the marks into the row of each arc.
// Sum over the arcs inside communities, R-MAT scale 23 (2.6e8 arcs): 6.57 ms
// with a warp per row, 1.05 ms so (0.78 ms is what gathering 2.6e8 labels from
// L2 takes by itself, at one 32-byte sector per clock and SM).
#pragma once
#include "common.cuh"

namespace cd {

constexpr int WALK_TILE = 128;  // arcs per step of a warp

constexpr int WALK_MAX = 4096;  // arcs per piece at most

// Arcs per piece (a multiple of WALK_TILE) for m arcs over `warps` warps, which
// take pieces round robin: four pieces a warp even out the parts of the graph
// whose rows are short (more offsets a tile) without many searches.
__host__ __device__ inline int64_t walk_piece(int64_t m, int64_t warps) {
  const int64_t tiles = (m + WALK_TILE - 1) / WALK_TILE;
  const int64_t per = (tiles + 4 * warps - 1) / (4 * warps);
  return (per < 1 ? 1 : per < WALK_MAX / WALK_TILE ? per : WALK_MAX / WALK_TILE) * WALK_TILE;
}

// The row of arc e (off[r] <= e < off[r + 1]); 0 <= e < off[n]. All lanes take part.
__device__ __forceinline__ int64_t warp_row_of(const int64_t* __restrict__ off, int64_t n, int64_t e) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = n;  // off[lo] <= e < off[hi]
  while (hi - lo > 1) {
    const int64_t step = (hi - lo + 31) >> 5;
    const int64_t p = lo + (lane + 1) * step;
    const unsigned below = __ballot_sync(FULL, p < hi && off[p] <= e);
    lo += __popc(below) * step;  // the offsets never decrease: the lanes below are a prefix
    hi = hi < lo + step ? hi : lo + step;
  }
  return lo;
}

// Rows of the tile's arcs ts + 4 lane + j, j = 0..3, into row[]; `cur` is the
// row of arc ts - 1 or ts and becomes that of the tile's last arc. `mark` is
// the warp's own WALK_TILE words (16-byte aligned). Rows of arcs at or past
// off[n] are meaningless.
__device__ __forceinline__ void warp_tile_rows(const int64_t* __restrict__ off, int64_t n, int64_t ts, int64_t& cur,
                                               int32_t* mark, int64_t row[4]) {
  const int lane = threadIdx.x & 31;
  *reinterpret_cast<int4*>(mark + 4 * lane) = make_int4(0, 0, 0, 0);
  __syncwarp();
  // Rows that start inside the tile. Empty rows share an offset: the last of
  // them wins. o < 0 only where the offsets decrease, which
  // cd_modularity_noalloc finds out in the same launch.
  bool more;
  {
    const int64_t j = cur + 1 + lane;
    const int64_t o = j < n ? off[j] - ts : WALK_TILE;
    const bool in = o >= 0 && o < WALK_TILE;
    if (in) atomicMax(&mark[o], 1 + lane);
    more = __all_sync(FULL, in);
  }
  for (int64_t nr = cur + 33; more; nr += 128) {  // short rows: 4 independent loads a lane
    if (nr > cur + 33 + 512) {  // a long run of empty rows (millions in a coarse R-MAT graph): search instead
      for (int j = 0; j < 4; ++j) {
        int64_t lo = cur, hi = n;  // off[lo] <= e < off[hi]
        const int64_t e = ts + 4 * lane + j;
        while (hi - lo > 1) {
          const int64_t mid = (lo + hi) >> 1;
          if (off[mid] <= e) lo = mid;
          else hi = mid;
        }
        row[j] = lo;
      }
      cur = __shfl_sync(FULL, (long long)row[3], 31);
      __syncwarp();  // as below: lanes have written marks, and shuffles order no memory
      return;
    }
    int64_t o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t j = nr + 32 * q + lane;
      o[q] = j < n ? off[j] - ts : WALK_TILE;
    }
    bool in = true;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      in = in && o[q] >= 0 && o[q] < WALK_TILE;
      if (in) atomicMax(&mark[o[q]], (int32_t)(nr - cur) + 32 * q + lane);
    }
    more = __all_sync(FULL, in);
  }
  __syncwarp();
  const int4 m = *reinterpret_cast<const int4*>(mark + 4 * lane);
  const int32_t a0 = m.x, a1 = max(a0, m.y), a2 = max(a1, m.z), a3 = max(a2, m.w);
  int32_t inc = a3;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(FULL, inc, o);
    if (lane >= o) inc = max(inc, y);
  }
  int32_t before = __shfl_up_sync(FULL, inc, 1);
  if (lane == 0) before = 0;
  row[0] = cur + max(before, a0);
  row[1] = cur + max(before, a1);
  row[2] = cur + max(before, a2);
  row[3] = cur + max(before, a3);
  cur += __shfl_sync(FULL, inc, 31);
  __syncwarp();  // the marks are cleared for the next tile
}

// The rows of the arcs ts + lane + 32 j, j = 0..3 (for stores that run along
// the lanes): warp_tile_rows, then a pass through the marks.
__device__ __forceinline__ void warp_tile_rows_strided(const int64_t* __restrict__ off, int64_t n, int64_t ts,
                                                       int64_t& cur, int32_t* mark, int64_t row[4]) {
  const int lane = threadIdx.x & 31;
  const int64_t base = cur;
  int64_t r[4];
  warp_tile_rows(off, n, ts, cur, mark, r);
  *reinterpret_cast<int4*>(mark + 4 * lane) =
      make_int4((int32_t)(r[0] - base), (int32_t)(r[1] - base), (int32_t)(r[2] - base), (int32_t)(r[3] - base));
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 4; ++j) row[j] = base + mark[lane + 32 * j];
  __syncwarp();
}

// emit(r, sum) once for every row r with arcs among the tile's (a row that goes
// on past the tile is emitted by each tile): the sum of val[] over the lanes'
// arcs of that row. Rows are as warp_tile_rows gave them (never decreasing over
// 4 lane + j); a lane's arcs past the end have the row -1 and val 0.
template <class F>
__device__ __forceinline__ void warp_rows_sum(const int64_t row[4], const unsigned long long val[4], F emit) {
  const int lane = threadIdx.x & 31;
  unsigned long long head = 0, tail = val[0];
#pragma unroll
  for (int j = 1; j < 4; ++j) {
    if (row[j] != row[j - 1]) {
      if (row[j - 1] == row[0]) head = tail;  // the lane's first row may have come in from the lane before
      else emit(row[j - 1], tail);
      tail = 0;
    }
    tail += val[j];
  }
  // tail: the lane's last row; segmented running sum over the lanes it spans
  const int64_t before = __shfl_up_sync(FULL, (long long)row[3], 1);
  const bool joined = lane > 0 && before == row[0];
  int open = joined && row[0] == row[3];  // the whole lane continues the lane before
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(FULL, tail, o);
    const int oy = __shfl_up_sync(FULL, open, o);
    if (lane >= o && open) {
      tail += y;
      open = oy;
    }
  }
  const unsigned long long carry = __shfl_up_sync(FULL, tail, 1);
  const int64_t after = __shfl_down_sync(FULL, (long long)row[0], 1);
  if (row[0] != row[3] && row[0] >= 0) emit(row[0], head + (joined ? carry : 0));
  if (row[3] >= 0 && (lane == 31 || after != row[3])) emit(row[3], tail);
}

// Sums by key of one CTA, added to a global array at the end: a popular key (a
// large community) then takes one global atomic per CTA instead of one per
// addition. Atomics on one address run one after another: 1e5 vertices in about
// a hundred communities took 44.6 us with an atomic per vertex. A key that finds
// no slot within four probes is added to the global array at once.
struct CtaSums {
  static constexpr int SLOTS = 512;
  uint32_t lo[SLOTS], hi[SLOTS];
  int32_t key[SLOTS];
  __device__ __forceinline__ void clear() {  // then __syncthreads()
    for (int i = threadIdx.x; i < SLOTS; i += blockDim.x) {
      key[i] = EMPTY;
      lo[i] = hi[i] = 0;
    }
  }
  // The slot the sum went to, -1: straight to the global array.
  __device__ __forceinline__ int add(unsigned long long* global, int32_t k, unsigned long long x) {
    unsigned h = ((uint32_t)k * 2654435761u) >> 23;
    for (int probe = 0; probe < 4; ++probe) {
      int32_t c = *(volatile int32_t*)&key[h];
      if (c == EMPTY) c = atomicCAS(&key[h], EMPTY, k);
      if (c == EMPTY || c == k) {
        add_words(&lo[h], &hi[h], x);
        return (int)h;
      }
      h = (h + 1) & (SLOTS - 1);
    }
    atomicAdd(&global[k], x);
    return -1;
  }
  __device__ __forceinline__ void flush(unsigned long long* global) {  // after __syncthreads()
    for (int i = threadIdx.x; i < SLOTS; i += blockDim.x)
      if (key[i] != EMPTY) atomicAdd(&global[key[i]], ((unsigned long long)hi[i] << 32) | lo[i]);
  }
};
static_assert(CtaSums::SLOTS == 512, "the hash keeps the top 9 bits");

}  // namespace cd
