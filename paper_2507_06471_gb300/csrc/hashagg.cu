// Louvain aggregation by hashing (Algorithm 3, Aggregation): the coarse graph
// without a sort.
//
// 1. A pass over the vertices notes each one's coarse vertex A = new(C[v]) and
//    sums the arcs and deg_w of every A; a scan of the arc sums gives each
//    community a contiguous segment of the arc space, and a second pass gives
//    every member its place in the segment (any order: nothing depends on it).
// 2. Every arc u->x of a member u writes (new(C[x]), w) into its place. The arcs
//    are split evenly over the warps and taken in the graph's own order, so the
//    columns are read and the segments written in runs (rowwalk.cuh).
// 3. Each segment is combined by its keys: up to 8 or 32 arcs by as many lanes
//    (a match, no table), up to 256 by a warp and up to AG_MID_MAX and AG_CTA_MAX
//    by CTAs of 128 and 512 threads with a shared-memory table (512 threads for a
//    few hundred arcs are mostly barriers: 1.58 ms of the case below with one
//    size, 1.07 + 0.27 with two); a larger segment is cut into AG_CHUNK-arc chunks,
//    each combined in shared memory, whose distinct entries are then merged in a
//    global table sized for the segment. The distinct (B, sum w) of a segment
//    are written back at its start.
// 4. The segments are compacted into the coarse CSR (k rows, columns in no
//    particular order; (A, A) collects every arc inside A, i.e. twice its
//    internal weight, the internal convention for loops).
//
// When vol(V) < 2^31 every weight and sum fits in 32 bits: the segments, the
// tables (one 64-bit word a slot, one atomic a merge) and the coarse weights are
// 32-bit then, 64-bit otherwise.
//
// Measured, R-MAT 22 weighted (1.3e8 arcs, 4.2e6 -> 2.7e6 vertices): a radix sort
// of the vertices, a warp per member row and per community, 12 bytes an arc and
// an ingest of the coarse arcs took 16.3 ms; this takes 4.4.
//
// The content of every row equals that of the sort-based aggregation; only the
// order of columns inside a row differs, and no later step depends on it.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "rowwalk.cuh"

namespace cd {
namespace {

constexpr int NT = 256;
constexpr int NW = NT / 32;
constexpr int AG_WARP_MAX = 256;   // arcs of a segment combined by one warp (512-slot table)
constexpr int AG_MID_MAX = 1024;   // by a CTA of 128 threads (2048-slot table)
constexpr int AG_CTA_MAX = 4096;   // by one of 512 (8192-slot table)
constexpr int AG_CHUNK = 4096;     // arcs per chunk of a larger segment
constexpr int AG_WCAP = 2 * AG_WARP_MAX;
constexpr int AG_SLICE = 1024;     // global-table slots per extraction item (tables are multiples)
constexpr int32_t AG_EMPTY = -1;
constexpr unsigned long long AG_EMPTY_SLOT = ~0ull;

// Counts on the device: segments per class, chunks, slots of the global tables.
enum { AC_T8 = 0, AC_T32, AC_WARP, AC_MID, AC_CTA, AC_BIG, AC_CHUNKS, AC_SLOTS, AC_N };
constexpr int AC_LISTS = 6;  // the first ones have a list of segments each

unsigned gcap(int64_t blocks, int64_t cap = 152 * 16) {
  if (blocks < 1) blocks = 1;
  return (unsigned)(blocks < cap ? blocks : cap);
}

__device__ __forceinline__ unsigned lg_for(int64_t x) {  // smallest lg >= 1 with 2^lg >= x
  return x <= 2 ? 1 : 64 - __clzll((unsigned long long)(x - 1));
}

// ------------------------------------------------------------------ steps 1-2

__global__ void __launch_bounds__(NT) k_ag_vertex(const int32_t* __restrict__ labels, const int32_t* __restrict__ newid,
                                                  const int64_t* __restrict__ off, const int64_t* __restrict__ degw,
                                                  int64_t n, int32_t* __restrict__ nl, unsigned long long* arcs,
                                                  unsigned long long* cdegw) {
  __shared__ CtaSums sa, sd;
  sa.clear();
  sd.clear();
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * NT;
  for (int64_t v = (int64_t)blockIdx.x * NT + threadIdx.x; v < n; v += stride) {
    const int32_t a = newid[labels[v]];
    const int64_t d = off[v + 1] - off[v];
    nl[v] = a;
    if (d > 0) {
      sa.add(arcs, a, (unsigned long long)d);
      sd.add(cdegw, a, (unsigned long long)degw[v]);
    }
  }
  __syncthreads();
  sa.flush(arcs);
  sd.flush(cdegw);
}

// delta[v] = (place of v's first arc in the segments) - off[v]. The members of
// one community that meet in a CTA take their places from one global atomic.
constexpr int AP_VERTS = 8 * NT;  // vertices per step of a CTA
__global__ void __launch_bounds__(NT) k_ag_place(const int32_t* __restrict__ nl, const int64_t* __restrict__ off,
                                                 int64_t n, const int64_t* __restrict__ sstart,
                                                 unsigned long long* taken, int64_t* __restrict__ delta) {
  constexpr int SLOTS = 1024;
  __shared__ uint32_t tot[SLOTS];  // 32-bit shared atomics: 64-bit ones take 25 times as long
  __shared__ unsigned long long base[SLOTS];
  __shared__ int32_t key[SLOTS];
  for (int64_t v0 = (int64_t)blockIdx.x * AP_VERTS; v0 < n; v0 += (int64_t)gridDim.x * AP_VERTS) {
    for (int i = threadIdx.x; i < SLOTS; i += NT) {
      key[i] = AG_EMPTY;
      tot[i] = 0;
    }
    __syncthreads();
    int32_t a[8];
    int16_t slot[8];
    unsigned long long at[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int64_t v = v0 + q * NT + threadIdx.x;
      a[q] = v < n ? nl[v] : -1;
      at[q] = v < n ? (unsigned long long)(off[v + 1] - off[v]) : 0;
      if (at[q] == 0) a[q] = -1;  // an isolated vertex has no place
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      slot[q] = -1;
      if (a[q] < 0) continue;
      unsigned h = ((uint32_t)a[q] * 2654435761u) >> 22;
      for (int probe = 0; probe < 4 && at[q] < (1u << 21); ++probe) {  // 2,048 such degrees stay below 2^32
        int32_t c = *(volatile int32_t*)&key[h];
        if (c == AG_EMPTY) c = atomicCAS(&key[h], AG_EMPTY, a[q]);
        if (c == AG_EMPTY || c == a[q]) {
          slot[q] = (int16_t)h;
          break;
        }
        h = (h + 1) & (SLOTS - 1);
      }
      if (slot[q] >= 0) at[q] = atomicAdd(&tot[slot[q]], (uint32_t)at[q]);
      else at[q] = atomicAdd(&taken[a[q]], at[q]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < SLOTS; i += NT)
      if (key[i] != AG_EMPTY) base[i] = atomicAdd(&taken[key[i]], (unsigned long long)tot[i]);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int64_t v = v0 + q * NT + threadIdx.x;
      if (a[q] < 0) continue;
      delta[v] = sstart[a[q]] + (int64_t)(at[q] + (slot[q] >= 0 ? base[slot[q]] : 0)) - off[v];
    }
    __syncthreads();
  }
}

// The arcs into their segments.
template <class W, class V>
__global__ void __launch_bounds__(NT) k_ag_scatter(const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                                                   const void* w, int64_t n, int64_t m, int64_t piece,
                                                   const int32_t* __restrict__ nl, const int64_t* __restrict__ delta,
                                                   int32_t* __restrict__ ab, V* __restrict__ aw) {
  __shared__ __align__(16) int32_t mark[NW][WALK_TILE];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t step = (((int64_t)gridDim.x * NT) >> 5) * piece;
  for (int64_t e0 = (((int64_t)blockIdx.x * NT + threadIdx.x) >> 5) * piece; e0 < m; e0 += step) {  // uniform in the warp
    const int64_t e1 = e0 + piece < m ? e0 + piece : m;
    int32_t bn[4];  // columns a tile ahead
#pragma unroll
    for (int j = 0; j < 4; ++j) bn[j] = e0 + lane + 32 * j < e1 ? __ldg(cols + e0 + lane + 32 * j) : -1;
    int64_t cur = warp_row_of(off, n, e0);
    for (int64_t ts = e0; ts < e1; ts += WALK_TILE) {
      int32_t b[4];
      V x[4];
      int64_t row[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t e = ts + lane + 32 * j;
        b[j] = bn[j];
        bn[j] = e + WALK_TILE < e1 ? __ldg(cols + e + WALK_TILE) : -1;
        x[j] = e < e1 ? (V)W::get(w, e) : 0;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = b[j] >= 0 ? nl[b[j]] : -1;
      warp_tile_rows_strided(off, n, ts, cur, mark[wid], row);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t e = ts + lane + 32 * j;
        if (e >= e1) continue;
        const int64_t p = delta[row[j]] + e;
        ab[p] = b[j];
        aw[p] = x[j];
      }
    }
  }
}

// ------------------------------------------------------------------ classes

// The segments into their classes' lists; a CTA appends to each list once per step.
constexpr int AF_SEGS = 8 * NT;
__global__ void __launch_bounds__(NT) k_ag_classes(const int64_t* __restrict__ sstart, int64_t k,
                                                   unsigned long long* cnt, int32_t* __restrict__ t8,
                                                   int32_t* __restrict__ t32, int32_t* __restrict__ wl,
                                                   int32_t* __restrict__ ml, int32_t* __restrict__ cl,
                                                   int32_t* __restrict__ ll,
                                                   int32_t* __restrict__ ch_seg, int64_t* __restrict__ ch_off) {
  __shared__ int n_of[8];
  __shared__ unsigned long long base[8];
  const int lane = threadIdx.x & 31;
  for (int64_t a0 = (int64_t)blockIdx.x * AF_SEGS; a0 < k; a0 += (int64_t)gridDim.x * AF_SEGS) {
    if (threadIdx.x < 8) n_of[threadIdx.x] = 0;
    __syncthreads();
    int8_t cls[8];
    int16_t rank[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int64_t a = a0 + q * NT + threadIdx.x;
      const int64_t len = a < k ? sstart[a + 1] - sstart[a] : 0;
      cls[q] = len == 0 ? -1 : len <= 8 ? AC_T8 : len <= 32 ? AC_T32 : len <= AG_WARP_MAX ? AC_WARP
             : len <= AG_MID_MAX ? AC_MID : len <= AG_CTA_MAX ? AC_CTA : AC_BIG;
      rank[q] = 0;
#pragma unroll
      for (int c = 0; c < AC_LISTS; ++c) {
        const unsigned m = __ballot_sync(FULL, cls[q] == c);
        if (!m) continue;
        int p = 0;
        if (lane == 0) p = atomicAdd(&n_of[c], __popc(m));
        p = __shfl_sync(FULL, p, 0);
        if (cls[q] == c) rank[q] = (int16_t)(p + __popc(m & ((1u << lane) - 1u)));
      }
      if (cls[q] == AC_BIG) {
        const int64_t nc = (len + AG_CHUNK - 1) / AG_CHUNK;
        const unsigned long long p = atomicAdd(&cnt[AC_CHUNKS], (unsigned long long)nc);
        for (int64_t j = 0; j < nc; ++j) {
          ch_seg[p + j] = (int32_t)a;
          ch_off[p + j] = j * AG_CHUNK;
        }
      }
    }
    __syncthreads();
    if (threadIdx.x < AC_LISTS && n_of[threadIdx.x]) base[threadIdx.x] = atomicAdd(&cnt[threadIdx.x], (unsigned long long)n_of[threadIdx.x]);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (cls[q] < 0) continue;
      int32_t* list = cls[q] == AC_T8 ? t8 : cls[q] == AC_T32 ? t32 : cls[q] == AC_WARP ? wl
                    : cls[q] == AC_MID ? ml : cls[q] == AC_CTA ? cl : ll;
      list[base[cls[q]] + rank[q]] = (int32_t)(a0 + q * NT + threadIdx.x);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ shared-memory combining

// Open addressing in a 2^lg-slot table holding at most half that many keys,
// so a free slot is always found. A probe is a load; only an empty slot is
// claimed with a compare-and-swap, and joins the occupied list.
template <class V>
__device__ __forceinline__ void tab_insert(int32_t* keys, V* vals, uint16_t* occ, int* occ_n,
                                           unsigned lg, int32_t key, V w) {
  const unsigned mask = (1u << lg) - 1u;
  unsigned h = ((uint32_t)key * 2654435761u) >> (32 - lg);
  for (unsigned probe = 0; probe <= mask; ++probe) {
    int32_t c = *(volatile int32_t*)&keys[h];
    if (c == AG_EMPTY) {
      c = atomicCAS(&keys[h], AG_EMPTY, key);
      if (c == AG_EMPTY) {
        occ[atomicAdd(occ_n, 1)] = (uint16_t)h;
        c = key;
      }
    }
    if (c == key) {
      atomicAdd(&vals[h], w);
      return;
    }
    h = (h + 1) & mask;
  }
}

// TW lanes per segment of at most TW arcs: equal keys meet by a match, and the
// first lane of each writes the sum.
template <int TW, class V>
__device__ __forceinline__ void tile_segments(const int64_t* __restrict__ sstart, const int32_t* __restrict__ list,
                                              int64_t count, int64_t warp, int64_t nwarps, int32_t* ab, V* aw,
                                              V* stage, int64_t* ucnt) {
  const int lane = threadIdx.x & 31;
  const int sub = lane & (TW - 1), tbase = lane - sub;
  const unsigned tmask = (TW == 32 ? FULL : ((1u << (TW & 31)) - 1u)) << tbase;
  constexpr int PER = 32 / TW;
  for (int64_t q0 = warp * PER; q0 < count; q0 += nwarps * PER) {  // uniform in the warp
    const int64_t q = q0 + lane / TW;
    int64_t p = 0;
    int len = 0;
    int32_t a = 0;
    if (q < count) {
      a = list[q];
      p = sstart[a];
      len = (int)(sstart[a + 1] - p);
    }
    const bool ok = sub < len;
    const int32_t key = ok ? ab[p + sub] : (int32_t)(0x80000000u | (unsigned)lane);
    const V w = ok ? aw[p + sub] : 0;
    const unsigned peers = __match_any_sync(FULL, key) & tmask;
    const int lead = __ffs(peers) - 1;
    stage[lane] = 0;
    __syncwarp();
    if (ok) atomicAdd(&stage[lead], w);
    __syncwarp();
    const unsigned leads = __ballot_sync(FULL, ok && lead == lane) & tmask;
    if (ok && lead == lane) {
      const int r = __popc(leads & ((1u << lane) - 1u));
      ab[p + r] = key;
      aw[p + r] = stage[lane];
    }
    if (sub == 0 && q < count) ucnt[a] = __popc(leads);
    __syncwarp();
  }
}

// Segments of at most AG_WARP_MAX arcs: combine, write the distinct entries
// back at the segment start and record their number.
template <class V> constexpr size_t ag_warp_smem() { return (size_t)NW * AG_WCAP * (sizeof(V) + 4 + 2); }
template <class V>
__global__ void __launch_bounds__(NT) k_ag_warp(const int64_t* __restrict__ sstart, const int32_t* __restrict__ t8,
                                                const int32_t* __restrict__ t32, const int32_t* __restrict__ wl,
                                                const unsigned long long* __restrict__ cnt, int32_t* ab, V* aw,
                                                int64_t* __restrict__ ucnt) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  V* vals = (V*)smem + (size_t)wid * AG_WCAP;
  int32_t* keys = (int32_t*)(smem + (size_t)NW * AG_WCAP * sizeof(V)) + (size_t)wid * AG_WCAP;
  uint16_t* occ = (uint16_t*)(smem + (size_t)NW * AG_WCAP * (sizeof(V) + 4)) + (size_t)wid * AG_WCAP;
  __shared__ int occ_n[NW];
  __shared__ V stage[NW][32];
  for (int j = lane; j < AG_WCAP; j += 32) {
    keys[j] = AG_EMPTY;
    vals[j] = 0;
  }
  if (lane == 0) occ_n[wid] = 0;
  __syncwarp();
  const int64_t warp = ((int64_t)blockIdx.x * NT + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * NT) >> 5;
  const int64_t nw = (int64_t)cnt[AC_WARP];
  for (int64_t q = warp; q < nw; q += nwarps) {
    const int32_t a = wl[q];
    const int64_t p = sstart[a];
    const int len = (int)(sstart[a + 1] - p);
    const unsigned lg = lg_for(2 * len);
    for (int j0 = lane; j0 < len; j0 += 128) {
      int32_t key[4];
      V w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool ok = j0 + 32 * u < len;
        key[u] = ok ? ab[p + j0 + 32 * u] : AG_EMPTY;
        w[u] = ok ? aw[p + j0 + 32 * u] : 0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (key[u] != AG_EMPTY) tab_insert(keys, vals, occ, &occ_n[wid], lg, key[u], w[u]);
    }
    __syncwarp();
    const int nocc = occ_n[wid];
    for (int j = lane; j < nocc; j += 32) {
      const int slot = occ[j];
      ab[p + j] = keys[slot];
      aw[p + j] = vals[slot];
      keys[slot] = AG_EMPTY;
      vals[slot] = 0;
    }
    __syncwarp();
    if (lane == 0) {
      ucnt[a] = nocc;
      occ_n[wid] = 0;
    }
    __syncwarp();
  }
  tile_segments<32, V>(sstart, t32, (int64_t)cnt[AC_T32], warp, nwarps, ab, aw, stage[wid], ucnt);
  tile_segments<8, V>(sstart, t8, (int64_t)cnt[AC_T8], warp, nwarps, ab, aw, stage[wid], ucnt);
}

// CTA of TH threads per block of up to MAX arcs: first (with 512 threads) the
// chunks of the large segments (a chunk's distinct count goes to dch and to the
// segment's upper bound ub), then the whole segments of `list`.
template <class V, int MAX> constexpr size_t ag_cta_smem() { return (size_t)2 * MAX * (sizeof(V) + 4 + 2); }
template <class V, int TH, int MAX, int CLASS>
__global__ void __launch_bounds__(TH) k_ag_cta(const int64_t* __restrict__ sstart, const int32_t* __restrict__ cl,
                                               const int32_t* __restrict__ ch_seg, const int64_t* __restrict__ ch_off,
                                               const unsigned long long* __restrict__ cnt, int32_t* ab, V* aw,
                                               int64_t* __restrict__ ucnt, int32_t* __restrict__ dch,
                                               unsigned long long* __restrict__ ub) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int AG_CNT = TH, AG_CCAP = 2 * MAX;
  V* vals = (V*)smem;
  int32_t* keys = (int32_t*)(smem + (size_t)AG_CCAP * sizeof(V));
  uint16_t* occ = (uint16_t*)(smem + (size_t)AG_CCAP * (sizeof(V) + 4));
  __shared__ int occ_n;
  const int64_t nch = CLASS == AC_CTA ? (int64_t)cnt[AC_CHUNKS] : 0, items = nch + (int64_t)cnt[CLASS];
  if (blockIdx.x >= items) return;
  for (int j = threadIdx.x; j < AG_CCAP; j += AG_CNT) {
    keys[j] = AG_EMPTY;
    vals[j] = 0;
  }
  if (threadIdx.x == 0) occ_n = 0;
  __syncthreads();
  for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const bool chunk = it < nch;
    const int32_t a = chunk ? ch_seg[it] : cl[it - nch];
    int64_t p = sstart[a], left = sstart[a + 1] - p;
    if (chunk) {
      p += ch_off[it];
      left -= ch_off[it];
    }
    const int len = left < MAX ? (int)left : MAX;
    const unsigned lg = lg_for(2 * len);
    for (int j0 = threadIdx.x; j0 < len; j0 += 4 * AG_CNT) {
      int32_t key[4];
      V w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool ok = j0 + AG_CNT * u < len;
        key[u] = ok ? ab[p + j0 + AG_CNT * u] : AG_EMPTY;
        w[u] = ok ? aw[p + j0 + AG_CNT * u] : 0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (key[u] != AG_EMPTY) tab_insert(keys, vals, occ, &occ_n, lg, key[u], w[u]);
    }
    __syncthreads();  // every entry read and inserted before the block is overwritten
    const int nocc = occ_n;
    for (int j = threadIdx.x; j < nocc; j += AG_CNT) {
      const int slot = occ[j];
      ab[p + j] = keys[slot];
      aw[p + j] = vals[slot];
      keys[slot] = AG_EMPTY;
      vals[slot] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      if (chunk) {
        dch[it] = nocc;
        atomicAdd(&ub[a], (unsigned long long)nocc);
      } else {
        ucnt[a] = nocc;
      }
      occ_n = 0;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ large segments

// Global table of a large segment: 2^lg >= 2 x (its upper bound of distinct
// keys) slots, at least AG_SLICE, placed at toff[a].
__global__ void k_ag_tables_size(const int32_t* __restrict__ ll, const unsigned long long* __restrict__ ub,
                                 int32_t* __restrict__ tlg, int64_t* __restrict__ toff, unsigned long long* cnt) {
  const int64_t nl = (int64_t)cnt[AC_BIG];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nl; q += stride) {
    const int32_t a = ll[q];
    unsigned lg = lg_for(2 * (int64_t)ub[a]);
    if (lg < 10) lg = 10;  // AG_SLICE
    tlg[a] = (int32_t)lg;
    toff[a] = (int64_t)atomicAdd(&cnt[AC_SLOTS], 1ull << lg);
  }
}

// A table's slices are owned by its segment.
__global__ void k_ag_tables_own(const int32_t* __restrict__ ll, int64_t nl, const int32_t* __restrict__ tlg,
                                const int64_t* __restrict__ toff, int32_t* __restrict__ owner) {
  for (int64_t q = blockIdx.x; q < nl; q += gridDim.x) {
    const int32_t a = ll[q];
    const int64_t s0 = toff[a] / AG_SLICE, ns = ((int64_t)1 << tlg[a]) / AG_SLICE;
    for (int64_t j = threadIdx.x; j < ns; j += blockDim.x) owner[s0 + j] = a;
  }
}

// CTA per chunk: its distinct entries into the segment's global table. 32-bit
// weights: a slot is one word (key << 32 | weight), claimed with its weight or
// added to with one atomic; the sums stay below 2^31, so the weight never
// carries into the key. 64-bit weights: key and weight in two arrays.
//
// The rows of the coarse graph come out in the order of these tables, so their
// hash must have nothing in common with that of the shared-memory tables that
// read such rows in chunks (smem_insert: the golden ratio's multiplier). With the
// golden ratio here too, 4,096 columns in a row had a few hundred homes at most
// among 8,192 slots, and an insert walked past hundreds. The hub builds of the
// first round with labels on R-MAT 26's coarse graph: 260 ms so, 152 with the rows
// extracted 32 slots at a time by whichever warp comes, 64 with SplitMix64's
// output function. (Another multiplier alone is as fast, but keys that are
// neighbours under one multiplier differ by few values, which crowd as well.)
__device__ __forceinline__ uint64_t merge_home(int32_t key, unsigned lg) {
  uint64_t z = (uint32_t)key;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return (z ^ (z >> 31)) >> (64 - lg);
}
template <class V>
__global__ void __launch_bounds__(NT) k_ag_merge(const int64_t* __restrict__ sstart, const int32_t* __restrict__ ch_seg,
                                                 const int64_t* __restrict__ ch_off, const int32_t* __restrict__ dch,
                                                 int64_t nch, const int32_t* __restrict__ ab,
                                                 const V* __restrict__ aw,
                                                 const int32_t* __restrict__ tlg, const int64_t* __restrict__ toff,
                                                 unsigned long long* gs, int32_t* gk) {
  for (int64_t it = blockIdx.x; it < nch; it += gridDim.x) {
    const int32_t a = ch_seg[it];
    const int64_t p = sstart[a] + ch_off[it];
    const int d = dch[it];
    const unsigned lg = (unsigned)tlg[a];
    const uint64_t mask = ((uint64_t)1 << lg) - 1;
    unsigned long long* slots = gs + toff[a];
    for (int j = threadIdx.x; j < d; j += NT) {
      const int32_t key = ab[p + j];
      const V w = aw[p + j];
      uint64_t h = merge_home(key, lg);
      for (uint64_t probe = 0; probe <= mask; ++probe) {
        if constexpr (sizeof(V) == 4) {
          const unsigned long long mine = ((unsigned long long)(uint32_t)key << 32) | w;
          unsigned long long c = *(volatile unsigned long long*)&slots[h];
          if (c == AG_EMPTY_SLOT) c = atomicCAS(&slots[h], AG_EMPTY_SLOT, mine);
          if (c == AG_EMPTY_SLOT) break;
          if ((int32_t)(c >> 32) == key) {
            atomicAdd(&slots[h], (unsigned long long)w);
            break;
          }
        } else {
          const int32_t prev = atomicCAS(&gk[toff[a] + h], AG_EMPTY, key);
          if (prev == AG_EMPTY || prev == key) {
            atomicAdd(&slots[h], (unsigned long long)w);
            break;
          }
        }
        h = (h + 1) & mask;
      }
    }
  }
}

// CTA per AG_SLICE slots of the global tables: the live entries go back into
// their segment (in any order).
template <class V>
__global__ void __launch_bounds__(NT) k_ag_extract(const int32_t* __restrict__ owner, int64_t nslices,
                                                   const unsigned long long* __restrict__ gs, const int32_t* __restrict__ gk,
                                                   const int64_t* __restrict__ sstart, int32_t* ab,
                                                   V* aw, int64_t* ucnt) {
  __shared__ int n_live;
  __shared__ unsigned long long base;
  const int lane = threadIdx.x & 31;
  constexpr int PER = AG_SLICE / NT;
  for (int64_t sl = blockIdx.x; sl < nslices; sl += gridDim.x) {
    const int32_t a = owner[sl];
    const int64_t p = sstart[a];
    if (threadIdx.x == 0) n_live = 0;
    __syncthreads();
    int32_t key[PER];
    V w[PER];
    int at[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int64_t slot = sl * AG_SLICE + q * NT + threadIdx.x;
      const unsigned long long x = gs[slot];
      if constexpr (sizeof(V) == 4) key[q] = x == AG_EMPTY_SLOT ? AG_EMPTY : (int32_t)(x >> 32);
      else key[q] = gk[slot];
      w[q] = (V)x;
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const unsigned bal = __ballot_sync(FULL, key[q] != AG_EMPTY);
      int b = 0;
      if (lane == 0 && bal) b = atomicAdd(&n_live, __popc(bal));
      at[q] = __shfl_sync(FULL, b, 0) + __popc(bal & ((1u << lane) - 1u));
    }
    __syncthreads();
    if (threadIdx.x == 0) base = n_live ? atomicAdd((unsigned long long*)&ucnt[a], (unsigned long long)n_live) : 0;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < PER; ++q)
      if (key[q] != AG_EMPTY) {
        ab[p + (int64_t)base + at[q]] = key[q];
        aw[p + (int64_t)base + at[q]] = w[q];
      }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ coarse CSR

// delta[A] = (start of A's segment) - (start of its coarse row); stat: the number
// of empty rows, the largest deg_w, the rows per degree bin and the hubs' arcs.
__global__ void __launch_bounds__(NT) k_ag_rows(const int64_t* __restrict__ sstart, const int64_t* __restrict__ coff,
                                                int64_t k, int64_t* __restrict__ delta, const unsigned long long* cdegw,
                                                int t_warp, int t_hub, unsigned long long* stat) {
  __shared__ unsigned long long s_max, s_hub;
  __shared__ int s_bin[NBINS + 1];  // [NBINS]: empty
  if (threadIdx.x <= NBINS) s_bin[threadIdx.x] = 0;
  if (threadIdx.x == 0) s_max = s_hub = 0;
  __syncthreads();
  unsigned long long mx = 0;
  const int64_t stride = (int64_t)gridDim.x * NT;
  for (int64_t a = (int64_t)blockIdx.x * NT + threadIdx.x; a < k; a += stride) {
    const int64_t c = coff[a], d = coff[a + 1] - c;
    delta[a] = sstart[a] - c;
    const int b = d == 0 ? NBINS : bin_of(d, t_warp, t_hub);
    atomicAdd(&s_bin[b], 1);
    if (b == B_HUB) atomicAdd(&s_hub, (unsigned long long)d);
    mx = cdegw[a] > mx ? cdegw[a] : mx;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(FULL, mx, o);
    mx = y > mx ? y : mx;
  }
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(&s_max, mx);
  __syncthreads();
  if (threadIdx.x < NBINS && s_bin[threadIdx.x]) atomicAdd(&stat[2 + threadIdx.x], (unsigned long long)s_bin[threadIdx.x]);
  if (threadIdx.x == 0) {
    if (s_bin[NBINS]) atomicAdd(&stat[0], (unsigned long long)s_bin[NBINS]);
    if (s_max) atomicMax(&stat[1], s_max);
    if (s_hub) atomicAdd(&stat[2 + NBINS], s_hub);
  }
}

// The distinct entries into the coarse rows, split evenly by entries.
template <class V, class WOUT>
__global__ void __launch_bounds__(NT) k_ag_compact(const int64_t* __restrict__ coff, int64_t k, int64_t nseg,
                                                   int64_t piece, const int64_t* __restrict__ delta,
                                                   const int32_t* __restrict__ ab, const V* __restrict__ aw,
                                                   int32_t* __restrict__ ccols, WOUT* __restrict__ cw) {
  __shared__ __align__(16) int32_t mark[NW][WALK_TILE];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t step = (((int64_t)gridDim.x * NT) >> 5) * piece;
  for (int64_t e0 = (((int64_t)blockIdx.x * NT + threadIdx.x) >> 5) * piece; e0 < nseg; e0 += step) {  // uniform in the warp
    const int64_t e1 = e0 + piece < nseg ? e0 + piece : nseg;
    int64_t cur = warp_row_of(coff, k, e0);
    for (int64_t ts = e0; ts < e1; ts += WALK_TILE) {
      int64_t row[4];
      warp_tile_rows_strided(coff, k, ts, cur, mark[wid], row);
      int32_t c[4];
      V x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t e = ts + lane + 32 * j;
        if (e >= e1) continue;
        const int64_t p = delta[row[j]] + e;
        c[j] = ab[p];
        x[j] = aw[p];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t e = ts + lane + 32 * j;
        if (e >= e1) continue;
        ccols[e] = c[j];
        cw[e] = (WOUT)x[j];
      }
    }
  }
}

// Inside aggregate_as: a CUDA error frees the scratch before returning.
#define AG_CHECK(call)                                         \
  do {                                                         \
    cudaError_t _e = (call);                                   \
    if (_e != cudaSuccess) return fail(set_cuda_error(_e));    \
  } while (0)

// V: type of the segments' weights. 32-bit ones become the coarse graph's own.
template <class V>
int aggregate_as(cd_graph* g, const int32_t* labels_dev, const int32_t* newid_dev, int64_t k, cd_graph** coarse_out) {
  constexpr bool NARROW = sizeof(V) == 4;
  cudaStream_t s = g->stream;
  const int64_t n = g->n, m = g->nnz;
  int rc = CD_OK;
  // scratch
  Arena scratch;
  int32_t *nl, *ab, *t8, *t32, *wl, *ml, *cl, *ll, *ch_seg, *dch, *tlg, *owner = nullptr, *gk = nullptr;
  int64_t *delta, *sstart, *ch_off, *toff, *ucnt;
  unsigned long long *arcs, *cnt, *ub, *gs = nullptr;
  V* aw;
  // the coarse graph
  int64_t *coarse_off = nullptr, *cdegw = nullptr;
  int32_t* ccols = nullptr;
  void* cw = nullptr;
  auto cleanup = [&]() {
    scratch.free(s);
    dev_free(gs, s);
    dev_free(gk, s);
    dev_free(owner, s);
  };
  auto fail = [&](int r) {
    cleanup();
    dev_free(coarse_off, s);
    dev_free(cdegw, s);
    dev_free(ccols, s);
    dev_free(cw, s);
    return r;
  };
  const int64_t max_big = m / (AG_CTA_MAX + 1) + 1;           // large segments at most
  const int64_t max_chunks = m / AG_CHUNK + max_big;          // their chunks at most
  const int64_t max_mid = std::min(k, m / (AG_WARP_MAX + 1) + 1);  // segments of each CTA class at most
  const int64_t max_cta = std::min(k, m / (AG_MID_MAX + 1) + 1);
  const bool big = m > AG_CTA_MAX;                            // there may be large segments
  scratch.add(&nl, n);
  scratch.add(&delta, std::max(n, k));
  scratch.add(&arcs, 3 * k);  // arcs per community, distinct entries, upper bounds: cleared together
  scratch.add(&sstart, k + 1);
  scratch.add(&cnt, AC_N + 2 + NBINS + 1);
  scratch.add(&ab, m);
  scratch.add(&aw, m);
  scratch.add(&t8, std::min(k, m + 1));
  scratch.add(&t32, std::min(k, m / 9 + 1));
  scratch.add(&wl, std::min(k, m / 33 + 1));
  scratch.add(&ml, max_mid);
  scratch.add(&cl, max_cta);
  scratch.add(&ll, max_big);
  scratch.add(&ch_seg, max_chunks);
  scratch.add(&ch_off, max_chunks);
  scratch.add(&dch, max_chunks);
  scratch.add(&tlg, big ? k : 1);
  scratch.add(&toff, big ? k : 1);
  if ((rc = scratch.make(s)) || (rc = dev_alloc_t(&cdegw, k, s)) || (rc = dev_alloc_t(&coarse_off, k + 1, s)))
    return fail(rc);
  ucnt = (int64_t*)arcs + k;
  ub = arcs + 2 * k;
  const int wbytes = g->wkind == W_UNIT ? 0 : g->wkind == W_I32 ? 4 : 8;
  const unsigned gv = gcap((n + NT - 1) / NT, 152 * 8);
  {
    KTimer t(g, K_AGG_EMIT, (double)n * (4 + 4 + 8 + 8 + 4 + 8) + (double)m * (4 + 4 + wbytes + 4 + sizeof(V)));
    AG_CHECK(cudaMemsetAsync(arcs, 0, 3 * k * 8, s));
    AG_CHECK(cudaMemsetAsync(cdegw, 0, k * 8, s));
    CD_LAUNCH(k_ag_vertex<<<gv, NT, 0, s>>>(labels_dev, newid_dev, g->off, g->degw, n, nl, arcs,
                                            (unsigned long long*)cdegw));
    if ((rc = exclusive_scan_i64((const int64_t*)arcs, sstart, k, sstart + k, s))) return fail(rc);
    AG_CHECK(cudaMemsetAsync(arcs, 0, k * 8, s));  // now the places taken per community
    CD_LAUNCH(k_ag_place<<<gcap((n + AP_VERTS - 1) / AP_VERTS, 152 * 6), NT, 0, s>>>(nl, g->off, n, sstart, arcs, delta));
    if (m > 0) {
      const unsigned gr = gcap((m + 8 * WALK_TILE - 1) / (8 * WALK_TILE), 152 * 8);
      const int64_t piece = walk_piece(m, (int64_t)gr * NW);
      if (g->wkind == W_UNIT)
        CD_LAUNCH((k_ag_scatter<WUnit, V><<<gr, NT, 0, s>>>(g->off, g->cols, g->w, n, m, piece, nl, delta, ab, aw)));
      else if (g->wkind == W_I32)
        CD_LAUNCH((k_ag_scatter<WI32, V><<<gr, NT, 0, s>>>(g->off, g->cols, g->w, n, m, piece, nl, delta, ab, aw)));
      else
        CD_LAUNCH((k_ag_scatter<WI64, V><<<gr, NT, 0, s>>>(g->off, g->cols, g->w, n, m, piece, nl, delta, ab, aw)));
    }
  }
  unsigned long long h[AC_N + 2 + NBINS + 1] = {};  // the counts; then empty rows, largest deg_w, degree bins, hub arcs
  int64_t nseg = 0;
  {
    KTimer t(g, K_AGG_REDUCE, (double)m * 2 * (4 + sizeof(V)) + (double)k * 32);
    AG_CHECK(cudaMemsetAsync(cnt, 0, sizeof(h), s));
    static PerDevice attrs;
    auto mid = k_ag_cta<V, 128, AG_MID_MAX, AC_MID>;
    auto cta = k_ag_cta<V, 512, AG_CTA_MAX, AC_CTA>;
    constexpr size_t msm = ag_cta_smem<V, AG_MID_MAX>(), csm = ag_cta_smem<V, AG_CTA_MAX>();
    if (!attrs.get()) {
      AG_CHECK(cudaFuncSetAttribute(k_ag_warp<V>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ag_warp_smem<V>()));
      AG_CHECK(cudaFuncSetAttribute(mid, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)msm));
      AG_CHECK(cudaFuncSetAttribute(cta, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)csm));
      attrs.set(1);
    }
    if (m > 0) {
      CD_LAUNCH(k_ag_classes<<<gcap((k + AF_SEGS - 1) / AF_SEGS, 152 * 8), NT, 0, s>>>(sstart, k, cnt, t8, t32, wl, ml, cl,
                                                                                    ll, ch_seg, ch_off));
      if (m > AG_MID_MAX)
        CD_LAUNCH((cta<<<gcap(max_cta + max_chunks, 152 * 2), 512, csm, s>>>(sstart, cl, ch_seg, ch_off, cnt, ab, aw, ucnt,
                                                                             dch, ub)));
      if (m > AG_WARP_MAX)
        CD_LAUNCH((mid<<<gcap(max_mid, 152 * 10), 128, msm, s>>>(sstart, ml, ch_seg, ch_off, cnt, ab, aw, ucnt, dch, ub)));
      CD_LAUNCH(k_ag_warp<V><<<gcap((k + NW - 1) / NW, 152 * 4), NT, ag_warp_smem<V>(), s>>>(sstart, t8, t32, wl, cnt, ab,
                                                                                          aw, ucnt));
    }
    if (big) {
      CD_LAUNCH(k_ag_tables_size<<<gcap((max_big + NT - 1) / NT), NT, 0, s>>>(ll, ub, tlg, toff, cnt));
      AG_CHECK(cudaMemcpyAsync(h, cnt, AC_N * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
      AG_CHECK(cudaStreamSynchronize(s));
      const int64_t nlarge = (int64_t)h[AC_BIG], nch = (int64_t)h[AC_CHUNKS], slots = (int64_t)h[AC_SLOTS];
      if (nlarge > 0) {
        const int64_t nslices = slots / AG_SLICE;
        if ((rc = dev_alloc_t(&gs, slots, s)) || (!NARROW && (rc = dev_alloc_t(&gk, slots, s))) ||
            (rc = dev_alloc_t(&owner, nslices, s)))
          return fail(rc);
        AG_CHECK(cudaMemsetAsync(gs, NARROW ? 0xff : 0, slots * sizeof(unsigned long long), s));
        if (!NARROW) AG_CHECK(cudaMemsetAsync(gk, 0xff, slots * sizeof(int32_t), s));
        CD_LAUNCH(k_ag_tables_own<<<gcap(nlarge, 152 * 8), NT, 0, s>>>(ll, nlarge, tlg, toff, owner));
        CD_LAUNCH(k_ag_merge<V><<<gcap(nch, 152 * 8), NT, 0, s>>>(sstart, ch_seg, ch_off, dch, nch, ab, aw, tlg, toff, gs,
                                                               gk));
        CD_LAUNCH(k_ag_extract<V><<<gcap(nslices, 152 * 8), NT, 0, s>>>(owner, nslices, gs, gk, sstart, ab, aw, ucnt));
      }
    }
    // 4: the coarse CSR
    if ((rc = exclusive_scan_i64(ucnt, coarse_off, k, coarse_off + k, s))) return fail(rc);
    CD_LAUNCH(k_ag_rows<<<gcap((k + NT - 1) / NT, 152 * 8), NT, 0, s>>>(sstart, coarse_off, k, delta,
                                                                      (const unsigned long long*)cdegw, g->t_warp, g->t_hub, cnt + AC_N));
    AG_CHECK(cudaMemcpyAsync(&nseg, coarse_off + k, 8, cudaMemcpyDeviceToHost, s));
    AG_CHECK(cudaMemcpyAsync(h + AC_N, cnt + AC_N, (2 + NBINS + 1) * 8, cudaMemcpyDeviceToHost, s));
    AG_CHECK(cudaStreamSynchronize(s));
    if ((rc = dev_alloc_t(&ccols, nseg + COL_PAD, s)) ||
        (rc = dev_alloc(&cw, (size_t)std::max<int64_t>(nseg, 1) * (NARROW ? 4 : 8), s)))
      return fail(rc);
    AG_CHECK(cudaMemsetAsync(ccols + nseg, 0, COL_PAD * sizeof(int32_t), s));
    if (nseg > 0) {
      const unsigned gr = gcap((nseg + 8 * WALK_TILE - 1) / (8 * WALK_TILE), 152 * 8);
      const int64_t piece = walk_piece(nseg, (int64_t)gr * NW);
      typedef typename std::conditional<NARROW, int32_t, int64_t>::type WOUT;
      CD_LAUNCH((k_ag_compact<V, WOUT><<<gr, NT, 0, s>>>(coarse_off, k, nseg, piece, delta, ab, aw, ccols, (WOUT*)cw)));
    }
    if (cudaGetLastError() != cudaSuccess) return fail(CD_ECUDA);
  }
  cleanup();
  // what an ingest of the coarse arcs would find: aggregation keeps vol(V), and deg_w was summed above
  unsigned long long stats[INGEST_STATS] = {};
  stats[0] = (unsigned long long)g->vol;
  stats[2] = h[AC_N];
  stats[3] = h[AC_N + 1];
  cd_graph* c = nullptr;
  rc = graph_adopt(s, k, nseg, coarse_off, ccols, cw, NARROW ? W_I32 : W_I64, &c, cdegw, stats, g, h + AC_N + 2);
  if (rc) return rc;
  c->timing = g->timing;
  c->ktiming = g->ktiming;
  c->cols_distinct = true;  // one arc per pair of communities
  *coarse_out = c;
  return CD_OK;
}

#undef AG_CHECK

}  // namespace

int aggregate_hash(cd_graph* g, const int32_t* labels_dev, const int32_t* newid_dev, int64_t k, cd_graph** coarse_out) {
  if (g->vol < ((int64_t)1 << 31)) return aggregate_as<uint32_t>(g, labels_dev, newid_dev, k, coarse_out);
  return aggregate_as<unsigned long long>(g, labels_dev, newid_dev, k, coarse_out);
}

}  // namespace cd
