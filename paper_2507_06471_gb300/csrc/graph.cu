// Graph ingest (Sec. II-A): device copy of a symmetric CSR, validation,
// weighted degrees deg_w(v) (loops counted twice) and vol(V); static degree
// bins for the scan kernels and the global hash tables of hub vertices.
//
// Internal weight convention: a loop arc v->v carries 2L, so that deg_w(v) is
// the plain row sum and aggregation/modularity sum arc weights without special
// cases. Upload doubles loop arcs; cd_graph_download halves them back.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>

#include "common.cuh"
#include "rowwalk.cuh"

namespace cd {

const char* const kKernelNames[K_COUNT] = {
    "ingest",     "scan_tile4", "scan_tile8", "scan_tile16", "scan_tile32", "scan_warp",
    "scan_blk128", "hub_build", "hub_eval",   "apply_moves", "renumber",    "agg_emit",
    "radix_sort", "agg_reduce", "modularity", "hub_mark", "frontier", "scan_blk512", "hub_prepare"};

static thread_local int g_last_cuda = 0;
static std::atomic<long long> g_launches{0};

void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

int set_cuda_error(cudaError_t e) {
  g_last_cuda = (int)e;
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return CD_ENOMEM;
  }
  return CD_ECUDA;
}

int dev_alloc(void** p, size_t bytes, cudaStream_t s) {
  // keep freed blocks in the device's default pool (threads that race here set the same)
  static PerDevice pool_set;
  if (!pool_set.get()) {
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, current_device()) == cudaSuccess) {
      uint64_t thr = UINT64_MAX;
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
    pool_set.set(1);
  }
  cudaError_t e = cudaMallocAsync(p, bytes, s);
  if (e != cudaSuccess) {
    *p = nullptr;
    return set_cuda_error(e);
  }
  return CD_OK;
}

void dev_free(void* p, cudaStream_t s) {
  if (p) cudaFreeAsync(p, s);
}

KTimer::KTimer(cd_graph* g_, int k_, double bytes_, cudaStream_t st_) : g(g_), k(k_), bytes(bytes_), st(st_) {
  if (g && g->ktiming) {
    if (!st) st = g->stream;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    cudaEventRecord(a, st);
  }
}

KTimer::~KTimer() {
  if (g && g->ktiming) {
    cudaEventRecord(b, st);
    g->pending.push_back({k, {a, b}});
    g->pending_bytes.push_back(bytes);
  }
}

void profile_reset(cd_graph* g) {
  for (int k = 0; k < K_COUNT; ++k) {
    memset(&g->prof[k], 0, sizeof(cd_kernel_profile));
    snprintf(g->prof[k].name, sizeof(g->prof[k].name), "%s", kKernelNames[k]);
  }
}

int profile_flush(cd_graph* g) {
  if (g->pending.empty()) return CD_OK;
  CD_CHECK(cudaStreamSynchronize(g->stream));
  for (size_t i = 0; i < g->pending.size(); ++i) {
    auto& p = g->pending[i];
    float ms = 0.f;
    cudaEventElapsedTime(&ms, p.second.first, p.second.second);
    cd_kernel_profile& kp = g->prof[p.first];
    kp.launches += 1;
    kp.total_ms += ms;
    kp.alg_bytes += g->pending_bytes[i];
    cudaEventDestroy(p.second.first);
    cudaEventDestroy(p.second.second);
  }
  g->pending.clear();
  g->pending_bytes.clear();
  return CD_OK;
}

namespace {

constexpr int NT = 256;
constexpr int NSTATS = INGEST_STATS;

__device__ __forceinline__ void fail(int32_t* status, int code) { atomicCAS(status, 0, code); }

// counts[NBINS]: arcs of the hubs.
__global__ void k_bin_count(const int64_t* __restrict__ off, int64_t n, int t_warp, int t_hub,
                            unsigned long long* counts) {
  __shared__ uint32_t sb[NBINS];
  if (threadIdx.x < NBINS) sb[threadIdx.x] = 0;
  __syncthreads();
  unsigned long long hub_arcs = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
    const int64_t d = off[v + 1] - off[v];
    if (d > 0) atomicAdd(&sb[bin_of(d, t_warp, t_hub)], 1u);
    if (d > t_hub) hub_arcs += (unsigned long long)d;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) hub_arcs += __shfl_xor_sync(FULL, hub_arcs, o);
  if ((threadIdx.x & 31) == 0 && hub_arcs) atomicAdd(&counts[NBINS], hub_arcs);
  __syncthreads();
  if (threadIdx.x < NBINS && sb[threadIdx.x]) atomicAdd(&counts[threadIdx.x], (unsigned long long)sb[threadIdx.x]);
}

// The resident loop's hubs, in any order.
__global__ void k_rh_collect(const int64_t* __restrict__ off, int64_t n, int t_hub, int32_t* __restrict__ v_out,
                             int32_t* count) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
    if (off[v + 1] - off[v] > t_hub) v_out[atomicAdd(count, 1)] = (int32_t)v;
}

// Items, slices and tables of nh <= RH_MAX_HUBS hubs: one CTA, four hubs a thread.
__global__ void __launch_bounds__(1024) k_rh_layout(const int64_t* __restrict__ off, ResidentHubs r) {
  __shared__ long long wsum[32][3];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  long long x[4][3], mine[3] = {0, 0, 0};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int h = threadIdx.x * 4 + q;
    const int64_t d = h < r.nh ? off[r.v[h] + 1] - off[r.v[h]] : 0;
    const int64_t cap = h < r.nh ? d + d / 2 + 64 : 0;  // at most two thirds full
    x[q][0] = (d + RH_CHUNK - 1) / RH_CHUNK;
    x[q][1] = (cap + RH_SLICE - 1) / RH_SLICE;
    x[q][2] = cap;
#pragma unroll
    for (int c = 0; c < 3; ++c) mine[c] += x[q][c];
  }
  long long inc[3] = {mine[0], mine[1], mine[2]};
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(FULL, inc[c], o);
      if (lane >= o) inc[c] += y;
    }
  if (lane == 31)
    for (int c = 0; c < 3; ++c) wsum[wid][c] = inc[c];
  __syncthreads();
  if (threadIdx.x == 0)
    for (int c = 0; c < 3; ++c) {
      long long run = 0;
      for (int w = 0; w < 32; ++w) {
        const long long y = wsum[w][c];
        wsum[w][c] = run;
        run += y;
      }
    }
  __syncthreads();
  long long at[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) at[c] = wsum[wid][c] + inc[c] - mine[c];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int h = threadIdx.x * 4 + q;
    if (h <= r.nh) {  // entry nh: the totals
      r.item[h] = (int32_t)at[0];
      r.slice[h] = (int32_t)at[1];
      r.tab[h] = at[2];
    }
    if (h < r.nh) {
      for (int i = 0; i < (int)x[q][0]; ++i) r.item_hub[at[0] + i] = h;
      for (int i = 0; i < (int)x[q][1]; ++i) r.slice_hub[at[1] + i] = h;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) at[c] += x[q][c];
  }
}

// `in` may be `out` (64-bit offsets are checked where they were copied to).
template <class OffT>
__global__ void k_offsets_check(const OffT* in, int64_t n, int64_t nnz, int64_t* out, int32_t* status) {
  int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += stride) {
    int64_t a = (int64_t)in[i];
    if (sizeof(OffT) != 8) out[i] = a;
    if (a < 0 || a > nnz) fail(status, CD_ENOTSYM);
    if (i < n && (int64_t)in[i + 1] < a) fail(status, CD_ENOTSYM);
    if (i == 0 && a != 0) fail(status, CD_ENOTSYM);
    if (i == n && a != nnz) fail(status, CD_ENOTSYM);
  }
}

// Ingest: bounds-check columns and weights, deg_w with loops twice, loop
// count, vol(V), per-bin vertex counts, and whether every row's columns are
// strictly increasing (then no row repeats a column). stats: [0] vol,
// [1] loops, [2] isolated, [3] largest deg_w, [4..4+NBINS) bin counts,
// [4+NBINS] rows not strictly increasing.
//
// A pass over the arcs, split evenly over the warps (rowwalk.cuh), checks them
// and sums the weights by row into deg_w (zero before); with unit weights only
// the loops are added. A pass over the vertices makes the statistics. Bound by
// the columns' latency and the row marks: R-MAT 24 (5.2e8 arcs) 3.8 -> 1.5 ms
// against rows by a lane, a warp or a CTA each with 64-bit shared counters;
// 613 vertices 21.5 -> 5.9 us, upload of R-MAT 2^20 796 -> 326 us.
constexpr int ST_UNSORTED = 4 + NBINS;

template <class W>
__global__ void __launch_bounds__(NT) k_ingest_arcs(const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                                                    const void* w, int64_t n, int64_t m, int64_t piece,
                                                    int loops_twice, unsigned long long* degw,
                                                    unsigned long long* stats, int32_t* status) {
  __shared__ __align__(16) int32_t mark[NT / 32][WALK_TILE];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t step = (((int64_t)gridDim.x * NT) >> 5) * piece;
  unsigned loops = 0;
  bool unsorted = false;
  for (int64_t e0 = (((int64_t)blockIdx.x * NT + threadIdx.x) >> 5) * piece; e0 < m; e0 += step) {  // uniform in the warp
    const int64_t e1 = e0 + piece < m ? e0 + piece : m;
    // the columns carry COL_PAD spare entries, and pieces start at multiples of WALK_TILE
    auto columns = [&](int64_t e) { return e < e1 ? __ldg(reinterpret_cast<const int4*>(cols + e)) : make_int4(0, 0, 0, 0); };
    int4 next = columns(e0 + 4 * lane);  // a tile ahead
    int64_t cur = warp_row_of(off, n, e0);
    // the arc before the piece, if it belongs to the same row
    int64_t last_row = e0 > 0 && off[cur] < e0 ? cur : -1;
    int32_t last_col = e0 > 0 ? cols[e0 - 1] : 0;
    for (int64_t ts = e0; ts < e1; ts += WALK_TILE) {
      const int64_t e = ts + 4 * lane;
      const int4 c4 = next;
      next = columns(e + WALK_TILE);
      int64_t x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = e + j < e1 ? W::get(w, e + j) : 1;
      const int32_t u[4] = {c4.x, c4.y, c4.z, c4.w};
      int64_t row[4];
      unsigned long long val[4];
      warp_tile_rows(off, n, ts, cur, mark[wid], row);
      int64_t pr = __shfl_up_sync(FULL, (long long)row[3], 1);
      int32_t pc = __shfl_up_sync(FULL, u[3], 1);
      if (lane == 0) {
        pr = last_row;
        pc = last_col;
      }
      last_row = __shfl_sync(FULL, (long long)row[3], 31);  // used only if the piece goes on, so of a whole tile
      last_col = __shfl_sync(FULL, u[3], 31);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        val[j] = 0;
        if (e + j >= e1) {
          row[j] = -1;
          continue;
        }
        if (u[j] < 0 || u[j] >= n) fail(status, CD_EBOUNDS);
        if (x[j] < 1) fail(status, CD_EINVAL);
        if (row[j] == (j ? row[j - 1] : pr) && (j ? u[j - 1] : pc) >= u[j]) unsorted = true;
        val[j] = (unsigned long long)x[j];
        if (u[j] == row[j]) {
          ++loops;
          if (loops_twice) {  // input convention: the loop arc carries L
            val[j] += (unsigned long long)x[j];
            if (W::unit) atomicAdd(&degw[row[j]], 1ull);
          }
        }
      }
      if (!W::unit) warp_rows_sum(row, val, [&](int64_t r, unsigned long long sum) { atomicAdd(&degw[r], sum); });
    }
  }
  loops = __reduce_add_sync(FULL, loops);
  unsorted = __any_sync(FULL, unsorted);
  if (lane == 0 && loops) atomicAdd(&stats[1], (unsigned long long)loops);
  if (lane == 0 && unsorted) atomicOr(&stats[ST_UNSORTED], 1ull);
}

// The statistics of the vertices; unit: deg_w holds the loops, the degree is added.
__global__ void __launch_bounds__(NT) k_ingest_rows(const int64_t* __restrict__ off, int64_t n, int unit,
                                                    unsigned long long* degw, unsigned long long* stats) {
  __shared__ uint32_t bins[NBINS + 1];  // the last one: isolated
  __shared__ unsigned long long part[2][NT / 32];
  for (int i = threadIdx.x; i <= NBINS; i += NT) bins[i] = 0;
  __syncthreads();
  unsigned long long vol = 0, top = 0;
  const int64_t stride = (int64_t)gridDim.x * NT;
  for (int64_t v = (int64_t)blockIdx.x * NT + threadIdx.x; v < n; v += stride) {
    const int64_t d = off[v + 1] - off[v];
    unsigned long long s = degw[v];
    if (unit) degw[v] = s += (unsigned long long)d;
    vol += s;
    top = s > top ? s : top;
    atomicAdd(&bins[d == 0 ? NBINS : bin_of(d)], 1u);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    vol += __shfl_xor_sync(FULL, vol, o);
    const unsigned long long t = __shfl_xor_sync(FULL, top, o);
    top = t > top ? t : top;
  }
  if ((threadIdx.x & 31) == 0) {
    part[0][threadIdx.x >> 5] = vol;
    part[1][threadIdx.x >> 5] = top;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < NT / 32; ++i) {
      vol += part[0][i];
      top = part[1][i] > top ? part[1][i] : top;
    }
    if (vol) atomicAdd(&stats[0], vol);
    if (top) atomicMax(&stats[3], top);
  }
  if (threadIdx.x <= NBINS && bins[threadIdx.x])
    atomicAdd(&stats[threadIdx.x < NBINS ? 4 + threadIdx.x : 2], (unsigned long long)bins[threadIdx.x]);
}

// Internal weights with loop arcs doubled (int64).
template <class W>
__global__ void __launch_bounds__(NT) k_double_loops(const int64_t* __restrict__ off,
                                                     const int32_t* __restrict__ cols,
                                                     const void* w, int64_t n,
                                                     int64_t* __restrict__ w64) {
  const int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < n; v += nwarps)
    for (int64_t e = off[v] + lane; e < off[v + 1]; e += 32) {
      int64_t x = W::get(w, e);
      w64[e] = cols[e] == v ? 2 * x : x;
    }
}

struct BinBase {
  int64_t b[NBINS + 1];
};

// The listed vertices by bin; cursor comes back with the vertices per bin. The
// hubs are only counted here (k_hub_list lists them in order). A CTA places
// 1,024 vertices at a time and takes their room with one atomic per bin: with one
// per warp the cursors' atomics, one after another, were the time (2.7e6
// vertices: 190 us, 21 so).
constexpr int FILL = 4;
__global__ void __launch_bounds__(NT) k_bin_fill(const int64_t* __restrict__ off, int64_t n, int t_warp,
                                                 int t_hub, BinBase base, unsigned long long* cursor,
                                                 int32_t* __restrict__ list) {
  __shared__ int cnt[NBINS];
  __shared__ int64_t at[NBINS];
  const int lane = threadIdx.x & 31;
  for (int64_t v0 = (int64_t)blockIdx.x * NT * FILL; v0 < n; v0 += (int64_t)gridDim.x * NT * FILL) {
    if (threadIdx.x < NBINS) cnt[threadIdx.x] = 0;
    __syncthreads();
    int b[FILL], rank[FILL];
#pragma unroll
    for (int k = 0; k < FILL; ++k) {
      const int64_t v = v0 + k * NT + threadIdx.x;
      const int64_t d = v < n ? off[v + 1] - off[v] : 0;
      b[k] = d > 0 ? bin_of(d, t_warp, t_hub) : -1;
      rank[k] = 0;
    }
#pragma unroll
    for (int k = 0; k < FILL; ++k) {
      const unsigned peers = __match_any_sync(FULL, b[k]);
      const int lead = __ffs(peers) - 1;
      int r = 0;
      if (lane == lead && b[k] >= 0) r = atomicAdd(&cnt[b[k]], __popc(peers));
      rank[k] = __shfl_sync(FULL, r, lead) + __popc(peers & ((1u << lane) - 1u));
    }
    __syncthreads();
    if (threadIdx.x < NBINS && cnt[threadIdx.x])
      at[threadIdx.x] = (int64_t)atomicAdd(&cursor[threadIdx.x], (unsigned long long)cnt[threadIdx.x]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < FILL; ++k)
      if (b[k] >= 0 && b[k] != B_HUB)
        list[base.b[b[k]] + at[b[k]] + rank[k]] = (int32_t)(v0 + k * NT + threadIdx.x);
  }
}

// Hubs are numbered in increasing vertex id, so the number of vertex u is its
// rank among the hubs: hub_pref[u / 32] (hubs below 32 (u / 32)) plus the hub
// bits below u in its word. The bits and their counts per word, a warp per word:
__global__ void __launch_bounds__(NT) k_hub_words(const int64_t* __restrict__ off, int64_t n, int t_hub,
                                                  uint32_t* __restrict__ bits, int64_t* __restrict__ count) {
  const int lane = threadIdx.x & 31;
  const int64_t words = (n + 31) / 32, nwarps = ((int64_t)gridDim.x * NT) >> 5;
  for (int64_t w = ((int64_t)blockIdx.x * NT + threadIdx.x) >> 5; w < words; w += nwarps) {
    const int64_t v = 32 * w + lane;
    const unsigned m = __ballot_sync(FULL, v < n && off[v + 1] - off[v] > t_hub);
    if (lane == 0) {
      bits[w] = m;
      count[w] = __popc(m);
    }
  }
}

// The hubs in order, and each one's table slots, build/mark items and evaluate
// items (scanned into the offsets of each afterwards).
__global__ void k_hub_list(const int64_t* __restrict__ off, int64_t words, const uint32_t* __restrict__ bits,
                           const int64_t* __restrict__ pref, uint32_t* __restrict__ hub_pref,
                           int32_t* __restrict__ hubs, int64_t* __restrict__ cap, int64_t* __restrict__ items,
                           int64_t* __restrict__ evs) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < words; w += stride) {
    int64_t h = pref[w];
    hub_pref[w] = (uint32_t)h;
    for (uint32_t m = bits[w]; m; m &= m - 1, ++h) {
      const int64_t v = 32 * w + __ffs(m) - 1;
      const int64_t d = off[v + 1] - off[v];
      const int64_t c = d + d / 2 + 64;  // live labels <= deg; the rest absorbs labels that come and go
      hubs[h] = (int32_t)v;
      cap[h] = c;
      items[h] = (d + HUB_CHUNK - 1) / HUB_CHUNK;
      evs[h] = (c + HUB_SLICE - 1) / HUB_SLICE;
    }
  }
}

// Warp per hub: its items.
__global__ void __launch_bounds__(NT) k_hub_items(const int64_t* __restrict__ off, const int32_t* __restrict__ hubs,
                                                  int64_t nh, const int64_t* __restrict__ item_first,
                                                  const int64_t* __restrict__ ev_first, int32_t* __restrict__ item_hub,
                                                  int64_t* __restrict__ item_arc, int32_t* __restrict__ ev_hub,
                                                  int64_t* __restrict__ ev_slot) {
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = ((int64_t)gridDim.x * NT) >> 5;
  for (int64_t h = ((int64_t)blockIdx.x * NT + threadIdx.x) >> 5; h < nh; h += nwarps) {
    const int64_t beg = off[hubs[h]], i0 = item_first[h], i1 = item_first[h + 1], e0 = ev_first[h], e1 = ev_first[h + 1];
    for (int64_t i = i0 + lane; i < i1; i += 32) {
      item_hub[i] = (int32_t)h;
      item_arc[i] = beg + (i - i0) * HUB_CHUNK;
    }
    for (int64_t e = e0 + lane; e < e1; e += 32) {
      ev_hub[e] = (int32_t)h;
      ev_slot[e] = (e - e0) * HUB_SLICE;
    }
  }
}

__global__ void k_download_w(const int64_t* __restrict__ off, const int32_t* __restrict__ cols,
                             const void* w, int wkind, int64_t n, int64_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < n; v += nwarps)
    for (int64_t e = off[v] + lane; e < off[v + 1]; e += 32) {
      int64_t x = wkind == W_UNIT ? 1 : wkind == W_I32 ? (int64_t)((const int32_t*)w)[e]
                                                       : ((const int64_t*)w)[e];
      out[e] = cols[e] == v ? x / 2 : x;  // loop arcs are stored doubled (2L)
    }
}

__global__ void k_narrow_w(const int64_t* __restrict__ w64, int64_t nnz, int32_t* __restrict__ w32) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += stride) w32[e] = (int32_t)w64[e];
}

__global__ void k_labels_check(const int32_t* __restrict__ lab, int64_t n, int32_t* status) {
  int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    if (lab[i] < 0 || lab[i] >= n) fail(status, CD_EINVAL);
}

unsigned grid_cap_u(int64_t blocks, int64_t cap) {
  if (blocks < 1) blocks = 1;
  return (unsigned)(blocks < cap ? blocks : cap);
}

unsigned grid_for(int64_t work, int per_block = NT) {
  int64_t b = (work + per_block - 1) / per_block;
  if (b < 1) b = 1;
  if (b > 152 * 32) b = 152 * 32;
  return (unsigned)b;
}

int read_status(cd_graph* g) {
  int32_t st = 0;
  CD_CHECK(cudaMemcpyAsync(&st, g->status, sizeof(int32_t), cudaMemcpyDeviceToHost, g->stream));
  CD_CHECK(cudaStreamSynchronize(g->stream));
  if (st) CD_CHECK(cudaMemsetAsync(g->status, 0, sizeof(int32_t), g->stream));
  return st;
}

void free_resident_hubs(cd_graph* g);

void free_arrays(cd_graph* g) {
  cudaStream_t s = g->stream;
  free_resident_hubs(g);
  void* ps[] = {g->off,  g->cols,  g->w,    g->degw,    g->bin_mem[0], g->bin_mem[1], g->run_mem, g->status,
                g->gid,  g->gbase, g->gvol, g->gfrozen, g->gcnt};
  for (void* p : ps) dev_free(p, s);
  if (g->h_ctr) cudaFreeHost(g->h_ctr);
}

void free_resident_hubs(cd_graph* g) {
  if (!g->rh) return;
  dev_free(g->rh->mem[0], g->stream);
  dev_free(g->rh->mem[1], g->stream);
  delete g->rh;
  g->rh = nullptr;
}

void free_bins(cd_graph* g) {
  cudaStream_t s = g->stream;
  free_resident_hubs(g);
  for (void*& p : g->bin_mem) {
    dev_free(p, s);
    p = nullptr;
  }
  g->bin_list = nullptr;
  g->act_list = nullptr;
  g->full_cnt = nullptr;
  g->act_ev = nullptr;
  g->act_small = nullptr;
  g->hub_cc = nullptr;
  g->hub_live = nullptr;
  g->hub_pref = nullptr;
  g->hub_bits = nullptr;
  g->hub_tab = nullptr;
  g->hub_slot = nullptr;
  g->hub_item_hub = nullptr;
  g->hub_item_arc = nullptr;
  g->hub_ev_hub = nullptr;
  g->hub_ev_slot = nullptr;
  g->hub_ev_first = nullptr;
  g->hub_part = nullptr;
  g->hub_cur = nullptr;
  g->hub_hascur = nullptr;
  g->hub_done = nullptr;
  g->hub_mv = nullptr;
  g->hub_rb = nullptr;
  g->hub_flist = nullptr;
  g->hub_fcnt = nullptr;
  g->hub_cl = nullptr;
  g->hub_used = nullptr;
  g->hub_item_first = nullptr;
  g->hub_blist = nullptr;
  g->hub_mlist = nullptr;
  g->hub_log = nullptr;
  g->hub_nl = g->hub_pl = nullptr;
  g->hub_nc = nullptr;
  g->hub_log_cap = 0;
  g->nhubs = g->hub_arcs = g->hub_slots = g->hub_items = g->hub_eval_items = 0;
}

int build_bins(cd_graph* g);

void take_bins(cd_graph* g, const unsigned long long* cnt) {
  g->bin_start[0] = 0;
  for (int b = 0; b < NBINS; ++b) g->bin_start[b + 1] = g->bin_start[b] + (int64_t)cnt[b];
  g->nhubs = (int64_t)cnt[B_HUB];
  g->hub_arcs = (int64_t)cnt[NBINS];
}

// Scalars, bins and hub structures of a graph whose CSR, weights and deg_w
// are in place; stats from the ingest kernels.
int finish_graph(cd_graph* g, const unsigned long long* stats, const unsigned long long* bins) {
  g->cols_distinct = stats[ST_UNSORTED] == 0;  // strictly increasing rows; aggregation sets it for coarse rows
  g->vol = (int64_t)stats[0];
  g->n_isolated = (int64_t)stats[2];
  g->max_degw = (int64_t)stats[3];
  if (stats[0] >= (1ull << 62)) return CD_EOVERFLOW;
  if (!bins) return build_bins(g);
  take_bins(g, bins);
  return CD_OK;
}

// Vertices per degree bin for (t_warp, t_hub).
int build_bins(cd_graph* g) {
  cudaStream_t s = g->stream;
  int rc;
  unsigned long long* d_cnt = nullptr;
  unsigned long long h_cnt[NBINS + 1] = {};
  if ((rc = dev_alloc_t(&d_cnt, NBINS + 1, s))) return rc;
  CD_CHECK(cudaMemsetAsync(d_cnt, 0, sizeof(h_cnt), s));
  if (g->n > 0)
    CD_LAUNCH(k_bin_count<<<grid_for(g->n), NT, 0, s>>>(g->off, g->n, g->t_warp, g->t_hub, d_cnt));
  CD_CHECK(cudaMemcpyAsync(h_cnt, d_cnt, sizeof(h_cnt), cudaMemcpyDeviceToHost, s));
  CD_CHECK(cudaStreamSynchronize(s));
  dev_free(d_cnt, s);
  take_bins(g, h_cnt);
  return CD_OK;
}

// The bin lists, and the hub histograms' layout.
constexpr int64_t HUB_LOG_DIV = 4;  // budget of logged hub updates per round: hub arcs / 4
int fill_bins(cd_graph* g) {
  cudaStream_t s = g->stream;
  const int64_t listed = g->bin_start[NBINS], nh = g->nhubs, words = (g->n + 31) / 32;
  int64_t* count = nullptr;  // hubs per word, then their prefix
  Arena a;
  a.add(&g->bin_list, listed);
  a.add(&g->act_list, listed);
  a.add(&g->full_cnt, NBINS + 2);
  const size_t zero0 = a.bytes;  // cleared from here ...
  if (nh > 0) {
    a.add(&g->hub_live, nh);
    a.add(&g->hub_rb, nh);
    a.add(&g->hub_used, nh);
    a.add(&g->hub_fcnt, 2);
    a.add(&g->hub_hascur, nh);
    a.add(&g->hub_done, nh);
    a.add(&g->hub_cur, nh);
  }
  const size_t zero1 = a.bytes;  // ... to here
  if (nh > 0) {
    a.add(&g->act_small, nh);  // any hub whose table in use is small
    a.add(&g->hub_cc, nh);
    a.add(&g->hub_pref, words);
    a.add(&g->hub_bits, words);
    a.add(&g->hub_tab, nh + 1);
    a.add(&g->hub_ev_first, nh + 1);
    a.add(&g->hub_item_first, nh + 1);
    a.add(&g->hub_mv, 2 * nh);
    a.add(&g->hub_flist, 2 * nh);
    a.add(&g->hub_cl, 5 * nh);
    a.add(&g->hub_nl, nh);
    a.add(&g->hub_nc, nh);
    a.add(&g->hub_pl, 2 * nh);
    a.add(&count, words);
  }
  int rc = a.make(s);
  if (rc) return rc;
  g->bin_mem[0] = a.mem;
  BinBase base;
  for (int b = 0; b <= NBINS; ++b) base.b[b] = g->bin_start[b];
  CD_CHECK(cudaMemsetAsync(g->full_cnt, 0, (NBINS + 2) * sizeof(unsigned long long), s));
  if (g->n > 0)
    CD_LAUNCH(k_bin_fill<<<grid_for(g->n), NT, 0, s>>>(g->off, g->n, g->t_warp, g->t_hub, base, g->full_cnt,
                                                       g->bin_list));
  CD_CHECK(cudaGetLastError());
  if (nh == 0) return CD_OK;
  // hubs: their list, tables and work items, laid out on the device (one read-back, the totals)
  int32_t* hubs = g->bin_list + g->bin_start[B_HUB];
  CD_LAUNCH(k_hub_words<<<grid_for(words * 32), NT, 0, s>>>(g->off, g->n, g->t_hub, g->hub_bits, count));
  if ((rc = exclusive_scan_i64(count, count, words, nullptr, s))) return rc;
  CD_LAUNCH(k_hub_list<<<grid_for(words), NT, 0, s>>>(g->off, words, g->hub_bits, count, g->hub_pref, hubs, g->hub_cc,
                                                      g->hub_nc, g->hub_cur));
  if ((rc = exclusive_scan_i64(g->hub_cc, g->hub_tab, nh, g->hub_tab + nh, s)) ||
      (rc = exclusive_scan_i64(g->hub_nc, g->hub_item_first, nh, g->hub_item_first + nh, s)) ||
      (rc = exclusive_scan_i64(g->hub_cur, g->hub_ev_first, nh, g->hub_ev_first + nh, s)))
    return rc;
  CD_CHECK(cudaMemcpyAsync(&g->hub_slots, g->hub_tab + nh, 8, cudaMemcpyDeviceToHost, s));
  CD_CHECK(cudaMemcpyAsync(&g->hub_items, g->hub_item_first + nh, 8, cudaMemcpyDeviceToHost, s));
  CD_CHECK(cudaMemcpyAsync(&g->hub_eval_items, g->hub_ev_first + nh, 8, cudaMemcpyDeviceToHost, s));
  CD_CHECK(cudaMemsetAsync((char*)a.mem + zero0, 0, zero1 - zero0, s));
  CD_CHECK(cudaStreamSynchronize(s));
  g->hub_wide = g->max_degw >= ((int64_t)1 << 32) ? 1 : 0;
  // a round applies at most hub_arcs / HUB_LOG_DIV logged updates (random probes
  // into the tables cost about as much as rebuilding the hubs); the hub of
  // every update beyond that budget is rebuilt from its row instead
  g->hub_log_cap = std::max<int64_t>(1, g->hub_slots * 2 / 3 / HUB_LOG_DIV);
  Arena w;
  w.add(&g->act_ev, g->hub_eval_items);
  w.add(&g->hub_slot, g->hub_slots * (1 + g->hub_wide));
  w.add(&g->hub_item_hub, g->hub_items);
  w.add(&g->hub_item_arc, g->hub_items);
  w.add(&g->hub_ev_hub, g->hub_eval_items);
  w.add(&g->hub_ev_slot, g->hub_eval_items);
  w.add(&g->hub_part, 3 * std::max(g->hub_eval_items, g->hub_items));
  w.add(&g->hub_blist, g->hub_items);
  w.add(&g->hub_mlist, g->hub_items);
  w.add(&g->hub_log, 2 * g->hub_log_cap);
  if ((rc = w.make(s))) return rc;
  g->bin_mem[1] = w.mem;
  CD_LAUNCH(k_hub_items<<<grid_for(nh * 32), NT, 0, s>>>(g->off, hubs, nh, g->hub_item_first, g->hub_ev_first,
                                                         g->hub_item_hub, g->hub_item_arc, g->hub_ev_hub, g->hub_ev_slot));
  CD_CHECK(cudaGetLastError());
  return CD_OK;
}

int ingest(cd_graph* g, int loops_twice, unsigned long long* stats_host, int32_t* status_host) {
  cudaStream_t s = g->stream;
  unsigned long long* d_stats = nullptr;
  Arena scratch;
  scratch.add(&d_stats, NSTATS);
  if (int rc = scratch.make(s)) return rc;
  CD_CHECK(cudaMemsetAsync(d_stats, 0, NSTATS * sizeof(unsigned long long), s));
  {
    KTimer t(g, K_UPLOAD, (double)g->nnz * (4 + (g->wkind == W_I32 ? 4 : g->wkind == W_I64 ? 8 : 0)) +
                              (double)g->n * 16);
    unsigned long long* degw = (unsigned long long*)g->degw;
    if (g->n > 0) CD_CHECK(cudaMemsetAsync(degw, 0, g->n * sizeof(int64_t), s));
    if (g->nnz > 0) {
      const unsigned gr = grid_cap_u((g->nnz + NT * 4 - 1) / (NT * 4), 152 * 6);
      const int64_t piece = walk_piece(g->nnz, (int64_t)gr * (NT / 32));
#define CD_INGEST(WT)                                                                                              \
  CD_LAUNCH(k_ingest_arcs<WT><<<gr, NT, 0, s>>>(g->off, g->cols, g->w, g->n, g->nnz, piece, loops_twice, degw,      \
                                                d_stats, g->status))
      if (g->wkind == W_UNIT) CD_INGEST(WUnit);
      else if (g->wkind == W_I32) CD_INGEST(WI32);
      else CD_INGEST(WI64);
#undef CD_INGEST
    }
    if (g->n > 0)
      CD_LAUNCH(k_ingest_rows<<<grid_cap_u((g->n + NT - 1) / NT, 152 * 8), NT, 0, s>>>(
          g->off, g->n, g->wkind == W_UNIT ? 1 : 0, degw, d_stats));
  }
  CD_CHECK(cudaGetLastError());
  CD_CHECK(cudaMemcpyAsync(stats_host, d_stats, (NSTATS) * sizeof(unsigned long long),
                           cudaMemcpyDeviceToHost, s));
  CD_CHECK(cudaMemcpyAsync(status_host, g->status, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  scratch.free(s);
  CD_CHECK(cudaStreamSynchronize(s));
  return CD_OK;
}

}  // namespace

int rebin(cd_graph* g, int t_warp, int t_hub) {
  if (t_warp < 32 || t_warp > WARP_MAX || t_hub < t_warp || t_hub > BLK4_MAX) return CD_EINVAL;
  g->bins_set = true;
  if (t_warp == g->t_warp && t_hub == g->t_hub) return CD_OK;
  CD_CHECK(cudaStreamSynchronize(g->stream));
  free_bins(g);
  g->t_warp = t_warp;
  g->t_hub = t_hub;
  return build_bins(g);
}

int ensure_bins(cd_graph* g) {
  if (g->bin_list) return CD_OK;
  const int rc = fill_bins(g);
  if (rc) {  // nothing half made stays; the counts do
    const int64_t nh = g->nhubs, ha = g->hub_arcs;
    free_bins(g);
    g->nhubs = nh;
    g->hub_arcs = ha;
  }
  return rc;
}

void drop_resident_hubs(cd_graph* g) { free_resident_hubs(g); }

int ensure_resident_hubs(cd_graph* g) {
  if (g->rh) return CD_OK;
  cudaStream_t s = g->stream;
  const int64_t nh = g->nhubs, items = g->hub_arcs / RH_CHUNK + nh;
  const int64_t slots = g->hub_arcs + g->hub_arcs / 2 + 64 * nh, slices = slots / RH_SLICE + nh;
  const bool wide = g->max_degw >= ((int64_t)1 << 32);
  ResidentHubs r;
  r.nh = (int32_t)nh;
  int rc;
  // 8-byte arrays first
  const size_t b8 = (size_t)((nh + 1) + 3 * slices + nh) * 8;
  const size_t b4 = (size_t)(nh + 2 * (nh + 1) + items + slices + 5 * nh + 1) * 4;
  if ((rc = dev_alloc(&r.mem[0], b8 + b4, s))) return rc;
  if ((rc = dev_alloc(&r.mem[1], (size_t)slots * (wide ? 12 : 8), s))) {
    dev_free(r.mem[0], s);
    return rc;
  }
  r.tab = (int64_t*)r.mem[0];
  r.part = r.tab + nh + 1;
  r.cur = r.part + 3 * slices;
  r.v = (int32_t*)(r.cur + nh);
  r.item = r.v + nh;
  r.slice = r.item + nh + 1;
  r.item_hub = r.slice + nh + 1;
  r.slice_hub = r.item_hub + items;
  r.done = r.slice_hub + slices;
  r.has = r.done + nh;
  r.moved = r.has + nh;
  r.to = r.moved + nh;
  r.from = r.to + nh;
  int32_t* count = r.from + nh;
  r.slot = (unsigned long long*)r.mem[1];
  r.key = wide ? (int32_t*)(r.slot + slots) : nullptr;
  auto run = [&]() -> int {
    CD_CHECK(cudaMemsetAsync(r.done, 0, (size_t)(2 * nh) * 4, s));  // done, has
    CD_CHECK(cudaMemsetAsync(count, 0, 4, s));
    CD_CHECK(cudaMemsetAsync(r.slot, wide ? 0 : 0xff, (size_t)slots * 8, s));
    if (wide) CD_CHECK(cudaMemsetAsync(r.key, 0xff, (size_t)slots * 4, s));
    CD_LAUNCH(k_rh_collect<<<grid_for(g->n), NT, 0, s>>>(g->off, g->n, g->t_hub, r.v, count));
    CD_LAUNCH(k_rh_layout<<<1, 1024, 0, s>>>(g->off, r));
    CD_CHECK(cudaGetLastError());
    return CD_OK;
  };
  if ((rc = run())) {
    dev_free(r.mem[0], s);
    dev_free(r.mem[1], s);
    return rc;
  }
  g->rh = new ResidentHubs(r);
  return CD_OK;
}

int ensure_run_state(cd_graph* g) {
  if (g->C) return CD_OK;
  const int64_t n32 = (g->n + 31) / 32 * 32;
  Arena a;
  a.add(&g->C, g->n);
  a.add(&g->sigma, g->n);
  a.add(&g->csize, g->n);
  a.add(&g->sigma32, g->vol < ((int64_t)1 << 31) ? g->n : 1);
  a.add(&g->flag[0], n32 / 32 + 1);
  a.add(&g->flag[1], n32 / 32 + 1);
  a.add(&g->mv_v, 3 * n32);
  a.add(&g->ctr, R_WORDS);
  const int rc = a.make(g->stream);
  if (rc) return rc;
  g->run_mem = a.mem;
  g->act_cnt = (unsigned long long*)g->ctr + R_ACT;
  g->hub_lcnt = (unsigned long long*)g->ctr + R_HUB_ITEMS;
  g->hub_ccnt = (unsigned long long*)g->ctr + R_HUB_CLASS;
  g->mv_c = g->mv_v + n32;
  g->mv_a = g->mv_v + 2 * n32;
  return CD_OK;
}

int check_labels(cd_graph* g, const int32_t* labels_dev) {
  if (g->n == 0) return CD_OK;
  CD_LAUNCH(k_labels_check<<<grid_for(g->n), NT, 0, g->stream>>>(labels_dev, g->n, g->status));
  CD_CHECK(cudaGetLastError());
  int st = read_status(g);
  return st ? st : CD_OK;
}

// Takes ownership of device arrays already in the internal convention (loop
// arcs carry 2L). If degw_pre is given (with its ingest stats) it is adopted
// too; otherwise deg_w is computed as the plain row sum.
int graph_adopt(cudaStream_t s, int64_t n, int64_t nnz, int64_t* off, int32_t* cols, void* w,
                int wkind, cd_graph** out, int64_t* degw_pre, const unsigned long long* stats_pre,
                const cd_graph* like, const unsigned long long* bins_pre) {
  cd_graph* g = new cd_graph();
  if (like) {
    g->t_warp = like->t_warp;
    g->t_hub = like->t_hub;
    g->bins_set = like->bins_set;
    g->workers = like->workers;
    if (!g->bins_set && nnz >= COARSE_HUB_ARCS && g->t_hub > COARSE_T_HUB && g->t_warp <= COARSE_T_HUB)
      g->t_hub = COARSE_T_HUB;
    if (g->t_hub != like->t_hub) bins_pre = nullptr;  // counted for the other threshold
  }
  g->stream = s;
  g->n = n;
  g->nnz = nnz;
  g->off = off;
  g->cols = cols;
  g->w = w;
  g->wkind = wkind;
  g->degw = degw_pre;
  profile_reset(g);
  int rc = dev_alloc_t(&g->status, 1, s);
  if (!rc && cudaMemsetAsync(g->status, 0, 4, s) != cudaSuccess) rc = CD_ECUDA;
  unsigned long long stats[NSTATS] = {};
  if (stats_pre) {
    memcpy(stats, stats_pre, sizeof(stats));
  } else {
    if (!rc) rc = dev_alloc_t(&g->degw, n, s);
    int32_t st = 0;
    if (!rc) rc = ingest(g, 0, stats, &st);
    if (!rc) rc = st;
  }
  // 64-bit weights whose every row sum (loops doubled included) is below 2^31
  // are kept in 32 bits: every arc weight is at most its row's deg_w
  if (!rc && g->wkind == W_I64 && g->w && nnz > 0 && stats[3] < (1ull << 31)) {
    int32_t* w32 = nullptr;
    rc = dev_alloc_t(&w32, nnz, s);
    if (!rc) {
      CD_LAUNCH(k_narrow_w<<<grid_for(nnz), NT, 0, s>>>((const int64_t*)g->w, nnz, w32));
      dev_free(g->w, s);
      g->w = w32;
      g->wkind = W_I32;
    }
  }
  if (!rc) rc = finish_graph(g, stats, bins_pre);
  if (rc) {
    free_arrays(g);
    delete g;
    return rc;
  }
  *out = g;
  return CD_OK;
}

}  // namespace cd

using namespace cd;

extern "C" {

int cd_params_default(cd_params* p) {
  if (!p) return CD_EINVAL;
  p->max_iter = 100;
  p->max_levels = 64;
  p->threshold = 0;
  p->tie_keep_current = 1;
  p->singleton_rule = 1;
  p->use_frontier = 1;
  p->timing = 0;
  p->sched_seed = 0x5EED5EEDull;
  p->aggregation = 0;
  p->asynchronous = 0;
  p->device_loop = 1;
  return CD_OK;
}

int cd_last_cuda_error(void) { return g_last_cuda; }

int64_t cd_launch_count(void) { return (int64_t)g_launches.load(); }

const char* cd_status_string(int st) {
  switch (st) {
    case CD_OK: return "ok";
    case CD_EINVAL: return "invalid argument (null pointer, size, weight < 1 or label out of range)";
    case CD_EBOUNDS: return "column id outside [0, n)";
    case CD_ENOMEM: return "device allocation failed";
    case CD_ECUDA: return "CUDA runtime error";
    case CD_EOVERFLOW: return "size overflow (vol(V) >= 2^62 or n >= 2^31)";
    case CD_ETIMEOUT: return "bounded device wait ran out";
    case CD_ENOTSYM: return "malformed CSR offsets";
    default: return "unknown status";
  }
}

int cd_csr_upload(const void* offsets, int offsets_is_i64, const int32_t* cols, const int32_t* w,
                  int64_t n, int64_t nnz, int ptrs_on_device, void* stream, cd_graph** out) {
  if (!out || n < 0 || nnz < 0 || !offsets || (nnz > 0 && !cols)) return CD_EINVAL;
  if (n >= (int64_t)INT32_MAX) return CD_EOVERFLOW;
  *out = nullptr;
  cudaStream_t s = (cudaStream_t)stream;
  cudaMemcpyKind kind = ptrs_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  cd_graph tmp;
  tmp.stream = s;
  tmp.n = n;
  tmp.nnz = nnz;
  profile_reset(&tmp);
  int rc = dev_alloc_t(&tmp.status, 1, s);
  int32_t* d_cols = nullptr;
  int64_t* d_off = nullptr;
  int32_t* d_w = nullptr;
  void* d_off_in = nullptr;
  if (!rc) rc = dev_alloc_t(&d_off, n + 1, s);
  if (!rc) rc = dev_alloc_t(&d_cols, nnz + COL_PAD, s);
  if (!rc && cudaMemsetAsync(d_cols + nnz, 0, COL_PAD * sizeof(int32_t), s) != cudaSuccess) rc = CD_ECUDA;
  if (!rc && w) rc = dev_alloc_t(&d_w, nnz, s);
  size_t ob = (size_t)(n + 1) * (offsets_is_i64 ? 8 : 4);
  if (!rc && !offsets_is_i64) rc = dev_alloc(&d_off_in, ob, s);
  auto cleanup = [&]() {
    dev_free(d_cols, s);
    dev_free(d_off, s);
    dev_free(d_w, s);
    dev_free(d_off_in, s);
    dev_free(tmp.status, s);
  };
  if (rc) {
    cleanup();
    return rc;
  }
  if (cudaMemsetAsync(tmp.status, 0, 4, s) != cudaSuccess ||
      cudaMemcpyAsync(offsets_is_i64 ? (void*)d_off : d_off_in, offsets, ob, kind, s) != cudaSuccess ||
      (nnz > 0 && cudaMemcpyAsync(d_cols, cols, (size_t)nnz * 4, kind, s) != cudaSuccess) ||
      (w && nnz > 0 && cudaMemcpyAsync(d_w, w, (size_t)nnz * 4, kind, s) != cudaSuccess)) {
    int e = set_cuda_error(cudaGetLastError());
    cleanup();
    return e;
  }
  if (offsets_is_i64)
    CD_LAUNCH(k_offsets_check<int64_t><<<grid_for(n + 1), NT, 0, s>>>(d_off, n, nnz, d_off,
                                                            tmp.status));
  else
    CD_LAUNCH(k_offsets_check<int32_t><<<grid_for(n + 1), NT, 0, s>>>((const int32_t*)d_off_in, n, nnz, d_off,
                                                            tmp.status));
  int32_t st = 0;
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(&st, tmp.status, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    cleanup();
    return CD_ECUDA;
  }
  dev_free(d_off_in, s);
  d_off_in = nullptr;
  if (st) {
    cleanup();
    return st;
  }
  // validate columns and weights, count loops, compute deg_w
  tmp.off = d_off;
  tmp.cols = d_cols;
  tmp.w = d_w;
  tmp.wkind = d_w ? W_I32 : W_UNIT;
  rc = dev_alloc_t(&tmp.degw, n, s);
  unsigned long long stats[NSTATS] = {};
  if (!rc) rc = ingest(&tmp, 1, stats, &st);
  if (!rc) rc = st;
  dev_free(tmp.status, s);
  tmp.status = nullptr;
  if (rc) {
    dev_free(tmp.degw, s);
    dev_free(d_cols, s);
    dev_free(d_off, s);
    dev_free(d_w, s);
    return rc;
  }
  // loops: switch to int64 weights with loop arcs doubled
  void* wint = d_w;
  int wk = d_w ? W_I32 : W_UNIT;
  if (stats[1] > 0) {
    int64_t* w64 = nullptr;
    rc = dev_alloc_t(&w64, nnz, s);
    if (rc) {
      dev_free(tmp.degw, s);
      dev_free(d_cols, s);
      dev_free(d_off, s);
      dev_free(d_w, s);
      return rc;
    }
    if (d_w)
      CD_LAUNCH(k_double_loops<WI32><<<grid_for(n * 32), NT, 0, s>>>(d_off, d_cols, d_w, n, w64));
    else
      CD_LAUNCH(k_double_loops<WUnit><<<grid_for(n * 32), NT, 0, s>>>(d_off, d_cols, nullptr, n, w64));
    dev_free(d_w, s);
    wint = w64;
    wk = W_I64;
  }
  // the ingest counted the degree bins, but not the arcs of the hubs
  unsigned long long bins[NBINS + 1] = {};
  for (int b = 0; b < NBINS; ++b) bins[b] = stats[4 + b];
  return graph_adopt(s, n, nnz, d_off, d_cols, wint, wk, out, tmp.degw, stats, nullptr,
                     bins[B_HUB] == 0 ? bins : nullptr);
}

int cd_graph_free(cd_graph* g) {
  if (!g) return CD_OK;
  free_arrays(g);
  for (auto& p : g->pending) {
    cudaEventDestroy(p.second.first);
    cudaEventDestroy(p.second.second);
  }
  cudaStreamSynchronize(g->stream);
  delete g;
  return CD_OK;
}

int cd_graph_info(const cd_graph* g, int64_t* n, int64_t* nnz, int64_t* vol) {
  if (!g) return CD_EINVAL;
  if (n) *n = g->n;
  if (nnz) *nnz = g->nnz;
  if (vol) *vol = g->vol;
  return CD_OK;
}

int cd_graph_download(const cd_graph* g, int64_t* off, int32_t* cols, int64_t* w, int on_device) {
  if (!g || !off || (g->nnz > 0 && !cols)) return CD_EINVAL;
  cudaStream_t s = g->stream;
  cudaMemcpyKind k = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  CD_CHECK(cudaMemcpyAsync(off, g->off, (g->n + 1) * 8, k, s));
  if (g->nnz > 0) CD_CHECK(cudaMemcpyAsync(cols, g->cols, g->nnz * 4, k, s));
  if (w && g->nnz > 0) {
    int64_t* tmp = nullptr;
    int rc = dev_alloc_t(&tmp, g->nnz, s);
    if (rc) return rc;
    CD_LAUNCH(k_download_w<<<grid_for(g->n * 32), NT, 0, s>>>(g->off, g->cols, g->w, g->wkind, g->n, tmp));
    CD_CHECK(cudaMemcpyAsync(w, tmp, g->nnz * 8, k, s));
    dev_free(tmp, s);
  }
  CD_CHECK(cudaStreamSynchronize(s));
  return CD_OK;
}

int cd_trace_get(const cd_graph* g, cd_round_trace* out, int32_t cap, int32_t* count) {
  if (!g || !count) return CD_EINVAL;
  *count = (int32_t)g->trace.size();
  for (int32_t i = 0; i < cap && i < (int32_t)g->trace.size(); ++i) out[i] = g->trace[i];
  return CD_OK;
}

int cd_profile_get(const cd_graph* g, cd_kernel_profile* out, int32_t cap, int32_t* count) {
  if (!g || !count) return CD_EINVAL;
  *count = K_COUNT;
  for (int32_t i = 0; i < cap && i < K_COUNT; ++i) out[i] = g->prof[i];
  return CD_OK;
}

}  // extern "C"
