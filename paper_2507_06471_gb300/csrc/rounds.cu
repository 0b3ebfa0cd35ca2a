// The round loop of a run or Louvain level as one resident kernel, for graphs
// without hubs or with few of them up to the sizes of resident_arcs: every round
// of Label Propagation (Algorithm 1) or local moving (Algorithm 2), synchronous,
// with the decisions, coins, counters and stop tests of the per-round kernels in
// scan.cu (the results are the same).
//
// Why: a round of a small graph, or a late round of a large one, examines few
// vertices, and its time is latency: a dozen launches of 3 to 8 us each, a
// compaction over all n list entries, a read-back and a synchronisation. The
// 10,000-vertex planted partition took 49 us a round that way (43 rounds, 2.1
// ms), the 1M-vertex LFR-style graph 165 us (233 rounds, 38.5 ms). So: 12 us a
// round (0.50 ms) and 75 us (17.4 ms). What bounds a small round is then the
// chain of one warp's work (flags, offsets, columns, labels, Sigma_tot: dependent
// loads) and the two barriers; what bounds a large one is the instructions of the
// table inserts.
//
// How: one cooperative launch of at most one wave of 256-thread CTAs. The
// vertices are dealt out in units of 1 to 32 consecutive ids round robin, so
// that every CTA gets an even share of whatever is active. In a round a CTA
//   1. takes its vertices' flags, sorts the flagged ones by degree bin into a list in
//      shared memory and scans them: a half CTA per vertex of degree t_warp+1
//      to 1,024, warps for degree 33..t_warp and 4/8/16/32-lane tiles below
//      (tasks taken from a counter in shared memory, longest first); it marks
//      the neighbours of its moves in the next map and keeps its moves;
//   2. meets the others at a barrier whose one atomic per CTA also sums moved +
//      deferred (the stop test);
//   3. applies its moves (labels, Sigma_tot, sizes), clears its part of the map
//      it read, and meets the others again.
// Hubs (degree above t_hub) that are examined in a round have their label
// histograms built in step 1, by items of 1,024 arcs dealt out over the half
// CTAs (combined in shared memory, then added to the hub's table in global
// memory); after the first barrier the tables are read by slices, cleared while
// read, and the last slice of a hub decides; a third barrier then comes before
// step 3. The per-round kernels keep the histograms from round to round instead,
// which pays on large graphs: see resident_rounds_apply.
// The grid has at most as many CTAs as are resident at once (cooperative
// launch), so the barrier's waits end; they are bounded all the same.
//
// Sigma_tot is kept in 32 bits when vol(V) < 2^31 (integers: exact), in 64
// otherwise.
#include <algorithm>

#include "scan.cuh"

namespace cd {
namespace {

constexpr int PNT = 256, PNW = PNT / 32;  // threads and warps of a CTA
constexpr int PCAP = WARP_CAP_SLOTS;      // table slots per warp; four warps' tables make a half CTA's
static_assert(4 * PCAP == BLK1_CAP_SLOTS, "a half CTA's table is its four warps' tables");
constexpr int CH_VERTS = 2048;            // vertices a CTA takes per step
constexpr int CH_PER_WARP = CH_VERTS / PNT;
// Arcs per CTA at least (or vertices enough for a step): a small graph gets fewer CTAs, which meet faster.
constexpr int64_t ARCS_PER_CTA = 512;
constexpr int PBINS = 6;                  // task order: half CTA, warp, 32, 16, 8, 4 lanes
// Arcs of a loop that takes a share of the GPU (the server's workers) at most:
// larger graphs are bound by the work of their rounds, and the per-round kernels
// of several workers fill the GPU better. 256 requests of up to 2e6 vertices,
// four workers: 67 requests/s with every loop on a quarter of the GPU, 105 with
// the large ones on all of it (graphs without hubs), 120 so.
constexpr int64_t SHARED_LOOP_ARCS = (int64_t)1 << 22;
// Isolated vertices at most, where they are the majority: the resident loop looks
// at every vertex's flag each round, the per-round kernels' lists leave them out.
// LPA with 1e6 arcs among 1e5 vertices: 2.85 -> 1.76 ms with 1e7 vertices in all,
// 3.08 -> 5.58 ms with 5e7. Graphs of few isolated vertices need no such line: the
// lists then hold every vertex and are gone through every round too (1e8 vertices
// of degree 3, a ring and a matching: LPA 93 -> 42 ms, local moving 138 -> 70; degree
// 2: 58 -> 30 and 62 -> 41). What limits those is their arcs, see resident_arcs.
constexpr int64_t MAX_ISOLATED = (int64_t)1 << 23;
// Arcs of a run at most. The resident loop saves what a round costs beside its
// work; the per-round kernels do the work itself faster (more warps per SM, rows dealt
// out as they are flagged and not by vertex, hub histograms kept from round to round),
// all the more without a frontier, where every round is a full one, and for local
// moving, whose rounds hold more work. Resident time over that of the per-round
// kernels (captured, below 2^22 arcs the host loop), at both sides of the lines:
//   hubs (R-MAT, edge factors 4 to 32)   LPA         1.5e6..8.2e6 0.40..0.93   1.5e7 1.22..1.43
//                                        local move  1.6e6..4.1e6 0.45..1.09   7e6..8.2e6 1.05..1.67
//     without a frontier                 LPA         1.6e6..4.1e6 0.46..0.82   7e6..8.2e6 0.94..1.39
//                                        local move  1.6e6..2.0e6 0.54..1.25   3.4e6..4.1e6 0.70..1.79
//   no hubs, mean degree 32 to 128       LPA         3e6..3.2e7 0.50..0.92     3.8e7..1.9e8 0.99..1.19
//                                        local move  3e6..1.3e7 0.44..0.91     1.9e7..1.9e8 1.06..1.45
//     8 to 20 (LFR-style 12)             LPA         to 1.6e8 0.30..0.99
//                                        local move  to 2.4e7 0.34..1.02       3.6e7..1.6e8 0.90..1.62
//     2 to 4                             both        to 3e8 0.27..1.00
//     without a frontier, any degree     LPA         to 1.6e7 0.35..1.06       1.9e7..1.6e8 0.91..1.29
//                                        local move  to 8e6 0.42..0.95         9.6e6..1.9e8 0.95..1.75
//   (4,000 stars of 400 arcs over a sparse graph, 4e6 arcs: local move 1.16, 1.29 without a frontier)
// Batched runs are held to 2^24 without a frontier only (Louvain: 1.1e7 0.89, 4.7e7
// and 5.7e7 1.09..1.15; with one 0.45..0.83 to 5.7e7): most of their graphs stop early.
constexpr int64_t MEAN_LOW = 4, MEAN_MID = 24;  // mean degrees of vertices that have arcs
inline int64_t resident_arcs(const cd_graph* g, const RunOpts& o, bool louv) {
  if (o.batched) return o.use_frontier ? INT64_MAX : (int64_t)1 << 24;
  int64_t most = (int64_t)1 << (g->nhubs ? 23 : 25);
  if (g->nhubs == 0 && o.use_frontier) {
    const int64_t linked = g->n - g->n_isolated;
    if (g->nnz <= (louv ? MEAN_LOW : MEAN_MID) * linked) return INT64_MAX;
    if (g->nnz <= MEAN_MID * linked) return most;
  }
  if (louv) most /= 2;
  return o.use_frontier ? most : most / 2;
}
constexpr int TRACE_COLS = 8;             // examined, arcs, moved, deferred, candidates, arcs of moved, -, -
constexpr int HEAD = 8;                   // int64 words before the trace: rounds, moves, status
constexpr int64_t WAIT_LIMIT = (int64_t)1 << 24;  // polls of one barrier at most (seconds), then CD_ETIMEOUT

struct LoopCtx {
  int64_t n, nwords, n32;  // vertices, flag words, vertices rounded up to whole words
  int64_t nunits;          // units of 1 << lgu consecutive vertices; unit q belongs to CTA q mod gridDim.x
  int32_t lgu;
  uint32_t* flag0;  // read in even rounds, written in odd ones
  uint32_t* flag1;
  int32_t max_iter, first_rows, t_warp, t_hub, per_graph;
  int64_t threshold;
  int64_t polls;              // of a barrier at most
  int32_t* last_change;       // per_graph: 1 + the last round in which a vertex of the graph wanted to move
  unsigned long long* bar;    // three words per round, zero
  unsigned long long* head;   // HEAD words, then TRACE_COLS per round, zero
  uint32_t* sigma32;          // NK: Sigma_tot
  ResidentHubs rh;            // rh.nh = 0: none
};

// Every CTA arrives once; `add` (changed vertices, < 2^32 in all) and `hubs`
// are summed over the CTAs (at most 2^15). False: a wait ran out.
__device__ __forceinline__ bool grid_meet(unsigned long long* word, unsigned add, unsigned hubs, unsigned& sum,
                                          unsigned& hub_sum, int64_t limit, int32_t* status) {
  __shared__ unsigned long long got;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(word, (1ull << 48) | ((unsigned long long)hubs << 32) | add);
    unsigned long long x;
    int64_t polls = 0;
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(word) : "memory");
      if ((x >> 48) >= gridDim.x || ++polls >= limit) break;
      __nanosleep(40);  // arrivals go to the same word
    }
    if ((x >> 48) < gridDim.x) {
      atomicCAS(status, 0, CD_ETIMEOUT);
      x = ~0ull;
    }
    __threadfence();
    got = x;
  }
  __syncthreads();
  const unsigned long long x = got;
  sum = (unsigned)x;
  hub_sum = (unsigned)(x >> 32) & 0xffffu;
  return x != ~0ull;
}

// Barrier of a half CTA (fixed numbers: a number in a register would reserve all sixteen).
__device__ __forceinline__ void half_sync(int half) {
  if (half) asm volatile("bar.sync 2, 128;" ::: "memory");
  else asm volatile("bar.sync 1, 128;" ::: "memory");
}

// One CTA's part of a round.
struct Tally {
  uint32_t act = 0, arcs = 0, cand = 0, def = 0, marcs = 0;
};

__device__ __forceinline__ void set_flag(uint32_t* nxt, int32_t u) { atomicOr(&nxt[u >> 5], 1u << (u & 31)); }

template <bool LOUV, class W, class V, bool NK>
struct Scan {
  typedef typename KeyOf<LOUV, NK>::T K;
  const ScanCtx& s;
  const LoopCtx& L;
  int round;
  bool first;        // every label is the vertex's own id and no row repeats a column
  uint32_t* nxt;     // null: no frontier
  int32_t* mv;       // this CTA's moves: vertex, new, old label in three arrays of mv_stride
  int64_t mv_stride;
  int* n_mv;         // in shared memory

  // The lanes with `want` hold a vertex v whose decision `target` differs from
  // its label: coin, move list, flag. Returns whether the lane's move commits.
  __device__ __forceinline__ bool act(bool want, int32_t v, int32_t cur, int32_t target) const {
    const int lane = threadIdx.x & 31;
    const bool commit = want && commit_coin(s.seed, s.level, round, local_id(s, v));
    const unsigned cm = __ballot_sync(FULL, commit);
    if (cm) {
      const int lead = __ffs(cm) - 1;
      int p0 = 0;
      if (lane == lead) p0 = atomicAdd(n_mv, __popc(cm));
      p0 = __shfl_sync(FULL, p0, lead);
      if (commit) {
        const int64_t p = p0 + __popc(cm & ((1u << lane) - 1u));
        mv[p] = v;
        mv[mv_stride + p] = target;
        mv[2 * mv_stride + p] = cur;
      }
    }
    if (want) {
      if (nxt) set_flag(nxt, v);
      if (L.per_graph) L.last_change[s.gid[v]] = round + 1;
    }
    return commit;
  }

  // 2^lgt lanes per vertex, one arc per lane; the warp takes 32 >> lgt vertices
  // of list[0, count) from `base` on.
  __device__ __forceinline__ void tile(const int32_t* list, int base, int count, int lgt, int64_t* stage,
                                       Tally& t) const {
    const int lane = threadIdx.x & 31;
    const int tw = 1 << lgt, sub = lane & (tw - 1), tbase = lane - sub;
    const unsigned tmask = (tw == 32 ? FULL : ((1u << tw) - 1u)) << tbase;
    const int i = base + (lane >> lgt);
    const bool on = i < count;
    const int32_t v = on ? list[i] : 0;
    int64_t beg = 0;
    int d = 0;
    if (on) {
      beg = __ldg(s.off + v);
      d = (int)(__ldg(s.off + v + 1) - beg);
    }
    const int32_t cur = on ? s.C[v] : 0;
    const bool has = on && sub < d;
    const int32_t u = has ? __ldg(s.cols + beg + sub) : v;
    const int64_t wt = has ? W::get(s.w, beg + sub) : 0;
    const int64_t dv = (LOUV && on) ? __ldg(s.degw + v) : 0;
    const int64_t volv = (LOUV && on) ? vol_of(s, v) : 0;
    const bool cand = has && u != v;
    const int32_t lbl = cand ? (first ? u : s.C[u]) : (int32_t)(0x80000000u | (unsigned)lane);
    const unsigned peers = __match_any_sync(FULL, lbl) & tmask;
    const int64_t gsum = group_sum<W>(peers, wt, stage, sizeof(V) == 4);
    const bool leader = cand && (__ffs(peers) - 1) == lane;
    const unsigned cm = __ballot_sync(FULL, cand && lbl == cur) & tmask;
    int64_t kcur = __shfl_sync(FULL, gsum, cm ? __ffs(cm) - 1 : lane);
    if (!cm) kcur = 0;
    const bool ok = leader && (!LOUV || lbl != cur);
    K bk = ok ? cand_key<LOUV, NK>(s, lbl, gsum, dv, volv) : no_key<K>();
    int32_t bc = ok ? lbl : NOCAND;
    reduce_best(bk, bc, tw);
    int32_t target = cur;
    if (on) target = decide<LOUV, NK>(s, v, cur, bk, bc, cm != 0, kcur, volv);
    const bool want = on && target != cur;
    const bool mine = act(want && sub == 0, v, cur, target);
    const bool commit = __shfl_sync(FULL, (int)mine, tbase) != 0;
    if (nxt && commit && has) set_flag(nxt, u);  // the neighbours of a moved vertex
    if (sub == 0 && on) {
      ++t.act;
      t.arcs += d;
      if (want && !mine) ++t.def;
      if (mine) t.marcs += d;
    }
    if (leader) ++t.cand;
  }

  // A warp takes the vertices list[base, base + vb): lane j loads vertex j's
  // header, the warp scans the rows one after another, and the decisions run
  // one lane per vertex.
  __device__ __forceinline__ void warp_batch(const int32_t* list, int base, int count, int vb, int32_t* keys, V* vals,
                                             uint16_t* occ, int* occ_n, Tally& t) const {
    const int lane = threadIdx.x & 31;
    const bool on = lane < vb && base + lane < count;
    const int32_t my_v = on ? list[base + lane] : 0;
    int64_t my_beg = 0, my_end = 0, my_dv = 0, my_vol = 0;
    int32_t my_cur = 0;
    if (on) {
      my_beg = __ldg(s.off + my_v);
      my_end = __ldg(s.off + my_v + 1);
      my_cur = s.C[my_v];
      if (LOUV) {
        my_dv = __ldg(s.degw + my_v);
        my_vol = vol_of(s, my_v);
      }
    }
    K my_bk = no_key<K>();
    int32_t my_bc = NOCAND;
    bool my_hc = false;
    int64_t my_kc = 0, ncand = 0;
    for (unsigned am = __ballot_sync(FULL, on); am; am &= am - 1) {
      const int j = __ffs(am) - 1;
      const int32_t v = __shfl_sync(FULL, my_v, j), cur = __shfl_sync(FULL, my_cur, j);
      const int64_t beg = __shfl_sync(FULL, my_beg, j), end = __shfl_sync(FULL, my_end, j);
      const int64_t dv = LOUV ? __shfl_sync(FULL, my_dv, j) : 0;
      const int64_t volv = LOUV ? __shfl_sync(FULL, my_vol, j) : 0;
      K bk = no_key<K>();
      int32_t bc = NOCAND;
      bool hc = false;
      int64_t kc = 0;
      if (first) {  // distinct labels along the row: no table
        for (int64_t e = beg + lane; e < end; e += 32) {
          const int32_t u = __ldg(s.cols + e);
          if (u == v) continue;
          const K key = cand_key<LOUV, NK>(s, u, W::get(s.w, e), dv, volv);
          ++ncand;
          if (better(key, u, bk, bc)) {
            bk = key;
            bc = u;
          }
        }
        reduce_best(bk, bc, 32);
      } else {
        const unsigned lg = 64 - __clzll((unsigned long long)(2 * (end - beg) - 1));  // 2^lg >= 2 deg
        group_insert<W, V, 32>(s, v, beg, end, lane, keys, vals, occ, occ_n, lg);
        __syncwarp();
        group_eval<LOUV, V, 32, NK>(s, cur, dv, volv, lane, keys, vals, occ, *occ_n, bk, bc, hc, kc, ncand);
        reduce_best(bk, bc, 32);
        const unsigned hm = __ballot_sync(FULL, hc);
        hc = hm != 0;
        if (hm) kc = __shfl_sync(FULL, kc, __ffs(hm) - 1);
        __syncwarp();
        if (lane == 0) *occ_n = 0;
        __syncwarp();
      }
      if (lane == j) {
        my_bk = bk;
        my_bc = bc;
        my_hc = hc;
        my_kc = kc;
      }
    }
    int32_t target = my_cur;
    if (on) target = decide<LOUV, NK>(s, my_v, my_cur, my_bk, my_bc, my_hc, my_kc, my_vol);
    const bool want = on && target != my_cur;
    const bool commit = act(want, my_v, my_cur, target);
    if (on) {
      const uint32_t d = (uint32_t)(my_end - my_beg);
      ++t.act;
      t.arcs += d;
      if (want && !commit) ++t.def;
      if (commit) t.marcs += d;
    }
    t.cand += (uint32_t)ncand;
    if (nxt)
      for (unsigned m = __ballot_sync(FULL, commit); m; m &= m - 1) {
        const int j = __ffs(m) - 1;
        const int64_t beg = __shfl_sync(FULL, my_beg, j), end = __shfl_sync(FULL, my_end, j);
        for (int64_t e = beg + lane; e < end; e += 32) set_flag(nxt, __ldg(s.cols + e));
      }
  }

  // A half CTA (128 threads, named barrier `half` + 1) scans vertex v with the
  // four warps' tables as one.
  struct HalfRed {
    K k[4];
    int64_t kc[4];
    int32_t c[4], hc[4];
    int32_t moved;
  };
  __device__ __forceinline__ void half_cta(int32_t v, int half, int32_t* keys, V* vals, uint16_t* occ, int* occ_n,
                                           HalfRed* red, Tally& t) const {
    const int lane = threadIdx.x & 31, gl = threadIdx.x & 127, wig = gl >> 5;
    const int64_t beg = __ldg(s.off + v), end = __ldg(s.off + v + 1);
    const int32_t cur = s.C[v];
    const int64_t dv = LOUV ? __ldg(s.degw + v) : 0;
    const int64_t volv = LOUV ? vol_of(s, v) : 0;
    const unsigned lg = 64 - __clzll((unsigned long long)(2 * (end - beg) - 1));
    group_insert<W, V, 128>(s, v, beg, end, gl, keys, vals, occ, occ_n, lg);
    half_sync(half);
    K bk = no_key<K>();
    int32_t bc = NOCAND;
    bool hc = false;
    int64_t kc = 0, ncand = 0;
    group_eval<LOUV, V, 128, NK>(s, cur, dv, volv, gl, keys, vals, occ, *occ_n, bk, bc, hc, kc, ncand);
    t.cand += (uint32_t)ncand;
    reduce_best(bk, bc, 32);
    unsigned hm = __ballot_sync(FULL, hc);
    if (hm) kc = __shfl_sync(FULL, kc, __ffs(hm) - 1);
    if (lane == 0) {
      red->k[wig] = bk;
      red->c[wig] = bc;
      red->hc[wig] = hm != 0;
      red->kc[wig] = kc;
    }
    half_sync(half);
    if (wig == 0) {
      bk = lane < 4 ? red->k[lane] : no_key<K>();
      bc = lane < 4 ? red->c[lane] : NOCAND;
      reduce_best(bk, bc, 32);
      hm = __ballot_sync(FULL, lane < 4 && red->hc[lane & 3]);
      kc = hm ? red->kc[__ffs(hm) - 1] : 0;
      int32_t target = cur;
      if (lane == 0) target = decide<LOUV, NK>(s, v, cur, bk, bc, hm != 0, kc, volv);
      const bool want = lane == 0 && target != cur;
      const bool commit = act(want, v, cur, target);
      if (lane == 0) {
        ++t.act;
        t.arcs += (uint32_t)(end - beg);
        if (want && !commit) ++t.def;
        if (commit) t.marcs += (uint32_t)(end - beg);
        *occ_n = 0;
        red->moved = commit;
      }
    }
    half_sync(half);
    if (red->moved && nxt)
      for (int64_t e = beg + gl; e < end; e += 128) set_flag(nxt, __ldg(s.cols + e));
    half_sync(half);  // red is written again for the next vertex
  }
};

__device__ __forceinline__ bool flagged(const uint32_t* map, int32_t v) {
  return !map || ((__ldcg(map + (v >> 5)) >> (v & 31)) & 1u);
}

// Add `w` arcs of `label` to hub h's table.
template <class V>
__device__ __forceinline__ void rh_add(const ResidentHubs& r, int64_t base, int64_t cap, int32_t label, V w) {
  int64_t at = hub_home(label, cap);
  for (int64_t probe = 0; probe < cap; ++probe) {  // at most two thirds of the slots fill: always ends
    if constexpr (sizeof(V) == 4) {
      unsigned long long* p = r.slot + base + at;
      unsigned long long x = *(volatile unsigned long long*)p;
      if (x == SLOT_EMPTY) {
        x = atomicCAS(p, SLOT_EMPTY, ((unsigned long long)(uint32_t)label << 32) | w);
        if (x == SLOT_EMPTY) return;
      }
      if ((int32_t)(x >> 32) == label) {
        atomicAdd(p, (unsigned long long)w);
        return;
      }
    } else {
      int32_t x = *(volatile int32_t*)(r.key + base + at);
      if (x == EMPTY) x = atomicCAS(r.key + base + at, EMPTY, label);
      if (x == EMPTY || x == label) {
        atomicAdd(r.slot + base + at, (unsigned long long)w);
        return;
      }
    }
    at = at + 1 == cap ? 0 : at + 1;
  }
}

// The items of examined hubs that fall to this half CTA: build. Returns whether there was one.
template <class W, class V>
__device__ __forceinline__ bool rh_build(const ScanCtx& s, const ResidentHubs& r, const uint32_t* map, int half,
                                         int32_t* keys, V* vals, uint16_t* occ, int* occ_n) {
  const int gl = threadIdx.x & 127;
  const int n_items = r.item[r.nh];
  bool any = false;
  for (int it = blockIdx.x * 2 + half; it < n_items; it += gridDim.x * 2) {
    const int h = __ldg(r.item_hub + it);
    const int32_t v = __ldg(r.v + h);
    if (!flagged(map, v) || (s.gfrozen && s.gfrozen[s.gid[v]])) continue;  // uniform in the half CTA
    any = true;
    const int64_t beg = __ldg(s.off + v) + (int64_t)(it - __ldg(r.item + h)) * RH_CHUNK, row_end = __ldg(s.off + v + 1);
    const int64_t end = beg + RH_CHUNK < row_end ? beg + RH_CHUNK : row_end;
    const int64_t base = __ldg(r.tab + h), cap = __ldg(r.tab + h + 1) - base;
    group_insert<W, V, 128>(s, v, beg, end, gl, keys, vals, occ, occ_n, 11);
    half_sync(half);
    const int n = *occ_n;
    for (int j = gl; j < n; j += 128) {
      const int q = occ[j];
      const int32_t label = keys[q];
      const V w = vals[q];
      keys[q] = EMPTY;
      vals[q] = 0;
      rh_add<V>(r, base, cap, label, w);
    }
    half_sync(half);
    if (gl == 0) *occ_n = 0;
    half_sync(half);
  }
  return any;
}
static_assert(RH_CHUNK <= BLK1_MAX, "an item fits a half CTA's table");

// One move per lane with `ok`: vertex v from community `from` to `to`.
template <bool LOUV, bool NK>
__device__ __forceinline__ void apply_moves(const ScanCtx& s, const LoopCtx& L, bool ok, int32_t v, int32_t to,
                                            int32_t from, int64_t* stage) {
  const int lane = threadIdx.x & 31;
  if (ok) s.C_w[v] = to;
  if constexpr (LOUV) {
    const int64_t d = ok ? __ldg(s.degw + v) : 0;
    // one atomic per distinct community of the warp: popular targets would serialise
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const int32_t key = side ? from : to;
      const unsigned peers = __match_any_sync(FULL, key);
      stage[lane] = side ? -d : d;
      __syncwarp();
      if (key >= 0 && (__ffs(peers) - 1) == lane) {
        int64_t sum = 0;
        for (unsigned m = peers; m; m &= m - 1) sum += stage[__ffs(m) - 1];
        if constexpr (NK) atomicAdd(&L.sigma32[key], (uint32_t)sum);
        else atomicAdd((unsigned long long*)&s.sigma_w[key], (unsigned long long)sum);
        atomicAdd(&s.csize_w[key], side ? -__popc(peers) : __popc(peers));
      }
      __syncwarp();
    }
  }
}

// Step 1's sorting: the flagged ones of the CTA's vertices c0 .. c0 + NG PNT into
// `list` by degree bin, with the bins' starts in first_of (cnt: vertices per
// bin, zero before). False: none. A warp without one skips what follows, and so
// does a group of 32 in it: late rounds have few, and this was most of a small
// graph's instructions.
template <int NG>
__device__ __forceinline__ bool collect(const ScanCtx& s, const LoopCtx& L, const uint32_t* map, uint32_t c0,
                                        uint32_t my_verts, int* cnt, int* start, int32_t* list,
                                        int first_of[PBINS + 1]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t i0 = c0 + wid * NG * 32 + lane;
  int32_t vk[NG];
#pragma unroll
  for (int k = 0; k < NG; ++k) {
    vk[k] = -1;
    const uint32_t i = i0 + 32 * k;
    if (i - lane >= my_verts) continue;  // uniform in the warp
    const uint32_t v = ((blockIdx.x + (i >> L.lgu) * gridDim.x) << L.lgu) + (i & ((1u << L.lgu) - 1u));
    if (i < my_verts && v < (uint32_t)L.n) vk[k] = (int32_t)v;
  }
  if (map) {
    uint32_t fw[NG];
#pragma unroll
    for (int k = 0; k < NG; ++k) fw[k] = vk[k] >= 0 ? __ldcg(map + (vk[k] >> 5)) : 0;
#pragma unroll
    for (int k = 0; k < NG; ++k)
      if (!((fw[k] >> (vk[k] & 31)) & 1u)) vk[k] = -1;
  }
  unsigned some = 0;  // the groups of 32 with a flagged vertex
#pragma unroll
  for (int k = 0; k < NG; ++k) some |= __any_sync(FULL, vk[k] >= 0) ? 1u << k : 0u;
  if (!__syncthreads_or(some != 0)) return false;
  int slot[NG];  // bin << 16 | rank, -1: none
#pragma unroll
  for (int k = 0; k < NG; ++k) {
    slot[k] = -1;
    if (!((some >> k) & 1u)) continue;
    if (vk[k] >= 0) {
      const int32_t v = vk[k];
      int64_t d = __ldg(s.off + v + 1) - __ldg(s.off + v);
      if (s.gfrozen && s.gfrozen[s.gid[v]]) d = 0;
      if (d > 0 && d <= L.t_hub) {  // hubs: by items
        const int bin = d <= 4 ? 5 : d <= 8 ? 4 : d <= 16 ? 3 : d <= 32 ? 2 : d <= L.t_warp ? 1 : 0;
        slot[k] = (bin << 16) | atomicAdd(&cnt[bin], 1);
      }
    }
  }
  __syncthreads();
  first_of[0] = 0;
#pragma unroll
  for (int q = 0; q < PBINS; ++q) first_of[q + 1] = first_of[q] + cnt[q];
  if (some) {
#pragma unroll
    for (int q = 0; q < PBINS; ++q)
      if (lane == q) start[q] = first_of[q];
    __syncwarp();
#pragma unroll
    for (int k = 0; k < NG; ++k)
      if (slot[k] >= 0) list[start[slot[k] >> 16] + (slot[k] & 0xffff)] = vk[k];
  }
  return true;
}

template <class V> constexpr size_t loop_smem() {
  return (size_t)PNW * PCAP * (sizeof(V) + 4 + 2) + (size_t)PNW * 32 * 8 + (size_t)CH_VERTS * 4;
}

template <bool LOUV, class W, class V, bool NK>
__global__ void __launch_bounds__(PNT, sizeof(V) == 4 ? 4 : 3) k_rounds(const __grid_constant__ ScanCtx s,
                                                                       const __grid_constant__ LoopCtx L) {
  typedef Scan<LOUV, W, V, NK> S;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ typename S::HalfRed red[2];
  __shared__ int occ_n[PNW];
  __shared__ int bincnt[2][8];  // by parity of the step: vertices per bin, then [7]: next task
  __shared__ int n_mv;
  // A CTA's counters of a round, then the high words of those that count arcs: 456 CTAs (the fewest that fill the GPU;
  // smaller grids have few arcs) of 2^31 vertices of up to 1,024 arcs may have 4.8e9 each. A thread's stay below 2^32.
  __shared__ uint32_t sums[5], sums_hi[5];
  __shared__ int hub_moves, s_last;
  __shared__ int start[PNW][8];
  __shared__ typename S::K red_k[PNW];
  __shared__ int32_t red_c[PNW];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, half = tid >> 7;
  V* vals0 = (V*)smem;
  int32_t* keys0 = (int32_t*)(smem + (size_t)PNW * PCAP * sizeof(V));
  int64_t* stage = (int64_t*)(smem + (size_t)PNW * PCAP * (sizeof(V) + 4)) + wid * 32;
  int32_t* list = (int32_t*)(smem + (size_t)PNW * PCAP * (sizeof(V) + 4) + (size_t)PNW * 32 * 8);
  uint16_t* occ0 = (uint16_t*)(list + CH_VERTS);
  for (int j = tid; j < PNW * PCAP; j += PNT) {
    keys0[j] = EMPTY;
    vals0[j] = 0;
  }
  if (tid < PNW) occ_n[tid] = 0;
  if (tid < 16) bincnt[tid >> 3][tid & 7] = 0;
  __syncthreads();
  // this CTA's units: blockIdx.x + i gridDim.x; its moves have room for all their vertices
  const int64_t G = gridDim.x, b = blockIdx.x;
  const uint32_t my_verts = (uint32_t)(L.nunits / G + (b < L.nunits % G ? 1 : 0)) << L.lgu;
  const int64_t mv_at = (b * (L.nunits / G) + (b < L.nunits % G ? b : L.nunits % G)) << L.lgu;
  int32_t* mv = s.mv_v + mv_at;
  const int64_t mv_stride = L.n32;
  int step = 0;
  int32_t round = 0;
  // the CTA's counters of a round, added to the round's trace row; returns moved + deferred
  auto account = [&](const Tally& t, int more_moves) -> unsigned {
    if (__any_sync(FULL, t.act | t.cand)) {
      const uint32_t c[5] = {t.act, t.arcs, t.cand, t.def, t.marcs};
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        unsigned long long x = __reduce_add_sync(FULL, q == 0 || q == 3 ? c[q] : c[q] & 0xffffu);
        if (q != 0 && q != 3) x += (unsigned long long)__reduce_add_sync(FULL, c[q] >> 16) << 16;
        if (lane == 0 && x) add_words(&sums[q], &sums_hi[q], x);
      }
    }
    __syncthreads();
    const int nm = more_moves ? hub_moves : n_mv;
    const unsigned changed = (unsigned)nm + sums[3];
    if (tid < 6) {
      const int q = tid < 2 ? tid : tid == 3 ? 3 : tid == 4 ? 2 : 4;
      const unsigned long long x = tid == 2 ? (unsigned long long)nm : ((unsigned long long)sums_hi[q] << 32) | sums[q];
      if (x) atomicAdd(&L.head[HEAD + (int64_t)round * TRACE_COLS + tid], x);
    }
    return changed;
  };
  for (; round < L.max_iter;) {
    uint32_t* cur_map = round & 1 ? L.flag1 : L.flag0;
    uint32_t* nxt_map = round & 1 ? L.flag0 : L.flag1;
    const bool frontier = s.mark != 0;
    if (tid == 0) n_mv = hub_moves = 0;
    if (tid < 5) sums[tid] = sums_hi[tid] = 0;
    const S sc{s, L, round, round == 0 && L.first_rows, frontier ? nxt_map : nullptr, mv, mv_stride, &n_mv};
    Tally t;
    bool hubs_here = false;
    if (L.rh.nh)
      hubs_here = rh_build<W, V>(s, L.rh, frontier ? cur_map : nullptr, half, keys0 + half * 4 * PCAP,
                                 vals0 + half * 4 * PCAP, occ0 + half * 4 * PCAP, &occ_n[half * 4]);
    for (uint32_t c0 = 0; c0 < my_verts; c0 += CH_VERTS) {
      int* cnt = bincnt[step & 1];
      int first_of[PBINS + 1];  // where each bin starts in the list
      const bool any = my_verts - c0 <= PNT
                           ? collect<1>(s, L, frontier ? cur_map : nullptr, c0, my_verts, cnt, start[wid], list, first_of)
                           : collect<CH_PER_WARP>(s, L, frontier ? cur_map : nullptr, c0, my_verts, cnt, start[wid], list,
                                                  first_of);
      if (!any) continue;
      if (tid < 8) bincnt[(step + 1) & 1][tid] = 0;  // the next step's
      __syncthreads();
      // half CTAs
      int n_half = first_of[1];
      if (!sc.first) {
        // a few: one half takes them while the other starts on the warps' tasks
        for (int i = n_half < 4 ? (half ? n_half : 0) : half; i < n_half; i += n_half < 4 ? 1 : 2)
          sc.half_cta(list[i], half, keys0 + half * 4 * PCAP, vals0 + half * 4 * PCAP, occ0 + half * 4 * PCAP,
                      &occ_n[half * 4], &red[half], t);
      } else {
        n_half = 0;  // rows without tables: the warps take them
      }
      // warps: batches of wb vertices of the warp bin, then tiles
      const int nw = first_of[2] - n_half;
      int wb = (nw + PNW - 1) / PNW;
      wb = wb < 1 ? 1 : wb > 32 ? 32 : wb;
      const int t_wb = (nw + wb - 1) / wb;
      const int t_32 = t_wb + cnt[2], t_16 = t_32 + (cnt[3] + 1) / 2, t_8 = t_16 + (cnt[4] + 3) / 4,
                t_4 = t_8 + (cnt[5] + 7) / 8;
      for (;;) {
        int task = 0;
        if (lane == 0) task = atomicAdd(&cnt[7], 1);
        task = __shfl_sync(FULL, task, 0);
        if (task >= t_4) break;
        if (task < t_wb) {
          sc.warp_batch(list, n_half + task * wb, first_of[2], wb, keys0 + wid * PCAP, vals0 + wid * PCAP,
                        occ0 + wid * PCAP, &occ_n[wid], t);
        } else {
          const int q = task < t_32 ? 2 : task < t_16 ? 3 : task < t_8 ? 4 : 5;
          const int t0 = q == 2 ? t_wb : q == 3 ? t_32 : q == 4 ? t_16 : t_8;
          const int f = q == 2 ? first_of[2] : q == 3 ? first_of[3] : q == 4 ? first_of[4] : first_of[5];
          const int e = q == 2 ? first_of[3] : q == 3 ? first_of[4] : q == 4 ? first_of[5] : first_of[6];
          sc.tile(list, f + ((task - t0) << (q - 2)), e, 7 - q, stage, t);
        }
      }
      ++step;
    }
    hubs_here = __syncthreads_or(hubs_here);
    const unsigned changed = account(t, 0);
    const int nm = n_mv;
    unsigned total, hubs, none;
    if (!grid_meet(L.bar + 3 * (int64_t)round, changed, hubs_here, total, hubs, L.polls, s.status)) return;
    if (hubs) {  // the same in every CTA: read the hubs' tables
      const ResidentHubs& r = L.rh;
      if (tid < 5) sums[tid] = sums_hi[tid] = 0;
      __syncthreads();
      Tally th;
      const int n_slices = r.slice[r.nh];
      for (int q = (int)b; q < n_slices; q += (int)G) {
        const int h = __ldg(r.slice_hub + q);
        const int32_t v = __ldg(r.v + h);
        if (!flagged(frontier ? cur_map : nullptr, v) || (s.gfrozen && s.gfrozen[s.gid[v]])) continue;  // uniform
        const int32_t cur = s.C[v];
        const int64_t dv = LOUV ? __ldg(s.degw + v) : 0;
        const int64_t volv = LOUV ? vol_of(s, v) : 0;
        const int first_slice = __ldg(r.slice + h), slices = __ldg(r.slice + h + 1) - first_slice;
        const int64_t base = __ldg(r.tab + h), cap = __ldg(r.tab + h + 1) - base;
        const int64_t s0 = (int64_t)(q - first_slice) * RH_SLICE, s1 = s0 + RH_SLICE < cap ? s0 + RH_SLICE : cap;
        typename S::K bk = no_key<typename S::K>();
        int32_t bc = NOCAND;
        for (int64_t e0 = s0 + tid; e0 < s1; e0 += 4 * PNT) {
          int32_t c[4];
          int64_t k[4], sg[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int64_t e = e0 + (int64_t)j * PNT;
            c[j] = -1;
            k[j] = 0;
            if (e >= s1) continue;
            if constexpr (sizeof(V) == 4) {
              const unsigned long long x = __ldcg(r.slot + base + e);
              if (x != SLOT_EMPTY) {
                c[j] = (int32_t)(x >> 32);
                k[j] = (int64_t)(uint32_t)x;
                r.slot[base + e] = SLOT_EMPTY;
              }
            } else {
              c[j] = __ldcg(r.key + base + e);
              if (c[j] != EMPTY) {
                k[j] = (int64_t)__ldcg(r.slot + base + e);
                r.key[base + e] = EMPTY;
                r.slot[base + e] = 0;
              }
            }
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) sg[j] = LOUV && c[j] >= 0 ? sig_of<NK>(s, c[j]) : 0;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (c[j] < 0) continue;
            ++th.cand;
            if (c[j] == cur) {
              r.cur[h] = k[j];
              r.has[h] = 1;
              if (LOUV) continue;
            }
            const typename S::K key = cand_key_sg<LOUV, NK>(sg[j], k[j], dv, volv);
            if (better(key, c[j], bk, bc)) {
              bk = key;
              bc = c[j];
            }
          }
        }
        reduce_best(bk, bc, 32);
        if (lane == 0) {
          red_k[wid] = bk;
          red_c[wid] = bc;
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) {
          for (int w = 1; w < PNW; ++w)
            if (better(red_k[w], red_c[w], bk, bc)) {
              bk = red_k[w];
              bc = red_c[w];
            }
          const i128 kk = (i128)bk;
          r.part[3 * (int64_t)q] = (int64_t)(kk >> 64);
          r.part[3 * (int64_t)q + 1] = (int64_t)(uint64_t)kk;
          r.part[3 * (int64_t)q + 2] = bc;
          __threadfence();
          s_last = atomicAdd(&r.done[h], 1) == slices - 1;
        }
        __syncthreads();
        if (s_last && wid == 0) {  // the hub's last slice: decide
          __threadfence();
          const volatile int64_t* part = r.part;
          typename S::K fk = no_key<typename S::K>();
          int32_t fc = NOCAND;
          for (int p = first_slice + lane; p < first_slice + slices; p += 32) {
            const i128 pk = (i128)(((unsigned __int128)(uint64_t)part[3 * (int64_t)p] << 64) |
                                   (uint64_t)part[3 * (int64_t)p + 1]);
            const int32_t pc = (int32_t)part[3 * (int64_t)p + 2];
            if (better((typename S::K)pk, pc, fk, fc)) {
              fk = (typename S::K)pk;
              fc = pc;
            }
          }
          reduce_best(fk, fc, 32);
          if (lane == 0) {
            const bool hc = *((volatile int32_t*)&r.has[h]) != 0;
            const int64_t kc = hc ? *((volatile int64_t*)&r.cur[h]) : 0;
            const int32_t target = decide<LOUV, NK>(s, v, cur, fk, fc, hc, kc, volv);
            const uint32_t d = (uint32_t)(__ldg(s.off + v + 1) - __ldg(s.off + v));
            ++th.act;
            th.arcs += d;
            if (target != cur) {
              if (frontier) set_flag(nxt_map, v);
              if (L.per_graph) L.last_change[s.gid[v]] = round + 1;
              if (commit_coin(s.seed, s.level, round, local_id(s, v))) {
                r.moved[h] = round + 1;
                r.to[h] = target;
                r.from[h] = cur;
                atomicAdd(&hub_moves, 1);
                th.marcs += d;
              } else {
                ++th.def;
              }
            }
            r.done[h] = 0;
            r.has[h] = 0;
          }
        }
        __syncthreads();  // red_k, s_last
      }
      const unsigned more = account(th, 1);
      unsigned hub_total;
      if (!grid_meet(L.bar + 3 * (int64_t)round + 1, more, 0, hub_total, none, L.polls, s.status)) return;
      total += hub_total;
      // the neighbours of the moved hubs
      if (frontier) {
        const int n_items = r.item[r.nh];
        for (int it = (int)b; it < n_items; it += (int)G) {
          const int h = __ldg(r.item_hub + it);
          if (__ldcg(r.moved + h) != round + 1) continue;
          const int32_t v = __ldg(r.v + h);
          const int64_t beg = __ldg(s.off + v) + (int64_t)(it - __ldg(r.item + h)) * RH_CHUNK;
          const int64_t row_end = __ldg(s.off + v + 1), end = beg + RH_CHUNK < row_end ? beg + RH_CHUNK : row_end;
          for (int64_t e = beg + tid; e < end; e += PNT) set_flag(nxt_map, __ldg(s.cols + e));
        }
      }
      // and their moves, dealt out over the warps of the grid
      for (int64_t h0 = (b * PNW + wid) * 32; h0 < r.nh; h0 += G * PNW * 32) {
        const int64_t h = h0 + lane;
        const bool ok = h < r.nh && __ldcg(r.moved + h) == round + 1;
        const int32_t v = ok ? r.v[h] : 0, to = ok ? __ldcg(r.to + h) : -1, from = ok ? __ldcg(r.from + h) : -1;
        apply_moves<LOUV, NK>(s, L, ok, v, to, from, stage);
      }
    }
    // the moves, and the flags that were read
    for (int base = wid * 32; base < nm; base += PNT) {
      const int i = base + lane;
      const bool ok = i < nm;
      apply_moves<LOUV, NK>(s, L, ok, ok ? mv[i] : 0, ok ? mv[mv_stride + i] : -1, ok ? mv[2 * mv_stride + i] : -1, stage);
    }
    if (frontier)
      for (int64_t w = b * PNT + tid; w < L.nwords; w += G * PNT) cur_map[w] = 0;
    ++round;
    if (LOUV ? total == 0 : (int64_t)total <= L.threshold) break;
    if (round < L.max_iter && !grid_meet(L.bar + 3 * (int64_t)round - 1, 0, 0, total, none, L.polls, s.status)) return;
  }
  if (b == 0 && tid == 0) L.head[0] = (unsigned long long)round;
}

// The state a run starts from: labels v, Sigma_tot = deg_w and sizes 1 (singletons) or Sigma_tot's copy of a given
// start; every vertex flagged; the barrier words, header and trace zero.
__global__ void __launch_bounds__(PNT) k_rounds_init(LoopCtx L, int32_t* C, int64_t* sigma, int32_t* csize,
                                                     const int64_t* __restrict__ degw, int louv, int singletons,
                                                     int64_t zero_words) {
  const int64_t stride = (int64_t)gridDim.x * PNT, tid = (int64_t)blockIdx.x * PNT + threadIdx.x;
  for (int64_t v = tid; v < L.n; v += stride) {
    int64_t sg = 0;
    if (singletons) {
      C[v] = (int32_t)v;
      if (louv) {
        sg = degw[v];
        if (!L.sigma32) sigma[v] = sg;
        csize[v] = 1;
      }
    } else if (louv) {
      sg = sigma[v];
    }
    if (louv && L.sigma32) L.sigma32[v] = (uint32_t)sg;
  }
  for (int64_t w = tid; w < L.nwords; w += stride) {
    L.flag0[w] = FULL;
    L.flag1[w] = 0;
  }
  for (int64_t i = tid; i < zero_words; i += stride) L.bar[i] = 0;  // the header and the trace follow the barrier words
  if (L.per_graph)
    for (int64_t i = tid; i < L.per_graph; i += stride) L.last_change[i] = 0;
  for (int64_t i = tid; i < L.rh.nh; i += stride) L.rh.moved[i] = 0;
}

int loop_sms() {
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, current_device());
  return sms;
}

template <bool LOUV, class W, class V, bool NK>
int launch_loop(cd_graph* g, const ScanCtx& s, LoopCtx L) {
  static PerDevice resident;  // CTAs at once
  auto kern = k_rounds<LOUV, W, V, NK>;
  constexpr size_t sm = loop_smem<V>();
  int r = resident.get();
  if (r == 0) {
    CD_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    int per = 0;
    CD_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, PNT, sm));
    r = std::max(1, per) * loop_sms();
    resident.set(r);
  }
  const int64_t useful = std::max(g->nnz / ARCS_PER_CTA, L.n / CH_VERTS);
  const int64_t fit = std::max(1, r / std::max(1, g->workers));
  const int64_t grid = g->loop_ctas ? g->loop_ctas : std::max<int64_t>(1, std::min(std::min(fit, L.n), useful));
  // the largest units that still give every CTA four
  L.lgu = 5;
  while (L.lgu > 0 && (L.n >> L.lgu) < 4 * grid) --L.lgu;
  L.nunits = (L.n + ((int64_t)1 << L.lgu) - 1) >> L.lgu;
  void* args[] = {(void*)&s, (void*)&L};
  const cudaError_t e =
      cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)grid), dim3(PNT), args, sm, g->stream);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
    cudaGetLastError();
    return LOOP_REFUSED;
  }
  CD_CHECK(e);
  note_launch();
  return CD_OK;
}

template <bool LOUV, bool NK>
int dispatch_loop(cd_graph* g, const ScanCtx& s, const LoopCtx& L) {
  const bool v32 = g->max_degw < ((int64_t)1 << 32);
  if (g->wkind == W_UNIT)
    return v32 ? launch_loop<LOUV, WUnit, uint32_t, NK>(g, s, L) : launch_loop<LOUV, WUnit, unsigned long long, NK>(g, s, L);
  if (g->wkind == W_I32)
    return v32 ? launch_loop<LOUV, WI32, uint32_t, NK>(g, s, L) : launch_loop<LOUV, WI32, unsigned long long, NK>(g, s, L);
  return v32 ? launch_loop<LOUV, WI64, uint32_t, NK>(g, s, L) : launch_loop<LOUV, WI64, unsigned long long, NK>(g, s, L);
}

// The parts of the context the resident kernel uses (its hubs and counters are in LoopCtx).
ScanCtx loop_ctx(cd_graph* g, const RunOpts& o, bool louv, bool nk) {
  ScanCtx s{};
  s.off = g->off;
  s.cols = g->cols;
  s.w = g->w;
  s.degw = g->degw;
  s.vol = g->vol;
  s.C = g->C;
  s.C_w = g->C;
  s.sigma = g->sigma;
  s.sigma_w = louv ? g->sigma : nullptr;
  s.sigma32 = nk ? g->sigma32 : nullptr;
  s.csize = g->csize;
  s.csize_w = g->csize;
  s.mark = o.use_frontier ? 1 : 0;
  s.mv_v = g->mv_v;
  s.status = g->status;
  s.seed = o.sched_seed;
  s.level = o.level;
  s.tie_keep = o.tie_keep_current;
  s.singleton_rule = o.singleton_rule;
  s.gid = o.batched ? g->gid : nullptr;
  s.gbase = o.batched ? g->gbase : nullptr;
  s.gvol = o.batched ? g->gvol : nullptr;
  s.gfrozen = o.batched ? g->gfrozen : nullptr;
  return s;
}

}  // namespace

bool resident_rounds_apply(const cd_graph* g, const RunOpts& o, bool louv, bool per_graph_stop) {
  return o.device_loop && !o.device_loop_all && !g->timing && !o.async_mode && o.max_iter > 0 && g->n > 0 &&
         g->n_isolated <= std::max(g->n - g->n_isolated, MAX_ISOLATED) &&
         (g->workers <= 1 || g->nnz <= SHARED_LOOP_ARCS) &&
         (g->nhubs == 0 || (g->nhubs <= RH_MAX_HUBS && g->nnz <= RH_MAX_ARCS)) &&
         g->nnz <= resident_arcs(g, o, louv) &&
         g->bin_start[B_BLK4 + 1] == g->bin_start[B_BLK4] && (!per_graph_stop || (o.threshold == 0 && o.use_frontier));
}

// All rounds of a run or level (see the head of this file). The labels (and,
// for a given start, sigma and csize) are set here or by the caller.
int resident_rounds(cd_graph* g, const RunOpts& o, bool louv, bool singletons, int64_t* moves_out, int32_t* rounds_out,
                    std::vector<int32_t>* graph_rounds) {
  const cudaStream_t st = g->stream;
  const bool per_graph = graph_rounds != nullptr;
  const bool nk = louv && g->vol < ((int64_t)1 << 31);
  int rc;
  LoopCtx L{};
  L.n = g->n;
  L.nwords = (g->n + 31) / 32;
  L.n32 = L.nwords * 32;
  L.flag0 = g->flag[0];
  L.flag1 = g->flag[1];
  L.max_iter = o.max_iter;
  L.polls = g->loop_polls ? g->loop_polls : WAIT_LIMIT;
  L.first_rows = singletons && g->cols_distinct;
  L.t_warp = g->t_warp;
  L.t_hub = g->t_hub;
  if (g->nhubs > 0) {
    if ((rc = ensure_resident_hubs(g))) return rc;
    L.rh = *g->rh;
  }
  L.threshold = o.threshold;
  L.per_graph = per_graph ? (int32_t)g->nb : 0;
  L.sigma32 = nk ? g->sigma32 : nullptr;
  const int64_t words = 3 * (int64_t)o.max_iter + HEAD + (int64_t)TRACE_COLS * o.max_iter;
  unsigned long long* work = nullptr;
  Arena scratch;
  scratch.add(&work, words);
  if (per_graph) scratch.add(&L.last_change, g->nb);
  if ((rc = scratch.make(st))) return rc;
  L.bar = work;
  L.head = work + 3 * (int64_t)o.max_iter;
  std::vector<unsigned long long> h;
  std::vector<int32_t> hl;
  int32_t status = 0;
  auto run = [&]() -> int {
    if (per_graph) CD_CHECK(cudaMemsetAsync(g->gfrozen, 0, g->nb, st));
    const unsigned gi = (unsigned)std::max<int64_t>(1, std::min<int64_t>((g->n + PNT - 1) / PNT, 152 * 8));
    CD_LAUNCH(k_rounds_init<<<gi, PNT, 0, st>>>(L, g->C, g->sigma, g->csize, g->degw, louv ? 1 : 0, singletons ? 1 : 0,
                                                words));
    const ScanCtx s = loop_ctx(g, o, louv, nk);
    int r = !louv ? dispatch_loop<false, false>(g, s, L) : nk ? dispatch_loop<true, true>(g, s, L)
                                                              : dispatch_loop<true, false>(g, s, L);
    if (r) return r;
    CD_CHECK(cudaGetLastError());
    // the header and the rounds of a usual run in one copy
    const int64_t some = std::min<int64_t>(o.max_iter, 128);
    h.resize(HEAD + TRACE_COLS * some);
    CD_CHECK(cudaMemcpyAsync(h.data(), L.head, h.size() * 8, cudaMemcpyDeviceToHost, st));
    CD_CHECK(cudaMemcpyAsync(&status, g->status, 4, cudaMemcpyDeviceToHost, st));
    if (per_graph) {
      hl.resize(g->nb);
      CD_CHECK(cudaMemcpyAsync(hl.data(), L.last_change, g->nb * 4, cudaMemcpyDeviceToHost, st));
    }
    CD_CHECK(cudaStreamSynchronize(st));
    if (!status && (int64_t)h[0] > some) {
      const int64_t all = (int64_t)h[0];
      h.resize(HEAD + TRACE_COLS * all);
      CD_CHECK(cudaMemcpyAsync(h.data(), L.head, h.size() * 8, cudaMemcpyDeviceToHost, st));
      CD_CHECK(cudaStreamSynchronize(st));
    }
    return status;
  };
  rc = run();
  scratch.free(st);
  if (rc == LOOP_REFUSED) return rc;
  if (rc) {  // the hubs' tables may hold entries of the round that was cut short
    drop_resident_hubs(g);
    if (status) cudaMemsetAsync(g->status, 0, sizeof(int32_t), st);
    return rc;
  }
  const int32_t rounds = (int32_t)h[0];
  int64_t moves = 0;
  for (int32_t r = 0; r < rounds; ++r) {
    const unsigned long long* t = h.data() + HEAD + (int64_t)TRACE_COLS * r;
    cd_round_trace tr;
    tr.level = o.level;
    tr.round = r;
    tr.active = (int64_t)t[0] + ((r == 0 || !o.use_frontier) ? g->n_isolated : 0);
    tr.arcs = (int64_t)t[1];
    tr.moved = (int64_t)t[2];
    tr.deferred = (int64_t)t[3];
    tr.cands = (int64_t)t[4];
    tr.moved_arcs = (int64_t)t[5];
    tr.scan_ms = tr.round_ms = 0.f;
    g->trace.push_back(tr);
    moves += tr.moved;
  }
  if (per_graph)  // a graph stops after its first round without a change
    for (int64_t b = 0; b < g->nb; ++b) (*graph_rounds)[b] = std::min(o.max_iter, hl[b] + 1);
  if (moves_out) *moves_out = moves;
  if (rounds_out) *rounds_out = rounds;
  return CD_OK;
}

}  // namespace cd

// For tests: the polls after which a barrier of g's resident loops gives up, and
// the CTAs they are launched with (0: as always).
extern "C" int cd_test_resident_loop(cd_graph* g, int64_t polls, int64_t ctas) {
  if (!g || polls < 0 || ctas < 0) return CD_EINVAL;
  g->loop_polls = polls;
  g->loop_ctas = ctas;
  return CD_OK;
}
