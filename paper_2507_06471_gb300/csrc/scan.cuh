// Device code shared by the scan kernels (scan.cu) and the resident round
// loop (rounds.cu): a round's context, the deferral coin, candidate keys and
// decisions, hub histograms, and the shared-memory label tables.
#pragma once
#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace cd {
namespace {

constexpr int NT = 256;  // threads of the tile and hub-evaluate kernels
constexpr int NW = NT / 32;
constexpr int WARP_CAP_SLOTS = 2 * WARP_MAX;   // table slots per warp-bin vertex
constexpr int BLK1_CAP_SLOTS = 2 * BLK1_MAX;   // per 128-thread group
constexpr int BLK4_CAP_SLOTS = 2 * BLK4_MAX;   // per 512-thread CTA

// ------------------------------------------------------------------ coin

// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014): draw number ctr of the
// stream with state `seed`; the move commits iff bit 63 is set.
__device__ __forceinline__ bool commit_coin(uint64_t seed, int level, int round, int32_t v) {
  uint64_t ctr = ((uint64_t)(uint32_t)level << 48) | ((uint64_t)(uint32_t)round << 32) | (uint32_t)v;
  uint64_t z = seed + (ctr + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (z >> 63) != 0;
}

// ------------------------------------------------------------------ keys

template <bool LOUV, bool NK> struct KeyOf { typedef int64_t T; };
template <> struct KeyOf<true, false> { typedef i128 T; };

__device__ __forceinline__ int64_t shfl_xor_key(int64_t x, int o) {
  return __shfl_xor_sync(FULL, (long long)x, o);
}
__device__ __forceinline__ i128 shfl_xor_key(i128 x, int o) {
  unsigned long long lo = (unsigned long long)x, hi = (unsigned long long)(x >> 64);
  lo = __shfl_xor_sync(FULL, lo, o);
  hi = __shfl_xor_sync(FULL, hi, o);
  return (i128)(((unsigned __int128)hi << 64) | lo);
}

// The key of "no candidate" (with the id NOCAND): below every candidate's key,
// so that comparing needs no case of its own.
template <class K> __device__ __forceinline__ K no_key();
template <> __device__ __forceinline__ int64_t no_key<int64_t>() { return INT64_MIN; }
template <> __device__ __forceinline__ i128 no_key<i128>() { return (i128)INT64_MIN << 64; }

// Is candidate (k1, c1) preferred over (k0, c0)? Larger key, then smaller id.
template <class K>
__device__ __forceinline__ bool better(K k1, int32_t c1, K k0, int32_t c0) {
  return k1 > k0 || (k1 == k0 && c1 < c0);
}

// The best of each group of `width` consecutive lanes, in every lane of it.
template <class K>
__device__ __forceinline__ void reduce_best(K& k, int32_t& c, int width) {
  if constexpr (sizeof(K) == 8) {
    if (width == 32) {  // whole warps: three hardware reductions instead of five exchanges of three words
      const int32_t hi = (int32_t)(k >> 32);
      const int32_t mh = __reduce_max_sync(FULL, hi);
      const uint32_t ml = __reduce_max_sync(FULL, hi == mh ? (uint32_t)k : 0u);
      const K best = (K)(((uint64_t)(uint32_t)mh << 32) | ml);
      c = __reduce_min_sync(FULL, k == best ? c : NOCAND);
      k = best;
      return;
    }
  }
  for (int o = width / 2; o > 0; o >>= 1) {
    K ok = shfl_xor_key(k, o);
    int32_t oc = __shfl_xor_sync(FULL, c, o);
    if (better(ok, oc, k, c)) {
      k = ok;
      c = oc;
    }
  }
}

struct ScanCtx {
  const int64_t* off;
  const int32_t* cols;
  const void* w;
  const int64_t* degw;
  int64_t vol;
  const int32_t* C;
  const int64_t* sigma;
  const uint32_t* sigma32;  // 32-bit copy of sigma for the gathers (vol(V) < 2^31, synchronous), or null
  const int32_t* csize;
  const uint32_t* flag_cur;  // bitmaps of n bits: examined this round / next round
  uint32_t* flag_nxt;
  int all_active;
  int mark;  // maintain the next-round flags (frontier on)
  int32_t* mv_v;
  int32_t* mv_c;
  unsigned long long* ctr;
  int32_t* status;
  uint64_t seed;
  int level, round, tie_keep, singleton_rule;
  int32_t* mv_a;
  // hubs
  const int32_t* hub_list;
  const uint32_t* hub_pref;
  const uint32_t* hub_bits;
  const int64_t* hub_tab;
  int64_t* hub_cc;                   // per hub: slots in use, [0, hub_cc) of its allocation (what lies past them is stale)
  int32_t* hub_live;                 // per hub: live entries counted by this round's evaluate items
  unsigned long long* hub_slot;
  int hub_wide;
  const int32_t* hub_item_hub;
  const int64_t* hub_item_arc;
  const int32_t* hub_ev_hub;
  const int64_t* hub_ev_slot;
  const int64_t* hub_ev_first;
  int64_t* hub_part;
  int64_t* hub_cur;
  int32_t* hub_hascur;
  int32_t* hub_done;
  int32_t* hub_mv;
  int32_t* hub_rb;                   // per hub: 1 = rebuild from its row, 2 = compact, before its next evaluation
  int32_t* hub_flist_w;              // hubs flagged this round (read back at the start of the next)
  unsigned long long* hub_fcnt_w;
  const int32_t* hub_flist_r;        // hubs flagged in the previous round
  const unsigned long long* hub_fcnt_r;
  int32_t* hub_used;                 // per hub: slots claimed since its last build
  int32_t* hub_nl;                   // per hub: live entries at its last evaluation in this run, -1: none yet
  int64_t* hub_nc;                   // per hub: slots its rebuild of this round lays out
  int32_t* hub_pl;                   // nhubs: hubs a CTA prepares this round; then nhubs: rebuilds that overflowed
  const int64_t* hub_item_first;     // nhubs+1: first build/mark item of each hub
  int32_t* hub_blist;                // build items of the hubs being rebuilt this round
  int32_t* hub_mlist;                // mark items of the hubs that moved this round
  unsigned long long* hub_lcnt;      // [0] build items, [1] mark items
  int32_t* hub_cl;                   // 5 x nhubs: hubs rebuilt per build class (one CTA small/large, clusters of 2, 4, 8)
  unsigned long long* hub_ccnt;      // 5: their counts; [5], [6]: those of hub_pl's two lists
  const int32_t* ev_list;            // evaluate items (of large hubs) to run this round
  const unsigned long long* ev_cnt;  // their number
  const int32_t* small_list;         // small hubs (one warp each) to evaluate this round
  const unsigned long long* small_cnt;
  const int32_t* hub_act;            // hubs examined this round (null: every hub)
  const unsigned long long* hub_act_cnt;
  int hub_upd;  // 0: neighbour moves do not update hub histograms (every hub is rebuilt next round)
  int64_t n_items, nhubs, n_ev_items;
  unsigned long long* hub_log;  // hub-histogram updates of this round, applied after the scans (null: at once)
  unsigned long long* hub_log_cnt;
  int64_t hub_log_cap;
  // asynchronous mode: a committed move is applied at once through these
  int async_mode;
  int32_t* C_w;
  int64_t* sigma_w;  // null for LPA
  int32_t* csize_w;
  // device-side round loop: the round number and the hub-update switch are
  // read from device memory (null: the host-side values above apply)
  const int32_t* round_p;
  const int32_t* hub_upd_p;
  // batched mode (gid == nullptr: one graph)
  const int32_t* gid;
  const int64_t* gbase;
  const int64_t* gvol;
  const uint8_t* gfrozen;
  unsigned long long* gcnt;
};

__device__ __forceinline__ int round_of(const ScanCtx& s) { return s.round_p ? *s.round_p : s.round; }
__device__ __forceinline__ bool hub_upd_of(const ScanCtx& s) {
  return s.hub_upd_p ? *s.hub_upd_p != 0 : s.hub_upd != 0;
}

// Flag vertex u for the next round (a bit in an L2-resident bitmap).
__device__ __forceinline__ void flag_next(const ScanCtx& s, int32_t u) {
  atomicOr(&s.flag_nxt[u >> 5], 1u << (u & 31));
}

// vol(V) of the graph v belongs to, and v's id inside that graph (the coin
// uses graph-local ids so that a batched run draws what a solo run draws).
__device__ __forceinline__ int64_t vol_of(const ScanCtx& s, int32_t v) {
  return s.gid ? s.gvol[s.gid[v]] : s.vol;
}
__device__ __forceinline__ int32_t local_id(const ScanCtx& s, int32_t v) {
  return s.gid ? v - (int32_t)s.gbase[s.gid[v]] : v;
}
// A vertex that wants to change label (moved or deferred) counts toward its
// graph's stop test.
__device__ __forceinline__ void count_change(const ScanCtx& s, int32_t v) {
  if (s.gcnt) atomicAdd(&s.gcnt[s.gid[v]], 1ull);
}

// Sigma_tot[c] for a candidate: from the 32-bit copy when there is one
// (half the bytes of the random gather).
template <bool NK>
__device__ __forceinline__ int64_t sig_of(const ScanCtx& s, int32_t c) {
  if constexpr (NK) {
    if (s.sigma32) return (int64_t)s.sigma32[c];
  }
  return s.sigma[c];
}

// vol(V) k - deg_w(v) Sigma_tot[c], or k for LPA. When vol(V) < 2^31 all four
// factors fit in 32 bits, so each product is one 32 x 32 -> 64 multiplication.
template <bool LOUV, bool NK>
__device__ __forceinline__ typename KeyOf<LOUV, NK>::T cand_key_sg(int64_t sig, int64_t k, int64_t d, int64_t vol) {
  if constexpr (LOUV && NK)
    return (int64_t)((uint64_t)(uint32_t)vol * (uint32_t)k) - (int64_t)((uint64_t)(uint32_t)d * (uint32_t)sig);
  else if constexpr (LOUV)
    return (i128)vol * k - (i128)d * sig;
  else
    return k;
}

template <bool LOUV, bool NK>
__device__ __forceinline__ typename KeyOf<LOUV, NK>::T cand_key(const ScanCtx& s, int32_t c, int64_t k,
                                                            int64_t d, int64_t vol) {
  if constexpr (LOUV)
    return cand_key_sg<LOUV, NK>(sig_of<NK>(s, c), k, d, vol);
  else
    return k;
}

// Final decision of vertex v from the best candidate.
template <bool LOUV, bool NK>
__device__ __forceinline__ int32_t decide(const ScanCtx& s, int32_t v, int32_t cur,
                                          typename KeyOf<LOUV, NK>::T bk, int32_t bc, bool has_cur,
                                          int64_t kcur, int64_t vol) {
  if (bc == NOCAND) return cur;
  if constexpr (!LOUV) {
    if (s.tie_keep && has_cur && kcur == bk) return cur;
    return bc;
  } else {
    int64_t d = s.degw[v];
    bool gain;
    if constexpr (NK) {
      // vol(V) < 2^31: vol k, d Sigma < 2^62 and Sigma[cur] >= d, so the sum stays inside (-2^63, 2^63)
      gain = bk - (int64_t)((uint64_t)(uint32_t)vol * (uint32_t)kcur) +
                 (int64_t)((uint64_t)(uint32_t)d * (uint32_t)(sig_of<NK>(s, cur) - d)) > 0;
    } else {
      gain = (i128)bk - (i128)vol * kcur + (i128)d * (s.sigma[cur] - d) > 0;
    }
    if (!gain) return cur;  // only strictly positive gains
    if (s.singleton_rule && bc > cur) {
      const int32_t na = s.csize[cur], nb = s.csize[bc];  // two loads in flight, not one after the other
      if (na == 1 && nb == 1) return cur;
    }
    return bc;
  }
}

// Asynchronous mode: v's move from `cur` to `target` takes effect now.
__device__ __forceinline__ void apply_now(const ScanCtx& s, int32_t v, int32_t cur, int32_t target) {
  s.C_w[v] = target;
  if (s.sigma_w) {
    const int64_t d = s.degw[v];
    atomicAdd((unsigned long long*)&s.sigma_w[cur], (unsigned long long)(-d));
    atomicAdd((unsigned long long*)&s.sigma_w[target], (unsigned long long)d);
    atomicSub(&s.csize_w[cur], 1);
    atomicAdd(&s.csize_w[target], 1);
  }
}

// One thread acts on a decision: append a committed move or count a deferral.
// Returns 1 if the move was deferred.
__device__ __forceinline__ int act_single(const ScanCtx& s, int32_t v, int32_t cur, int32_t target) {
  if (target == cur) return 0;
  if (s.mark) flag_next(s, v);
  count_change(s, v);
  if (commit_coin(s.seed, s.level, round_of(s), local_id(s, v))) {
    unsigned long long pos = atomicAdd(&s.ctr[C_MOVES], 1ull);
    s.mv_v[pos] = v;
    s.mv_c[pos] = target;
    s.mv_a[pos] = cur;
    if (s.async_mode) apply_now(s, v, cur, target);
    return 0;
  }
  return 1;
}

__device__ __forceinline__ void flush_counters(const ScanCtx& s, int bin, int64_t act, int64_t arcs,
                                               int64_t cands, int64_t def, int64_t marcs) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    act += __shfl_xor_sync(FULL, act, o);
    arcs += __shfl_xor_sync(FULL, arcs, o);
    cands += __shfl_xor_sync(FULL, cands, o);
    def += __shfl_xor_sync(FULL, def, o);
    marcs += __shfl_xor_sync(FULL, marcs, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (act) atomicAdd(&s.ctr[C_BIN0 + 3 * bin], (unsigned long long)act);
    if (arcs) atomicAdd(&s.ctr[C_BIN0 + 3 * bin + 1], (unsigned long long)arcs);
    if (cands) atomicAdd(&s.ctr[C_BIN0 + 3 * bin + 2], (unsigned long long)cands);
    if (def) atomicAdd(&s.ctr[C_DEFERRED], (unsigned long long)def);
    if (marcs) atomicAdd(&s.ctr[C_MARCS], (unsigned long long)marcs);
  }
}

__device__ __forceinline__ bool is_active(const ScanCtx& s, int32_t v) {
  if (s.gfrozen && s.gfrozen[s.gid[v]]) return false;
  return s.all_active || ((s.flag_cur[v >> 5] >> (v & 31)) & 1u);
}

// Group weight of the lanes in `peers` (equal labels; every lane takes part):
// popcount for unit weights, else sums over the warp's staging row. When every
// deg_w < 2^32 (v32) the lanes add into their group's first word, one shared
// atomic each; walking the peers instead takes as many dependent loads as the
// largest group has lanes, which is the whole row once labels have settled.
template <class W>
__device__ __forceinline__ int64_t group_sum(unsigned peers, int64_t wt, int64_t* stage, bool v32) {
  if constexpr (W::unit) {
    return (int64_t)__popc(peers);
  } else {
    const int lane = threadIdx.x & 31;
    if (v32) {  // uniform
      uint32_t* row = (uint32_t*)stage;
      row[lane] = 0;
      __syncwarp();
      atomicAdd(&row[__ffs(peers) - 1], (uint32_t)wt);
      __syncwarp();
      const uint32_t sum = row[__ffs(peers) - 1];
      __syncwarp();
      return (int64_t)sum;
    }
    stage[lane] = wt;
    __syncwarp();
    int64_t s = 0;
    unsigned m = peers;
    while (m) {
      s += stage[__ffs(m) - 1];
      m &= m - 1;
    }
    __syncwarp();
    return s;
  }
}

// ------------------------------------------------------------------ hub histograms

constexpr unsigned long long SLOT_EMPTY = ~0ull;

// Flag hub h for the start of the next round: HUB_REBUILD (an update was
// lost; it is rebuilt from its row and not updated until then) or
// HUB_COMPACT (it is consistent but too full; its live entries are rehashed).
// A hub is queued once, when it is first flagged.
constexpr int32_t HUB_REBUILD = 1, HUB_COMPACT = 2;

__device__ __forceinline__ void hub_flag(const ScanCtx& s, int32_t h, int32_t how) {
  const int32_t old = how == HUB_REBUILD ? atomicExch(&s.hub_rb[h], HUB_REBUILD) : atomicCAS(&s.hub_rb[h], 0, how);
  if (old == 0) s.hub_flist_w[atomicAdd(s.hub_fcnt_w, 1ull)] = h;
}

// Slot of `label` in a table of `cap` slots (hub histograms, here and in the
// shared-memory layouts built for them).
__device__ __forceinline__ int64_t hub_home(int32_t label, int64_t cap) {
  return (int64_t)(((uint64_t)((uint32_t)label * 2654435761u) * (uint64_t)cap) >> 32);
}

// An update gives up after HUB_PROBE_MAX probes (the hub is rebuilt), and a
// hub whose claimed slots pass 7/8 of its capacity is compacted: labels that
// leave keep their slot (count 0), so a table fills up over the rounds and
// linear-probe chains would otherwise grow without bound.
constexpr int HUB_PROBE_MAX = 64;
constexpr int64_t HUB_SKIP_DIV = 16;     // Louvain (measured: 4 and 64 slower)
constexpr int64_t HUB_SKIP_DIV_LPA = 4;  // LPA (measured: 16 slower by 12%)

// k_{h,label} += w in hub h's histogram (w may be negative: a neighbour left
// `label`; the count then stays >= 0). A packed slot is updated with one
// 64-bit atomic: the count lives in the low word and never carries or borrows
// into the label. A build (BUILD) probes the whole table, which at most two
// thirds of its slots can fill; an update gives up after HUB_PROBE_MAX probes
// or when a label to decrement is missing, and then flags the hub.
template <bool BUILD>
__device__ __forceinline__ void hub_hist_add(const ScanCtx& s, int32_t h, int32_t label, int64_t w) {
  if (!BUILD && s.hub_rb[h] == HUB_REBUILD) return;
  const int64_t base = s.hub_tab[h];
  const int64_t cap = s.hub_cc[h];
  const int64_t lim = BUILD ? cap : (cap < HUB_PROBE_MAX ? cap : HUB_PROBE_MAX);
  int64_t slot = hub_home(label, cap);
  bool claimed = false;
  if (!s.hub_wide) {
    unsigned long long* words = s.hub_slot + base;
    for (int64_t probe = 0; probe < lim; ++probe) {
      unsigned long long cur = words[slot];
      if (cur == SLOT_EMPTY) {
        if (w <= 0) break;
        cur = atomicCAS(&words[slot], SLOT_EMPTY,
                        ((unsigned long long)(uint32_t)label << 32) | (unsigned long long)(uint32_t)w);
        if (cur == SLOT_EMPTY) {
          claimed = true;
          break;
        }
      }
      if ((int32_t)(cur >> 32) == label) {
        atomicAdd(&words[slot], (unsigned long long)w);
        return;
      }
      slot = slot + 1 == cap ? 0 : slot + 1;
    }
  } else {
    unsigned long long* words = s.hub_slot + 2 * base;  // (label, count) pairs
    for (int64_t probe = 0; probe < lim; ++probe) {
      unsigned long long cur = words[2 * slot];
      if (cur == SLOT_EMPTY) {
        if (w <= 0) break;
        cur = atomicCAS(&words[2 * slot], SLOT_EMPTY, (unsigned long long)(uint32_t)label);
        if (cur == SLOT_EMPTY) {
          claimed = true;
          cur = (uint32_t)label;
        }
      }
      if ((int32_t)(uint32_t)cur == label) {
        atomicAdd(&words[2 * slot + 1], (unsigned long long)w);
        if (!claimed) return;
        break;
      }
      slot = slot + 1 == cap ? 0 : slot + 1;
    }
  }
  if (claimed) {
    const int32_t used = atomicAdd(&s.hub_used[h], 1) + 1;
    if (!BUILD && (int64_t)used * 8 > cap * 7) hub_flag(s, h, HUB_COMPACT);
    return;
  }
  hub_flag(s, h, HUB_REBUILD);
}

// Read slot i of a hub table at `base`: (label or -1 if empty, count).
__device__ __forceinline__ void hub_slot_read(const ScanCtx& s, int64_t base, int64_t i, int32_t& c,
                                              int64_t& k) {
  if (!s.hub_wide) {
    const unsigned long long x = s.hub_slot[base + i];
    c = x == SLOT_EMPTY ? -1 : (int32_t)(x >> 32);
    k = (int64_t)(x & 0xffffffffull);
  } else {
    const unsigned long long x = s.hub_slot[2 * (base + i)];
    c = x == SLOT_EMPTY ? -1 : (int32_t)(uint32_t)x;
    k = (int64_t)s.hub_slot[2 * (base + i) + 1];
  }
}

// A committed move of a neighbour of u (label A -> c over an arc of weight
// w) changes u's histogram if u is a hub. The hub bitmap (n bits) stays in L2.
__device__ __forceinline__ void hub_neighbour_moved(const ScanCtx& s, int32_t u, int32_t A, int32_t c,
                                                    int64_t w) {
  if (!hub_upd_of(s)) return;
  const uint32_t bits = __ldg(&s.hub_bits[u >> 5]);
  if (!((bits >> (u & 31)) & 1u)) return;
  const int32_t h = (int32_t)(__ldg(&s.hub_pref[u >> 5]) + __popc(bits & ((1u << (u & 31)) - 1u)));
  if (s.hub_log) {
    // appended as (h, A) and (c, w) words by the lanes that got here together;
    // applied by k_hub_apply_log with every thread busy
    cg::coalesced_group grp = cg::coalesced_threads();
    unsigned long long pos = 0;
    if (grp.thread_rank() == 0) pos = atomicAdd(s.hub_log_cnt, (unsigned long long)grp.size());
    pos = grp.shfl(pos, 0) + grp.thread_rank();
    if ((int64_t)pos < s.hub_log_cap) {
      s.hub_log[2 * pos] = ((unsigned long long)(uint32_t)h << 32) | (uint32_t)A;
      s.hub_log[2 * pos + 1] = ((unsigned long long)(uint32_t)c << 32) | (unsigned long long)(uint32_t)w;
    } else {
      hub_flag(s, h, HUB_REBUILD);  // log full: rebuild this hub from its row instead
    }
    return;
  }
  hub_hist_add<false>(s, h, A, -w);
  hub_hist_add<false>(s, h, c, w);
}

// ------------------------------------------------------------------ shared-memory tables

// Open addressing with linear probing; capacity 2^lg >= 2 x the arcs inserted,
// so a free slot is always found within `cap` probes. A probe is a plain load;
// only an empty slot is claimed with a compare-and-swap. A newly claimed slot
// is appended to the table's occupied list, so that reading the table costs
// the number of distinct labels rather than its capacity.
template <class V>
__device__ __forceinline__ void smem_insert(int32_t* keys, V* vals, uint16_t* occ, int* occ_n,
                                            unsigned lg, int32_t key, V w, int32_t* status) {
  const unsigned mask = (1u << lg) - 1u;
  unsigned h = ((uint32_t)key * 2654435761u) >> (32 - lg);
  for (unsigned probe = 0; probe <= mask; ++probe) {
    int32_t k = *(volatile int32_t*)&keys[h];
    if (k == EMPTY) {
      k = atomicCAS(&keys[h], EMPTY, key);
      if (k == EMPTY) {
        occ[atomicAdd(occ_n, 1)] = (uint16_t)h;
        k = key;
      }
    }
    if (k == key) {
      atomicAdd(vals + h, w);
      return;
    }
    h = (h + 1) & mask;
  }
  atomicCAS(status, 0, CD_ETIMEOUT);  // table full: impossible with cap >= 2 deg
}

__device__ __forceinline__ unsigned ceil_log2(int64_t x) {
  unsigned lg = 0;
  while (((int64_t)1 << lg) < x) ++lg;
  return lg < 1 ? 1 : lg;
}

// Synchronise the GROUP threads sharing a table: a warp, the whole CTA, or a
// named barrier (ids 1..15) for a sub-CTA group.
template <int GROUP, int NTB>
__device__ __forceinline__ void group_sync(int gid) {
  if constexpr (GROUP == 32)
    __syncwarp();
  else if constexpr (GROUP == NTB)
    __syncthreads();
  else
    asm volatile("bar.sync %0, %1;" ::"r"(gid + 1), "n"(GROUP) : "memory");
}

// Insert the arcs [beg, end) of vertex v into a group's table. Columns are
// read 16 bytes at a time (4 arcs per lane, 4 label gathers in flight), and
// every arc goes into the table by itself: combining the equal labels of a
// warp first (a match, then a walk over the peers) took several times the
// instructions of the shared atomics it saved.
// Column arrays carry COL_PAD spare entries, so a 16-byte load that starts
// before `end` stays inside the allocation.
template <class W, class V, int GROUP>
__device__ __forceinline__ void group_insert(const ScanCtx& s, int32_t v, int64_t beg, int64_t end,
                                             int gl, int32_t* keys, V* vals, uint16_t* occ, int* occ_n,
                                             unsigned lg) {
  const int lane = threadIdx.x & 31;
  const int wig = gl >> 5;
  const int64_t a0 = beg & ~(int64_t)3;
  for (int64_t wb = a0 + (int64_t)wig * 128; wb < end; wb += (int64_t)GROUP * 4) {
    const int64_t base = wb + 4 * lane;
    const int4 c4 = base < end ? __ldg(reinterpret_cast<const int4*>(s.cols + base)) : make_int4(0, 0, 0, 0);
    const int32_t cs[4] = {c4.x, c4.y, c4.z, c4.w};
    int32_t lbl[4];
    V wt[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t e = base + j;
      const bool has = e >= beg && e < end;
      lbl[j] = has && cs[j] != v ? s.C[cs[j]] : -1;
      wt[j] = (has && !W::unit) ? (V)W::get(s.w, e) : (V)1;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (lbl[j] >= 0) smem_insert(keys, vals, occ, occ_n, lg, lbl[j], wt[j], s.status);
  }
}

// Read a group's table through its occupied list: every listed slot is a
// candidate; the slot is cleared for the next vertex.
template <bool LOUV, class V, int GROUP, bool NK>
__device__ __forceinline__ void group_eval(const ScanCtx& s, int32_t cur, int64_t dv, int64_t vol,
                                           int gl, int32_t* keys, V* vals, const uint16_t* occ, int nocc,
                                           typename KeyOf<LOUV, NK>::T& bk, int32_t& bc, bool& hc,
                                           int64_t& kc, int64_t& ncand) {
  constexpr int EB = 2;  // candidates per thread per batch: the Sigma_tot gathers go out together
  for (int j0 = gl; j0 < nocc; j0 += EB * GROUP) {
    int32_t c[EB];
    int64_t k[EB], sg[EB];
#pragma unroll
    for (int q = 0; q < EB; ++q) {
      const int j = j0 + q * GROUP;
      c[q] = -1;
      k[q] = 0;
      if (j < nocc) {
        const int slot = occ[j];
        c[q] = keys[slot];
        k[q] = (int64_t)vals[slot];
        keys[slot] = EMPTY;
        vals[slot] = 0;
      }
    }
#pragma unroll
    for (int q = 0; q < EB; ++q) sg[q] = (LOUV && c[q] >= 0) ? sig_of<NK>(s, c[q]) : 0;
#pragma unroll
    for (int q = 0; q < EB; ++q) {
      if (c[q] < 0) continue;
      ++ncand;
      if (c[q] == cur) {
        hc = true;
        kc = k[q];
        if (LOUV) continue;
      }
      const typename KeyOf<LOUV, NK>::T key = cand_key_sg<LOUV, NK>(sg[q], k[q], dv, vol);
      if (better(key, c[q], bk, bc)) {
        bk = key;
        bc = c[q];
      }
    }
  }
}

// What a scan needs of a vertex before reading its row.
struct VHdr {
  int64_t beg, end, dv, vol;
  int32_t cur;
  bool act;
};

template <bool LOUV>
__device__ __forceinline__ VHdr load_hdr(const ScanCtx& s, int32_t v, bool valid) {
  VHdr h;
  h.act = valid && is_active(s, v);
  h.beg = valid ? s.off[v] : 0;
  h.end = valid ? s.off[v + 1] : 0;
  h.cur = valid ? s.C[v] : 0;
  h.dv = (LOUV && valid) ? s.degw[v] : 0;
  h.vol = (LOUV && valid) ? vol_of(s, v) : 0;
  return h;
}

}  // namespace
}  // namespace cd
