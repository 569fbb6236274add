// Local moving, the parts that its host-driven rounds (local_move.cu) and its
// resident rounds (lm_rounds.cu) share: the decision policy, the application of
// a sub-round's decisions, the moves to empty communities and the round's
// tracking state.  The rules are stated in local_move.cu.
#pragma once
#include <algorithm>
#include <cstdlib>

#include "decide.cuh"
#include "solver.h"
#include "track.cuh"

namespace mslice {

struct TierOff {
  int32_t off[NTIERS];
};

__device__ __forceinline__ int bucket_seg(const LevelDev& g, const uint8_t* tier, uint64_t seed, uint64_t tag,
                                          uint64_t it, uint64_t lvl, uint64_t r, int K, const int32_t* active,
                                          int64_t v) {
  if (active && !active[node_inst(g, (int32_t)v)]) return SEG_FROZEN;  // converged instance: frozen
  return vertex_class(seed, tag, it, lvl, r, local_id(g, (int32_t)v), K) * NTIERS + tier[v];
}

// sum_s Lambda_s k_{v,s} (X_s - self*k_{v,s}) with X_s = table(c, s).
// (od is applied by the caller.)
template <bool DENSE>
__device__ __forceinline__ u128 null_sum(const LevelDev& g, const u128* lam, const SigStore& h, int32_t v, int32_t c,
                                         bool self) {
  int64_t b, e;
  slice_range(g, v, b, e);
  u128 t = 0;
  for (int64_t j = b; j < e; ++j) {
    int32_t s;
    long long k;
    slice_entry(g, v, j, s, k);
    long long x = sst_get<DENSE>(h, c, s);
    if (self) x -= k;
    t += lam[s] * (u128)(ull)k * (u128)(ull)x;
  }
  return t;
}

// The same over the entries t, t + nt, ... of v's list, U at a time: their
// table loads are in flight together before the first is used (a walk of one
// entry at a time waits for two dependent loads each).  The resident kernels take
// four.  The large levels' kernels keep the plain walk: the registers of four cost
// the group kernels a fifth of their speed, and took the dense block kernels from 64
// registers to 74 (tier 3) and to 248 bytes of spills (tier 4): rows of 300 entries
// with lists of 8 decided in 1.97 ms a round instead of 1.78 (N = 50,000).
template <bool DENSE, int U>
__device__ __forceinline__ u128 null_sum_part(const LevelDev& g, const u128* lam, const SigStore& h, int32_t v,
                                              int32_t c, bool self, int t, int nt) {
  int64_t b, e;
  slice_range(g, v, b, e);
  u128 acc = 0;
  for (int64_t j0 = b + t; j0 < e; j0 += (int64_t)U * nt) {
    int32_t s[U];
    long long k[U];
    Slot f[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t j = j0 + (int64_t)u * nt;
      k[u] = 0;
      if (j < e) slice_entry(g, v, j, s[u], k[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k[u] > 0) f[u] = sst_first<DENSE>(h, c, s[u]);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k[u] > 0) {
        long long x = sst_resolve<DENSE>(h, c, s[u], f[u]);
        if (self) x -= k[u];
        acc += lam[s[u]] * (u128)(ull)k[u] * (u128)(ull)x;
      }
  }
  return acc;
}

// L0: a level-0 policy.  Its nodes hold one (snapshot, strength)
// entry each, so the code that walks lists is left out and (hashed tables) the
// snapshot's region is looked up once per node instead of once per candidate; the group
// kernels, capped at 64 registers, spill 52 bytes instead of 116.
template <bool DENSE, bool L0 = false>
struct LMPolicy {
  static constexpr int MIN_BLOCKS = DENSE ? MSLICE_DENSE_MIN_BLOCKS : MSLICE_GROUP_MIN_BLOCKS;
  static constexpr int BLOCK_MIN_BLOCKS = L0 ? 6 : 4;
  LevelDev g;
  const int32_t* labels;
  const int32_t* size;
  SigStore sig;
  const u128* lam;
  int32_t* target;
  TrackView trk;

  typedef Slot Probe;
  // Per node: own community and its size; at level 0 the node's snapshot s,
  // strength k and A = nd * Lambda_s * k (nd: od, or 1 for the global null
  // model), so a candidate costs one probe and
  // one 128x64-bit product.
  struct VCtx {
    int32_t a, size_a, s;
    bool single;
    long long k;
    Omega om;
    u128 A;
    uint64_t base, size;  // L0: the snapshot's hash region
  };

  __device__ bool begin(int32_t) const { return true; }
  __device__ VCtx vctx(int32_t v) const {
    VCtx c;
    c.a = labels[v];
    c.size_a = size[c.a];
    c.single = L0 || g.is0 != 0;
    c.s = 0;
    c.k = 0;
    c.A = 0;
    c.om = node_omega(g, v);
    if (c.single) {
      c.k = g.k0[v];
      c.s = node_slice0(g, v);
      if constexpr (L0 && !DENSE) hash_region(sig.h, pack_cs(0, c.s), c.base, c.size);
      if (c.k > 0) c.A = (u128)(ull)null_scale(g, c.om) * lam[c.s] * (u128)(ull)c.k;
    }
    return c;
  }
  __device__ void skip(int32_t v) const { target[v] = NO_MOVE; }
  __device__ bool edge(int32_t, const VCtx& vc, int64_t e, int32_t& key, long long& w) const {
    int32_t u;
    if (!edge_at<L0>(g, e, u, w, vc.om)) return false;
    key = labels[u];
    return true;
  }
  __device__ int32_t own_key(int32_t v) const { return labels[v]; }
  __device__ i128 key_of(int32_t v, const VCtx& vc, int32_t c, long long W, bool self) const {
    const u128 ns = null_sum<DENSE>(g, lam, sig, v, c, self);
    return (((i128)W) << P_BITS) - (i128)((u128)(ull)null_scale(g, vc.om) * ns);
  }
  __device__ Probe probe(int32_t, const VCtx& vc, int32_t c) const {
    if (vc.single && vc.k > 0) {
      if constexpr (L0 && !DENSE)
        return hash_first_at(sig.h, pack_cs(c, vc.s), vc.base, vc.size);
      else
        return sst_first<DENSE>(sig, c, vc.s);
    }
    return Slot{EMPTY_KEY, 0};
  }
  __device__ Cand cand(int32_t v, const VCtx& vc, int32_t c, long long W, const Probe& pr) const {
    if (L0 || vc.single) {
      const long long x = vc.k > 0 ? sst_resolve<DENSE>(sig, c, vc.s, pr) : 0;
      return Cand{(((i128)W) << P_BITS) - (i128)(vc.A * (u128)(ull)x), c};
    }
    return Cand{key_of(v, vc, c, W, false), c};
  }
  __device__ i128 own(int32_t v, const VCtx& vc, long long Wown) const {
    if (L0 || vc.single) {
      const long long x = vc.k > 0 ? sst_get<DENSE>(sig, vc.a, vc.s) - vc.k : 0;
      return (((i128)Wown) << P_BITS) - (i128)(vc.A * (u128)(ull)x);
    }
    return key_of(v, vc, vc.a, Wown, true);
  }
  // slice-parallel scoring (block tiers, aggregated levels)
  __device__ int64_t slice_count(int32_t v) const { return L0 || g.is0 ? 0 : g.sptr[v + 1] - g.sptr[v]; }
  __device__ bool own_walks_slices() const { return true; }
  template <int U>
  __device__ u128 null_part(int32_t v, const VCtx&, int32_t c, bool self, int t, int nt) const {
    return null_sum_part<DENSE, U>(g, lam, sig, v, c, self, t, nt);
  }
  __device__ Cand cand_ns(int32_t, const VCtx& vc, int32_t c, long long W, const u128& ns) const {
    return Cand{(((i128)W) << P_BITS) - (i128)((u128)(ull)null_scale(g, vc.om) * ns), c};
  }
  __device__ i128 own_ns(int32_t, const VCtx& vc, long long Wown, const u128& ns) const {
    return (((i128)Wown) << P_BITS) - (i128)((u128)(ull)null_scale(g, vc.om) * ns);
  }
  __device__ void finish(int32_t v, const Cand& best, long long, const i128& Ga, const VCtx& vc) const {
    const int32_t a = vc.a;
    const bool has = best.label != INT32_MAX;
    const i128 Gmax = (has && best.G > Ga) ? best.G : Ga;
    int32_t t = NO_MOVE;
    if (vc.size_a > 1 && Gmax < 0) {
      t = TO_EMPTY;
    } else if (has && best.G > Ga) {
      if (!(vc.size_a == 1 && best.label > a && size[best.label] == 1)) t = best.label;
    }
    target[v] = t;
    if (t == NO_MOVE && track_mode(trk) != TRACK_OFF)
      track_record<L0>(trk, g, vc.om, v, vc.size_a == 1, has, Ga, best.G);
  }
};

// The bucket lists of a round, for nodes that join them while it runs.
struct BucketLists {
  int32_t* lists;
  int64_t row_stride;
  int32_t* cursors;
  TierOff off;
  const uint16_t* seg;
};

// Appends node u (segment sg, class and tier) to its class's list.
__device__ __forceinline__ void bucket_append(const BucketLists& bl, int sg, int32_t u) {
  const int q = sg / NTIERS, t = sg % NTIERS;
  bl.lists[(int64_t)q * bl.row_stride + bl.off.off[t] + atomicAdd(&bl.cursors[sg], 1)] = u;
}

// The (snapshot, strength) lists of a warp's movers move between the two
// communities' rows.  The lists' entries are dealt to the lanes as one sequence
// (a mover of 30 entries walked by its own thread held the warp for 60 dependent
// loads).  All lanes of the warp call it; a lane without a mover has b == e.
__device__ __forceinline__ void move_slices(const LevelDev& g, const SigStore& sig, int32_t v, int32_t a, int32_t t,
                                            int64_t b, int64_t e, int lane) {
  int incl = (int)(e - b);
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += y;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  for (int i0 = 0; i0 < total; i0 += 32) {
    const int i = i0 + lane;
    int m = 0;  // the mover holding entry i: the lanes before it sum to at most i
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
      const int x = __shfl_sync(0xffffffffu, incl, m + d - 1);
      if (x <= i) m += d;
    }
    m = min(m, 31);
    const int before = m > 0 ? 1 : 0;
    const int prev = __shfl_sync(0xffffffffu, incl, m - before);
    const int32_t vm = __shfl_sync(0xffffffffu, v, m), am = __shfl_sync(0xffffffffu, a, m),
                  tm = __shfl_sync(0xffffffffu, t, m);
    const int64_t bm = __shfl_sync(0xffffffffu, b, m);
    if (i < total) {
      int32_t s;
      long long k;
      slice_entry(g, vm, bm + (i - (before ? prev : 0)), s, k);
      ss_add(sig, am, s, -k);
      if (tm >= 0) ss_add(sig, tm, s, k);
    }
  }
}

// Tracked rounds: the strength a mover takes through its null slices counts
// against their budgets.  At level 0 (one slice a node, lists in node order)
// most movers of a warp share a slice: their strengths are added up first.
__device__ __forceinline__ void track_moved(const TrackView& trk, int32_t s, long long k) {
  const long long old = (long long)atomicAdd((ull*)&trk.E[s], (ull)k);
  if (old + k > trk.B[s]) trk.state[TRACK_PAST] = 1;
}

// One neighbour u of a mover (from, to) over weight w; see track_push.
__device__ __forceinline__ void track_push_one(const TrackView& trk, const BucketLists& bl, int q, int32_t u,
                                               long long d, long long slack) {
  if (slack < 0) return;
  const long long old = (long long)atomicAdd((ull*)&trk.slack[u], (ull)(-d));
  if (old >= 0 && old < d) {
    const int sg = bl.seg[u];
    if ((sg & SEG_SETTLED) && sg != SEG_FROZEN) {
      const int sgu = sg & ~(int)SEG_SETTLED;
      if (sgu / NTIERS > q) bucket_append(bl, sgu, u);
    }
  }
}

// A warp takes its movers' moves off the margins of their neighbours; a settled
// one that has to decide after all joins the list of its class when that is still
// to come in this round (it decides in the next one otherwise: its class has been
// decided, from the state before this move).  (The label of a neighbour that moves
// in this sub-round may be read before or after its move: that neighbour has to
// decide either way.)  The movers' rows are dealt to the lanes as one sequence,
// four entries a lane at a time, so that the loads of four neighbours are in
// flight: mover by mover, a warp with a few hubs held the sub-round for 0.3 ms.
// All lanes of the warp call it; a lane without a mover has no entries.
__device__ __forceinline__ void track_push(const TrackView& trk, const LevelDev& g, const int32_t* labels,
                                           const BucketLists& bl, int q, int32_t v, int32_t from, int32_t to,
                                           int64_t rb, int64_t re, int lane) {
  constexpr int U = 4;
  const Omega om = re > rb ? node_omega(g, v) : Omega{g.on, g.od};
  if (__any_sync(0xffffffffu, re - rb > (1 << 25))) {  // (their sum must fit 32 bits)
    for (int src = 0; src < 32; ++src) {
      const int32_t f = __shfl_sync(0xffffffffu, from, src), t = __shfl_sync(0xffffffffu, to, src);
      const int64_t b = __shfl_sync(0xffffffffu, rb, src), e = __shfl_sync(0xffffffffu, re, src);
      const Omega os{__shfl_sync(0xffffffffu, om.on, src), __shfl_sync(0xffffffffu, om.od, src)};
      for (int64_t x = b + lane; x < e; x += 32) {
        int32_t u;
        long long w;
        if (edge_at(g, x, u, w, os))
          track_push_one(trk, bl, q, u, track_drop(trk, labels[u], f, t, w), *(volatile long long*)&trk.slack[u]);
      }
    }
    return;
  }
  int incl = (int)(re - rb);
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += y;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  for (int i0 = 0; i0 < total; i0 += 32 * U) {
    int32_t us[U], fs[U], ts[U], cs[U];
    long long ws[U], sl[U];
    bool ok[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int i = i0 + 32 * k + lane;
      int m = 0;  // the mover whose entry i is: the lanes before it hold at most i
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1)
        if (__shfl_sync(0xffffffffu, incl, m + d - 1) <= i) m += d;
      m = min(m, 31);
      const int before = __shfl_sync(0xffffffffu, incl, m > 0 ? m - 1 : 0);
      fs[k] = __shfl_sync(0xffffffffu, from, m);
      ts[k] = __shfl_sync(0xffffffffu, to, m);
      const int64_t b = __shfl_sync(0xffffffffu, rb, m);
      Omega os = om;
      if (g.od_i) {
        os.on = __shfl_sync(0xffffffffu, om.on, m);
        os.od = __shfl_sync(0xffffffffu, om.od, m);
      }
      ok[k] = i < total && edge_at(g, b + (i - (m > 0 ? before : 0)), us[k], ws[k], os);
    }
#pragma unroll
    for (int k = 0; k < U; ++k)
      if (ok[k]) {
        cs[k] = labels[us[k]];
        sl[k] = *(volatile long long*)&trk.slack[us[k]];
      }
#pragma unroll
    for (int k = 0; k < U; ++k)
      if (ok[k]) track_push_one(trk, bl, q, us[k], track_drop(trk, cs[k], fs[k], ts[k], ws[k]), sl[k]);
  }
}

// Node idx of the lists of tiers [t0, t1), and their length.
__device__ __forceinline__ bool seg_item(const TierSegs& sg, int t0, int t1, int64_t idx, int32_t& v) {
#pragma unroll
  for (int t = 0; t < NTIERS; ++t) {
    if (t < t0 || t >= t1) continue;
    const int cnt = *sg.count[t];
    if (idx < cnt) {
      v = sg.list[t][idx];
      return true;
    }
    idx -= cnt;
  }
  return false;
}

__device__ __forceinline__ int seg_total(const TierSegs& sg, int t0, int t1) {
  int t = 0;
#pragma unroll
  for (int i = 0; i < NTIERS; ++i)
    if (i >= t0 && i < t1) t += *sg.count[i];
  return t;
}

// Applies the sub-round's decisions: labels, community sizes and Sigma, and
// resets each applied decision.  Moves to an empty community only leave here
// (their label is assigned by lm_empty).  Tracked rounds also lower the margins
// of the movers' neighbours.
// TRACK = false leaves the tracking out (its registers cost an untracked round's
// pass a third of its time).
template <bool TRACK>
__device__ __forceinline__ void lm_apply(const LevelDev& g, const TierSegs& sg, int32_t* labels, int32_t* size,
                                         const SigStore& sig, int32_t* target, ull* moved, int32_t* empties,
                                         int32_t* inst_moved, const TrackView& trk, const BucketLists& bl, int q) {
  const bool track = TRACK && track_mode(trk) != TRACK_OFF;
  const int lane = threadIdx.x & 31;
  const int warps = gridDim.x * (blockDim.x >> 5), warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  int local = 0, local_empty = 0;
  // A warp takes 32 list items at a time.  A tracked round walks its movers'
  // rows as well: there the tiers come one after another, heaviest first, fewer
  // items at a time, and a short list is dealt out to all warps.
  int used = 0;  // claims of the tiers before: the next tiers' start with other warps
  for (int part = 0; part < (track ? 3 : 1); ++part) {
    const int t0 = !track ? 0 : part == 0 ? 3 : part == 1 ? 2 : 0;
    const int t1 = !track || part == 0 ? NTIERS : part == 1 ? 3 : 2;
    const int total = seg_total(sg, t0, t1);
    const int most = !track || part == 2 ? 32 : part == 1 ? 4 : 1;
    const int take = track ? max(1, min(most, (total + warps - 1) / warps)) : 32;
    const int first = (warp + warps - used % warps) % warps;
    used += (total + take - 1) / take;
    for (int64_t base = (int64_t)first * take; base < total; base += (int64_t)warps * take) {
      const int64_t idx = base + lane;
      int32_t v = 0, t = NO_MOVE, a = 0;
      int64_t b = 0, e = 0, rb = 0, re = 0;
      if (lane < take && idx < total && seg_item(sg, t0, t1, idx, v)) t = target[v];
#if MSLICE_CHECKED
      if (t != NO_MOVE && (t >= g.N || (t < 0 && t != TO_EMPTY))) {
        atomicOr(g.chk, ERR_BOUNDS);
        t = NO_MOVE;
      }
#endif
      if (t != NO_MOVE) {
        if (inst_moved) inst_moved[node_inst(g, v)] = 1;
        a = labels[v];
        atomicSub(&size[a], 1);
        slice_range(g, v, b, e);
        if (g.is0 && e > b) {
          const int32_t s = node_slice0(g, v);
          const long long k = g.k0[v];
          ss_add(sig, a, s, -k);
          if (t >= 0) ss_add(sig, t, s, k);
        }
        if (track) {
          rb = g.rowptr[v];
          re = g.rowptr[v + 1];
          trk.slack[v] = TRACK_DEAD;
        }
      }
      if (track) {
        const unsigned mv = __ballot_sync(0xffffffffu, t != NO_MOVE);
        if (mv && g.is0) {
          const int32_t s = t != NO_MOVE ? node_slice0(g, v) : -1;
          const long long k = t != NO_MOVE ? g.k0[v] : 0;
          const int32_t s0 = __shfl_sync(0xffffffffu, s, __ffs(mv) - 1);
          const long long k0 = warp_sum(s == s0 ? k : 0ll);
          if (lane == 0) track_moved(trk, s0, k0);
          if (t != NO_MOVE && s != s0) track_moved(trk, s, k);
        } else if (t != NO_MOVE) {
          for (int64_t j = b; j < e; ++j) {
            int32_t s;
            long long k;
            slice_entry(g, v, j, s, k);
            track_moved(trk, s, k);
          }
        }
        if (mv) track_push(trk, g, labels, bl, q, v, a, t, rb, re, lane);
      }
      if (!g.is0) move_slices(g, sig, v, a, t, b, e, lane);
      if (t >= 0) {
        atomicAdd(&size[t], 1);
        labels[v] = t;
        target[v] = NO_MOVE;
        local++;
      } else if (t == TO_EMPTY) {
        local_empty++;
      }
    }
  }
  local = warp_sum(local);
  local_empty = warp_sum(local_empty);
  if ((threadIdx.x & 31) == 0) {
    if (local) atomicAdd(moved, (ull)local);
    if (local_empty) atomicAdd(empties, local_empty);
  }
}

template <class T>
__device__ __forceinline__ T block_scan_excl(T x, T* sm, T& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T incl = x;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T y = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += y;
  }
  if (lane == 31) sm[w] = incl;
  __syncthreads();
  if (w == 0) {
    const int nw = blockDim.x >> 5;
    const T a = lane < nw ? sm[lane] : T(0);
    T ai = a;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const T y = __shfl_up_sync(0xffffffffu, ai, d);
      if (lane >= d) ai += y;
    }
    if (lane < nw) sm[lane] = ai - a;
    if (lane == nw - 1) sm[32] = ai;
  }
  __syncthreads();
  const T r = incl - x + sm[w];
  total = sm[32];
  __syncthreads();
  return r;
}

// A pruned round whose movement has passed a budget: the settled nodes of class q
// (the next one) whose margin does not cover what their slices have moved past
// their budgets rejoin its lists (see track.cuh).  Four nodes a thread at a time,
// and a node's margin is read only when a slice of it has passed its budget.
__device__ __forceinline__ void track_rescan(const TrackView& trk, const LevelDev& g, const BucketLists& bl, int q) {
  constexpr int U = 4;
  if (track_mode(trk) != TRACK_PRUNE || !trk.state[TRACK_PAST]) return;
  const int64_t threads = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v0 < g.N; v0 += U * threads) {
    int sgs[U];
#pragma unroll
    for (int k = 0; k < U; ++k) sgs[k] = v0 + k * threads < g.N ? bl.seg[v0 + k * threads] : SEG_FROZEN;
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (!(sgs[k] & SEG_SETTLED) || sgs[k] == SEG_FROZEN) continue;
      const int sgv = sgs[k] & ~(int)SEG_SETTLED;
      if (sgv / NTIERS != q) continue;
      const int32_t v = (int32_t)(v0 + k * threads);
      double x = 0;
      if (g.is0) {
        const int32_t s = node_slice0(g, v);
        const long long over = trk.E[s] - trk.B[s];
        if (over > 0) x = (double)trk.lam[s] * (double)g.k0[v] * (double)over;
      } else {
        int64_t b, e;
        slice_range(g, v, b, e);
        for (int64_t j = b; j < e; ++j) {
          int32_t s;
          long long kk;
          slice_entry(g, v, j, s, kk);
          const long long over = trk.E[s] - trk.B[s];
          if (over > 0) x += (double)trk.lam[s] * (double)kk * (double)over;
        }
      }
      if (x <= 0) continue;
      const long long m = trk.slack[v];
      if (m >= 0 && m < track_cost(x * (double)null_scale(g, node_omega(g, v)) * trk.scale, 0.0))
        bucket_append(bl, sgv, v);
    }
  }
}

// Moves to an empty community, by a whole grid (bar: its barrier); called when
// the sub-round has some.  Within each instance, in ascending node order,
// the movers take the ascending labels of that instance that are free once
// every other move is applied and the movers have left.
//   blk:      2*gridDim.x ints (per-chunk counts)
//   freelist: all free labels in ascending order; mrank: movers' global ranks
//   icnt:     4*B + 2 ints (per-instance counts, then their prefixes); zero
//             on entry and left zero on exit
template <class Bar>
__device__ __forceinline__ void lm_empty(const LevelDev& g, int32_t B, int32_t* target, int32_t* labels, int32_t* size,
                                         const SigStore& sig, int32_t* blk, int32_t* freelist, int32_t* mrank, int32_t* icnt,
                                         Bar&& bar) {
  __shared__ int32_t sm[33];
  const int64_t N = g.N, nb = gridDim.x;
  const int64_t chunk = (N + nb - 1) / nb;
  const int64_t lo = min(N, (int64_t)blockIdx.x * chunk), hi = min(N, lo + chunk);
  int32_t* fcnt = icnt;           // free labels per instance
  int32_t* mcnt = icnt + B;       // movers per instance
  int32_t* fbase = icnt + 2 * B;  // exclusive prefixes (B + 1 each)
  int32_t* mbase = icnt + 3 * B + 1;
  int cf = 0, ce = 0;
  // (warp-uniform loop) consecutive nodes mostly share an instance: the lanes
  // of the same one are counted with one atomic.  A late iteration has hundreds
  // of thousands of free labels, and one atomic each on B counters took 0.3 ms
  // of a batch of 36 instances (N = 1.5 M, now 0.03 ms).
  for (int64_t i0 = lo + (threadIdx.x & ~31); i0 < hi; i0 += blockDim.x) {
    const int64_t i = i0 + (threadIdx.x & 31);
    const bool in = i < hi;
    const bool f = in && size[i] == 0, m = in && target[i] == TO_EMPTY;
    cf += f;
    ce += m;
    if (B > 1) {
      const int32_t inst = in ? node_inst(g, (int32_t)i) : -1;
      const unsigned peers = __match_any_sync(0xffffffffu, inst);
      const int nf = __popc(__ballot_sync(0xffffffffu, f) & peers), nm = __popc(__ballot_sync(0xffffffffu, m) & peers);
      if (in && (threadIdx.x & 31) == __ffs(peers) - 1) {
        if (nf) atomicAdd(&fcnt[inst], nf);
        if (nm) atomicAdd(&mcnt[inst], nm);
      }
    }
  }
  int tf, te;
  block_scan_excl(cf, sm, tf);
  block_scan_excl(ce, sm, te);
  if (threadIdx.x == 0) {
    blk[blockIdx.x] = tf;
    blk[nb + blockIdx.x] = te;
  }
  bar();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    int32_t a = 0, b = 0;
    for (int32_t i = 0; i < B; ++i) {
      fbase[i] = a;
      mbase[i] = b;
      if (B > 1) {
        a += fcnt[i];
        b += mcnt[i];
      }
    }
    fbase[B] = a;
    mbase[B] = b;
  }
  int pf = 0, pe = 0;
  for (int b = threadIdx.x; b < blockIdx.x; b += blockDim.x) {
    pf += blk[b];
    pe += blk[nb + b];
  }
  int tot_pf, tot_pe;
  block_scan_excl(pf, sm, tot_pf);
  block_scan_excl(pe, sm, tot_pe);
  pf = tot_pf;
  pe = tot_pe;
  for (int64_t base = lo; base < hi; base += blockDim.x) {
    const int64_t i = base + threadIdx.x;
    const int f = (i < hi && size[i] == 0) ? 1 : 0;
    const int m = (i < hi && target[i] == TO_EMPTY) ? 1 : 0;
    int totf, totm;
    const int rf = block_scan_excl(f, sm, totf);
    const int rm = block_scan_excl(m, sm, totm);
    if (f) freelist[pf + rf] = (int32_t)i;
    if (m) mrank[i] = pe + rm;
    pf += totf;
    pe += totm;
  }
  bar();
  for (int64_t v = lo + threadIdx.x; v < hi; v += blockDim.x) {
    if (target[v] != TO_EMPTY) continue;
    const int32_t inst = B > 1 ? node_inst(g, (int32_t)v) : 0;
    const int32_t L = freelist[fbase[inst] + (mrank[v] - mbase[inst])];
    labels[v] = L;
    size[L] = 1;
    int64_t b, en;
    slice_range(g, (int32_t)v, b, en);
    for (int64_t j = b; j < en; ++j) {
      int32_t s;
      long long k;
      slice_entry(g, (int32_t)v, j, s, k);
      ss_add(sig, L, s, k);
    }
    target[v] = NO_MOVE;
  }
  bar();
  if (blockIdx.x == 0)
    for (int32_t i = threadIdx.x; i < 4 * B + 2; i += blockDim.x) icnt[i] = 0;
}

// The tracking state of a round from that of the round before (prev) and what
// that round did.
//   - Tracking starts when the movement, going on as in the last two rounds,
//     is expected to stay under a sixteenth of the nodes, and stops past a
//     quarter: the movers' pushes and the drift of the null sums would leave
//     few nodes settled for what they cost.
//   - Pruning that leaves three nodes in four in the lists is given up until
//     the movement has fallen to a quarter, or for a number of rounds that
//     doubles each time (communities can swap nodes for dozens of rounds).
//   - After TRACK_FAILS levels of a kind (level 0, or aggregated) in a row whose
//     pruning was given up like that, the next ones of that kind begin with a pause
//     (see track_start): where margins are small beside the drift, every level of a
//     solve records and prunes in vain.  The Constant Potts Model with gamma = 1 on
//     T = 16, n = 100,000: 418 ms without this, 395 after 2 levels, 398 after 3; T = 64,
//     n = 100,000, where later levels' pruning works, lost 7% after 1 level and up to
//     2% after 2.
//   - Levels with fewer entries, or with short rows (the decisions cost little
//     more than the tracking), are not tracked, unless strength lists of two or
//     more entries a node make their decisions dear (TRACK_MIN_LOOKUPS).
// Measured: a start below a quarter paid a useless recording round at 14.5%
// movement (T = 64, n = 100,000), hence the sixteenth of the expected movement.
// Levels of 2^22, 2^20 and 2^18 entries as the least to track: within 1% of one
// another; tracking every level of 2^16 nodes: 0.85x on a long contact sequence
// and 0.89x on n = 1,000 graphs, whose pushes cost more than their decisions. With
// the strength-list rule the contact sequence went from 162 to 150 ms.
constexpr int64_t TRACK_MIN_ENTRIES = 1 << 20, TRACK_MIN_DEGREE = 8;
constexpr int64_t TRACK_MIN_LOOKUPS = 1 << 21;
constexpr double TRACK_START = 1.0 / 16, TRACK_STOP = 1.0 / 4;
constexpr int TRACK_FIRST_PAUSE = 8, TRACK_FAILS = 3;

struct TrackState {
  int32_t mode, pause, next_pause, moved, pause_moved;
};

// How a level's tracking starts: the mode of its first round, the rounds left
// untracked at least, and the length of the next pause.
struct TrackStart {
  int32_t mode, pause, next_pause;
};

__host__ __device__ __forceinline__ TrackState track_next(const int32_t* prev, bool first, const TrackStart& start,
                                                          long long moved, long long listed) {
  TrackState s{start.mode, start.pause, start.next_pause, 0, 0};
  if (first) return s;
  const long long settled = prev[TRACK_SETTLED];
  const int32_t before = prev[TRACK_MODE], last = prev[TRACK_MOVED];
  const double active = (double)(listed + settled);
  const double expect = last > 0 ? (double)moved * (double)moved / (double)last : (double)moved;
  s.pause = prev[TRACK_PAUSE];
  s.next_pause = prev[TRACK_NEXT_PAUSE];
  s.pause_moved = prev[TRACK_PAUSE_MOVED];
  s.moved = (int32_t)moved;
  if (before == TRACK_PRUNE && listed > 3 * settled) {
    s.pause = s.next_pause;
    s.next_pause = s.next_pause < (1 << 19) ? 2 * s.next_pause : 1 << 20;
    s.pause_moved = (int32_t)moved;
  }
  if (s.pause > 0) {
    s.pause--;
    if (4 * moved < s.pause_moved) s.pause = 0;
  }
  if (s.pause > 0)
    s.mode = TRACK_OFF;
  else if (before == TRACK_OFF)
    s.mode = expect < TRACK_START * active ? TRACK_RECORD : TRACK_OFF;
  else
    s.mode = (double)moved < TRACK_STOP * active ? TRACK_PRUNE : TRACK_OFF;
  return s;
}

// fails: levels of this kind in a row whose pruning was given up.
inline TrackStart track_start(bool from_singletons, int fails) {
  if (fails < TRACK_FAILS) return TrackStart{from_singletons ? TRACK_OFF : TRACK_RECORD, 0, TRACK_FIRST_PAUSE};
  const int32_t pause = TRACK_FIRST_PAUSE << std::min(fails - TRACK_FAILS, 16);
  return TrackStart{TRACK_OFF, pause, 2 * pause};
}

// The count after a level that ended in `state` with `listed` nodes in its last
// round's lists; start: how it began.
inline int track_fails(int fails, const TrackStart& start, const int32_t* state, long long listed) {
  if (state[TRACK_MODE] == TRACK_PRUNE)
    return listed > 3 * (long long)state[TRACK_SETTLED] ? fails + 1 : 0;
  // (in a pause that began in this level)
  return state[TRACK_PAUSE] > 0 && state[TRACK_NEXT_PAUSE] > start.next_pause ? fails + 1 : fails;
}

__device__ __forceinline__ void track_store(int32_t* state, const TrackState& s) {
  state[TRACK_MODE] = s.mode;
  state[TRACK_PAUSE] = s.pause;
  state[TRACK_NEXT_PAUSE] = s.next_pause;
  state[TRACK_MOVED] = s.moved;
  state[TRACK_PAUSE_MOVED] = s.pause_moved;
}

template <bool DENSE, bool L0 = false>
inline LMPolicy<DENSE, L0> lm_policy(const Solver& S, const Level& L, const int32_t* labels, const TrackView& trk) {
  LMPolicy<DENSE, L0> pol;
  pol.g = L.d;
  pol.labels = labels;
  pol.size = S.size;
  pol.sig = S.sig;
  pol.lam = S.lam;
  pol.target = S.target;
  pol.trk = trk;
  return pol;
}

inline TierOff tier_offsets(const Solver& S) {
  TierOff to;
  for (int t = 0; t < NTIERS; ++t) to.off[t] = S.tier_off[t];
  return to;
}

// The tracking view of round r: budgets, movement and state words alternate
// between two sets (trk: the view of even rounds).
inline TrackView track_at(const TrackView& trk, int32_t Tn, int r) {
  TrackView t = trk;
  if (!t.state) return t;
  const int64_t p = r & 1;
  t.state = trk.state + p * TRACK_WORDS;
  t.E = trk.E + p * Tn;
  t.B = trk.B + p * Tn;
  t.Ep = trk.E + (1 - p) * Tn;
  t.Bp = trk.B + (1 - p) * Tn;
  return t;
}

// Work to decide in a round (entries, and a node counted as so many) up to
// which rounds are resident, and the same for a level's refinement.  A round of
// launches costs 160 us however little it decides, a resident one 60-80 us, but
// on one 512-thread block per SM; with the bound at 2^21, 2^22 or 6 million the
// solves took the same time, at 16 million a batch of 36 was 4% slower.
constexpr int64_t RESIDENT_MAX_WORK = (int64_t)1 << 22, RESIDENT_NODE_WORK = 16;
constexpr int64_t RESIDENT_REFINE_WORK = (int64_t)1 << 21;

// The bound in force: MSLICE_RESIDENT_MAX_WORK lowers it (0: nothing is resident).
inline int64_t resident_work(int64_t bound) {
  const char* e = std::getenv("MSLICE_RESIDENT_MAX_WORK");
  return e ? std::min<int64_t>(bound, std::atoll(e)) : bound;
}

// Bytes behind the list lengths for a resident launch's control words.
constexpr size_t RESIDENT_CTL_BYTES = 1024;
// Words of a dense table up to which a resident launch builds it itself.
constexpr int64_t RESIDENT_BUILD_MAX = (int64_t)1 << 20;

// Rounds in one launch (lm_rounds.cu): from round r, up to r_end, while nodes
// move, no hash region needs a rebuild and no round lists more than max_listed
// nodes.  Synchronises.
struct ResidentIn {
  int r = 0, r_end = 0;
  bool first = false;        // r is the level's first round
  bool build = false;        // sizes and (dense) Sigma are to be built first
  TrackStart start{TRACK_OFF, 0, TRACK_FIRST_PAUSE};
  long long prev_moved = 0, prev_listed = 0;
  long long max_listed = 0;
};
struct ResidentOut {
  int64_t rounds = 0, moves = 0, last_moved = 0, last_listed = 0, communities = 0;
  int32_t state[TRACK_WORDS] = {};  // of the last round
  ull used = 0;
  unsigned status = 0;
};
void resident_rounds(Solver& S, const Level& L, int32_t* labels, int it, int lvl, const TrackView& trk,
                     const ResidentIn& in, const int32_t* active, ResidentOut& out);

}  // namespace mslice
