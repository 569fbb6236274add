// Which nodes a round of local moving can leave undecided.
//
// A node that decided to stay keeps staying until something its decision
// reads has changed enough.  When v decides to stay in community a, its margin
//   M = G(v,a) - max(0, max over its other candidates c of G(v,c)) >= 0
// (0: the empty community and every community v has no edge to, whose keys are
// at most 0).  Two things lower it later:
//   - a neighbour u (weight w) moves from b to t: the key of staying falls by
//     2^64 w when b = a, the key of t rises by 2^64 w when t != a: at most
//     2w, w, and 0 when u joins a.  Each mover takes that off the margins of
//     its neighbours (track_push);
//   - the null sums move.  With E_s the strength that has moved in null slice
//     s, no Sigma_{c,s} has changed by more than E_s, so both keys together
//     have changed by at most 2 nd Lambda_s k_{v,s} E_s.
// While the margin minus both stays >= 0, the decision rule's outcome is "stay"
// and v is left out of the round ("settled").  All roundings are downward, so
// leaving v out never changes a result.  A node alone in its community has no
// empty candidate (staying is worth 0, its candidates -M or less), and a
// neighbour's move can give it a candidate of any key up to 2^64 w: its margin
// is capped below one weight unit, so that any neighbour's move ends it.
//
// E_s is charged ahead: a margin is kept net of a budget B_s of movement for
// the whole round, so the lists are made once, at the round's start.  After
// movement past a budget (the flag), settled nodes whose margin does not cover
// the excess rejoin the lists before their class decides (track_rescan); a margin
// that a push takes below 0 makes its node rejoin at once.
//
// Modes of a round (device word, so that device-driven rounds need no host):
//   OFF     most nodes move: nothing is recorded, every node decides
//   RECORD  every node decides and records its margin
//   PRUNE   settled nodes are left out
// A round's decisions, by far its most expensive part, shrink from all nodes to
// those near a change.  Power-law graph, T = 16, n = 100,000 (1.6 M nodes, 33 M
// entries), level 0: after 6 of 19 rounds 90% of the nodes are settled, after 9
// 99%; a round goes from 1.3 ms to 0.17 ms (its launches), the level from 26.9
// to 16.2 ms, the second iteration's from 8.1 to 3.5 ms, the solve from 93.7 to
// 69.1 ms.  T = 64, n = 100,000 (6.4 M nodes): 459 to 258 ms.
#pragma once
#include "level.h"

namespace mslice {

enum : int32_t { TRACK_OFF = 0, TRACK_RECORD = 1, TRACK_PRUNE = 2 };

constexpr long long TRACK_DEAD = -(1ll << 62);   // margin of a node that has to decide
constexpr long long TRACK_CAP = 1ll << 30;       // largest stored margin
constexpr long long TRACK_MAX_DROP = 1ll << 31;  // a push of more ends any margin
constexpr int TRACK_MAX_SLICES = 32;             // nodes with longer strength lists always decide
constexpr uint16_t SEG_SETTLED = 0x8000;         // bucket segment of a settled node (class and tier kept)
constexpr uint16_t SEG_FROZEN = 0xffff;          // node of a converged instance

// Words of TrackView::state.
enum {
  TRACK_MODE = 0,        // mode of the round
  TRACK_PAST = 1,        // a budget has been passed in this round
  TRACK_SETTLED = 2,     // nodes settled at the round's start
  TRACK_PAUSE = 3,       // rounds left before tracking is tried again
  TRACK_NEXT_PAUSE = 4,  // length of the next pause
  TRACK_MOVED = 5,       // moves of the round before the last
  TRACK_PAUSE_MOVED = 6, // moves of the round that started the pause
  TRACK_WORDS = 8
};

struct TrackView {
  int32_t* state = nullptr;       // words below (nullptr: not tracking)
  long long* slack = nullptr;     // margins in units of 2^-F weight units, net of the round's budgets
  long long* E = nullptr;         // per null slice: strength moved in this round
  long long* B = nullptr;         // per null slice: budget of this round
  const long long* Ep = nullptr;  // the same of the round before (rounds alternate between two sets)
  const long long* Bp = nullptr;
  const long long* base = nullptr;  // per null slice: smallest budget
  const u128* lam = nullptr;
  int F = 0;                      // margin unit: 2^-F weight units
  double scale = 0;               // 2^(F-63): margin units per 2^64 of key, doubled
};

__device__ __forceinline__ int32_t track_mode(const TrackView& t) { return t.state ? t.state[TRACK_MODE] : TRACK_OFF; }

// Costs of xp and credits of xn margin units (both >= 0), each rounded against
// the node past every rounding of the products that made it (relative 2^-53
// each).
__device__ __forceinline__ long long track_cost(double xp, double xn) {
  const double up = xp > 0 ? xp * (1.0 + 0x1p-40) + 1.0 : 0.0, down = xn * (1.0 - 0x1p-40) - 1.0;
  const long long c = up >= 0x1p60 ? 1ll << 60 : (long long)ceil(up);
  const long long d = down >= 0x1p60 ? 1ll << 60 : down > 0 ? (long long)down : 0;
  return c - d;
}

// Margin cost of what is left of the budgets (B_s - E_s; a credit past them)
// for node v; false when the node's list is too long to be tracked.
template <bool L0>
__device__ __forceinline__ bool track_budget_cost(const TrackView& t, const LevelDev& g, const Omega& om, int32_t v,
                                                  long long& cost) {
  if constexpr (L0) {
    const int32_t s = node_slice0(g, v);
    const double x = (double)t.lam[s] * (double)g.k0[v] * (double)(t.B[s] - t.E[s]) *
                     ((double)null_scale(g, om) * t.scale);
    cost = track_cost(x > 0 ? x : 0, x < 0 ? -x : 0);
    return true;
  }
  int64_t b, e;
  slice_range(g, v, b, e);
  if (e - b > TRACK_MAX_SLICES) return false;
  double xp = 0, xn = 0;
  for (int64_t j = b; j < e; ++j) {
    int32_t s;
    long long k;
    slice_entry(g, v, j, s, k);
    const double x = (double)t.lam[s] * (double)k * (double)(t.B[s] - t.E[s]);
    xp += x > 0 ? x : 0;
    xn -= x < 0 ? x : 0;
  }
  const double f = (double)null_scale(g, om) * t.scale;
  cost = track_cost(xp * f, xn * f);
  return true;
}

// Margin of a node that decided to stay: Ga its key of staying, Gb its best
// other candidate's key when has.
template <bool L0>
__device__ __forceinline__ void track_record(const TrackView& t, const LevelDev& g, const Omega& om, int32_t v,
                                             bool alone, bool has, const i128& Ga, const i128& Gb) {
  // (alone without a candidate: a node without edges)
  const i128 M = has ? Ga - (alone || Gb > 0 ? Gb : (i128)0) : alone ? (i128)1 << 100 : Ga;
  long long m = TRACK_DEAD;
  if (M >= 0) {
    const i128 u = M >> (P_BITS - t.F);
    m = u > (i128)TRACK_CAP ? TRACK_CAP : (long long)u;
    long long cost;
    if (track_budget_cost<L0>(t, g, om, v, cost)) {
      const long long cap = !alone ? TRACK_CAP : t.F > 0 ? (1ll << t.F) - 1 : 0;
      m -= cost;
      m = m < cap ? m : cap;
    } else {
      m = TRACK_DEAD;
    }
  }
  t.slack[v] = m;
}

// A round's budget of a null slice: half of what moved in the round before
// (movement mostly falls faster than that), and the smallest budget.
__device__ __forceinline__ long long track_budget(const TrackView& t, int32_t s) { return t.Ep[s] / 2 + t.base[s]; }

// Round start: the budgets of slices first, first + step, ...; nothing has
// moved yet.
__device__ __forceinline__ void track_budgets(const TrackView& t, int32_t mode, int32_t Tn, int32_t first,
                                              int32_t step) {
  if (mode == TRACK_OFF) return;
  for (int32_t s = first; s < Tn; s += step) {
    t.E[s] = 0;
    t.B[s] = mode == TRACK_RECORD ? t.base[s] : track_budget(t, s);
  }
}

// Round start: charges the node's margin with the last round's movement and the
// change of the budgets, and says whether the node is settled for the round.
// (m: its margin; k0: its strength at level 0, both loaded ahead)
__device__ __forceinline__ bool track_settled(const TrackView& t, const LevelDev& g, int32_t v, long long m,
                                              int64_t k0) {
  if (m < 0) return false;
  double x = 0;
  // (a budget that shrinks is not credited: the cap of a node alone in its
  // community has to hold)
  if (g.is0) {
    const int32_t s = node_slice0(g, v);
    const long long grown = t.Ep[s] + track_budget(t, s) - t.Bp[s];
    if (grown > 0) x = (double)t.lam[s] * (double)k0 * (double)grown;
  } else {
    int64_t b, e;
    slice_range(g, v, b, e);  // (at most TRACK_MAX_SLICES: longer lists are recorded dead)
    for (int64_t j = b; j < e; ++j) {
      int32_t s;
      long long k;
      slice_entry(g, v, j, s, k);
      const long long grown = t.Ep[s] + track_budget(t, s) - t.Bp[s];
      if (grown > 0) x += (double)t.lam[s] * (double)k * (double)grown;
    }
  }
  if (x > 0) {
    m -= track_cost(x * (double)null_scale(g, node_omega(g, v)) * t.scale, 0.0);
    if (m < 0) m = TRACK_DEAD;
    t.slack[v] = m;
  }
  return m >= 0;
}

// What a mover (from b to t) takes off the margin of a neighbour in community
// c over an edge of weight w.
__device__ __forceinline__ long long track_drop(const TrackView& t, int32_t c, int32_t from, int32_t to, long long w) {
  if (c == to) return t.F > 0 ? 1ll << t.F : 1;  // (a neighbour alone until now must decide)
  if (t.F >= 0) {
    if (w >= (TRACK_MAX_DROP >> (t.F + 1))) return TRACK_MAX_DROP;
    return (c == from ? 2 * w : w) << t.F;
  }
  const long long d = (w >> (-t.F - 1)) + 2;  // >= 2w 2^F
  return d < TRACK_MAX_DROP ? d : TRACK_MAX_DROP;
}

}  // namespace mslice
