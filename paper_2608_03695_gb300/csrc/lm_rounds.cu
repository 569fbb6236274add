// Resident rounds of local moving: one cooperative launch runs a level's rounds
// until nothing moves (or the host has to step in), with grid barriers where
// the host-driven rounds of local_move.cu have kernel boundaries.
//
// A host-driven round is about 28 launches and a synchronisation, 160 us however
// little there is to decide; most rounds of most levels (all of a small graph's,
// and the pruned tail of a large level) have a few microseconds of work.  Here a
// round costs 2K + 1 grid barriers.  The price is occupancy: every degree tier
// is decided by the same blocks of 512 threads, one per SM (their tables take
// 107 KB of shared memory), which keeps fewer nodes in flight than the tiers'
// own kernels; rounds with more than RESIDENT_MAX_WORK to decide
// are left to those (see local_move()).
//
// Double buffering by the round's parity replaces the clearing launches: lists'
// lengths, move counts and tracking words of the other parity are cleared by
// block 0 between the round's first and second barrier, when every block has
// read what it needs of them.
#include <cstddef>
#include <cstring>

#include "../../include/mslice.h"
#include "resident.cuh"

namespace mslice {

namespace {

// Device words of a launch.
struct ResidentCtl {
  ull moved[2];            // moves of the round, by parity (moves to empty communities apart)
  int32_t empties[2][64];  // moves to empty communities per sub-round
  // results
  long long rounds, moves, last_moved, last_listed;
  ull communities;  // non-empty at the end
  ull used;         // the hash's rebuild flag
  unsigned status;
  int32_t state[TRACK_WORDS];
};
static_assert(sizeof(ResidentCtl) <= RESIDENT_CTL_BYTES, "room behind the list lengths");

struct ResidentArgs {
  LevelDev g;
  int32_t *labels, *size, *target;
  SigStore sig;
  const uint8_t* tier;
  uint16_t* seg;
  int32_t* lists;
  int64_t row_stride;
  TierOff off;
  int32_t* cursors;    // 2 x K x NTIERS
  int32_t* inst_moved; // 2 x B (nullptr: single solve)
  int32_t* lm_active;
  const int32_t* active;
  int32_t B;
  TrackView trk;       // of even rounds
  int32_t Tn;
  TrackStart start;
  int32_t first;                 // the level's first round is this launch's
  long long prev_moved, prev_listed;  // of the round before this launch
  uint64_t seed, it, lvl;
  int32_t r0, r_end, K;
  long long max_listed;          // leave after a round that listed more nodes
  int32_t *gkeys;
  long long* gvals;
  const int64_t* goff;
  unsigned* status;
  const ull* sig_used;           // nullptr: dense tables
  int32_t build;                 // sizes and (dense) Sigma are to be built first
  int32_t *blk, *freelist, *mrank, *icnt;
  ResidentCtl* ctl;
};

template <class Pol>
__global__ void __launch_bounds__(RT, 1) k_lm_rounds(Pol pol, ResidentArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  long long* hv = reinterpret_cast<long long*>(smem);
  int32_t* hk = reinterpret_cast<int32_t*>(smem + R_SLOTS * sizeof(long long));
  uint16_t* cl = reinterpret_cast<uint16_t*>(smem + R_SLOTS * (sizeof(long long) + sizeof(int32_t)));
  __shared__ int32_t ncand[RW * 4];
  __shared__ int32_t block_ncand;
  __shared__ Cand red[RW];
  __shared__ ull usm[2 * RW];
  __shared__ i128 own_sm;
  __shared__ int32_t seg_cnt[64 * NTIERS], seg_base[64 * NTIERS];
  __shared__ int32_t mode_sh;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < R_SLOTS; i += RT) {
    hk[i] = -1;
    hv[i] = 0;
  }
  for (int i = threadIdx.x; i < RW * 4; i += RT) ncand[i] = 0;
  if (threadIdx.x == 0) block_ncand = 0;
  if (a.build) {
    // community sizes and Sigma of the labels: five launches less a level
    const int64_t tid = (int64_t)blockIdx.x * RT + threadIdx.x, threads = (int64_t)gridDim.x * RT;
    for (int64_t i = tid; i < a.g.N; i += threads) a.size[i] = 0;
    for (int64_t i = tid; i < a.sig.rows * a.sig.T; i += threads) a.sig.d[i] = 0;
    resident_bar();
    if (a.g.is0) {
      for (int64_t v = tid; v < a.g.N; v += threads) {
        const int32_t c = a.labels[v];
        atomicAdd(&a.size[c], 1);
        if (a.g.k0[v] > 0) ss_add(a.sig, c, node_slice0(a.g, (int32_t)v), a.g.k0[v]);
      }
    } else {
      for (int64_t v = tid >> 3; v < a.g.N; v += threads >> 3) {
        const int32_t c = a.labels[v];
        if ((lane & 7) == 0) atomicAdd(&a.size[c], 1);
        for (int64_t j = a.g.sptr[v] + (lane & 7); j < a.g.sptr[v + 1]; j += 8) ss_add(a.sig, c, a.g.sidx[j], a.g.sval[j]);
      }
    }
    // (complete at the barrier after the first round's lists)
  }
  const int nseg = a.K * NTIERS;
  long long moved = a.prev_moved, listed = a.prev_listed, moves = 0;
  int32_t r = a.r0;
  for (;;) {
    const int p = r & 1;
    TrackView trk = a.trk;
    int32_t mode = TRACK_OFF;
    if (a.trk.state) {
      trk.state = a.trk.state + p * TRACK_WORDS;
      trk.E = a.trk.E + (int64_t)p * a.Tn;
      trk.B = a.trk.B + (int64_t)p * a.Tn;
      trk.Ep = a.trk.E + (int64_t)(1 - p) * a.Tn;
      trk.Bp = a.trk.B + (int64_t)(1 - p) * a.Tn;
      if (threadIdx.x == 0) {
        const TrackState st =
            track_next(a.trk.state + (1 - p) * TRACK_WORDS, a.first && r == a.r0, a.start, moved, listed);
        mode_sh = st.mode;
        if (blockIdx.x == 0) track_store(trk.state, st);
      }
      __syncthreads();
      mode = mode_sh;
      track_budgets(trk, mode, a.Tn, blockIdx.x * RT + threadIdx.x, gridDim.x * RT);
    }
    const BucketLists bl{a.lists, a.row_stride, a.cursors + p * nseg, a.off, a.seg};
    const bool first_here = r == a.r0;
    const bool prune = mode == TRACK_PRUNE;
    const int32_t* prev_moved = a.inst_moved && !first_here ? a.inst_moved + (1 - p) * a.B : nullptr;
    int settled = 0;
    resident_list(a.g.N, nseg, a.lists, a.row_stride, a.off, bl.cursors, seg_cnt, seg_base, [&](int32_t v) {
      int s = prev_moved && !prev_moved[node_inst(a.g, v)]
                  ? (int)SEG_FROZEN
                  : bucket_seg(a.g, a.tier, a.seed, 0, a.it, a.lvl, (uint64_t)r, a.K, a.active, v);
      if (prune && s < nseg && track_settled(trk, a.g, v, trk.slack[v], a.g.is0 ? a.g.k0[v] : 0)) {
        s |= SEG_SETTLED;
        ++settled;
      }
      a.seg[v] = (uint16_t)s;
      return s;
    });
    if (prune) {
      settled = warp_sum(settled);
      if (lane == 0 && settled) atomicAdd(&trk.state[TRACK_SETTLED], settled);
    }
    resident_bar();
    pol.trk = trk;
    if (blockIdx.x == 0) {
      // the other parity's words: read by every block before the barrier above
      if (a.inst_moved)
        for (int32_t i = threadIdx.x; i < a.B; i += RT) {
          if (!first_here && !a.inst_moved[(1 - p) * a.B + i]) a.lm_active[i] = 0;
          a.inst_moved[(1 - p) * a.B + i] = 0;
        }
      for (int i = threadIdx.x; i < nseg; i += RT) a.cursors[(1 - p) * nseg + i] = 0;
      for (int i = threadIdx.x; i < a.K; i += RT) a.ctl->empties[1 - p][i] = 0;
      if (threadIdx.x == 0) {
        a.ctl->moved[1 - p] = 0;
        if (a.trk.state)
          a.trk.state[(1 - p) * TRACK_WORDS + TRACK_PAST] = a.trk.state[(1 - p) * TRACK_WORDS + TRACK_SETTLED] = 0;
      }
    }
    for (int q = 0; q < a.K; ++q) {
      const TierSegs sg = resident_segs(a.lists, a.row_stride, a.off, bl.cursors, q);
      resident_deal(
          sg,
          [&](int32_t v) {
            if (table_bits_for_degree(a.g.rowptr[v + 1] - a.g.rowptr[v]) <= TIER4_SMEM_BITS)
              block_decide_node<Pol, RT, 4>(pol, v, hk, hv, cl, &block_ncand, red, usm, &own_sm);
            else
              block_decide_scratch<Pol, RT, 4>(pol, v, a.gkeys, a.gvals, a.goff, a.status, red, usm, &own_sm);
          },
          [&](int32_t v) {
            group_decide_node<Pol, 32, T2_BITS, 2>(pol, v, hk + w * R_PER_WARP, hv + w * R_PER_WARP,
                                                   cl + w * (R_PER_WARP / 2), &ncand[w * 4], lane, 0xffffffffu);
          },
          [&](int32_t v, int gi, int gl) {
            const int o = w * R_PER_WARP + gi * 64;
            group_decide_node<Pol, 8, 6, 4>(pol, v, hk + o, hv + o, cl + w * (R_PER_WARP / 2) + gi * 32,
                                            &ncand[w * 4 + gi], gl, 0xffu << (gi * 8));
          });
      resident_bar();
      lm_apply<true>(a.g, sg, a.labels, a.size, a.sig, a.target, &a.ctl->moved[p], &a.ctl->empties[p][q],
               a.inst_moved ? a.inst_moved + p * a.B : nullptr, trk, bl, q);
      resident_bar();
      const bool past = mode == TRACK_PRUNE && trk.state[TRACK_PAST];
      const bool empties = a.ctl->empties[p][q] > 0;
      if (past) track_rescan(trk, a.g, bl, q + 1);
      if (empties)
        lm_empty(a.g, a.B, a.target, a.labels, a.size, a.sig, a.blk, a.freelist, a.mrank, a.icnt,
                 [] { resident_bar(); });
      else if (past)
        resident_bar();
    }
    // ---- end of the round (every block reads the same words; nobody writes
    // them before the next round's first barrier)
    moved = (long long)a.ctl->moved[p];
    for (int q = 0; q < a.K; ++q) moved += a.ctl->empties[p][q];
    listed = 0;
    for (int i = 0; i < nseg; ++i) listed += bl.cursors[i];
    moves += moved;
    ++r;
    if (moved == 0 || r >= a.r_end || listed > a.max_listed || (a.sig_used && *a.sig_used) || *a.status) break;
  }
  {
    int n = 0;
    for (int64_t v = (int64_t)blockIdx.x * RT + threadIdx.x; v < a.g.N; v += (int64_t)gridDim.x * RT)
      n += a.size[v] > 0;
    n = warp_sum(n);
    if (lane == 0 && n) atomicAdd(&a.ctl->communities, (ull)n);
  }
  if (blockIdx.x == 0) {
    if (a.inst_moved) {
      const int p = (r - 1) & 1;
      for (int32_t i = threadIdx.x; i < a.B; i += RT) {
        if (!a.inst_moved[p * a.B + i]) a.lm_active[i] = 0;
        a.inst_moved[p * a.B + i] = 0;
      }
    }
    if (threadIdx.x == 0) {
      a.ctl->rounds = r - a.r0;
      a.ctl->moves = moves;
      a.ctl->last_moved = moved;
      a.ctl->last_listed = listed;
      a.ctl->used = a.sig_used ? *a.sig_used : 0;
      a.ctl->status = *a.status;
      if (a.trk.state)
        for (int i = 0; i < TRACK_WORDS; ++i) a.ctl->state[i] = a.trk.state[((r - 1) & 1) * TRACK_WORDS + i];
    }
  }
}

template <class Pol>
void launch_rounds(Ctx& c, const Pol& pol, const ResidentArgs& a, unsigned grid) {
  const size_t bytes = TIER4_SMEM_BYTES;
  check_cuda(cudaFuncSetAttribute(k_lm_rounds<Pol>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes),
             "resident rounds' shared memory");
  launch_coop(c, k_lm_rounds<Pol>, dim3(grid), dim3(RT), bytes, pol, a);
}

}  // namespace

void resident_rounds(Solver& S, const Level& L, int32_t* labels, int it, int lvl, const TrackView& trk,
                     const ResidentIn& in, const int32_t* active, ResidentOut& out) {
  Ctx& c = *S.c;
  ResidentArgs a{};
  a.g = L.d;
  a.labels = labels;
  a.size = S.size;
  a.target = S.target;
  a.sig = S.sig;
  a.tier = S.tier;
  a.seg = S.bseg;
  a.lists = S.lists;
  a.row_stride = S.N0;
  a.off = tier_offsets(S);
  a.cursors = S.cursors;
  a.inst_moved = S.B > 1 ? S.inst_moved : nullptr;
  a.lm_active = S.lm_active;
  a.active = active;
  a.B = S.B;
  a.trk = trk;
  a.Tn = S.Tn;
  a.start = in.start;
  a.first = in.first ? 1 : 0;
  a.prev_moved = in.prev_moved;
  a.prev_listed = in.prev_listed;
  a.seed = S.p.seed;
  a.it = (uint64_t)it;
  a.lvl = (uint64_t)lvl;
  a.r0 = in.r;
  a.r_end = in.r_end;
  a.K = S.p.K;
  a.max_listed = in.max_listed;
  a.gkeys = S.gkeys;
  a.gvals = S.gvals;
  a.goff = S.goff;
  a.status = c.d_status;
  a.sig_used = S.sig.d ? nullptr : S.sig_used;
  a.blk = S.empty_blk;
  a.freelist = S.freelist;
  a.mrank = S.tmp32b;
  a.icnt = S.inst_cnt;
  // (the control words lie behind the two sets of list lengths: one clear)
  const size_t lengths = (2 * (size_t)S.p.K * NTIERS * sizeof(int32_t) + 15) & ~(size_t)15;
  a.ctl = reinterpret_cast<ResidentCtl*>(reinterpret_cast<char*>(S.cursors) + lengths);
  a.build = in.build ? 1 : 0;
  check_cuda(cudaMemsetAsync(S.cursors, 0, lengths + sizeof(ResidentCtl), c.stream), "memset");
  const unsigned grid = resident_grid(L.d.N, (int64_t)S.tier_cnt[3] + S.tier_cnt[4], S.p.K, coop_share(S.sms));
  if (S.sig.d)
    launch_rounds(c, lm_policy<true>(S, L, labels, trk), a, grid);
  else
    launch_rounds(c, lm_policy<false>(S, L, labels, trk), a, grid);
  ResidentCtl h;
  const size_t at = offsetof(ResidentCtl, rounds);
  std::memcpy(&h.rounds, readback(c, &a.ctl->rounds, sizeof(ResidentCtl) - at), sizeof(ResidentCtl) - at);
  out.rounds = h.rounds;
  out.moves = h.moves;
  out.last_moved = h.last_moved;
  out.last_listed = h.last_listed;
  out.communities = (int64_t)h.communities;
  out.used = h.used;
  out.status = h.status;
  std::memcpy(out.state, h.state, sizeof(out.state));
}

}  // namespace mslice
