// Local moving (the Louvain/Leiden move phase, Sec. 3.2) of multislice
// modularity (Eq. multislice-modularity) under the synchronous schedule:
// in round r every node draws a class in [0, K) from the counter-based hash;
// in sub-round q the nodes of class q decide against the state at the start
// of the sub-round, then every decision is applied at once.
//
// Exact move key of node v for community c (c\v: v excluded):
//   G(v,c) = 2^64 W(v,c\v) - od * sum_s Lambda_s k_{v,s} Sigma_{c\v,s}
// with W in units of 1/od (intra-snapshot weight w counts od*w, a coupling
// entry counts on) and Lambda_s = floor(gn 2^64 / (gd 2m_s)).  G is 2^64*od
// times the modularity gain up to a per-node constant, with gamma/2m_s
// quantised to Lambda_s/2^64.  Best = largest key, ties to the smallest
// label; a node that is not alone may also move to an empty community
// (key 0, losing ties); it moves only on a strict improvement; a node alone
// in its community joins another singleton community only if that label is
// smaller (otherwise two neighbouring singletons could swap forever).
//
// Global null model (plain modularity of the supra-graph, Eq. modularity):
// one null slice per instance, strengths k' = od*k + on*(coupling edges),
// Lambda' = floor(gn 2^64 / (gd 2M')), 2M' = od*2mu, and the null term's
// scale od becomes 1 (Omega::nd):  G(v,c) = 2^64 W(v,c\v) - Lambda' k'_v
// Sigma'_{c\v}.
//
// Sigma_{c,s} lives in a hash keyed (c, s) and is kept exact by the integer
// atomics of every move; it is rebuilt from the labels only at the start of
// a level and when tombstone keys fill half of the table.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include "../../include/mslice.h"
#include "lm.cuh"

namespace cg = cooperative_groups;

namespace mslice {

namespace {

constexpr int APPLY_THREADS = 256;
constexpr int EMPTY_THREADS = 512;

unsigned fixed_grid(int per_sm) { return 152u * (unsigned)per_sm; }

// Tier of every node by degree, and by slice work at aggregated levels
// (sptr non-null: see work_tier).
__global__ void k_tier(const int64_t* rowptr, const int64_t* sptr, int32_t N, TierCuts cuts, uint8_t* tier,
                       int32_t* cnt, int64_t* gsize) {
  const int lane = threadIdx.x & 31;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < N; base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = base + threadIdx.x;
    int t = -1;
    if (v < N) {
      const int64_t d = rowptr[v + 1] - rowptr[v];
      t = work_tier(d, sptr ? sptr[v + 1] - sptr[v] : 0, cuts);
      tier[v] = (uint8_t)t;
      int64_t S = 0;
      if (t == NTIERS - 1) {
        S = 2;
        while (S < 2 * d) S <<= 1;
      }
      gsize[v] = S;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, t);
    if (t >= 0 && lane == __ffs(peers) - 1) atomicAdd(&cnt[t], __popc(peers));
  }
}

// Buckets the nodes of this round by (class, tier): row q of `lists` holds
// class q, tier t at [tier_off[t], tier_off[t] + count).  Order inside a
// bucket does not matter: decisions read only the sub-round snapshot.
// Bucketing in node order, in three steps over chunks of BUCKET_CHUNK
// consecutive nodes: count every chunk's nodes per (class, tier) segment,
// scan the counts of each segment over the chunks, then write every chunk's
// nodes at its offsets.  The lists come out in ascending node order, so the
// nodes a decision kernel holds in flight at any moment (a window of the
// list) are close in node order and their gathers (neighbour labels in the
// same snapshots, the snapshots' community-table regions) stay in L2.  A
// chunk is one block; ranks inside a chunk come from shared-memory atomics
// (order inside a chunk does not matter).
constexpr int BUCKET_THREADS = 256;
constexpr int BUCKET_ITEMS = 16;
constexpr int64_t BUCKET_CHUNK = (int64_t)BUCKET_THREADS * BUCKET_ITEMS;
constexpr int BUCKET_MAX_SEGS = 64 * NTIERS;  // segments (K * NTIERS) for K <= 64

// Step 1: segment of every node and counts[s * nchunks + chunk].  In a pruned
// round (trk) a settled node keeps its segment, marked, and is not counted.
__global__ void __launch_bounds__(BUCKET_THREADS)
    k_bucket_count(LevelDev g, const uint8_t* tier, uint64_t seed, uint64_t tag, uint64_t it, uint64_t lvl, uint64_t r,
                   int K, const int32_t* active, TrackView trk, uint16_t* seg, int32_t* counts,
                   int64_t nchunks) {
  __shared__ int32_t cnt[BUCKET_MAX_SEGS];
  const int nseg = K * NTIERS;
  const bool prune = track_mode(trk) == TRACK_PRUNE;
  int settled = 0;
  for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
    for (int i = threadIdx.x; i < nseg; i += BUCKET_THREADS) cnt[i] = 0;
    __syncthreads();
    constexpr int U = 4;  // nodes whose margins are loaded together
    for (int k0 = 0; k0 < BUCKET_ITEMS; k0 += U) {
      const int64_t v0 = ch * BUCKET_CHUNK + (int64_t)k0 * BUCKET_THREADS + threadIdx.x;
      if (v0 >= g.N) break;
      long long ms[U] = {};
      int64_t ks[U] = {};
      if (prune) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int64_t v = v0 + (int64_t)u * BUCKET_THREADS;
          if (v < g.N) {
            ms[u] = trk.slack[v];
            if (g.is0) ks[u] = g.k0[v];
          }
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t v = v0 + (int64_t)u * BUCKET_THREADS;
        if (v >= g.N) break;
        int sg = bucket_seg(g, tier, seed, tag, it, lvl, r, K, active, v);
        if (prune && sg < nseg && track_settled(trk, g, (int32_t)v, ms[u], ks[u])) {
          sg |= SEG_SETTLED;
          ++settled;
        }
        seg[v] = (uint16_t)sg;
        if (sg < nseg) atomicAdd(&cnt[sg], 1);
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nseg; i += BUCKET_THREADS) counts[(int64_t)i * nchunks + ch] = cnt[i];
    __syncthreads();
  }
  if (prune) {
    settled = warp_sum(settled);
    if ((threadIdx.x & 31) == 0 && settled) atomicAdd(&trk.state[TRACK_SETTLED], settled);
  }
}

// Step 2: one block per segment turns its counts into exclusive offsets over
// the chunks and stores the segment's size in cursors[s].
__global__ void __launch_bounds__(1024) k_bucket_scan(int32_t* counts, int64_t nchunks, int32_t* cursors) {
  __shared__ int32_t part[32];
  __shared__ int32_t carry;
  const int s = blockIdx.x;
  int32_t* c = counts + (int64_t)s * nchunks;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t base = 0; base < nchunks; base += blockDim.x) {
    const int64_t i = base + threadIdx.x;
    const int32_t x = i < nchunks ? c[i] : 0;
    int32_t incl = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    if (lane == 31) part[w] = incl;
    __syncthreads();
    if (w == 0) {
      const int32_t p = lane < (int)(blockDim.x >> 5) ? part[lane] : 0;
      int32_t pi = p;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, pi, d);
        if (lane >= d) pi += y;
      }
      part[lane] = pi - p;
    }
    __syncthreads();
    if (i < nchunks) c[i] = carry + part[w] + incl - x;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry += part[w] + incl;
    __syncthreads();
  }
  if (threadIdx.x == 0) cursors[s] = carry;
}

// Step 3: every chunk writes its nodes at its offsets.
__global__ void __launch_bounds__(BUCKET_THREADS)
    k_bucket_write(int32_t N, const uint16_t* seg, const int32_t* counts, int64_t nchunks, int K, int32_t* lists,
                   int64_t row_stride, TierOff tier_off) {
  __shared__ int32_t pos[BUCKET_MAX_SEGS];
  const int nseg = K * NTIERS;
  for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
    for (int i = threadIdx.x; i < nseg; i += BUCKET_THREADS) pos[i] = counts[(int64_t)i * nchunks + ch];
    __syncthreads();
    for (int k = 0; k < BUCKET_ITEMS; ++k) {
      const int64_t v = ch * BUCKET_CHUNK + (int64_t)k * BUCKET_THREADS + threadIdx.x;
      if (v >= N) break;
      const int sg = seg[v];
      if (sg >= nseg) continue;
      const int q = sg / NTIERS, t = sg % NTIERS;
      lists[(int64_t)q * row_stride + tier_off.off[t] + atomicAdd(&pos[sg], 1)] = (int32_t)v;
    }
    __syncthreads();
  }
}

__global__ void k_hash_clear(HashView h) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  if (h.narrow) {
    Slot8* sl = slots8(h);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < h.cap; i += stride)
      sl[i] = Slot8{EMPTY_KEY8, 0};
  } else {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < h.cap; i += stride)
      h.slots[i] = Slot{EMPTY_KEY, 0};
  }
}

// Aggregated levels: G lanes per node, sharing its list.
template <int G>
__global__ void k_sigma_insert_group(LevelDev g, const int32_t* labels, SigStore h, int32_t* size) {
  const int lane = threadIdx.x % G;
  const int64_t groups = (int64_t)gridDim.x * blockDim.x / G;
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G; v < g.N; v += groups) {
    const int32_t c = labels[v];
    if (size && lane == 0) atomicAdd(&size[c], 1);
    int64_t b, e;
    slice_range(g, (int32_t)v, b, e);
    for (int64_t j = b + lane; j < e; j += G) {
      int32_t s;
      long long k;
      slice_entry(g, (int32_t)v, j, s, k);
      ss_add(h, c, s, k);
    }
  }
}

__global__ void k_sigma_insert(LevelDev g, const int32_t* labels, SigStore h, int32_t* size) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < g.N; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t c = labels[v];
    if (size) atomicAdd(&size[c], 1);
    int64_t b, e;
    slice_range(g, (int32_t)v, b, e);
    for (int64_t j = b; j < e; ++j) {
      int32_t s;
      long long k;
      slice_entry(g, (int32_t)v, j, s, k);
      ss_add(h, c, s, k);
    }
  }
}

__global__ void k_count_sizes(const int32_t* size, int64_t N, ull* out) {
  int n = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x)
    n += size[v] > 0;
  n = warp_sum(n);
  if ((threadIdx.x & 31) == 0 && n) atomicAdd(out, (ull)n);
}

// Round start (one block) of a tracked round: its tracking state, budgets and
// counters, and the other parity's accumulators cleared for the round after.
__global__ void __launch_bounds__(512) k_round_begin(TrackView trk, int32_t* state_prev, int32_t Tn, int first,
                                                     TrackStart start, long long moved, long long listed,
                                                     int32_t* counters) {
  __shared__ int32_t mode_sh;
  if (threadIdx.x == 0) {
    const TrackState st = track_next(state_prev, first, start, moved, listed);
    mode_sh = st.mode;
    track_store(trk.state, st);
    trk.state[TRACK_PAST] = trk.state[TRACK_SETTLED] = 0;
    state_prev[TRACK_PAST] = state_prev[TRACK_SETTLED] = 0;
    counters[0] = counters[1] = counters[2] = 0;
  }
  __syncthreads();
  track_budgets(trk, mode_sh, Tn, threadIdx.x, blockDim.x);
}

// lm_active[i] stays 1 only for instances that moved in the round; clears
// the flags for the next round.
__global__ void k_round_freeze(int32_t* lm_active, int32_t* inst_moved, int32_t B) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < B) {
    if (!inst_moved[i]) lm_active[i] = 0;
    inst_moved[i] = 0;
  }
}

template <bool TRACK>
__global__ void k_lm_apply(LevelDev g, TierSegs sg, int32_t* labels, int32_t* size, SigStore sig, int32_t* target,
                           int32_t* counters, int32_t* inst_moved, TrackView trk, BucketLists bl, int q) {
  lm_apply<TRACK>(g, sg, labels, size, sig, target, (ull*)counters, &counters[2], inst_moved, trk, bl, q);
}

// The rest of a host-driven sub-round (one cooperative launch; it returns at
// once when there is nothing to do): settled nodes that rejoin the next class's
// lists, and the moves to an empty community.
__global__ void __launch_bounds__(EMPTY_THREADS) k_empty_pass(LevelDev g, int32_t B, int32_t* target, int32_t* labels,
                                                              int32_t* size, SigStore sig, int32_t* counters,
                                                              int32_t* blk, int32_t* freelist, int32_t* mrank,
                                                              int32_t* icnt, TrackView trk, BucketLists bl,
                                                              int q_next) {
  track_rescan(trk, g, bl, q_next);
  const int n_empty = counters[2];
  if (n_empty == 0) return;
  lm_empty(g, B, target, labels, size, sig, blk, freelist, mrank, icnt, [] { cg::this_grid().sync(); });
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // (every block has read counters[2] before the barriers)
    atomicAdd((ull*)counters, (ull)n_empty);
    counters[2] = 0;
  }
}

}  // namespace

LevelDev level0_view(const SupraGraph& G, long long on, long long od) {
  LevelDev d;
  d.N = (int32_t)G.N;
  d.n = (int32_t)(G.n > 0 ? G.n : 1);
  d.is0 = 1;
  d.rowptr = G.rowptr;
  d.adj0 = G.adj;
  d.k0 = G.k;
  d.on = on;
  d.od = od;
  return d;
}

LevelDev level0_view(const SupraGraph& G, const Solver& S) {
  LevelDev d = level0_view(G, S.p.on, S.p.od);
  if (G.B > 1) {
    d.slice0 = G.slice0;
    d.inst = G.inst0;
    d.inst_off = G.inst_off0;
    d.on_i = S.on_d;
    d.od_i = S.od_d;
  }
  if (S.cw_d) {
    d.cw = S.cw_d;
    d.ncw = G.ncw;
  }
  if (S.p.cpm) d.k0 = S.kn;  // CPM: every node weighs 1, snapshots as null slices
  if (S.p.global_null) {
    // one null slice per instance: the instance id (batches) or 0 (v / N)
    d.global_null = 1;
    d.k0 = S.kn;
    if (G.B > 1)
      d.slice0 = G.inst0;
    else
      d.n = (int32_t)(G.N > 0 ? G.N : 1);
  }
  return d;
}

void solver_alloc(Solver& S) {
  Ctx& c = *S.c;
  const int64_t N = S.N0 > 0 ? S.N0 : 1;
  S.target = c.ws->get<int32_t>("s_target", N);
  S.size = c.ws->get<int32_t>("s_size", N);
  S.tmp32a = c.ws->get<int32_t>("s_tmpa", N + 1);
  S.tmp32b = c.ws->get<int32_t>("s_tmpb", N + 1);
  S.freelist = c.ws->get<int32_t>("s_free", N + 1);
  S.tier = c.ws->get<uint8_t>("s_tier", N);
  S.cls = c.ws->get<uint8_t>("s_cls", N);
  S.bseg = c.ws->get<uint16_t>("s_bseg", N);
  S.bcounts = c.ws->get<int32_t>("s_bcounts", (size_t)S.p.K * NTIERS * ((N + BUCKET_CHUNK - 1) / BUCKET_CHUNK));
  S.lists = c.ws->get<int32_t>("s_lists", (size_t)N * S.p.K);
  S.cursors = c.ws->get<int32_t>("s_cursors", 2 * NTIERS * S.p.K + NTIERS + 4 + RESIDENT_CTL_BYTES / sizeof(int32_t));
  S.counters = c.ws->get<int32_t>("s_counters", 8);
  S.sig_used = c.ws->get<ull>("s_sig_used", 1);
  S.goff = c.ws->get<int64_t>("s_goff", N + 1);
  S.R = c.ws->get<int32_t>("s_R", N);
  S.sizeR = c.ws->get<int32_t>("s_sizeR", N);
  S.Wc = c.ws->get<long long>("s_Wc", N);
  S.Wout = c.ws->get<long long>("s_Wout", N);
  S.Wsel = c.ws->get<long long>("s_Wsel", N);
  S.rhs = c.ws->get<ull>("s_rhs", 2 * N);
  S.elig = c.ws->get<uint8_t>("s_elig", N);
  S.wc = c.ws->get<uint8_t>("s_wc", N);
  int max_blocks = 0;
  check_cuda(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&max_blocks, k_empty_pass, EMPTY_THREADS, 0), "occupancy");
  int dev = 0, sms = 0;
  check_cuda(cudaGetDevice(&dev), "device");
  check_cuda(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "attribute");
  S.sms = sms;
  S.empty_grid = std::max(1, std::min(max_blocks, 2) * sms);
  S.empty_blk = c.ws->get<int32_t>("s_empty_blk", 2 * (size_t)std::max(S.empty_grid, sms));
  S.wqueue = c.ws->get<int32_t>("s_wqueue", NTIERS);
  S.lm_active = c.ws->get<int32_t>("s_lm_active", S.B);
  S.inst_moved = c.ws->get<int32_t>("s_inst_moved", 2 * (size_t)S.B);
  check_cuda(cudaMemsetAsync(S.inst_moved, 0, 2 * (size_t)S.B * sizeof(int32_t), c.stream), "memset");
  S.inst_cnt = c.ws->get<int32_t>("s_inst_cnt", 4 * (size_t)S.B + 2);
  check_cuda(cudaMemsetAsync(S.inst_cnt, 0, (4 * (size_t)S.B + 2) * sizeof(int32_t), c.stream), "memset");
  fill_i32(c, S.target, NO_MOVE, N);
  check_cuda(cudaMemsetAsync(S.counters, 0, 8 * sizeof(int32_t), c.stream), "memset");
}

void prepare_level(Solver& S, const Level& L) {
  Ctx& c = *S.c;
  const int32_t N = L.d.N;
  configure_stores(S, N);
  if (L.tiers_known) {
    int32_t off = 0;
    for (int t = 0; t < NTIERS; ++t) {
      S.tier_cnt[t] = L.tier_cnt[t];
      S.tier_off[t] = off;
      off += L.tier_cnt[t];
    }
    return;
  }
  int32_t* cnt = S.cursors;  // reused: tier counts
  check_cuda(cudaMemsetAsync(cnt, 0, NTIERS * sizeof(int32_t), c.stream), "memset");
  int64_t* gsize = reinterpret_cast<int64_t*>(c.ws->get<int64_t>("s_gsize", (size_t)(N > 0 ? N : 1)));
  if (N > 0)
    launch(c, k_tier, dim3(grid_for(N, 256) < 4096 ? grid_for(N, 256) : 4096), dim3(256), 0, L.d.rowptr,
           (const int64_t*)(L.d.is0 ? nullptr : L.d.sptr), N, S.p.cuts, S.tier, cnt, gsize);
  int64_t* gtotal = c.ws->get<int64_t>("s_gtotal", 1);
  scan_excl(c, gsize, S.goff, N, gtotal);
  check_cuda(cudaMemcpyAsync(S.goff + N, gtotal, sizeof(int64_t), cudaMemcpyDeviceToDevice, c.stream), "copy");
  struct {
    int32_t cnt[NTIERS];
    int32_t pad;
    int64_t gt;
  } hb;
  check_cuda(cudaMemcpyAsync(&hb.cnt, cnt, NTIERS * sizeof(int32_t), cudaMemcpyDeviceToHost, c.stream), "copy");
  check_cuda(cudaMemcpyAsync(&hb.gt, gtotal, sizeof(int64_t), cudaMemcpyDeviceToHost, c.stream), "copy");
  sync(c);
  int32_t off = 0;
  for (int t = 0; t < NTIERS; ++t) {
    S.tier_cnt[t] = hb.cnt[t];
    S.tier_off[t] = off;
    off += hb.cnt[t];
  }
  if (hb.gt > S.gcap) {
    S.gcap = hb.gt;
    S.gkeys = c.ws->get<int32_t>("s_gkeys", S.gcap);
    S.gvals = c.ws->get<long long>("s_gvals", S.gcap);
    if (S.p.theta_num > 0) S.gwts = c.ws->get<ull>("s_gwts", S.gcap);
  }
}

// Level-0 nodes of every null slice: the snapshot's n (Q_MS and CPM, whose
// null slices are the snapshots) or the instance's n*T (the global model,
// one null slice per instance).
static std::vector<int64_t> null_slice_nodes(const Solver& S) {
  const SupraGraph& G = *S.G0;
  std::vector<int64_t> out(S.Tn > 0 ? S.Tn : 1, 0);
  for (int32_t i = 0; i < G.B; ++i) {
    const InstInfo& in = G.inst[i];
    if (S.p.global_null) {
      if (i < (int32_t)out.size()) out[i] = in.n * in.T;
    } else {
      for (int32_t s = in.soff; s < in.soff + in.T && s < (int32_t)out.size(); ++s) out[s] = in.n;
    }
  }
  return out;
}

// Mass of every null slice, the bound on every sum its table keys hold: 2m_s
// (Q_MS), the node count n (CPM, whose strengths are 1) or the instance's 2M'
// in units of 1/omega_den (the global model; INT64_MAX past 2^62).
static std::vector<int64_t> null_slice_masses(const Solver& S) {
  const SupraGraph& G = *S.G0;
  std::vector<int64_t> out(S.Tn > 0 ? S.Tn : 1, 0);
  for (int32_t i = 0; i < G.B; ++i) {
    const InstInfo& in = G.inst[i];
    if (S.p.global_null) {
      u128 sum2m = 0;
      for (int32_t s = in.soff; s < in.soff + in.T; ++s) sum2m += (u128)(ull)G.two_m_host[s];
      const u128 m = (u128)(ull)S.od_h[i] * sum2m + (u128)(ull)S.csum_h[i];
      if (i < (int32_t)out.size()) out[i] = m >= ((u128)1 << 62) ? INT64_MAX : (int64_t)m;
    } else {
      for (int32_t s = in.soff; s < in.soff + in.T && s < (int32_t)out.size(); ++s)
        out[s] = S.p.cpm ? in.n : G.two_m_host[s];
    }
  }
  return out;
}

// What the margins of local moving are kept against (see track.cuh), once per
// solve.  A slice's smallest budget is 1/4096 of its mass, or four average
// nodes' strength up to 1/256: a quiet round stays inside it, and it costs a
// settled node little margin (at 1/256 throughout, 2.6% of the nodes of the
// T = 64, n = 100,000 power-law graph were in every round's lists).  Slices of a
// handful of edges get a 1/16, up to 8.
void setup_tracking(Solver& S) {
  Ctx& c = *S.c;
  const SupraGraph& G = *S.G0;
  const std::vector<int64_t> mass = null_slice_masses(S), nodes = null_slice_nodes(S);
  S.track_base_h.resize(mass.size());
  for (size_t s = 0; s < mass.size(); ++s)
    S.track_base_h[s] = std::max<int64_t>({mass[s] >> 12, std::min(mass[s] >> 8, mass[s] / std::max<int64_t>(1, nodes[s] / 4)),
                                           std::min<int64_t>(mass[s] >> 4, 8)});
  S.track_base = c.ws->get<long long>("s_track_base", mass.size());
  check_cuda(cudaMemcpyAsync(S.track_base, S.track_base_h.data(), mass.size() * sizeof(long long),
                             cudaMemcpyHostToDevice, c.stream), "copy");
  S.total_strength = 0;
  for (int32_t i = 0; i < G.B; ++i) {
    const InstInfo& in = G.inst[i];
    double sum2m = 0;
    for (int32_t s = in.soff; s < in.soff + in.T; ++s) sum2m += (double)G.two_m_host[s];
    S.total_strength += (double)S.od_h[i] * sum2m + (double)S.csum_h[i];
  }
}

void configure_stores(Solver& S, int64_t N) {
  Ctx& c = *S.c;
  const int64_t T = S.Tn;
  S.sig = SigStore{};
  S.kr = SigStore{};
  S.sig.T = S.kr.T = (int32_t)T;
  const int64_t need = (N > 0 ? N : 1) * T;
  int64_t limit = DENSE_LIMIT;
  if (const char* e = std::getenv("MSLICE_DENSE_LIMIT")) limit = std::atoll(e);
  if (need <= limit) {
    if (need > S.dense_cap) {
      S.sig_d = c.ws->get<long long>("s_sig_d", need);
      S.kr_d = c.ws->get<long long>("s_kr_d", need);
      S.dense_cap = need;
    }
    S.sig.d = S.sig_d;
    S.kr.d = S.kr_d;
    S.sig.rows = S.kr.rows = (N > 0 ? N : 1);
    return;
  }
  if (S.region_T != T) {
    // hash tables keyed by (label, null slice), one region per null slice
    // sized for its level-0 nodes: at most one live key per (node, slice)
    // entry of that slice plus the keys one round of moves creates; a
    // rebuild is triggered once a region has taken half of its slots
    const std::vector<int64_t> ns = null_slice_nodes(S);
    S.region_h.assign(ns.size() + 1, 0);
    for (size_t s = 0; s < ns.size(); ++s)
      S.region_h[s + 1] = S.region_h[s] + (uint64_t)(2 * ns[s] + 2 * ((ns[s] + S.p.K - 1) / S.p.K) + 64);
    const uint64_t cap = S.region_h.back();
    uint64_t* region = c.ws->get<uint64_t>("s_region", S.region_h.size());
    check_cuda(cudaMemcpyAsync(region, S.region_h.data(), S.region_h.size() * sizeof(uint64_t),
                               cudaMemcpyHostToDevice, c.stream), "copy");
    ull* rused = S.sig_used ? c.ws->get<ull>("s_region_used", ns.size()) : nullptr;
    if (rused) check_cuda(cudaMemsetAsync(rused, 0, ns.size() * sizeof(ull), c.stream), "memset");
    S.sig_h = HashView{c.ws->get<Slot>("s_sig", cap), cap, c.d_status, S.sig_used, region, rused};
    S.kr_h = HashView{c.ws->get<Slot>("s_kr", cap), cap, c.d_status, nullptr, region, nullptr};
    S.region_T = T;
  }
  // 8-byte slots when no null slice's mass reaches 2^32 (no sum can)
  bool narrow = true;
  for (int64_t m : null_slice_masses(S)) narrow = narrow && m < ((int64_t)1 << 32);
  if (const char* e = std::getenv("MSLICE_WIDE_SLOTS")) narrow = narrow && std::atoi(e) == 0;
  S.sig_h.narrow = S.kr_h.narrow = narrow ? 1 : 0;
  S.sig_h.nregions = S.kr_h.nregions = (int32_t)(S.region_h.size() - 1);
  S.sig.h = S.sig_h;
  S.kr.h = S.kr_h;
}

// Empties a store (dense rows zeroed, hash slots freed).
void clear_store(Solver& S, const SigStore& st) {
  Ctx& c = *S.c;
  if (st.d)
    check_cuda(cudaMemsetAsync(st.d, 0, (size_t)st.rows * st.T * sizeof(long long), c.stream), "memset");
  else
    launch(c, k_hash_clear, dim3(fixed_grid(8)), dim3(256), 0, st.h);
}

// Sigma (and, optionally, the community sizes) from the labels.
static void rebuild_sigma(Solver& S, const Level& L, const int32_t* labels, bool sizes) {
  Ctx& c = *S.c;
  const int32_t N = L.d.N;
  if (sizes) check_cuda(cudaMemsetAsync(S.size, 0, (N > 0 ? N : 1) * sizeof(int32_t), c.stream), "memset");
  if (S.sig_used) check_cuda(cudaMemsetAsync(S.sig_used, 0, sizeof(ull), c.stream), "memset");
  if (!S.sig.d && S.sig.h.region_used)
    check_cuda(cudaMemsetAsync(S.sig.h.region_used, 0, (S.region_h.size() - 1) * sizeof(ull), c.stream), "memset");
  clear_store(S, S.sig);
  if (N > 0)
    if (L.d.is0)
      launch(c, k_sigma_insert, dim3(grid_for(N, 256)), dim3(256), 0, L.d, labels, S.sig, sizes ? S.size : nullptr);
    else if (L.ns < 4 * (int64_t)N)  // (lists of one or two entries mostly)
      launch(c, k_sigma_insert_group<4>, dim3(fixed_grid(8)), dim3(256), 0, L.d, labels, S.sig,
             sizes ? S.size : nullptr);
    else
      launch(c, k_sigma_insert_group<32>, dim3(fixed_grid(8)), dim3(256), 0, L.d, labels, S.sig,
             sizes ? S.size : nullptr);
}

void sigma_rebuild(Solver& S, const Level& L, const int32_t* labels) { rebuild_sigma(S, L, labels, false); }

TierSegs bucket_segments(Solver& S, int q) {
  TierSegs sg;
  for (int t = 0; t < NTIERS; ++t) {
    sg.list[t] = S.lists + (int64_t)q * S.N0 + S.tier_off[t];
    sg.count[t] = S.cursors + NTIERS * q + t;
  }
  sg.queue = S.wqueue;
  return sg;
}

static void bucket_tracked(Solver& S, const Level& L, uint64_t tag, int it, int lvl, int r, const int32_t* active,
                           const TrackView& trk) {
  Ctx& c = *S.c;
  const TierOff to = tier_offsets(S);
  const int64_t N = L.d.N;
  if (N == 0) {
    check_cuda(cudaMemsetAsync(S.cursors, 0, NTIERS * S.p.K * sizeof(int32_t), c.stream), "memset");
    return;
  }
  const int64_t nchunks = (N + BUCKET_CHUNK - 1) / BUCKET_CHUNK;
  const unsigned grid = (unsigned)std::min<int64_t>(nchunks, fixed_grid(16));
  launch(c, k_bucket_count, dim3(grid), dim3(BUCKET_THREADS), 0, L.d, (const uint8_t*)S.tier, S.p.seed, tag,
         (uint64_t)it, (uint64_t)lvl, (uint64_t)r, S.p.K, active, trk, S.bseg, S.bcounts, nchunks);
  launch(c, k_bucket_scan, dim3(S.p.K * NTIERS), dim3(1024), 0, S.bcounts, nchunks, S.cursors);
  launch(c, k_bucket_write, dim3(grid), dim3(BUCKET_THREADS), 0, L.d.N, (const uint16_t*)S.bseg,
         (const int32_t*)S.bcounts, nchunks, S.p.K, S.lists, (int64_t)S.N0, to);
}

void bucket(Solver& S, const Level& L, uint64_t tag, int it, int lvl, int r, const int32_t* active) {
  bucket_tracked(S, L, tag, it, lvl, r, active, TrackView{});
}

int64_t count_communities(Solver& S, int64_t N) {
  Ctx& c = *S.c;
  if (N == 0) return 0;
  ull* d = c.ws->get<ull>("cd_tot", 1);
  check_cuda(cudaMemsetAsync(d, 0, sizeof(ull), c.stream), "memset");
  launch(c, k_count_sizes, dim3(std::min(grid_for(N, 1024), fixed_grid(4))), dim3(256), 0, (const int32_t*)S.size, N, d);
  return (int64_t)*static_cast<const ull*>(readback(c, d, sizeof(ull)));
}

// The tracking state of a level (see track.cuh).  Margins live in a
// refinement array, which is only read after local moving.  Their unit is set
// so that a node of average strength has about 2^20 of them.
static TrackView track_view(Solver& S, const Level& L) {
  Ctx& c = *S.c;
  TrackView t;
  t.state = c.ws->get<int32_t>("s_track_state", 2 * TRACK_WORDS);
  t.slack = S.Wsel;
  t.E = c.ws->get<long long>("s_track_E", 2 * (size_t)S.Tn);
  t.B = c.ws->get<long long>("s_track_B", 2 * (size_t)S.Tn);
  t.base = S.track_base;
  t.lam = S.lam;
  const double avg = S.total_strength / (double)(L.d.N > 0 ? L.d.N : 1);
  int bits = 0;
  while (bits < 60 && avg > (double)(1ll << bits)) ++bits;
  t.F = std::max(-40, std::min(16, 20 - bits));
  t.scale = std::ldexp(1.0, t.F - 63);
  return t;
}

// Chooses the degree cuts of the decision tiers for this solve: every
// candidate decides the K sub-rounds of round r twice (decisions only,
// nothing is applied, so the state is untouched) and the candidate with the
// fastest pass is kept.  Decisions do not depend on the tier that makes
// them, so neither does the result.
template <class Decide>
static void autotune_cuts(Solver& S, const Level& L, int it, int r, const int32_t* active, Decide&& decide) {
  Ctx& c = *S.c;
  // (cut 2 in units of the tier-2 capacity: T2 = TIER_MAX[2])
  constexpr int T2 = TIER_MAX[2];
  static const TierCuts kCand[] = {{{16, 32, T2, 1024}}, {{12, 32, T2, 1024}}, {{16, 24, T2, 1024}},
                                   {{16, 32, T2, 512}},  {{12, 24, T2, 512}},  {{16, 32, T2 * 3 / 4, 1024}}};
  cudaEvent_t e0, e1;
  check_cuda(cudaEventCreate(&e0), "event");
  check_cuda(cudaEventCreate(&e1), "event");
  float best = 0;
  TierCuts chosen = kCand[0];
  // the first pass warms the caches and is not counted
  for (int k = -1; k < (int)(sizeof(kCand) / sizeof(kCand[0])); ++k) {
    S.p.cuts = kCand[k < 0 ? 0 : k];
    prepare_level(S, L);
    bucket(S, L, 0, it, 0, r, active);
    float ms = 0;
    for (int rep = 0; rep < 2; ++rep) {
      check_cuda(cudaEventRecord(e0, c.stream), "event");
      for (int q = 0; q < S.p.K; ++q) decide(bucket_segments(S, q));
      check_cuda(cudaEventRecord(e1, c.stream), "event");
      check_cuda(cudaEventSynchronize(e1), "event");
      float x = 0;
      check_cuda(cudaEventElapsedTime(&x, e0, e1), "event time");
      ms = rep == 0 ? x : std::min(ms, x);
    }
    if (k >= 0 && (k == 0 || ms < best)) {
      best = ms;
      chosen = kCand[k];
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  S.p.cuts = chosen;
  S.p.autotune = false;
  prepare_level(S, L);
  fill_i32(c, S.target, NO_MOVE, L.d.N);
}

MoveOut local_move(Solver& S, const Level& L, int32_t* labels, int it, int lvl, int max_rounds) {
  Ctx& c = *S.c;
  MoveOut out;
  const int32_t N = L.d.N;
  if (N == 0) {
    // an empty level runs one round that moves nothing
    if (max_rounds > 0) {
      out.rounds = 1;
      S.lm_rounds++;
    }
    return out;
  }
  const bool tuning = S.p.autotune && lvl == 0;
  // Rounds are resident (lm_rounds.cu) while they have at most
  // RESIDENT_MAX_WORK to decide, by the level's average degree:
  // every round of a level that small, and the others once a pruned round has
  // listed few enough nodes.  Not while the level-0 decisions are being timed
  // or the tier cuts tuned.
  const bool may_reside = !tuning && !(c.profile && lvl == 0);
  const long long few = resident_work(RESIDENT_MAX_WORK) / (L.nnz / N + RESIDENT_NODE_WORK);
  // community sizes and Sigma of the level's initial labels (refinement
  // reads Sigma even when no round runs), unless the first resident launch
  // builds them
  bool build = max_rounds > 0 && may_reside && N <= few && S.sig.d && S.sig.rows * S.sig.T <= RESIDENT_BUILD_MAX;
  if (!build) rebuild_sigma(S, L, labels, true);
  if (max_rounds <= 0) return out;
  // Margins are recorded once few nodes move: from the level's first round,
  // except where the level starts from singletons (its first rounds move most
  // nodes), and not on a level whose tier cuts are still being tuned.
  // (MSLICE_TRACK_MIN_ENTRIES: tracks every level of that many entries)
  const char* track_min = std::getenv("MSLICE_TRACK_MIN_ENTRIES");
  const bool worth = track_min ? L.nnz >= std::atoll(track_min)
                               : (L.nnz >= TRACK_MIN_ENTRIES && L.nnz >= TRACK_MIN_DEGREE * (int64_t)N &&
                                  L.ns <= 4 * (int64_t)N) ||
                                     (L.ns >= 2 * (int64_t)N && L.nnz + L.nnz / N * L.ns >= TRACK_MIN_LOOKUPS);
  const TrackView trk = !worth || tuning ? TrackView{} : track_view(S, L);
  int& fails = S.track_fails[lvl > 0];
  const TrackStart start = track_start(lvl == 0 && it == 0 && !S.warm, fails);
  if (trk.state)
    check_cuda(cudaMemsetAsync(trk.state, 0, 2 * TRACK_WORDS * sizeof(int32_t), c.stream), "memset");
  // Batch: an instance whose round moved nothing is at a fixed point of
  // this level (its decisions read only its own state, which no longer
  // changes), so it is left out of the remaining rounds.
  const bool batch = S.B > 1;
  if (batch)
    check_cuda(cudaMemcpyAsync(S.lm_active, S.inst_active, S.B * sizeof(int32_t), cudaMemcpyDeviceToDevice, c.stream),
               "copy");
  const int32_t* active = batch ? S.lm_active : S.inst_active;
  const int nseg = S.p.K * NTIERS;
  auto decide = [&](const TierSegs& sg, const TrackView& t) {
    if (S.sig.d && L.d.is0)
      decide_all(c, lm_policy<true, true>(S, L, labels, t), sg, S.tier_cnt, S.gkeys, S.gvals, S.goff);
    else if (S.sig.d)
      decide_all(c, lm_policy<true>(S, L, labels, t), sg, S.tier_cnt, S.gkeys, S.gvals, S.goff);
    else if (L.d.is0)
      decide_all(c, lm_policy<false, true>(S, L, labels, t), sg, S.tier_cnt, S.gkeys, S.gvals, S.goff);
    else
      decide_all(c, lm_policy<false>(S, L, labels, t), sg, S.tier_cnt, S.gkeys, S.gvals, S.goff);
  };
  long long moved = 0, listed = N;  // of the last round
  bool first_round = true, rebuild = false;
  int32_t state[TRACK_WORDS] = {};  // tracking words of the last round
  int r = 0;
  while (r < max_rounds) {
    if (rebuild) rebuild_sigma(S, L, labels, false);
    if (may_reside && listed <= few) {
      ResidentIn in;
      in.r = r;
      in.r_end = max_rounds;
      in.first = first_round;
      in.build = build;
      build = false;
      in.start = start;
      in.prev_moved = moved;
      in.prev_listed = listed;
      in.max_listed = 2 * few;  // (some slack, so that rounds do not change hands to and fro)
      ResidentOut ro;
      resident_rounds(S, L, labels, it, lvl, trk, in, active, ro);
      S.lm_rounds += ro.rounds;
      S.lm_edges += ro.rounds * L.nnz_eff;
      out.rounds += ro.rounds;
      out.moves += ro.moves;
      r += (int)ro.rounds;
      first_round = false;
      if (ro.status) check_status(c, "local moving");
      if (ro.rounds < 1) fail(MSLICE_ECUDA, "resident rounds ran no round");
      moved = ro.last_moved;
      listed = ro.last_listed;
      out.communities = ro.communities;
      std::memcpy(state, ro.state, sizeof(state));
      rebuild = !S.sig.d && ro.used > 0;
      if (moved == 0) break;
      if (r >= max_rounds) out.capped = true;
      continue;
    }
    // tuning waits for round 2, when the partition looks like the later rounds'
    if (S.p.autotune && lvl == 0 && r == 2)
      autotune_cuts(S, L, it, r, active, [&](const TierSegs& sg) { decide(sg, TrackView{}); });
    S.lm_rounds++;
    S.lm_edges += L.nnz_eff;
    out.communities = -1;
    const bool prof = c.profile && lvl == 0;
    const size_t spans = prof ? c.prof_spans->size() : 0;
    if (prof) c.prof_bytes += 12 * L.nnz_eff + 40 * (int64_t)N;
    // One round: buckets, K sub-rounds of decisions, applies and moves to
    // empty communities; its moves, the table fill, the status word, the list
    // lengths and the tracking mode go to the pinned buffer.
    const TrackView tr = track_at(trk, S.Tn, r);
    // (the mode k_round_begin comes to, from the same words)
    const bool tracked = tr.state && track_next(state, first_round, start, moved, listed).mode != TRACK_OFF;
    const BucketLists bl{S.lists, (int64_t)S.N0, S.cursors, tier_offsets(S), S.bseg};
    if (tr.state)
      launch(c, k_round_begin, dim3(1), dim3(512), 0, tr, track_at(trk, S.Tn, r + 1).state, S.Tn, (int)first_round,
             start, moved, listed, S.counters);
    else
      check_cuda(cudaMemsetAsync(S.counters, 0, 3 * sizeof(int32_t), c.stream), "memset");
    bucket_tracked(S, L, 0, it, lvl, r, active, tr);
    for (int q = 0; q < S.p.K; ++q) {
      const TierSegs sg = bucket_segments(S, q);
      if (prof) {
        cudaEvent_t e0, e1;
        check_cuda(cudaEventCreate(&e0), "event");
        check_cuda(cudaEventCreate(&e1), "event");
        check_cuda(cudaEventRecord(e0, c.stream), "event");
        decide(sg, tr);
        check_cuda(cudaEventRecord(e1, c.stream), "event");
        c.prof_spans->push_back({e0, e1});
      } else {
        decide(sg, tr);
      }
      launch(c, tracked ? k_lm_apply<true> : k_lm_apply<false>, dim3(fixed_grid(4)), dim3(APPLY_THREADS), 0, L.d, sg, labels, S.size, S.sig, S.target,
             S.counters, batch ? S.inst_moved : nullptr, tr, bl, q);
      // (all of the co-resident grid, unless other solves share the SMs)
      const int32_t share = coop_share(S.sms);
      launch_coop(c, k_empty_pass, dim3(share < S.sms ? std::min(share, S.empty_grid) : S.empty_grid), dim3(EMPTY_THREADS), 0, L.d, S.B, S.target, labels, S.size,
                  S.sig, S.counters, S.empty_blk, S.freelist, S.tmp32b, S.inst_cnt, tr, bl, q + 1);
    }
    if (batch)
      launch(c, k_round_freeze, dim3(grid_for(S.B, 256)), dim3(256), 0, S.lm_active, S.inst_moved, S.B);
    char* h = static_cast<char*>(c.pinned);
    struct {
      int64_t moved;
      ull used;
      unsigned status;
      int32_t pad_;
      int32_t state[TRACK_WORDS];
    } rb{};
    std::memcpy(h, &rb, sizeof(rb));
    check_cuda(cudaMemcpyAsync(h, S.counters, sizeof(int64_t), cudaMemcpyDeviceToHost, c.stream), "copy");
    check_cuda(cudaMemcpyAsync(h + 8, S.sig_used, sizeof(ull), cudaMemcpyDeviceToHost, c.stream), "copy");
    check_cuda(cudaMemcpyAsync(h + 16, c.d_status, sizeof(unsigned), cudaMemcpyDeviceToHost, c.stream), "copy");
    if (tr.state) {
      check_cuda(cudaMemcpyAsync(h + 24, tr.state, sizeof(rb.state), cudaMemcpyDeviceToHost, c.stream), "copy");
      check_cuda(cudaMemcpyAsync(h + sizeof(rb), S.cursors, nseg * sizeof(int32_t), cudaMemcpyDeviceToHost, c.stream), "copy");
    }
    sync(c);
    std::memcpy(&rb, h, sizeof(rb));
    if (rb.status) check_status(c, "local moving");
    rebuild = !S.sig.d && rb.used > 0;  // a region has taken half of its slots
    moved = rb.moved;
    listed = N;
    if (tr.state) {
      std::memcpy(state, rb.state, sizeof(state));
      const int32_t* cur = reinterpret_cast<const int32_t*>(h + sizeof(rb));
      listed = 0;
      for (int i = 0; i < nseg; ++i) listed += cur[i];
    }
    if (prof && tr.state && rb.state[TRACK_MODE] == TRACK_PRUNE) {
      // the decision timing covers the rounds in which every node decides
      for (size_t k = spans; k < c.prof_spans->size(); ++k) {
        cudaEventDestroy((*c.prof_spans)[k].first);
        cudaEventDestroy((*c.prof_spans)[k].second);
      }
      c.prof_spans->resize(spans);
      c.prof_bytes -= 12 * L.nnz_eff + 40 * (int64_t)N;
    }
    first_round = false;
    out.rounds++;
    out.moves += moved;
    ++r;
    if (moved == 0) break;
    if (r == max_rounds) out.capped = true;
  }
  S.lm_moves += out.moves;
  if (trk.state) fails = track_fails(fails, start, state, listed);
  return out;
}

}  // namespace mslice
