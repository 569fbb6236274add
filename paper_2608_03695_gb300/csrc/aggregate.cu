// Aggregation (Louvain/Leiden, Sec. 3.2): one node per refined
// sub-community, numbered by ascending sub-community label.  Contraction
// without a sort: the level's nodes are bucketed by new id (member lists),
// then one warp or block per new node walks its members' rows and sums the
// weights per neighbouring new node in a shared-memory table; rows with more
// than 4096 entries use tables in global scratch and are spread over the
// whole grid.  Self-loops are dropped: no key or check reads them, and Q is
// always evaluated on level 0.  The same pass sums the members' snapshot
// strengths k_{x,s}.  Rows are written once to an upper-bound layout and
// compacted.  The order of a row's entries is not defined; nothing that
// reads a level depends on it (sums are exact integers and every scan is
// order-free).  The initial label of a new node is the smallest new id
// inside its local-moving community.
#include <algorithm>
#include <cstring>

#include "../../include/mslice.h"
#include "resident.cuh"

namespace mslice {

namespace {

__global__ void k_present(const int32_t* sizeR, int32_t N, int32_t* flag) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
    flag[i] = sizeR[i] > 0 ? 1 : 0;
}

constexpr int CW_BITS = 9;        // warp tier: rows with at most 256 entries / snapshot entries
constexpr int CW_WARPS = 8;
constexpr int CB_BITS = 13;       // block tier: at most 4096
constexpr int CB_THREADS = 512;
constexpr int CW_MAX = 1 << (CW_BITS - 1), CB_MAX = 1 << (CB_BITS - 1);

// Per node: its new id; per new node: members, stored entries and snapshot
// entries (upper bounds of its output).
__global__ void k_contract_prep(LevelDev g, const int32_t* R, const int32_t* newid, int32_t* xmap, int32_t* mcnt,
                                long long* dsum, int32_t* scnt) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < g.N; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t x = newid[R[v]];
    xmap[v] = x;
    atomicAdd(&mcnt[x], 1);
    atomicAdd((ull*)&dsum[x], (ull)(g.rowptr[v + 1] - g.rowptr[v]));
    int64_t b, e;
    slice_range(g, (int32_t)v, b, e);
    if (e > b) atomicAdd(&scnt[x], (int32_t)(e - b));
  }
}

__global__ void k_contract_members(int32_t N, const int32_t* xmap, const int64_t* moff, int32_t* mfill, int32_t* mem) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t x = xmap[v];
    mem[moff[x] + atomicAdd(&mfill[x], 1)] = (int32_t)v;
  }
}

// Slots of a big row's global table for n entries: every entry could be a
// distinct key, so twice n keeps the load at most one half (short probe
// sequences; the power of two above 2n used before took up to twice this).
__device__ __forceinline__ int64_t big_table_slots(int64_t n) { return 2 * n + 16; }

// Rows by size: tier 0 (<= CW_MAX), 1 (<= CB_MAX), 2 (larger; its tables of
// big_table_slots(size) slots in global scratch).
__global__ void k_contract_tier(int32_t Np, const long long* dsum, const int32_t* scnt, int32_t* lists,
                                int32_t* tcnt, int64_t* gsize, int64_t* ssize) {
  const int lane = threadIdx.x & 31;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < Np; base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t x = base + threadIdx.x;
    int t = -1;
    if (x < Np) {
      const long long need = max(dsum[x], (long long)scnt[x]);
      t = need <= CW_MAX ? 0 : (need <= CB_MAX ? 1 : 2);
      gsize[x] = t == 2 ? big_table_slots(dsum[x]) : 0;
      ssize[x] = t == 2 ? big_table_slots(scnt[x]) : 0;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, t);
    const int leader = __ffs(peers) - 1;
    int pos = 0;
    if (t >= 0 && lane == leader) pos = atomicAdd(&tcnt[t], __popc(peers));
    pos = __shfl_sync(peers, pos, leader);
    if (t >= 0) lists[(int64_t)t * Np + pos + __popc(peers & ((1u << lane) - 1u))] = (int32_t)x;
  }
}

// Insert-or-add into a shared table of `cap` (a power of two) slots.
__device__ __forceinline__ int64_t ctab_add(int32_t* hk, long long* hv, int64_t cap, int32_t key, long long w,
                                            bool& fresh) {
  const uint64_t mask = (uint64_t)cap - 1;
  const int bits = 63 - __clzll((long long)cap);
  uint64_t i = ((uint64_t)(uint32_t)key * 0x9E3779B97F4A7C15ull) >> (64 - bits);
  for (uint64_t p = 0; p <= mask; ++p) {
    const int32_t prev = atomicCAS(&hk[i], -1, key);
    if (prev == -1 || prev == key) {
      shared_add64(&hv[i], w);
      fresh = prev == -1;
      return (int64_t)i;
    }
    i = (i + 1) & mask;
  }
  fresh = false;
  return -1;
}

// Insert-or-add into a global table of `cap` slots (any size): home by a
// multiplicative hash and a multiply-high range reduction, linear probing.
__device__ __forceinline__ int64_t gtab_add(int32_t* hk, long long* hv, int64_t cap, int32_t key, long long w,
                                            bool& fresh) {
  uint64_t i = __umul64hi((uint64_t)(uint32_t)key * 0x9E3779B97F4A7C15ull, (uint64_t)cap);
  for (int64_t p = 0; p < cap; ++p) {
    const int32_t prev = atomicCAS(&hk[i], -1, key);
    if (prev == -1 || prev == key) {
      atomicAdd((ull*)&hv[i], (ull)w);
      fresh = prev == -1;
      return (int64_t)i;
    }
    i = (i + 1 == (uint64_t)cap) ? 0 : i + 1;
  }
  fresh = false;
  return -1;
}

// One row by a warp (at most CW_MAX stored and snapshot entries).  Members are
// fetched 32 at a time with their row bounds; lanes stride over each member's
// entries.  K, V (2^CW_BITS slots), CL and *ncl: the warp's shared table, free on
// entry and left free.
struct RowOut {
  const int64_t *eoff, *soff;  // the rows' places in the upper-bound layout
  int32_t* tcol;
  long long* tw;
  int32_t* ecnt;
  int32_t* tsidx;
  long long* tsval;
  int32_t* scnt;
};

__device__ __forceinline__ void contract_row_warp(const LevelDev& g, const int32_t* xmap, const int64_t* moff,
                                                  const int32_t* mem, int32_t x, int32_t* K, long long* V,
                                                  uint16_t* CL, int32_t* ncl, const RowOut& o) {
  constexpr int SLOTS = 1 << CW_BITS;
  const int lane = threadIdx.x & 31;
  const int64_t mb = moff[x], me = moff[x + 1];
  int n = 0;
  for (int64_t j0 = mb; j0 < me; j0 += 32) {
    const int64_t jj = j0 + lane;
    int32_t mv = 0;
    int64_t rb = 0, re = 0;
    if (jj < me) {
      mv = mem[jj];
      rb = g.rowptr[mv];
      re = g.rowptr[mv + 1];
    }
    const int cm = (int)min((int64_t)32, me - j0);
    for (int t = 0; t < cm; ++t) {
      const int32_t v = __shfl_sync(0xffffffffu, mv, t);
      const int64_t b = __shfl_sync(0xffffffffu, rb, t), e = __shfl_sync(0xffffffffu, re, t);
      const Omega om = node_omega(g, v);
      for (int64_t base = b; base < e; base += 32) {
        const int64_t i = base + lane;
        bool fresh = false;
        int64_t slot = 0;
        if (i < e) {
          int32_t u;
          long long W;
          if (edge_at(g, i, u, W, om)) {
            const int32_t y = xmap[u];
            if (y != x) slot = ctab_add(K, V, SLOTS, y, W, fresh);
#if MSLICE_CHECKED
            if (y != x && slot < 0) atomicOr(g.chk, ERR_BOUNDS);
#endif
          }
        }
        const unsigned bal = __ballot_sync(0xffffffffu, fresh);
        if (fresh) CL[n + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)slot;
        n += __popc(bal);
      }
    }
  }
  __syncwarp();
  const int64_t eo = o.eoff[x];
  for (int k = lane; k < n; k += 32) {
    const int slot = CL[k];
    o.tcol[eo + k] = K[slot];
    o.tw[eo + k] = V[slot];
    K[slot] = -1;
    V[slot] = 0;
  }
  if (lane == 0) o.ecnt[x] = n;
  __syncwarp();
  // snapshot strengths: lane per member
  for (int64_t j = mb + lane; j < me; j += 32) {
    const int32_t v = mem[j];
    int64_t b, e;
    slice_range(g, v, b, e);
    for (int64_t q = b; q < e; ++q) {
      int32_t sl;
      long long k;
      slice_entry(g, v, q, sl, k);
      bool fresh;
      const int64_t slot = ctab_add(K, V, SLOTS, sl, k, fresh);
#if MSLICE_CHECKED
          if (slot < 0) atomicOr(g.chk, ERR_BOUNDS);
#endif
      if (fresh) CL[atomicAdd(ncl, 1)] = (uint16_t)slot;
    }
  }
  __syncwarp();
  const int ns = *ncl;
  const int64_t so = o.soff[x];
  for (int k = lane; k < ns; k += 32) {
    const int slot = CL[k];
    o.tsidx[so + k] = K[slot];
    o.tsval[so + k] = V[slot];
    K[slot] = -1;
    V[slot] = 0;
  }
  __syncwarp();
  if (lane == 0) {
    o.scnt[x] = ns;
    *ncl = 0;
  }
  __syncwarp();
}

// One warp per new node x (tier 0).
__global__ void __launch_bounds__(CW_WARPS * 32)
    k_contract_warp(LevelDev g, const int32_t* xmap, const int64_t* moff, const int32_t* mem, const int32_t* list,
                    const int32_t* count_ptr, const int64_t* eoff, const int64_t* soff, int32_t* tcol, long long* tw,
                    int32_t* ecnt, int32_t* tsidx, long long* tsval, int32_t* scnt_out) {
  constexpr int SLOTS = 1 << CW_BITS;
  __shared__ int32_t hk[CW_WARPS][SLOTS];
  __shared__ long long hv[CW_WARPS][SLOTS];
  __shared__ uint16_t cl[CW_WARPS][SLOTS / 2];
  __shared__ int32_t ncl[CW_WARPS];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t* K = hk[w];
  long long* V = hv[w];
  uint16_t* CL = cl[w];
  for (int i = lane; i < SLOTS; i += 32) {
    K[i] = -1;
    V[i] = 0;
  }
  if (lane == 0) ncl[w] = 0;
  __syncwarp();
  const int count = *count_ptr;
  const int64_t warps = (int64_t)gridDim.x * CW_WARPS;
  for (int64_t idx = (int64_t)blockIdx.x * CW_WARPS + w; idx < count; idx += warps) {
    contract_row_warp(g, xmap, moff, mem, list[idx], K, V, CL, &ncl[w],
                      RowOut{eoff, soff, tcol, tw, ecnt, tsidx, tsval, scnt_out});
  }
}

// One block per new node x of tier 1: a table of 2^CB_BITS slots in shared
// memory.  Warps take members in turn; lanes stride over entries.  Blocks
// claim their rows one at a time from a counter (queue), which keeps them
// busy until the list is done whatever the spread of row sizes.
__global__ void __launch_bounds__(CB_THREADS)
    k_contract_block(LevelDev g, const int32_t* xmap, const int64_t* moff, const int32_t* mem, const int32_t* list,
                     const int32_t* count_ptr, const int64_t* eoff, const int64_t* soff, int32_t* tcol, long long* tw,
                     int32_t* ecnt, int32_t* tsidx, long long* tsval, int32_t* scnt_out, int32_t* queue) {
  extern __shared__ __align__(16) unsigned char csm[];
  __shared__ int32_t ncnt;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr int NW = CB_THREADS / 32;
  const int count = *count_ptr;
  constexpr int64_t cap = (int64_t)1 << CB_BITS;
  long long* V = reinterpret_cast<long long*>(csm);
  int32_t* K = reinterpret_cast<int32_t*>(V + cap);
  uint32_t* CL = reinterpret_cast<uint32_t*>(K + cap);  // listed slots
  for (int64_t i = threadIdx.x; i < cap; i += blockDim.x) {
    K[i] = -1;
    V[i] = 0;
  }
  __shared__ int32_t claim;
  if (threadIdx.x == 0) claim = -1;
  for (int idx; (idx = block_claim(queue, count, &claim)) >= 0;) {
    const int32_t x = list[idx];
    if (threadIdx.x == 0) ncnt = 0;
    __syncthreads();
    const int64_t mb = moff[x], me = moff[x + 1];
    for (int64_t j = mb + w; j < me; j += NW) {
      const int32_t v = mem[j];
      const int64_t b = g.rowptr[v], e = g.rowptr[v + 1];
      const Omega om = node_omega(g, v);
      for (int64_t i = b + lane; i < e; i += 32) {
        int32_t u;
        long long W;
        if (edge_at(g, i, u, W, om)) {
          const int32_t y = xmap[u];
          if (y != x) {
            bool fresh;
            const int64_t slot = ctab_add(K, V, cap, y, W, fresh);
#if MSLICE_CHECKED
            if (slot < 0) atomicOr(g.chk, ERR_BOUNDS);
#endif
            if (fresh) CL[atomicAdd(&ncnt, 1)] = (uint32_t)slot;
          }
        }
      }
    }
    __syncthreads();
    const int n = ncnt;
    const int64_t eo = eoff[x];
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const uint32_t slot = CL[k];
      tcol[eo + k] = K[slot];
      tw[eo + k] = V[slot];
      K[slot] = -1;
      V[slot] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      ecnt[x] = n;
      ncnt = 0;
    }
    __syncthreads();
    for (int64_t j = mb + threadIdx.x; j < me; j += blockDim.x) {
      const int32_t v = mem[j];
      int64_t b, e;
      slice_range(g, v, b, e);
      for (int64_t q = b; q < e; ++q) {
        int32_t sl;
        long long k;
        slice_entry(g, v, q, sl, k);
        bool fresh;
        const int64_t slot = ctab_add(K, V, cap, sl, k, fresh);
#if MSLICE_CHECKED
            if (slot < 0) atomicOr(g.chk, ERR_BOUNDS);
#endif
        if (fresh) CL[atomicAdd(&ncnt, 1)] = (uint32_t)slot;
      }
    }
    __syncthreads();
    const int ns = ncnt;
    const int64_t so = soff[x];
    for (int k = threadIdx.x; k < ns; k += blockDim.x) {
      const uint32_t slot = CL[k];
      tsidx[so + k] = K[slot];
      tsval[so + k] = V[slot];
      K[slot] = -1;
      V[slot] = 0;
    }
    if (threadIdx.x == 0) scnt_out[x] = ns;
    __syncthreads();
  }
}

// Tier 2 (rows of more than CB_MAX entries) is spread over the whole grid:
// warps take the members of all such rows in turn and insert into the row's
// tables in global scratch (edges and snapshot strengths in separate tables,
// pre-filled with free slots), listing claimed slots with per-row counters;
// a second kernel writes each row out.  big: the tier's rows; mpre: prefix of
// their member counts (nbig + 1 entries).
__global__ void k_big_members(const int32_t* big, const int32_t* nbig_ptr, const int64_t* moff, int64_t* cnt) {
  const int nbig = *nbig_ptr;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nbig; i += (int64_t)gridDim.x * blockDim.x)
    cnt[i] = moff[big[i] + 1] - moff[big[i]];
}

// Members of tier-2 rows are taken BI_CHUNK at a time by a block, which sums
// their entries per target in shared memory first (the members of one coarse
// community mostly reach the same few others, so adding every entry straight
// into the global table serialised on a few slots) and then adds each
// distinct target once to the row's global table.  An entry whose probe in
// the shared table runs past BI_PROBES slots goes to the global table
// directly; sums are integers, so the split changes nothing.
constexpr int BI_BITS = 11, BI_SBITS = 8, BI_CHUNK = 64, BI_PROBES = 16;
constexpr size_t BI_SMEM = ((size_t)1 << BI_BITS) * (sizeof(int32_t) + sizeof(long long) + sizeof(uint16_t)) +
                           ((size_t)1 << BI_SBITS) * (sizeof(int32_t) + sizeof(long long) + sizeof(uint16_t));

// Insert-or-add into a shared table of 2^bits slots, listing a newly taken
// slot in L (n: its length); false when the probe limit is reached (nothing
// added).
__device__ __forceinline__ bool stab_add(int32_t* K, long long* V, uint16_t* L, int* n, int bits, int32_t key,
                                         long long w) {
  const unsigned mask = (1u << bits) - 1u;
  unsigned i = ((uint32_t)key * 0x9E3779B1u) >> (32 - bits);
  for (int p = 0; p < BI_PROBES; ++p) {
    const int32_t prev = atomicCAS(&K[i], -1, key);
    if (prev == -1 || prev == key) {
      shared_add64(&V[i], w);
      if (prev == -1) L[atomicAdd(n, 1)] = (uint16_t)i;
      return true;
    }
    i = (i + 1) & mask;
  }
  return false;
}

__device__ __forceinline__ void big_add(int32_t* hk, long long* hv, uint32_t* hl, int64_t o, int64_t cap,
                                        int32_t* cnt, int32_t key, long long w, const LevelDev& g) {
  bool fresh;
  const int64_t slot = gtab_add(hk + o, hv + o, cap, key, w, fresh);
#if MSLICE_CHECKED
  if (slot < 0) atomicOr(g.chk, ERR_BOUNDS);
#endif
  if (fresh) hl[o + atomicAdd(cnt, 1)] = (uint32_t)slot;
}

__global__ void __launch_bounds__(256)
    k_big_insert(LevelDev g, const int32_t* xmap, const int64_t* moff, const int32_t* mem, const int32_t* big,
                 const int32_t* nbig_ptr, const int64_t* mpre, const int64_t* gofs, const int64_t* gsize, int32_t* gk,
                 long long* gv, uint32_t* gl, int32_t* gcnt, const int64_t* sofs, const int64_t* ssize, int32_t* sk,
                 long long* sv, uint32_t* sl, int32_t* scnt) {
  extern __shared__ __align__(16) unsigned char bi_smem[];
  constexpr int EB = 1 << BI_BITS, SB = 1 << BI_SBITS;
  long long* EV = reinterpret_cast<long long*>(bi_smem);
  long long* SV = EV + EB;
  int32_t* EK = reinterpret_cast<int32_t*>(SV + SB);
  int32_t* SK = EK + EB;
  uint16_t* EL = reinterpret_cast<uint16_t*>(SK + SB);
  uint16_t* SL = EL + EB;
  __shared__ int row_sh, ne, ns;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  for (int i = threadIdx.x; i < EB; i += blockDim.x) {
    EK[i] = -1;
    EV[i] = 0;
  }
  for (int i = threadIdx.x; i < SB; i += blockDim.x) {
    SK[i] = -1;
    SV[i] = 0;
  }
  if (threadIdx.x == 0) ne = ns = 0;
  const int nbig = *nbig_ptr;
  const int64_t total = mpre[nbig];
  const int64_t chunks = (total + BI_CHUNK - 1) / BI_CHUNK;
  for (int64_t ch = blockIdx.x; ch < chunks; ch += gridDim.x) {
    const int64_t f0 = ch * BI_CHUNK, f1 = f0 + BI_CHUNK < total ? f0 + BI_CHUNK : total;
    if (threadIdx.x == 0) {
      int lo = 0, hi = nbig - 1;  // the big row holding member f0
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (mpre[mid] <= f0) lo = mid; else hi = mid - 1;
      }
      row_sh = lo;
    }
    __syncthreads();
    // the rows overlapping [f0, f1), one at a time (block-uniform)
    for (int lo = row_sh; lo < nbig && mpre[lo] < f1; ++lo) {
      const int64_t a = mpre[lo] > f0 ? mpre[lo] : f0, b = mpre[lo + 1] < f1 ? mpre[lo + 1] : f1;
      const int32_t x = big[lo];
      const int64_t o = gofs[x], cap = gsize[x], so = sofs[x], scap = ssize[x];
      for (int64_t f = a + warp; f < b; f += nwarps) {
        const int32_t v = mem[moff[x] + (f - mpre[lo])];
        const Omega om = node_omega(g, v);
        for (int64_t i = g.rowptr[v] + lane; i < g.rowptr[v + 1]; i += 32) {
          int32_t u;
          long long W;
          if (edge_at(g, i, u, W, om)) {
            const int32_t y = xmap[u];
            if (y != x && !stab_add(EK, EV, EL, &ne, BI_BITS, y, W)) big_add(gk, gv, gl, o, cap, &gcnt[lo], y, W, g);
          }
        }
        int64_t sb, se;
        slice_range(g, v, sb, se);
        for (int64_t q = sb + lane; q < se; q += 32) {
          int32_t s;
          long long k;
          slice_entry(g, v, q, s, k);
          if (!stab_add(SK, SV, SL, &ns, BI_SBITS, s, k)) big_add(sk, sv, sl, so, scap, &scnt[lo], s, k, g);
        }
      }
      __syncthreads();
      const int me = ne, ms = ns;
      __syncthreads();  // every thread has the counts before they are reset
      if (threadIdx.x == 0) ne = ns = 0;
      for (int j = threadIdx.x; j < me; j += blockDim.x) {
        const int i = EL[j];
        big_add(gk, gv, gl, o, cap, &gcnt[lo], EK[i], EV[i], g);
        EK[i] = -1;
        EV[i] = 0;
      }
      for (int j = threadIdx.x; j < ms; j += blockDim.x) {
        const int i = SL[j];
        big_add(sk, sv, sl, so, scap, &scnt[lo], SK[i], SV[i], g);
        SK[i] = -1;
        SV[i] = 0;
      }
      __syncthreads();
    }
  }
}

__global__ void k_big_output(const int32_t* big, const int32_t* nbig_ptr, const int64_t* gofs, const int32_t* gk,
                             const long long* gv, const uint32_t* gl, const int32_t* gcnt, const int64_t* sofs,
                             const int32_t* sk,
                             const long long* sv, const uint32_t* sl, const int32_t* scnt, const int64_t* eoff,
                             const int64_t* soff, int32_t* tcol, long long* tw, int32_t* ecnt, int32_t* tsidx,
                             long long* tsval, int32_t* scnt_out) {
  const int nbig = *nbig_ptr;
  for (int i = blockIdx.x; i < nbig; i += gridDim.x) {
    const int32_t x = big[i];
    const int64_t o = gofs[x], eo = eoff[x], so = soff[x], sb = sofs[x];
    const int n = gcnt[i], ns = scnt[i];
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const uint32_t slot = gl[o + k];
      tcol[eo + k] = gk[o + slot];
      tw[eo + k] = gv[o + slot];
    }
    for (int k = threadIdx.x; k < ns; k += blockDim.x) {
      const uint32_t slot = sl[sb + k];
      tsidx[so + k] = sk[sb + slot];
      tsval[so + k] = sv[sb + slot];
    }
    if (threadIdx.x == 0) {
      ecnt[x] = n;
      scnt_out[x] = ns;
    }
  }
}

// One row, by a warp, from the upper-bound layout (RowOut) to its final place.
struct RowPlace {
  const int64_t *rowptr, *sptr;
  int32_t* col;
  long long* W;
  int32_t* sidx;
  long long* sval;
};

__device__ __forceinline__ void contract_row_place(const RowOut& f, const RowPlace& t, int64_t x) {
  const int lane = threadIdx.x & 31;
  const int64_t a = f.eoff[x], o = t.rowptr[x];
  const int n = f.ecnt[x];
  for (int k = lane; k < n; k += 32) {
    t.col[o + k] = f.tcol[a + k];
    t.W[o + k] = f.tw[a + k];
  }
  const int64_t sa = f.soff[x], so = t.sptr[x];
  const int ns = f.scnt[x];
  for (int k = lane; k < ns; k += 32) {
    t.sidx[so + k] = f.tsidx[sa + k];
    t.sval[so + k] = f.tsval[sa + k];
  }
}

__global__ void k_contract_compact(int32_t Np, RowOut from, RowPlace to) {
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t x = (((int64_t)blockIdx.x * blockDim.x) >> 5) + (threadIdx.x >> 5); x < Np; x += warps)
    contract_row_place(from, to, x);
}

__global__ void k_min_init(const int32_t* P, const int32_t* R, const int32_t* newid, int32_t N, int32_t* minid) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x)
    // (looked up first: one atomic a node serialised on large communities)
    if (newid[R[v]] < __ldcg(&minid[P[v]])) atomicMin(&minid[P[v]], newid[R[v]]);
}

__global__ void k_next_labels(const int32_t* P, const int32_t* R, const int32_t* newid, const int32_t* minid,
                              int32_t N, int32_t* next) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x)
    next[newid[R[v]]] = minid[P[v]];
}

// Batches: instance of every new node and the first new id of every instance.
__global__ void k_next_inst(LevelDev g, const int32_t* R, const int32_t* newid, int32_t* inst_next, int32_t* off_next) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < g.N; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t x = newid[R[v]];
    const int32_t i = g.inst[v];
    inst_next[x] = i;
    // (most nodes find a smaller id there: one atomic each on B words took
    // 0.15 ms of a level of 0.7 M nodes)
    if (x < off_next[i]) atomicMin(&off_next[i], x);
  }
}

__global__ void k_compose(const int32_t* R, const int32_t* newid, int64_t N0, int32_t* node_of0) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N0; v += (int64_t)gridDim.x * blockDim.x)
    node_of0[v] = newid[R[node_of0[v]]];
}

// ---------------------------------------------------------------------------
// The whole aggregation of a small level in one cooperative launch: the path
// below is about 28 launches and three synchronisations (0.26 ms however small
// the level); here they are eight grid barriers and one synchronisation, with
// the rows' scratch allocated by upper bound.  Rows are summed by a warp or a
// block; a row that needs more distinct targets than the block's table holds, or is
// so long that one block would hold up the level, sends the level to the general
// path.  The next level's degree tiers are found on the way.
static_assert(R_PER_WARP >= 1 << CW_BITS, "a warp's share of the block's table holds a warp's row");
constexpr int64_t RESIDENT_ROW_MAX = 1 << 15;  // entries of a row one block sums

struct AggCtl {
  int32_t np, general, nblock, pad_;
  int32_t tier[NTIERS], pad2_[3];
  int64_t mu, ms;
};

struct AggArgs {
  LevelDev g;
  const int32_t *R, *sizeR, *P;
  int32_t T;  // null slices
  int32_t *newid, *minid, *xmap, *mcnt, *scnt, *mem, *big;
  long long* dsum;
  int64_t *moff, *eoff, *soff;
  int32_t *tcol, *ecnt, *tsidx, *scnt_out;
  long long *tw, *tsval;
  int64_t *rowptr, *sptr;
  int32_t *col, *sidx;  // col: nullptr where the rows are moved by a launch of its own
  long long *W, *sval;
  int32_t* next_labels;
  int32_t *inst_next, *off_next;
  int32_t B;
  uint8_t* tier;
  TierCuts cuts;
  long long* blk;  // 3 words per block
  AggCtl* ctl;
};

// Exclusive prefix of this block's share over the blocks (blk[0..gridDim.x)),
// and the total over all blocks.
__device__ __forceinline__ long long blocks_before(const long long* blk, long long* sm, long long& total) {
  long long before = 0, all = 0;
  for (int b = threadIdx.x; b < gridDim.x; b += RT) {
    const long long x = blk[b];
    all += x;
    if (b < blockIdx.x) before += x;
  }
  long long tb;
  block_scan_excl(before, sm, tb);
  block_scan_excl(all, sm, total);
  return tb;
}

__global__ void __launch_bounds__(RT, 1) k_aggregate(AggArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  long long* hv = reinterpret_cast<long long*>(smem);
  int32_t* hk = reinterpret_cast<int32_t*>(smem + R_SLOTS * sizeof(long long));
  uint16_t* cl = reinterpret_cast<uint16_t*>(hk + R_SLOTS);
  __shared__ long long sm[33];
  __shared__ int32_t ncl[RW];
  __shared__ int32_t ncnt, tiers[NTIERS];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t tid = (int64_t)blockIdx.x * RT + threadIdx.x, threads = (int64_t)gridDim.x * RT;
  const int32_t N = a.g.N;
  const int nb = gridDim.x;
  for (int i = threadIdx.x; i < R_SLOTS; i += RT) {
    hk[i] = -1;
    hv[i] = 0;
  }
  if (threadIdx.x < RW) ncl[threadIdx.x] = 0;
  if (threadIdx.x < NTIERS) tiers[threadIdx.x] = 0;
  // ---- new ids: ranks of the present sub-community labels
  {
    const int32_t chunk = (N + nb - 1) / nb;
    const int32_t lo = min((int64_t)N, (int64_t)blockIdx.x * chunk), hi = min((int64_t)N, (int64_t)lo + chunk);
    long long cnt = 0, tot;
    for (int32_t i = lo + threadIdx.x; i < hi; i += RT) cnt += a.sizeR[i] > 0;
    block_scan_excl(cnt, sm, tot);
    if (threadIdx.x == 0) a.blk[blockIdx.x] = tot;
    for (int64_t i = tid; i <= N; i += threads) {
      a.mcnt[i] = a.scnt[i] = 0;
      a.dsum[i] = 0;
      if (i < N) a.minid[i] = INT32_MAX;
    }
    resident_bar();
    long long np;
    long long at = blocks_before(a.blk, sm, np);
    if (tid == 0) a.ctl->np = (int32_t)np;
    if (np == N) return;  // (every block alike) nothing merged
    for (int32_t base = lo; base < hi; base += RT) {
      const int32_t i = base + threadIdx.x;
      const long long f = i < hi && a.sizeR[i] > 0 ? 1 : 0;
      long long t;
      const long long r = block_scan_excl(f, sm, t);
      if (i < hi) a.newid[i] = (int32_t)(at + r);
      at += t;
    }
    if (a.inst_next)
      for (int64_t i = tid; i <= a.B; i += threads) a.off_next[i] = (int32_t)np;
  }
  resident_bar();
  // ---- members, entries and snapshot entries of every new node
  for (int64_t v = tid; v < N; v += threads) {
    const int32_t x = a.newid[a.R[v]];
    a.xmap[v] = x;
    atomicAdd(&a.mcnt[x], 1);
    atomicAdd((ull*)&a.dsum[x], (ull)(a.g.rowptr[v + 1] - a.g.rowptr[v]));
    int64_t b, e;
    slice_range(a.g, (int32_t)v, b, e);
    if (e > b) atomicAdd(&a.scnt[x], (int32_t)(e - b));
    if (x < __ldcg(&a.minid[a.P[v]])) atomicMin(&a.minid[a.P[v]], x);
    if (a.inst_next) {
      const int32_t i = a.g.inst[v];
      a.inst_next[x] = i;
      if (x < a.off_next[i]) atomicMin(&a.off_next[i], x);
    }
  }
  resident_bar();
  const int32_t Np = a.ctl->np;
  const int32_t chunk = (Np + nb - 1) / nb;
  const int32_t lo = min((int64_t)Np, (int64_t)blockIdx.x * chunk), hi = min((int64_t)Np, (int64_t)lo + chunk);
  {
    long long m = 0, d = 0, c = 0, t;
    for (int32_t x = lo + threadIdx.x; x < hi; x += RT) {
      const long long dx = a.dsum[x], cx = a.scnt[x];
      m += a.mcnt[x];
      d += dx;
      c += cx;
      if (max(dx, cx) > CW_MAX) {
        a.big[atomicAdd(&a.ctl->nblock, 1)] = x;
        // slots: distinct targets, and snapshots (addressed directly up to
        // R_SLOTS of them)
        if (min(dx, (long long)Np) > R_SLOTS / 2 || (a.T > R_SLOTS && min(cx, (long long)a.T) > R_SLOTS / 2) ||
            max(dx, cx) > RESIDENT_ROW_MAX)
          a.ctl->general = 1;
      }
    }
    block_scan_excl(m, sm, t);
    if (threadIdx.x == 0) a.blk[blockIdx.x] = t;
    block_scan_excl(d, sm, t);
    if (threadIdx.x == 0) a.blk[nb + blockIdx.x] = t;
    block_scan_excl(c, sm, t);
    if (threadIdx.x == 0) a.blk[2 * nb + blockIdx.x] = t;
  }
  resident_bar();
  if (a.ctl->general) return;  // (every block alike)
  {
    long long tm, td, tc;
    long long am = blocks_before(a.blk, sm, tm), ad = blocks_before(a.blk + nb, sm, td),
              ac = blocks_before(a.blk + 2 * nb, sm, tc);
    for (int32_t base = lo; base < hi; base += RT) {
      const int32_t x = base + threadIdx.x;
      const bool in = x < hi;
      long long t;
      const long long rm = block_scan_excl(in ? (long long)a.mcnt[x] : 0ll, sm, t);
      if (in) {
        a.moff[x] = am + rm;
        a.mcnt[x] = 0;  // (fill counts of the member lists)
      }
      am += t;
      const long long rd = block_scan_excl(in ? a.dsum[x] : 0ll, sm, t);
      if (in) a.eoff[x] = ad + rd;
      ad += t;
      const long long rc = block_scan_excl(in ? (long long)a.scnt[x] : 0ll, sm, t);
      if (in) a.soff[x] = ac + rc;
      ac += t;
    }
    if (tid == 0) a.moff[Np] = tm;
    for (int64_t v = tid; v < N; v += threads) a.next_labels[a.xmap[v]] = a.minid[a.P[v]];
  }
  resident_bar();
  for (int64_t v = tid; v < N; v += threads) {
    const int32_t x = a.xmap[v];
    a.mem[a.moff[x] + atomicAdd(&a.mcnt[x], 1)] = (int32_t)v;
  }
  resident_bar();
  // ---- rows: a block each for the long ones, then a warp each
  const RowOut o{a.eoff, a.soff, a.tcol, a.tw, a.ecnt, a.tsidx, a.tsval, a.scnt_out};
  const int nbig = a.ctl->nblock;
  for (int i = blockIdx.x; i < nbig; i += nb) {
    const int32_t x = a.big[i];
    if (threadIdx.x == 0) ncnt = 0;
    __syncthreads();
    const int64_t mb = a.moff[x], me = a.moff[x + 1];
    for (int64_t j = mb + w; j < me; j += RW) {
      const int32_t v = a.mem[j];
      const int64_t b = a.g.rowptr[v], e = a.g.rowptr[v + 1];
      const Omega om = node_omega(a.g, v);
      for (int64_t q = b + lane; q < e; q += 32) {
        int32_t u;
        long long W;
        if (edge_at(a.g, q, u, W, om)) {
          const int32_t y = a.xmap[u];
          if (y != x) {
            bool fresh;
            const int64_t slot = ctab_add(hk, hv, R_SLOTS, y, W, fresh);
#if MSLICE_CHECKED
            if (slot < 0) atomicOr(a.g.chk, ERR_BOUNDS);
#endif
            if (fresh) cl[atomicAdd(&ncnt, 1)] = (uint16_t)slot;
          }
        }
      }
    }
    __syncthreads();
    const int n = ncnt;
    for (int k = threadIdx.x; k < n; k += RT) {
      const int slot = cl[k];
      a.tcol[a.eoff[x] + k] = hk[slot];
      a.tw[a.eoff[x] + k] = hv[slot];
      hk[slot] = -1;
      hv[slot] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      a.ecnt[x] = n;
      ncnt = 0;
    }
    __syncthreads();
    if (a.T <= R_SLOTS) {
      for (int64_t j = mb + w; j < me; j += RW) {
        const int32_t v = a.mem[j];
        int64_t b, e;
        slice_range(a.g, v, b, e);
        for (int64_t q = b + lane; q < e; q += 32) {
          int32_t sl;
          long long k;
          slice_entry(a.g, v, q, sl, k);
          shared_add64(&hv[sl], k);  // (strengths are positive)
        }
      }
      __syncthreads();
      for (int sl = threadIdx.x; sl < a.T; sl += RT) {
        const long long k = hv[sl];
        if (k == 0) continue;
        const int at = atomicAdd(&ncnt, 1);
        a.tsidx[a.soff[x] + at] = sl;
        a.tsval[a.soff[x] + at] = k;
        hv[sl] = 0;
      }
    } else {
      for (int64_t j = mb + w; j < me; j += RW) {
        const int32_t v = a.mem[j];
        int64_t b, e;
        slice_range(a.g, v, b, e);
        for (int64_t q = b + lane; q < e; q += 32) {
          int32_t sl;
          long long k;
          slice_entry(a.g, v, q, sl, k);
          bool fresh;
          const int64_t slot = ctab_add(hk, hv, R_SLOTS, sl, k, fresh);
#if MSLICE_CHECKED
          if (slot < 0) atomicOr(a.g.chk, ERR_BOUNDS);
#endif
          if (fresh) cl[atomicAdd(&ncnt, 1)] = (uint16_t)slot;
        }
      }
      __syncthreads();
      for (int k = threadIdx.x; k < ncnt; k += RT) {
        const int slot = cl[k];
        a.tsidx[a.soff[x] + k] = hk[slot];
        a.tsval[a.soff[x] + k] = hv[slot];
        hk[slot] = -1;
        hv[slot] = 0;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) a.scnt_out[x] = ncnt;
    __syncthreads();
  }
  for (int32_t x = (nb - 1 - blockIdx.x) * RW + w; x < Np; x += nb * RW)
    if (max(a.dsum[x], (long long)a.scnt[x]) <= CW_MAX)
      contract_row_warp(a.g, a.xmap, a.moff, a.mem, x, hk + w * R_PER_WARP, hv + w * R_PER_WARP,
                        cl + w * (R_PER_WARP / 2), &ncl[w], o);
  resident_bar();
  // ---- the rows' final places; the next level's tiers
  {
    long long d = 0, c = 0, t;
    for (int32_t x = lo + threadIdx.x; x < hi; x += RT) {
      d += a.ecnt[x];
      c += a.scnt_out[x];
    }
    block_scan_excl(d, sm, t);
    if (threadIdx.x == 0) a.blk[blockIdx.x] = t;
    block_scan_excl(c, sm, t);
    if (threadIdx.x == 0) a.blk[nb + blockIdx.x] = t;
  }
  resident_bar();
  long long td, tc;
  long long ad = blocks_before(a.blk, sm, td), ac = blocks_before(a.blk + nb, sm, tc);
  for (int32_t base = lo; base < hi; base += RT) {
    const int32_t x = base + threadIdx.x;
    const bool in = x < hi;
    const int n = in ? a.ecnt[x] : 0, ns = in ? a.scnt_out[x] : 0;
    long long t;
    const long long rd = block_scan_excl((long long)n, sm, t);
    if (in) a.rowptr[x] = ad + rd;
    ad += t;
    const long long rc = block_scan_excl((long long)ns, sm, t);
    if (in) a.sptr[x] = ac + rc;
    ac += t;
    if (in) {
      const int tr = work_tier(n, ns, a.cuts);
      a.tier[x] = (uint8_t)tr;
      atomicAdd(&tiers[tr], 1);
    }
  }
  __syncthreads();
  if (a.col) {
    const RowPlace place{a.rowptr, a.sptr, a.col, a.W, a.sidx, a.sval};
    for (int32_t x = lo + w; x < hi; x += RW) contract_row_place(o, place, x);
  }
  if (threadIdx.x < NTIERS && tiers[threadIdx.x]) atomicAdd(&a.ctl->tier[threadIdx.x], tiers[threadIdx.x]);
  if (tid == 0) {
    a.rowptr[Np] = a.ctl->mu = td;
    a.sptr[Np] = a.ctl->ms = tc;
  }
}

unsigned gsz(int64_t n) {
  int64_t g = (n + 255) / 256;
  if (g > 152 * 16) g = 152 * 16;
  return (unsigned)(g < 1 ? 1 : g);
}

}  // namespace

// What every aggregated level shares with the level it came from.
static void next_level(const Level& L, Level& next, int32_t Np, int64_t mu, int64_t ms, const int64_t* rowptr,
                       const int32_t* col, const long long* W, const int64_t* sptr, const int32_t* sidx,
                       const long long* sval, const int32_t* inst, const int32_t* inst_off) {
  next = Level{};
  next.d.N = Np;
  next.d.is0 = 0;
  next.d.on = L.d.on;
  next.d.od = L.d.od;
  next.d.global_null = L.d.global_null;
  next.d.on_i = L.d.on_i;
  next.d.od_i = L.d.od_i;
  next.d.chk = L.d.chk;
  next.d.inst = inst;
  next.d.inst_off = inst_off;
  next.d.rowptr = rowptr;
  next.d.col = col;
  next.d.W = W;
  next.d.sptr = sptr;
  next.d.sidx = sidx;
  next.d.sval = sval;
  next.nnz = next.nnz_eff = mu;
  next.ns = ms;
}

// Levels up to this many work units (entries, and RESIDENT_NODE_WORK a node) are
// aggregated in one launch.
constexpr int64_t RESIDENT_AGGREGATE_WORK = (int64_t)1 << 21;
// Up to this many entries and strengths (12 bytes each) the rows go straight to
// their places, in arrays sized by upper bound; past it they are moved once their
// number is known.  A served window of 8 x 4,000 nodes, admitted at 19.2 MB, holds
// 18.8 MB; 19.3 with 2^17, and 20.3 with every array by upper bound.  All of them
// moved: n = 1,000, T = 4 1% longer.
constexpr int64_t RESIDENT_PLACE_MAX = (int64_t)1 << 15;

enum class Resident { DONE, SAME, GENERAL };  // SAME: nothing merged; GENERAL: not for one launch

static Resident aggregate_resident(Solver& S, const Level& L, const int32_t* P, Level& next, const std::string& slot,
                                   int32_t* next_labels, int32_t* node_of0) {
  Ctx& c = *S.c;
  const int32_t N = L.d.N;
  const size_t n1 = (size_t)N + 1, nnz = (size_t)std::max<int64_t>(1, L.nnz), ns = (size_t)std::max<int64_t>(1, L.ns);
  AggArgs a{};
  a.g = L.d;
  a.R = S.R;
  a.sizeR = S.sizeR;
  a.P = P;
  a.T = S.Tn;
  a.newid = S.tmp32b;
  a.minid = S.tmp32a;
  a.xmap = c.ws->get<int32_t>("ag_xmap", N);
  a.mcnt = c.ws->get<int32_t>("ag_mcnt", n1);
  a.scnt = c.ws->get<int32_t>("ag_scnt", n1);
  a.dsum = c.ws->get<long long>("ag_dsum", n1);
  a.moff = c.ws->get<int64_t>("ag_moff", n1);
  a.eoff = c.ws->get<int64_t>("ag_eoff", n1);
  a.soff = c.ws->get<int64_t>("ag_soff", n1);
  a.mem = c.ws->get<int32_t>("ag_mem", N);
  a.big = S.freelist;
  a.tcol = c.ws->get<int32_t>("ag_tcol", nnz);
  a.tw = c.ws->get<long long>("ag_tw", nnz);
  a.tsidx = c.ws->get<int32_t>("ag_tsidx", ns);
  a.tsval = c.ws->get<long long>("ag_tsval", ns);
  a.ecnt = c.ws->get<int32_t>("ag_ecnt", n1);
  a.scnt_out = c.ws->get<int32_t>("ag_scnt_out", n1);
  a.rowptr = c.ws->get<int64_t>(slot + "_rowptr", n1);
  a.sptr = c.ws->get<int64_t>(slot + "_sptr", n1);
  // The next level's rows stay allocated while it is solved (and the server admits
  // requests by what a solve holds), so only few entries are given room by their
  // upper bound.
  const bool placed = L.nnz + L.ns <= RESIDENT_PLACE_MAX;
  const auto place = [&](int64_t entries, int64_t strengths) {
    a.col = c.ws->get<int32_t>(slot + "_col", entries);
    a.W = c.ws->get<long long>(slot + "_W", entries);
    a.sidx = c.ws->get<int32_t>(slot + "_sidx", strengths);
    a.sval = c.ws->get<long long>(slot + "_sval", strengths);
  };
  if (placed) place(L.nnz, L.ns);
  a.next_labels = next_labels;
  a.B = S.B;
  if (L.d.inst) {
    a.inst_next = c.ws->get<int32_t>(slot + "_inst", (size_t)N);
    a.off_next = c.ws->get<int32_t>(slot + "_ioff", (size_t)S.B + 1);
  }
  a.tier = S.tier;
  a.cuts = S.p.cuts;
  a.blk = c.ws->get<long long>("ag_blk", 3 * (size_t)S.sms);
  a.ctl = reinterpret_cast<AggCtl*>(c.ws->get_bytes("ag_ctl", sizeof(AggCtl)));
  check_cuda(cudaMemsetAsync(a.ctl, 0, sizeof(AggCtl), c.stream), "memset");
  check_cuda(cudaFuncSetAttribute(k_aggregate, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TIER4_SMEM_BYTES),
             "resident aggregation's shared memory");
  const int64_t want = std::max<int64_t>((L.nnz + 4095) / 4096, (N + RT - 1) / RT);
  launch_coop(c, k_aggregate, dim3((unsigned)std::max<int64_t>(1, std::min<int64_t>(want, coop_share(S.sms)))), dim3(RT),
              TIER4_SMEM_BYTES, a);
  AggCtl h;
  std::memcpy(&h, readback(c, a.ctl, sizeof(AggCtl)), sizeof(AggCtl));
  if (h.np == N) return Resident::SAME;
  if (h.general) return Resident::GENERAL;
  if (!placed) {
    place(h.mu, h.ms);
    launch(c, k_contract_compact, dim3(gsz((int64_t)h.np * 32)), dim3(256), 0, h.np,
           RowOut{a.eoff, a.soff, a.tcol, a.tw, a.ecnt, a.tsidx, a.tsval, a.scnt_out},
           RowPlace{a.rowptr, a.sptr, a.col, a.W, a.sidx, a.sval});
  }
  if (node_of0)
    launch(c, k_compose, dim3(gsz(S.N0)), dim3(256), 0, (const int32_t*)S.R, (const int32_t*)a.newid, S.N0, node_of0);
  next_level(L, next, h.np, h.mu, h.ms, a.rowptr, a.col, a.W, a.sptr, a.sidx, a.sval, a.inst_next, a.off_next);
  // (a level with top-tier nodes still lays out their scratch tables)
  next.tiers_known = h.tier[NTIERS - 1] == 0;
  for (int t = 0; t < NTIERS; ++t) next.tier_cnt[t] = h.tier[t];
  return Resident::DONE;
}

bool aggregate(Solver& S, const Level& L, const int32_t* P, Level& next, const std::string& slot,
               int32_t* next_labels, int32_t* node_of0, int64_t* checksum) {
  Ctx& c = *S.c;
  const int32_t N = L.d.N;
  if (L.nnz + RESIDENT_NODE_WORK * (int64_t)N <= resident_work(RESIDENT_AGGREGATE_WORK)) {
    const Resident r = aggregate_resident(S, L, P, next, slot, next_labels, node_of0);
    if (r == Resident::SAME) return false;
    if (r == Resident::DONE) {
      if (checksum) *checksum = (int64_t)level_checksum(S, next);
      return true;
    }
  }
  // new ids = ranks of the present sub-community labels
  int32_t* flag = S.tmp32a;
  int32_t* newid = S.tmp32b;
  launch(c, k_present, dim3(gsz(N)), dim3(256), 0, (const int32_t*)S.sizeR, N, flag);
  int32_t* d_np = c.ws->get<int32_t>("ag_np", 1);
  scan_excl(c, flag, newid, N, d_np);
  const int32_t Np = *static_cast<const int32_t*>(readback(c, d_np, sizeof(int32_t)));
  if (Np == N) return false;

  // ---- contraction: member lists, rows summed per neighbouring new node ----
  const int64_t np1 = (int64_t)Np + 1;
  int32_t* xmap = c.ws->get<int32_t>("ag_xmap", N);
  int32_t* mcnt = c.ws->get<int32_t>("ag_mcnt", np1);
  int32_t* scnt = c.ws->get<int32_t>("ag_scnt", np1);
  long long* dsum = c.ws->get<long long>("ag_dsum", np1);
  check_cuda(cudaMemsetAsync(mcnt, 0, np1 * sizeof(int32_t), c.stream), "memset");
  check_cuda(cudaMemsetAsync(scnt, 0, np1 * sizeof(int32_t), c.stream), "memset");
  check_cuda(cudaMemsetAsync(dsum, 0, np1 * sizeof(long long), c.stream), "memset");
  launch(c, k_contract_prep, dim3(gsz(N)), dim3(256), 0, L.d, (const int32_t*)S.R, (const int32_t*)newid, xmap, mcnt,
         dsum, scnt);
  int64_t* moff = c.ws->get<int64_t>("ag_moff", np1);
  int64_t* eoff = c.ws->get<int64_t>("ag_eoff", np1);
  int64_t* soff = c.ws->get<int64_t>("ag_soff", np1);
  scan_excl(c, (const int32_t*)mcnt, moff, np1, (int64_t*)nullptr);
  scan_excl(c, (const int64_t*)dsum, eoff, np1, (int64_t*)nullptr);
  scan_excl(c, (const int32_t*)scnt, soff, np1, (int64_t*)nullptr);
  int32_t* mem = c.ws->get<int32_t>("ag_mem", N);
  check_cuda(cudaMemsetAsync(mcnt, 0, np1 * sizeof(int32_t), c.stream), "memset");
  launch(c, k_contract_members, dim3(gsz(N)), dim3(256), 0, N, (const int32_t*)xmap, (const int64_t*)moff, mcnt, mem);
  int32_t* lists = c.ws->get<int32_t>("ag_lists", 3 * (size_t)Np);
  int32_t* tcnt = c.ws->get<int32_t>("ag_tcnt", 4);
  int64_t* gsize = c.ws->get<int64_t>("ag_gsize", np1);
  int64_t* gofs = c.ws->get<int64_t>("ag_gofs", np1);
  int64_t* ssize = c.ws->get<int64_t>("ag_ssize", np1);
  int64_t* sofs = c.ws->get<int64_t>("ag_sofs", np1);
  check_cuda(cudaMemsetAsync(tcnt, 0, 4 * sizeof(int32_t), c.stream), "memset");
  check_cuda(cudaMemsetAsync(gsize + Np, 0, sizeof(int64_t), c.stream), "memset");
  check_cuda(cudaMemsetAsync(ssize + Np, 0, sizeof(int64_t), c.stream), "memset");
  launch(c, k_contract_tier, dim3(gsz(Np)), dim3(256), 0, Np, (const long long*)dsum, (const int32_t*)scnt, lists, tcnt,
         gsize, ssize);
  int64_t* d_gtot = c.ws->get<int64_t>("ag_gtot", 2);
  scan_excl(c, (const int64_t*)gsize, gofs, np1, d_gtot);
  scan_excl(c, (const int64_t*)ssize, sofs, np1, d_gtot + 1);
  struct {
    int32_t t[4];
    int64_t gtot, stot;
  } hd;
  check_cuda(cudaMemcpyAsync(c.pinned, tcnt, 4 * sizeof(int32_t), cudaMemcpyDeviceToHost, c.stream), "copy");
  check_cuda(cudaMemcpyAsync(static_cast<char*>(c.pinned) + 16, d_gtot, 2 * sizeof(int64_t), cudaMemcpyDeviceToHost,
                             c.stream), "copy");
  sync(c);
  std::memcpy(&hd, c.pinned, sizeof(hd));
  const int64_t cap = L.nnz > 0 ? L.nnz : 1;
  const int64_t scap = L.ns > 0 ? L.ns : 1;
  int32_t* tcol = c.ws->get<int32_t>("ag_tcol", cap);
  long long* tw = c.ws->get<long long>("ag_tw", cap);
  int32_t* tsidx = c.ws->get<int32_t>("ag_tsidx", scap);
  long long* tsval = c.ws->get<long long>("ag_tsval", scap);
  int32_t* ecnt = c.ws->get<int32_t>("ag_ecnt", np1);
  int32_t* scnt_out = c.ws->get<int32_t>("ag_scnt_out", np1);
  check_cuda(cudaMemsetAsync(ecnt + Np, 0, sizeof(int32_t), c.stream), "memset");
  check_cuda(cudaMemsetAsync(scnt_out + Np, 0, sizeof(int32_t), c.stream), "memset");
  if (hd.t[0] > 0)
    launch(c, k_contract_warp, dim3(152 * 4), dim3(CW_WARPS * 32), 0, L.d, (const int32_t*)xmap, (const int64_t*)moff,
           (const int32_t*)mem, (const int32_t*)lists, (const int32_t*)tcnt, (const int64_t*)eoff,
           (const int64_t*)soff, tcol, tw, ecnt, tsidx, tsval, scnt_out);
  const size_t cb_smem = ((size_t)1 << CB_BITS) * (sizeof(long long) + sizeof(int32_t)) +
                         (size_t)CB_MAX * sizeof(int32_t);
  if (hd.t[1] > 0) {
    check_cuda(cudaFuncSetAttribute(k_contract_block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cb_smem),
               "attribute");
    int32_t* queue = c.ws->get<int32_t>("ag_queue", 1);
    check_cuda(cudaMemsetAsync(queue, 0, sizeof(int32_t), c.stream), "memset");
    launch(c, k_contract_block, dim3(152 * 2), dim3(CB_THREADS), cb_smem, L.d, (const int32_t*)xmap,
           (const int64_t*)moff, (const int32_t*)mem, (const int32_t*)(lists + Np), (const int32_t*)(tcnt + 1),
           (const int64_t*)eoff, (const int64_t*)soff, tcol, tw, ecnt, tsidx, tsval, scnt_out, queue);
  }
  if (hd.t[2] > 0) {
    if (hd.gtot > ((int64_t)1 << 31) * 8) fail(MSLICE_ENOMEM, "aggregation scratch too large");
    const int32_t nbig = hd.t[2];
    const int32_t* big = lists + 2 * (int64_t)Np;
    const int32_t* nbig_d = tcnt + 2;
    int32_t* gk = c.ws->get<int32_t>("ag_gk", hd.gtot);
    long long* gv = c.ws->get<long long>("ag_gv", hd.gtot);
    uint32_t* gl = c.ws->get<uint32_t>("ag_gl", hd.gtot);
    int32_t* sk = c.ws->get<int32_t>("ag_sk", hd.stot);
    long long* sv = c.ws->get<long long>("ag_sv", hd.stot);
    uint32_t* sl = c.ws->get<uint32_t>("ag_sl", hd.stot);
    int32_t* cnts = c.ws->get<int32_t>("ag_bigcnt", 2 * (size_t)nbig);
    int64_t* mcnt_big = c.ws->get<int64_t>("ag_bigm", (size_t)nbig + 1);
    int64_t* mpre = c.ws->get<int64_t>("ag_bigpre", (size_t)nbig + 1);
    check_cuda(cudaMemsetAsync(gk, 0xff, hd.gtot * sizeof(int32_t), c.stream), "memset");
    check_cuda(cudaMemsetAsync(gv, 0, hd.gtot * sizeof(long long), c.stream), "memset");
    check_cuda(cudaMemsetAsync(sk, 0xff, hd.stot * sizeof(int32_t), c.stream), "memset");
    check_cuda(cudaMemsetAsync(sv, 0, hd.stot * sizeof(long long), c.stream), "memset");
    check_cuda(cudaMemsetAsync(cnts, 0, 2 * (size_t)nbig * sizeof(int32_t), c.stream), "memset");
    check_cuda(cudaMemsetAsync(mcnt_big + nbig, 0, sizeof(int64_t), c.stream), "memset");
    launch(c, k_big_members, dim3(gsz(nbig)), dim3(256), 0, big, nbig_d, (const int64_t*)moff, mcnt_big);
    scan_excl(c, (const int64_t*)mcnt_big, mpre, (int64_t)nbig + 1, (int64_t*)nullptr);
    check_cuda(cudaFuncSetAttribute(k_big_insert, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BI_SMEM),
               "attribute");
    launch(c, k_big_insert, dim3(152 * 4), dim3(256), BI_SMEM, L.d, (const int32_t*)xmap, (const int64_t*)moff,
           (const int32_t*)mem, big, nbig_d, (const int64_t*)mpre, (const int64_t*)gofs, (const int64_t*)gsize, gk,
           gv, gl, cnts, (const int64_t*)sofs, (const int64_t*)ssize, sk, sv, sl, cnts + nbig);
    launch(c, k_big_output, dim3(std::min<int32_t>(nbig, 152 * 4)), dim3(256), 0, big, nbig_d,
           (const int64_t*)gofs, (const int32_t*)gk, (const long long*)gv, (const uint32_t*)gl,
           (const int32_t*)cnts, (const int64_t*)sofs, (const int32_t*)sk, (const long long*)sv, (const uint32_t*)sl,
           (const int32_t*)(cnts + nbig), (const int64_t*)eoff, (const int64_t*)soff, tcol, tw, ecnt, tsidx, tsval,
           scnt_out);
  }

  int64_t* rowptr = c.ws->get<int64_t>(slot + "_rowptr", (size_t)np1);
  int64_t* sptr = c.ws->get<int64_t>(slot + "_sptr", (size_t)np1);
  int64_t* d_tot = c.ws->get<int64_t>("ag_tot", 2);
  scan_excl(c, (const int32_t*)ecnt, rowptr, np1, d_tot);
  scan_excl(c, (const int32_t*)scnt_out, sptr, np1, d_tot + 1);
  const int64_t* tots = static_cast<const int64_t*>(readback(c, d_tot, 2 * sizeof(int64_t)));
  const int64_t mu = tots[0], ms = tots[1];
  int32_t* col = c.ws->get<int32_t>(slot + "_col", mu);
  long long* W = c.ws->get<long long>(slot + "_W", mu);
  int32_t* sidx = c.ws->get<int32_t>(slot + "_sidx", ms);
  long long* sval = c.ws->get<long long>(slot + "_sval", ms);
  launch(c, k_contract_compact, dim3(gsz((int64_t)Np * 32)), dim3(256), 0, Np,
         RowOut{eoff, soff, tcol, tw, ecnt, tsidx, tsval, scnt_out}, RowPlace{rowptr, sptr, col, W, sidx, sval});

  int32_t *inst_next = nullptr, *off_next = nullptr;
  if (L.d.inst) {
    inst_next = c.ws->get<int32_t>(slot + "_inst", (size_t)Np);
    off_next = c.ws->get<int32_t>(slot + "_ioff", (size_t)S.B + 1);
    fill_i32(c, off_next, Np, (int64_t)S.B + 1);
    launch(c, k_next_inst, dim3(gsz(N)), dim3(256), 0, L.d, (const int32_t*)S.R, (const int32_t*)newid, inst_next,
           off_next);
  }
  next_level(L, next, Np, mu, ms, rowptr, col, W, sptr, sidx, sval, inst_next, off_next);

  // ---- initial labels, level map ----
  int32_t* minid = flag;  // reuse
  fill_i32(c, minid, INT32_MAX, N);
  launch(c, k_min_init, dim3(gsz(N)), dim3(256), 0, P, (const int32_t*)S.R, (const int32_t*)newid, N, minid);
  launch(c, k_next_labels, dim3(gsz(N)), dim3(256), 0, P, (const int32_t*)S.R, (const int32_t*)newid,
         (const int32_t*)minid, N, next_labels);
  if (node_of0)
    launch(c, k_compose, dim3(gsz(S.N0)), dim3(256), 0, (const int32_t*)S.R, (const int32_t*)newid, S.N0, node_of0);
  if (checksum) *checksum = (int64_t)level_checksum(S, next);
  return true;
}

}  // namespace mslice
