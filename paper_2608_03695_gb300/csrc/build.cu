// Supra-graph builder (Eq. supra-adjacency): the level-0 CSR over N = n*T
// supra-nodes.  Row v = s*n + i holds, in ascending column order, the
// coupling entries to the copies of i in earlier snapshots, the snapshot-s row
// of i shifted by s*n, and the coupling entries to later copies.  Ordinal
// coupling (Eq. supra-adjacency) couples s with s-1 and s+1; categorical
// coupling (the all-pairs omega^(sr) of Eq. multislice-modularity) with every
// other snapshot.  Entries are 8-byte {col, w} pairs; w <= 0 flags a coupling
// entry and names its pair's slot (-w-1) in a table of omega numerators, so
// omega (uniform or per pair) is applied at solve time and a sweep needs no
// rebuild.
#include "build.h"

#include "../../include/mslice.h"

#include <algorithm>
#include <numeric>

namespace mslice {

namespace {

struct SliceTable {
  const int64_t* const* indptr;
  const int32_t* const* indices;
  const int32_t* const* weights;
};

// indptr of every snapshot: starts at 0, non-decreasing, ends at nnz_s.  status[1]:
// some row is a hub's.
__global__ void k_check_indptr(SliceTable st, const int64_t* nnz, int32_t T, int64_t n, unsigned* status) {
  const int64_t total = n * (int64_t)T;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < total; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t s = (int32_t)(v / n);
    const int64_t i = v - (int64_t)s * n;
    const int64_t a = st.indptr[s][i], b = st.indptr[s][i + 1];
    bool bad = (b < a) || (a < 0) || (b > nnz[s]);
    if (i == 0 && a != 0) bad = true;
    if (i == n - 1 && b != nnz[s]) bad = true;
    if (bad) atomicOr(status, ERR_BAD_INPUT);
    if (b - a > HUB_ROW) status[1] = 1;
  }
}

// Coupled snapshots of snapshot s: [lo, s) below and (s, hi) above.
__device__ __forceinline__ void coupled_range(int32_t coupling, int32_t T, int32_t s, int32_t& lo, int32_t& hi) {
  lo = coupling == 0 ? (s > 0 ? s - 1 : 0) : 0;
  hi = coupling == 0 ? (s + 2 < T ? s + 2 : T) : T;
}

// The flag of the coupling entry from snapshot s to r: -(slot + 1).
__device__ __forceinline__ int32_t coupling_flag(int32_t coupling, int32_t T, int32_t s, int32_t r) {
  return coupling == 0 ? -((s < r ? s : r) + 1) : -(s * T + r + 1);
}

// Rows: G lanes per supra-row check the snapshot row and write the
// supra-row in the same pass: rowptr (in closed form: first[s] entries come
// before snapshot s, and every row of a snapshot has the same coupling entries),
// the shifted entries, the coupling flags and k_v = sum of the row's weights.
// A row must be sorted strictly ascending, in range, without a self-loop, with
// w >= 1 and the mirrored entry (j, i) present with the same weight.  Only the
// entries above the diagonal look for their mirror image: when each finds one
// (distinct entries have distinct ones) and as many entries lie below the
// diagonal as above (balance ends at 0), every entry below is such an image.
// The searches bound the pass (about four dependent lookups each, a few rows
// away in L2); checking and copying apart, with a search per entry and a scan
// for the row pointers, took 1.6 ms for 31 M entries.
// G = 8, where rows are short and there are more of them than warps: with a warp
// each, most lanes of a warp have no entry.  Rows of more than BUILD_LONG entries
// are then taken by the whole warp (with 8 lanes a row of 1,400 entries alone took
// as long as the rest of the pass), and rows of more than HUB_ROW by blocks of
// their own (k_build_hubs): a warp takes the long ones of its four rows one after
// another, and where hubs are neighbours in node order that alone was the pass.
// G = 32 (a warp a row), where the rows are long on average or there are warps for
// all of them.
// Builds, four long rows a warp in turn -> now (a warp a row before that): hubs of
// 100,000, 60,000, 20,000 and 40 of 3,000 (N = 300,000) 12.0 -> 0.77 ms (6.9); 12
// hubs of 6,000 (N = 60,000) 1.60 -> 0.58 (0.88); one snapshot of 1,500 nodes,
// every second pair linked, 0.77 -> 0.60 (0.61).  Hubs from 512 entries on: 3%
// slower on a power-law graph of n = 100,000 (rows up to 1,400, 2,560 of them).
constexpr int64_t BUILD_LONG = 64;
constexpr int BUILD_HUB_PARTS = 8;                // blocks that share a hub's row
constexpr int64_t BUILD_WARPS = 152 * (2048 / 32);  // resident at a time

// Entries from + gl, from + gl + step, ... (up to `to`) of row i of a snapshot
// (entries from a on): checked and written at out.
__device__ __forceinline__ void build_entries(const int64_t* ip, const int32_t* ix, const int32_t* wt, int32_t n,
                                              int32_t i, int64_t a, int64_t from, int64_t to, int2* out, int32_t off,
                                              int gl, int step, long long& ksum, int& above, bool& bad) {
  for (int64_t e = from + gl; e < to; e += step) {
    const int32_t j = ix[e];
    const int32_t w = wt[e];
    out[e - a] = make_int2(j + off, w);
    ksum += w;
    if (j < 0 || j >= n || j == i || w < 1) {
      bad = true;
      continue;
    }
    if (e > a && ix[e - 1] >= j) bad = true;
    above += j > i ? 1 : -1;
    if (j < i) continue;
    // binary search for i in row j
    int64_t x = ip[j], y = ip[j + 1];
    const int64_t end = y;
    while (x < y) {
      const int64_t mid = (x + y) >> 1;
      if (ix[mid] < i)
        x = mid + 1;
      else
        y = mid;
    }
    if (x >= end || ix[x] != i || wt[x] != w) bad = true;
  }
}

// What the rows' passes found (per warp): entries above less those below the
// diagonal, and anything malformed.
__device__ __forceinline__ void build_verdict(long long above, bool bad, ull* balance, unsigned* status) {
  above = warp_sum(above);
  const bool any = __any_sync(0xffffffffu, bad);
  if ((threadIdx.x & 31) == 0) {
    if (above) atomicAdd(balance, (ull)above);
    if (any) atomicOr(status, ERR_BAD_INPUT);
  }
}

// hubs: room for every row of more than HUB_ROW entries, hubs' number at
// *nhubs; nullptr: those rows are taken here too.
template <int G>
__global__ void k_build_rows(SliceTable st, int32_t T, int64_t n, int32_t coupling, const int64_t* first,
                             int64_t* rowptr, int2* adj, int64_t* k, int32_t* hubs, ull* nhubs, ull* balance,
                             unsigned* status) {
  const int64_t total = n * (int64_t)T;
  const int lane = threadIdx.x & 31, gl = lane % G;
  const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << (lane - gl);
  const int64_t groups = (int64_t)gridDim.x * blockDim.x / G;
  const int32_t n32 = (int32_t)n;
  long long above_sum = 0;
  bool bad = false;
  // (warp-uniform loop)
  for (int64_t v0 = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / G; v0 < total; v0 += groups) {
    const int64_t v = v0 + lane / G;
    const bool ok = v < total;
    const int32_t s = ok ? (int32_t)v / n32 : 0, i = ok ? (int32_t)v - s * n32 : 0;
    const int64_t* ip = st.indptr[s];
    const int64_t a = ok ? ip[i] : 0, b = ok ? ip[i + 1] : 0;
    const bool hub = hubs && b - a > HUB_ROW;
    int32_t lo, hi;
    coupled_range(coupling, T, s, lo, hi);
    int64_t out = first[s] + a + i * (int64_t)(hi - lo - 1);
    const int32_t off = s * n32;
    long long ksum = 0;
    int above = 0;
    if (ok) {
      if (gl == 0) {
        rowptr[v] = out;
        if (hub) hubs[atomicAdd(nhubs, 1ull)] = (int32_t)v;
      }
      for (int32_t r = lo + gl; r < s; r += G)
        adj[out + (r - lo)] = make_int2(r * n32 + i, coupling_flag(coupling, T, s, r));
      out += s - lo;
      for (int32_t r = s + 1 + gl; r < hi; r += G)
        adj[out + (b - a) + (r - s - 1)] = make_int2(r * n32 + i, coupling_flag(coupling, T, s, r));
      if (!hub && (G == 32 || b - a <= BUILD_LONG))
        build_entries(ip, st.indices[s], st.weights[s], n32, i, a, a, b, adj + out, off, gl, G, ksum, above, bad);
    }
    if constexpr (G < 32) {
      unsigned wide = __ballot_sync(0xffffffffu, gl == 0 && !hub && b - a > BUILD_LONG);
      while (wide) {
        const int src = __ffs(wide) - 1;
        wide &= wide - 1;
        const int32_t ss = __shfl_sync(0xffffffffu, s, src), is = __shfl_sync(0xffffffffu, i, src);
        const int64_t as = __shfl_sync(0xffffffffu, a, src), bs = __shfl_sync(0xffffffffu, b, src),
                      os = __shfl_sync(0xffffffffu, out, src);
        long long kw = 0;
        build_entries(st.indptr[ss], st.indices[ss], st.weights[ss], n32, is, as, as, bs, adj + os, ss * n32, lane, 32,
                      kw, above, bad);
        kw = warp_sum(kw);
        if (lane == src) ksum = kw;  // (the others of the group hold 0)
      }
    }
#pragma unroll
    for (int m = G / 2; m >= 1; m >>= 1) ksum += __shfl_xor_sync(gmask, ksum, m);
    if (ok && gl == 0) k[v] = ksum;  // (0 so far for a hub)
    above_sum += above;
  }
  build_verdict(above_sum, bad, balance, status);
}

// The snapshot rows of the hubs: blocks (x, 0 .. BUILD_HUB_PARTS - 1) share one.
__global__ void __launch_bounds__(256)
    k_build_hubs(SliceTable st, int32_t T, int64_t n, int32_t coupling, const int64_t* rowptr, int2* adj, int64_t* k,
                 const int32_t* hubs, const ull* nhubs, ull* balance, unsigned* status) {
  const int32_t n32 = (int32_t)n;
  const int64_t count = (int64_t)*nhubs;
  long long above_sum = 0;
  bool bad = false;
  for (int64_t h = blockIdx.x; h < count; h += gridDim.x) {
    const int32_t v = hubs[h], s = v / n32, i = v - s * n32;
    const int64_t a = st.indptr[s][i], b = st.indptr[s][i + 1];
    const int64_t part = (b - a + gridDim.y - 1) / gridDim.y;
    const int64_t from = min(b, a + blockIdx.y * part), to = min(b, from + part);
    int32_t lo, hi;
    coupled_range(coupling, T, s, lo, hi);
    long long ksum = 0;
    int above = 0;
    build_entries(st.indptr[s], st.indices[s], st.weights[s], n32, i, a, from, to, adj + rowptr[v] + (s - lo), s * n32,
                  threadIdx.x, blockDim.x, ksum, above, bad);
    ksum = warp_sum(ksum);
    if ((threadIdx.x & 31) == 0 && ksum) atomicAdd((ull*)&k[v], (ull)ksum);
    above_sum += above;
  }
  build_verdict(above_sum, bad, balance, status);
}

// 2m_s = sum of k_v over the rows of snapshot s: blockIdx.y is the snapshot,
// blocks stride over its rows, one atomic per block.
__global__ void k_slice_mass(const int64_t* k, int64_t n, ull* two_m) {
  __shared__ ull sm[32];
  const int32_t s = blockIdx.y;
  ull t = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    t += (ull)k[(int64_t)s * n + i];
  t = warp_sum(t);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x < 32) {
    ull x = threadIdx.x < (blockDim.x >> 5) ? sm[threadIdx.x] : 0ull;
    x = warp_sum(x);
    if (threadIdx.x == 0 && x) atomicAdd(&two_m[s], x);
  }
}

__global__ void k_lambda(const int64_t* two_m, int32_t T, const int32_t* slice_inst, const long long* gn,
                         const long long* gd, u128* lam) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= T) return;
  const int32_t i = slice_inst ? slice_inst[s] : 0;
  const long long t = two_m[s];
  lam[s] = t > 0 ? (((u128)(ull)gn[i]) << P_BITS) / ((u128)(ull)gd[i] * (u128)(ull)t) : (u128)0;
}

// Copies one instance into the concatenated arrays (coupling flags move to
// the instance's slots of the batch's table).
__global__ void k_append(int64_t Ni, const int64_t* rowptr, const int2* adj, const int64_t* k, int64_t n, int32_t inst,
                         int64_t noff, int64_t eoff, int32_t soff, int32_t cwoff, int64_t* rowptr_o, int2* adj_o,
                         int64_t* k_o, int32_t* slice0, int32_t* inst0) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < Ni; v += (int64_t)gridDim.x * blockDim.x) {
    rowptr_o[noff + v] = rowptr[v] + eoff;
    k_o[noff + v] = k[v];
    slice0[noff + v] = soff + (int32_t)(v / n);
    inst0[noff + v] = inst;
  }
  const int64_t nnz = rowptr[Ni];
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x) {
    const int2 x = adj[e];
    adj_o[eoff + e] = make_int2(x.x + (int32_t)noff, x.y <= 0 ? x.y - cwoff : x.y);
  }
}

__global__ void k_slice_inst(int32_t* slice_inst, int32_t soff, int32_t T, int32_t inst) {
  for (int s = threadIdx.x; s < T; s += blockDim.x) slice_inst[soff + s] = inst;
}

unsigned gs(int64_t n, int per) {
  int64_t g = (n + per - 1) / per;
  if (g > 152 * 16) g = 152 * 16;
  return (unsigned)(g < 1 ? 1 : g);
}

}  // namespace

void build_supra(Ctx& c, const std::vector<const int64_t*>& indptr, const std::vector<const int32_t*>& indices,
                 const std::vector<const int32_t*>& weights, const std::vector<int64_t>& nnz, int64_t n,
                 SupraGraph& g, int32_t coupling) {
  const int32_t T = (int32_t)indptr.size();
  if (coupling != 0 && (int64_t)T * T >= INT32_MAX) fail(MSLICE_EINVAL, "categorical coupling needs T*T < 2^31");
  g.T = T;
  g.coupling = coupling;
  g.ncw = coupling_slots(coupling, T);
  g.n = n;
  g.N = n * T;
  // device table of snapshot pointers
  const int64_t** d_ip = c.ws->get<const int64_t*>("b_ip", T);
  const int32_t** d_ix = c.ws->get<const int32_t*>("b_ix", T);
  const int32_t** d_wt = c.ws->get<const int32_t*>("b_wt", T);
  int64_t* d_nnz = c.ws->get<int64_t>("b_nnz", T);
  check_cuda(cudaMemcpyAsync(d_ip, indptr.data(), T * sizeof(void*), cudaMemcpyHostToDevice, c.stream), "copy");
  check_cuda(cudaMemcpyAsync(d_ix, indices.data(), T * sizeof(void*), cudaMemcpyHostToDevice, c.stream), "copy");
  check_cuda(cudaMemcpyAsync(d_wt, weights.data(), T * sizeof(void*), cudaMemcpyHostToDevice, c.stream), "copy");
  check_cuda(cudaMemcpyAsync(d_nnz, nnz.data(), T * sizeof(int64_t), cudaMemcpyHostToDevice, c.stream), "copy");
  SliceTable st{d_ip, d_ix, d_wt};
  check_cuda(cudaMemsetAsync(c.d_status, 0, 2 * sizeof(unsigned), c.stream), "memset");
  g.hubs = false;
  if (g.N > 0) {
    unsigned hubs = 0;
    launch(c, k_check_indptr, dim3(gs(g.N, 256)), dim3(256), 0, st, (const int64_t*)d_nnz, T, n, c.d_status);
    check_status(c, "snapshot row pointers", &hubs);
    g.hubs = hubs != 0;
  }
  // entries before every snapshot, and in all
  std::vector<int64_t> first(T + 1, 0);
  for (int32_t s = 0; s < T; ++s) {
    const int64_t partners = coupling == 0 ? (s > 0 ? 1 : 0) + (s + 1 < T ? 1 : 0) : T - 1;
    first[s + 1] = first[s] + nnz[s] + n * partners;
  }
  g.nnz = n > 0 ? first[T] : 0;
  int64_t* d_first = c.ws->get<int64_t>("b_first", T + 1);
  check_cuda(cudaMemcpyAsync(d_first, first.data(), (T + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, c.stream),
             "copy");
  g.rowptr = static_cast<int64_t*>(g.mem.get_bytes("rowptr0", (g.N + 1) * sizeof(int64_t)));
  check_cuda(cudaMemcpyAsync(g.rowptr + g.N, &g.nnz, sizeof(int64_t), cudaMemcpyHostToDevice, c.stream), "copy");
  g.adj = static_cast<int2*>(g.mem.get_bytes("adj0", (g.nnz ? g.nnz : 1) * sizeof(int2)));
  g.k = static_cast<int64_t*>(g.mem.get_bytes("k0", (g.N ? g.N : 1) * sizeof(int64_t)));
  g.two_m = static_cast<int64_t*>(g.mem.get_bytes("two_m", T * sizeof(int64_t)));
  check_cuda(cudaMemsetAsync(g.two_m, 0, T * sizeof(int64_t), c.stream), "memset");
  if (g.N > 0) {
    ull* balance = c.ws->get<ull>("b_balance", 2);
    ull* nhubs = balance + 1;
    check_cuda(cudaMemsetAsync(balance, 0, 2 * sizeof(ull), c.stream), "memset");
    const int64_t entries = std::accumulate(nnz.begin(), nnz.end(), (int64_t)0);
    const bool all_warps = g.N <= BUILD_WARPS;
    int32_t* hubs = g.hubs && !all_warps ? c.ws->get<int32_t>("b_hubs", entries / HUB_ROW + 1) : nullptr;
    if (all_warps || entries > BUILD_LONG * g.N)
      launch(c, k_build_rows<32>, dim3(gs(g.N * 32, 256)), dim3(256), 0, st, T, n, coupling, (const int64_t*)d_first,
             g.rowptr, g.adj, g.k, hubs, nhubs, balance, c.d_status);
    else
      launch(c, k_build_rows<8>, dim3(gs(g.N * 8, 256)), dim3(256), 0, st, T, n, coupling, (const int64_t*)d_first,
             g.rowptr, g.adj, g.k, hubs, nhubs, balance, c.d_status);
    if (hubs)
      launch(c, k_build_hubs, dim3(76, BUILD_HUB_PARTS), dim3(256), 0, st, T, n, coupling, (const int64_t*)g.rowptr,
             g.adj, g.k, (const int32_t*)hubs, (const ull*)nhubs, balance, c.d_status);
    unsigned gx = (unsigned)std::min<int64_t>((n + 255) / 256, 64);
    launch(c, k_slice_mass, dim3(gx, T), dim3(256), 0, (const int64_t*)g.k, n, (ull*)g.two_m);
    const bool mirrored = *static_cast<const ull*>(readback(c, balance, sizeof(ull))) == 0;
    check_status(c, "snapshot rows");
    if (!mirrored) fail(MSLICE_EINVAL, "snapshot rows: malformed input");
  }
  g.two_m_host.resize(T);
  check_cuda(cudaMemcpyAsync(g.two_m_host.data(), g.two_m, T * sizeof(int64_t), cudaMemcpyDeviceToHost, c.stream),
             "copy");
  sync(c);
  g.nnz_intra = g.nnz - coupling_entries(coupling, n, T);
  g.B = 1;
  g.inst.assign(1, InstInfo{n, 0, T, 0, coupling, 0});
}

void compute_lambda(Ctx& c, const SupraGraph& g, const long long* gn, const long long* gd, u128* lam) {
  launch(c, k_lambda, dim3(grid_for(g.T, 128)), dim3(128), 0, (const int64_t*)g.two_m, g.T,
         (const int32_t*)g.slice_inst, gn, gd, lam);
}

void concat_instances(Ctx& c, const std::vector<const SupraGraph*>& parts, SupraGraph& out) {
  const int32_t B = (int32_t)parts.size();
  out.B = B;
  out.inst.assign(B, InstInfo{});
  int64_t N = 0, nnz = 0, nnz_intra = 0, ncw = 0;
  int32_t T = 0;
  bool hubs = false;
  for (int32_t i = 0; i < B; ++i) {
    out.inst[i] = InstInfo{parts[i]->n, N, parts[i]->T, T, parts[i]->coupling, ncw};
    N += parts[i]->N;
    nnz += parts[i]->nnz;
    nnz_intra += parts[i]->nnz_intra;
    hubs = hubs || parts[i]->hubs;
    T += parts[i]->T;
    ncw += parts[i]->ncw;
  }
  if (ncw >= INT32_MAX) fail(MSLICE_EINVAL, "the batch's coupling tables need fewer than 2^31 slots");
  out.ncw = ncw;
  out.hubs = hubs;
  out.coupling = -1;  // per instance
  out.N = N;
  out.T = T;
  out.n = parts.empty() ? 0 : parts[0]->n;
  out.nnz = nnz;
  out.nnz_intra = nnz_intra;
  out.rowptr = static_cast<int64_t*>(out.mem.get_bytes("rowptr0", (N + 1) * sizeof(int64_t)));
  out.adj = static_cast<int2*>(out.mem.get_bytes("adj0", (nnz ? nnz : 1) * sizeof(int2)));
  out.k = static_cast<int64_t*>(out.mem.get_bytes("k0", (N ? N : 1) * sizeof(int64_t)));
  out.two_m = static_cast<int64_t*>(out.mem.get_bytes("two_m", (T ? T : 1) * sizeof(int64_t)));
  out.slice0 = static_cast<int32_t*>(out.mem.get_bytes("slice0", (N ? N : 1) * sizeof(int32_t)));
  out.inst0 = static_cast<int32_t*>(out.mem.get_bytes("inst0", (N ? N : 1) * sizeof(int32_t)));
  out.inst_off0 = static_cast<int32_t*>(out.mem.get_bytes("inst_off0", (B + 1) * sizeof(int32_t)));
  out.slice_inst = static_cast<int32_t*>(out.mem.get_bytes("slice_inst", (T ? T : 1) * sizeof(int32_t)));
  std::vector<int32_t> offs(B + 1);
  int64_t eoff = 0;
  out.two_m_host.clear();
  for (int32_t i = 0; i < B; ++i) {
    const SupraGraph& p = *parts[i];
    offs[i] = (int32_t)out.inst[i].noff;
    if (p.N > 0)
      launch(c, k_append, dim3(gs(std::max<int64_t>(p.N, p.nnz), 256)), dim3(256), 0, p.N, (const int64_t*)p.rowptr,
             (const int2*)p.adj, (const int64_t*)p.k, p.n, i, out.inst[i].noff, eoff, out.inst[i].soff,
             (int32_t)out.inst[i].cwoff, out.rowptr, out.adj, out.k, out.slice0, out.inst0);
    if (p.T > 0) {
      check_cuda(cudaMemcpyAsync(out.two_m + out.inst[i].soff, p.two_m, p.T * sizeof(int64_t),
                                 cudaMemcpyDeviceToDevice, c.stream), "copy");
      launch(c, k_slice_inst, dim3(1), dim3(256), 0, out.slice_inst, out.inst[i].soff, p.T, i);
    }
    for (int64_t t : p.two_m_host) out.two_m_host.push_back(t);
    eoff += p.nnz;
  }
  offs[B] = (int32_t)N;
  check_cuda(cudaMemcpyAsync(out.rowptr + N, &nnz, sizeof(int64_t), cudaMemcpyHostToDevice, c.stream), "copy");
  check_cuda(cudaMemcpyAsync(out.inst_off0, offs.data(), (B + 1) * sizeof(int32_t), cudaMemcpyHostToDevice, c.stream),
             "copy");
  sync(c);
}

}  // namespace mslice
