// Multislice modularity (Eq. multislice-modularity) of a level-0 labelling,
// from exact integer sums:
//   2mu Q = I + omega*J - gamma * sum_s S_s / 2m_s
//   I   = intra-snapshot weight over ordered pairs inside one community,
//   J   = ordered coupling pairs inside one community (general coupling:
//         omega*J = Jw/od, Jw the sum of the pairs' numerators),
//   S_s = sum_c Sigma_{c,s}^2 (128-bit),
//   2mu = sum_s 2m_s + n * sum_{s,r} omega^(sr)  (2*omega*n*(T-1) ordinal).
// Per-snapshot gamma: each slice term is multiplied by its gamma before the
// ascending sum, and the sum is subtracted as it is.
// Temporal CPM: S_s counts nodes (Sigma = node counts) and its slice term is
// S_s itself (a mass of 1) for every snapshot.
// The FP64 combination follows one fixed order (slice terms in ascending s,
// then omega*J, the numerator, the division), with explicitly rounded
// operations so no contraction changes the result.
//
// Global null model (plain modularity of the supra-graph, Eq. modularity):
//   Q = (I + omega*J) / 2mu - gamma * S' / (2M')^2,
//   S' = sum_c Sigma'_c^2 with Sigma' in units of 1/od, 2M' = od*2mu;
// FP64 order: I + omega*J, divided by 2mu; S' divided by the product
// 2M'*2M' (each converted first); times gamma; subtracted.
//
// Also: canonical relabelling (first occurrence order) and the order-free
// level checksum used by the step-level tests.
#include <cstring>
#include <vector>

#include "solver.h"

namespace mslice {

namespace {

// I and J of every instance (IJ: 2 words per instance): G lanes a row, as in
// k_build_rows: 8 where rows are short and there are more of them than warps, with
// the whole warp for a row of more than IJ_LONG entries and blocks of their own
// (k_IJ_hubs) for rows of more than HUB_ROW; a warp a row otherwise (from 32
// entries on average: at 62 a row 0.32 ms against 0.34).  Hubs of 100,000, 60,000,
// 20,000 and 40 of 3,000 (N = 300,000): Q 2.26 ms with a warp's four long rows in
// turn, 1.33 with a warp a row, 0.27 now.  A warp's rows ascend, and so do their
// instances: sums go out when the instance changes and at the end (one atomic a
// row on B words took 1.5 ms of a batch of 36, N = 1.5 M).
constexpr int64_t IJ_LONG = 64, IJ_DENSE = 32;
constexpr int IJ_HUB_PARTS = 8;
constexpr int64_t IJ_WARPS = 152 * (2048 / 32);  // resident at a time

__device__ __forceinline__ void ij_row(const LevelDev& g, const int32_t* labels, int32_t c, int64_t b, int64_t e,
                                       int t, int nt, ull& I, ull& J) {
  for (int64_t q = b + t; q < e; q += nt) {
    const int2 x = g.adj0[q];
    if (labels[x.x] == c) {
      if (x.y > 0)
        I += (ull)x.y;
      else
        J += g.cw ? (ull)g.cw[-x.y - 1] : 1ull;  // weighted by the pair's numerator with a table
    }
  }
}

// hubs, nhubs: see k_build_rows.
template <int G>
__global__ void k_IJ(LevelDev g, const int32_t* labels, ull* IJ, int32_t B, int32_t* hubs, ull* nhubs) {
  const int lane = threadIdx.x & 31, gl = lane % G;
  const int64_t groups = (int64_t)gridDim.x * blockDim.x / G;
  ull I = 0, J = 0;
  int32_t cur = 0;  // instance the warp's sums belong to
  auto flush = [&] {
    I = warp_sum(I);
    J = warp_sum(J);
    if (lane == 0) {
      if (I) atomicAdd(&IJ[2 * cur], I);
      if (J) atomicAdd(&IJ[2 * cur + 1], J);
    }
    I = J = 0;
  };
  for (int64_t v0 = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / G; v0 < g.N; v0 += groups) {
    const int64_t v = v0 + lane / G;
    const bool ok = v < g.N;
    const int64_t b = ok ? g.rowptr[v] : 0, e = ok ? g.rowptr[v + 1] : 0;
    const bool hub = hubs && e - b > HUB_ROW;
    const int32_t c = ok ? labels[v] : 0;
    const int32_t inst = B > 1 ? node_inst(g, (int32_t)(ok ? v : v0)) : 0;
    const int32_t first = __shfl_sync(0xffffffffu, inst, 0);
    const bool alike = __all_sync(0xffffffffu, inst == first);
    if (first != cur || !alike) {
      flush();
      cur = first;
    }
    if (hub && gl == 0) hubs[atomicAdd(nhubs, 1ull)] = (int32_t)v;
    if (!hub && (G == 32 || e - b <= IJ_LONG)) ij_row(g, labels, c, b, e, gl, G, I, J);
    if constexpr (G < 32) {
      unsigned wide = __ballot_sync(0xffffffffu, gl == 0 && !hub && e - b > IJ_LONG);
      while (wide) {
        const int src = __ffs(wide) - 1;
        wide &= wide - 1;
        ull Iw = 0, Jw = 0;
        ij_row(g, labels, __shfl_sync(0xffffffffu, c, src), __shfl_sync(0xffffffffu, b, src),
               __shfl_sync(0xffffffffu, e, src), lane, 32, Iw, Jw);
        Iw = warp_sum(Iw);
        Jw = warp_sum(Jw);
        if (lane == src) {
          I += Iw;
          J += Jw;
        }
      }
    }
    if (!alike) {  // rows of several instances: each lane's sums go out alone
      if (I) atomicAdd(&IJ[2 * inst], I);
      if (J) atomicAdd(&IJ[2 * inst + 1], J);
      I = J = 0;
    }
  }
  flush();
}

// The hubs' rows: blocks (x, 0 .. IJ_HUB_PARTS - 1) share one.
__global__ void __launch_bounds__(256)
    k_IJ_hubs(LevelDev g, const int32_t* labels, ull* IJ, int32_t B, const int32_t* hubs, const ull* nhubs) {
  const int64_t count = (int64_t)*nhubs;
  for (int64_t h = blockIdx.x; h < count; h += gridDim.x) {
    const int32_t v = hubs[h];
    const int64_t b = g.rowptr[v], e = g.rowptr[v + 1];
    const int64_t part = (e - b + gridDim.y - 1) / gridDim.y;
    const int64_t from = min(e, b + blockIdx.y * part), to = min(e, from + part);
    ull I = 0, J = 0;
    ij_row(g, labels, labels[v], from, to, threadIdx.x, blockDim.x, I, J);
    I = warp_sum(I);
    J = warp_sum(J);
    if ((threadIdx.x & 31) == 0) {
      const int32_t inst = B > 1 ? node_inst(g, v) : 0;
      if (I) atomicAdd(&IJ[2 * inst], I);
      if (J) atomicAdd(&IJ[2 * inst + 1], J);
    }
  }
}

// S_s += Sigma_{c,s}^2 over the table; per-block partial sums in shared
// memory when T is small enough, global 128-bit atomics otherwise.
__global__ void k_S(SigStore h, int32_t T, ull* S) {
  extern __shared__ ull sm[];  // 2*T words when used
  const bool use_sm = T <= 1024;
  if (use_sm) {
    for (int i = threadIdx.x; i < 2 * T; i += blockDim.x) sm[i] = 0;
    __syncthreads();
  }
  const uint64_t span = ss_span(h);
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < span; i += (uint64_t)gridDim.x * blockDim.x) {
    int32_t cc, s;
    long long val;
    if (!ss_entry(h, i, cc, s, val)) continue;
    const u128 sq = (u128)(ull)val * (u128)(ull)val;
    if (use_sm)
      atomic_add_u128(&sm[2 * s], sq);
    else
      atomic_add_u128(&S[2 * s], sq);
  }
  if (use_sm) {
    __syncthreads();
    for (int s = threadIdx.x; s < T; s += blockDim.x) {
      const u128 x = ((u128)sm[2 * s + 1] << 64) | sm[2 * s];
      if (x) atomic_add_u128(&S[2 * s], x);
    }
  }
}

struct QInst {
  int64_t n;
  int32_t T, soff;
  long long gn, gd, on, od;
  long long csum;      // n * sum_{s,r} omega_num^(sr): the coupling part of 2mu, in units of 1/od
  int32_t table, gtab;  // the instance has its own omega^(sr) table / per-snapshot gamma
};

// omega*J of an instance: with its own table, (double)Jw/od; otherwise
// (on*J)/od.  IJ's second word holds Jw when the solve has a coupling table
// (weighted) -- an instance without one then had every pair weigh on, so
// J = Jw/on.
__device__ __forceinline__ double omega_J(const QInst& p, ull Jword, int32_t weighted) {
  if (p.table) return __ddiv_rn(__ull2double_rn(Jword), __ll2double_rn(p.od));
  const ull J = weighted ? (p.on > 0 ? Jword / (ull)p.on : 0ull) : Jword;
  return __ddiv_rn(__dmul_rn(__ll2double_rn(p.on), __ull2double_rn(J)), __ll2double_rn(p.od));
}

// Q of every instance (one thread each), in the fixed FP64 order.  S holds
// one 128-bit sum per null slice: per snapshot (Q_MS) or per instance
// (global model).  gs: per-snapshot gamma (num, den) pairs, when any
// instance has them.
// The slice terms of Q_MS, one thread per snapshot: S_s / 2m_s (CPM: S_s,
// a mass of 1), times gamma_s when the instance has per-snapshot gamma.
// k_Q adds them in ascending s, so the result is that of one sequential
// evaluation.
__global__ void k_slice_terms(const ull* S, const int64_t* two_m, int32_t T, const int32_t* slice_inst,
                              const QInst* qi, int32_t cpm, const long long* gs, double* terms) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < T; s += gridDim.x * blockDim.x) {
    const long long t = two_m[s];
    double term = 0.0;
    if (t > 0 || cpm) {
      const u128 x = ((u128)S[2 * s + 1] << 64) | S[2 * s];
      term = cpm ? u128_to_double(x) : __ddiv_rn(u128_to_double(x), __ll2double_rn(t));
      if (qi[slice_inst ? slice_inst[s] : 0].gtab)
        term = __dmul_rn(__ddiv_rn(__ll2double_rn(gs[2 * s]), __ll2double_rn(gs[2 * s + 1])), term);
    }
    terms[s] = term;
  }
}

__global__ void k_Q(const ull* IJ, const ull* S, const int64_t* two_m, const QInst* qi, int32_t B, int32_t global,
                    int32_t cpm, int32_t weighted, const double* terms, double* Q) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B) return;
  const QInst p = qi[i];
  if (global) {
    long long sum2m = 0;
    for (int s = p.soff; s < p.soff + p.T; ++s) sum2m += two_m[s];
    const long long twoM = p.od * sum2m + p.csum;
    if (twoM == 0) {
      Q[i] = 0.0;
      return;
    }
    const u128 x = ((u128)S[2 * i + 1] << 64) | S[2 * i];
    const double wJ = omega_J(p, IJ[2 * i + 1], weighted);
    const double gam = __ddiv_rn(__ll2double_rn(p.gn), __ll2double_rn(p.gd));
    const double twomu = __ddiv_rn(__ll2double_rn(twoM), __ll2double_rn(p.od));
    const double first = __ddiv_rn(__dadd_rn(__ull2double_rn(IJ[2 * i]), wJ), twomu);
    const double tM = __ll2double_rn(twoM);
    const double null = __ddiv_rn(u128_to_double(x), __dmul_rn(tM, tM));
    Q[i] = __dsub_rn(first, __dmul_rn(gam, null));
    return;
  }
  double nullsum = 0.0;
  long long sum2m = 0;
  // (eight loads in flight: the additions are a chain, the loads need not be)
  for (int s0 = p.soff; s0 < p.soff + p.T; s0 += 8) {
    long long t[8];
    double term[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const bool in = s0 + u < p.soff + p.T;
      t[u] = in ? two_m[s0 + u] : 0;
      term[u] = in ? terms[s0 + u] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (s0 + u >= p.soff + p.T) break;
      sum2m += t[u];
      if (t[u] > 0 || cpm) nullsum = __dadd_rn(nullsum, term[u]);  // ascending s
    }
  }
  const double wJ = omega_J(p, IJ[2 * i + 1], weighted);
  const double gam = __ddiv_rn(__ll2double_rn(p.gn), __ll2double_rn(p.gd));
  const long long twomu_num = p.od * sum2m + p.csum;
  if (twomu_num == 0) {
    Q[i] = 0.0;
    return;
  }
  const double twomu = __ddiv_rn(__ll2double_rn(twomu_num), __ll2double_rn(p.od));
  const double num = __dsub_rn(__dadd_rn(__ull2double_rn(IJ[2 * i]), wJ), p.gtab ? nullsum : __dmul_rn(gam, nullsum));
  Q[i] = __ddiv_rn(num, twomu);
}

__global__ void k_first(const int32_t* x, int64_t N, int32_t* first) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x)
    // (the smallest index is mostly there already; one atomic a node serialised
    // on the largest communities, 1.2 ms for 2.4 M nodes)
    if ((int32_t)v < __ldcg(&first[x[v]])) atomicMin(&first[x[v]], (int32_t)v);
}

__global__ void k_first_flag(const int32_t* x, const int32_t* first, int64_t N, int32_t* flag) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x)
    flag[v] = first[x[v]] == (int32_t)v ? 1 : 0;
}

// Renumbered labels, counted from the instance's first community.
__global__ void k_canon(const int32_t* x, const int32_t* first, const int32_t* rank, int64_t N, const int32_t* inst,
                        const int32_t* inst_off, int32_t* out) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x)
    out[v] = rank[first[x[v]]] - (inst ? rank[inst_off[inst[v]]] : 0);
}

__global__ void k_checksum(LevelDev g, ull* out) {
  ull h = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < g.N; v += (int64_t)gridDim.x * blockDim.x) {
    for (int64_t e = g.rowptr[v]; e < g.rowptr[v + 1]; ++e)
      h += mix64(mix64(mix64((ull)g.W[e]) ^ (ull)g.col[e]) ^ (ull)v);
    for (int64_t j = g.sptr[v]; j < g.sptr[v + 1]; ++j)
      h += mix64(mix64(mix64((ull)g.sval[j]) ^ (ull)g.sidx[j]) ^ ((ull)v + 0x9E3779B97F4A7C15ULL));
  }
  h = warp_sum(h);
  if ((threadIdx.x & 31) == 0) atomicAdd(out, h);
}

unsigned gsz(int64_t n) {
  int64_t g = (n + 255) / 256;
  if (g > 152 * 16) g = 152 * 16;
  return (unsigned)(g < 1 ? 1 : g);
}

}  // namespace

void modularity(Solver& S, const int32_t* labels0, double* Q) {
  Ctx& c = *S.c;
  const SupraGraph& G = *S.G0;
  const int32_t B = G.B;
  LevelDev g = level0_view(G, S);  // (S.Tn / S.kn set up by setup_null_model)
  configure_stores(S, G.N);
  sigma_rebuild(S, Level{g}, labels0);
  const int32_t Tn = S.Tn;
  // I and J per instance, S per null slice, the hubs' number
  const size_t accs = 2 * (size_t)B + 2 * (size_t)Tn;
  ull* acc = c.ws->get<ull>("q_acc", accs + 1);
  double* dQ = c.ws->get<double>("q_out", B);
  QInst* dqi = c.ws->get<QInst>("q_inst", B);
  std::vector<QInst> qi(B);
  for (int32_t i = 0; i < B; ++i) {
    const InstInfo& in = G.inst[i];
    qi[i] = QInst{in.n, in.T, in.soff, S.gn_h[i], S.gd_h[i], S.on_h[i], S.od_h[i], S.csum_h[i],
                  (int32_t)S.has_cw_h[i], (int32_t)S.has_gs_h[i]};
  }
  check_cuda(cudaMemcpyAsync(dqi, qi.data(), B * sizeof(QInst), cudaMemcpyHostToDevice, c.stream), "copy");
  check_cuda(cudaMemsetAsync(acc, 0, (accs + 1) * sizeof(ull), c.stream), "memset");
  if (G.N > 0) {
    const bool all_warps = G.N <= IJ_WARPS;
    int32_t* hubs = G.hubs && !all_warps ? c.ws->get<int32_t>("q_hubs", G.nnz / HUB_ROW + 1) : nullptr;
    if (all_warps || G.nnz > IJ_DENSE * G.N)
      launch(c, k_IJ<32>, dim3(gsz(G.N * 32)), dim3(256), 0, g, labels0, acc, B, hubs, acc + accs);
    else
      launch(c, k_IJ<8>, dim3(gsz(G.N * 8)), dim3(256), 0, g, labels0, acc, B, hubs, acc + accs);
    if (hubs)
      launch(c, k_IJ_hubs, dim3(76, IJ_HUB_PARTS), dim3(256), 0, g, labels0, acc, B, (const int32_t*)hubs,
             (const ull*)(acc + accs));
  }
  const size_t smem = Tn <= 1024 ? 2 * (size_t)Tn * sizeof(ull) : 0;
  const int64_t span = S.sig.d ? S.sig.rows * S.sig.T : (int64_t)S.sig.h.cap;
  launch(c, k_S, dim3(gsz(span)), dim3(256), smem, S.sig, Tn, acc + 2 * B);
  double* terms = c.ws->get<double>("q_terms", G.T > 0 ? G.T : 1);
  if (!S.p.global_null && G.T > 0)
    launch(c, k_slice_terms, dim3(grid_for(G.T, 256)), dim3(256), 0, (const ull*)(acc + 2 * B),
           (const int64_t*)G.two_m, G.T, (const int32_t*)(G.B > 1 ? G.slice_inst : nullptr), (const QInst*)dqi,
           (int32_t)(S.p.cpm ? 1 : 0), (const long long*)S.gs_d, terms);
  launch(c, k_Q, dim3(grid_for(B, 128)), dim3(128), 0, (const ull*)acc, (const ull*)(acc + 2 * B),
         (const int64_t*)G.two_m, (const QInst*)dqi, B, (int32_t)(S.p.global_null ? 1 : 0), (int32_t)(S.p.cpm ? 1 : 0),
         (int32_t)(S.cw_d ? 1 : 0), (const double*)terms, dQ);
  // B values go straight to the caller's (pageable) array
  check_cuda(cudaMemcpyAsync(Q, dQ, B * sizeof(double), cudaMemcpyDeviceToHost, c.stream), "copy");
  sync(c);
}

void canonicalise(Solver& S, const int32_t* x, int32_t* out, int64_t N) {
  Ctx& c = *S.c;
  if (N == 0) return;
  int32_t* first = S.tmp32a;
  int32_t* rank = S.tmp32b;
  fill_i32(c, first, INT32_MAX, N);
  launch(c, k_first, dim3(gsz(N)), dim3(256), 0, x, N, first);
  int32_t* flag = S.freelist;
  launch(c, k_first_flag, dim3(gsz(N)), dim3(256), 0, x, (const int32_t*)first, N, flag);
  // rank has N + 1 entries: rank[N] counts every community
  check_cuda(cudaMemsetAsync(flag + N, 0, sizeof(int32_t), c.stream), "memset");
  scan_excl(c, flag, rank, N + 1, (int32_t*)nullptr);
  const SupraGraph& G = *S.G0;
  launch(c, k_canon, dim3(gsz(N)), dim3(256), 0, x, (const int32_t*)first, (const int32_t*)rank, N,
         (const int32_t*)G.inst0, (const int32_t*)G.inst_off0, out);
}

uint64_t level_checksum(Solver& S, const Level& L) {
  Ctx& c = *S.c;
  ull* d = c.ws->get<ull>("ck_out", 1);
  check_cuda(cudaMemsetAsync(d, 0, sizeof(ull), c.stream), "memset");
  if (L.d.N > 0) launch(c, k_checksum, dim3(gsz(L.d.N)), dim3(256), 0, L.d, d);
  return *static_cast<const ull*>(readback(c, d, sizeof(ull)));
}

}  // namespace mslice
