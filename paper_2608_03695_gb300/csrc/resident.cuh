// What the resident kernels share (lm_rounds.cu, refine.cu): one cooperative
// launch that runs a phase of a small level from end to end, with grid barriers
// where the launches of the large levels' path are.  One block of 512 threads
// per SM at most; its decision tables (8,192 slots) serve a block per node, a
// warp per node (512 slots each) or 8 lanes per node (64 slots each).
#pragma once
#include <cooperative_groups.h>

#include <algorithm>

#include "lm.cuh"

namespace mslice {

constexpr int RT = 512;  // threads per block
constexpr int RW = RT / 32;
constexpr int R_SLOTS = TIER4_SMEM_SLOTS;
constexpr int R_PER_WARP = R_SLOTS / RW;
constexpr int R_BUCKET_ITEMS = 4;
static_assert(R_PER_WARP >= 1 << T2_BITS, "a warp's share of the block's table holds tier 2's");

__device__ __forceinline__ void resident_bar() {
  if (gridDim.x == 1)
    __syncthreads();
  else
    cooperative_groups::this_grid().sync();
}

// Lists the nodes v in [0, N) by segment: seg_of(v) gives the segment and, at
// least nseg, leaves the node out.  A block's share at a time: segments counted
// in shared memory (cnt, base: nseg words each), one reservation per block and
// segment.
template <class SegOf>
__device__ __forceinline__ void resident_list(int64_t N, int nseg, int32_t* lists, int64_t row_stride,
                                              const TierOff& off, int32_t* cursors, int32_t* cnt, int32_t* base,
                                              SegOf&& seg_of) {
  const int64_t chunk = (int64_t)RT * R_BUCKET_ITEMS;
  for (int64_t c0 = (int64_t)blockIdx.x * chunk; c0 < N; c0 += (int64_t)gridDim.x * chunk) {
    for (int i = threadIdx.x; i < nseg; i += RT) cnt[i] = 0;
    __syncthreads();
    int sg[R_BUCKET_ITEMS], rank[R_BUCKET_ITEMS];
#pragma unroll
    for (int k = 0; k < R_BUCKET_ITEMS; ++k) {
      const int64_t v = c0 + (int64_t)k * RT + threadIdx.x;
      sg[k] = v < N ? seg_of((int32_t)v) : SEG_FROZEN;
      if (sg[k] < nseg) rank[k] = atomicAdd(&cnt[sg[k]], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nseg; i += RT) base[i] = cnt[i] ? atomicAdd(&cursors[i], cnt[i]) : 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < R_BUCKET_ITEMS; ++k)
      if (sg[k] < nseg) {
        const int q = sg[k] / NTIERS, t = sg[k] % NTIERS;
        lists[(int64_t)q * row_stride + off.off[t] + base[sg[k]] + rank[k]] =
            (int32_t)(c0 + (int64_t)k * RT + threadIdx.x);
      }
    __syncthreads();
  }
}

// The lists of class q.
__device__ __forceinline__ TierSegs resident_segs(int32_t* lists, int64_t row_stride, const TierOff& off,
                                                  const int32_t* cursors, int q) {
  TierSegs sg;
#pragma unroll
  for (int t = 0; t < NTIERS; ++t) {
    sg.list[t] = lists + (int64_t)q * row_stride + off.off[t];
    sg.count[t] = cursors + q * NTIERS + t;
  }
  return sg;
}

// The nodes of one class, dealt out by tier: a block per node of tiers 4 and 3,
// a warp per node of tier 2, 8 lanes per node of tiers 1 and 0.  The last blocks
// take the first of tier 2, and the low tiers start with the warps after those:
// a node is a chain of dependent loads of 5-15 us, so two in one warp while
// others idle double the sub-round.  For the same reason the low tiers get a warp
// per node while there are as many warps: the four groups of a warp whose nodes
// walk lists of different lengths take turns (1,000 nodes x 4 snapshots 5.2 ->
// 4.8 ms a solve; at two or more nodes a warp 8 lanes each are faster again).
template <class ByBlock, class ByWarp, class ByEight>
__device__ __forceinline__ void resident_deal(const TierSegs& sg, ByBlock&& by_block, ByWarp&& by_warp,
                                              ByEight&& by_eight) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int t = NTIERS - 1; t >= NTIERS - 2; --t) {
    const int n = *sg.count[t];
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
      const int32_t v = sg.list[t][i];
      __syncthreads();
      by_block(v);
    }
  }
  __syncthreads();
  const int gw = (gridDim.x - 1 - blockIdx.x) * RW + w, warps = gridDim.x * RW;
  const int n2 = *sg.count[2];
  for (int i = gw; i < n2; i += warps) by_warp(sg.list[2][i]);
  const int n0 = *sg.count[0], n = n0 + *sg.count[1];
  const int gi = lane >> 3, g0 = (gw + warps - n2 % warps) % warps;
  if (n <= warps) {
    if (g0 < n) by_warp(g0 < n0 ? sg.list[0][g0] : sg.list[1][g0 - n0]);
    return;
  }
  for (int i = g0 * 4 + gi; i < n; i += warps * 4) by_eight(i < n0 ? sg.list[0][i] : sg.list[1][i - n0], gi, lane & 7);
  __syncwarp();
}

// Blocks for a level of N nodes, `big` of them decided by a block: a block or a
// warp per node of a class, up to one block per SM (fewer blocks make the
// barriers cheaper).
inline unsigned resident_grid(int64_t N, int64_t big, int32_t K, int32_t sms) {
  const int64_t blocks = (big + K - 1) / K, warps = (N - big + K - 1) / K;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(blocks + (warps + RW - 1) / RW, sms));
}

}  // namespace mslice
