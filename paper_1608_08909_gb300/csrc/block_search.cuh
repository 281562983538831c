// Breadth-first search of a small graph by one block, everything in shared
// memory: the max/min chains and distance rows of graphs of up to some ten
// thousand nodes are chains of short levels, so a level's latency is all that
// counts -- shared-memory reads, one block barrier per level (three rotating
// queue lengths) and one queue atomic per warp.
#pragma once
#include <type_traits>

#include "common.cuh"

namespace ssm {

constexpr int kBsInf = 0x7FFFFFFF;  // the key of a node that no search has reached
constexpr int kBsWide = 256;        // frontiers above this: two lanes a node, else eight
constexpr int kBsPerLane = 8;       // rows above this many entries per lane are walked by the whole warp,
constexpr int kBsLongSlots = 8;     // with this many entries per lane in flight
constexpr int kBsHub = 1024;        // rows above this: all warps of the block, after the level's other rows
constexpr int kBsMaxHubs = 32;      // (as many in a level; further ones like the rest)
constexpr int kBsHubBits = 24;      // a queue length's upper bits count the hubs that still add to it

struct BlockSearch {
  int *key;             // [n] a node's key: distance * 2^shift + source
  const int *off;       // [n + 1] row offsets
  const uint16_t *nbr;  // neighbours (in shared or global memory)
  uint16_t *q0, *q1;    // [n] queues
  int *len;             // [3] queue lengths, zero but for the search's own use
  int *hub;             // [kBsMaxHubs] hubs of a level
};

// The search from p with the keys level << shift | source: it lowers keys in
// place and goes on only from nodes whose key it lowered.  Narrow levels take
// eight lanes a node (a mesh's 14 nodes in one step of latency), wide ones two
// (leaves of a hub would leave seven of eight idle).  A hub's row, in one warp 55
// steps on a star of 14,000 nodes, waits until the level's other rows are done
// and is then every warp's.  slot is the queue length
// in use, carried from search to search.  Called by every thread of the block, with a
// barrier between two calls and none of p's key's readers after it; the keys
// are final when it returns.  HUBS: whether a row is above kBsHub (looking out
// for them costs 7 % of a narrow level).
template <bool HUBS>
__device__ __forceinline__ void block_search(const BlockSearch &B, int p, int shift, int source, int &slot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    B.key[p] = source;
    B.q0[0] = (uint16_t)p;
    B.len[slot] = 1;
  }
  __syncthreads();
  for (int level = 1;; ++level) {
    const int nslot = slot == 2 ? 0 : slot + 1;
    uint16_t *const qc = level & 1 ? B.q0 : B.q1, *const qn = level & 1 ? B.q1 : B.q0;
    // whole warps: lowers the neighbours at j, j + 32, ... below e to nk, U in
    // flight, and queues those it lowered in q, of length *len
    auto visit = [&](auto slots, int j, int e, int nk, uint16_t *q_, int *len) {
      constexpr int U = decltype(slots)::value;
      int u[U];
      unsigned m[U], total = 0u;
#pragma unroll
      for (int q = 0; q < U; ++q) u[q] = j + 32 * q < e ? B.nbr[j + 32 * q] : -1;
#pragma unroll
      for (int q = 0; q < U; ++q)
        if (u[q] >= 0 && !(B.key[u[q]] > nk && atomicMin(B.key + u[q], nk) > nk)) u[q] = -1;
#pragma unroll
      for (int q = 0; q < U; ++q) {
        m[q] = __ballot_sync(0xffffffffu, u[q] >= 0);
        total += __popc(m[q]);
      }
      if (total == 0u) return;
      int base = 0;
      if (lane == 0) base = atomicAdd(len, (int)total);
      if (HUBS) base &= (1 << kBsHubBits) - 1;
      base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
      for (int q = 0; q < U; ++q) {
        if (u[q] >= 0) q_[base + __popc(m[q] & ((1u << lane) - 1u))] = (uint16_t)u[q];
        base += __popc(m[q]);
      }
    };
    int ncur = B.len[slot];
    if (HUBS && ncur >> kBsHubBits) {  // the last level's hubs first
      const int nh = min(ncur >> kBsHubBits, kBsMaxHubs);
      for (int h = 0; h < nh; ++h) {
        const int v = B.hub[h], je = B.off[v + 1];
        for (int j = B.off[v] + 32 * kBsLongSlots * warp; j < je; j += (int)blockDim.x * kBsLongSlots)
          visit(std::integral_constant<int, kBsLongSlots>(), j + lane, je, ((level - 1) << shift) | source, qc, B.len + slot);
      }
      __syncthreads();
      ncur = B.len[slot] & ((1 << kBsHubBits) - 1);
    }
    if (ncur == 0) break;
    if (threadIdx.x == 0) B.len[nslot == 2 ? 0 : nslot + 1] = 0;
    const int nk = (level << shift) | source;
    const int gs = ncur > kBsWide ? 1 : 3, sub = lane & ((1 << gs) - 1);
    for (int t0 = warp << (5 - gs); t0 < ncur; t0 += (int)blockDim.x >> gs) {
      const int t = t0 + (lane >> gs);
      int v = 0, b = 0, e = 0;
      if (t < ncur) {
        v = qc[t];
        b = B.off[v];
        e = B.off[v + 1];
      }
      const bool lng = e - b > (kBsPerLane << gs);
      for (int j = lng ? e : b + sub; __any_sync(0xffffffffu, j < e); j += 1 << gs) visit(std::integral_constant<int, 1>(), j, e, nk, qn, B.len + nslot);
      for (unsigned m = __ballot_sync(0xffffffffu, lng && sub == 0); m; m &= m - 1u) {
        const int jb = __shfl_sync(0xffffffffu, b, __ffs(m) - 1), je = __shfl_sync(0xffffffffu, e, __ffs(m) - 1);
        if (HUBS && je - jb > kBsHub) {
          const int hv = __shfl_sync(0xffffffffu, v, __ffs(m) - 1);
          int h = 0;
          if (lane == 0) {
            h = atomicAdd(B.len + nslot, 1 << kBsHubBits) >> kBsHubBits;
            if (h < kBsMaxHubs) B.hub[h] = hv;
            else atomicSub(B.len + nslot, 1 << kBsHubBits);
          }
          if (__shfl_sync(0xffffffffu, h, 0) < kBsMaxHubs) continue;
        }
        for (int j = jb; j < je; j += 32 * kBsLongSlots) visit(std::integral_constant<int, kBsLongSlots>(), j + lane, je, nk, qn, B.len + nslot);
      }
    }
    __syncthreads();
    slot = nslot;
  }
}

// whether any row is above kBsHub, for every thread of the block
__device__ __forceinline__ bool block_search_hubs(const int *off, int n) {
  bool hub = false;
  for (int i = threadIdx.x; i < n; i += blockDim.x) hub |= off[i + 1] - off[i] > kBsHub;
  return __syncthreads_or(hub ? 1 : 0) != 0;
}

// shared memory of keys, offsets and queues of n nodes
__host__ __device__ constexpr int64_t block_search_bytes(int64_t n) { return 8 * (n + 1) + 4 * n; }

}  // namespace ssm
