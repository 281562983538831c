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

struct BlockSearch {
  int *key;             // [n] a node's key: distance * 2^shift + source
  const int *off;       // [n + 1] row offsets
  const uint16_t *nbr;  // neighbours (in shared or global memory)
  uint16_t *q0, *q1;    // [n] queues
  int *len;             // [3] queue lengths, zero but for the search's own use
};

// The search from p with the keys level << shift | source: it lowers keys in
// place and goes on only from nodes whose key it lowered.  Narrow levels take
// eight lanes a node (a mesh's 14 nodes in one step of latency), wide ones two
// (leaves of a hub would leave seven of eight idle).  slot is the queue length
// in use, carried from search to search.  Called by every thread of the block, with a
// barrier between two calls and none of p's key's readers after it; the keys
// are final when it returns.
__device__ __forceinline__ void block_search(const BlockSearch &B, int p, int shift, int source, int &slot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    B.key[p] = source;
    B.q0[0] = (uint16_t)p;
    B.len[slot] = 1;
  }
  __syncthreads();
  for (int level = 1;; ++level) {
    const int ncur = B.len[slot], nslot = slot == 2 ? 0 : slot + 1;
    if (ncur == 0) break;
    if (threadIdx.x == 0) B.len[nslot == 2 ? 0 : nslot + 1] = 0;
    const uint16_t *qc = level & 1 ? B.q0 : B.q1;
    uint16_t *qn = level & 1 ? B.q1 : B.q0;
    const int nk = (level << shift) | source;
    // whole warps: lowers the neighbours at j, j + 32, ... below e, U in
    // flight, and queues those it lowered
    auto visit = [&](auto slots, int j, int e) {
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
      if (lane == 0) base = atomicAdd(B.len + nslot, (int)total);
      base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
      for (int q = 0; q < U; ++q) {
        if (u[q] >= 0) qn[base + __popc(m[q] & ((1u << lane) - 1u))] = (uint16_t)u[q];
        base += __popc(m[q]);
      }
    };
    const int gs = ncur > kBsWide ? 1 : 3, sub = lane & ((1 << gs) - 1);
    for (int t0 = warp << (5 - gs); t0 < ncur; t0 += (int)blockDim.x >> gs) {
      const int t = t0 + (lane >> gs);
      int b = 0, e = 0;
      if (t < ncur) {
        const int v = qc[t];
        b = B.off[v];
        e = B.off[v + 1];
      }
      const bool lng = e - b > (kBsPerLane << gs);
      for (int j = lng ? e : b + sub; __any_sync(0xffffffffu, j < e); j += 1 << gs) visit(std::integral_constant<int, 1>(), j, e);
      for (unsigned m = __ballot_sync(0xffffffffu, lng && sub == 0); m; m &= m - 1u) {
        const int jb = __shfl_sync(0xffffffffu, b, __ffs(m) - 1), je = __shfl_sync(0xffffffffu, e, __ffs(m) - 1);
        for (int j = jb; j < je; j += 32 * kBsLongSlots) visit(std::integral_constant<int, kBsLongSlots>(), j + lane, je);
      }
    }
    __syncthreads();
    slot = nslot;
  }
}

// shared memory of keys, offsets and queues of n nodes
__host__ __device__ constexpr int64_t block_search_bytes(int64_t n) { return 8 * (n + 1) + 4 * n; }

}  // namespace ssm
