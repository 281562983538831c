// Max/min pivots and pivot distances of graphs that one block's shared memory
// holds (keys, offsets, queues and 16-bit neighbours: 12 bytes a node and 2 an
// edge end, up to some 14,000 nodes).  A level of the cluster's max/min or of
// a block per source with its graph in L2 costs 1.2 to 1.8 us in latency,
// however small the level; here it is 0.2 to 0.3 us (block_search.cuh).
//   * k_small_maxmin: one block, the chain of k pruned searches
//   * k_small_bfs: a block per source at a time
// Max/min / distances, ms with the call's host work, in the cluster and by pulled
// levels or a block per source, and here: 32 x 32 grid, k = 50: 0.92 / 0.33 ->
// 0.26 / 0.07; rgg, n = 8,000, k = 200: 3.33 / 0.61 -> 1.32 / 0.26; ba, n = 5,000,
// k = 200: 1.34 / 0.20 -> 0.55 / 0.16; star, n = 14,000, k = 50: 0.24 / 0.12 ->
// 0.13 / 0.08; path, n = 14,000, k = 50: 55.6 / 17.3 -> 16.8 / 5.8.
#include <algorithm>

#include "bfs.cuh"
#include "block_search.cuh"

namespace ssm {

constexpr int kSmallThreads = 512;
constexpr int64_t kSmallSmem = 227 * 1024 - 1024;

static int64_t small_bytes(int32_t n, int64_t m2) { return block_search_bytes(n) + 2 * m2; }

bool small_graph_fits(int32_t n, int64_t m2) { return small_bytes(n, m2) <= kSmallSmem; }

struct SmallArgs {
  int32_t n, k, start;
  int64_t m2;
  const int32_t *rowptr, *colidx, *sources;
  int32_t *pivots;
  uint16_t *dist;
  int32_t *status;
};

// the graph into shared memory (a neighbour outside the graph: recorded, read as node 0)
__device__ __forceinline__ BlockSearch small_load(const SmallArgs &A, unsigned char *sm, int *len, int *hub) {
  const int n = A.n;
  int *off = reinterpret_cast<int *>(sm) + n + 1;
  uint16_t *q = reinterpret_cast<uint16_t *>(off + n + 1), *nbr = q + 2 * n;
  for (int i = threadIdx.x; i <= n; i += kSmallThreads) off[i] = max(0, min(__ldg(A.rowptr + i), (int)A.m2));
  const int m2 = (int)A.m2;
  bool bad = false;
  for (int t0 = threadIdx.x; t0 < m2; t0 += 8 * kSmallThreads) {  // eight loads in flight
    unsigned c[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) c[q] = (unsigned)__ldg(A.colidx + min(t0 + q * kSmallThreads, m2 - 1));
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      bad |= c[q] >= (unsigned)n;
      if (t0 + q * kSmallThreads < m2) nbr[t0 + q * kSmallThreads] = (uint16_t)(c[q] < (unsigned)n ? c[q] : 0u);
    }
  }
  if (bad) dev_fail(A.status, SSM_E_GRAPH);
  if (threadIdx.x < 3) len[threadIdx.x] = 0;
  return BlockSearch{reinterpret_cast<int *>(sm), off, nbr, q, q + n, len, hub};
}

__global__ void __launch_bounds__(kSmallThreads) k_small_maxmin(SmallArgs A) {
  extern __shared__ __align__(16) unsigned char sg_smem[];
  __shared__ int s_len[3], s_hub[kBsMaxHubs];
  __shared__ unsigned s_best[2];
  const BlockSearch B = small_load(A, sg_smem, s_len, s_hub);
  const int n = A.n;
  for (int i = threadIdx.x; i < n; i += kSmallThreads) B.key[i] = kBsInf;
  if (threadIdx.x < 2) s_best[threadIdx.x] = 0u;
  __syncthreads();
  const bool hubs = block_search_hubs(B.off, n);
  int slot = 0, p = A.start;
  for (int a = 0; a < A.k; ++a) {
    if (threadIdx.x == 0) A.pivots[a] = p;
    if (a > 0 && a == A.k - 1) break;  // the last pivot needs no search
    if (hubs) block_search<true>(B, p, 0, 0, slot);
    else block_search<false>(B, p, 0, 0, slot);
    if (threadIdx.x == 0) s_best[(a + 1) & 1] = 0u;  // last read before this search
    // the farthest node, ties to the lowest id (distances and ids below 2^16)
    unsigned best = 0u;
    for (int i = threadIdx.x; i < n; i += kSmallThreads)
      best = max(best, ((unsigned)min(B.key[i], 0xFFFF) << 16) | (0xFFFFu - (unsigned)i));
    best = __reduce_max_sync(0xffffffffu, best);
    if ((threadIdx.x & 31) == 0) atomicMax(s_best + (a & 1), best);
    __syncthreads();
    best = s_best[a & 1];
    if ((best >> 16) == 0xFFFFu) {  // some node was not reached
      if (threadIdx.x == 0) dev_fail(A.status, SSM_E_DISCONNECTED);
      break;
    }
    p = (int)(0xFFFFu - (best & 0xFFFFu));
  }
}

__global__ void __launch_bounds__(kSmallThreads) k_small_bfs(SmallArgs A) {
  extern __shared__ __align__(16) unsigned char sg_smem[];
  __shared__ int s_len[3], s_hub[kBsMaxHubs];
  const BlockSearch B = small_load(A, sg_smem, s_len, s_hub);
  const int n = A.n;
  __syncthreads();
  const bool hubs = block_search_hubs(B.off, n);
  int slot = 0;
  bool lost = false;
  for (int si = blockIdx.x; si < A.k; si += gridDim.x) {
    for (int i = threadIdx.x; i < n; i += kSmallThreads) B.key[i] = kBsInf;
    int p = __ldg(A.sources + si);
    if ((unsigned)p >= (unsigned)n) {  // a source outside the graph: recorded, searched from node 0
      if (threadIdx.x == 0) dev_fail(A.status, SSM_E_ARG);
      p = 0;
    }
    __syncthreads();
    if (hubs) block_search<true>(B, p, 0, 0, slot);
    else block_search<false>(B, p, 0, 0, slot);
    uint16_t *row = A.dist + (size_t)si * n;
    for (int i = threadIdx.x; i < n; i += kSmallThreads) {
      const int d = B.key[i];
      lost |= d == kBsInf;
      row[i] = (uint16_t)min(d, 0xFFFF);
    }
    __syncthreads();
  }
  if (lost) dev_fail(A.status, SSM_E_DISCONNECTED);
}

int launch_small_maxmin(int32_t n, int64_t m2, const int32_t *rowptr, const int32_t *colidx, int32_t k, int32_t start,
                        int32_t *pivots, int32_t *status, cudaStream_t s) {
  const SmallArgs A{n, k, start, m2, rowptr, colidx, nullptr, pivots, nullptr, status};
  SSM_TRY_CUDA(allow_dynamic_smem((const void *)k_small_maxmin));
  note_launch(), k_small_maxmin<<<1, kSmallThreads, (size_t)small_bytes(n, m2), s>>>(A);
  SSM_TRY_CUDA(cudaGetLastError());
  note_pivot_config(1, 4);
  return SSM_OK;
}

// blocks that run at once
static int small_bfs_slots(size_t smem) {
  int per_sm = 0;
  if (allow_dynamic_smem((const void *)k_small_bfs) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_small_bfs, kSmallThreads, smem) != cudaSuccess)
    (void)cudaGetLastError();
  return std::max(1, per_sm) * num_sms();
}

// Up to four sources per block: with more, four blocks per SM on a graph in L2
// (bfs.cu) catch up where only one graph per SM fits here (1,024 sources,
// 100 x 100 grid: 0.82 there, 0.86 ms here); one where rows are long, since the
// other way looks at an edge for 32 sources at once (clique of 300: 200 sources
// 0.11 there, 0.13 here; 50 sources 0.10, 0.09)
bool small_bfs_fits(int32_t n, int64_t m2, int32_t k) {
  const int64_t rounds = m2 > 128 * (int64_t)n ? 1 : 4;
  return small_graph_fits(n, m2) && k <= rounds * (int64_t)small_bfs_slots((size_t)small_bytes(n, m2));
}

int launch_small_bfs(int32_t n, int64_t m2, const int32_t *rowptr, const int32_t *colidx, int32_t k,
                     const int32_t *sources, uint16_t *dist, int32_t *status, cudaStream_t s) {
  const SmallArgs A{n, k, 0, m2, rowptr, colidx, sources, nullptr, dist, status};
  const size_t smem = (size_t)small_bytes(n, m2);
  note_launch(), k_small_bfs<<<std::min(k, small_bfs_slots(smem)), kSmallThreads, smem, s>>>(A);
  SSM_TRY_CUDA(cudaGetLastError());
  return SSM_OK;
}

}  // namespace ssm
