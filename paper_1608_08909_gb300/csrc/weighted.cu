// Weighted graphs (Algorithm 1 line 2: "weighted MSSP"; Section 3's weights
// with general edge lengths).
//
// Edge lengths l_ij are float32.  A distance is the least float32 path sum:
// d(v) = fl(d(u) + l_uv) along a path walked from the source, minimised over
// paths.  Rounding is monotone and never decreases a sum, so every search
// that only lowers labels and stops when no edge can lower one reaches that
// same minimum; the label-correcting search below and a Dijkstra therefore
// agree bit for bit.
//
//   ssm_edge_lengths        lengths of the CSR edges from the input list
//                           (a repeated edge keeps its shortest length)
//   k_sssp_multi            one block per source: rounds of relaxations of
//                           a frontier queue, labels lowered by atomicMin
//                           on their bit patterns (non-negative floats order
//                           like their bits); with the label row holding
//                           min over the earlier pivots it is max/min's
//                           pruned search (k_sssp_maxmin, for graphs whose
//                           labels do not fit one cluster's shared memory)
//   k_wmm_argmax            the next max/min pivot: max over v of
//                           (mind_v, -v) as one 64-bit key
//   k_wregion_keys, bitonic sort, k_wcounts
//                           regions (ties to the lowest pivot index) and
//                           s_ia = |{j in R(a) : 2 d_ja <= d_ia}| by binary
//                           search in each region's sorted distances; s = 0
//                           where the pivot is i or a neighbour of i
//   k_wsweep, k_wsweep_f32  Eq. 4 with w_ij = l_ij^-2 and w'_ia = s_ia/d_ia^2
//                           (FP64 as written; FP32 with w' formed once per
//                           call and one rsqrt per term)
#include <algorithm>

#include "common.cuh"
#include "weighted.cuh"

namespace ssm {

constexpr unsigned kInfBits = 0x7f800000u;
constexpr int kSsspThreads = 512;  // of a search's block (half as many when there are many sources)

// ------------------------------------------------------------ edge lengths
__global__ void k_fill_u32(int64_t count, unsigned *__restrict__ p, unsigned v) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count; t += (int64_t)gridDim.x * blockDim.x)
    p[t] = v;
}

__device__ __forceinline__ int find_in_row(const int32_t *__restrict__ colidx, int b, int e, int v) {
  while (b < e) {
    const int mid = b + ((e - b) >> 1);
    const int c = __ldg(colidx + mid);
    if (c == v) return mid;
    if (c < v) b = mid + 1;
    else e = mid;
  }
  return -1;
}

__global__ void k_elen_set(int32_t n, int64_t m_in, const int32_t *__restrict__ src, const int32_t *__restrict__ dst,
                           const float *__restrict__ len, const int32_t *__restrict__ rowptr,
                           const int32_t *__restrict__ colidx, unsigned *__restrict__ elen,
                           unsigned *__restrict__ lmax, int32_t *__restrict__ status) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m_in; e += (int64_t)gridDim.x * blockDim.x) {
    const int u = src[e], v = dst[e];
    if (u < 0 || u >= n || v < 0 || v >= n) {
      dev_fail(status, SSM_E_GRAPH);
      continue;
    }
    if (u == v) continue;
    const float l = len[e];
    if (!(l >= 1.17549435e-38f) || !(l <= 3.4e38f)) {
      dev_fail(status, SSM_E_ARG);
      continue;
    }
    const unsigned lb = __float_as_uint(l);
    atomicMax(lmax, lb);
    const int tu = find_in_row(colidx, rowptr[u], rowptr[u + 1], v);
    const int tv = find_in_row(colidx, rowptr[v], rowptr[v + 1], u);
    if (tu < 0 || tv < 0) {
      dev_fail(status, SSM_E_GRAPH);
      continue;
    }
    atomicMin(elen + tu, lb);
    atomicMin(elen + tv, lb);
  }
}

__global__ void k_elen_check(int32_t n, int64_t m2, const unsigned *__restrict__ elen,
                             const unsigned *__restrict__ lmax, int32_t *__restrict__ status) {
  if (blockIdx.x == 0 && threadIdx.x == 0 && (double)n * (double)__uint_as_float(*lmax) >= 1e37)
    dev_fail(status, SSM_E_ARG);
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m2; t += (int64_t)gridDim.x * blockDim.x)
    if (elen[t] == kInfBits) dev_fail(status, SSM_E_GRAPH);  // a CSR edge missing from the list
}

// ------------------------------------------------------------ SSSP
// Near-far label-correcting search (two-bucket Delta-stepping), one block per
// source: only labels below a threshold T are relaxed in a round ("near"); a
// node lowered to a label at or above T waits in the far pile; when the near
// queue is empty T grows by Delta (at least to the smallest far label plus
// Delta) and the far pile is split again.  Plain rounds over every improved
// node re-relaxed each node about 20 times on a 262K-node geometric graph;
// the threshold keeps the search close to label-setting order while each round
// still relaxes a whole band of nodes.  Any order that relaxes until nothing
// improves reaches the same least path sums.
//
// While a search runs a node's word holds its label's bits << 1 | queued, so
// lowering a label and marking the node is one atomicMin with bits << 1 | 1
// (labels are non-negative floats; an equal label leaves the mark alone), and
// the value it returns says whether the node has to be queued.  A marked node
// whose label is below T is in the near queue, one at or above T in the far
// pile; a far node lowered below T is queued near as well, and its far entry is
// dropped at the split (the mark is gone by then).  So a node is in each queue
// at most once.
//
// A round is bound by its chain of dependent accesses (a block's search has
// some 860 rounds of a few hundred nodes on that graph): queue entry, row range
// and mark, edges, heads' words, atomicMin.  The queues sit in shared memory (a
// long one goes on in the block's global slot), the rows of a warp's entries
// are spread over its lanes, and kSsspU edges per lane are in flight at once;
// heads are read first, and only those that would be lowered see an atomicMin
// (one in five).  With one edge per lane at a time, queues and membership bits
// in global memory 200 sources on the 262K-node graph took 18.4 ms, now 8.0 (a
// round 20,000 cycles, three steps of some 5,500 per warp: the words of 200
// sources do not fit L2), and 1024 sources 66.9, now 31.
constexpr int kSsspQ = 1024;  // entries of a queue kept in shared memory
constexpr int kSsspU = 4;     // edges per lane in flight

__host__ __device__ inline size_t sssp_qbytes(int32_t n) { return (((size_t)n * 4) + 255) & ~size_t(255); }
size_t sssp_slot_bytes(int32_t n) { return 4 * sssp_qbytes(n); }

// A block's queues: near by parity, far by parity.  An entry is a node, a near
// entry in shared memory its row range as well.
struct SsspQueues {
  int4 (*near_sm)[kSsspQ];
  int32_t (*far_sm)[kSsspQ];
  int32_t *gl;
  size_t stride;  // of the global parts
  const int32_t *rowptr;
  __device__ __forceinline__ int4 get_near(int q, unsigned t) const {
    if (t < kSsspQ) return near_sm[q][t];
    const int v = __ldcg(gl + q * stride + t);
    return make_int4(v, __ldg(rowptr + v), __ldg(rowptr + v + 1), 0);
  }
  __device__ __forceinline__ void put_near(int q, unsigned t, int4 e) const {
    if (t < kSsspQ) near_sm[q][t] = e;
    else __stcg(gl + q * stride + t, e.x);
  }
  __device__ __forceinline__ int32_t get_far(int q, unsigned t) const {
    return t < kSsspQ ? far_sm[q][t] : __ldcg(gl + (2 + q) * stride + t);
  }
  __device__ __forceinline__ void put_far(int q, unsigned t, int32_t v) const {
    if (t < kSsspQ) far_sm[q][t] = v;
    else __stcg(gl + (2 + q) * stride + t, v);
  }
};

// The whole warp: places in a queue (counter in shared memory) for the flagged
// (lane, slot) pairs, one atomic for all of them; places[q] is set where flag[q]
template <int U>
__device__ __forceinline__ void sssp_places(const bool (&flag)[U], unsigned *counter, unsigned (&place)[U]) {
  const unsigned lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
  unsigned mask[U], total = 0;
#pragma unroll
  for (int q = 0; q < U; ++q) {
    mask[q] = __ballot_sync(0xffffffffu, flag[q]);
    total += __popc(mask[q]);
  }
  if (!total) return;
  unsigned at = 0;
  if (lane == 0) at = atomicAdd(counter, total);
  at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
  for (int q = 0; q < U; ++q) {
    place[q] = at + __popc(mask[q] & below);
    at += __popc(mask[q]);
  }
}

// One search from `source` into row (words as above).  init: every label is
// +inf first; otherwise the row's labels stay (max/min's pruned search: only
// nodes the new pivot is strictly closer to change).  delta is the band width.
// No word is marked on entry and on return.
__device__ void sssp_block(int32_t n, const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                           const unsigned *__restrict__ elen, int32_t source, unsigned *__restrict__ row, bool init,
                           float delta, char *slot, int32_t *__restrict__ status) {
  __shared__ int4 s_near_q[2][kSsspQ];
  __shared__ int32_t s_far_q[2][kSsspQ];
  __shared__ unsigned s_near[2], s_far, s_keep, s_least;
  const SsspQueues Q{s_near_q, s_far_q, (int32_t *)slot, sssp_qbytes(n) / 4, rowptr};
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  __syncthreads();  // the previous search of this block is over
  if (init)
    for (int v = threadIdx.x; v < n; v += blockDim.x) __stcg(row + v, kInfBits << 1);
  __syncthreads();
  if (threadIdx.x == 0) {
    __stcg(row + source, 1u);
    s_near_q[0][0] = make_int4(source, __ldg(rowptr + source), __ldg(rowptr + source + 1), 0);
    s_near[0] = 1u;
    s_near[1] = 0u;
    s_far = 0u;
    s_least = 0xFFFFFFFFu;
  }
  float T = delta;
  int cur = 0, fcur = 0;
  // every round relaxes at least one node whose label is then final for the
  // band, so the rounds are bounded; the cap only guards against a fault
  const int64_t cap = 64ll * ((int64_t)n + 16);
  for (int64_t round = 0;; ++round) {
    __syncthreads();  // the queue of this pass is complete
    unsigned count = s_near[cur];
    if (count == 0) {
      const unsigned nfar = s_far, least = s_least;
      if (nfar == 0) break;
      // next band: T >= smallest far label + delta (least is at or below it);
      // the marked entries of the far pile go to the near queue or the other pile
      T = fmaxf(T + delta, least == 0xFFFFFFFFu ? 0.0f : __uint_as_float(least) + delta);
      // where delta vanishes against the labels, take the next float above
      // the smallest far label so that at least that node moves on
      if (least != 0xFFFFFFFFu && !(T > __uint_as_float(least))) T = __uint_as_float(least + 1u);
      const unsigned tbits = __float_as_uint(T);
      __syncthreads();
      if (threadIdx.x == 0) {
        s_keep = 0u;
        s_least = 0xFFFFFFFFu;
      }
      __syncthreads();
      for (unsigned t = threadIdx.x; t < nfar; t += blockDim.x) {
        const int v = Q.get_far(fcur, t);
        const unsigned w = __ldcg(row + v);
        if (!(w & 1u)) continue;
        if ((w >> 1) < tbits) {
          Q.put_near(cur, atomicAdd(&s_near[cur], 1u), make_int4(v, __ldg(rowptr + v), __ldg(rowptr + v + 1), 0));
        } else {
          Q.put_far(fcur ^ 1, atomicAdd(&s_keep, 1u), v);
          atomicMin(&s_least, w >> 1);
        }
      }
      __syncthreads();
      if (threadIdx.x == 0) s_far = s_keep;
      fcur ^= 1;
      count = s_near[cur];
      if (count == 0) continue;
      __syncthreads();
    }
    if (round > cap) {
      if (threadIdx.x == 0) dev_fail(status, SSM_E_NUMERIC);
      break;
    }
    const unsigned tbits = __float_as_uint(T);
    unsigned *const next = &s_near[cur ^ 1];
    // entries per warp and step: a small round is spread over all warps
    const unsigned ipw = min(32u, (count + nwarps - 1u) / nwarps);
    for (unsigned base = warp * ipw; base < count; base += nwarps * ipw) {
      int b = 0, e = 0;
      unsigned dv = 0;
      if (lane < ipw && base + lane < count) {
        // the edges need the row range only: they are on their way together
        // with the label (a near entry's node is always marked)
        const int4 en = Q.get_near(cur, base + lane);
        b = en.y;
        e = en.z;
        dv = atomicAnd(row + en.x, ~1u) >> 1;
      }
      int incl = e - b;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane >= o) incl += t;
      }
      const int total = __shfl_sync(0xffffffffu, incl, 31);
      // up to 32 edges (a path's rounds): no read before the atomicMin, whose
      // round trip is then the longest in the chain that is left
      if (total <= 32) {
        const int t = (int)lane;
        bool act = t < total;
        int lo = 0;
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1) {
          const int pv = __shfl_sync(0xffffffffu, incl, lo + step - 1);
          if (pv <= t) lo += step;
        }
        const int at = lo > 31 ? 31 : lo;
        const int pos = __shfl_sync(0xffffffffu, e, at) - (__shfl_sync(0xffffffffu, incl, at) - t);
        const int u = act ? __ldg(colidx + pos) : 0;
        const unsigned len = act ? __ldg(elen + pos) : 0u;
        const unsigned nb = __float_as_uint(__fadd_rn(__uint_as_float(__shfl_sync(0xffffffffu, dv, at)), __uint_as_float(len)));
        act = act && nb < kInfBits;
        const unsigned old = act ? atomicMin(row + u, 2u * nb + 1u) : 0u;
        const int rb = act ? __ldg(rowptr + u) : 0, re = act ? __ldg(rowptr + u + 1) : 0;
        const bool lower = act && (old >> 1) > nb, was = (old & 1u) != 0u, below = nb < tbits;
        const bool near[1] = {lower && below && (!was || (old >> 1) >= tbits)}, far[1] = {lower && !below && !was};
        unsigned place[1] = {};
        sssp_places(near, next, place);
        if (near[0]) Q.put_near(cur ^ 1, place[0], make_int4(u, rb, re, 0));
        sssp_places(far, &s_far, place);
        if (far[0]) Q.put_far(fcur, place[0], u);
        const unsigned least = __reduce_min_sync(0xffffffffu, lower && !below ? nb : 0xFFFFFFFFu);
        if (lane == 0 && least != 0xFFFFFFFFu) atomicMin(&s_least, least);
        continue;
      }
      for (int s0 = 0; s0 < total; s0 += 32 * kSsspU) {
        int u[kSsspU], at[kSsspU];
        unsigned nb[kSsspU], len[kSsspU];
        bool act[kSsspU];
#pragma unroll
        for (int q = 0; q < kSsspU; ++q) {
          const int t = s0 + 32 * q + (int)lane;
          act[q] = t < total;
          int lo = 0;  // row = first lane whose inclusive prefix exceeds t
#pragma unroll
          for (int step = 16; step >= 1; step >>= 1) {
            const int pv = __shfl_sync(0xffffffffu, incl, lo + step - 1);
            if (pv <= t) lo += step;
          }
          at[q] = lo > 31 ? 31 : lo;
          const int o_end = __shfl_sync(0xffffffffu, e, at[q]), o_incl = __shfl_sync(0xffffffffu, incl, at[q]);
          const int pos = o_end - (o_incl - t);
          u[q] = act[q] ? __ldg(colidx + pos) : 0;
          len[q] = act[q] ? __ldg(elen + pos) : 0u;
        }
        unsigned old[kSsspU];
#pragma unroll
        for (int q = 0; q < kSsspU; ++q) old[q] = act[q] ? __ldcg(row + u[q]) : 0u;
#pragma unroll
        for (int q = 0; q < kSsspU; ++q) {
          nb[q] = __float_as_uint(__fadd_rn(__uint_as_float(__shfl_sync(0xffffffffu, dv, at[q])), __uint_as_float(len[q])));
          act[q] = act[q] && (old[q] >> 1) > nb[q];
        }
#pragma unroll
        for (int q = 0; q < kSsspU; ++q)
          if (act[q]) old[q] = atomicMin(row + u[q], 2u * nb[q] + 1u);
        // the lowered heads' row ranges, should they be queued (asked for with the
        // words, for every head, they cost 10 % more than their latency hid)
        int rb[kSsspU], re[kSsspU];
#pragma unroll
        for (int q = 0; q < kSsspU; ++q) {
          rb[q] = act[q] ? __ldg(rowptr + u[q]) : 0;
          re[q] = act[q] ? __ldg(rowptr + u[q] + 1) : 0;
        }
        unsigned least = 0xFFFFFFFFu, place[kSsspU] = {};
        bool near[kSsspU], far[kSsspU];
#pragma unroll
        for (int q = 0; q < kSsspU; ++q) {
          const bool lower = act[q] && (old[q] >> 1) > nb[q], was = (old[q] & 1u) != 0u, below = nb[q] < tbits;
          near[q] = lower && below && (!was || (old[q] >> 1) >= tbits);
          far[q] = lower && !below && !was;
          if (lower && !below) least = min(least, nb[q]);
        }
        sssp_places(near, next, place);
#pragma unroll
        for (int q = 0; q < kSsspU; ++q)
          if (near[q]) Q.put_near(cur ^ 1, place[q], make_int4(u[q], rb[q], re[q], 0));
        sssp_places(far, &s_far, place);
#pragma unroll
        for (int q = 0; q < kSsspU; ++q)
          if (far[q]) Q.put_far(fcur, place[q], u[q]);
        least = __reduce_min_sync(0xffffffffu, least);
        if (lane == 0 && least != 0xFFFFFFFFu) atomicMin(&s_least, least);
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) s_near[cur] = 0u;
    cur ^= 1;
  }
}

// band width of the near-far search: kDeltaScale times the mean edge length
constexpr float kDeltaScale = 8.0f;

// delta from the mean edge length: per-block sums, added in block order by the
// last block (one block over all edges took 1.16 ms on 2.1 M of them)
constexpr int kMeanBlocks = 28;
struct MeanWs {
  float delta;
  unsigned done, next;  // zero before the launch; blocks finished, sources handed out
  double part[kMeanBlocks];
};
static_assert(sizeof(MeanWs) <= 256, "the mean's workspace is 256 bytes");

__global__ void __launch_bounds__(1024) k_mean_length(int32_t n, const int32_t *__restrict__ rowptr,
                                                      const float *__restrict__ elen, MeanWs *__restrict__ ws) {
  __shared__ double red[32];
  __shared__ unsigned s_ticket;
  const int64_t m2 = rowptr[n];
  double acc = 0.0;
  float sum = 0.0f;
  int run = 0;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m2; t += (int64_t)gridDim.x * blockDim.x) {
    sum += __ldg(elen + t);
    if (++run == 16) {  // short runs in FP32: the band width needs no more
      acc += (double)sum;
      sum = 0.0f;
      run = 0;
    }
  }
  acc += (double)sum;
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    ws->part[blockIdx.x] = t;
    __threadfence();
    s_ticket = atomicAdd(&ws->done, 1u);
  }
  __syncthreads();
  if (s_ticket != gridDim.x - 1 || threadIdx.x != 0) return;
  __threadfence();
  double t = 0.0;
  for (unsigned q = 0; q < gridDim.x; ++q) t += __ldcg(ws->part + q);
  const float mean = m2 > 0 ? (float)(t / (double)m2) : 1.0f;
  ws->delta = mean > 0.0f ? kDeltaScale * mean : 1.0f;
}

static int launch_mean_length(int32_t n, const int32_t *rowptr, const float *elen, MeanWs *ws, cudaStream_t s) {
  SSM_TRY_CUDA(cudaMemsetAsync(&ws->done, 0, 2 * sizeof(unsigned), s));
  note_launch(), k_mean_length<<<kMeanBlocks, 1024, 0, s>>>(n, rowptr, elen, ws);
  return SSM_OK;
}

// d_ip mode: a block takes one source after another; dist rows [k][n] hold words
// (k_sssp_labels turns them into labels)
__global__ void __launch_bounds__(kSsspThreads, 2) k_sssp_multi(int32_t n, const int32_t *__restrict__ rowptr,
                                                             const int32_t *__restrict__ colidx,
                                                             const unsigned *__restrict__ elen, int32_t k,
                                                             const int32_t *__restrict__ sources,
                                                             unsigned *__restrict__ dist, MeanWs *__restrict__ ws,
                                                             char *slots, size_t slot_bytes,
                                                             int32_t *__restrict__ status) {
  __shared__ int s_a;
  const float dl = ws->delta;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_a = (int)atomicAdd(&ws->next, 1u);
    __syncthreads();
    const int a = s_a;
    if (a >= k) break;
    const int s = sources[a];
    if (s < 0 || s >= n) {
      if (threadIdx.x == 0) dev_fail(status, SSM_E_ARG);
      continue;
    }
    sssp_block(n, rowptr, colidx, elen, s, dist + (size_t)a * n, true, dl, slots + blockIdx.x * slot_bytes, status);
  }
}

// max/min mode (one block): the source is the pivot encoded in *key (or
// `start` when key is null); the search lowers mind in place
__global__ void __launch_bounds__(kSsspThreads) k_sssp_maxmin(int32_t n, const int32_t *__restrict__ rowptr,
                                                              const int32_t *__restrict__ colidx,
                                                              const unsigned *__restrict__ elen, int32_t start,
                                                              const unsigned long long *__restrict__ key,
                                                              int32_t *__restrict__ pivot_out,
                                                              unsigned *__restrict__ mind,
                                                              const float *__restrict__ delta, char *slots, bool init,
                                                              int32_t *__restrict__ status) {
  const int s = key ? (int)(0xFFFFFFFFu - (unsigned)(*key & 0xFFFFFFFFull)) : start;
  if (s < 0 || s >= n) {
    if (threadIdx.x == 0) dev_fail(status, SSM_E_ARG);
    return;
  }
  if (threadIdx.x == 0) *pivot_out = s;
  sssp_block(n, rowptr, colidx, elen, s, mind, init, *delta, slots, status);
}

// *key = max over v of (bits(mind_v) << 32 | (2^32 - 1 - v)): the largest
// label, ties to the lowest node id; an unreachable node (+inf) is an error
__global__ void k_wmm_argmax(int32_t n, const unsigned *__restrict__ mind, unsigned long long *__restrict__ key,
                             int32_t *__restrict__ status) {
  unsigned long long best = 0;
  bool inf = false;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const unsigned b = mind[v] >> 1;
    inf |= b >= kInfBits;
    const unsigned long long kk = ((unsigned long long)b << 32) | (0xFFFFFFFFu - (unsigned)v);
    best = kk > best ? kk : best;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_xor_sync(0xffffffffu, best, o);
    best = t > best ? t : best;
  }
  if ((threadIdx.x & 31) == 0) atomicMax(key, best);
  if (inf) dev_fail(status, SSM_E_DISCONNECTED);
}

// words to labels, four at a time where the table allows it; an unreachable
// node is an error
__global__ void k_sssp_labels(int64_t count, unsigned *__restrict__ dist, int32_t *__restrict__ status) {
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, gs = (int64_t)gridDim.x * blockDim.x;
  const int64_t quads = (reinterpret_cast<uintptr_t>(dist) & 15u) == 0 ? count / 4 : 0;
  bool inf = false;
  uint4 *d4 = reinterpret_cast<uint4 *>(dist);
  for (int64_t t = gt; t < quads; t += gs) {
    uint4 w = d4[t];
    w.x >>= 1;
    w.y >>= 1;
    w.z >>= 1;
    w.w >>= 1;
    inf |= max(max(w.x, w.y), max(w.z, w.w)) >= kInfBits;
    d4[t] = w;
  }
  for (int64_t t = 4 * quads + gt; t < count; t += gs) {
    const unsigned w = dist[t] >> 1;
    inf |= w >= kInfBits;
    dist[t] = w;
  }
  if (inf) dev_fail(status, SSM_E_DISCONNECTED);
}

// Blocks of half the width, four at once on an SM and not two, where there are
// many sources and their rounds are narrow: 1024 sources take 2.6 against 3.1 ms on
// 20K nodes, but 43 against 32 ms on 262K.  As many blocks as run at once: each
// has its queues in the workspace.
struct SsspShape {
  int threads, blocks;
};
static SsspShape sssp_shape(int32_t n, int32_t k) {
  const bool half = k > 2 * num_sms() && n < 65536;
  return {half ? kSsspThreads / 2 : kSsspThreads, std::max(1, std::min<int>(k, num_sms() * (half ? 4 : 2)))};
}

size_t sssp_ws_bytes(int32_t n, int32_t k) { return 256 + sssp_slot_bytes(n) * (size_t)sssp_shape(n, k).blocks; }

int launch_sssp(int32_t n, const int32_t *rowptr, const int32_t *colidx, const float *elen, int32_t k,
                const int32_t *sources, float *dist, int32_t *status, void *ws, size_t ws_bytes, cudaStream_t s) {
  const SsspShape shape = sssp_shape(n, k);
  const size_t sb = sssp_slot_bytes(n);
  if (ws_bytes < sssp_ws_bytes(n, k))
    return fail(SSM_E_NOMEM, "sssp: workspace %zu bytes, need %zu", ws_bytes, sssp_ws_bytes(n, k));
  MeanWs *mean = (MeanWs *)ws;
  char *slots = (char *)ws + 256;
  if (int rc = launch_mean_length(n, rowptr, elen, mean, s)) return rc;
  note_launch(), k_sssp_multi<<<shape.blocks, shape.threads, 0, s>>>(n, rowptr, colidx, (const unsigned *)elen, k, sources,
                                                       (unsigned *)dist, mean, slots, sb, status);
  const int64_t cnt = (int64_t)k * n;
  note_launch(), k_sssp_labels<<<(unsigned)std::min<int64_t>((cnt / 4 + 255) / 256 + 1, (int64_t)num_sms() * 16), 256, 0, s>>>(
      cnt, (unsigned *)dist, status);
  SSM_TRY_CUDA(cudaGetLastError());
  return SSM_OK;
}

// ------------------------------------------------------------ regions and s
__global__ void k_wregion_keys(int32_t n, int32_t k, const float *__restrict__ dist, int32_t *__restrict__ region,
                               unsigned long long *__restrict__ keys, int64_t npad) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npad; i += (int64_t)gridDim.x * blockDim.x) {
    if (i >= n) {
      keys[i] = ~0ull;
      continue;
    }
    int best = 0;
    float bd = __ldg(dist + i);
    for (int a = 1; a < k; ++a) {
      const float d = __ldg(dist + (size_t)a * n + i);
      if (d < bd) {
        bd = d;
        best = a;
      }
    }
    region[i] = best;
    keys[i] = ((unsigned long long)best << 32) | __float_as_uint(bd);
  }
}

// bitonic sort of npad (a power of two, at least 2048) 64-bit keys, ascending
constexpr int kSortChunk = 2048;

__device__ __forceinline__ void cmp_swap(unsigned long long &x, unsigned long long &y, bool up) {
  if ((x > y) == up) {
    const unsigned long long t = x;
    x = y;
    y = t;
  }
}

// stages kk = 2 .. 2048 inside each 2048-key chunk (directions by global index)
__global__ void __launch_bounds__(1024) k_bitonic_local(unsigned long long *__restrict__ keys) {
  __shared__ unsigned long long sk[kSortChunk];
  const int64_t base = (int64_t)blockIdx.x * kSortChunk;
  sk[threadIdx.x] = keys[base + threadIdx.x];
  sk[threadIdx.x + 1024] = keys[base + threadIdx.x + 1024];
  __syncthreads();
  for (int kk = 2; kk <= kSortChunk; kk <<= 1)
    for (int j = kk >> 1; j > 0; j >>= 1) {
      const int t = threadIdx.x;
      const int i = ((t / j) * 2 * j) + (t % j);
      const bool up = (((base + i) & kk) == 0);
      cmp_swap(sk[i], sk[i + j], up);
      __syncthreads();
    }
  keys[base + threadIdx.x] = sk[threadIdx.x];
  keys[base + threadIdx.x + 1024] = sk[threadIdx.x + 1024];
}

__global__ void k_bitonic_global(unsigned long long *__restrict__ keys, int64_t npad, int64_t kk, int64_t j) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < npad / 2; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = ((t / j) * 2 * j) + (t % j);
    const bool up = ((i & kk) == 0);
    unsigned long long x = keys[i], y = keys[i + j];
    cmp_swap(x, y, up);
    keys[i] = x;
    keys[i + j] = y;
  }
}

// the steps j = 1024 .. 1 of stage kk inside each chunk
__global__ void __launch_bounds__(1024) k_bitonic_merge_local(unsigned long long *__restrict__ keys, int64_t kk) {
  __shared__ unsigned long long sk[kSortChunk];
  const int64_t base = (int64_t)blockIdx.x * kSortChunk;
  sk[threadIdx.x] = keys[base + threadIdx.x];
  sk[threadIdx.x + 1024] = keys[base + threadIdx.x + 1024];
  __syncthreads();
  for (int j = kSortChunk >> 1; j > 0; j >>= 1) {
    const int t = threadIdx.x;
    const int i = ((t / j) * 2 * j) + (t % j);
    const bool up = (((base + i) & kk) == 0);
    cmp_swap(sk[i], sk[i + j], up);
    __syncthreads();
  }
  keys[base + threadIdx.x] = sk[threadIdx.x];
  keys[base + threadIdx.x + 1024] = sk[threadIdx.x + 1024];
}

static int launch_sort(unsigned long long *keys, int64_t npad, cudaStream_t s) {
  const unsigned chunks = (unsigned)(npad / kSortChunk);
  note_launch(), k_bitonic_local<<<chunks, 1024, 0, s>>>(keys);
  const unsigned gb = (unsigned)std::min<int64_t>((npad / 2 + 255) / 256, (int64_t)num_sms() * 16);
  for (int64_t kk = 2 * kSortChunk; kk <= npad; kk <<= 1) {
    for (int64_t j = kk >> 1; j >= kSortChunk; j >>= 1) note_launch(), k_bitonic_global<<<gb, 256, 0, s>>>(keys, npad, kk, j);
    note_launch(), k_bitonic_merge_local<<<chunks, 1024, 0, s>>>(keys, kk);
  }
  SSM_TRY_CUDA(cudaGetLastError());
  return SSM_OK;
}

// seg[a] = first key position of region a (a = 0..k; padding keys sort last)
__global__ void k_seg_start(int32_t k, const unsigned long long *__restrict__ keys, int64_t npad,
                            int64_t *__restrict__ seg) {
  for (int a = blockIdx.x * blockDim.x + threadIdx.x; a <= k; a += gridDim.x * blockDim.x) {
    const unsigned long long want = (unsigned long long)a << 32;
    int64_t lo = 0, hi = npad;
    while (lo < hi) {
      const int64_t mid = lo + ((hi - lo) >> 1);
      if (keys[mid] < want) lo = mid + 1;
      else hi = mid;
    }
    seg[a] = lo;
  }
}

// s_ia for one pivot (blockIdx.x) and a range of nodes: the entries of region a
// with 2 d_ja <= d_ia are a prefix of its sorted segment, found by binary search
// in shared memory; of a segment of more than kCountSeg entries, every
// stride-th is there, and the search ends in global memory between two of them.
// One search over global memory per (pivot, node), with a binary search of the
// node's row for the pivot, took 1.62 ms on 52 M pairs, now 0.26; the pivot and its
// neighbours, where s is 0, are cleared afterwards (k_wcounts_near).
constexpr int kCountSeg = 8192;
__global__ void __launch_bounds__(256) k_wcounts(int32_t n, const float *__restrict__ dist,
                                                 const unsigned long long *__restrict__ keys,
                                                 const int64_t *__restrict__ seg, uint32_t *__restrict__ s_out) {
  __shared__ float sd[kCountSeg];
  const int a = blockIdx.x;
  const int64_t lo = seg[a];
  const int len = (int)(seg[a + 1] - lo);
  const int stride = (len + kCountSeg - 1) / kCountSeg, kept = stride > 1 ? (len + stride - 1) / stride : len;
  auto twice = [&](int t) { return __fmul_rn(2.0f, __uint_as_float((unsigned)__ldg(keys + lo + t))); };
  for (int t0 = threadIdx.x; t0 < kept; t0 += 8 * (int)blockDim.x) {  // eight loads in flight
    float v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = twice(min(t0 + q * (int)blockDim.x, kept - 1) * stride);
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (t0 + q * (int)blockDim.x < kept) sd[t0 + q * (int)blockDim.x] = v[q];
  }
  __syncthreads();
  const float *d = dist + (size_t)a * n;
  uint32_t *out = s_out + (size_t)a * n;
  for (int64_t i = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.y * blockDim.x) {
    const float di = __ldg(d + i);
    int b = 0, e = kept;
    while (b < e) {
      const int mid = (b + e) >> 1;
      if (sd[mid] <= di) b = mid + 1;
      else e = mid;
    }
    if (stride > 1 && b > 0) {  // entry (b - 1) stride is below, entry b stride is not
      e = min(b * stride, len);
      b = (b - 1) * stride + 1;
      while (b < e) {
        const int mid = (b + e) >> 1;
        if (twice(mid) <= di) b = mid + 1;
        else e = mid;
      }
    }
    out[i] = (uint32_t)b;
  }
}

// blocks (pivot, part of its row): with one of 128 threads, a hub among the pivots
// took 0.28 ms over its 200,000 neighbours
__global__ void k_wcounts_near(int32_t n, const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                               const int32_t *__restrict__ pivots, uint32_t *__restrict__ s_out) {
  const int p = pivots[blockIdx.x];
  if ((unsigned)p >= (unsigned)n) return;
  uint32_t *out = s_out + (size_t)blockIdx.x * n;
  if (threadIdx.x == 0 && blockIdx.y == 0) out[p] = 0u;
  const int e = rowptr[p + 1];
#pragma unroll 4
  for (int t = rowptr[p] + (int)(blockIdx.y * blockDim.x + threadIdx.x); t < e; t += (int)(gridDim.y * blockDim.x))
    out[__ldg(colidx + t)] = 0u;
}

// ------------------------------------------------------------ the sweep
constexpr int kWSweepThreads = 256;

// relative change: block sums; the last block adds them, a fixed share per
// thread and a fixed tree (added by one thread they took 45 us of a 183 us
// iteration on 1,023 blocks)
__device__ void wsweep_change(double dn, double dd, double *__restrict__ part, unsigned *__restrict__ done,
                              double *__restrict__ rel) {
  __shared__ double red[2][kWSweepThreads / 32];
  __shared__ unsigned s_ticket;
  auto block_sum = [&](double &x, double &y) {  // in thread 0
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    if ((threadIdx.x & 31) == 0) {
      red[0][threadIdx.x >> 5] = x;
      red[1][threadIdx.x >> 5] = y;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      x = y = 0.0;
      for (int w = 0; w < kWSweepThreads / 32; ++w) {
        x += red[0][w];
        y += red[1][w];
      }
    }
    __syncthreads();
  };
  block_sum(dn, dd);
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = dn;
    part[2 * blockIdx.x + 1] = dd;
    __threadfence();
    s_ticket = atomicAdd(done, 1u);
  }
  __syncthreads();
  if (s_ticket != gridDim.x - 1) return;
  __threadfence();
  double a0 = 0.0, a1 = 0.0;
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
    a0 += __ldcg(part + 2 * b);
    a1 += __ldcg(part + 2 * b + 1);
  }
  block_sum(a0, a1);
  if (threadIdx.x == 0) {
    *rel = a1 > 0.0 ? sqrt(a0) / sqrt(a1) : 0.0;
    *done = 0;
  }
}

// Eq. 4 for one node in FP64, every operation rounded on its own in the
// order of the plain FP64 definition (bit-identical to it)
template <class T2>
struct WArith;

template <>
struct WArith<double2> {
  using R = double;
  __device__ static R add(R a, R b) { return __dadd_rn(a, b); }
  __device__ static R sub(R a, R b) { return __dsub_rn(a, b); }
  __device__ static R mul(R a, R b) { return __dmul_rn(a, b); }
  __device__ static R div(R a, R b) { return __ddiv_rn(a, b); }
  __device__ static R sqrt_(R a) { return __dsqrt_rn(a); }
};

template <class T2>
__global__ void __launch_bounds__(kWSweepThreads) k_wsweep(int32_t n, const int32_t *__restrict__ rowptr,
                                                           const int32_t *__restrict__ colidx,
                                                           const float *__restrict__ elen, int32_t k,
                                                           const int32_t *__restrict__ pivots,
                                                           const float *__restrict__ dist,
                                                           const uint32_t *__restrict__ s_tab,
                                                           const T2 *__restrict__ X, T2 *__restrict__ Y,
                                                           double *__restrict__ part, unsigned *__restrict__ done,
                                                           double *__restrict__ rel) {
  using A = WArith<T2>;
  using R = typename A::R;
  extern __shared__ __align__(16) unsigned char wsm[];
  T2 *xp = reinterpret_cast<T2 *>(wsm);
  for (int a = threadIdx.x; a < k; a += blockDim.x) xp[a] = X[__ldg(pivots + a)];
  __syncthreads();
  double dn = 0.0, dd = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const T2 xi = X[i];
    R nx = 0, ny = 0, den = 0;
    for (int t = __ldg(rowptr + i); t < __ldg(rowptr + i + 1); ++t) {
      const int j = __ldg(colidx + t);
      const R l = (R)__ldg(elen + t);
      const R w = A::div((R)1, A::mul(l, l));
      const T2 xj = X[j];
      const R dx = A::sub(xi.x, xj.x), dy = A::sub(xi.y, xj.y);
      const R r = A::sqrt_(A::add(A::mul(dx, dx), A::mul(dy, dy)));
      if (r > (R)0) {
        nx = A::add(nx, A::mul(w, A::add(xj.x, A::div(A::mul(l, dx), r))));
        ny = A::add(ny, A::mul(w, A::add(xj.y, A::div(A::mul(l, dy), r))));
      } else {
        nx = A::add(nx, A::mul(w, xj.x));
        ny = A::add(ny, A::mul(w, xj.y));
      }
      den = A::add(den, w);
    }
    for (int a = 0; a < k; ++a) {
      const uint32_t sc = __ldg(s_tab + (size_t)a * n + i);
      if (sc == 0) continue;  // the pivot is i itself or one of its neighbours
      const R d = (R)__ldg(dist + (size_t)a * n + i);
      const R w = A::div((R)sc, A::mul(d, d));
      const T2 xq = xp[a];
      const R dx = A::sub(xi.x, xq.x), dy = A::sub(xi.y, xq.y);
      const R r = A::sqrt_(A::add(A::mul(dx, dx), A::mul(dy, dy)));
      if (r > (R)0) {
        nx = A::add(nx, A::mul(w, A::add(xq.x, A::div(A::mul(d, dx), r))));
        ny = A::add(ny, A::mul(w, A::add(xq.y, A::div(A::mul(d, dy), r))));
      } else {
        nx = A::add(nx, A::mul(w, xq.x));
        ny = A::add(ny, A::mul(w, xq.y));
      }
      den = A::add(den, w);
    }
    T2 y = xi;
    if (den > (R)0) {
      y.x = A::div(nx, den);
      y.y = A::div(ny, den);
    }
    Y[i] = y;
    const double ex = (double)y.x - (double)xi.x, ey = (double)y.y - (double)xi.y;
    dn += ex * ex + ey * ey;
    dd += (double)xi.x * (double)xi.x + (double)xi.y * (double)xi.y;
  }
  wsweep_change(dn, dd, part, done, rel);
}

// FP32 form: w'_ia = s_ia / d_ia^2 formed once per call into wtab (0 where
// the pivot term is skipped), then per term one rsqrt and multiply-adds:
// u = 1/r, B = w' d u, numerator = sum w' x_p + sum B (x_i - x_p) (kept as
// two sums so that nothing cancels); r = 0 contributes w' x_p only.  A thread
// owns one node; eight pivots' (d, w') pairs are loaded before they are used.
__global__ void k_wprep(int64_t count, const float *__restrict__ dist, const uint32_t *__restrict__ s_tab,
                        float *__restrict__ wtab) {
  auto weight = [](uint32_t sc, float d) { return sc ? (float)sc / (d * d) : 0.0f; };
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, gs = (int64_t)gridDim.x * blockDim.x;
  const bool quads_ok = ((reinterpret_cast<uintptr_t>(dist) | reinterpret_cast<uintptr_t>(s_tab)) & 15u) == 0;
  const int64_t quads = quads_ok ? count / 4 : 0;  // wtab is 256-byte aligned
#pragma unroll 2
  for (int64_t t = gt; t < quads; t += gs) {
    const float4 d = __ldg(reinterpret_cast<const float4 *>(dist) + t);
    const uint4 c = __ldg(reinterpret_cast<const uint4 *>(s_tab) + t);
    reinterpret_cast<float4 *>(wtab)[t] = make_float4(weight(c.x, d.x), weight(c.y, d.y), weight(c.z, d.z), weight(c.w, d.w));
  }
  for (int64_t t = 4 * quads + gt; t < count; t += gs) wtab[t] = weight(s_tab[t], dist[t]);
}

constexpr int kWPrefetch = 8;

__global__ void __launch_bounds__(kWSweepThreads) k_wsweep_f32(int32_t n, const int32_t *__restrict__ rowptr,
                                                               const int32_t *__restrict__ colidx,
                                                               const float *__restrict__ elen, int32_t k,
                                                               const int32_t *__restrict__ pivots,
                                                               const float *__restrict__ dist,
                                                               const float *__restrict__ wtab,
                                                               const float2 *__restrict__ X, float2 *__restrict__ Y,
                                                               double *__restrict__ part, unsigned *__restrict__ done,
                                                               double *__restrict__ rel) {
  extern __shared__ __align__(16) unsigned char wsm[];
  float2 *xp = reinterpret_cast<float2 *>(wsm);
  for (int a = threadIdx.x; a < k; a += blockDim.x) xp[a] = X[__ldg(pivots + a)];
  __syncthreads();
  double dn = 0.0, dd = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float2 xi = X[i];
    float wx = 0.f, wy = 0.f, bx = 0.f, by = 0.f, den = 0.f;
    const float *dcol = dist + i;
    const float *wcol = wtab + i;
    // the first pivots' (d, w') are requested before the neighbour gathers,
    // and every batch's loads are issued before the previous batch is used
    float dq[kWPrefetch], wq[kWPrefetch];
#pragma unroll
    for (int q = 0; q < kWPrefetch; ++q) {
      const bool ok = q < k;
      dq[q] = ok ? __ldg(dcol + (size_t)q * n) : 0.f;
      wq[q] = ok ? __ldg(wcol + (size_t)q * n) : 0.f;
    }
    for (int t = __ldg(rowptr + i); t < __ldg(rowptr + i + 1); ++t) {
      const float l = __ldg(elen + t);
      const float w = 1.0f / (l * l);
      const float2 xj = X[__ldg(colidx + t)];
      const float dx = xi.x - xj.x, dy = xi.y - xj.y;
      const float r2 = dx * dx + dy * dy;
      const float B = r2 > 0.f ? w * l * rsqrtf(r2) : 0.f;
      wx += w * xj.x;
      wy += w * xj.y;
      bx += B * dx;
      by += B * dy;
      den += w;
    }
    for (int a0 = 0; a0 < k; a0 += kWPrefetch) {
      float dn_[kWPrefetch], wn_[kWPrefetch];
#pragma unroll
      for (int q = 0; q < kWPrefetch; ++q) {
        const bool ok = a0 + kWPrefetch + q < k;
        dn_[q] = ok ? __ldg(dcol + (size_t)(a0 + kWPrefetch + q) * n) : 0.f;
        wn_[q] = ok ? __ldg(wcol + (size_t)(a0 + kWPrefetch + q) * n) : 0.f;
      }
#pragma unroll
      for (int q = 0; q < kWPrefetch; ++q) {
        if (a0 + q >= k) break;
        const float2 p = xp[a0 + q];
        const float w = wq[q];
        const float dx = xi.x - p.x, dy = xi.y - p.y;
        const float r2 = dx * dx + dy * dy;
        const float B = r2 > 0.f ? w * dq[q] * rsqrtf(r2) : 0.f;
        wx += w * p.x;
        wy += w * p.y;
        bx += B * dx;
        by += B * dy;
        den += w;
      }
#pragma unroll
      for (int q = 0; q < kWPrefetch; ++q) {
        dq[q] = dn_[q];
        wq[q] = wn_[q];
      }
    }
    float2 y = xi;
    if (den > 0.f) {
      y.x = (wx + bx) / den;
      y.y = (wy + by) / den;
    }
    Y[i] = y;
    const double ex = (double)y.x - (double)xi.x, ey = (double)y.y - (double)xi.y;
    dn += ex * ex + ey * ey;
    dd += (double)xi.x * (double)xi.x + (double)xi.y * (double)xi.y;
  }
  wsweep_change(dn, dd, part, done, rel);
}

}  // namespace ssm

// =========================================================== C ABI
SSM_API int ssm_edge_lengths(int32_t n, int64_t m_in, const int32_t *src, const int32_t *dst, const float *len,
                             int64_t m, const int32_t *rowptr, const int32_t *colidx, float *elen, int32_t *status,
                             void *ws, size_t ws_bytes, cudaStream_t s) {
  using namespace ssm;
  if (n < 1 || m_in < 0 || m < 0 || !rowptr || !colidx || !elen || !status || !ws || (m_in > 0 && (!src || !dst || !len)))
    return fail(SSM_E_ARG, "ssm_edge_lengths: null pointer or bad size");
  if (ws_bytes < 256) return fail(SSM_E_NOMEM, "ssm_edge_lengths: workspace %zu bytes, need 256", ws_bytes);
  unsigned *lmax = (unsigned *)ws;
  const int64_t m2 = 2 * m;
  const unsigned gb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((std::max(m2, m_in) + 255) / 256,
                                                                        (int64_t)num_sms() * 8));
  SSM_TRY_CUDA(cudaMemsetAsync(lmax, 0, sizeof(unsigned), s));
  if (m2 > 0) note_launch(), k_fill_u32<<<gb, 256, 0, s>>>(m2, (unsigned *)elen, kInfBits);
  if (m_in > 0)
    note_launch(), k_elen_set<<<gb, 256, 0, s>>>(n, m_in, src, dst, len, rowptr, colidx, (unsigned *)elen, lmax, status);
  note_launch(), k_elen_check<<<gb, 256, 0, s>>>(n, m2, (const unsigned *)elen, lmax, status);
  SSM_TRY_CUDA(cudaGetLastError());
  return SSM_OK;
}

SSM_API size_t ssm_pivot_sssp_workspace(int32_t n, int32_t k) {
  if (n < 1 || k < 1) return 0;
  return ssm::sssp_ws_bytes(n, k);
}

SSM_API int ssm_pivot_sssp(int32_t n, int64_t m, const int32_t *rowptr, const int32_t *colidx, const float *elen,
                           int32_t k, const int32_t *sources, float *dist, int32_t *status, void *ws, size_t ws_bytes,
                           cudaStream_t s) {
  using namespace ssm;
  (void)m;
  if (n < 1 || k < 1 || !rowptr || !colidx || !elen || !sources || !dist || !status || !ws)
    return fail(SSM_E_ARG, "ssm_pivot_sssp: null pointer or bad size");
  return launch_sssp(n, rowptr, colidx, elen, k, sources, dist, status, ws, ws_bytes, s);
}

namespace ssm {
struct WmmWs {
  unsigned *mind;
  unsigned long long *keys;
  MeanWs *mean;
  char *slot;  // the single-block search's queues, or the cluster's spill area
};
static size_t carve_wmm(Carver &c, WmmWs &w, int32_t n, int32_t k) {
  w.mind = c.take<unsigned>((size_t)n);
  w.keys = c.take<unsigned long long>((size_t)k);
  w.mean = c.take<MeanWs>(1);
  w.slot = c.take<char>(std::max(sssp_slot_bytes(n), wmaxmin_spill_entries(n) * sizeof(int32_t)));
  return c.size();
}
}  // namespace ssm

SSM_API size_t ssm_select_pivots_weighted_workspace(int32_t n, int32_t k) {
  if (n < 1 || k < 1) return 0;
  ssm::Carver c(nullptr, 0);
  ssm::WmmWs w;
  return ssm::carve_wmm(c, w, n, k);
}

SSM_API int ssm_select_pivots_weighted(int32_t n, int64_t m, const int32_t *rowptr, const int32_t *colidx,
                                       const float *elen, int32_t k, int32_t start, int32_t *pivots,
                                       int32_t *status, void *ws, size_t ws_bytes, cudaStream_t s) {
  using namespace ssm;
  (void)m;
  if (n < 1 || !rowptr || !colidx || !elen || !pivots || !status || !ws)
    return fail(SSM_E_ARG, "ssm_select_pivots_weighted: null pointer or n < 1");
  if (k < 1 || k > n || start < 0 || start >= n)
    return fail(SSM_E_ARG, "ssm_select_pivots_weighted: need 1 <= k <= n and 0 <= start < n");
  Carver c(ws, ws_bytes);
  WmmWs w;
  carve_wmm(c, w, n, k);
  if (!c.ok) return fail(SSM_E_NOMEM, "ssm_select_pivots_weighted: workspace %zu bytes, need %zu", ws_bytes, c.size());
  if (int rc = launch_mean_length(n, rowptr, elen, w.mean, s)) return rc;
  float *const delta = &w.mean->delta;
  // in one cluster when the labels fit its shared memory; larger graphs search
  // pivot by pivot in one block over global memory
  bool ran = false;
  if (int rc = launch_wmaxmin_cluster(n, rowptr, colidx, elen, k, start, pivots, delta, (int32_t *)w.slot, status, s, &ran))
    return rc;
  if (ran) return SSM_OK;
  SSM_TRY_CUDA(cudaMemsetAsync(w.keys, 0, (size_t)k * sizeof(unsigned long long), s));
  note_launch(), k_sssp_maxmin<<<1, kSsspThreads, 0, s>>>(n, rowptr, colidx, (const unsigned *)elen, start, nullptr,
                                                        pivots, w.mind, delta, w.slot, true, status);
  const unsigned ab = (unsigned)std::max(1, std::min((n + 255) / 256, num_sms() * 4));
  for (int a = 1; a < k; ++a) {
    note_launch(), k_wmm_argmax<<<ab, 256, 0, s>>>(n, w.mind, w.keys + a, status);
    note_launch(), k_sssp_maxmin<<<1, kSsspThreads, 0, s>>>(n, rowptr, colidx, (const unsigned *)elen, 0, w.keys + a,
                                                          pivots + a, w.mind, delta, w.slot, false, status);
  }
  if (k == 1) note_launch(), k_wmm_argmax<<<ab, 256, 0, s>>>(n, w.mind, w.keys, status);  // reachability check
  SSM_TRY_CUDA(cudaGetLastError());
  return SSM_OK;
}

namespace ssm {
static int64_t sort_size(int32_t n) {
  int64_t p = kSortChunk;
  while (p < n) p <<= 1;
  return p;
}
struct WcntWs {
  unsigned long long *keys;
  int64_t *seg;
};
static size_t carve_wcnt(Carver &c, WcntWs &w, int32_t n, int32_t k) {
  w.keys = c.take<unsigned long long>((size_t)sort_size(n));
  w.seg = c.take<int64_t>((size_t)k + 1);
  return c.size();
}
}  // namespace ssm

SSM_API size_t ssm_weighted_counts_workspace(int32_t n, int32_t k) {
  if (n < 1 || k < 1) return 0;
  ssm::Carver c(nullptr, 0);
  ssm::WcntWs w;
  return ssm::carve_wcnt(c, w, n, k);
}

SSM_API int ssm_weighted_counts(int32_t n, const int32_t *rowptr, const int32_t *colidx, int32_t k,
                                const int32_t *pivots, const float *dist, int32_t *region, uint32_t *s_tab,
                                int32_t *status, void *ws, size_t ws_bytes, cudaStream_t s) {
  using namespace ssm;
  if (n < 1 || k < 1 || !rowptr || !colidx || !pivots || !dist || !region || !s_tab || !status || !ws)
    return fail(SSM_E_ARG, "ssm_weighted_counts: null pointer or bad size");
  Carver c(ws, ws_bytes);
  WcntWs w;
  carve_wcnt(c, w, n, k);
  if (!c.ok) return fail(SSM_E_NOMEM, "ssm_weighted_counts: workspace %zu bytes, need %zu", ws_bytes, c.size());
  const int64_t npad = sort_size(n);
  const int sms = num_sms();
  note_launch(), k_wregion_keys<<<(unsigned)std::min<int64_t>((npad + 255) / 256, (int64_t)sms * 8), 256, 0, s>>>(
      n, k, dist, region, w.keys, npad);
  if (int rc = launch_sort(w.keys, npad, s)) return rc;
  note_launch(), k_seg_start<<<std::max(1, (k + 256) / 256), 256, 0, s>>>(k, w.keys, npad, w.seg);
  // 2048 nodes a block (a star's one large region is then some n / 2048 blocks' work),
  // fewer where there would be less than two blocks per SM
  const int64_t parts = std::max<int64_t>(((int64_t)n + 2047) / 2048, std::min<int64_t>(((int64_t)n + 255) / 256, (2 * sms + k - 1) / k));
  note_launch(), k_wcounts<<<dim3((unsigned)k, (unsigned)std::min<int64_t>(parts, 65535)), 256, 0, s>>>(n, dist, w.keys, w.seg, s_tab);
  note_launch(), k_wcounts_near<<<dim3((unsigned)k, (unsigned)std::max(4, 2048 / k)), 128, 0, s>>>(n, rowptr, colidx, pivots, s_tab);
  SSM_TRY_CUDA(cudaGetLastError());
  return SSM_OK;
}

namespace ssm {
static int wsweep_blocks(int32_t n) { return std::max(1, std::min((n + kWSweepThreads - 1) / kWSweepThreads, num_sms() * 8)); }
struct WSweepWs {
  void *buf;
  double *part;
  unsigned *done;
  float *wtab;
};
static size_t carve_wsweep(Carver &c, WSweepWs &w, int32_t n, int32_t k, int32_t precision) {
  w.buf = c.take<char>((size_t)n * (precision == 64 ? 16 : 8));
  w.part = c.take<double>(2 * (size_t)wsweep_blocks(n));
  w.done = c.take<unsigned>(1);
  w.wtab = precision == 32 ? c.take<float>((size_t)k * n) : nullptr;
  return c.size();
}
}  // namespace ssm

SSM_API size_t ssm_iterate_weighted_workspace(int32_t n, int32_t k, int32_t precision) {
  if (n < 1 || k < 1 || (precision != 32 && precision != 64)) return 0;
  ssm::Carver c(nullptr, 0);
  ssm::WSweepWs w;
  return ssm::carve_wsweep(c, w, n, k, precision);
}

SSM_API int ssm_iterate_weighted(int32_t n, const int32_t *rowptr, const int32_t *colidx, const float *elen,
                                 int32_t k, const int32_t *pivots, const float *dist, const uint32_t *s_tab, void *pos,
                                 int32_t precision, int32_t iters, double *rel_change, int32_t *status, void *ws,
                                 size_t ws_bytes, cudaStream_t s) {
  using namespace ssm;
  if (n < 1 || k < 1 || !rowptr || !colidx || !elen || !pivots || !dist || !s_tab || !pos || !status || !ws ||
      !rel_change || iters < 0)
    return fail(SSM_E_ARG, "ssm_iterate_weighted: null pointer or bad size");
  if (precision != 32 && precision != 64) return fail(SSM_E_ARG, "ssm_iterate_weighted: precision must be 32 or 64");
  const size_t esz = precision == 64 ? 16 : 8;
  if ((size_t)k * esz > 200 * 1024) return fail(SSM_E_ARG, "ssm_iterate_weighted: k too large for the pivot stage");
  Carver c(ws, ws_bytes);
  WSweepWs w;
  carve_wsweep(c, w, n, k, precision);
  if (!c.ok) return fail(SSM_E_NOMEM, "ssm_iterate_weighted: workspace %zu bytes, need %zu", ws_bytes, c.size());
  SSM_TRY_CUDA(cudaMemsetAsync(w.done, 0, sizeof(unsigned), s));
  SSM_TRY_CUDA(cudaMemsetAsync(rel_change, 0, sizeof(double), s));
  const int nb = wsweep_blocks(n);
  const size_t smem = (size_t)k * esz;
  if (precision == 64) {
    SSM_TRY_CUDA(allow_dynamic_smem((const void *)k_wsweep<double2>));
  } else {
    SSM_TRY_CUDA(allow_dynamic_smem((const void *)k_wsweep_f32));
    if (iters > 0) {
      const int64_t cnt = (int64_t)k * n;
      note_launch(), k_wprep<<<(unsigned)std::min<int64_t>((cnt + 255) / 256, (int64_t)num_sms() * 8), 256, 0, s>>>(
          cnt, dist, s_tab, w.wtab);
    }
  }
  void *bufs[2] = {pos, w.buf};
  for (int it = 0; it < iters; ++it) {
    void *in = bufs[it & 1], *out = bufs[(it & 1) ^ 1];
    if (precision == 64)
      note_launch(), k_wsweep<double2><<<nb, kWSweepThreads, smem, s>>>(n, rowptr, colidx, elen, k, pivots, dist, s_tab,
                                                                  (const double2 *)in, (double2 *)out, w.part, w.done,
                                                                  rel_change);
    else
      note_launch(), k_wsweep_f32<<<nb, kWSweepThreads, smem, s>>>(n, rowptr, colidx, elen, k, pivots, dist, w.wtab,
                                                             (const float2 *)in, (float2 *)out, w.part, w.done,
                                                             rel_change);
  }
  if (iters & 1) SSM_TRY_CUDA(cudaMemcpyAsync(pos, w.buf, (size_t)n * esz, cudaMemcpyDeviceToDevice, s));
  SSM_TRY_CUDA(cudaGetLastError());
  return SSM_OK;
}
