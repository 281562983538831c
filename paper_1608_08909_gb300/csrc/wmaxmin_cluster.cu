// Max/min-sp pivot sampling (Section 4.1) on weighted graphs inside one
// thread-block cluster.
//
// The sampling is a chain of k searches, each lowering mind[v], the least
// float32 path sum from v to a pivot chosen so far, where the new pivot is
// strictly closer.  A search needs at least as many dependent rounds as its
// shortest paths have edges (about 860 for the first one on a geometric graph
// of 262K nodes, some 8,000 for 200 pivots), so its cost is the latency of a
// round.  With one block, labels, queues and membership bits in global memory
// a round was five dependent L2 round trips (15 us); here it is one L2 round
// trip for the edges and three through distributed shared memory:
//   * node v belongs to CTA v mod C of a C-CTA cluster (C = 16 or 8); its word
//     sits in that CTA's shared memory: bits of mind << 1 | queued.  Lowering a
//     label and marking the node as queued is one DSMEM atomicMin with
//     bits << 1 | 1 (labels are non-negative floats, so their bits order like
//     the labels, and an equal label never changes the mark); the value it
//     returns tells whether the node has to be pushed;
//   * a node is pushed, with its row range, into its owner's near queue of the
//     next round (label below the threshold T) or far pile (label at or above
//     T): a DSMEM atomicAdd for the place and a DSMEM store.  A queued node
//     whose label is below T is in the near queue, one at or above T in the far
//     pile; a far node lowered below T is pushed to the near queue as well, and
//     its far entry is dropped (its mark is cleared) when the pile is split;
//   * when the near queue is empty everywhere, T moves on (at least to the least
//     far label plus the band width) and every CTA splits its own pile;
//   * with its pushes of a round every CTA publishes the least label it sent to
//     a far pile, so T needs no exchange of its own: a round and a split each
//     end with one hardware cluster barrier.
// Any order of relaxations reaches the same least path sums, so the pivots are
// those of every other correct search.  Entries beyond a queue's
// shared-memory part go to a global spill area (an owner's node is in each
// queue at most once, so `slots` entries per queue always suffice).
// Measured (262K-node geometric graph, k = 200): 123 ms in one block, 23.4 ms here
// (about 2.9 us a round; 16 CTAs of 512 threads: 23.4, of 256: 26.6, of 1024: 25.8).
#include <algorithm>

#include "cluster.cuh"
#include "common.cuh"
#include "weighted.cuh"

namespace ssm {

constexpr int kWcThreads = 512;
constexpr int kWcMaxCluster = 16;
constexpr int kWcQcapMax = 2048;  // entries of a queue kept in shared memory
constexpr int kWcQcapMin = 256;
constexpr int kWcU = 1;  // edge slots per lane at a time
constexpr float kWcBand = 3.0f;
constexpr unsigned kWcInfBits = 0x7f800000u;

struct WcArgs {
  int32_t n;
  const int32_t *rowptr, *colidx;
  const unsigned *elen;
  int32_t k, start;
  int32_t *pivots;
  const float *delta;
  int32_t *spill;  // [C][4][slots] node ids: near queues by parity, far piles by parity
  int32_t *status;
  int32_t cshift, slots, qcap;
};

struct WcSmem {
  unsigned *word;           // [slots] bits of mind << 1 | queued
  int4 *near_q;             // [2][qcap] (v, row begin, row end, -)
  int4 *far_q;              // [2][qcap]
  unsigned long long *pub;  // [2][16] published by every CTA, by round parity: least far label << 32 | nodes pushed near
  unsigned *t3;             // [3] own near queue lengths, rotating with the round (raised by the pushing CTAs)
  unsigned *tf;             // own far pile length (raised by the pushing CTAs)
  unsigned *p3;             // [3] near nodes this CTA pushed, rotating
  unsigned *m3;             // [3] least far label this CTA pushed, rotating
};

// the place of queue `which` (0, 1 near; 2, 3 far) entry idx of CTA o
__device__ __forceinline__ void wc_store(const WcArgs &A, const WcSmem &S, unsigned which, unsigned o, unsigned idx, int4 e) {
  const unsigned qcap = (unsigned)A.qcap;
  int4 *q = (which < 2u ? S.near_q : S.far_q) + (which & 1u) * qcap;
  if (idx < qcap) dsmem_st_v4(dsmem_addr(q + idx, o), e);
  else if (idx - qcap < (unsigned)A.slots) A.spill[((size_t)o * 4u + which) * (unsigned)A.slots + (idx - qcap)] = e.x;
}

// own entry idx of queue `which`
__device__ __forceinline__ int4 wc_entry(const WcArgs &A, const WcSmem &S, unsigned which, unsigned r, unsigned idx) {
  const unsigned qcap = (unsigned)A.qcap;
  if (idx < qcap) return ((which < 2u ? S.near_q : S.far_q) + (which & 1u) * qcap)[idx];
  const int v = __ldcg(A.spill + ((size_t)r * 4u + which) * (unsigned)A.slots + (idx - qcap));
  return make_int4(v, __ldg(A.rowptr + v), __ldg(A.rowptr + v + 1), 0);
}

// up to kWcU edges per lane of round L: the heads' words are lowered, and the
// heads that were not queued where they now belong are pushed
__device__ __forceinline__ void wc_round(const WcArgs &A, const WcSmem &S, unsigned cs, unsigned L, unsigned fpar,
                                         unsigned tbits, const int (&v)[kWcU], const unsigned (&nb)[kWcU],
                                         const bool (&act)[kWcU]) {
  const unsigned lane = threadIdx.x & 31u, cmask = (1u << cs) - 1u, nxt = L + 1u;
  unsigned old[kWcU];
  int rb[kWcU], re[kWcU];
#pragma unroll
  for (int u = 0; u < kWcU; ++u)
    old[u] = dsmem_atomic_min_if(act[u], dsmem_addr(S.word + ((unsigned)v[u] >> cs), (unsigned)v[u] & cmask), 2u * nb[u] + 1u);
  // the row range of a head arrives while its word is on its way
#pragma unroll
  for (int u = 0; u < kWcU; ++u) {
    rb[u] = act[u] ? __ldg(A.rowptr + v[u]) : 0;
    re[u] = act[u] ? __ldg(A.rowptr + v[u] + 1) : 0;
  }
  bool near[kWcU], far[kWcU];
  unsigned idx[kWcU];
#pragma unroll
  for (int u = 0; u < kWcU; ++u) {
    const bool lower = act[u] && (old[u] >> 1) > nb[u], was = (old[u] & 1u) != 0u;
    near[u] = lower && nb[u] < tbits && (!was || (old[u] >> 1) >= tbits);
    far[u] = lower && nb[u] >= tbits && !was;
    idx[u] = dsmem_atomic_add_if(near[u] || far[u], dsmem_addr(near[u] ? S.t3 + nxt % 3u : S.tf, (unsigned)v[u] & cmask), 1u);
  }
  unsigned pushed = 0, least = 0xFFFFFFFFu;
#pragma unroll
  for (int u = 0; u < kWcU; ++u) {
    if (near[u] || far[u])
      wc_store(A, S, near[u] ? (nxt & 1u) : 2u + fpar, (unsigned)v[u] & cmask, idx[u], make_int4(v[u], rb[u], re[u], 0));
    pushed += __popc(__ballot_sync(0xffffffffu, near[u]));
    // a far node lowered again makes its label count too
    if (act[u] && (old[u] >> 1) > nb[u] && nb[u] >= tbits) least = min(least, nb[u]);
  }
  least = __reduce_min_sync(0xffffffffu, least);
  if (lane == 0) {
    if (pushed) atomicAdd(S.p3 + nxt % 3u, pushed);
    if (least != 0xFFFFFFFFu) atomicMin(S.m3 + nxt % 3u, least);
  }
}

__global__ void __launch_bounds__(kWcThreads, 1) k_wmaxmin_cluster(WcArgs A) {
  extern __shared__ __align__(16) unsigned char wc_smem[];
  __shared__ unsigned s_t3[3], s_p3[3], s_m3[3], s_tf, s_keep, s_min;
  __shared__ unsigned long long s_wbest[kWcThreads / 32];
  __shared__ unsigned long long s_best[kWcMaxCluster];
  const unsigned cs = (unsigned)A.cshift, C = 1u << cs, cmask = C - 1u;
  const unsigned r = cluster_rank();
  const unsigned tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const unsigned n = (unsigned)A.n;
  const unsigned own = n > r ? ((n - 1u - r) >> cs) + 1u : 0u;
  WcSmem S;
  S.word = reinterpret_cast<unsigned *>(wc_smem);
  S.near_q = reinterpret_cast<int4 *>(S.word + A.slots);
  S.far_q = S.near_q + 2 * (size_t)A.qcap;
  S.pub = reinterpret_cast<unsigned long long *>(S.far_q + 2 * (size_t)A.qcap);
  S.t3 = s_t3;
  S.tf = &s_tf;
  S.p3 = s_p3;
  S.m3 = s_m3;
  // a wider band than the per-source search: a round here costs its barrier, not
  // its relaxations (23.8 ms against 25.6 with the same band, 23.8 with twice it)
  const float delta = kWcBand * *A.delta;

  // counters of the next search: reset before the cluster barrier that precedes it
  auto reset_search = [&]() {
    if (tid < (unsigned)kWcMaxCluster) S.pub[tid] = ((unsigned long long)0xFFFFFFFFu << 32) | (tid == 0 ? 1u : 0u);
    if (tid < 3) {
      s_t3[tid] = s_p3[tid] = 0u;
      s_m3[tid] = 0xFFFFFFFFu;
    }
    if (tid == 3) s_tf = 0u;
  };
  for (unsigned t = tid; t < own; t += blockDim.x) S.word[t] = kWcInfBits << 1;
  reset_search();
  cluster_sync();  // every CTA of the cluster runs before any DSMEM access

  unsigned p = (unsigned)A.start;
  bool bad = false;
  for (int j = 0; j < A.k; ++j) {
    if (r == 0 && tid == 0) A.pivots[j] = (int32_t)p;
    const bool last = j == A.k - 1;
    if (last && j > 0) break;  // the final pivot needs no search
    if (tid == 0 && r == (p & cmask)) {
      S.word[p >> cs] = 1u;
      S.near_q[0] = make_int4((int)p, __ldg(A.rowptr + p), __ldg(A.rowptr + p + 1), 0);
      s_t3[0] = 1u;
    }
    __syncthreads();
    float T = delta;
    unsigned fpar = 0, gfar = 0xFFFFFFFFu;
    // a round relaxes a node whose label is final for its band, or moves T on: the
    // rounds are bounded, and the cap only guards against a fault
    const unsigned cap = 64u * (n + 16u);  // n is below 2^20: the words fit 16 CTAs
    for (unsigned L = 0;; ++L) {
      const unsigned long long pb = lane < C ? S.pub[(L & 1u) * 16u + lane] : (unsigned long long)0xFFFFFFFFu << 32;
      const unsigned tot = __reduce_add_sync(0xffffffffu, (unsigned)pb);
      gfar = min(gfar, __reduce_min_sync(0xffffffffu, (unsigned)(pb >> 32)));
      if (tot == 0 && gfar == 0xFFFFFFFFu) break;  // the same published words in every CTA: uniform
      if (L >= cap) {
        if (r == 0 && tid == 0) dev_fail(A.status, SSM_E_NUMERIC);
        bad = true;
        break;
      }
      if (tid == 0) {  // read during round L - 1; raised again from round L + 1 on
        s_t3[(L + 2u) % 3u] = 0u;
        s_p3[(L + 2u) % 3u] = 0u;
        s_m3[(L + 2u) % 3u] = 0xFFFFFFFFu;
      }
      if (tot == 0) {
        // the next band: own pile split into the near queue of round L + 1 and
        // the other pile.  gfar is at or below the least label in any pile
        const unsigned count = min(s_tf, own);
        T = fmaxf(T + delta, __uint_as_float(gfar) + delta);
        if (!(T > __uint_as_float(gfar))) T = __uint_as_float(gfar + 1u);
        const unsigned tbits = __float_as_uint(T);
        if (tid == 0) {
          s_keep = 0u;
          s_min = 0xFFFFFFFFu;
        }
        __syncthreads();
        for (unsigned t = tid; t < count; t += blockDim.x) {
          const int4 e = wc_entry(A, S, 2u + fpar, r, t);
          const unsigned w = S.word[(unsigned)e.x >> cs];
          if (!(w & 1u)) continue;  // reached and relaxed since: not far any more
          if ((w >> 1) < tbits) {
            wc_store(A, S, (L + 1u) & 1u, r, atomicAdd(s_t3 + (L + 1u) % 3u, 1u), e);
            atomicAdd(s_p3 + (L + 1u) % 3u, 1u);
          } else {
            wc_store(A, S, 2u + (fpar ^ 1u), r, atomicAdd(&s_keep, 1u), e);
            atomicMin(&s_min, w >> 1);
          }
        }
        __syncthreads();
        if (tid == 0) {
          s_tf = s_keep;
          s_m3[(L + 1u) % 3u] = s_min;
        }
        fpar ^= 1u;
        gfar = 0xFFFFFFFFu;
      } else {
        const unsigned cnt = s_t3[L % 3u], tbits = __float_as_uint(T);
        unsigned ipw = 1;  // entries per warp: small rounds are spread over all warps
        while (ipw < 32u && ipw * nwarps < cnt) ipw <<= 1;
        for (unsigned base = warp * ipw; base < cnt; base += nwarps * ipw) {
          int beg = 0, end = 0;
          unsigned dv = 0;
          if (lane < ipw && base + lane < cnt) {
            const int4 e = wc_entry(A, S, L & 1u, r, base + lane);
            const unsigned w = atomicAnd(S.word + ((unsigned)e.x >> cs), ~1u);
            if (w & 1u) {
              beg = e.y;
              end = e.z;
              dv = w >> 1;
            }
          }
          if (ipw == 1u) {
            const int b = __shfl_sync(0xffffffffu, beg, 0), en = __shfl_sync(0xffffffffu, end, 0);
            const float d0 = __uint_as_float(__shfl_sync(0xffffffffu, dv, 0));
            for (int t0 = b; t0 < en; t0 += 32 * kWcU) {
              int v[kWcU];
              unsigned nb[kWcU];
              bool act[kWcU];
#pragma unroll
              for (int u = 0; u < kWcU; ++u) {
                const int t = t0 + 32 * u + (int)lane;
                act[u] = t < en;
                v[u] = act[u] ? __ldg(A.colidx + t) : 0;
                nb[u] = act[u] ? __float_as_uint(__fadd_rn(d0, __uint_as_float(__ldg(A.elen + t)))) : 0u;
              }
#pragma unroll
              for (int u = 0; u < kWcU; ++u) act[u] = act[u] && nb[u] < kWcInfBits;
              wc_round(A, S, cs, L, fpar, tbits, v, nb, act);
            }
            continue;
          }
          int incl = end - beg;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if ((int)lane >= o) incl += t;
          }
          const int total = __shfl_sync(0xffffffffu, incl, 31);
          for (int t0 = 0; t0 < total; t0 += 32 * kWcU) {
            int v[kWcU];
            unsigned nb[kWcU];
            bool act[kWcU];
#pragma unroll
            for (int u = 0; u < kWcU; ++u) {
              const int t = t0 + 32 * u + (int)lane;
              act[u] = t < total;
              int lo = 0;  // row = first lane whose inclusive prefix exceeds t
#pragma unroll
              for (int step = 16; step >= 1; step >>= 1) {
                const int pv = __shfl_sync(0xffffffffu, incl, lo + step - 1);
                if (pv <= t) lo += step;
              }
              const int at = lo > 31 ? 31 : lo;
              const int o_end = __shfl_sync(0xffffffffu, end, at), o_incl = __shfl_sync(0xffffffffu, incl, at);
              const float d0 = __uint_as_float(__shfl_sync(0xffffffffu, dv, at));
              const int pos = o_end - (o_incl - t);
              v[u] = act[u] ? __ldg(A.colidx + pos) : 0;
              nb[u] = act[u] ? __float_as_uint(__fadd_rn(d0, __uint_as_float(__ldg(A.elen + pos)))) : 0u;
            }
#pragma unroll
            for (int u = 0; u < kWcU; ++u) act[u] = act[u] && nb[u] < kWcInfBits;
            wc_round(A, S, cs, L, fpar, tbits, v, nb, act);
          }
        }
      }
      __syncthreads();  // own push counts are final
      if (tid < C)
        dsmem_st_u64(dsmem_addr(S.pub + ((L + 1u) & 1u) * 16u + r, tid),
                     ((unsigned long long)s_m3[(L + 1u) % 3u] << 32) | s_p3[(L + 1u) % 3u]);
      cluster_sync();
    }
    if (bad) break;

    // argmax of mind over the cluster, ties to the lowest node id
    unsigned long long key = 0;
    for (unsigned t = tid; t < own; t += blockDim.x) {
      const unsigned long long c = ((unsigned long long)(S.word[t] >> 1) << 32) | (unsigned long long)(~(r + (t << cs)));
      key = c > key ? c : key;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long t = __shfl_xor_sync(0xffffffffu, key, o);
      key = t > key ? t : key;
    }
    if (lane == 0) s_wbest[warp] = key;
    __syncthreads();
    if (warp == 0) {
      key = lane < nwarps ? s_wbest[lane] : 0ull;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, key, o);
        key = t > key ? t : key;
      }
      if (lane < C) dsmem_st_u64(dsmem_addr(s_best + r, lane), key);
    }
    reset_search();  // the rounds are over in every CTA (they ended at a cluster barrier)
    cluster_sync();
    key = 0;
    for (unsigned x = 0; x < C; ++x) key = s_best[x] > key ? s_best[x] : key;
    if ((unsigned)(key >> 32) >= kWcInfBits) {  // some node was never reached
      if (r == 0 && tid == 0) dev_fail(A.status, SSM_E_DISCONNECTED);
      break;
    }
    if (last) break;
    p = ~(unsigned)key;
  }
  cluster_sync();  // no CTA leaves while another may still read its shared memory
}

// ------------------------------------------------------------------- host
struct WcShape {
  int C = 0, slots = 0, qcap = 0;
  size_t smem = 0;
};

// 16 CTAs before 8; C == 0 when no cluster holds the words in shared memory
static WcShape wc_shape(int32_t n) {
  WcShape none;
  int dev = 0, smem_max = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return none;
  if (cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return none;
  const size_t budget = (size_t)smem_max - 2 * 1024;  // static shared memory of the kernel
  const void *kern = (const void *)k_wmaxmin_cluster;
  for (int C : {16, 8}) {
    WcShape sh;
    sh.slots = (int)((((int64_t)n + C - 1) / C + 7) / 8 * 8);
    const size_t fixed = (size_t)sh.slots * 4 + 32 * sizeof(unsigned long long);
    if (fixed >= budget) continue;
    sh.qcap = (int)std::min<size_t>(kWcQcapMax, (budget - fixed) / (4 * sizeof(int4)));
    if (sh.qcap < kWcQcapMin) continue;
    sh.smem = fixed + (size_t)4 * sh.qcap * sizeof(int4);
    if (C > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      (void)cudaGetLastError();
      continue;
    }
    if (allow_dynamic_smem(kern) != cudaSuccess) {
      (void)cudaGetLastError();
      continue;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3(kWcThreads);
    cfg.dynamicSmemBytes = sh.smem;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      continue;
    }
    if (clusters < 1) continue;
    sh.C = C;
    return sh;
  }
  return none;
}

// node ids of spilled queue entries: four queues of every node's slot (slots
// are rounded up to eight per CTA)
size_t wmaxmin_spill_entries(int32_t n) { return 4 * ((size_t)n + 16 * kWcMaxCluster); }

int launch_wmaxmin_cluster(int32_t n, const int32_t *rowptr, const int32_t *colidx, const float *elen, int32_t k,
                           int32_t start, int32_t *pivots, const float *delta, int32_t *spill, int32_t *status,
                           cudaStream_t s, bool *ran) {
  *ran = false;
  const WcShape sh = wc_shape(n);
  if (sh.C == 0) return SSM_OK;
  WcArgs A;
  A.n = n; A.rowptr = rowptr; A.colidx = colidx; A.elen = (const unsigned *)elen; A.k = k; A.start = start;
  A.pivots = pivots; A.delta = delta; A.spill = spill; A.status = status;
  A.cshift = sh.C == 16 ? 4 : 3;
  A.slots = sh.slots;
  A.qcap = sh.qcap;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)sh.C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)sh.C);
  cfg.blockDim = dim3(kWcThreads);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  note_launch();
  SSM_TRY_CUDA(cudaLaunchKernelEx(&cfg, k_wmaxmin_cluster, A));
  *ran = true;
  return SSM_OK;
}

}  // namespace ssm
