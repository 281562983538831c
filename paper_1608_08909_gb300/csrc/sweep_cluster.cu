// The FP32 Jacobi sweeps of Eq. 4 for a small graph, all iterations in one
// launch of one thread-block cluster.
//
// On a graph of a few thousand nodes an iteration on the whole GPU is two
// kernels that each wait for the other (14 us at n = 1024, k = 50, of which the
// arithmetic is well below one).  Here a cluster of C CTAs (16 or 8) keeps
// everything in shared memory: every CTA holds the positions of all nodes (two
// buffers), the (w', w' d) table of every pivot and distance, and for the nodes
// it owns (every C-th, so that the hubs of a heavy-tailed graph are spread) the
// table places of their d_ip and their neighbours.  Positions are kept CTA by
// CTA: node v at (v mod C) per + v div C.  A lane has two consecutive nodes (packed FP32x2), so a pivot's
// position is one broadcast and its table row is shared by 64 nodes; the warps
// of a 64-node block share its pivots and neighbours (warp w every W-th), rows
// above `lng` entries are a warp's work each (hubs: below), and a node's W + 1 partial sums
// are added in order.  (Lanes sharing a node, each with its own pivots, took
// 1.4 to 5 times as long: every pivot position and table entry was a gather.)
// A CTA stores its new positions into the other buffer of every CTA (distributed
// shared memory; warps that would be idle each serve some of the receivers), and
// an iteration ends at the hardware's cluster barrier: every CTA makes the same
// number of them, also one that owns no node, and none writes to another after
// the last.  X^{t+1} goes into the buffer that was read before the last barrier.
//
// The update is the single-graph sweep's form about x_i: x_i + (sum_a (B - w)
// (x_i - x_p) + sum_j (x_j - x_i)(1 - 1/r)) / den, B = w d / r, with r^2 + 1e-24
// so that coincident points add nothing; only the order of a node's sum differs
// (fixed here too).  Bound by latency: shared-memory gathers, a block barrier,
// the stores and the cluster barrier.  Measured (us an iteration, two kernels on
// the whole GPU, here): grid of 1,024 nodes, k = 50: 14.1, 2.3; Barabasi-Albert
// graph of 8,000 nodes, k = 60: 18.8, 8.6; of 4,096 nodes, k = 200: 25.2, 7.8.
//
// Rows above kScHub entries, where a CTA has few of them, are cut into segments
// that all its warps share (star of 8,000 nodes: 20.5, and 21 with a warp per
// row; 6.9 so).  A CTA keeps the neighbours that its shared memory has room for
// and reads the others from L2 in every iteration, which 16 SMs of one GPC do at
// some 0.5 TB/s.
#include <algorithm>

#include "cluster.cuh"
#include "common.cuh"
#include "sweep.cuh"

namespace ssm {

constexpr int kScThreads = 1024;  // half as many where a CTA has fewer than kScWide (node, pivot) pairs
constexpr int kScWide = 8192;
// The longest row that one lane per warp walks: twice the mean degree (a warp takes
// 0.03 us over a row whatever its length: 8,000 nodes of degree 60, k = 2: 12.9 us an
// iteration so, 19.6 with rows above 16 a warp's, 14.5 in two kernels), at least
// kScLong; kScLong where the mean is above kScLaneMean
constexpr int kScLong = 16;
constexpr int kScLaneMean = 64;
constexpr int kScHub = kMidDeg;   // longest row that one warp walks, if a CTA has few that are longer
constexpr int kScMaxHubs = 64;    // (above this many they fill the warps as they are)
constexpr int kScHubSegs = 128;   // a hub's entries per warp: so that these and one per hub are enough,
constexpr int kScMinSeg = 256;    // and at least this many
constexpr int kScMaxCluster = 16;
constexpr int kScMaxN = 8192;     // node ids in 16 bits
constexpr int kScMaxD = 4095;     // d^2 exact in FP32
constexpr int kScMinIters = 4;    // the tables are formed by every launch
// Above that mean an iteration takes a CTA some 0.1 us per thousand neighbours and
// 0.03 a row, two kernels at least 14 (k = 2) to 19 us (k = 50): rows count for
// kScRowCost neighbours (more than their time, for the tables of a short run), and
// above kScMaxDense the two kernels are taken.  (Here and there, k = 2 / 50: 4,000
// nodes of degree 200 12.4 / 12.4 and 13.6 / 19; of degree 400 19 / 19 and 14 / 20;
// 8,000 of degree 100 23 / 26 and 15 / 19; clique of 1,500 16.5 / 17 and 15.5 / 19.)
constexpr int64_t kScRowCost = 500, kScMaxDense = 187700;
constexpr float kScR2Floor = 1e-24f;

struct ScArgs {
  int32_t n, k, dmax, per, perp, warps, iters;  // nodes per CTA (perp: up to whole blocks), warps per 64-node block
  int32_t lng;   // longest row that one lane per warp walks
  int32_t ecap;  // neighbour ids of a CTA kept in shared memory
  int32_t hubs;  // there are rows above kScHub: the hubs' lists are part of the shared memory
  const int32_t *rowptr, *colidx, *pivots, *cnt_off;
  const uint32_t *cnt;
  const uint16_t *dip;
  float2 *pos;
  double tol;
  int32_t *iters_done;
  double *rel_change;
  int32_t *status;
};

// rows of a CTA that all its warps share, in segments
struct ScHubs {
  float2 sum[kScHubSegs + kScMaxHubs];
  int seg[kScHubSegs + kScMaxHubs];  // node | number of the segment << 16
  int node[kScMaxHubs], first[kScMaxHubs];  // a hub, and the place of its first segment
};

__device__ __forceinline__ float sc_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void dsmem_st_f2(uint32_t a, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

__device__ __forceinline__ void dsmem_st_d2(uint32_t a, double x, double y) {
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(x), "d"(y) : "memory");
}

// the term of a neighbour at place j about x
__device__ __forceinline__ void sc_edge(const float2 *Xc, int j, float2 x, float &sx, float &sy) {
  const float2 q = Xc[j];
  const float ex = q.x - x.x, ey = q.y - x.y;
  const float r2 = fmaf(ex, ex, ey * ey);
  const float f = r2 > 0.f ? 1.f - sc_rsqrt(r2) : 0.f;
  sx = fmaf(ex, f, sx);
  sy = fmaf(ey, f, sy);
}

// the whole warp: the terms of the neighbours whose places are place[b .. e - 1],
// or (place null) those of the graph's entries col[b .. e - 1], at(id) their
// places, about the node at place `self` (whose own term, past the end, is
// zero); the sum in every lane
template <class At>
__device__ __forceinline__ float2 sc_row(const float2 *Xc, const uint16_t *place, const int32_t *__restrict__ col, int b,
                                         int e, int self, At at) {
  constexpr int U = 8;  // neighbours per lane in flight
  const float2 x = Xc[self];
  float sx = 0.f, sy = 0.f;
  const int lane = (int)(threadIdx.x & 31u);
  auto edges = [&](const int (&j)[U]) {
#pragma unroll
    for (int q = 0; q < U; ++q) sc_edge(Xc, j[q], x, sx, sy);
  };
  if (place && e - b <= 16 * U) {
    for (int t = b + lane; t < e; t += 32) sc_edge(Xc, place[t], x, sx, sy);
  } else if (place) {
    for (int t0 = b; t0 < e; t0 += 32 * U) {
      int j[U];
#pragma unroll
      for (int q = 0; q < U; ++q) j[q] = t0 + 32 * q + lane < e ? place[t0 + 32 * q + lane] : self;
      edges(j);
    }
  } else {
    int v[U];  // the next ids are on their way while these are used
#pragma unroll
    for (int q = 0; q < U; ++q) v[q] = __ldg(col + min(b + lane + 32 * q, e - 1));
    for (int t0 = b; t0 < e; t0 += 32 * U) {
      int j[U];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        j[q] = t0 + 32 * q + lane < e ? at(v[q]) : self;
        v[q] = __ldg(col + min(t0 + 32 * (U + q) + lane, e - 1));
      }
      edges(j);
    }
  }
  __syncwarp();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sx += __shfl_xor_sync(0xffffffffu, sx, o);
    sy += __shfl_xor_sync(0xffffffffu, sy, o);
  }
  return make_float2(sx, sy);
}

__global__ void __launch_bounds__(kScThreads, 1) k_sweep_cluster(ScArgs A) {
  extern __shared__ __align__(16) unsigned char sc_smem[];
  __shared__ double s_red[2][kScThreads / 32];
  __shared__ __align__(16) double2 s_part[2][kScMaxCluster];
  const int n = A.n, k = A.k, D = A.dmax + 1;
  unsigned C;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
  const size_t stride = (size_t)A.per * C;  // the last CTAs' places may be one short
  float2 *X = reinterpret_cast<float2 *>(sc_smem);            // [2][stride]
  float2 *tab = X + 2 * stride;                               // [k][D] (-w, w d)
  float2 *part = tab + (size_t)k * D;                         // [warps + 1][perp] partial sums; the last: long rows
  float *den = reinterpret_cast<float *>(part + (size_t)(A.warps + 1) * A.perp);  // [perp]
  int32_t *rows = reinterpret_cast<int32_t *>(den + A.perp);  // [perp + 1] row starts, local
  int32_t *lrows = rows + A.perp + 2;                         // [perp] long rows
  int32_t *start = lrows + A.perp;                            // [perp] entry of the graph's rows less the local one
  int32_t *pnode = start + A.perp;                            // [k]
  uint16_t *place = reinterpret_cast<uint16_t *>(pnode + ((k + 1) & ~1));  // [k][perp]
  ScHubs *hub = reinterpret_cast<ScHubs *>(place + (size_t)k * A.perp);
  uint16_t *cols = reinterpret_cast<uint16_t *>(hub + (A.hubs ? 1 : 0));  // [ecap]
  __shared__ int s_nlong, s_nhub, s_hubsum, s_nseg;
  const unsigned r = cluster_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int T = (int)blockDim.x;
  const int i0 = (int)r * A.per, own = n > (int)r ? (n - 1 - (int)r) / (int)C + 1 : 0;  // nodes r, r + C, ...
  const int cs = 31 - __clz((int)C);
  auto at = [&](int v) { return (v & ((int)C - 1)) * A.per + (v >> cs); };

  for (int i = tid; i < n; i += T) X[at(i)] = A.pos[i];
  // w = s / d^2, w d = s / d from exact operands (s <= n, d^2 < 2^24), each rounded once
  for (int t = tid; t < k * D; t += T) {
    const int a = t / D, d = t - a * D;
    const int o = __ldg(A.cnt_off + a), ecc = __ldg(A.cnt_off + a + 1) - o - 1;
    float2 w = make_float2(0.f, 0.f);
    if (d >= 2) {
      const float s = (float)__ldg(A.cnt + o + min(d >> 1, ecc)), fd = (float)d;
      w = make_float2(-__fdiv_rn(s, fd * fd), __fdiv_rn(s, fd));
    }
    tab[t] = w;
  }
  for (int a = tid; a < k; a += T) {
    int p = __ldg(A.pivots + a);
    if ((unsigned)p >= (unsigned)n) {  // a pivot id outside the graph: recorded, read as node 0
      dev_fail(A.status, SSM_E_ARG);
      p = 0;
    }
    pnode[a] = at(p);
  }
  if (tid == 0) {
    s_nlong = s_nhub = s_hubsum = s_nseg = 0;
    rows[0] = 0;
  }
  if (warp == 0) {  // local row starts
    int sum = 0;
    for (int b = 0; b < A.perp; b += 32) {
      const int li = b + lane, v = li * (int)C + (int)r;
      int deg = li < own ? __ldg(A.rowptr + v + 1) - __ldg(A.rowptr + v) : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, deg, o);
        if (lane >= o) deg += t;
      }
      rows[li + 1] = sum + deg;
      sum += __shfl_sync(0xffffffffu, deg, 31);
    }
  }
  __syncthreads();
  auto here = [&](int li) { return rows[li + 1] <= A.ecap; };  // a row's neighbours are kept; else read from the graph
  auto keep = [&](int li, int first, int step) {  // a row's neighbours, eight loads in flight
    if (!here(li)) return;
    const int32_t *col = A.colidx + start[li];
    const int e = rows[li + 1];
    for (int t = rows[li] + first; t < e; t += 8 * step) {
      int v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = __ldg(col + min(t + q * step, e - 1));
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (t + q * step < e) cols[t + q * step] = (uint16_t)at(v[q]);
    }
  };
  for (int li = tid; li < own; li += T) {
    const int e = __ldg(A.rowptr + li * (int)C + (int)r), t0 = rows[li], len = rows[li + 1] - t0;
    start[li] = e - t0;
    if (len <= A.lng) keep(li, 0, 1);
    if (len > kScHub) {
      atomicAdd(&s_nhub, 1);
      atomicAdd(&s_hubsum, len);
    }
  }
  __syncthreads();
  const int nhub = A.hubs && s_nhub <= kScMaxHubs ? s_nhub : 0, hublen = nhub ? kScHub : 0x7FFFFFFF;
  const int seg = max(kScMinSeg, (s_hubsum + kScHubSegs - 1) / kScHubSegs);
  __syncthreads();
  if (tid == 0) s_nhub = 0;
  __syncthreads();
  // long rows and hubs, in any order: every row is a sum of its own
  for (int li = tid; li < own; li += T) {
    const int len = rows[li + 1] - rows[li];
    if (len > hublen) {
      const int h = atomicAdd(&s_nhub, 1), c = (len + seg - 1) / seg, first = atomicAdd(&s_nseg, c);
      hub->node[h] = li;
      hub->first[h] = first;
      for (int q = 0; q < c; ++q) hub->seg[first + q] = li | q << 16;
    } else if (len > A.lng) {
      lrows[atomicAdd(&s_nlong, 1)] = li;
    }
  }
  __syncthreads();
  for (int q = warp; q < s_nlong; q += T / 32) keep(lrows[q], lane, 32);  // long rows, a warp each
  for (int h = 0; h < nhub; ++h) keep(hub->node[h], tid, T);              // hubs, all threads
  for (int t = tid; t < A.perp * k; t += T) {
    const int a = t / A.perp, li = t - a * A.perp;
    unsigned d = li < own ? __ldg(A.dip + (size_t)a * n + li * (int)C + (int)r) : 0u;
    if (d > (unsigned)A.dmax) {  // a wrong dmax hint: recorded, clamped
      dev_fail(A.status, SSM_E_ARG);
      d = (unsigned)A.dmax;
    }
    place[t] = (uint16_t)(a * D + (int)d);
  }
  __syncthreads();
  for (int li = tid; li < A.perp; li += T) {  // denominators: they do not change between iterations
    const int deg = rows[li + 1] - rows[li];
    float acc = 0.f;
    for (int a = 0; a < k; ++a) acc -= tab[place[a * A.perp + li]].x;
    den[li] = acc + (float)deg;
    part[(size_t)A.warps * A.perp + li] = make_float2(0.f, 0.f);
  }
  const int W = A.warps, blocks = A.perp / 64, blk = warp / W, wb = warp - blk * W;
  const int l0 = 64 * blk + 2 * lane;  // this lane's nodes l0, l0 + 1 (blk < blocks)
  // warps of own nodes, and how many warps share the stores of one of them
  const int nw = (own + 31) / 32, share = nw > 0 ? max(1, min((int)C, T / 32 / nw)) : 1;
  cluster_sync();  // every CTA of the cluster runs, and has read pos, before any remote write

  int it = 0;
  for (; it < A.iters; ++it) {
    const float2 *Xc = X + (size_t)(it & 1) * stride;
    float2 *Xn = X + (size_t)((it & 1) ^ 1) * stride;
    const bool change = A.tol > 0.0 || it + 1 == A.iters;
    if (blk < blocks) {
      const float2 x0 = l0 < own ? Xc[i0 + l0] : make_float2(0.f, 0.f), x1 = l0 + 1 < own ? Xc[i0 + l0 + 1] : make_float2(0.f, 0.f);
      const float2 xi = make_float2(x0.x, x1.x), yi = make_float2(x0.y, x1.y), tiny = make_float2(kScR2Floor, kScR2Floor);
      float2 ax = make_float2(0.f, 0.f), ay = ax;
#pragma unroll 4
      for (int a = wb; a < k; a += W) {
        const unsigned pl = *reinterpret_cast<const unsigned *>(place + a * A.perp + l0);
        const float2 w0 = tab[pl & 0xFFFFu], w1 = tab[pl >> 16], p = Xc[pnode[a]];
        const float2 dx = __fadd2_rn(xi, make_float2(-p.x, -p.x)), dy = __fadd2_rn(yi, make_float2(-p.y, -p.y));
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, tiny));
        const float2 c = __ffma2_rn(make_float2(w0.y, w1.y), make_float2(sc_rsqrt(r2.x), sc_rsqrt(r2.y)),
                                    make_float2(w0.x, w1.x));  // B - w
        ax = __ffma2_rn(c, dx, ax);
        ay = __ffma2_rn(c, dy, ay);
      }
      float sx[2] = {ax.x, ax.y}, sy[2] = {ay.x, ay.y};
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int rb = rows[l0 + q], re = rows[l0 + q + 1];
        if (re - rb <= A.lng) {
          const bool in = re <= A.ecap;
          for (int t = rb + wb; t < re; t += W)
            sc_edge(Xc, in ? cols[t] : at(__ldg(A.colidx + start[l0 + q] + t)), q ? x1 : x0, sx[q], sy[q]);
        }
        part[(size_t)wb * A.perp + l0 + q] = make_float2(sx[q], sy[q]);
      }
    }
    for (int q = warp; q < s_nlong; q += T / 32) {
      const int li = lrows[q];
      const float2 v = sc_row(Xc, here(li) ? cols : nullptr, A.colidx + start[li], rows[li], rows[li + 1], i0 + li, at);
      if (lane == 0) part[(size_t)W * A.perp + li] = v;
    }
    if (nhub) {  // a segment per warp, then a hub per warp
      for (int q = warp; q < s_nseg; q += T / 32) {
        const int li = hub->seg[q] & 0xFFFF, b = rows[li] + (hub->seg[q] >> 16) * seg;
        const float2 v = sc_row(Xc, here(li) ? cols : nullptr, A.colidx + start[li], b, min(b + seg, rows[li + 1]), i0 + li, at);
        if (lane == 0) hub->sum[q] = v;
      }
      __syncthreads();
      for (int h = warp; h < nhub; h += T / 32) {
        const int li = hub->node[h], c = (rows[li + 1] - rows[li] + seg - 1) / seg;
        float sx = 0.f, sy = 0.f;
        for (int q = lane; q < c; q += 32) {
          sx += hub->sum[hub->first[h] + q].x;
          sy += hub->sum[hub->first[h] + q].y;
        }
        __syncwarp();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          sx += __shfl_xor_sync(0xffffffffu, sx, o);
          sy += __shfl_xor_sync(0xffffffffu, sy, o);
        }
        if (lane == 0) part[(size_t)W * A.perp + li] = make_float2(sx, sy);
      }
    }
    __syncthreads();
    float cn = 0.f, cd = 0.f;
    for (int u = warp; u < nw * share; u += T / 32) {
      const int sh = u / nw, li = (u - sh * nw) * 32 + lane;
      if (li >= own) continue;
      const float2 x = Xc[i0 + li];
      float ax = 0.f, ay = 0.f;
#pragma unroll 4
      for (int w = 0; w <= W; ++w) {
        const float2 v = part[(size_t)w * A.perp + li];
        ax += v.x;
        ay += v.y;
      }
      const float dn = den[li];
      const float ex = dn > 0.f ? ax / dn : 0.f, ey = dn > 0.f ? ay / dn : 0.f;
      for (unsigned c = (unsigned)sh; c < C; c += (unsigned)share)
        dsmem_st_f2(dsmem_addr(Xn + i0 + li, c), make_float2(x.x + ex, x.y + ey));
      if (sh > 0) continue;
      const float chk = ax + ay;
      if (!(chk == chk)) dev_fail(A.status, SSM_E_NUMERIC);
      cn = fmaf(ex, ex, fmaf(ey, ey, cn));
      cd = fmaf(x.x, x.x, fmaf(x.y, x.y, cd));
    }
    __syncwarp();
    if (change) {  // ||X^{t+1} - X^t||_F / ||X^t||_F: lanes, warps and CTAs in a fixed order
      double tn = (double)cn, td = (double)cd;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        tn += __shfl_xor_sync(0xffffffffu, tn, o);
        td += __shfl_xor_sync(0xffffffffu, td, o);
      }
      if (lane == 0) {
        s_red[0][warp] = tn;
        s_red[1][warp] = td;
      }
      __syncthreads();
      if (warp == 0) {
        tn = lane < T / 32 ? s_red[0][lane] : 0.0;
        td = lane < T / 32 ? s_red[1][lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          tn += __shfl_xor_sync(0xffffffffu, tn, o);
          td += __shfl_xor_sync(0xffffffffu, td, o);
        }
        if ((unsigned)lane < C) dsmem_st_d2(dsmem_addr(&s_part[it & 1][r], (unsigned)lane), tn, td);
      }
    }
    __syncwarp();
    cluster_sync();  // X^{t+1} and the partial sums are everywhere
    if (change) {
      double num = 0.0, dn = 0.0;
      for (unsigned c = 0; c < C; ++c) {
        num += s_part[it & 1][c].x;
        dn += s_part[it & 1][c].y;
      }
      const double rel = dn > 0.0 ? sqrt(num) / sqrt(dn) : 0.0;
      if (r == 0 && tid == 0) {
        *A.rel_change = rel;
        *A.iters_done = it + 1;
      }
      if (A.tol > 0.0 && rel < A.tol) {  // the same sums in every CTA: uniform
        ++it;
        break;
      }
    }
  }
  const float2 *Xf = X + (size_t)(it & 1) * stride;
  for (int t = tid; t < own; t += T) A.pos[t * (int)C + (int)r] = Xf[i0 + t];
}

static size_t sc_smem_bytes(int32_t C, int32_t per, int32_t k, int32_t D, int32_t perp, int32_t warps, int32_t hubs) {
  return (hubs ? sizeof(ScHubs) : 0) + ((size_t)2 * per * C + (size_t)k * D + (size_t)(warps + 1) * perp) * sizeof(float2) + (size_t)perp * 4 +
         (size_t)(3 * perp + 2) * 4 + (size_t)((k + 1) & ~1) * 4 + (size_t)perp * k * 2;
}

int launch_sweep_cluster(int32_t n, int64_t m, const int32_t *rowptr, const int32_t *colidx, int32_t k,
                         const int32_t *pivots, const uint16_t *dip, const int32_t *cnt_off, const uint32_t *cnt,
                         int32_t dmax, int32_t long_rows, float2 *pos, int32_t iters, double tol, int32_t *iters_done,
                         double *rel_change, int32_t *status, cudaStream_t s, int *blocks) {
  *blocks = 0;
  if (n > kScMaxN || dmax > kScMaxD || iters < kScMinIters || (int64_t)k * (dmax + 1) > 65535) return SSM_OK;
  int dev = 0, smem_max = 0;
  SSM_TRY_CUDA(cudaGetDevice(&dev));
  SSM_TRY_CUDA(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  const size_t budget = (size_t)smem_max - 2 * 1024;  // static shared memory of the kernel
  const void *kern = (const void *)k_sweep_cluster;
  for (int C : {16, 8}) {
    ScArgs A;
    A.hubs = long_rows > 0;
    A.per = (n + C - 1) / C;
    A.perp = (A.per + 63) / 64 * 64;
    const int threads = (int64_t)A.per * k < kScWide ? kScThreads / 2 : kScThreads;
    A.warps = std::max(1, threads / 32 / (A.perp / 64));
    if (A.perp / 64 > threads / 32) continue;  // a warp has one block of nodes
    // fewer partial sums where the table leaves no room for them
    while (A.warps > 1 && sc_smem_bytes(C, A.per, k, dmax + 1, A.perp, A.warps, A.hubs) > budget) A.warps /= 2;
    const size_t fixed = sc_smem_bytes(C, A.per, k, dmax + 1, A.perp, A.warps, A.hubs);
    if (fixed > budget) continue;
    A.ecap = (int32_t)std::min<size_t>((budget - fixed) / 2, (size_t)(2 * m));
    const int64_t mean = 2 * m / n;
    A.lng = mean > kScLaneMean ? kScLong : (int32_t)std::max<int64_t>(kScLong, 2 * mean);
    if (mean > kScLaneMean && kScRowCost * A.per + 2 * m / C > kScMaxDense) continue;
    const size_t smem = fixed + (size_t)A.ecap * 2;
    A.n = n; A.k = k; A.dmax = dmax; A.iters = iters; A.rowptr = rowptr; A.colidx = colidx; A.pivots = pivots;
    A.cnt_off = cnt_off; A.cnt = cnt; A.dip = dip; A.pos = pos; A.tol = tol; A.iters_done = iters_done;
    A.rel_change = rel_change; A.status = status;
    if (C > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      (void)cudaGetLastError();
      continue;
    }
    SSM_TRY_CUDA(allow_dynamic_smem(kern));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      continue;
    }
    if (clusters < 1) continue;
    note_launch();
    SSM_TRY_CUDA(cudaLaunchKernelEx(&cfg, k_sweep_cluster, A));
    *blocks = C;
    return SSM_OK;
  }
  return SSM_OK;
}

}  // namespace ssm
