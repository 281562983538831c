// Pivot sampling "k-means sp" (Section 4.1): k max/min-sp pivots are refined
// by k-means over the shortest-path entries of those pivots.
//
// Node i is the point y_i = (d_0i, ..., d_{k-1,i}) of Z^k (column i of the
// pivot-major d_ip table); cluster a starts with centre y_{p_a}.  A centre is
// kept as an exact integer sum S_a (k entries) and a member count n_a, so
// every data-dependent sum is an exact integer and does not depend on the
// order in which the GPU forms it:
//   t_ia = y_i . S_a                                   (exact, 64-bit)
//   g(i,a) = alpha_a - beta_a * t_ia                   (FP64, two roundings)
//   alpha_a = sum_b (S_ab / n_a)^2 in b order, beta_a = 2 / n_a
// g(i,a) is ||y_i - S_a/n_a||^2 minus the common ||y_i||^2; node i joins the
// cluster with the least g, ties to the lowest a.  Passes repeat (at most
// max_iter; the paper caps its k-means at 50) until a pass after the first
// changes no node; between passes S_a, n_a become the members' sum and count
// (a cluster left empty keeps its centre).  The new pivot of cluster a is the
// member minimising the exact integer n_a ||y_i||^2 - 2 t_ia, ties to the
// lowest node id; an empty cluster keeps its max/min pivot.
//
// GB300 layout.  The assignment is the dense part (n k^2 products per pass)
// and runs on the tensor cores as a filter whose error is bounded:
//  * y is centred, y' = y - m with m half the largest distance (a common shift
//    of points and centres moves every g(i,.) of a node by the same amount),
//    and kept once per call as FP16 (exact) in the shared-memory image of the
//    operand, 128 nodes per tile;
//  * a centre's entries S_ab / n_a - m are rounded to multiples of 2^-f and
//    cut into two signed digits of w bits (w <= 12: exact in FP16), f and w
//    from k and the largest distance so that a sum of k products stays at or
//    below 2^24: every FP32 accumulator then holds an exact integer;
//  * from the two accumulators a thread forms h_a, an FP32 value within tau_i
//    / 2 of g(i,a) less the common shift, keeps the two least, and when they
//    are more than tau_i apart the least is the least g as well.  tau_i bounds
//    twice the rounding of the centres (2^-f sum_b |y'_ib|), of the FP32
//    evaluation and of the FP64 definition itself;
//  * the other nodes (a few in a thousand on a small-world graph, a few in a
//    hundred on a large-diameter one) are listed and decided by the definition
//    itself, a warp each, in exact integers and FP64 (k_km_resolve).
// So the assignment is the definition's for every node, whatever the filter's
// width.  k_km_assign_tc holds the centres' digits of all clusters in shared
// memory (k <= 208) and streams the node tiles: one thread copies, one issues
// the MMAs (M = 128 nodes, N = both digits of half the clusters), and eight warps
// per half read its accumulators while the other half is multiplied.
// The centres are updated by the nodes that changed cluster only (integer
// atomics on the members' sums: order-free).
// Where the filter does not apply (k > 208, or distances so large that a digit
// would have fewer than 7 bits) k_km_assign evaluates every g in 64-bit integer
// multiply-adds and FP64: a block takes 64 nodes x 64 clusters, 4 x 4 per
// thread; which of the two runs is decided on the device (the largest distance
// is not known to the host).
// Measured (GB300, Barabasi-Albert graph of 2^20 nodes, k = 200, 50 passes): 487 ms
// with every g in integers and FP64 on the CUDA cores and the centres summed
// from all nodes in each pass (7.4 + 2.2 ms a pass), 12.6 ms now.  Of a pass'
// 0.20-0.24 ms the filter takes 142 us (the MMAs 2,600 of 4,900 cycles per tile,
// the rest waiting for the next tile's entries and for the accumulators to be
// read; reading the images alone would take 64 us of HBM), the open nodes
// 22-34 us, the moves 85 us (pass 2) to 22 us (pass 50), the centres 6 us.
// Every pass is launched up front and stops on the device (no host round
// trip), so the call is asynchronous.
// The filter's arrays take as much memory as the table itself; a caller who has
// less than they need gets the integer products instead.
// Exactness needs n * max(d) < 2^32 (32-bit centre sums) and
// n * k * max(d)^2 < 2^53 (t and n_a ||y||^2 exact in FP64 / int64); both are
// checked on the device (SSM_E_ARG).
#include <cuda_fp16.h>

#include <algorithm>

#include "common.cuh"
#include "tc.cuh"

namespace ssm {

constexpr int kKmMaxK = 1024;
constexpr int kKmNodes = 64;     // k_km_assign: nodes per tile
constexpr int kKmClusters = 64;  // clusters per shared-memory chunk
constexpr int kKmThreads = 256;  // 16 node groups x 16 cluster groups, 4 x 4 each
constexpr int kKmChunk = 64;     // pivots (entries of y) staged at a time

// k_km_assign_tc: the operand images.  Rows (nodes or clusters) in groups of
// eight, entries (pivots) in groups of eight: a core matrix is 8 rows x 16
// bytes, contiguous; groups of rows follow one another, then groups of entries
constexpr int kKtMaxK = 208;                       // both digits of the centres and one node tile fill the shared memory
constexpr int kKtTile = 128;                       // nodes per tile (M)
constexpr int kKtGroups = 4;                       // groups of clusters, four warps each
constexpr int kKtHalves = 2;                       // two groups share accumulators and MMAs
constexpr int kKtThreads = 32 * (4 * kKtGroups + 3);
constexpr int kKtParts = 4;                        // parts of a node image that are copied and released on their own
constexpr unsigned kKtStepBytes = kKtTile * 32u;   // node tile, 16 entries (one MMA's K)
constexpr int kKtMinBits = 7;                      // least digit width the filter is used with
constexpr int kKtMaxStrips = 4;                    // strips of 16 clusters in a group (13 over 4, rounded up)
constexpr unsigned kKtCols = 256;                  // TMEM columns between the halves' accumulators
constexpr float kKtFar = 1e38f;                    // h of a column that is no cluster

__host__ __device__ inline int kt_pad(int k) { return (k + 15) / 16 * 16; }
__host__ __device__ inline unsigned kt_tile_bytes(int k) { return (unsigned)(kt_pad(k) / 16) * kKtStepBytes; }
// clusters kt_split(k, g) .. kt_split(k, g + 1) - 1 are group g (whole strips; some are empty when k <= 48)
__host__ __device__ inline int kt_split(int k, int g) {
  const int strips = kt_pad(k) / 16;
  return 16 * ((strips * g + kKtGroups - 1) / kKtGroups);
}
__host__ __device__ inline unsigned kt_digit_bytes(int k) { return (unsigned)kt_pad(k) * (unsigned)kt_pad(k) * 4u; }
// the first cluster of half h
__host__ __device__ inline int kt_half(int k, int h) { return kt_split(k, h * (kKtGroups / kKtHalves)); }
// row of cluster a's digit (0 high, 1 low) in the centres' image: a half's high
// digits, its low digits, then the other half's
__device__ __forceinline__ int kt_row(int k, int a, int dig) {
  const int h = a >= kt_half(k, 1) ? 1 : 0, lo = kt_half(k, h), num = kt_half(k, h + 1) - lo;
  return 2 * lo + dig * num + (a - lo);
}
// byte offset of entry b of row r in an image with `rows` rows
__host__ __device__ inline unsigned kt_at(int rows, int r, int b) {
  return (((unsigned)(b >> 3) * (unsigned)(rows >> 3) + (unsigned)(r >> 3)) << 7) + ((unsigned)(r & 7) << 4) +
         ((unsigned)(b & 7) << 1);
}

// per call, from k and the largest distance (k_km_init)
struct KmFilter {
  int32_t on;     // the tensor-core filter is used
  int32_t m;      // shift of the distances
  int32_t w;      // bits per digit
  float up;       // 2^f
  float s0, s1;   // -2^(1-f), -2^(1-f+w): weights of the two accumulators in h
  float t0, t1;   // tau_i = t0 + t1 sum_b |y'_ib|
};

struct KmState {
  unsigned *S;               // [k][kt_pad(k)] centre sums (row a = cluster a, zeros past k)
  unsigned *ST;              // [k][k] the same transposed (row b = pivot b)
  unsigned *M;               // [k][k] sums over the present members
  unsigned *cnt;             // [k] member counts of the centres
  unsigned *mcnt;            // [k] present members
  double *alpha, *beta;      // [k]
  double *sq;                // [k][k] squares of the centres' entries (alpha's terms), with the filter
  int32_t *stop;             // set when the passes are over (or on an error)
  unsigned *dmax;            // largest d_ip entry
  KmFilter *filt;
  unsigned *moved;           // [2] by pass parity: entries of `list`
  unsigned *open, *wide;     // [2] entries at the front (few candidates) and at the back (all clusters) of `unsure`
  int4 *list;                // [n] (node, previous cluster, new cluster, -) of nodes that changed
  int2 *unsure;              // [n] (node, candidates: four bytes) of nodes the filter leaves open
  float *tau;                // [n]
  float *hbase;              // [kt_pad(k)] sum_b (centre - m)^2 (kKtFar past k)
  unsigned char *digits;     // centres' digit image, 2 kt_pad(k) rows
  unsigned char *image;      // node images, one per tile
  long long *vbest;          // [k] pivot choice: least n_a ||y||^2 - 2 t
  int32_t *pbest;            // [k] lowest node id attaining it
  long long *vnode;          // [n] that value per node
};

// largest entry: 16-byte loads, packed 16-bit maxima
__global__ void k_km_dmax(int64_t count, const uint16_t *__restrict__ dip, unsigned *__restrict__ out) {
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, gs = (int64_t)gridDim.x * blockDim.x;
  const int64_t head = min(count, (int64_t)(((16u - (unsigned)((uintptr_t)dip & 15u)) & 15u) / 2u));
  const int64_t quads = (count - head) / 8;
  const uint4 *q = reinterpret_cast<const uint4 *>(dip + head);
  unsigned m2 = 0u;
#pragma unroll 4
  for (int64_t t = gt; t < quads; t += gs) {
    const uint4 v = __ldg(q + t);
    m2 = __vmaxu2(m2, __vmaxu2(__vmaxu2(v.x, v.y), __vmaxu2(v.z, v.w)));
  }
  unsigned m = max(m2 & 0xFFFFu, m2 >> 16);
  const int64_t rest = head + 8 * quads;
  for (int64_t t = gt; t < head; t += gs) m = max(m, (unsigned)__ldg(dip + t));
  for (int64_t t = rest + gt; t < count; t += gs) m = max(m, (unsigned)__ldg(dip + t));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

// centre a = y of pivot a; the exactness bounds are checked and the filter's
// width is chosen here
__global__ void k_km_init(int32_t n, int32_t k, int tc, const uint16_t *__restrict__ dip,
                          const int32_t *__restrict__ piv, KmState W, int32_t *__restrict__ status) {
  const unsigned dmx = *W.dmax;
  const double dm = (double)dmx;
  if ((double)n * dm >= 4294967296.0 || (double)n * (double)k * dm * dm >= 9007199254740992.0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      dev_fail(status, SSM_E_ARG);
      *W.stop = 1;
      W.filt->on = 0;
    }
    return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    KmFilter F = {};
    F.m = (int32_t)((dmx + 1u) / 2u);
    const int64_t c = max(1, F.m);  // |y'| and |centre - m| are at most c
    int w = 12;
    while (w > 1 && (int64_t)k * c * (1ll << (w - 1)) > (1ll << 24)) --w;
    F.w = w;
    F.on = tc && c <= 2048 && w >= kKtMinBits ? 1 : 0;
    int f = 0;
    if (F.on) {  // the largest f with c 2^f <= 2^(2w-1) - 2^w
      const int64_t top = (1ll << (2 * w - 1)) - (1ll << w);
      while ((c << (f + 1)) <= top) ++f;
    }
    F.up = (float)(1ll << f);
    F.s0 = -2.0f / F.up;
    F.s1 = F.s0 * (float)(1 << w);
    // |h - (g - shift)| is at most the centres' rounding (2 * 2^-f / 2 per entry of
    // y'), four FP32 roundings of values up to k c^2 + 2 c sum|y'|, and the
    // rounding of g itself (k + 8 FP64 roundings of values up to k max(d)^2,
    // the shift's share included); tau is twice that, rounded up
    const double fc = (double)c, fp = 4.0 / 16777216.0;
    const double own = (double)k * dm * dm * (double)(k + 8) * 4.5e-16;
    F.t1 = (float)(2.002 * (1.0 / (double)(1ll << f) + 2.0 * fc * fp));
    F.t0 = (float)(2.002 * ((double)k * fc * fc * fp + own));
    *W.filt = F;
  }
  for (int a = blockIdx.x; a < k; a += gridDim.x) {
    int p = __ldg(piv + a);
    if ((unsigned)p >= (unsigned)n) {
      if (threadIdx.x == 0) {
        dev_fail(status, SSM_E_ARG);
        *W.stop = 1;
      }
      p = 0;
    }
    for (int b = threadIdx.x; b < k; b += blockDim.x) {
      W.S[(size_t)a * kt_pad(k) + b] = __ldg(dip + (size_t)b * n + p);
      W.M[(size_t)a * k + b] = 0u;
    }
    for (int b = k + threadIdx.x; b < kt_pad(k); b += blockDim.x) W.S[(size_t)a * kt_pad(k) + b] = 0u;
    if (threadIdx.x == 0) {
      W.cnt[a] = 1u;
      W.mcnt[a] = 0u;
    }
  }
}

// y' of every node in FP16, tile by tile in the operand image, and tau.  A
// thread takes a node and every second group of eight pivots: the loads of a
// warp are 64 consecutive bytes of a row, its stores 512 consecutive bytes.
// Bound by HBM (2 k n bytes in, 2 kt_pad(k) n out, once per call).
__global__ void __launch_bounds__(256) k_km_image(int32_t n, int32_t k, const uint16_t *__restrict__ dip, KmState W) {
  __shared__ int part[kKtTile];
  const KmFilter F = *W.filt;
  if (!F.on) return;
  const int r = threadIdx.x & (kKtTile - 1), h = threadIdx.x >> 7;
  const int groups = kt_pad(k) / 8;
  for (int64_t tile = blockIdx.x; tile * kKtTile < n; tile += gridDim.x) {
    const int64_t i = tile * kKtTile + r;
    unsigned char *img = W.image + tile * kt_tile_bytes(k);
    int sum = 0;
    for (int gq = h; gq < groups; gq += 2) {
      unsigned word[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        int y[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int b = 8 * gq + 2 * e + q;
          y[q] = b < k && i < n ? (int)__ldg(dip + (size_t)b * n + i) - F.m : 0;
          sum += abs(y[q]);
        }
        const __half2 v = __halves2half2(__int2half_rn(y[0]), __int2half_rn(y[1]));
        word[e] = *reinterpret_cast<const unsigned *>(&v);
      }
      *reinterpret_cast<uint4 *>(img + kt_at(kKtTile, r, 8 * gq)) = make_uint4(word[0], word[1], word[2], word[3]);
    }
    if (h) part[r] = sum;
    __syncthreads();
    if (!h && i < n) W.tau[i] = F.t0 + F.t1 * (float)(sum + part[r]);
    __syncthreads();
  }
}

// Before pass `pass` (1, 2, ...; one block per cluster): the members' sums
// become the centre (an emptied cluster keeps its centre); alpha_a, beta_a in
// the order the definition states (the quotients and squares in parallel, the
// sum by one thread -- with the filter one of k_km_assign_tc); the centre's digits and h's constant.  The passes are
// over when one after the first changed nothing.  commit_only: the last call.
__global__ void __launch_bounds__(256) k_km_centres(int32_t k, int32_t pass, int32_t commit_only, KmState W,
                                                    int32_t *__restrict__ iters) {
  __shared__ double sq[kKmMaxK];
  __shared__ double red[8];
  const int a = blockIdx.x, tid = threadIdx.x;
  // every block reads the same words (block 0 alone writes stop, to the same verdict)
  if (__ldcg(W.stop)) return;
  const int prev = (pass - 1) & 1;
  const bool over = pass > 2 && __ldcg(W.moved + prev) == 0u;
  if (over) {
    if (a == 0 && tid == 0) *W.stop = 1;
    return;
  }
  if (a == 0 && tid == 0 && !commit_only) {
    *iters = pass;
    W.moved[pass & 1] = 0u;
    W.open[pass & 1] = 0u;
    W.wide[pass & 1] = 0u;
  }
  const unsigned mc = W.mcnt[a];
  const unsigned ca = mc ? mc : W.cnt[a];
  const double c = (double)ca;
  const KmFilter F = *W.filt;
  const int pad = kt_pad(k);
  double acc = 0.0;
  for (int b = tid; b < k; b += blockDim.x) {
    const unsigned s = mc ? W.M[(size_t)a * k + b] : W.S[(size_t)a * pad + b];
    W.S[(size_t)a * pad + b] = s;
    W.ST[(size_t)b * k + a] = s;
    const double q = __ddiv_rn((double)s, c);
    sq[b] = __dmul_rn(q, q);
    if (F.on) {
      W.sq[(size_t)a * k + b] = sq[b];
      const double v = q - (double)F.m;
      acc += v * v;
      const int Q = __double2int_rn(v * (double)F.up);
      const int half = 1 << (F.w - 1);
      const int q1 = (Q + half) >> F.w;  // Q = q1 2^w + q0, -half <= q0 < half
      const int q0 = Q - (q1 << F.w);
      *reinterpret_cast<__half *>(W.digits + kt_at(2 * pad, kt_row(k, a, 0), b)) = __int2half_rn(q1);
      *reinterpret_cast<__half *>(W.digits + kt_at(2 * pad, kt_row(k, a, 1), b)) = __int2half_rn(q0);
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((tid & 31) == 0) red[tid >> 5] = acc;
  __syncthreads();
  if (tid == 0) {
    W.cnt[a] = ca;
    W.beta[a] = __ddiv_rn(2.0, c);
    if (F.on) {
      double h = 0.0;
      for (int q = 0; q < 8; ++q) h += red[q];
      W.hbase[a] = (float)h;
    } else {
      double al = 0.0;
#pragma unroll 8
      for (int b = 0; b < k; ++b) al = __dadd_rn(al, sq[b]);
      W.alpha[a] = al;
    }
  }
}

// ------------------------------------------------------------ the filter
// shared-memory descriptor of an operand image (K-major, no swizzle): core
// matrices of adjacent row groups 128 bytes apart, of adjacent entry groups
// `kstride` bytes apart; version 1
__device__ __forceinline__ uint64_t kt_desc(uint32_t addr, uint32_t kstride) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(kstride >> 4) << 16) | ((uint64_t)(128u >> 4) << 32) |
         ((uint64_t)1 << 46);
}
// instruction descriptor: FP16 A and B (K-major), FP32 accumulator, M = 128, N
__device__ __forceinline__ uint32_t kt_idesc(int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24);
}

// two least values seen and the place of the least
struct KmTop {
  float b1 = kKtFar, b2 = kKtFar;
  int arg = 0;
  __device__ __forceinline__ void see(float h, int at) {
    const bool less = h < b1;
    b2 = fminf(b2, fmaxf(b1, h));
    b1 = fminf(b1, h);
    if (less) arg = at;
  }
};

// the accumulators of one group, `cols` clusters (a multiple of 16): high
// digits, and low digits `low` columns further.  Even and odd columns are kept apart so that two
// chains of minima run side by side.
__device__ __forceinline__ KmTop kt_scan(uint32_t tmem, int low, int cols, const float *hb, float s0, float s1) {
  KmTop even, odd;
#pragma unroll
  for (int g = 0; g < kKtMaxStrips; ++g) {
    if (16 * g < cols) {
      uint32_t h[16], l[16];
      tc_ld16(tmem + (unsigned)(16 * g), h);
      tc_ld16(tmem + (unsigned)(low + 16 * g), l);
      tc_ld_wait(h);
      tc_ld_wait(l);
      const float4 *h4 = reinterpret_cast<const float4 *>(hb + 16 * g);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float4 b = h4[e];
        auto at = [&](int q, float base) {
          return fmaf(__uint_as_float(l[4 * e + q]), s0, fmaf(__uint_as_float(h[4 * e + q]), s1, base));
        };
        even.see(at(0, b.x), 16 * g + 4 * e);
        odd.see(at(1, b.y), 16 * g + 4 * e + 1);
        even.see(at(2, b.z), 16 * g + 4 * e + 2);
        odd.see(at(3, b.w), 16 * g + 4 * e + 3);
      }
    }
  }
  even.b2 = fminf(fminf(even.b2, odd.b2), fmaxf(even.b1, odd.b1));
  if (odd.b1 < even.b1) {
    even.b1 = odd.b1;
    even.arg = odd.arg;
  }
  return even;
}

// Warps 0-15: four per group of clusters, warp w on the TMEM lanes (nodes)
// 32 (w mod 4) .. + 31; the last group also gives the nodes' verdicts.  Warp 16,
// one thread: MMAs; warp 17, one thread: copies; warp 18: the sums alpha of the
// definition (a chain of k FP64 additions per cluster that only k_km_resolve
// reads).  One CTA per SM.  A node image is copied and released in kKtParts
// parts, so the next tile's entries arrive while the second half is multiplied.
__global__ void __launch_bounds__(kKtThreads, 1) k_km_assign_tc(int32_t n, int32_t k, int32_t pass, KmState W,
                                                               int32_t *__restrict__ assign,
                                                               int32_t *__restrict__ status) {
  extern __shared__ __align__(128) unsigned char kt_smem[];
  __shared__ __align__(16) float s_hb[kKtMaxK];
  __shared__ float2 s_two[kKtGroups - 1][kKtTile];  // the other groups' two least values
  __shared__ unsigned char s_arg[kKtGroups - 1][kKtTile];
  enum {
    kDigits,
    kFull,
    kNodes = kFull + kKtHalves,
    kFree = kNodes + kKtParts,
    kEmpty = kFree + kKtParts,
    kTaken = kEmpty + kKtHalves,
    kSlot,
    kBars
  };
  __shared__ __align__(8) uint64_t s_bar[kBars];
  __shared__ uint32_t s_tmem;
  if (__ldcg(W.stop)) return;
  const KmFilter F = *W.filt;
  const int tiles = (int)(((int64_t)n + kKtTile - 1) / kKtTile);
  if (!F.on || (int)blockIdx.x >= tiles) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int pad = kt_pad(k), steps = pad / 16;
  const uint32_t dbytes = kt_digit_bytes(k), ybytes = kt_tile_bytes(k);
  const uint32_t sB = tc_smem(kt_smem), sY = sB + dbytes;
  auto bar = [&](int q) { return tc_smem(&s_bar[q]); };
  for (int t = tid; t < pad; t += blockDim.x) s_hb[t] = t < k ? W.hbase[t] : kKtFar;
  if (warp == 16) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(tc_smem(&s_tmem)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int q = 0; q < kBars; ++q)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar(q)),
                   "r"(q < kEmpty ? 1u : q < kTaken ? 4u * (kKtGroups / kKtHalves) : q < kSlot ? 4u : 4u * (kKtGroups - 1)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = s_tmem;
  bool ok = true;

  if (warp == 18) {
    for (int a = (int)blockIdx.x + (int)gridDim.x * lane; a < k; a += 32 * (int)gridDim.x) {
      const double *sq = W.sq + (size_t)a * k;
      double al = 0.0;
#pragma unroll 8
      for (int b = 0; b < k; ++b) al = __dadd_rn(al, sq[b]);
      W.alpha[a] = al;
    }
  } else if (warp == 17) {
    if (lane == 0) {
      tc_bulk_load(sB, W.digits, dbytes, bar(kDigits));
      int it = 0;
      for (int64_t tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x, ++it) {
        const unsigned char *img = W.image + tile * ybytes;
        for (int q = 0; q < kKtParts; ++q) {
          const int a = steps * q / kKtParts, b = steps * (q + 1) / kKtParts;
          if (a == b) continue;
          // the part is free when the previous tile's MMAs on it are done
          if (it > 0 && !(ok = tc_wait(bar(kFree + q), (unsigned)(it - 1) & 1u))) break;
          tc_bulk_load(sY + (unsigned)a * kKtStepBytes, img + (unsigned)a * kKtStepBytes,
                       (unsigned)(b - a) * kKtStepBytes, bar(kNodes + q));
        }
        if (tile + gridDim.x < tiles) tc_bulk_prefetch(img + (size_t)gridDim.x * ybytes, ybytes);
      }
      // whatever happened above, no copy is in flight when the CTA ends (the
      // last copy into each part; bounded waits)
      const int last = ok ? it - 1 : it - 2;
      tc_wait(bar(kDigits), 0u);
      if (last >= 0)
        for (int q = 0; q < kKtParts; ++q)
          if (steps * q / kKtParts != steps * (q + 1) / kKtParts) tc_wait(bar(kNodes + q), (unsigned)last & 1u);
    }
  } else if (warp == 16) {
    // the whole warp runs this loop, so that the descriptors stay in uniform
    // registers
    int it = 0;
    bool issued = false;
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    for (int64_t tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x, ++it) {
      if (it == 0 && !(ok = tc_wait_warp(bar(kDigits), 0u))) break;
#pragma unroll 1
      for (int g = 0; g < kKtHalves && ok; ++g) {
        // the half's accumulators have been read
        if (it > 0 && !(ok = tc_wait_warp(bar(kEmpty + g), (unsigned)(it - 1) & 1u))) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const int lo = kt_half(k, g), N = 2 * (kt_half(k, g + 1) - lo);
        const uint32_t acc = tm + kKtCols * (unsigned)g, idesc = kt_idesc(N);
        uint64_t da = kt_desc(sY, kKtTile * 16u);
        uint64_t db = kt_desc(sB + (unsigned)lo * 32u, (unsigned)pad * 32u);  // 2 lo rows on, 16 bytes a row
        const uint64_t db_step = (unsigned)pad * 64u >> 4;
        uint32_t add = 0u;
        for (int q = 0; q < kKtParts; ++q) {
          const int s_lo = steps * q / kKtParts, s_hi = steps * (q + 1) / kKtParts;
          if (s_lo == s_hi) continue;
          if (g == 0 && !(ok = tc_wait_warp(bar(kNodes + q), (unsigned)it & 1u))) break;
          issued = true;
          if (N > 0)
            for (int st = s_lo; st < s_hi; ++st) {
              tc_mma_f16_warp(acc, da, db, idesc, add);
              da += kKtStepBytes >> 4;
              db += db_step;
              add = 1u;
            }
          if (g == kKtHalves - 1) tc_commit_warp(bar(kFree + q));
        }
        if (ok) tc_commit_warp(bar(kFull + g));
      }
    }
    // nothing is in flight when the CTA ends: the last commit covers every MMA before it
    if (ok) {
      ok = tc_wait_warp(bar(kFull + kKtHalves - 1), (unsigned)(it - 1) & 1u);
    } else if (issued) {
      tc_commit_warp(bar(kDigits));  // completes phase 1 of a barrier used once
      tc_wait(bar(kDigits), 1u);
    }
  } else {
    const int grp = warp >> 2, half = grp / (kKtGroups / kKtHalves);
    const bool last = grp == kKtGroups - 1;
    const int row = 32 * (warp & 3) + lane;
    const int c_lo = kt_split(k, grp), cols = kt_split(k, grp + 1) - c_lo;
    const int h_lo = kt_half(k, half), h_cols = kt_half(k, half + 1) - h_lo;
    const uint32_t lanes =
        tmem + ((uint32_t)(32 * (warp & 3)) << 16) + kKtCols * (unsigned)half + (unsigned)(c_lo - h_lo);
    const unsigned below = (1u << lane) - 1u;
    // the lists' places of the previous tile's nodes are on their way while
    // this tile's accumulators are read
    unsigned mm = 0, mf = 0, mw = 0, pm = 0, pf = 0, pw = 0;
    int4 em = make_int4(0, 0, 0, 0);
    int2 eu = make_int2(0, 0);
    auto append = [&]() {
      const unsigned qm = __shfl_sync(0xffffffffu, pm, 0);
      if (mm >> lane & 1u) W.list[qm + __popc(mm & below)] = em;
      if (mf | mw) {
        const unsigned qf = __shfl_sync(0xffffffffu, pf, 0), qw = __shfl_sync(0xffffffffu, pw, 0);
        if (mf >> lane & 1u) W.unsure[qf + __popc(mf & below)] = eu;
        if (mw >> lane & 1u) W.unsure[(unsigned)n - 1u - (qw + __popc(mw & below))] = eu;
      }
      mm = mf = mw = 0u;
    };
    int it = 0;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++it) {
      const int64_t i = tile * kKtTile + row;
      const bool live = i < n;
      const float tau = last && live ? W.tau[i] : 0.0f;
      const int old = last && live ? assign[i] : 0;
      if (!(ok = tc_wait_warp(bar(kFull + half), (unsigned)it & 1u))) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
      const KmTop own = kt_scan(lanes, h_cols, cols, s_hb + c_lo, F.s0, F.s1);
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0) tc_arrive(bar(kEmpty + half));
      if (!last) {
        // the slots of the previous tile have been taken
        if (it > 0 && !(ok = tc_wait_warp(bar(kTaken), (unsigned)(it - 1) & 1u))) break;
        s_two[grp][row] = make_float2(own.b1, own.b2);
        s_arg[grp][row] = (unsigned char)(c_lo + own.arg);
        __syncwarp();
        if (lane == 0) tc_arrive(bar(kSlot));
        continue;
      }
      append();
      if (!(ok = tc_wait_warp(bar(kSlot), (unsigned)it & 1u))) break;
      float2 two[kKtGroups];
      int at[kKtGroups];
#pragma unroll
      for (int g = 0; g < kKtGroups - 1; ++g) {
        two[g] = s_two[g][row];
        at[g] = s_arg[g][row];
      }
      two[kKtGroups - 1] = make_float2(own.b1, own.b2);
      at[kKtGroups - 1] = c_lo + own.arg;
      __syncwarp();
      if (lane == 0) tc_arrive(bar(kTaken));
      float b1 = two[0].x, b2 = two[0].y;
      int a = at[0];
#pragma unroll
      for (int g = 1; g < kKtGroups; ++g) {
        b2 = fminf(fminf(b2, two[g].y), fmaxf(b1, two[g].x));
        if (two[g].x < b1) {
          b1 = two[g].x;
          a = at[g];
        }
      }
      const bool sure = live && b2 - b1 > tau, moved = sure && old != a;
      if (moved) assign[i] = a;
      // who can be the least: the groups' least within tau, or any cluster when
      // a group's second is (written so that anything unordered counts as near)
      unsigned cand = 0u;
      bool all = false;
#pragma unroll
      for (int g = 0; g < kKtGroups; ++g) {
        cand |= (two[g].x - b1 > tau ? 255u : (unsigned)at[g]) << (8 * g);
        all |= !(two[g].y - b1 > tau);
      }
      em = make_int4((int)i, old, a, 0);
      eu = make_int2((int)i, (int)cand);
      mm = __ballot_sync(0xffffffffu, moved);
      mf = __ballot_sync(0xffffffffu, live && !sure && !all);
      mw = __ballot_sync(0xffffffffu, live && !sure && all);
      if (lane == 0) {
        if (mm) pm = atomicAdd(W.moved + (pass & 1), (unsigned)__popc(mm));
        if (mf) pf = atomicAdd(W.open + (pass & 1), (unsigned)__popc(mf));
        if (mw) pw = atomicAdd(W.wide + (pass & 1), (unsigned)__popc(mw));
      }
    }
    if (last) append();
  }
  if (!ok) dev_fail(status, SSM_E_TIMEOUT);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 16) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// Too many nodes are left with all clusters: k_km_assign takes the whole pass, at
// 8 ns a node (k = 200), where k_km_resolve takes 36 for such a node.  (A star:
// all leaves are equally far from all centres; 2^18 leaves, two passes: 11.0 -> 3.0 ms.)
__device__ __forceinline__ bool km_mostly_wide(const KmState &W, int32_t n, int32_t pass) {
  return __ldcg(W.wide + (pass & 1)) > (unsigned)n / 6u;
}

// one assignment pass without the filter, 64 nodes at a time: the distances of
// the tile and the sums of 64 clusters are staged 64 pivots at a time
__global__ void __launch_bounds__(kKmThreads) k_km_assign(int32_t n, int32_t k, int32_t pass,
                                                         const uint16_t *__restrict__ dip, KmState W,
                                                         int32_t *__restrict__ assign) {
  __shared__ __align__(16) unsigned Y[kKmChunk][kKmNodes];     // d of the tile's nodes, pivots b0 .. b0+63
  __shared__ __align__(16) unsigned Sc[kKmChunk][kKmClusters];  // S_ab of 64 clusters, same pivots
  __shared__ double bg[16][kKmNodes];                          // per cluster group: best g of each node
  __shared__ int ba[16][kKmNodes];                             // and its cluster
  __shared__ double s_best[kKmNodes];
  __shared__ int s_arg[kKmNodes];
  {
    const bool wide = km_mostly_wide(W, n, pass);  // the three loads together
    const int stop = __ldcg(W.stop), on = W.filt->on;
    if (stop || (on && !wide)) return;
  }
  const int tid = threadIdx.x;
  const int tn = tid & 15, ta = tid >> 4;  // node group (4 nodes), cluster group (4 clusters)
  for (int n0 = blockIdx.x * kKmNodes; n0 < n; n0 += gridDim.x * kKmNodes) {
    if (tid < kKmNodes) {
      s_best[tid] = 0.0;
      s_arg[tid] = -1;
    }
    for (int c0 = 0; c0 < k; c0 += kKmClusters) {
      unsigned long long acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
      for (int b0 = 0; b0 < k; b0 += kKmChunk) {
        __syncthreads();  // the previous chunk is consumed
        for (int t = tid; t < kKmChunk * kKmNodes; t += kKmThreads) {
          const int b = t / kKmNodes, v = t - b * kKmNodes;
          Y[b][v] = (b0 + b < k && n0 + v < n) ? (unsigned)__ldg(dip + (size_t)(b0 + b) * n + n0 + v) : 0u;
        }
        for (int t = tid; t < kKmChunk * kKmClusters; t += kKmThreads) {
          const int b = t / kKmClusters, q = t - b * kKmClusters;
          Sc[b][q] = (b0 + b < k && c0 + q < k) ? W.ST[(size_t)(b0 + b) * k + c0 + q] : 0u;
        }
        __syncthreads();
        const int nb = min(kKmChunk, k - b0);
#pragma unroll 4
        for (int b = 0; b < nb; ++b) {
          const uint4 y = reinterpret_cast<const uint4 *>(Y[b])[tn];
          const uint4 sv4 = reinterpret_cast<const uint4 *>(Sc[b])[ta];
          const unsigned yv[4] = {y.x, y.y, y.z, y.w}, sv[4] = {sv4.x, sv4.y, sv4.z, sv4.w};
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] += (unsigned long long)yv[i] * sv[j];
        }
      }
      // per node, the best of this thread's 4 clusters (ascending a, strict <)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        double best = 0.0;
        int arg = -1;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int a = c0 + 4 * ta + j;
          if (a < k) {
            const double g = __dsub_rn(W.alpha[a], __dmul_rn(W.beta[a], (double)acc[i][j]));
            if (arg < 0 || g < best) {
              best = g;
              arg = a;
            }
          }
        }
        bg[ta][4 * tn + i] = best;
        ba[ta][4 * tn + i] = arg;
      }
      __syncthreads();
      // cluster groups in ascending a after the running best (strict <)
      if (tid < kKmNodes) {
        double best = s_best[tid];
        int arg = s_arg[tid];
        for (int q = 0; q < 16; ++q) {
          const int a = ba[q][tid];
          if (a < 0) continue;
          const double g = bg[q][tid];
          if (arg < 0 || g < best) {
            best = g;
            arg = a;
          }
        }
        s_best[tid] = best;
        s_arg[tid] = arg;
      }
    }
    __syncthreads();
    if (tid < kKmNodes) {  // warps 0 and 1, whole
      const int i = n0 + tid;
      const int a = s_arg[tid], old = i < n ? assign[i] : a;
      if (old != a) assign[i] = a;
      const unsigned mm = __ballot_sync(0xffffffffu, old != a);
      unsigned pm = 0;
      if ((tid & 31) == 0 && mm) pm = atomicAdd(W.moved + (pass & 1), (unsigned)__popc(mm));
      pm = __shfl_sync(0xffffffffu, pm, 0);
      if (old != a) W.list[pm + __popc(mm & ((1u << (tid & 31)) - 1u))] = make_int4(i, old, a, 0);
    }
  }
}

// ------------------------------------------------------------ after a pass
// words of the k x k members' sums, up to a 16-byte boundary
__host__ __device__ inline unsigned km_sum_words(int k) { return ((unsigned)k * (unsigned)k + 3u) & ~3u; }

// distance of pivot b to node i, from the filter's image (a node's entries lie
// 16 bytes at a time) or from the table
__device__ __forceinline__ unsigned km_dist(const KmState &W, const KmFilter &F, const uint16_t *__restrict__ dip,
                                            int32_t n, int32_t k, int b, int i) {
  if (!F.on) return __ldg(dip + (size_t)b * n + i);
  const unsigned char *img = W.image + (size_t)(i / kKtTile) * kt_tile_bytes(k);
  const int v = __half2int_rn(*reinterpret_cast<const __half *>(img + kt_at(kKtTile, i & (kKtTile - 1), b)));
  return (unsigned)(v + F.m);
}

// The nodes the filter left open, decided by the definition: t in 64-bit
// integers, g in FP64, ties to the lowest cluster; lanes over pivots, clusters
// one after another.  A node with up to four candidates is a warp's work, one
// with all clusters a block's.  Those that changed cluster join the list.
__global__ void __launch_bounds__(256, 3) k_km_resolve(int32_t n, int32_t k, int32_t pass,
                                                    const uint16_t *__restrict__ dip, KmState W,
                                                    int32_t *__restrict__ assign) {
  __shared__ double s_best[8];
  __shared__ int s_at[8];
  const KmFilter F = *W.filt;
  const unsigned nopen = __ldcg(W.open + (pass & 1)), nwide = __ldcg(W.wide + (pass & 1));
  if (__ldcg(W.stop) || !F.on || km_mostly_wide(W, n, pass)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kRegs = (kKtMaxK + 31) / 32;
  unsigned y[kRegs];
  auto load = [&](int i) {
#pragma unroll
    for (int q = 0; q < kRegs; ++q) y[q] = lane + 32 * q < k ? km_dist(W, F, dip, n, k, lane + 32 * q, i) : 0u;
  };
  double best = 0.0;
  int arg = 0x7fffffff;
  auto better = [&](double g, int a) {
    if (a != 0x7fffffff && (arg == 0x7fffffff || g < best || (g == best && a < arg))) {
      best = g;
      arg = a;
    }
  };
  // kTake clusters (negative: none) side by side, so that their sums' loads
  // are in flight together; lane slot + c keeps cluster c's t, so that a warp
  // forms its g's in one go (an FP64 instruction costs the same for one lane as
  // for 32; every lane forming every g, a node took 15 us, one cluster after
  // another 40 us)
  constexpr int kTake = 5;
  unsigned long long mine = 0ull;
  int at = -1;
  auto take = [&](const int (&a)[kTake], int slot) {
    unsigned long long acc[kTake];
#pragma unroll
    for (int c = 0; c < kTake; ++c) {
      acc[c] = 0ull;
#pragma unroll
      for (int q = 0; q < kRegs; ++q)
        if (lane + 32 * q < k)
          acc[c] += (unsigned long long)y[q] * __ldg(W.S + (size_t)max(a[c], 0) * kt_pad(k) + lane + 32 * q);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int c = 0; c < kTake; ++c) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
#pragma unroll
    for (int c = 0; c < kTake; ++c)
      if (lane == slot + c) {
        mine = acc[c];
        at = a[c];
      }
  };
  auto choose = [&]() {
    arg = 0x7fffffff;
    if (at >= 0) better(__dsub_rn(__ldg(W.alpha + at), __dmul_rn(__ldg(W.beta + at), (double)mine)), at);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double g = __shfl_xor_sync(0xffffffffu, best, o);
      const int a = __shfl_xor_sync(0xffffffffu, arg, o);
      better(g, a);
    }
    at = -1;
  };
  auto settle = [&](int i) {  // one thread
    const int old = assign[i];
    if (old != arg) {
      assign[i] = arg;
      W.list[atomicAdd(W.moved + (pass & 1), 1u)] = make_int4(i, old, arg, 0);
    }
  };
  for (unsigned t = blockIdx.x * 8u + (unsigned)warp; t < nopen; t += gridDim.x * 8u) {
    const int2 e = W.unsure[t];
    load(e.x);
    int a[kTake];
#pragma unroll
    for (int c = 0; c < kTake; ++c) {
      a[c] = c < kKtGroups ? (int)((unsigned)e.y >> (8 * c) & 255u) : 255;
      if (a[c] >= k) a[c] = -1;
    }
    take(a, 0);
    choose();
    if (lane == 0) settle(e.x);
  }
  // blocks from the other end, so that few nodes of either kind meet in one block
  for (unsigned t = gridDim.x - 1u - blockIdx.x; t < nwide; t += gridDim.x) {
    const int2 e = W.unsure[(unsigned)n - 1u - t];
    load(e.x);
    int slot = 0;
    static_assert((kKtMaxK + 7) / 8 <= 32, "a warp's clusters fit its lanes");
    for (int a0 = warp; a0 < k; a0 += 8 * kTake, slot += kTake) {
      int a[kTake];
#pragma unroll
      for (int c = 0; c < kTake; ++c) a[c] = a0 + 8 * c < k ? a0 + 8 * c : -1;
      take(a, slot);
    }
    choose();
    if (lane == 0) {
      s_best[warp] = best;
      s_at[warp] = arg;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w) better(s_best[w], s_at[w]);
      settle(e.x);
    }
    __syncthreads();
  }
}

// The members' sums after the moves of the listed nodes: a warp per node,
// atomics on the k x k sums in L2 (2.8 ns a node when many run at once)
__device__ __forceinline__ void km_move_direct(int32_t n, int32_t k, const uint16_t *__restrict__ dip, const KmState &W,
                                               const KmFilter &F, unsigned count) {
  const int lane = threadIdx.x & 31;
  const unsigned per = blockDim.x >> 5, w0 = blockIdx.x * per + (threadIdx.x >> 5), ws = gridDim.x * per;
  for (unsigned t = w0; t < count; t += ws) {
    const int4 e = W.list[t];
#pragma unroll 4
    for (int b = lane; b < k; b += 32) {
      const unsigned y = km_dist(W, F, dip, n, k, b, e.x);
      atomicAdd(W.M + (size_t)e.z * k + b, y);
      if (e.y >= 0) atomicAdd(W.M + (size_t)e.y * k + b, 0u - y);
    }
    if (lane == 0) {
      atomicAdd(W.mcnt + e.z, 1u);
      if (e.y >= 0) atomicAdd(W.mcnt + e.y, 0u - 1u);
    }
  }
}

__global__ void __launch_bounds__(256) k_km_move(int32_t n, int32_t k, int32_t pass, const uint16_t *__restrict__ dip,
                                                 KmState W) {
  if (__ldcg(W.stop)) return;
  km_move_direct(n, k, dip, W, *W.filt, __ldcg(W.moved + (pass & 1)));
}

// The same with the k x k sums of a CTA in shared memory, added to the global
// sums by one bulk reduction at the end (k <= kKtMaxK, nodes in the filter's
// image).  Fewer than kKmMoveFew nodes are moved directly: clearing and adding
// 160 KB per CTA takes some 25 us.
constexpr int kKmMoveThreads = 1024;
constexpr unsigned kKmMoveFew = 8192, kKmMoveNodes = 256;  // ... and the least nodes per CTA

__global__ void __launch_bounds__(kKmMoveThreads, 1) k_km_move_smem(int32_t n, int32_t k, int32_t pass,
                                                                    const uint16_t *__restrict__ dip, KmState W) {
  extern __shared__ __align__(128) unsigned km_sums[];
  if (__ldcg(W.stop)) return;
  const unsigned count = __ldcg(W.moved + (pass & 1));
  const KmFilter F = *W.filt;
  if (!F.on || count < kKmMoveFew) {
    km_move_direct(n, k, dip, W, F, count);
    return;
  }
  const unsigned ctas = min(gridDim.x, (count + kKmMoveNodes - 1u) / kKmMoveNodes);
  if (blockIdx.x >= ctas) return;
  const unsigned words = km_sum_words(k);
  unsigned *const scnt = km_sums + words;
  for (unsigned t = threadIdx.x; t < words + (unsigned)k; t += blockDim.x) km_sums[t] = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned w0 = blockIdx.x * (kKmMoveThreads / 32u) + (threadIdx.x >> 5), ws = ctas * (kKmMoveThreads / 32u);
  constexpr int kRegs = (kKtMaxK + 31) / 32;
  // two nodes ahead: the list entry; one ahead: its distances
  const int4 none = make_int4(0, 0, 0, 0);
  int4 e = w0 < count ? W.list[w0] : none, e1 = w0 + ws < count ? W.list[w0 + ws] : none;
  unsigned y[kRegs];
  auto load = [&](int i, unsigned (&v)[kRegs]) {
#pragma unroll
    for (int q = 0; q < kRegs; ++q) v[q] = lane + 32 * q < k ? km_dist(W, F, dip, n, k, lane + 32 * q, i) : 0u;
  };
  if (w0 < count) load(e.x, y);
  for (unsigned t = w0; t < count; t += ws) {
    const int4 cur = e;
    e = e1;
    unsigned y1[kRegs];
    load(e.x, y1);  // node 0 past the end
    e1 = t + 2 * ws < count ? W.list[t + 2 * ws] : none;
#pragma unroll
    for (int q = 0; q < kRegs; ++q)
      if (lane + 32 * q < k) {
        atomicAdd(km_sums + cur.z * k + lane + 32 * q, y[q]);
        if (cur.y >= 0) atomicAdd(km_sums + cur.y * k + lane + 32 * q, 0u - y[q]);
        y[q] = y1[q];
      }
    if (lane == 0) {
      atomicAdd(scnt + cur.z, 1u);
      if (cur.y >= 0) atomicAdd(scnt + cur.y, 0u - 1u);
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0) {
    tc_bulk_add_u32(W.M, tc_smem(km_sums), words * 4u);
    tc_bulk_store_wait();
  }
  for (int a = threadIdx.x; a < k; a += blockDim.x)
    if (scnt[a]) atomicAdd(W.mcnt + a, scnt[a]);
}

// new pivots, step 1: v_i = n_a ||y_i||^2 - 2 t_ia for the node's cluster a
// (a warp per node, eight entries per lane and step), and the least v per
// cluster (per block first)
__global__ void __launch_bounds__(256) k_km_pick_value(int32_t n, int32_t k, const uint16_t *__restrict__ dip,
                                                       const int32_t *__restrict__ assign, KmState W) {
  __shared__ long long least[kKmMaxK];
  const KmFilter F = *W.filt;
  for (int a = threadIdx.x; a < k; a += blockDim.x) least[a] = 0x7FFFFFFFFFFFFFFFll;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t w0 = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5), ws = (int64_t)gridDim.x * 8;
  for (int64_t i = w0; i < n; i += ws) {
    const int a = assign[i];
    if (a < 0) continue;
    const unsigned *Sa = W.S + (size_t)a * kt_pad(k);
    unsigned long long yy = 0ull, t = 0ull;
    for (int b = 8 * lane; b < k; b += 256) {
      const uint4 u0 = __ldg(reinterpret_cast<const uint4 *>(Sa + b)), u1 = __ldg(reinterpret_cast<const uint4 *>(Sa + b) + 1);
      const unsigned su[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
      unsigned y[8];
      if (F.on) {  // the image's entries past k meet zero sums
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(W.image + (size_t)(i / kKtTile) * kt_tile_bytes(k) +
                                                              kt_at(kKtTile, (int)(i & (kKtTile - 1)), b)));
        const unsigned vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const __half2 h = *reinterpret_cast<const __half2 *>(&vv[q]);
          y[2 * q] = (unsigned)(__half2int_rn(__low2half(h)) + F.m);
          y[2 * q + 1] = (unsigned)(__half2int_rn(__high2half(h)) + F.m);
        }
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) y[q] = b + q < k ? (unsigned)__ldg(dip + (size_t)(b + q) * n + i) : 0u;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (b + q < k) {
          yy += (unsigned long long)y[q] * y[q];
          t += (unsigned long long)y[q] * su[q];
        }
    }
    long long v = (long long)((unsigned long long)W.cnt[a] * yy) - 2ll * (long long)t;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) {
      W.vnode[i] = v;
      if (v < least[a]) atomicMin(least + a, v);
    }
  }
  __syncthreads();
  for (int a = threadIdx.x; a < k; a += blockDim.x)
    if (least[a] != 0x7FFFFFFFFFFFFFFFll) atomicMin(W.vbest + a, least[a]);
}

// step 2: the lowest node id attaining the least v
__global__ void k_km_pick_node(int32_t n, const int32_t *__restrict__ assign, KmState W) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int a = assign[i];
    if (a >= 0 && W.vnode[i] == W.vbest[a]) atomicMin(W.pbest + a, (int)i);
  }
}

__global__ void k_km_pick_out(int32_t k, const int32_t *__restrict__ piv_in, const KmState W,
                              int32_t *__restrict__ piv_out) {
  for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < k; a += gridDim.x * blockDim.x) {
    const int p = W.pbest[a];
    piv_out[a] = p != 0x7FFFFFFF ? p : __ldg(piv_in + a);
  }
}

__global__ void k_km_fill(int32_t k, KmState W) {
  for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < k; a += gridDim.x * blockDim.x) {
    W.vbest[a] = 0x7FFFFFFFFFFFFFFFll;
    W.pbest[a] = 0x7FFFFFFF;
  }
}

// tc: with the filter's arrays, which hold a copy of the whole table
static size_t carve_kmeans(Carver &c, KmState &W, int32_t **assign_ws, int32_t n, int32_t k, bool tc) {
  W.S = c.take<unsigned>((size_t)k * kt_pad(k));
  W.ST = c.take<unsigned>((size_t)k * k);
  W.M = c.take<unsigned>(km_sum_words(k));
  W.cnt = c.take<unsigned>((size_t)k);
  W.mcnt = c.take<unsigned>((size_t)k);
  W.alpha = c.take<double>((size_t)k);
  W.beta = c.take<double>((size_t)k);
  W.sq = tc ? c.take<double>((size_t)k * k) : nullptr;
  W.stop = c.take<int32_t>(1);
  W.dmax = c.take<unsigned>(1);
  W.filt = c.take<KmFilter>(1);
  W.moved = c.take<unsigned>(2);
  W.open = c.take<unsigned>(2);
  W.wide = c.take<unsigned>(2);
  W.list = c.take<int4>((size_t)n);
  W.vnode = reinterpret_cast<long long *>(W.list);  // the moves are over when the pivots are chosen
  W.unsure = tc ? c.take<int2>((size_t)n) : nullptr;
  W.tau = tc ? c.take<float>((size_t)n) : nullptr;
  W.hbase = tc ? c.take<float>((size_t)kt_pad(k)) : nullptr;
  W.digits = tc ? c.take<unsigned char>((size_t)kt_digit_bytes(k)) : nullptr;
  W.image = tc ? c.take<unsigned char>(((size_t)n + kKtTile - 1) / kKtTile * kt_tile_bytes(k)) : nullptr;
  W.vbest = c.take<long long>((size_t)k);
  W.pbest = c.take<int32_t>((size_t)k);
  *assign_ws = c.take<int32_t>((size_t)n);
  return c.size();
}

}  // namespace ssm

SSM_API size_t ssm_kmeans_pivots_workspace(int32_t n, int32_t k) {
  if (n < 1 || k < 1) return 0;
  ssm::Carver c(nullptr, 0);
  ssm::KmState W;
  int32_t *a;
  return ssm::carve_kmeans(c, W, &a, n, k, k <= ssm::kKtMaxK);
}

SSM_API size_t ssm_kmeans_pivots_workspace_least(int32_t n, int32_t k) {
  if (n < 1 || k < 1) return 0;
  ssm::Carver c(nullptr, 0);
  ssm::KmState W;
  int32_t *a;
  return ssm::carve_kmeans(c, W, &a, n, k, false);
}

SSM_API int ssm_kmeans_pivots(int32_t n, int32_t k, const uint16_t *dip, const int32_t *pivots_in, int32_t max_iter,
                              int32_t *pivots_out, int32_t *assign, int32_t *iters, int32_t *status, void *ws,
                              size_t ws_bytes, cudaStream_t s) {
  using namespace ssm;
  if (n < 1 || !dip || !pivots_in || !pivots_out || !iters || !status || !ws)
    return fail(SSM_E_ARG, "ssm_kmeans_pivots: null pointer or bad size");
  if (k < 1 || k > kKmMaxK || k > n) return fail(SSM_E_ARG, "ssm_kmeans_pivots: need 1 <= k <= min(n, %d)", kKmMaxK);
  if (max_iter < 1) return fail(SSM_E_ARG, "ssm_kmeans_pivots: max_iter must be >= 1");
  // without room for the filter every pass takes the integer products, with the
  // same results
  const bool tc = k <= kKtMaxK && ws_bytes >= ssm_kmeans_pivots_workspace(n, k);
  Carver c(ws, ws_bytes);
  KmState W;
  int32_t *asg_ws = nullptr;
  carve_kmeans(c, W, &asg_ws, n, k, tc);
  if (!c.ok) return fail(SSM_E_NOMEM, "ssm_kmeans_pivots: workspace %zu bytes, need %zu", ws_bytes, c.size());
  int32_t *asg = assign ? assign : asg_ws;
  const int sms = num_sms();
  SSM_TRY_CUDA(cudaMemsetAsync(W.dmax, 0, sizeof(unsigned), s));
  SSM_TRY_CUDA(cudaMemsetAsync(W.stop, 0, sizeof(int32_t), s));
  SSM_TRY_CUDA(cudaMemsetAsync(iters, 0, sizeof(int32_t), s));
  SSM_TRY_CUDA(cudaMemsetAsync(asg, 0xFF, (size_t)n * sizeof(int32_t), s));  // -1: no cluster yet
  const int64_t kn = (int64_t)k * n;
  note_launch(), k_km_dmax<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>((kn / 8 + 255) / 256, sms * 8)), 256, 0, s>>>(
      kn, dip, W.dmax);
  note_launch(), k_km_init<<<std::min(k, sms * 4), 256, 0, s>>>(n, k, tc ? 1 : 0, dip, pivots_in, W, status);
  const int kt_tiles = (int)(((int64_t)n + kKtTile - 1) / kKtTile);
  const int tiles = (int)(((int64_t)n + kKmNodes - 1) / kKmNodes);
  const size_t smem = tc ? (size_t)kt_digit_bytes(k) + kt_tile_bytes(k) : 0;
  if (tc) {
    SSM_TRY_CUDA(allow_dynamic_smem((const void *)k_km_assign_tc));
    SSM_TRY_CUDA(allow_dynamic_smem((const void *)k_km_move_smem));
    SSM_TRY_CUDA(cudaMemsetAsync(W.digits, 0, (size_t)kt_digit_bytes(k), s));  // rows and entries past k
    note_launch(), k_km_image<<<std::min(kt_tiles, sms * 32), 256, 0, s>>>(n, k, dip, W);
  }
  const int resolve_blocks = (int)std::min<int64_t>(((int64_t)n + 7) / 8, (int64_t)sms * 8);
  for (int pass = 1; pass <= max_iter; ++pass) {
    note_launch(), k_km_centres<<<k, 256, 0, s>>>(k, pass, 0, W, iters);
    if (tc) note_launch(), k_km_assign_tc<<<std::min(kt_tiles, sms), kKtThreads, smem, s>>>(n, k, pass, W, asg, status);
    note_launch(), k_km_assign<<<tc ? std::min(tiles, sms * 3) : tiles, kKmThreads, 0, s>>>(n, k, pass, dip, W, asg);
    if (tc) {
      note_launch(), k_km_resolve<<<std::min(resolve_blocks, sms * 3), 256, 0, s>>>(n, k, pass, dip, W, asg);
      note_launch(), k_km_move_smem<<<sms, kKmMoveThreads, ((size_t)km_sum_words(k) + (size_t)k) * sizeof(unsigned), s>>>(n, k, pass, dip, W);
    } else {
      note_launch(), k_km_move<<<resolve_blocks, 256, 0, s>>>(n, k, pass, dip, W);
    }
  }
  note_launch(), k_km_centres<<<k, 256, 0, s>>>(k, max_iter + 1, 1, W, iters);  // the last members' sums
  note_launch(), k_km_fill<<<(k + 255) / 256, 256, 0, s>>>(k, W);
  const int nb = (int)std::min<int64_t>(((int64_t)n + 255) / 256, (int64_t)sms * 8);
  note_launch(), k_km_pick_value<<<(int)std::min<int64_t>(((int64_t)n + 7) / 8, (int64_t)sms * 8), 256, 0, s>>>(
      n, k, dip, asg, W);
  note_launch(), k_km_pick_node<<<nb, 256, 0, s>>>(n, asg, W);
  note_launch(), k_km_pick_out<<<(k + 255) / 256, 256, 0, s>>>(k, pivots_in, W, pivots_out);
  SSM_TRY_CUDA(cudaGetLastError());
  return SSM_OK;
}
