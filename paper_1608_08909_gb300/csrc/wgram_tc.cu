// The centred Gram matrix of weighted PivotMDS on the tensor cores.
//
// G_ab = sum_i V_ia V_ib of integers |V| < 2^55 (wgram_tc.cuh), wanted to FP64
// accuracy.  V is cut into seven signed digits of eight bits, V = sum_p 256^(6-p)
// v_p with -128 <= v_p <= 128 (the bytes of V + 0x80808080808080, less 128 each),
// all exact in FP16, and
//   G = sum_s 256^(12-s) sum_{p+q=s} v_p^T v_q.
// Classes s = 0 .. 8 are formed (39 digit pairs): what is left off is below
// 2^-68 of the range's square per node, and below 2^-53 of a diagonal entry also
// where one of 65,536 nodes is far from the others, those equally far.  (With
// classes 0 .. 6, 1.7 ms, that table's eigenvalue was 2e-12 off, and with lengths
// over four decades 4e-15 where an FP64 product is at 4e-16.)  An FP32
// accumulator holds an exact integer: it is read out before 2^14 times its pairs
// and nodes passes 2^24, into 32-bit sums, and those go into 64-bit sums in
// global memory with integer atomics (order-free), four per entry.
//
// A CTA has one class and a range of nodes (as many CTAs per class as its work
// asks for).  Per unit of 32 nodes a warp loads two pivots' rows at a time (128
// consecutive bytes each), forms the fixed point, and writes the digits of the
// class as FP16 planes, one 16-byte core-matrix row per pivot and eight nodes
// (K-major, no swizzle; node groups 32 bytes further apart than the rows need,
// so that the four of a warp's store meet no bank twice).  The planes are
// double-buffered: the MMAs (M = 128 pivots, N = all of them; the second tile,
// the last 128 pivots, only against those from 128 on) run while the next unit
// is converted.  Both operands of every pair are planes of the same buffer.
// Bound by the conversion (7,400 to 10,000 cycles a unit and CTA at k = 200) and,
// for the classes of many pairs, the MMAs.  Measured (262K nodes, k = 200): 2.2 ms,
// against 16.2 in FP64.
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "tc.cuh"
#include "wgram_tc.cuh"

namespace ssm {

constexpr int kWgThreads = 512;
constexpr int kWgUnit = 32;     // nodes per unit (two MMAs of K = 16)
constexpr int kWgClasses = 9;   // s = 0 .. 8
constexpr int kWgRowPairs = 7;  // row pairs per warp (104 over 16 warps, rounded up)
constexpr int kWgSums = 120;    // read-outs per 32-bit sum: 120 2^24 < 2^31
constexpr unsigned long long kWgBias = 0x80808080808080ull;
constexpr unsigned kWgDigits = 7;

struct WgSplit {
  int32_t start[kWgClasses + 1];  // CTAs of the classes
};

__host__ __device__ inline int wg_pad(int k) { return (k + 15) / 16 * 16; }
__host__ __device__ inline int wg_rows(int k) { return wg_pad(k) > 128 ? wg_pad(k) : 128; }
__host__ __device__ inline unsigned wg_group(int k) { return (unsigned)wg_rows(k) * 16u + 32u; }  // bytes, eight nodes
__host__ __device__ inline unsigned wg_plane(int k) { return 4u * wg_group(k); }
__host__ __device__ inline unsigned wg_smem(int k) {
  return 2u * kWgDigits * wg_plane(k) + (unsigned)(wg_pad(k) > 128 ? wg_pad(k) - 128 : 0) * 128u * 4u + (unsigned)wg_rows(k) * 8u;
}

__device__ __forceinline__ uint64_t wg_desc(uint32_t addr, uint32_t kstride) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(kstride >> 4) << 16) | ((uint64_t)(128u >> 4) << 32) |
         ((uint64_t)1 << 46);
}
__device__ __forceinline__ uint32_t wg_idesc(int N) { return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24); }

// the FP16 pair of digit p of two biased values
__device__ __forceinline__ uint32_t wg_digit(unsigned long long a, unsigned long long b, int p) {
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
  uint32_t w;
  switch (p) {
    case 0: w = __byte_perm(ah, bh, 0x7632) | 0x64006400u; break;  // nine bits: 0 .. 256
    case 1: w = (__byte_perm(ah, bh, 0x0501) & 0x00FF00FFu) | 0x64006400u; break;
    case 2: w = (__byte_perm(ah, bh, 0x0400) & 0x00FF00FFu) | 0x64006400u; break;
    case 3: w = (__byte_perm(al, bl, 0x0703) & 0x00FF00FFu) | 0x64006400u; break;
    case 4: w = (__byte_perm(al, bl, 0x0602) & 0x00FF00FFu) | 0x64006400u; break;
    case 5: w = (__byte_perm(al, bl, 0x0501) & 0x00FF00FFu) | 0x64006400u; break;
    default: w = (__byte_perm(al, bl, 0x0400) & 0x00FF00FFu) | 0x64006400u; break;
  }
  const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&w), __half2half2(__ushort_as_half(0x6480)));  // 1024 + 128
  return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ void wg_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])
               :
               : "memory");
}

__global__ void __launch_bounds__(kWgThreads, 1) k_wgram_tc(int32_t n, int32_t k, const float *__restrict__ dist,
                                                           const unsigned *__restrict__ dmax,
                                                           const long long *__restrict__ centre, WgSplit split,
                                                           unsigned long long *__restrict__ acc,
                                                           int32_t *__restrict__ status) {
  extern __shared__ __align__(128) unsigned char wg_raw[];
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ uint32_t s_tmem;
  int cls = 0;
  while ((int)blockIdx.x >= split.start[cls + 1]) ++cls;
  const int64_t units = ((int64_t)n + kWgUnit - 1) / kWgUnit;
  const int64_t j = (int)blockIdx.x - split.start[cls], m = split.start[cls + 1] - split.start[cls];
  const int64_t u0 = units * j / m, u1 = units * (j + 1) / m;
  if (u0 >= u1) return;  // uniform: the whole CTA leaves before any TMEM use
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int pad = wg_pad(k), R = wg_rows(k), n1 = max(0, pad - 128);
  const uint32_t group = wg_group(k), plane = wg_plane(k);
  const int dlo = max(0, cls - ((int)kWgDigits - 1)), dhi = cls - dlo;  // digits p with a partner cls - p
  const int planes = dhi - dlo + 1;
  const int flush = 512 / kWgUnit * 2 / planes;                          // units per read-out: planes 2^14 nodes <= 2^24
  const uint32_t base = tc_smem(wg_raw);
  int *const sum1 = reinterpret_cast<int *>(wg_raw + 2u * kWgDigits * plane);        // [n1][128] second tile's sums, a thread's own
  unsigned long long *const shift = reinterpret_cast<unsigned long long *>(sum1 + n1 * 128);  // [R] bias - centre
  const int f = wfix_f(*dmax);
  for (int t = tid; t < n1 * 128; t += kWgThreads) sum1[t] = 0;
  for (int r = tid; r < R; r += kWgThreads) shift[r] = kWgBias - (r < k ? (unsigned long long)__ldg(centre + r) : 0ull);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(tc_smem(&s_tmem)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int q = 0; q < 2; ++q) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&s_bar[q])));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);

  // this warp's row pairs 2 (warp + 16 i), + 1; a lane loads node `lane` of both
  float d[2 * kWgRowPairs];
  auto load = [&](int64_t u, int q) {
    const int64_t i = u * kWgUnit + lane;
    const int r = 2 * (warp + 16 * (q >> 1)) + (q & 1);
    return r < k && i < n && u < u1 ? __ldg(dist + (size_t)r * n + i) : 0.f;
  };
  int sum0[7][8];
#pragma unroll
  for (int t = 0; t < 7; ++t)
#pragma unroll
    for (int e = 0; e < 8; ++e) sum0[t][e] = 0;
  const int q4 = warp & 3, cg = warp >> 2;  // TMEM lanes 32 q4 .. + 31; strips of eight columns cg, cg + 4, ...
  const int row = 32 * q4 + lane;
  const uint32_t tlane = tmem + ((uint32_t)(32 * q4) << 16);
  // 64-bit sums: classes 0-2 in units of 256^10, 3-4 of 256^8, 5-6 of 256^6, 7-8 of 256^4
  const int part = cls < 3 ? 0 : (cls - 1) / 2;
  const int up = 8 * (2 + 2 * part - cls);
  auto emit = [&]() {
    unsigned long long *out = acc + (size_t)part * k * k;
    auto add = [&](int a, int b, int v) {
      if (a < k && b < k && a <= b && v != 0) atomicAdd(out + (size_t)a * k + b, (unsigned long long)((long long)v << up));
    };
#pragma unroll
    for (int t = 0; t < 7; ++t)
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int b = 8 * (cg + 4 * t) + e;
        if (b < pad) add(row, b, sum0[t][e]);
        sum0[t][e] = 0;
      }
    for (int c = cg; 8 * c < n1; c += 4)
      for (int e = 0; e < 8; ++e) {
        int &v = sum1[(8 * c + e) * 128 + row];
        const int a = R - 128 + row;
        if (a >= 128) add(a, 128 + 8 * c + e, v);  // the tile's other rows are the first tile's
        v = 0;
      }
  };

#pragma unroll
  for (int q = 0; q < 2 * kWgRowPairs; ++q) d[q] = load(u0, q);
  bool ok = true;
  int since = 0, reads = 0;
  int64_t it = 0;
  for (int64_t u = u0; u < u1; ++u, ++it) {
    const int buf = (int)(it & 1);
    const uint32_t mb = tc_smem(&s_bar[buf]);
    const bool freed = it < 2 || tc_wait_warp(mb, (unsigned)((it - 2) >> 1) & 1u);
    unsigned char *const dst = wg_raw + (size_t)buf * kWgDigits * plane;
    const bool in = u * kWgUnit + lane < n;
    auto convert = [&](auto least) {  // digits from `least` on
#pragma unroll
    for (int i = 0; i < kWgRowPairs; ++i) {
      const int r0 = 2 * (warp + 16 * i);
      if (r0 < R) {
        unsigned long long v0 = (unsigned long long)wfix(d[2 * i], f) + shift[r0];
        unsigned long long v1 = (unsigned long long)wfix(d[2 * i + 1], f) + shift[r0 + 1];
        d[2 * i] = load(u + 1, 2 * i);  // the next unit's, while the other rows are converted
        d[2 * i + 1] = load(u + 1, 2 * i + 1);
        if (!in || r0 >= k) v0 = kWgBias;
        if (!in || r0 + 1 >= k) v1 = kWgBias;
        // even lanes keep row r0 of nodes lane, lane + 1, odd lanes row r0 + 1 of lane - 1, lane
        const bool odd = (lane & 1) != 0;
        const unsigned long long got = __shfl_xor_sync(0xffffffffu, odd ? v0 : v1, 1);
        const unsigned long long a = odd ? got : v0, b = odd ? v1 : got;
        unsigned char *const at = dst + (unsigned)(lane >> 3) * group + (unsigned)(r0 + (odd ? 1 : 0)) * 16u +
                                  (unsigned)((lane & 7) >> 1) * 4u;
#pragma unroll
        for (int p = decltype(least)::value; p < (int)kWgDigits; ++p)
          if (p <= dhi) *reinterpret_cast<uint32_t *>(at + (unsigned)p * plane) = wg_digit(a, b, p);
      }
    }
    };
    if (dlo == 0) convert(std::integral_constant<int, 0>());
    else if (dlo == 1) convert(std::integral_constant<int, 1>());
    else convert(std::integral_constant<int, 2>());
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the planes are read by the tensor cores
    asm volatile("tcgen05.fence::before_thread_sync;");
    const int stuck = __syncthreads_or(freed ? 0 : 1);
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (stuck) {
      ok = false;
      break;
    }
    if (warp == 0) {
      const uint32_t bs = base + (unsigned)buf * kWgDigits * plane;
      uint32_t add = since > 0 ? 1u : 0u;
      for (int p = dlo; p <= dhi; ++p) {
        const uint32_t pa = bs + (unsigned)p * plane, pb = bs + (unsigned)(cls - p) * plane;
#pragma unroll
        for (int st = 0; st < 2; ++st) {
          const uint32_t off = (unsigned)st * 2u * group;
          tc_mma_f16_warp(tmem, wg_desc(pa + off, group), wg_desc(pb + off, group), wg_idesc(pad), add);
          if (n1 > 0)
            tc_mma_f16_warp(tmem + 256u, wg_desc(pa + off + (unsigned)(R - 128) * 16u, group),
                            wg_desc(pb + off + 128u * 16u, group), wg_idesc(n1), add);
          add = 1u;
        }
      }
      tc_commit_warp(mb);
    }
    if (++since == flush || u + 1 == u1) {
      const bool done = tc_wait_warp(mb, (unsigned)(it >> 1) & 1u);
      if (!__syncthreads_and(done ? 1 : 0)) {
        ok = false;
        ++it;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
      for (int t = 0; t < 7; ++t)
        if (8 * (cg + 4 * t) < pad) {
          uint32_t v[8];
          wg_ld8(tlane + (unsigned)(8 * (cg + 4 * t)), v);
#pragma unroll
          for (int e = 0; e < 8; ++e) sum0[t][e] += __float2int_rn(__uint_as_float(v[e]));
        }
      for (int c = cg; 8 * c < n1; c += 4) {
        uint32_t v[8];
        wg_ld8(tlane + 256u + (unsigned)(8 * c), v);
#pragma unroll
        for (int e = 0; e < 8; ++e) sum1[(8 * c + e) * 128 + row] += __float2int_rn(__uint_as_float(v[e]));
      }
      since = 0;
      if (++reads == kWgSums || u + 1 == u1) {
        emit();
        reads = 0;
      }
      // the accumulators are free for the next unit's MMAs, which follow its barrier
    }
  }
  if (!ok) {
    if (tid == 0) dev_fail(status, SSM_E_TIMEOUT);
    // let what is still in flight finish (bounded) before the TMEM goes
    if (it > 0) tc_wait(tc_smem(&s_bar[(it - 1) & 1]), (unsigned)((it - 1) >> 1) & 1u);
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

__global__ void k_wgram_final(int32_t k, const unsigned *__restrict__ dmax, const unsigned long long *__restrict__ acc,
                              double *__restrict__ G) {
  const int64_t kk = (int64_t)k * k;
  const double unit = wfix_bad(*dmax) ? __longlong_as_double(0x7FF8000000000000ll) : scalbn(1.0, 32 - 2 * wfix_f(*dmax));
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < kk; t += (int64_t)gridDim.x * blockDim.x) {
    const int a = (int)(t / k), b = (int)(t - (int64_t)a * k);
    if (a > b) continue;
    auto part = [&](int q) { return (double)(long long)acc[q * kk + t]; };
    const double g = (scalbn(part(0), 48) + (scalbn(part(1), 32) + (scalbn(part(2), 16) + part(3)))) * unit;
    G[(size_t)a * k + b] = g;
    G[(size_t)b * k + a] = g;
  }
}

size_t wgram_tc_acc_words(int32_t k) { return 4 * (size_t)k * k; }

int launch_wgram_tc(int32_t n, int32_t k, const float *dist, const unsigned *dmax, const long long *centre,
                    unsigned long long *acc, double *G, int32_t *status, cudaStream_t s) {
  // cycles per unit of a class (conversion, MMAs, its share of a read-out) in
  // hundredths of the longest one's, from one class at a time at k = 200; at k = 60,
  // 100 and 128 the shares are the same within 5 %
  const int cost[kWgClasses] = {74, 80, 82, 88, 91, 95, 100, 92, 86};
  int total = 0;
  for (int c : cost) total += c;
  const int sms = std::max(num_sms(), 2 * kWgClasses);
  WgSplit split;
  int sum = 0;
  for (int c = 0; c <= kWgClasses; ++c) {
    split.start[c] = (int32_t)((int64_t)sms * sum / total);
    if (c < kWgClasses) sum += cost[c];
  }
  SSM_TRY_CUDA(allow_dynamic_smem((const void *)k_wgram_tc));
  SSM_TRY_CUDA(cudaMemsetAsync(acc, 0, wgram_tc_acc_words(k) * sizeof(unsigned long long), s));
  note_launch(), k_wgram_tc<<<sms, kWgThreads, wg_smem(k), s>>>(n, k, dist, dmax, centre, split, acc, status);
  const int64_t kk = (int64_t)k * k;
  note_launch(), k_wgram_final<<<(unsigned)((kk + 255) / 256), 256, 0, s>>>(k, dmax, acc, G);
  SSM_TRY_CUDA(cudaGetLastError());
  return SSM_OK;
}

}  // namespace ssm
