// Fixed point of the squared weighted distances, and their centred Gram matrix
// on the tensor cores (wgram_tc.cu), for weighted PivotMDS.
#pragma once
#include "common.cuh"

namespace ssm {

// the exponent f from the largest |distance| (its bits): the largest with every
// X = d^2 2^f below 2^55 (the square of a distance above dmax / 16 is then exact).
// A table with an infinity or a NaN gives a NaN product, which
// the eigen-solve refuses.
__device__ __forceinline__ bool wfix_bad(unsigned dmax_bits) { return dmax_bits >= 0x7F800000u; }
__device__ __forceinline__ int wfix_f(unsigned dmax_bits) {
  const unsigned long long m = (dmax_bits & 0x7FFFFFu) | 0x800000u;
  return 54 - 2 * ((int)(dmax_bits >> 23) - 127) - ((m * m) >> 47 ? 1 : 0);
}

// round(d^2 2^f), d a normal float (below that: 0)
__device__ __forceinline__ long long wfix(float d, int f) {
  const unsigned b = __float_as_uint(d) & 0x7FFFFFFFu;
  const int e = (int)(b >> 23);
  if (e == 0) return 0ll;
  const unsigned long long m = (b & 0x7FFFFFu) | 0x800000u;
  const int sh = -(2 * (e - 150) + f);  // d^2 = m^2 2^(2 (e - 150)); at least -8 for d <= dmax
  if (sh > 48) return 0ll;
  return sh <= 0 ? (long long)((m * m) << -sh) : (long long)((m * m + (1ull << (sh - 1))) >> sh);
}

// G'_ab = sum_i V_ia V_ib 2^(-2 f), V = X - centre, into the symmetric k x k
// matrix G for k up to kWgMaxK; acc holds wgram_tc_acc_words(k) 64-bit words.
constexpr int kWgMaxK = 208;
size_t wgram_tc_acc_words(int32_t k);
int launch_wgram_tc(int32_t n, int32_t k, const float *dist, const unsigned *dmax, const long long *centre,
                    unsigned long long *acc, double *G, int32_t *status, cudaStream_t s);

}  // namespace ssm
