// A few consecutive 16-bit distances of the d_ip table, two per 32-bit word, by
// the widest loads that the row's alignment admits.  No load reaches past the
// k n entries of the table.  (Compiles as plain C++ as well, with a table that
// checks every access: tests/test_dip_part.py.)
#pragma once
#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define SSM_HD __host__ __device__ __forceinline__
#else
#define SSM_HD inline
#endif

namespace ssm {

// loads of d_ip: 16 bytes at a time (2: n a multiple of 8 and dip on 16 bytes),
// aligned words, shifted where the row starts in the middle of one (1: dip on 4
// bytes), or single entries (0)
enum DipLoads : int32_t { kDipEntries = 0, kDipWords = 1, kDipQuads = 2 };

// the 2 W entries of d_ip from entry `first` on, two per word (0 from the left-th on)
template <int W>
struct DipPart {
  unsigned w[W];
};

// T.entry(i): entry i; T.word(i): entries 2 i, 2 i + 1; T.words<W>(first, w): 2 W
// entries from first (a multiple of 2 W) on
template <int W, class T>
SSM_HD DipPart<W> dip_part(const T &dip, size_t first, int left, int32_t loads) {
  DipPart<W> v;
  if (loads == kDipQuads) {  // all of them are there, or none
    if (left) {
      dip.template words<W>(first, v.w);
    } else {
#ifdef __CUDACC__
#pragma unroll
#endif
      for (int t = 0; t < W; ++t) v.w[t] = 0u;
    }
  } else if (loads == kDipWords && left == 2 * W && (first & 1u) == 0) {  // whole words
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int t = 0; t < W; ++t) v.w[t] = dip.word((first >> 1) + t);
  } else if (loads == kDipWords) {
    const int odd = (int)(first & 1u);
    unsigned w[W + 1];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int t = 0; t < W + 1; ++t) {
      const int lo = 2 * t - odd;  // the word's entries: lo and lo + 1 from first on
      // where only the lower one is wanted it is loaded alone: the upper one may
      // be past the table
      w[t] = !(left > 0 && lo < left) ? 0u : lo + 1 < left ? dip.word((first >> 1) + t) : (unsigned)dip.entry(first + lo);
    }
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int t = 0; t < W; ++t) {
      const unsigned x = odd ? (w[t] >> 16) | (w[t + 1] << 16) : w[t];
      v.w[t] = 2 * t + 1 < left ? x : 2 * t < left ? x & 0xFFFFu : 0u;
    }
  } else {
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int t = 0; t < W; ++t) {
      const unsigned lo = 2 * t < left ? (unsigned)dip.entry(first + 2 * t) : 0u;
      const unsigned hi = 2 * t + 1 < left ? (unsigned)dip.entry(first + 2 * t + 1) : 0u;
      v.w[t] = lo | (hi << 16);
    }
  }
  return v;
}

// how many of the nodes 2 W g .. 2 W (g + 1) - 1 there are
template <int W>
SSM_HD int part_left(int n, int64_t g) {
  const int64_t left = n - 2 * W * g;
  return (int)(left < 0 ? 0 : left < 2 * W ? left : 2 * W);
}

}  // namespace ssm
