"""The sweep's wide loads of d_ip (csrc/dip_part.cuh), compiled for the host with
a table that checks every access: no load leaves the k n entries, and the words
hold what single entries give."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1608_08909_gb300", "csrc")

HARNESS = r"""
#include "dip_part.cuh"
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
using namespace ssm;
struct Table {
  const std::vector<uint16_t> &d;
  uint16_t entry(size_t i) const { return d.at(i); }
  unsigned word(size_t i) const { return d.at(2 * i) | (unsigned)d.at(2 * i + 1) << 16; }
  template <int W>
  void words(size_t first, unsigned (&w)[W]) const {
    if (first % (2 * W)) abort();  // misaligned
    for (int t = 0; t < W; ++t) w[t] = word(first / 2 + t);
  }
};
template <int W>
void rows(int n, int k, int loads) {
  std::vector<uint16_t> d((size_t)n * k);
  for (size_t i = 0; i < d.size(); ++i) d[i] = (uint16_t)(i * 40503u + 7u);
  const Table t{d};
  for (int a = 0; a < k; ++a)
    for (int64_t g = 0; 2 * W * g < n + 256; ++g) {  // tiles go past the last node
      const DipPart<W> v = dip_part<W>(t, (size_t)a * n + 2 * W * g, part_left<W>(n, g), loads);
      for (int q = 0; q < 2 * W; ++q) {
        const int64_t i = 2 * W * g + q;
        const unsigned got = v.w[q / 2] >> (16 * (q & 1)) & 0xFFFFu;
        if (got != (i < n ? d[(size_t)a * n + i] : 0u)) {
          std::printf("n %d k %d W %d loads %d node %lld\n", n, k, W, loads, (long long)i);
          std::exit(1);
        }
      }
    }
}
int main() {
  for (int n = 1; n <= 40; ++n)
    for (int k = 1; k <= 5; ++k)
      for (int loads = 0; loads <= (n % 8 == 0 ? 2 : 1); ++loads) {
        rows<1>(n, k, loads);
        rows<4>(n, k, loads);
      }
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host C++ compiler")
def test_distance_loads_stay_inside_the_table(tmp_path):
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
