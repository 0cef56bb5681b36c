"""Layouts that the host side and several kernels share, checked by a small program compiled from the
library's own header: what one warp loads at a time is one contiguous row."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

TWIST = r"""
#include <cstdio>
#include <vector>
#include "fdas_internal.h"
// 0: every twiddle has a place of its own and every warp load is contiguous (float4 by float4)
int check(int L, int n1, bool columns) {
  const int N2 = L / n1, h2 = N2 / 2;
  std::vector<int> seen(2 * L, 0);
  for (int n2 = 0; n2 < N2; ++n2)
    for (int k1 = 0; k1 < n1; ++k1) {
      const int at = fdas::twist_re(n2, k1, n1, h2);
      if (at < 0 || at + 2 >= 2 * L || seen[at]++ || seen[at + 2]++) return 1;
      // the pair (j, j + h2) is one float4: re, re, im, im
      if (n2 < h2 && (at % 4 != 0 || fdas::twist_re(n2 + h2, k1, n1, h2) != at + 1)) return 2;
    }
  if (columns) {   // lane t loads column pair r*n1 + t for one k1 at a time
    for (int r = 0; r < h2 / n1; ++r)
      for (int k1 = 0; k1 < n1; ++k1)
        for (int t = 0; t < n1; ++t)
          if (fdas::twist_re(r * n1 + t, k1, n1, h2) != fdas::twist_re(r * n1, k1, n1, h2) + 4 * t) return 3;
  } else {         // lane k1 loads pair j
    for (int j = 0; j < h2; ++j)
      for (int k1 = 0; k1 < n1; ++k1)
        if (fdas::twist_re(j, k1, n1, h2) != fdas::twist_re(j, 0, n1, h2) + 4 * k1) return 4;
  }
  return 0;
}
int main() {
  const int len[6] = {256, 512, 1024, 2048, 4096, 8192}, lanes[6] = {8, 16, 32, 32, 64, 128};
  const bool columns[6] = {true, true, false, true, false, false};
  for (int i = 0; i < 6; ++i)
    if (int rc = check(len[i], lanes[i], columns[i])) return std::printf("L = %d: %d\n", len[i], rc), 1;
  return 0;
}
"""

STACK = r"""
#include <cstdio>
#include <vector>
#include "fdas_internal.h"
int main() {
  std::vector<int> seen(fdas::kStackHalves, 0);
  for (int layer = 0; layer < 2; ++layer)
    for (int o = 0; o < 32; ++o)
      for (int i = 0; i < 32; ++i)
        for (int k = 0; k < 9; ++k) {
          const int at = fdas::stack_at(layer, o, i, k);
          if (at < 0 || at >= fdas::kStackHalves || seen[at]++) return std::puts("place"), 1;
        }
  // plane j, row 32 b + o: tap 11 - b of input channels 8j .. 8j + 7, and nothing where that is no tap
  for (int at = 0; at < fdas::kStackHalves; ++at) {
    const int e = at % 8, row = at / 8 % 480, j = at / (8 * 480) % 4, layer = at / (8 * 480 * 4), k = 11 - row / 32;
    const bool tap = k >= 0 && k < 9;
    if (seen[at] != (tap ? 1 : 0)) return std::puts("zero blocks"), 1;
    if (tap && fdas::stack_at(layer, row % 32, 8 * j + e, k) != at) return std::puts("row"), 1;
  }
  return 0;
}
"""

SEGMENTS = r"""
#include <cstdio>
#include "fdas_internal.h"
int main() {
  for (int sms : {148, 152})
    for (int most : {2, 4, 16})
      for (int64_t nseg = 1; nseg < 3000; nseg += 1 + nseg / 40)
        for (int Z = 1; Z <= 401; Z += 2) {
          const int s = fdas::wide_segments(nseg, Z, most, sms);
          const auto units = [&](int k) { return (nseg + k - 1) / k * Z; };
          const bool full = s == most, fits = units(s) <= sms, half_fits = s > 1 && units(s / 2) <= sms;
          if (s < 1 || s > most || most % s || !(full || fits) || half_fits)
            return std::printf("%ld segments x %d, %d: %d\n", (long)nseg, Z, most, s), 1;
        }
  return 0;
}
"""

SPLIT = r"""
#include <cstdio>
#include "fdas_internal.h"
// Longest CTA in positions when every group's start but the CTA's first counts 1.3 of them.
template <class First>
double longest(int64_t grid, int Z, const First& first) {
  double worst = 0;
  for (int64_t k = 0; k < grid; ++k) {
    const int64_t u0 = first(k), u1 = first(k + 1);
    if (u1 <= u0) continue;
    const double t = (double)(u1 - u0) + 1.3 * (double)((u1 - 1) / Z - u0 / Z);
    if (t > worst) worst = t;
  }
  return worst;
}
int main() {
  for (int64_t grid : {148, 152})
    for (int64_t ng = 1; ng < 40; ++ng)
      for (int Z = 1; Z <= 401; Z += 2) {
        const int64_t units = ng * Z;
        if (units <= grid) continue;
        const int cost = fdas::group_cost_of(units, ng, grid);
        const int64_t total = units + cost * ng, span = total / grid;
        struct { int64_t span; int span_extra, group_cost; } split{span, (int)(total % grid), cost};
        auto first = [&](int64_t k) { return fdas::first_unit_of(split, Z, (unsigned)k); };
        if (first(0) != 0 || first(grid) != units) return std::printf("ends: %ld x %d\n", (long)ng, Z), 1;
        for (int64_t k = 0; k < grid; ++k)
          if (first(k + 1) < first(k)) return std::printf("order: %ld x %d\n", (long)ng, Z), 1;
        const double plain = longest(grid, Z, [&](int64_t k) { return k * units / grid; });
        if (longest(grid, Z, first) > plain + 1e-9) return std::printf("longer: %ld x %d\n", (long)ng, Z), 1;
      }
  return 0;
}
"""


def run(tmp_path, source):
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(source)
    inc = ["-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(ROOT, "paper_1711_10855_gb300", "csrc")]
    subprocess.run([NVCC, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", *inc, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_twiddle_table_is_contiguous_over_the_lanes_of_a_load(tmp_path):
    run(tmp_path, TWIST)


def test_inference_weight_image_is_a_straight_copy(tmp_path):
    run(tmp_path, STACK)


def test_fewest_segments_per_cta_while_every_unit_has_an_sm(tmp_path):
    run(tmp_path, SEGMENTS)


def test_unit_split_is_never_longer_than_equal_ranges(tmp_path):
    run(tmp_path, SPLIT)
