"""The double-float conversions of csrc/df.cuh against the language's own, for
every exponent of a double and of a float: widening is equal bit for bit;
splitting gives the nearest float and the nearest float to the rest (at a tie of
the leading part either neighbour, the two parts still adding up exactly)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), os.pardir, "paper_1905_07622_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cmath>
#include <cstring>
#include <random>
#include "df.cuh"
static double dbl(unsigned long long w) { double d; std::memcpy(&d, &w, 8); return d; }
static float flt(unsigned int w) { float f; std::memcpy(&f, &w, 4); return f; }
int main() {
  std::mt19937_64 g(11);
  long bad_split = 0, bad_widen = 0;
  const unsigned long long low[] = {0, 1, 0x0fffffff, 0x10000000, 0x10000001, 0x1fffffff, 0x20000000, 0x30000000};
  for (unsigned long long e = 0; e < 2048; ++e)
    for (int t = 0; t < 400; ++t) {
      unsigned long long m = g() & 0xfffffffffffffull;
      if (t < 64) m = (m & ~0x3fffffffull) | low[t % 8];
      if (t >= 64 && t < 72) m = 0xfffffe0000000ull + low[t % 8];  // a carry into the exponent
      const double d = dbl((g() & 1) << 63 | e << 52 | (m & 0xfffffffffffffull));
      float h, l;
      heat::df_split(d, h, l);
      const float h0 = (float)d, l0 = (float)(d - (double)h0);
      if (std::isnan(d)) { bad_split += !std::isnan(h); continue; }
      const bool tie = (m & 0x1fffffff) == 0x10000000;
      if (std::isinf(h0) || !tie) bad_split += !(h == h0 && (l == l0 || (std::isnan(l) && std::isnan(l0))));
      else bad_split += !((double)h + (double)l == (double)h0 + (double)l0 && std::fabs((double)l) == std::fabs((double)l0));
      bad_split += heat::df_narrow(d) != h;
    }
  for (unsigned int e = 0; e < 512; ++e)
    for (int t = 0; t < 400; ++t) {
      const float f = flt(e << 23 | (t < 2 ? t * 0x7fffff : (unsigned int)(g() & 0x7fffff)));
      const double w = heat::df_widen(f), w0 = (double)f;
      bad_widen += !(w == w0 || (std::isnan(w) && std::isnan(w0)));
    }
  std::printf("%ld %ld\n", bad_split, bad_widen);
  return 0;
}
"""


def test_conversions_equal_the_plain_ones(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "df_convert.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "df_convert"
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", os.path.abspath(CSRC), str(src), "-o", str(exe)], check=True,
                   capture_output=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["0", "0"]
