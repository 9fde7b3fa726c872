"""csrc/wm_quotient.h on the host: the quotient equals IEEE division for every reciprocal
within an ulp that the device may start from (a subnormal quotient within its last bit)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_24882_gb300", "csrc")
SRC = r"""
#include <cstdint>
#include <cstdio>
#include <cstring>
#include "wm_quotient.h"
static float f(uint32_t u) { float x; std::memcpy(&x, &u, 4); return x; }
static uint32_t u(float x) { uint32_t v; std::memcpy(&v, &x, 4); return v; }
int main() {
  uint64_t s = 88172645463325252ull;
  long bad = 0;
  for (long i = 0; i < 3000000; ++i) {
    s ^= s << 13, s ^= s >> 7, s ^= s << 17;
    const uint32_t e = 64 + (uint32_t)((s >> 50) % 183);  // d from 2^-63 to 2^120
    const uint32_t ea = 27 + (uint32_t)((s >> 40) % 130);  // |a| from 2^-100 to 2^30
    uint32_t m = (uint32_t)s & 0x7fffff, k = (uint32_t)(s >> 23) & 0x7fffff;
    if (i % 7 == 0) m = 0x7fffff - m % 4;  // mantissas at both ends
    if (i % 11 == 0) k = k % 4;
    if (i % 13 == 0) k = 0x7fffff - k % 4;
    const float a = (i & 1 ? -1.f : 1.f) * f(ea << 23 | m), d = f(e << 23 | k);
    const float y = (float)(1.0 / (double)d);
    for (int o = -1; o <= 1; ++o) {
      const float q = wm_quotient_from(a, d, f(u(y) + o)), t = a / d;
      bad += std::fabs(t) >= 0x1p-126f ? q != t : !(std::fabs(q - t) <= 0x1p-149f);
    }
  }
  bad += wm_quotient_from(0.f, 3.f, 1.f / 3.f) != 0.f;
  std::printf("%ld\n", bad);
  return bad != 0;
}
"""


def test_quotient_is_correctly_rounded(tmp_path):
    cxx = shutil.which("g++") or pytest.skip("no g++")
    src = tmp_path / "q.cpp"
    src.write_text(SRC)
    exe = str(tmp_path / "q")
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-I", CSRC, "-o", exe, str(src)], check=True)
    assert subprocess.run([exe], capture_output=True, text=True).stdout.strip() == "0"
