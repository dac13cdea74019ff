"""double -> float on the bits rounds as the conversion does.

csrc/float_bits.h is plain integer code: built here as C++ and compared with the
processor's conversion over random bits of every exponent, the neighbourhoods of ties
and of the ends of the normal range, zeros, subnormals, infinities and NaN.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "float_bits.h"
#include <math.h>
#include <initializer_list>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
static long long normal = 0;
static bool same(uint64_t b) {
  double d;
  memcpy(&d, &b, 8);
  const float f = (float)d;
  uint32_t want;
  memcpy(&want, &f, 4);
  bool ok;
  const unsigned got = mg::d2f_nearest_bits((unsigned)(b >> 32), (unsigned)b, &ok);
  if (ok) return ++normal, got == want;
  // left to the conversion: nothing that is normal in both formats by a wide margin
  return !(fabs(d) >= 0x1p-126 && fabs(d) < 0x1.fffffep127);
}
int main() {
  uint64_t s = 88172645463325252ull;
  auto next = [&] { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; };
  for (int e = 0; e < 2048; ++e)
    for (int i = 0; i < 3000; ++i) {
      uint64_t b = (next() & 0x800fffffffffffffull) | ((uint64_t)e << 52);
      if (i % 3 == 1) b = (b & ~0x1fffffffull) | 0x10000000ull;            // a tie
      if (i % 3 == 2) b |= (uint64_t)(next() & 1 ? 0xfffffe0000000ull : 0) | 0x0fffffffull;
      for (int k = -1; k <= 1; ++k)
        if (!same(b + k)) return printf("%016llx\n", (unsigned long long)(b + k)), 1;
    }
  for (uint64_t b : {0ull, 0x8000000000000000ull, 0x7ff0000000000000ull, 0xfff8000000000000ull, 0x47efffffe0000000ull,
                     0x47efffffefffffffull, 0x47effffff0000000ull, 0x380fffffffffffffull, 0x3810000000000000ull})
    if (!same(b)) return printf("%016llx\n", (unsigned long long)b), 1;
  bool ok;
  mg::d2f_nearest_bits(0x80000000u, 0u, &ok);
  if (!ok) return printf("zero\n"), 1;
  printf("%lld\n", normal);
  return 0;
}
"""


def test_rounds_as_the_conversion(tmp_path):
    src, exe = tmp_path / "bits.cpp", tmp_path / "bits"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2110_00328_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 1000000
