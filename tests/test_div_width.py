"""The trace divides directions by the grid width with a reciprocal and one exact-remainder correction; it must
round like the division for every width (the same operations in C, on the CPU)."""
import ctypes
import os
import subprocess

SRC = r"""
#include <math.h>
#include <string.h>
static float div_width(float a, float w, float inv) {
  const float q = a * inv;
  return copysignf(fmaf(fmaf(-q, w, a), inv, q), a);
}
long check(unsigned seed, int per_width) {
  long bad = 0;
  for (int w = 2; w <= 32769; ++w) {
    const float W = (float)w, inv = 1.0f / W;
    for (int t = 0; t < per_width; ++t) {
      seed = seed * 1664525u + 1013904223u;
      /* magnitudes 2^-27 to 2^14, every mantissa, both signs; zeros now and then */
      unsigned b = (seed & 0x807fffffu) | ((100u + (seed >> 9) % 41u) << 23);
      if (t == 0) b = seed & 0x80000000u;
      float a;
      memcpy(&a, &b, 4);
      const float x = div_width(a, W, inv), y = a / W;
      if (memcmp(&x, &y, 4)) ++bad;
    }
  }
  return bad;
}
"""


def test_div_width_rounds_like_the_division(tmp_path):
    src, lib = tmp_path / "d.c", tmp_path / "d.so"
    src.write_text(SRC)
    subprocess.run(["gcc", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-o", str(lib), str(src), "-lm"], check=True,
                   env=dict(os.environ))
    fn = ctypes.CDLL(str(lib)).check
    fn.restype, fn.argtypes = ctypes.c_long, [ctypes.c_uint, ctypes.c_int]
    assert fn(12345, 300) == 0
