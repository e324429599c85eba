"""The trace's own div_width, taken from its source and compiled for the CPU with the intrinsics' meaning (one rounding
each), must round like the division for every grid width that the pyramid's levels hold."""
import ctypes
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1811_02357_gb300", "csrc")

FRAME = r"""
#include <math.h>
#include <string.h>
#define __device__
#define __forceinline__ static inline
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
%s
extern "C" long check(unsigned seed, int widest, int per_width) {
  long bad = 0;
  for (int w = 2; w <= widest; ++w) {
    const float W = (float)w, inv = %s;
    for (int t = 0; t < per_width; ++t) {
      seed = seed * 1664525u + 1013904223u;
      /* magnitudes 2^-27 to 2^14, every mantissa, both signs; zeros now and then */
      unsigned b = (seed & 0x807fffffu) | ((100u + (seed >> 9) %% 41u) << 23);
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


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _wrong(tmp_path, body, inv):
    src, so = tmp_path / "d.cpp", tmp_path / "d.so"
    src.write_text(FRAME % (body, inv))
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-o", str(so), str(src), "-lm"], check=True)
    fn = ctypes.CDLL(str(so)).check
    fn.restype, fn.argtypes = ctypes.c_long, [ctypes.c_uint, ctypes.c_int, ctypes.c_int]
    levels = int(re.search(r"constexpr int kMaxLevels = (\d+);", _source("geom.cuh")).group(1))
    return fn(4321, (1 << (levels - 1)) + 1, 300)


def test_the_source_rounds_like_the_division(tmp_path):
    text = _source("trace.cu")
    body = re.search(r"__device__ __forceinline__ float div_width\(.*?\n}\n", text, re.S).group(0)
    inv = re.search(r"o\.inv_w = (.*?);", text).group(1).replace("c.W", "w")
    assert _wrong(tmp_path, body, inv) == 0
