"""The adjoint's quotients from a reciprocal (quot, k_adjoint.cu) against the
FP32 division they stand for.  The function's own text is compiled for the host
(fmaf and unfused products round there as on the GPU) and compared over

* random significands, adversarial ones (near one, near two) among them, with
  dividends of 2^-100 .. 2^100 and divisors of 1 .. 2^60: equal bits,
* zeros, infinities and NaN in either operand: equal (NaN for NaN),
* dividends down to the smallest subnormal, divisors up to the largest finite:
  one unit in the last place.  For tiny dividends the remainder's rounding (to
  2^-149, error 2^-150) times r <= 1 joins the final rounding; for divisors
  above 2^126 the reciprocal is subnormal, good to 2^-21, and the correction
  leaves 2^-42.
"""
import os
import re
import shutil
import subprocess

import pytest

CU = os.path.join(os.path.dirname(__file__), "..", "paper_2208_08038_gb300", "csrc", "k_adjoint.cu")

MAIN = r"""
static float fb(uint32_t u) { float f; memcpy(&f, &u, 4); return f; }
static uint32_t bits(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
static uint64_t st = 88172645463325252ULL;
static uint64_t rnd(void) { st ^= st << 13; st ^= st >> 7; st ^= st << 17; return st; }
static uint32_t mant(int k, uint64_t v) {
  uint32_t m = (uint32_t)v & 0x7fffffu;
  return k == 1 ? m | 0x7fff00u : (k == 2 ? m & 0xffu : m);
}
static int same(float a, float b) { return (a != a && b != b) || a == b; }
static long ulps(float a, float b) {  /* same sign */
  long d = (long)(bits(a) & 0x7fffffffu) - (long)(bits(b) & 0x7fffffffu);
  return d < 0 ? -d : d;
}

int main(void) {
  long n = 0, bad = 0, badspec = 0, badtiny = 0;
  for (long k = 0; k < 40000000; ++k) {
    uint64_t v = rnd();
    uint32_t sx = (uint32_t)(v >> 63) << 31;
    float x = fb(sx | (uint32_t)(127 - 100 + (v >> 46) % 201) << 23 | mant(k % 3, v));
    float b = fb((uint32_t)(127 + (v >> 56) % 61) << 23 | mant((k / 3) % 3, v >> 23));
    if (b < 1.0f) continue;
    if (bits(quot(x, b, 1.0f / b)) != bits(x / b)) ++bad;
    ++n;
  }
  const float X[] = {0.0f, -0.0f, 1.5f, -2.75e30f, INFINITY, -INFINITY, NAN};
  const float Bs[] = {1.0f, 1.25f, 3.0e18f, 3.4e38f, INFINITY, NAN};
  for (int i = 0; i < 7; ++i)
    for (int j = 0; j < 6; ++j)
      if (!same(quot(X[i], Bs[j], 1.0f / Bs[j]), X[i] / Bs[j]) && !(j == 3 && ulps(quot(X[i], Bs[j], 1.0f / Bs[j]), X[i] / Bs[j]) <= 1))
        ++badspec;
  for (long k = 0; k < 20000000; ++k) {
    uint64_t v = rnd();
    float x = fb((uint32_t)(v >> 63) << 31 | (uint32_t)((v >> 46) % 40) << 23 | mant(k % 3, v));
    float b = fb((uint32_t)(127 + (v >> 56) % 127) << 23 | mant((k / 3) % 3, v >> 23));
    if (k & 1) x *= 0x1p+120f;
    if (ulps(quot(x, b, 1.0f / b), x / b) > 1) ++badtiny;
  }
  printf("%ld %ld %ld %ld\n", n, bad, badspec, badtiny);
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("gcc") is None, reason="needs gcc")
def test_quotient_from_reciprocal(tmp_path):
    body = re.search(r"__device__ __forceinline__ float quot\(.*?\n}\n", open(CU).read(), re.S).group(0)
    src, exe = os.path.join(tmp_path, "quot.c"), os.path.join(tmp_path, "quot")
    open(src, "w").write("#include <math.h>\n#include <stdint.h>\n#include <stdio.h>\n#include <string.h>\n"
                         "#define __device__ static\n#define __forceinline__\n"
                         "#define __fmul_rn(a, b) ((a) * (b))\n" + body + MAIN)
    subprocess.run(["gcc", "-O2", "-std=c99", "-ffp-contract=off", src, "-o", exe, "-lm"], check=True)
    n, bad, badspec, badtiny = map(int, subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split())
    assert n > 30_000_000
    assert (bad, badspec, badtiny) == (0, 0, 0)
