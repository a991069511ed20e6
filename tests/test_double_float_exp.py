"""The double-float exponential, checked on the CPU from the kernel source
itself: dl_exp and its table are cut out of the sources, compiled into a host
harness with g++ (each operation rounds as the device's does), and compared
with long double for 2^18 arguments per factor of four from 2^-14 to 69 (beyond,
the low part of e^-a is a denormal).

Error bound, relative to the result. Before the table: the argument's low part
and m ln2/1024's, up to 2^-24 |a| together, are added with one rounding, 2^-49
|a|, and the constant itself is known to 2^-50: less than 2^-48 |a|. From there
on, with |r| <= ln2/2048: r^2/2 + r^3/6 with two roundings of 2^-24 and r^4/24 left
out, 7.4e-15; one more at its addition, the table's low part and its addition,
3 x 2^-49; the last sum of what is below 2^-23, 2^-48: 1.63e-14 in all."""
import os
import shutil
import subprocess

import pytest

from test_comb_index import CSRC, _function

HARNESS = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#define __device__
#define __forceinline__ inline
struct float2 { float x, y; };
struct df { float hi, lo; };
typedef df dl;
struct LeanExp { float c_hi, c_lo, inv; };
constexpr int kExpBits = 10, kExpEntries = 1 << kExpBits;
static float __fmul_rn(float a, float b) { return a * b; }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static int __float_as_int(float f) { int i; memcpy(&i, &f, 4); return i; }
static float __int_as_float(int i) { float f; memcpy(&f, &i, 4); return f; }
static df df_make(float h, float l) { return {h, l}; }
static df fast_two_sum(float a, float b) { const float s = a + b; return {s, b - (s - a)}; }
static const float2 tab[kExpEntries] = {
#include "exp_table.inc"
};
@FUNCTION@
static df split(long double x) { const float h = (float)x; return {h, (float)(x - (long double)h)}; }
int main()
{
  const long double ln2 = logl(2.0L);
  const df c = split(ln2 / kExpEntries);
  const LeanExp K = {c.hi, c.lo, (float)(kExpEntries / ln2)};
  uint64_t s = 88172645463325252ull;
  for (double lo = 0x1p-14; lo < 69.0; lo *= 4.0) {
    const double hi = fmin(4.0 * lo, 69.0);
    double worst = 0.0;
    for (int i = 0; i < 1 << 18; ++i) {
      s ^= s << 13; s ^= s >> 7; s ^= s << 17;
      const df a = split(-(long double)(lo + (hi - lo) * ((s >> 11) * 0x1p-53)));
      const long double v = (long double)a.hi + a.lo, want = expl(v);
      const df r = dl_exp(a, K, tab);
      const double err = (double)fabsl((((long double)r.hi + r.lo) - want) / want);
      worst = fmax(worst, err / (double)(1.63e-14L - 0x1p-48L * v));
    }
    printf("%g %g %.3f\n", lo, hi, worst);
  }
  const df zero = dl_exp({-87.5f, 0.0f}, K, tab), top = dl_exp({88.5f, 0.0f}, K, tab), one = dl_exp({0.0f, 0.0f}, K, tab);
  return zero.hi == 0.0f && zero.lo == 0.0f && std::isinf(top.hi) && one.hi == 1.0f && one.lo == 0.0f ? 0 : 1;
}
"""


def test_error_bound(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    src = open(os.path.join(CSRC, "lean64.cuh")).read()
    text = HARNESS.replace("@FUNCTION@", _function(src, "__device__ __forceinline__ dl dl_exp("))
    path = tmp_path / "exp.cpp"
    path.write_text(text)
    exe = str(tmp_path / "exp")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(path), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    for line in out.stdout.splitlines():
        assert float(line.split()[2]) <= 1.0, out.stdout
