"""The quantiser's quotient x / scale: the product with the rounded reciprocal
and one correction by its fused-multiply-add residual.  Checked with the
host's IEEE fmaf against the fp32 division for every mantissa of the scale
and, around every value and every rounding midpoint of the e4m3 format
(mantissas k / 16), the seven floats x next to it.  Powers of two scale all
of it exactly in the range in which the kernel uses it.  The sign of zero is
kept as well."""
import os
import platform
import shutil
import subprocess
import tempfile

import pytest

SRC = r"""
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
static float f_of(uint32_t u) { float f; memcpy(&f, &u, 4); return f; }
static uint32_t u_of(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
static float quotient(float x, float s, float y) {
  const float q0 = x * y;
  return fmaf(fmaf(q0, s, -x), -y, q0);
}
int main(void) {
  long bad = 0, tot = 0;
  for (uint32_t i = 0; i < (1u << 23); i++) {
    const float s = f_of(0x3f800000u | i), y = 1.0f / s;
    for (int k = 0; k < 16; k++) {
      const float x0 = (float)((1.0 + k / 16.0) * (double)s);
      for (int d = -3; d <= 3; d++) {
        const float x = f_of(u_of(x0) + d);
        tot++;
        if (u_of(quotient(x, s, y)) != u_of(x / s)) bad++;
      }
    }
    if (u_of(quotient(-0.0f, s, y)) != u_of(-0.0f) || u_of(quotient(0.0f, s, y)) != 0) bad++;
  }
  printf("%ld %ld\n", tot, bad);
  return 0;
}
"""


def test_corrected_product_is_the_quotient_around_values_and_midpoints():
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        pytest.skip("no C compiler")
    flags = ["-O2", "-ffp-contract=off"]
    if platform.machine() in ("x86_64", "AMD64"):
        flags.append("-mfma")  # fmaf as one instruction; without it the library's fmaf is exact but slow
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "t.c"), os.path.join(d, "t")
        open(src, "w").write(SRC)
        subprocess.run([cc, *flags, "-o", exe, src, "-lm"], check=True)
        out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=600).stdout.split()
    assert int(out[0]) == (1 << 23) * 16 * 7 and int(out[1]) == 0
