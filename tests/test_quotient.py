"""The FP32 sweeps divide by the diagonal d of a uniform tree as fma(x, zh, x zl),
zh + zl = 1 / d in two floats: the correctly rounded quotient for every
significand of x, at every diagonal a uniform tree can have (2D: 8/3; 3D: 8/3
3^-depth, depth 0 to 7)."""
from __future__ import annotations

import shutil
import subprocess

import pytest

SOURCE = r"""
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
int main(void) {
  long bad = 0;
  for (int c = 0; c < 9; ++c) {
    double h = 1.0;
    for (int i = 0; i < c; ++i) h *= 3.0;
    h = 1.0 / h;
    const float d = (float)(c == 8 ? 4.0 * (4.0 / 6.0) : 8.0 * (4.0 / 12.0) * h);
    const float zh = 1.0f / d, zl = (float)(1.0 / (double)d - (double)zh);
    for (uint32_t m = 0; m < (1u << 23); ++m) {
      const uint32_t bits = 0x3f800000u | m;
      float x;
      memcpy(&x, &bits, 4);
      const float e = x * zl;
      bad += fmaf(x, zh, e) != x / d;
    }
  }
  printf("%ld\n", bad);
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("gcc") is None, reason="needs gcc")
def test_quotient_is_correctly_rounded(tmp_path):
    src, exe = tmp_path / "quotient.c", tmp_path / "quotient"
    src.write_text(SOURCE)
    subprocess.run(["gcc", "-O2", "-std=c11", "-ffp-contract=off", "-o", str(exe), str(src), "-lm"], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert int(out) == 0
