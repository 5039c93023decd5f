"""The quotient n / f of the founders' weights by a known divisor f = sqrt(fan-in)
(csrc/eco_params.cu, divide_by_known: one correction of n times the rounded
reciprocal) equals the IEEE quotient for every significand of n and every
fan-in that a configuration allows: D of 3 k^2 + 4, 3 k^2 + 8 and 4 k^2 + 16
for odd k up to 31, D without a patch, and H.  Exhaustive, in C, on the CPU."""
import ctypes
import subprocess

SRC = r"""
#include <math.h>
#include <stdint.h>
#include <string.h>
long mismatches(int fan) {
  const float f = sqrtf((float)fan), r = 1.0f / f;
  long bad = 0;
#pragma omp parallel for reduction(+ : bad)
  for (uint32_t m = 0; m < (1u << 23); ++m) {
    const uint32_t b = 0x3f800000u + m;
    float n;
    memcpy(&n, &b, 4);
    const float q = n * r;
    bad += fmaf(fmaf(-q, f, n), r, q) != n / f;
  }
  return bad;
}
"""


def test_every_significand_and_fan_in(tmp_path):
    (tmp_path / "d.c").write_text(SRC)
    so = str(tmp_path / "d.so")
    subprocess.run(["gcc", "-O2", "-ffp-contract=off", "-fopenmp", "-shared", "-fPIC", str(tmp_path / "d.c"), "-o", so, "-lm"],
                   check=True)
    lib = ctypes.CDLL(so)
    lib.mismatches.restype = ctypes.c_long
    fans = {4, 8, 16, 32, 64, 128}
    for k in range(1, 32, 2):
        fans |= {3 * k * k + 4, 3 * k * k + 8, 4 * k * k + 16}
    assert {f: n for f in sorted(fans) if (n := lib.mismatches(f))} == {}
