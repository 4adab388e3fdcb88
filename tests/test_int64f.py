"""The integer-arithmetic binary64 functions of csrc/fvna_int64f.cuh return the
bits of the correctly rounded operation: compiled for the host and compared
with the host's own division, square root and product, over random operands,
operands at the ends of a binade, few-bit ones, and seeds displaced by up to
two units either way (more than the hardware approximations err)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1311_3004_gb300", "csrc")

SRC = r"""
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
static int g_off = 0;
#define INT64F_SEED_OFF g_off
#include "fvna_int64f.cuh"
using namespace fvna::int64f;
static u64 st = 88172645463325252ull;
static u64 rnd() { st ^= st << 13; st ^= st >> 7; st ^= st << 17; return st * 2685821657736338717ull; }
static double operand(u64 lo, u64 n) {
  u64 m = rnd() >> 12, k = rnd() % 8;
  if (k == 0) m &= 0xffffffull << 28;
  if (k == 1) m = 0;
  if (k == 2) m = ~0ull;
  if (k == 3) m = rnd() % 16;
  if (k == 4) m = 0xfffffffffffffull - rnd() % 16;
  if (k == 5) m = (1ull << (rnd() % 52)) - (rnd() & 1);
  return of_bits((m & 0xfffffffffffffull) | ((lo + rnd() % n) << 52) | ((rnd() & 1) << 63));
}
int main(int, char **v) {
  const long n = atol(v[1]);
  g_off = atoi(v[2]);
  long bad[4] = {0, 0, 0, 0};
  for (long i = 0; i < n; i++) {
    const bool near1 = i & 1;
    double x = operand(near1 ? 1021 : 520, near1 ? 5 : 1000);
    double y = operand(near1 ? 1021 : 520, near1 ? 5 : 1000);
    bad[0] += bits_of(rcp_mid(x)) != bits_of(1.0 / x);
    bad[1] += bits_of(div_normal(bits_of(x), bits_of(y))) != bits_of(x / y);
    bad[2] += bits_of(sqrt_mid(fabs(x))) != bits_of(sqrt(fabs(x)));
    x = operand(near1 ? 1021 : 517, near1 ? 5 : 517);
    y = operand(near1 ? 1021 : 517, near1 ? 5 : 517);
    if (rnd() % 9 == 0) x = (rnd() & 1) ? 0.0 : -0.0;
    if (rnd() % 9 == 0) y = (rnd() & 1) ? 0.0 : -0.0;
    bad[3] += bits_of(mulz(x, y)) != bits_of(x * y);
  }
  printf("%ld %ld %ld %ld\n", bad[0], bad[1], bad[2], bad[3]);
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    d = tmp_path_factory.mktemp("int64f")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-o",
                    str(d / "t"), str(d / "t.cpp")], check=True)
    return str(d / "t")


@pytest.mark.parametrize("off", [-2, -1, 0, 1, 2])
def test_bits_of_the_rounded_operation(exe, off):
    out = subprocess.run([exe, "4000000", str(off)], check=True, capture_output=True, text=True)
    assert out.stdout.split() == ["0", "0", "0", "0"]
