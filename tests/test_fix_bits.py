"""The fixed-point arithmetic of csrc/alb_fix.cuh against 64-bit arithmetic.

The header compiles as plain host C++; a small driver built here with g++
compares each function with long double results over its whole accepted range:
the exponential within the 5e-10 the header states (its parts: 2^-33 rounding,
FP32 polynomial, truncation to 2^-63 at the smallest population), the
multiplicative update within 2^-23 of its step, conversions to and from Q63 exactly or to
the stated absolute error. Runs on the CPU only.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER_DIR = os.path.join(ROOT, "paper_2009_13426_gb300", "csrc")

DRIVER = r"""
#include <math.h>
#include <stdio.h>
#include "alb_fix.cuh"
using namespace alb;
static const uint64_t TAB[FIXT_N] = {ALB_FIXT_TABLE_VALUES};
static uint64_t st = 0x9e3779b97f4a7c15ull;
static uint64_t next() {  /* splitmix64 */
  uint64_t z = (st += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
static double uni() { return (double)(next() >> 11) * 0x1p-53; }
int main() {
  const long double ONE = 9223372036854775808.0L;  /* 2^63 */
  /* exponential: every table edge with its neighbours, then random exponents */
  long double worst = 0;
  auto ex = [&](uint32_t y) {
    const long double want = exp2l(-(long double)y / 33554432.0L);
    const long double e = fabsl((long double)fix_exp(y, TAB) / ONE / want - 1);
    if (e > worst) worst = e;
  };
  for (uint32_t j = 0; j < FIX_Y_END; j += 1u << 16)
    for (int d = -2; d <= 2; ++d)
      if (j + d < FIX_Y_END) ex(j + d);
  ex(FIX_Y_END - 1);
  for (int k = 0; k < 3000000; ++k) ex((uint32_t)(next() % FIX_Y_END));
  printf("exp %Lg\n", worst);
  /* update: populations of every size, steps of both signs and all sizes */
  worst = 0;
  for (int k = 0; k < 3000000; ++k) {
    const uint64_t P = fix_exp((uint32_t)(next() % FIX_Y_END), TAB);
    const float bound = (float)(FIX_STEP_MAX * (k & 1 ? uni() : pow(2.0, -30 * uni())));
    const float d = (float)(k & 2 ? -bound * uni() : bound * (k & 4 ? 1.0 : uni()));
    const FixStep fs = fix_step(bound);
    const long double want = (long double)P * expl(-(long double)d);
    /* in units of the bound, beside the truncations to 2^-63 */
    const long double e = (fabsl((long double)fix_scale(P, d, fs) - want) - 2) / want / bound;
    if (e > worst) worst = e;
  }
  printf("scale %Lg\n", worst);
  /* to FP32 and FP64: correctly rounded */
  long bad = 0;
  for (int k = 0; k < 3000000; ++k) {
    uint64_t P = next() >> (next() % 62);
    if (!P) P = 1;
    if (k % 5 == 0) P = (P & ~0xffull) | 0x80;  /* near ties */
    if (k % 7 == 0) P = (1ull << (next() % 63)) + (next() % 3) - 1;
    if (!P) P = 1;
    if (fix_to_f32(P) != (float)P * 0x1p-63f) ++bad;
    if (fix_to_f64(P) != (double)P * 0x1p-63) ++bad;
  }
  printf("convert %ld\n", bad);
  /* doubles to Q63 modulo 2^64 (targets up to a few tens), and residuals */
  long double wt = 0, wr = 0;
  for (int k = 0; k < 3000000; ++k) {
    const double v = (uni() - 0.5) * pow(2.0, 7 - 60 * uni());
    const uint64_t q = fix_of_f64(v);
    /* v reduced to [-1, 1): exact in long double */
    const long double w = (long double)v - 2 * floorl(((long double)v + 1) / 2);
    const long double g = (long double)(int64_t)q / ONE;
    long double e = fabsl(g - w);
    if (e > 1) e = fabsl(e - 2);
    if (e > wt) wt = e;
    const double r = (uni() - 0.5) * pow(2.0, -1 - 50 * uni());
    const long double er = fabsl((long double)fix_residual_f32(fix_of_f64(r)) - (long double)r);
    const long double lim = fabsl((long double)r) * 0x1p-23L + 0x1p-55L;
    if (er / lim > wr) wr = er / lim;
  }
  printf("target %Lg\nresidual %Lg\nzero %d\n", wt, wr, fix_of_f64(0.0) == 0 && fix_of_f64(-0.0) == 0);
  return 0;
}
"""


@pytest.fixture(scope="module")
def report(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fix")
    src = d / "driver.cpp"
    src.write_text(DRIVER)
    exe = d / "driver"
    subprocess.run([cxx, "-O2", "-std=c++17", "-x", "c++", "-I", HEADER_DIR, str(src), "-o",
                    str(exe)], check=True, capture_output=True, text=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return {line.split()[0]: float(line.split()[1]) for line in out.splitlines()}


def test_exponential_within_its_bound(report):
    assert 0 < report["exp"] <= 5e-10


def test_update_within_its_bound(report):
    # of the bound on the step: the FP32 polynomial and its product (2^-23
    # together), the cubic's remainder (bound^3 / 24), the rounding of the factor
    # to 2^-29 of the bound
    assert report["scale"] <= 2.0 ** -23 + 9e-4 ** 3 / 24 + 2.0 ** -29


def test_conversions_round_once(report):
    assert report["convert"] == 0


def test_targets_and_residuals(report):
    assert report["target"] <= 2.0 ** -63 * 1.001
    assert report["residual"] <= 1.0
    assert report["zero"] == 1
