"""Sine and cosine of a double-float (the rollout of the FP32 path), compiled for the
host: within a double-float's own rounding of the exact value.

Bound: a value of at most 1 rounds to hi + lo with an error of at most half a unit
of lo, 2^-50; the FP64 function and the sum of the argument's two floats add at most
four units of 2^-53."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_10711_gb300", "csrc")

SHIM = r"""
#pragma once
#include <cmath>
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
#define __align__(n) alignas(n)
static inline float __fmul_rn(float a, float b) { volatile float r = a * b; return r; }
static inline float __fadd_rn(float a, float b) { volatile float r = a + b; return r; }
static inline float __fsub_rn(float a, float b) { volatile float r = a - b; return r; }
static inline float __fdiv_rn(float a, float b) { volatile float r = a / b; return r; }
static inline float __fsqrt_rn(float a) { volatile float r = std::sqrt(a); return r; }
static inline float __frsqrt_rn(float a) { volatile float r = 1.0f / std::sqrt(a); return r; }
static inline float __frcp_rn(float a) { volatile float r = 1.0f / a; return r; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline float __double2float_rn(double a) { return (float)a; }
"""

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "ucn_df.cuh"
using namespace ucn;
int main() {
  unsigned long long s = 1;
  long double worst = 0;
  for (double range : {0.5, 1.6, 3.2, 10.0})
    for (int i = 0; i < 200000; ++i) {
      s = s * 6364136223846793005ull + 1442695040888963407ull;
      const DF a = df_from(range * (2.0 * (double)(s >> 11) / 9007199254740992.0 - 1.0));
      DF sn, cs;
      df_sincos(a, sn, cs);
      const long double x = (long double)a.hi + a.lo;
      worst = fmaxl(worst, fmaxl(fabsl((long double)sn.hi + sn.lo - sinl(x)), fabsl((long double)cs.hi + cs.lo - cosl(x))));
    }
  printf("%.6Le\n", worst);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_sine_and_cosine_within_their_rounding(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(SHIM)
    (tmp_path / "main.cpp").write_text('#include <initializer_list>\n#include "cuda_runtime.h"\n#include <math.h>\n' + MAIN)
    exe = str(tmp_path / "sc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I" + str(tmp_path), "-I" + CSRC,
                    str(tmp_path / "main.cpp"), "-o", exe], check=True)
    worst = float(subprocess.run([exe], check=True, capture_output=True, text=True).stdout)
    assert worst <= 2.0 ** -50 + 4 * 2.0 ** -53, worst
