"""The double-float exponential, compiled for the host (every operation of it is an
IEEE one): its Taylor polynomial is summed in double-float from the first term to
the last, the same bits as Horner's rule written out here."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_29318_gb300", "csrc")

SHIMS = r"""
#include <cmath>
#include <cstdio>
#include <random>
using std::fabs; using std::fma; using std::isfinite;
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fdiv_rn(float a, float b) { return a / b; }
static inline float __fsqrt_rn(float a) { return std::sqrt(a); }
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline float __shfl_sync(unsigned, float v, int) { return v; }
static inline float __shfl_down_sync(unsigned, float v, unsigned) { return v; }
static inline float __shfl_xor_sync(unsigned, float v, int) { return v; }
"""

MAIN = r"""
using ff::dfloat;
static dfloat horner(dfloat x) {
  const float n = rintf(x.h * 1.44269504f);
  const dfloat nl = ff::df_mul(dfloat(n), dfloat(0.6931471805599453));
  const dfloat f = ff::df_add(x, dfloat(-nl.h, -nl.l));
  double fact[14] = {1.0};
  for (int k = 1; k < 14; ++k) fact[k] = fact[k - 1] * k;
  dfloat p(1.0 / fact[13]);
  for (int k = 12; k >= 0; --k) p = ff::df_add(ff::df_mul(p, f), dfloat(1.0 / fact[k]));
  return dfloat(ldexpf(p.h, (int)n), ldexpf(p.l, (int)n));
}
int main() {
  std::mt19937_64 g(1);
  int differ = 0;
  double worst = 0.0;
  for (int i = 0; i < 400000; ++i) {
    const double top = i % 4 == 0 ? 0.3 : i % 4 == 1 ? 1.0 : i % 4 == 2 ? 9.0 : 70.0;
    const dfloat x(-top * (double)(g() >> 11) / 9007199254740992.0);
    const dfloat a = ff::df_exp(x), b = horner(x);
    differ += a.h != b.h || a.l != b.l;
    const double want = std::exp((double)x.h + (double)x.l);
    worst = fmax(worst, fabs(((double)a.h + (double)a.l - want) / want) / (1.0 + top));
  }
  printf("%d %.3e\n", differ, worst);
}
"""


def test_every_term_in_double_float(tmp_path):
    """Of the error, n ln 2 contributes n (2^-48 + 2^-47) at most (the constant's rounding and the
    product's), the reduction and eight significant steps of Horner's rule 2^-45 in all."""
    cuda = next((p for p in ("/usr/local/cuda/include", "/usr/local/cuda/targets/sbsa-linux/include")
                 if os.path.exists(os.path.join(p, "cuda_runtime.h"))), None)
    if shutil.which("g++") is None or cuda is None:
        pytest.skip("needs g++ and CUDA's headers")
    src = tmp_path / "t.cpp"
    src.write_text("#include <cuda_runtime.h>\n" + SHIMS + '#include "dfloat.cuh"\n' + MAIN)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", cuda, "-I", CSRC,
                    str(src), "-o", str(exe)], check=True, capture_output=True, text=True)
    differ, worst = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert int(differ) == 0
    assert float(worst) < 2.0 ** -45
