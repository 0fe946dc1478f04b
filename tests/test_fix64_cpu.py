"""Kernel values of the float64 sums (fix64.cuh), compiled for the host, against
long double: the relative error stays at float64's rounding however small the
value is.

Bound: 2^-53 for the rounding to 53 bits; w has 57 fraction bits, at most 3
units of them lost, and a root within 2^-58 of w < 2^5: together ln 2 (3 2^-57 +
2^-53); the exponential and Matern's product stay below 2^-57.  With the first
three below 2^-53 (1 + 0.13 + 0.70) the sum is below 2^-52.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "paper_2402_09531_gb300/csrc/fix64.cuh"
using namespace dw;
using namespace dw::fx;
static u64 table[kTable];

static long double exact(int kernel, long double r, long double sigma) {
  const long double t = r / sigma;
  if (kernel == DWFMM_K_GAUSS) return expl(-0.5L * t * t);
  if (kernel == DWFMM_K_EXP) return expl(-t);
  const long double s = sqrtl(3.0L) * t;
  return (1.0L + s) * expl(-s);
}

template <int KER>
double worst(int d, double edge, double sigma, int pairs, double close, double* smallest) {
  std::mt19937_64 gen(d * 1000 + pairs);
  std::uniform_real_distribution<double> u(0.0, 1.0);
  const int F = units_exponent(edge * std::sqrt(static_cast<double>(d)) * (1.0 + 1e-6));
  Consts c;
  if (!make_consts(KER, sigma, F, c)) return -1.0;
  double bad = 0.0;
  for (int i = 0; i < pairs; ++i) {
    u64 A[2] = {0, 0}, C[2] = {0, 0};
    s64 B[2] = {0, 0};
    long double r2 = 0.0L;
    // corner to corner for every eighth pair, from one site on for `close`
    for (int k = 0; k < d; ++k) {
      const double far = i % 8 == 0 ? 1.0 : u(gen);
      const double x = edge * (i % 8 == 0 ? 1e-3 * u(gen) : u(gen));
      const double y = close > 0.0 ? std::min(edge, x + edge * close * u(gen)) : edge * (1.0 - 1e-3 * (1.0 - far)) * far;
      const s64 X = static_cast<s64>(to_units(x, F)), Y = static_cast<s64>(to_units(y, F));
      const int h = static_cast<int>(X >> 30) - static_cast<int>(Y >> 30);
      const int l = static_cast<int>(X & 0x3fffffff) - static_cast<int>(Y & 0x3fffffff);
      for (int q = 0; q < 2; ++q) {
        A[q] += static_cast<u64>(static_cast<s64>(h) * h);
        B[q] += static_cast<s64>(h) * l;
        C[q] += static_cast<u64>(static_cast<s64>(l) * l);
      }
      const long double df = ldexpl(static_cast<long double>(X - Y), -F);
      r2 += df * df;
    }
    double out[2];
    phi64<KER, 2>(A, B, C, c, table, out);
    const long double want = exact(KER, sqrtl(r2), sigma);
    if (out[0] != out[1]) return 2.0;
    bad = std::max(bad, static_cast<double>(fabsl(out[0] / want - 1.0L)));
    *smallest = std::min(*smallest, out[0]);
  }
  return bad;
}

int main() {
  make_table(table);
  double all = 0.0, least = 1.0;
  int used = 0;
  const double sigmas[] = {0.51, 0.75, 1.0, 3.0, 100.0, 1e4};
  const double edges[] = {1e-3, 1.0, 1.9, 3.7, 7.9};
  const double closes[] = {0.0, 0.1, 1e-4, 1e-9, 1e-16};
  for (int d : {1, 3, 4, 8, 16})
    for (double s : sigmas)
      for (double e : edges)
        for (double cl : closes) {
          const double w[3] = {worst<DWFMM_K_EXP>(d, e, s, 4000, cl, &least), worst<DWFMM_K_MATERN32>(d, e, s, 4000, cl, &least),
                               worst<DWFMM_K_GAUSS>(d, e, s, 4000, cl, &least)};
          for (double v : w)
            if (v >= 0.0) {
              ++used;
              all = std::max(all, v);
            }
        }
  printf("%d %.4f %.3e\n", used, all * 0x1p53, least);
  return 0;
}
"""


def test_relative_error_of_kernel_values(tmp_path):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", ROOT, "-I", os.path.join(cuda, "include"), str(src), "-o", str(exe)],
                   check=True)
    used, bad, least = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert int(used) > 1000
    assert float(least) < 2.0 ** -28      # the range's lower end is reached
    assert float(bad) <= 2.0, (used, bad, least)
