"""The FP64 build's square root, arctangent and logarithm (csrc/dmath.cuh)
compiled for the host, against long double."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_17084_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include <random>
#include "dmath.cuh"
int main() {
  static dm::Tables T;
  dm::fill_tables(&T);
  std::mt19937_64 g(1);
  std::uniform_real_distribution<double> U(0, 1);
  double es = 0, ea = 0, el = 0;
  for (int i = 0; i < 2000000; ++i) {
    const double x = pow(10, -21 + 23 * U(g));
    es = fmax(es, fabs((double)((long double)dm::root(x) / sqrtl(x) - 1)));
    const double b = (U(g) * 2 - 1) * pow(10, -40 * U(g) * (i & 1)), a = (U(g) * 2 - 1) * pow(10, -40 * U(g) * (i >> 1 & 1));
    ea = fmax(ea, fabs((double)(dm::arg(b, a, T.at) - atan2l(b, a))));
    const double N = pow(10, -12 + 13 * U(g)), D = i & 1 ? N * (1 + pow(10, -8 * U(g))) : pow(10, -12 + 13 * U(g));
    const long double L = logl(N) - logl(D);
    el = fmax(el, (double)(fabsl(dm::log_ratio(N, D, T.lg) - L) / fmaxl(1, fabsl(L))));
  }
  const double P = 3.14159265358979323846;
  const bool edges = dm::arg(0.0, 1.0, T.at) == 0 && dm::arg(0.0, -1.0, T.at) == P && dm::arg(2.0, 0.0, T.at) == P / 2 &&
                     dm::arg(-1e-24, 0.0, T.at) == -P / 2 && dm::arg(0.0, 0.0, T.at) == 0 &&
                     dm::max2(-0.0, 0.0) == 0 && !dm::gt(0.0, -0.0) && dm::gt(1.0, -2.0) && dm::gt(-1.0, -2.0);
  printf("%g %g %g %d\n", es, ea, el, (int)edges);
}
"""


def test_functions(tmp_path):
    cuda = "/usr/local/cuda/include"
    if not os.path.exists(cuda):
        pytest.skip("no CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.check_call(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-I", cuda, "-I", CSRC, "-D__forceinline__=inline",
                           "-D__host__=", "-D__device__=", str(src), "-o", str(exe)])
    es, ea, el, edges = subprocess.check_output([str(exe)], text=True).split()
    assert float(es) < 2.3e-16  # one rounding and a half
    assert float(ea) < 9e-16    # two roundings at pi's magnitude
    assert float(el) < 9e-16    # two roundings, relative above 1
    assert edges == "1"


GEOMETRY = r"""
#include <cstdio>
#include <random>
#include "dmath.cuh"
int main() {
  std::mt19937_64 g(2);
  std::uniform_real_distribution<double> U(0, 1);
  double eq = 0, ei = 0, el = 0, es = 0;
  for (int i = 0; i < 2000000; ++i) {
    // quotients of distances from 1 down to 1e-40, |a| from |b| down to 1e-13 of it
    const double b = pow(10, -40 * U(g)) * (i & 1 ? -1 : 1), a = b * (i & 2 ? U(g) : pow(10, -13 * U(g)));
    if (fabs(a) < fabs(b)) eq = fmax(eq, fabs((double)(dm::quot(a, b) - (long double)a / b)));
    const double len = pow(10, 0.5 - 30 * U(g));
    ei = fmax(ei, fabs((double)(dm::inverse(len) * (long double)len - 1)));
    const double d2 = pow(10, 1 - 60 * U(g));
    el = fmax(el, fabs((double)(dm::length(d2) / sqrtl(d2) - 1)));
    const double x = pow(10, -24 + 3 * U(g));
    es = fmax(es, fabs((double)(dm::root(x) / sqrtl(x) - 1)));
  }
  printf("%g %g %g %g\n", eq, ei, el, es);
}
"""


def test_quotients_and_lengths_of_the_grid(tmp_path):
    cuda = "/usr/local/cuda/include"
    if not os.path.exists(cuda):
        pytest.skip("no CUDA headers")
    src, exe = tmp_path / "g.cpp", tmp_path / "g"
    src.write_text(GEOMETRY)
    subprocess.check_call(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-I", cuda, "-I", CSRC, "-D__forceinline__=inline",
                           "-D__host__=", "-D__device__=", str(src), "-o", str(exe)])
    eq, ei, el, es = (float(v) for v in subprocess.check_output([str(exe)], text=True).split())
    assert eq < 1.2e-16  # one rounding of 1
    assert ei < 2.3e-16  # a rounding and a half
    assert el < 2.3e-16
    assert es < 6e-15    # down to 1e-24, as root's comment says
