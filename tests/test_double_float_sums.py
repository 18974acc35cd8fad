"""Double-float sums and sums of products (csrc/df32.cuh), compiled for the host: the same C
functions on the CPU, whose float arithmetic rounds as the device's does.

 - operator+ keeps the relative accuracy of its result where the high parts cancel: the sum
   of the low parts is exact, so 2^-47 of the result is left (a plain FP32 sum of the low
   parts leaves 2^-24).
 - a sum of products is no less accurate than a chain of renormalised multiply-adds
   (df_fma) at every length: 10 % on the root mean square for the sampling of 4000 sums
   (the two are equal at two and four products)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2312_13051_gb300", "csrc")

MAIN = r"""
#include <cmath>
#include <cstdio>
#include <random>
#define __host__
#define __device__
#define __forceinline__ inline
%s
typedef long double ld;
static ld val(df a) { return (ld)a.hi + (ld)a.lo; }
static df from(double x) { const float h = float(x); return df(h, float(x - double(h))); }
int main() {
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> u(-1, 1);
  double worst = 0;
  for (int t = 0; t < 200000; ++t) {  // equal high parts of opposite sign, low parts of their own
    const df a = from(u(g)), b(-a.hi, float(a.hi * 5.9e-8 * u(g)));
    const ld ex = ((ld)a.hi + b.hi) + ((ld)a.lo + b.lo), got = ((ld)(a + b).hi - ex) + (a + b).lo;
    if (ex != 0) worst = std::fmax(worst, double(fabsl(got) / fabsl(ex)));
  }
  std::printf("add %%.3e\n", worst);
  for (int sign = 0; sign < 2; ++sign)
    for (int K : {2, 4, 8, 24, 62, 128, 512, 2048}) {
      double r[2] = {0, 0};
      std::uniform_real_distribution<double> v(sign ? 0 : -1, 1);
      const int T = K > 200 ? 400 : 4000;
      for (int t = 0; t < T; ++t) {
        df chain(0.f), pair(0.f);
        ld ex = 0, sum = 0;
        for (int k = 0; k < K; k += 2) {
          const df a = from(v(g)), b = from(v(g)), c = from(v(g)), d = from(v(g));
          ex += val(a) * val(b) + val(c) * val(d);
          sum += fabsl(val(a) * val(b)) + fabsl(val(c) * val(d));
          chain = df_fma(c, d, df_fma(a, b, chain));
          df_mac2(pair, a, b, c, d);
        }
        const double e0 = double((val(chain) - ex) / sum), e1 = double((val(pair) - ex) / sum);
        r[0] += e0 * e0;
        r[1] += e1 * e1;
      }
      std::printf("sum %%d %%d %%.4f\n", sign, K, std::sqrt(r[1] / r[0]));
    }
}
"""


def _function(src, head):
    a = src.index(head)
    return src[a:src.index("\n}\n", a) + 3]


def test_double_float_sums(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src = open(os.path.join(CSRC, "df32.cuh")).read()
    basics = src[src.index("struct df {"):src.index("// Complex double-float.")]
    parts = [basics, _function(src, "__device__ __forceinline__ df df_fma("),
             _function(src, "__device__ __forceinline__ void df_mac2(")]
    main = tmp_path / "sums.cpp"
    main.write_text(MAIN % "\n".join(parts))
    exe = tmp_path / "sums"
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-o", str(exe), str(main)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [line.split() for line in out.splitlines()]
    assert float(rows[0][1]) <= 2.0 ** -47
    ratios = {(int(r[1]), int(r[2])): float(r[3]) for r in rows[1:]}
    assert len(ratios) == 16 and max(ratios.values()) <= 1.1, ratios
