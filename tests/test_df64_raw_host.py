"""The double-single sum and product without renormalisation (df_add_raw,
df_mul_raw in csrc/chhs_df64.cuh), compiled for the host from the same source
and checked against long double: each to 2^-44 of the larger operand (or of
the product), also on pairs whose low part a cancellation has left as large as
the high part; the bound is the one df_add and df_mul are held to."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
HEADER = os.path.join(os.path.dirname(HERE), "paper_1611_02967_gb300", "csrc", "chhs_df64.cuh")

PROGRAM = r'''
#include HEADER_PATH
#include <cmath>
#include <cstdio>
#include <random>
using namespace chhs_dev;
int main() {
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> u(-1, 1);
  long double w_add = 0, w_mul = 0, w_face = 0;
  for (int k = 0; k < 300000; ++k) {
    const double x = u(g) * std::pow(10.0, (int)(g() % 20) - 10), y = u(g) * std::pow(10.0, (int)(g() % 20) - 10);
    const df64 a = df_split(x), b = df_split(y);
    const long double m = std::max(std::fabs((long double)x), std::fabs((long double)y));
    const df64 s = df_add_raw(a, b), p = df_mul_raw(a, b);
    w_add = std::max(w_add, std::fabs((long double)s.hi + s.lo - ((long double)x + y)) / m);
    w_mul = std::max(w_mul, std::fabs((long double)p.hi + p.lo - (long double)x * y) / std::fabs((long double)x * y));
    // a face's v = d + a (e + c a d) with d the difference of nearby values
    const double near = x * (1.0 + 1e-6 * u(g)), e0 = u(g), e1 = e0 * (1.0 + 1e-5 * u(g)), al = u(g), c = 1.5;
    const df64 d = df_sub_raw(df_split(near), a), e = df_sub_raw(df_split(e1), df_split(e0)), A = df_split(al);
    const df64 w = df_add_raw(df_mul_raw(df_split(c), df_mul_raw(A, d)), e), v = df_add_raw(df_mul_raw(A, w), d);
    const long double D = (long double)near - x, W = (long double)c * al * D + ((long double)e1 - e0);
    const long double scale = std::fabs((long double)x) * 3 + std::fabs((long double)e0);
    w_face = std::max(w_face, std::fabs((long double)v.hi + v.lo - (D + al * W)) / scale);
  }
  const df64 inf = df_sub_raw(df_split(INFINITY), df_split(1.0));
  printf("%Lg %Lg %Lg %d\n", w_add, w_mul, w_face, !std::isfinite(inf.hi + inf.lo));
  return 0;
}
'''


def test_raw_sum_product_and_face(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM.replace("HEADER_PATH", '"%s"' % HEADER))
    exe = tmp_path / "t"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", str(src), "-o", str(exe)], check=True)
    w_add, w_mul, w_face, non_finite = subprocess.run([str(exe)], capture_output=True, text=True,
                                                      check=True).stdout.split()
    assert float(w_add) <= 2.0 ** -44 and float(w_mul) <= 2.0 ** -43 and float(w_face) <= 2.0 ** -43
    assert int(non_finite) == 1
