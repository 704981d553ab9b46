"""The number of V-cycles predicted before the next stopping norm
(csrc/chhs_predict.cuh), compiled for the host from the same source: equal to
the double-precision prediction for random norms and contractions, for ones
placed at its ties (to a few parts in 2^20 ... 2^52), and for norms and
tolerances near the ends of the double range."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
HEADER = os.path.join(os.path.dirname(HERE), "paper_1611_02967_gb300", "csrc", "chhs_predict.cuh")

PROGRAM = r'''
#include HEADER_PATH
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
using namespace chhs_dev;
int wrong = 0, n = 0;
void check(double r, double rmax, double tol, double tol_max, double num, double den, int ran, int cap) {
  // as the loop decided it in double precision throughout
  const double rho = std::fmin(std::fmax(std::pow(num / den, 1.0 / ran), 1e-3), 0.9), lr = std::log(rho);
  double need = r > tol ? std::log(tol / r) / lr : 0.0;
  if (rmax > tol_max) need = std::fmax(need, std::log(tol_max / rmax) / lr);
  const int want = std::max(1, (int)std::min((double)cap, std::floor(need + 0.5)));
  const int got = predict_inner(r, rmax, tol, tol_max, num, den, ran, std::max(cap, 1));
  wrong += got != std::min(want, std::max(cap, 1));
  ++n;
}
int main() {
  std::mt19937_64 g(3);
  std::uniform_real_distribution<double> u(0, 1);
  for (int k = 0; k < 400000; ++k) {
    const double tol = std::pow(10.0, -14 + 10 * u(g)), r = tol * std::pow(10.0, 8 * u(g) - 0.5);
    const double den = r * std::pow(10.0, 3 * u(g) - 0.3), tol_max = k & 1 ? 50 * tol : INFINITY;
    check(r, r * (1 + 80 * u(g)), tol, tol_max, r, den, 1 + (int)(4 * u(g)), (int)(5 * u(g)));
  }
  for (int k = 0; k < 400000; ++k) {  // need + 1/2 a whole number, a little to either side
    const int ran = 1 + (int)(4 * u(g)), whole = 2 + (int)(3 * u(g));
    const double tol = std::pow(10.0, -13 + 8 * u(g)), rho = 0.01 + 0.88 * u(g);
    const double r = tol * std::pow(rho, -(whole - 0.5)) * (1 + std::pow(2.0, -20 - 32 * u(g)) * (k & 1 ? 1 : -1));
    check(r, r, tol, INFINITY, r, r / std::pow(rho, ran), ran, 4);
    check(tol, r, tol, tol * (1 + 1e-9 * u(g)), r, r / std::pow(rho, ran), ran, 4);
  }
  for (int k = 0; k < 100000; ++k) {
    const double tol = std::pow(10.0, -300 + 590 * u(g)), r = tol * (1 + u(g) * 100), den = r * (1 + 20 * u(g));
    check(r, r, tol, INFINITY, r, den, 1, 4);
  }
  printf("%d %d\n", wrong, n);
  return 0;
}
'''


def test_equals_the_double_precision_prediction(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM.replace("HEADER_PATH", '"%s"' % HEADER))
    exe = tmp_path / "t"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", str(src), "-o", str(exe)], check=True)
    wrong, n = map(int, subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split())
    assert n == 1300000 and wrong == 0
