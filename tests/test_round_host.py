"""f64_to_f32_rn (csrc/chhs_df64.cuh), compiled for the host from the same
source: the conversion to single precision bit for bit, over random bit
patterns, ties and their neighbours in even and odd significands, carries into
the exponent, the ends of the normal and subnormal ranges, zeros, infinities and
NaNs (which stay NaNs)."""
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
int wrong = 0;
void check(uint64_t b) {
  double x;
  memcpy(&x, &b, 8);
  const float got = f64_to_f32_rn(x), want = (float)x;
  if (std::isnan(want)) wrong += !std::isnan(got);
  else wrong += memcmp(&got, &want, 4) != 0;
}
int main() {
  std::mt19937_64 g(7);
  for (int k = 0; k < 2000000; ++k) check(g());
  for (int e = 870; e <= 1160; ++e)
    for (int k = 0; k < 400; ++k) {
      const uint64_t sign = g() & (1ull << 63), top = (k & 3) ? g() & 0x7FFFFFull : 0x7FFFFFull;
      for (uint64_t low : {0ull, 1ull, 0x0FFFFFFFull, 0x10000000ull, 0x10000001ull, 0x1FFFFFFFull, (unsigned long long)(g() & 0x1FFFFFFFull)})
        check(sign | (uint64_t)e << 52 | top << 29 | low);
    }
  for (double x : {0.0, -0.0, (double)INFINITY, -(double)INFINITY, (double)NAN, -(double)NAN}) check(df_bits(x));
  check(0x7FF0000000000001ull);
  check(0xFFF0000020000000ull);
  printf("%d\n", wrong);
  return 0;
}
'''


def test_is_the_conversion(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM.replace("HEADER_PATH", '"%s"' % HEADER))
    exe = tmp_path / "t"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", str(src), "-o", str(exe)], check=True)
    assert int(subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout) == 0
