"""Division by a multiplication (csrc/niti_div.h), which all tile and k-block coordinates of the tcgen05 kernel go through:
exact at the ends of the dividends' range and beside every multiple, for small, large and random divisors."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include "niti_div.h"
#include <cstdio>
static long long bad = 0, seen = 0;
static void check(long long n, long long d, Div v) {
  if (n < 0 || n > 0x7fffffffLL) return;
  ++seen;
  if (div_by((int)n, v) != (int)(n / d) && bad++ < 5) printf("%lld / %lld\n", n, d);
}
static void divisor(long long d) {
  const Div v = make_div(d);
  const long long top = 0x7fffffffLL, q = top / d;
  const long long factors[] = {0, 1, 2, 3, q / 3, q / 2, q - 1, q, q + 1};
  for (long long f : factors)
    for (int o = -2; o <= 2; ++o) check(f * d + o, d, v);
  for (int o = 0; o < 3; ++o) check(top - o, d, v);
}
int main() {
  for (long long d = 1; d <= 200000; ++d) divisor(d);
  for (int s = 1; s <= 31; ++s)
    for (int o = -3; o <= 3; ++o)
      if ((1LL << s) + o >= 1 && (1LL << s) + o <= 1LL << 31) divisor((1LL << s) + o);
  unsigned long long x = 88172645463325252ull;
  for (int i = 0; i < 400000; ++i) {
    x ^= x << 13; x ^= x >> 7; x ^= x << 17;
    divisor(1 + (long long)((x >> 33) >> (i % 31)));
  }
  for (int d = 1; d < 300; ++d) {
    const Div v = make_div(d);
    for (long long n = 0; n < 70000; ++n) check(n, d, v);
  }
  printf("%lld wrong of %lld\n", bad, seen);
  return bad != 0;
}
"""


def test_division_by_multiplication_is_exact(tmp_path):
    src, exe = tmp_path / "div.cc", tmp_path / "div"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2009_13108_b200", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    done = subprocess.run([str(exe)], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout
