"""The integer evaluation of binary64 sums and squares (csrc/fixadd.cuh), compiled for the
host, against the IEEE operations it stands for: equal bit for bit wherever it reports that
it handles its operands, over exponent differences, cancellations, ties and signs, and
refusing zeros, subnormals, infinities and NaN."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_02495_gb300", "csrc")

SRC = r"""
#include "fixadd.cuh"
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <limits>
#include <random>
using namespace swept::fix;
static uint64_t bits(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
int main(int argc, char** argv) {
  const int kind = atoi(argv[1]);
  std::mt19937_64 g(17 + kind);
  long handled = 0, wrong = 0, total = 0;
  const int spread[6] = {1, 2, 4, 12, 25, 30};  // exponents within spread of each other
  for (long it = 0; it < 1000000; ++it, ++total) {
    double v[5];
    const int base = kind == 8 ? (int)(g() % 2000) - 1000 : (int)(g() % 41) - 20;
    for (int i = 0; i < 5; ++i) {
      uint64_t m = g() >> 12;
      if (kind == 6) m = ((g() & 1) ? (1ull << (g() % 53)) - (g() % 3) : (g() % 5) << (g() % 41)) & ((1ull << 52) - 1);
      v[i] = std::ldexp(1.0 + m * 0x1p-52, base - (int)(g() % (kind < 6 ? spread[kind] : 3)));
      if (g() & 1) v[i] = -v[i];
    }
    if (kind == 7) {  // smooth fields: differences far below the values
      const double c = 1.0 + (g() >> 12) * 0x1p-52, h = std::ldexp((double)(g() >> 40), -24 - (int)(g() % 20));
      for (int i = 0; i < 5; ++i) v[i] = c + (i - 2) * h + (i - 2) * (i - 2) * h * std::ldexp(1.0, -(int)(g() % 8));
    }
    double d2, d4, q;
    double bd;
    if (second_fourth(v[0], v[1], v[2], v[3], v[4], d2, d4, &bd)) wrong += bits(bd) != bits(v[1] - v[3]);
    if (second_fourth(v[0], v[1], v[2], v[3], v[4], d2, d4)) {
      ++handled;
      const double s1 = v[3] + v[1], s2 = v[4] + v[0];
      wrong += bits(d2) != bits(std::fma(-2.0, v[2], s1));
      wrong += bits(d4) != bits(std::fma(6.0, v[2], std::fma(-4.0, s1, s2)));
    }
    if (square(v[0], q)) wrong += bits(q) != bits(v[0] * v[0]);
    if (it % 8 == 0) {  // a column run of four points, rows of stride 3: (w, own, e)
      double a[12], col[4], sum[4];
      for (int i = 0; i < 12; ++i) a[i] = v[g() % 5] * (1.0 + (double)(g() >> 40) * 0x1p-26);
      for (int i = 0; i < 4; ++i) col[i] = a[3 * i + 1];
      if (cross_sums<4, 3>(a, a + 2, v[0], v[4], col, sum))
        for (int i = 0; i < 4; ++i)
          wrong += bits(sum[i]) != bits((a[3 * i] + a[3 * i + 2]) + ((i ? col[i - 1] : v[0]) + (i < 3 ? col[i + 1] : v[4])));
    }
    // half: any bit pattern, and the smallest exponents
    uint64_t p = g();
    if (it & 1) p &= 0x803fffffffffffffull;
    double h;
    memcpy(&h, &p, 8);
    if (h == h) wrong += bits(half(h)) != bits(0.5 * h);
    if (std::fabs(h) > 1e-37 && std::fabs(h) < 1e38)
      wrong += std::fabs((double)float_bits(h) - h) > 0x1p-23 * std::fabs(h) || std::fabs((double)float_bits(h)) > std::fabs(h);
    const float fb = float_bits(v[1]);
    wrong += !(std::fabs((double)fb) <= std::fabs(v[1]) && std::fabs((double)fb - v[1]) <= 0x1p-23 * std::fabs(v[1])) && kind != 8;
    // a value outside the range in any place is refused
    const double out[5] = {0.0, -0.0, 1e-310, std::numeric_limits<double>::infinity(), std::nan("")};
    v[g() % 5] = out[g() % 5];
    wrong += second_fourth(v[0], v[1], v[2], v[3], v[4], d2, d4);
  }
  printf("%ld %ld %ld\n", total, handled, wrong);
  return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixadd")
    src = d / "t.cpp"
    src.write_text(SRC)
    out = str(d / "t")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", out], check=True)
    return out


# kinds 0-5: exponent spreads; 6: structured significands (ties, carries); 7: smooth; 8: all exponents
@pytest.mark.parametrize("kind,least", [(0, 0.99), (1, 0.99), (2, 0.99), (3, 0.99), (4, 0.99), (5, 0.4), (6, 0.3),
                                        (7, 0.9), (8, 0.9)])
def test_equals_ieee(exe, kind, least):
    total, handled, wrong = map(int, subprocess.run([exe, str(kind)], check=True, capture_output=True,
                                                    text=True).stdout.split())
    assert wrong == 0
    assert handled >= least * total
