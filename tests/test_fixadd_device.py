"""The integer evaluation of binary64 sums, squares and halves (csrc/fixadd.cuh), the same operands
through the host's and the device's instructions (PTX carry chains, funnel shifts, bit-field masks):
equal bit for bit to the IEEE operations wherever it reports that it handles its operands.  Kinds:
exponent spreads, ties and carries, smooth fields, all exponents, zeros and exact cancellation."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_02495_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "fixadd.cuh"
#ifdef __CUDACC__
#define BOTH __host__ __device__
#else
#define BOTH
#endif
using namespace swept::fix;
struct Rng {  // splitmix64
  uint64_t s;
  BOTH uint64_t operator()() {
    uint64_t z = (s += 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
  }
};
BOTH inline uint64_t bits(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
BOTH inline double of_bits(uint64_t u) { double x; memcpy(&x, &u, 8); return x; }
// operands of one point: 0..4 spreads 1, 4, 12, 25, 30; 5 ties and carries; 6 smooth; 7 all exponents; 8 zeros and
// exact cancellation
BOTH inline void draw(int kind, Rng& g, double (&v)[5]) {
  const int spread[5] = {1, 4, 12, 25, 30};
  const int base = kind == 7 ? (int)(g() % 2000) - 1000 : (int)(g() % 41) - 20;
  for (int i = 0; i < 5; ++i) {
    uint64_t m = g() >> 12;
    if (kind == 5) m = ((g() & 1) ? (1ull << (g() % 53)) - (g() % 3) : (g() % 5) << (g() % 41)) & ((1ull << 52) - 1);
    v[i] = of_bits((uint64_t)(1023 + base - (int)(g() % (kind < 5 ? spread[kind] : 3))) << 52 | m | (g() << 63));
  }
  if (kind == 6) {
    const double c = 1.0 + (g() >> 12) * 0x1p-52, h = (double)(g() >> 40) * 0x1p-36;
    for (int i = 0; i < 5; ++i) v[i] = c + (i - 2) * h;
  }
  if (kind == 8)
    for (int i = 1; i < 5; ++i) {
      const int what = (int)(g() % 6);
      v[i] = what == 0 ? 0.0 : (what == 1 ? -v[0] : (what == 2 ? v[0] : v[i]));
      if (what == 3 && g() % 8 == 0) v[i] = -0.0;
    }
}
// wrong results of one draw; `handled` counts the points and runs that were not refused
BOTH inline unsigned check(int kind, Rng& g, unsigned* handled) {
  double v[5], d2, d4, bd, q;
  draw(kind, g, v);
  unsigned wrong = 0;
  if (second_fourth(v[0], v[1], v[2], v[3], v[4], d2, d4, &bd)) {
    ++*handled;
    const double s1 = v[3] + v[1], s2 = v[4] + v[0];
    wrong += bits(bd) != bits(v[1] - v[3]);
    wrong += bits(d2) != bits(fma(-2.0, v[2], s1));
    wrong += bits(d4) != bits(fma(6.0, v[2], fma(-4.0, s1, s2)));
  }
  if (square(v[0], q)) wrong += bits(q) != bits(v[0] * v[0]);
  const double p = of_bits(g() & (g() & 1 ? ~0ull : 0x803fffffffffffffull));
  if (p == p) wrong += bits(half(p)) != bits(0.5 * p);
  double a[12], col[4], sum[4];
  for (int i = 0; i < 12; ++i) a[i] = v[g() % 5] * (kind == 8 ? 1.0 : 1.0 + (double)(g() >> 40) * 0x1p-26);
  for (int i = 0; i < 4; ++i) col[i] = a[3 * i + 1];
  if (cross_sums<4, 3>(a, a + 2, v[0], v[4], col, sum)) {
    ++*handled;
    for (int i = 0; i < 4; ++i)
      wrong += bits(sum[i]) != bits((a[3 * i] + a[3 * i + 2]) + ((i ? col[i - 1] : v[0]) + (i < 3 ? col[i + 1] : v[4])));
  }
  return wrong;
}
constexpr int kThreads = 256, kBlocks = 64, kEach = 32;
#ifdef __CUDACC__
__global__ void run(int kind, unsigned long long* out) {
  unsigned wrong = 0, handled = 0;
  Rng g{(uint64_t)(blockIdx.x * kThreads + threadIdx.x) * 1000003ull + kind};
  for (int i = 0; i < kEach; ++i) wrong += check(kind, g, &handled);
  atomicAdd(out, wrong);
  atomicAdd(out + 1, handled);
}
#endif
int main(int, char** argv) {
  const int kind = atoi(argv[1]);
  unsigned long long out[2] = {0, 0};
#ifdef __CUDACC__
  unsigned long long* d;
  if (cudaMalloc(&d, sizeof out) || cudaMemset(d, 0, sizeof out)) return 1;
  run<<<kBlocks, kThreads>>>(kind, d);
  if (cudaMemcpy(out, d, sizeof out, cudaMemcpyDeviceToHost)) return 2;
#else
  for (int t = 0; t < kBlocks * kThreads; ++t) {
    unsigned handled = 0;
    Rng g{(uint64_t)t * 1000003ull + kind};
    for (int i = 0; i < kEach; ++i) out[0] += check(kind, g, &handled);
    out[1] += handled;
  }
#endif
  printf("%llu %llu\n", out[0], out[1]);
  return 0;
}
"""
TOTAL = 2 * 256 * 64 * 32  # points and runs
# least part handled: a spread of 30 exponents leaves few runs of 14 values, ties cancel, zeros refuse points
KINDS = [(0, 0.98), (1, 0.98), (2, 0.98), (3, 0.9), (4, 0.1), (5, 0.3), (6, 0.3), (7, 0.85), (8, 0.05)]


def counts(exe, kind):
    return tuple(map(int, subprocess.run([exe, str(kind)], check=True, capture_output=True, text=True).stdout.split()))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixhost")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")],
                   check=True)
    return str(d / "t")


@pytest.fixture(scope="module")
def device(tmp_path_factory):
    from paper_1612_02495_gb300 import build as libbuild

    d = tmp_path_factory.mktemp("fixdev")
    (d / "t.cu").write_text(SRC)
    subprocess.run([libbuild._nvcc(), *libbuild.ARCH, "-O3", "-std=c++17", "--fmad=false", "-I", CSRC, str(d / "t.cu"), "-o",
                    str(d / "t")], check=True)
    return str(d / "t")


@pytest.mark.parametrize("kind,least", KINDS)
def test_host(host, kind, least):
    wrong, handled = counts(host, kind)
    assert wrong == 0 and handled >= least * TOTAL


@pytest.mark.gpu
@pytest.mark.parametrize("kind", [k for k, _ in KINDS])
def test_device(host, device, kind):
    wrong, handled = counts(device, kind)
    assert wrong == 0
    assert handled == counts(host, kind)[1]  # the same points refused
