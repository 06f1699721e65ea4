"""The first two positions of window row 0 are free in every pass of a radius-2 scheme: the FP64 KS
tiers keep their count of failed trips there (KsNote, csrc/kernels.cuh).  Every load, store and
tier of every pass kind is walked through on the host, over tile widths, wide last tiles and
remainders."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_02495_gb300", "csrc")

SRC = r"""
#include <cstdint>
#include <cstdio>
#include "swept_geom.cuh"
#include "swept_phases.cuh"
using namespace swept;
static long hits = 0, out = 0;
struct Cx {
  static constexpr int kR = 2, kC = 1;
  Geom g;
  template <class F> void for_range(int lo, int hi, F&& f) { for (int i = lo; i < hi; ++i) f(i); }
  void sync() {}
  void touch(int r, int j) { hits += r == 0 && j < 2; out += j < 0 || j >= g.M; }
  void load_u(int r, int, int j, int64_t) { touch(r, j); }
  void store_u(int r, int, int j, int64_t) { touch(r, j); }
  void load_edge(int r, int, int j, int64_t) { touch(r, j); }
  void store_edge(int r, int, int j, int64_t) { touch(r, j); }
  void level(int s, int, int lo, int hi, int64_t, int) {
    for (int j = lo; j < hi; ++j) {
      touch(s & 1, j);
      for (int d = -2; d <= 2; ++d) touch((s - 1) & 1, j + d);
    }
  }
};
int main() {
  long passes = 0;
  for (int W = 8; W <= 128; W += 8)
    for (int X = 0; X < W; X += X < 4 ? 1 : 5)
      for (int hh = 1; hh <= W / 4; ++hh) {
        Geom g{};
        g.R = 2, g.S = 2, g.C = 1, g.W = W, g.h = W / 4, g.nt = 3, g.X = X, g.N = 3 * W + X;
        g.M = (W + X + 5) / 2 * 2, g.E = 2 * g.h * 4, g.bc = 0, g.chunk = 1;
        for (int b = 0; b < 3; ++b) {
          Cx cx{g};
          if (hh < g.h) {
            run_up(cx, g, b, hh, true);
            run_diamond(cx, g, b, 1, MODE_GAP, hh);
            passes += 2;
            continue;
          }
          run_up(cx, g, b, hh, false);
          for (int odd = 0; odd < 2; ++odd) {
            run_diamond(cx, g, b, odd, MODE_DIAMOND, hh);
            run_diamond(cx, g, b, odd, MODE_DOWN, hh);
          }
          passes += 5;
        }
      }
  printf("%ld %ld %ld\n", passes, hits, out);
}
"""


def test_row0_start_is_free(tmp_path):
    src, exe = tmp_path / "t.cpp", str(tmp_path / "t")
    src.write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(CSRC, "..", "..", "include"), str(src), "-o",
                    exe], check=True)
    passes, hits, out = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert passes > 10000 and hits == 0 and out == 0
