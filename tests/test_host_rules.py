"""Layouts and predicates that the kernels share with plain C++: compiled with the host
compiler and checked exhaustively over small values, without a GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2412_09734_gb300", "csrc")


@pytest.fixture
def run_cpp(tmp_path):
    """Compiles a program against the kernel sources' headers; returns its output's lines."""
    def go(source):
        src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
        src.write_text(source)
        subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
        return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    return go


def test_batch_work_arrays_stay_apart_and_inside_the_buffer(run_cpp):
    lines = run_cpp(r"""
#include <cstdio>
#include "batch_work.h"
int main() {
  for (size_t m = 0; m < 40; m += 1 + m / 3)
    for (size_t n = 0; n < 150; n += 1 + n / 4)
      for (size_t za = 16; za < 90; za += 1 + (za - 16) / 2) {
        mpax::BatchWork w(m, n, za);
        std::printf("%zu %zu %zu %zu", m, n, za, w.total);
        const size_t at[15][2] = {{w.val, za}, {w.valt, za}, {w.c, n}, {w.l, n}, {w.u, n},
                                  {w.lc, m}, {w.uc, m}, {w.w, n}, {w.xa, n}, {w.xhat, n},
                                  {w.gbuf, n}, {w.ya, m}, {w.yhat, m}, {w.gys, m}, {w.gxs, n}};
        for (auto& a : at) std::printf(" %zu %zu", a[0], a[1]);
        std::printf("\n");
      }
}
""")
    rows = [[int(v) for v in line.split()] for line in lines if line]
    assert len(rows) > 1000
    for m, n, za, total, *at in rows:
        end = 0
        for start, length in sorted(zip(at[::2], at[1::2])):
            assert start % 16 == 0 and start >= end, (m, n, za)
            end = start + length
        assert end <= total, (m, n, za)


def test_power_round_decides_alike_before_and_after_its_own_end(run_cpp):
    """The launch of round t may read `done` before or after its first block writes t: both
    must run the round.  A later round's launches stop; a running iteration's do not."""
    lines = run_cpp(r"""
#include <cstdio>
#include "rules.h"
int main() {
  for (int done = 0; done < 6; ++done)
    for (int t = 1; t < 6; ++t)
      std::printf("%d %d %d\n", done, t, (int)mpax::power_round_over(done, t));
}
""")
    over = {(d, t): o for d, t, o in (map(int, line.split()) for line in lines if line)}
    for t in range(1, 6):
        assert over[0, t] == over[t, t] == 0
        assert all(over[d, t] == 1 for d in range(1, t))


def test_scaled_value_from_float_pairs_is_the_fp64_product(run_cpp):
    """Bit for bit, for values and factors over the whole float range and near 1, and for
    zeros, infinities and NaN."""
    lines = run_cpp(r"""
#include <cstdio>
#include <cstring>
#include <random>
#include "float_pair.h"
struct Pair { float x, y; };
static long bad = 0;
static void check(float a, double r, double c) {
  const float got = mpax::scale_pair(a, mpax::float_pair<Pair>(r), mpax::float_pair<Pair>(c), &r, &c);
  const float want = (float)(((double)a * r) * c);
  if (got != got && want != want) return;
  if (std::memcmp(&got, &want, 4) != 0 && bad++ < 5) std::printf("%a %a %a\n", a, r, c);
}
int main() {
  std::mt19937_64 g(1);
  std::uniform_real_distribution<double> u(0.0, 1.0);
  auto pick = [&](double lo, double hi) {
    return std::ldexp(1.0 + u(g), (int)std::floor(lo + (hi - lo) * u(g)));
  };
  for (long i = 0; i < 3000000; ++i) {
    check((float)pick(-149, 128) * (i & 1 ? 1.0f : -1.0f), pick(-149, 100), pick(-149, 100));
    check((float)pick(-4, 4), pick(-4, 4), pick(-4, 4));
    check((float)pick(90, 128), pick(-128, -90), pick(-3, 3));
  }
  for (float a : {0.0f, -0.0f, INFINITY, -INFINITY, NAN, 1.0f})
    for (double r : {0.0, 1.0, 1e-40, 1e30})
      for (double c : {0.0, 1.0, 1e-40, 1e30})
        check(a, r, c);
  std::printf("bad %ld\n", bad);
}
""")
    assert lines[-2] == "bad 0", lines
