"""The dash walk's three forms on the CPU (csrc/ps_dash_walk.cuh): wherever the FP32
prefilter or the double-float walk decides a quad, it decides as the FP64 rule does, and
the cut vertices that it vouches for are the FP64 rule's to the bit."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2007_00308_gb300", "csrc")

MAIN = r"""
#include "ps_dash_walk.cuh"
#include <cstdio>
#include <cstdlib>
#include <random>
using namespace ps;
int main(int argc, char** argv) {
  const float offset = (float)atof(argv[1]);
  float pat[32];
  int np = 0;
  for (int i = 2; i < argc; ++i) pat[np++] = (float)atof(argv[i]);
  DashPattern P{};
  if (!dash_pattern(P, pat, np, offset)) return 2;
  std::mt19937_64 rng(7);
  auto uni = [&](double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); };
  long n = 0, quick = 0, sure = 0, cut = 0, vouched = 0, bad = 0;
  for (int it = 0; it < 200000; ++it) {
    // a start from 0 to 2^18 periods in, on a stretch end now and then; zero-length
    // quads, ordinary ones and some that hold many periods
    float sa = (float)(std::exp2(uni(-6, 18)) * P.period);
    if (it % 5 == 0) sa = (float)(std::floor(sa / P.period) * P.period + P.cum[it % (P.m2 + 1)] - P.offset);
    if (it % 97 == 0) sa = 0.f;
    float len = (float)(std::exp2(uni(-12, it % 50 ? 1 : 6)) * P.period);
    if (it % 11 == 0) len = 0.f;
    float sb = sa + len;
    if (it % 7 == 0) sb = (float)(std::floor(sb / P.period) * P.period + P.cum[it % (P.m2 + 1)] - P.offset);
    if (sb < sa) sb = sa;
    float4 v0, v1;
    v0.x = (float)uni(-50, 4100); v0.y = (float)uni(0, 1); v0.z = it % 3 ? 7.5f : 0.f; v0.w = (float)uni(0, 1e6);
    v1.x = v0.x + (float)uni(-1, 1); v1.y = (float)uni(0, 1); v1.z = 8.25f; v1.w = v0.w;
    const bool capped = it & 1;
    ++n;
    DashWalk x;
    x.start(P, sa, sb);
    double lo, hi;
    bool c0, c1;
    const int q = dash_quick(P, sa, sb);
    if (q >= 0) {  // whole or nothing, and no caps
      ++quick;
      int m = 0;
      while (x.next(P, true, lo, hi, c0, c1)) {
        ++m;
        if (lo != sa || hi != sb || c0 || c1) ++bad;
      }
      if (m != q) ++bad;
      x.start(P, sa, sb);
    }
    DashWalkDF w;
    w.start(P, sa, sb);
    DF a, b;
    bool at_a, at_b, d0, d1, differ = false;
    long mine = 0;
    while (w.next(P, capped, a, b, at_a, at_b, d0, d1)) {
      if (!x.next(P, capped, lo, hi, c0, c1)) { differ = true; break; }
      differ |= c0 != d0 || c1 != d1 || (at_a != (lo > sa)) || (at_b != (hi < sb));
      if (!(sb > sa)) continue;
      const DF d = df_diff(sb, sa);
      const float fe = 2.f * w.err / d.hi;
      const double dd = (double)sb - (double)sa;
      for (int end = 0; end < 2; ++end) {
        if (!(end ? at_b : at_a)) continue;
        bool ok = true;
        const DF e = end ? b : a;
        const float4 p = cut_rib(v0, v1, df_div(df_add_f(e, -sa), d), fe, ok);
        ok &= e.hi + (e.lo + w.err) == e.hi && e.hi + (e.lo - w.err) == e.hi;
        ++mine;
        if (!ok) continue;
        ++vouched;
        const double f = ((end ? hi : lo) - (double)sa) / dd;
        const float* A = &v0.x;
        const float* B = &v1.x;
        const float* G = &p.x;
        for (int c = 0; c < 4; ++c) {
          const double dv = (double)B[c] - (double)A[c];
          if ((float)((double)A[c] + f * dv) != G[c]) differ = true;
        }
        if ((float)(end ? hi : lo) != e.hi) differ = true;
      }
    }
    if (w.sure) {
      ++sure;
      cut += mine;
      if (x.next(P, capped, lo, hi, c0, c1)) differ = true;
      if (differ) ++bad;
    }
  }
  printf("%ld %ld %ld %ld %ld %ld\n", n, quick, sure, cut, vouched, bad);
  return 0;
}
"""

PATTERNS = [("0", "12 6"), ("3.25", "9 3 1 3"), ("-1.7", "7.3 2.1"), ("0.01", "0.1 0.2 0.3 0.05"),
            ("2", "5 0 0 5"), ("0.001", "0 3 4 2"), ("0", "3"), ("1e6", "2.5 1.25 0.3"),
            ("0", " ".join(["1", "0.5"] * 16)), ("0", "1e-3 2e-3"), ("5", "1e5 3e5")]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("dash_walk")
    src, exe = d / "main.cpp", d / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", f"-I{CSRC}",
                    "-I/usr/local/cuda/include", str(src), "-o", str(exe)], check=True)
    return exe


@pytest.mark.parametrize("offset,pattern", PATTERNS)
def test_prefilter_and_pair_walk_follow_the_fp64_rule(program, offset, pattern):
    r = subprocess.run([str(program), offset, *pattern.split()], check=True, capture_output=True, text=True)
    n, quick, sure, cut, vouched, bad = map(int, r.stdout.split())
    print(offset, pattern, r.stdout.strip())
    assert bad == 0
    assert n == 200000 and quick > 0 and vouched <= cut
    # (patterns off the FP32 grid leave their exact coincidences to the FP64 walk)
    assert sure > 0.5 * n and vouched > 0.5 * cut
