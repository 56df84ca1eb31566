"""The packed pair arithmetic of csrc/ps_df.cuh on the CPU: two pairs side by side go through the
same steps as one (equal to the bit), exact where it says so, and sine and cosine of a pair within
their error bound."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2007_00308_gb300", "csrc")

MAIN = r"""
#include "ps_df.cuh"
#include <cstdio>
#include <cstring>
#include <random>
using namespace ps;
static const float4 tab[512] = {PS_SINCOS_TABLE_VALUES};
static bool same(float a, float b) { return std::memcmp(&a, &b, 4) == 0 || (a == 0.f && b == 0.f); }
int main() {
  std::mt19937_64 rng(11);
  auto uni = [&](double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); };
  auto val = [&](int it) {  // magnitudes 2^-20 to 2^12, zeros, and neighbours that cancel
    if (it % 13 == 0) return 0.f;
    return (float)((rng() & 1 ? 1 : -1) * std::exp2(uni(-20, 12)));
  };
  auto pair = [&](int it) { const float h = val(it); return DF{h, (float)(h * uni(-1, 1) * 2.9e-8)}; };
  long bad = 0, inexact = 0;
  for (int it = 0; it < 300000; ++it) {
    const DF x0 = pair(it), x1 = pair(it + 5), y = pair(it + 9), z0 = pair(it + 3), z1 = pair(it + 7);
    const DFP x{F2{x0.hi, x1.hi}, F2{x0.lo, x1.lo}}, z{F2{z0.hi, z1.hi}, F2{z0.lo, z1.lo}};
    const float near = it % 3 ? z1.hi : x1.hi * (1.f + 1e-6f);
    const DFP t = two_sum2(x.hi, F2{z0.hi, near}), d = two_diff2(x.hi, F2{z0.hi, near});
    const DF t0 = two_sum(x0.hi, z0.hi), t1 = two_sum(x1.hi, near), d0 = two_sum(x0.hi, -z0.hi), d1 = two_sum(x1.hi, -near);
    bad += !same(t.hi.x, t0.hi) + !same(t.lo.x, t0.lo) + !same(t.hi.y, t1.hi) + !same(t.lo.y, t1.lo);
    bad += !same(d.hi.x, d0.hi) + !same(d.lo.x, d0.lo) + !same(d.hi.y, d1.hi) + !same(d.lo.y, d1.lo);
    inexact += (double)d.hi.y + (double)d.lo.y != (double)x1.hi - (double)near;
    Acc2 A = acc_first2(x, y);
    acc_prod2(A, z, x0);
    Acc a0 = acc_first(x0, y), a1 = acc_first(x1, y);
    acc_prod(a0, z0, x0);
    acc_prod(a1, z1, x0);
    bad += !same(A.s.x, a0.s) + !same(A.e.x, a0.e) + !same(A.s.y, a1.s) + !same(A.e.y, a1.e);
    // a + g + x y against a sum in long double: one rounding and the pairs' own error
    const F2 v = sum_prod_round2(two_sum2(F2{z0.hi, near}, x.hi), x.lo, z, y);
    const long double w = (long double)z0.hi + x0.hi + x0.lo + ((long double)z0.hi + z0.lo) * ((long double)y.hi + y.lo);
    const long double mag = fabsl((long double)z0.hi) + fabsl(x0.hi) + fabsl((long double)z0.hi * y.hi);
    inexact += fabsl(v.x - w) > 0x1p-24L * fabsl(w) * 1.0001L + 0x1p-44L * mag + 1e-40L;
  }
  long off = 0;
  for (int it = 0; it < 300000; ++it) {
    const float h = it % 100 ? (float)uni(-20, 20) : (float)((it / 100 % 64) * 0.0122718463030851296);
    const DF x{h, (float)(h * uni(-1, 1) * 2.9e-8)};
    DF s, c;
    df_sincos(x, tab, s, c);
    const long double a = (long double)x.hi + x.lo;
    off += fabsl((long double)s.hi + s.lo - sinl(a)) > 2e-14L || fabsl((long double)c.hi + c.lo - cosl(a)) > 2e-14L;
  }
  std::printf("%ld %ld %ld\n", bad, inexact, off);
  return 0;
}
"""


def test_packed_pairs_are_the_scalar_ones(tmp_path):
    src = tmp_path / "m.cpp"
    src.write_text(MAIN)
    inc = [f"-I{CSRC}", "-I/usr/local/cuda/include"]
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", *inc, str(src), "-o", str(tmp_path / "m")])
    out = subprocess.check_output([str(tmp_path / "m")], text=True).split()
    assert out == ["0", "0", "0"]
