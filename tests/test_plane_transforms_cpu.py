"""The two-pass transforms of the fixed-point plane kernels at every side the library accepts, replayed
on the host from pcf_fx.cuh: the plan covers the length, every slot of a row is used once and lies in
the row, twiddle indexes stay in the table, and both directions agree with the DFT.

Tolerance: inputs sum to 2^61 units; a pass rounds each value a few times by at most one unit, so
that R + S roundings of the first and the second pass stay below 2^-54 of that sum."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SIDES = [18, 24, 36, 54, 72, 108, 16, 32, 48, 64, 96, 128]

SOURCE = r"""
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "pcf_fx.cuh"
using namespace pcf;
typedef long double LD;
typedef std::complex<LD> C;
static const LD kPi = 3.14159265358979323846264338327950288L;
static fxtw twiddle(int q, int L, bool inv) {
  const LD a = (inv ? 2 : -2) * kPi * q / L;
  const auto split = [](LD v, int* h, int* l) {
    const long long z = std::llrint(std::ldexp(v, 62));
    *l = (int)(uint32_t)(uint64_t)z;
    *h = (int)((z - *l) >> 32);
  };
  fxtw w;
  split(std::cos(a), &w.ch, &w.cl);
  split(std::sin(a), &w.sh, &w.sl);
  return w;
}
template <int R, int S, bool INV>
static double run(int L) {
  std::mt19937_64 gen(L);
  std::vector<int> used(L, 0);
  for (int b = 0; b < R; ++b)
    for (int e = 0; e < S; ++e) {
      const int s = fx_slot<S>(b, e);
      if (s < 0 || s >= L || used[s]++) return 1e9;
    }
  double worst = 0;
  for (int trial = 0; trial < 20; ++trial) {
    std::vector<fxc> buf(L);
    std::vector<C> x(L);
    for (int i = 0; i < L; ++i) {
      const fxc v{(long long)gen() / (8 * L), (long long)gen() / (8 * L)};
      buf[fx_slot<S>(i / S, i % S)] = v;
      x[i] = C(v.x, v.y);
    }
    for (int n = 0; n < S; ++n) {
      fxc v[R];
      for (int q = 0; q < R; ++q) v[q] = buf[fx_slot<S>(q, n)];
      FxDft<R, INV>::run(v);
      for (int k = 0; k < R; ++k) {
        if (n * k >= L) return 1e9;
        buf[fx_slot<S>(k, n)] = k ? fx_cmul(v[k], twiddle(n * k, L, INV)) : v[k];
      }
    }
    for (int b = 0; b < R; ++b) {
      fxc v[S];
      for (int e = 0; e < S; ++e) v[e] = buf[fx_slot<S>(b, e)];
      FxDft<S, INV>::run(v);
      for (int e = 0; e < S; ++e) buf[fx_slot<S>(b, e)] = v[e];
    }
    for (int i = 0; i < L; ++i) {  // output i = b + R k
      C s = 0;
      for (int n = 0; n < L; ++n) {
        const LD a = (INV ? 2 : -2) * kPi * (i * n % L) / L;
        s += x[n] * C(std::cos(a), std::sin(a));
      }
      const fxc o = buf[fx_slot<S>(i % R, i / R)];
      worst = std::max(worst, (double)(std::abs(s - C(o.x, o.y)) / std::ldexp((LD)1, 61)));
    }
  }
  return worst;
}
template <int R, int S>
static double both(int L) { return std::max(run<R, S, true>(L), run<R, S, false>(L)); }
int main(int argc, char** argv) {
  for (int i = 1; i < argc; ++i) {
    const int L = std::atoi(argv[i]);
    const FxPlan p = fx_plan(L);
    double e = 1e9;
    if (p.R * p.S == L && p.R % 2 == 0) switch (p.R * 100 + p.S) {
      case 208: e = both<2, 8>(L); break;
      case 408: e = both<4, 8>(L); break;
      case 608: e = both<6, 8>(L); break;
      case 808: e = both<8, 8>(L); break;
      case 1208: e = both<12, 8>(L); break;
      case 1608: e = both<16, 8>(L); break;
      case 603: e = both<6, 3>(L); break;
      case 406: e = both<4, 6>(L); break;
      case 606: e = both<6, 6>(L); break;
      case 609: e = both<6, 9>(L); break;
      case 1206: e = both<12, 6>(L); break;
      case 1209: e = both<12, 9>(L); break;
    }
    std::printf("%d %.17g\n", L, e);
  }
}
"""


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-x", "c++", "-I", os.path.join(ROOT, "paper_2306_00165_gb300", "csrc"),
                    str(d / "fx.cpp"), "-o", str(d / "fx")], check=True)
    out = subprocess.run([str(d / "fx"), *map(str, SIDES)], check=True, capture_output=True, text=True).stdout
    return {int(a): float(b) for a, b in (line.split() for line in out.splitlines())}


def test_sides_are_all_that_the_library_accepts():
    import paper_2306_00165_gb300 as pcf
    pcf._build.build()
    lib = pcf.load_library()
    for axis in (0, 2):
        ok = []
        for n in range(1, 300):
            g = [16, 33, 16]
            g[axis] = n
            if lib.pcf_state_len(*g) > 0:
                ok.append(n)
        assert ok == sorted(SIDES)


@pytest.mark.parametrize("side", SIDES)
def test_transform_of_every_accepted_side(errors, side):
    assert errors[side] <= 2.0 ** -54
