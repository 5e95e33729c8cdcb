"""The fixed-point matrix-vector product of the FP64 forms (fx_words and fx_fold of pcf_fx.cuh), replayed on
the host in 128-bit integers: words fit 32 bits, both sums stay inside 64 bits, and the error is at most
2^-55.9 of (largest entry) x (sum of the column's magnitudes), with low words at their largest, for every
length up to 65 terms: 65 x 2^54 of 2^116 for the product left out, 2^54 for the rounding."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "pcf_fx.cuh"
using namespace pcf;
typedef __int128 wide;
int main() {
  std::mt19937_64 gen(1);
  double worst = 0;
  for (int K = 1; K <= 65; ++K)
    for (int t = 0; t < 400; ++t) {
      wide exact = 0, H = 0, Cr = 0;
      for (int k = 0; k < K; ++k) {
        // entries up to 2^57, column values that sum to less than 2^59
        const fx xm = ((1LL << 59) - (1LL << 44)) / K;
        fx a = t % 4 == 0 ? 1LL << 57 : (fx)(gen() >> 7), x = t % 4 == 0 ? xm : (fx)(gen() % (unsigned long long)xm);
        if (t % 4 == 1) {  // low words at their largest, of one sign
          a = (a & ~((1LL << 28) - 1)) | ((1LL << 27) - 1);
          if (x >= 1LL << 28) x = (x & ~((1LL << 28) - 1)) | ((1LL << 27) - 1);
        }
        if (t % 4 == 3) {
          if (gen() & 1) a = -a;
          if (gen() & 1) x = -x;
        }
        int ah, al, xh, xl;
        fx_words(a, &ah, &al);
        fx_words(x, &xh, &xl);
        if ((((fx)ah << 28) + al) != a || (((fx)xh << 28) + xl) != x) return 1;
        exact += (wide)a * x;
        H += (wide)ah * xh;
        Cr += (wide)ah * xl + (wide)al * xh;
        const wide lim = (wide)1 << 63;
        if (H * 2 >= lim || -H * 2 >= lim || Cr + (1 << 26) >= lim || -Cr >= lim) return 2;
      }
      const wide got = (wide)fx_fold((fx)H, (fx)Cr) << 55;
      worst = std::fmax(worst, std::fabs((double)(got - exact)) / std::ldexp(1.0, 116));
    }
  std::printf("%.17g\n", worst);
}
"""


def test_matrix_vector_product(tmp_path):
    (tmp_path / "dot.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2306_00165_gb300", "csrc"),
                    str(tmp_path / "dot.cpp"), "-o", str(tmp_path / "dot")], check=True)
    out = subprocess.run([str(tmp_path / "dot")], check=True, capture_output=True, text=True).stdout
    assert float(out) <= 2.0 ** -55.9
