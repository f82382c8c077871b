"""Host-side check (no GPU) of the z transforms' fixed-point products: the tables and arithmetic of the CUDA kernel,
compiled for the host from its own header, against extended sums, for every matrix of the z transforms, odd and
even column counts and the largest one, with flat, decaying, graded, tiny and huge columns.

Bar, set before the first run: an entry of a column and of a matrix is rounded to 2^-57 of the largest scaled one, the
dropped products add at most 2^-58 each, and halving and the conversion to FP64 round the result: an error of at most
(2 K + 16) 2^-57 times the largest scaled entry, plus 2^-53 of the result.  The 2-norm error over columns that decay like 1/n^2,
as resolved fields do, is no larger than that of FP64 sums from N = 16 on."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2506_14792_gb300", "csrc")

PROGRAM = r'''
#include <cstdio>
#include <cstdlib>
#include <random>
#include "rb_kernels.cuh"
#include "rb_setup.h"
using namespace spadj;
using namespace spadj::rbk;
int main(int argc, char** argv) {
  std::mt19937 g(3);
  std::normal_distribution<double> q;
  for (int arg = 1; arg < argc; ++arg) {
    const int N = std::atoi(argv[arg]), Mz = 3 * N / 2, Mh = Mz / 2;
    const auto o = rbhost::build_operators(N, Mz, 1.0);
    for (int mat = 0; mat < 6; ++mat) {
      const bool expand = mat < 3;
      const int r = expand ? Mh : N, c = expand ? N : Mh;
      std::vector<double> A((size_t)r * c);
      for (int n = 0; n < N; ++n)
        for (int j = 0; j < Mh; ++j) {
          const double v = mat % 3 == 0 ? o.Cz[(size_t)j * N + n] : mat % 3 == 1 ? o.Cdz[(size_t)j * N + n] : o.Gz[(size_t)n * Mz + j];
          A[expand ? (size_t)j * N + n : (size_t)n * Mh + j] = v;
        }
      const std::vector<double> t = z_table(A, r, c);
      const int2* w = reinterpret_cast<const int2*>(t.data() + (size_t)r * c);
      const int* ex = reinterpret_cast<const int*>(t.data() + (size_t)r * c + z_limb_entries(r, c));
      for (int kind = 0; kind < 6; ++kind) {
        double worst = 0, ef = 0, ed = 0;
        for (int rep = 0; rep < 8; ++rep) {
          std::vector<double> x(c);
          int emax = -4096;
          double big = 0;
          for (int k = 0; k < c; ++k) {
            x[k] = q(g) * (kind == 1 ? 1 / ((1.0 + k) * (1 + k)) : kind == 2 ? std::exp(-0.4 * k) : kind == 3 ? std::exp(-12.0 * (k % 5)) : kind == 4 ? 1e-290 : kind == 5 ? 1e290 : 1.0);
            unsigned long long b;
            std::memcpy(&b, &x[k], 8);
            const int e = (int)(b >> 52) & 0x7ff;
            if (e) emax = std::max(emax, e + ex[k]);
            big = std::max(big, std::fabs(x[k]) * std::ldexp(1.0, ex[k]));
          }
          double nf = 0, nd = 0, nn = 0;
          for (int i = 0; i < r; ++i) {
            ZAcc s[4];
            double h[2] = {0, 0};
            long double T = 0;
            for (int k = 0; k < c; ++k) {
              const int hf = k >= c / 2;
              const ZLimb z = z_limbs(z_fixed(x[k], ex[k], emax));
              s[2 * hf + (expand ? k & 1 : 0)].add(z.h, z.l, w[2 * ((size_t)(k - hf * (c / 2)) * r + i) + hf]);
              h[k & 1] = std::fma(A[(size_t)i * c + k], x[k], h[k & 1]);
              T += (long double)A[(size_t)i * c + k] * x[k];
            }
            const long long E = z_half(s[0].sum(), s[2].sum()), O = z_half(s[1].sum(), s[3].sum());
            const double F = expand ? fx_to_double(z_half(E, O), emax + 2 - 1079) : fx_to_double(E, emax + 1 - 1079);
            const double D = h[0] + h[1];
            const double bar = (2.0 * c + 16) * std::ldexp(big, -57) + std::ldexp(std::fabs((double)T), -53);
            worst = std::max(worst, std::fabs((double)(F - T)) / bar);
            nf += (double)((F - T) / big * ((F - T) / big));
            nd += (double)((D - T) / big * ((D - T) / big));
            nn += (double)(T / big * (T / big));
          }
          ef += std::sqrt(nf / nn) / 8;
          ed += std::sqrt(nd / nn) / 8;
        }
        std::printf("%d %d %d %g %g %g\n", N, mat, kind, worst, ef, ed);
      }
    }
  }
  return 0;
}
'''


def test_products_against_extended_sums(tmp_path):
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc not available")
    src = tmp_path / "z.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "z")
    subprocess.run(["nvcc", "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-o", exe, str(src),
                    os.path.join(CSRC, "rb_setup.cpp")], check=True, capture_output=True)
    sizes = [8, 12, 16, 20, 40, 64, 128]
    out = subprocess.run([exe] + [str(n) for n in sizes], check=True, capture_output=True, text=True).stdout
    rows = [[float(v) for v in line.split()] for line in out.strip().splitlines()]
    assert len(rows) == len(sizes) * 36
    for N, mat, kind, worst, ef, ed in rows:
        assert worst <= 1.0, (N, mat, kind, worst)
        if kind == 1 and N >= 16:
            assert ef <= ed, (N, mat, ef, ed)
