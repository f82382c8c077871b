"""Host-side check (no GPU) of every single row of the z transforms' fixed-point products, with their third limbs: the
tables and arithmetic of the CUDA kernel, compiled for the host from its own header, against extended sums.

Bar, set before the first run.  A product's limbs leave out less than 2^-84 of the largest scaled entry, and so does a staged
entry's last limb; the sum of K of them is rounded to FP64 once.  So a row's error is at most 2^-53 of its value plus
(2 K + 16) 2^-84 of the largest scaled entry (the extended sum's own error, K 2^-63 of sum |a||x|, is added to the bar).
For columns like those of resolved fields (flat, decaying like 1/n^2 or geometrically from either end) that is at most
2^-52.5 of the row's own sum |a||x|, also in the derivative's rows far below their columns' largest entries."""
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
      const int* wt = reinterpret_cast<const int*>(t.data() + z_tail_offset(r, c));
      if (z_tail_offset(r, c) + z_limb_entries(r, c) / 2 != t.size()) std::abort();
      for (int kind = 0; kind < 8; ++kind) {
        double worst = 0, rel = 0, rel64 = 0;
        for (int rep = 0; rep < 8; ++rep) {
          std::vector<double> x(c);
          int emax = -4096;
          double big = 0;
          for (int k = 0; k < c; ++k) {
            const int b = c - 1 - k;
            x[k] = q(g) * (kind == 1 ? 1 / ((1.0 + k) * (1 + k)) : kind == 2 ? std::exp(-0.4 * k) : kind == 3 ? std::exp(-0.4 * b)
                           : kind == 4 ? std::exp(-12.0 * (k % 5)) : kind == 5 ? 1e-300 * (k % 3 ? 1.0 : 1e-18) : kind == 6 ? 1e290 : 1.0);
            if (kind == 7 && k != (rep * 7) % c) x[k] *= 1e-9;  // one column alone, the others far below
            unsigned long long bits;
            std::memcpy(&bits, &x[k], 8);
            if (bits << 1) emax = std::max(emax, std::max((int)(bits >> 52) & 0x7ff, 1) + ex[k]);
            big = std::max(big, std::fabs(x[k]) * std::ldexp(1.0, ex[k]));
          }
          for (int i = 0; i < r; ++i) {
            ZAcc3 s[4];
            double h[2] = {0, 0};
            long double T = 0, S = 0;
            for (int k = 0; k < c; ++k) {
              const int hf = k >= c / 2;
              const size_t at = 2 * ((size_t)(k - hf * (c / 2)) * r + i) + hf;
              const ZLimb z = z_limbs(z_fixed(x[k], ex[k], emax));
              s[2 * hf + (expand ? k & 1 : 0)].add(z.h, z.l, z_tail(x[k], ex[k], emax), w[at], wt[at]);
              h[k & 1] = std::fma(A[(size_t)i * c + k], x[k], h[k & 1]);
              T += (long double)A[(size_t)i * c + k] * x[k];
              S += fabsl((long double)A[(size_t)i * c + k] * x[k]);
            }
            const ZWide E = z_half(s[0].wide(), s[2].wide()), O = z_half(s[1].wide(), s[3].wide());
            const double F = expand ? z_to_double(z_half(E, O), emax + 2 - 1079) : z_to_double(E, emax + 1 - 1079);
            const long double bar = ldexpl(fabsl(T), -53) + (2.0 * c + 16) * ldexpl(big, -84) + c * ldexpl(S, -63) + 0x1p-1074L;
            worst = std::max(worst, (double)(fabsl(F - T) / bar));
            if (S > 0x1p-960L) {
              rel = std::max(rel, (double)(fabsl(F - T) / S));
              rel64 = std::max(rel64, (double)(fabsl(h[0] + h[1] - T) / S));
            }
            // the mirrored grid row of an expansion: E - O
            if (expand) {
              long double Tm = 0;
              for (int k = 0; k < c; ++k) Tm += (k & 1 ? -1 : 1) * (long double)A[(size_t)i * c + k] * x[k];
              const double Fm = z_to_double(z_half(E, z_neg(O)), emax + 2 - 1079);
              const long double bm = ldexpl(fabsl(Tm), -53) + (2.0 * c + 16) * ldexpl(big, -84) + c * ldexpl(S, -63) + 0x1p-1074L;
              worst = std::max(worst, (double)(fabsl(Fm - Tm) / bm));
            }
          }
        }
        std::printf("%d %d %d %g %g %g\n", N, mat, kind, worst, rel, rel64);
      }
    }
  }
  return 0;
}
'''


def test_every_row_against_extended_sums(tmp_path):
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc not available")
    src = tmp_path / "z.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "z")
    subprocess.run(["nvcc", "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-o", exe, str(src),
                    os.path.join(CSRC, "rb_setup.cpp")], check=True, capture_output=True)
    sizes = [8, 12, 16, 20, 40, 64, 96, 128]
    out = subprocess.run([exe] + [str(n) for n in sizes], check=True, capture_output=True, text=True).stdout
    rows = [[float(v) for v in line.split()] for line in out.strip().splitlines()]
    assert len(rows) == len(sizes) * 48
    for N, mat, kind, worst, rel, rel64 in rows:
        assert worst <= 1.0, (N, mat, kind, worst)
        if kind < 4:
            assert rel <= 2.0 ** -52.5, (N, mat, kind, rel, rel64)
