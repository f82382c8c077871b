"""Host-side check (no GPU) of the eigenproblems' banded pencils: the parts they are assembled from, entry by entry against
the recombined and reordered operators written out as dense matrices, for both flows, both kinds of pencil and odd and even
N; and that building them costs no more than the operators they are built from (a problem's creation is mostly that)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2506_14792_gb300", "csrc")

PROGRAM = r'''
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "couette_setup.h"
#include "rb_setup.h"
using namespace spadj;
using namespace spadj::couhost;
typedef std::vector<double> V;

static double now() { return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count(); }

int main() {
  for (int N : {8, 9, 30})
    for (int base = 0; base < 2; ++base)
      for (int mean = 0; mean < 2; ++mean) {
        const int nv = 4 * N + 7;
        const auto o = rbhost::build_operators(N, 3 * N / 2, 1.0);
        V Um, UP;
        base_flow(o, base, Um, UP);
        // the pencil's parts, rows u, v, w, continuity, boundary values, gauge; columns u, v, w, p, tau
        std::vector<V> A(kBandParts, V((size_t)nv * nv, 0.0));
        auto at = [&](int t, int r, int c) -> double& { return A[t][(size_t)r * nv + c]; };
        for (int r = 0; r < N; ++r)
          for (int c = 0; c < N; ++c) {
            const int q = r * N + c;
            for (int f = 0; f < 3; ++f) {
              at(kPartShift, f * N + r, f * N + c) = o.SS[q];
              at(kPartVisc, f * N + r, f * N + c) = -o.DD[q];
              at(kPartAlpha, f * N + r, f * N + c) = Um[q];
            }
            at(kPartConst, r, 2 * N + c) = UP[q];
            at(kPartConst, 2 * N + r, 3 * N + c) = o.SD[q];
            at(kPartConst, 3 * N + r, 2 * N + c) = o.D0[q];
            at(kPartAlpha, r, 3 * N + c) = at(kPartBeta, N + r, 3 * N + c) = o.SS[q];
            at(kPartAlpha, 3 * N + r, c) = at(kPartBeta, 3 * N + r, N + c) = o.S0[q];
          }
        for (int f = 0; f < 3; ++f) {
          at(kPartVisc, f * N + o.lift_row, 4 * N + 2 * f) = -o.lift_val;
          at(kPartConst, f * N + N - 1, 4 * N + 2 * f + 1) = 1.0;
          for (int n = 0; n < N; ++n) {
            at(kPartConst, 4 * N + 2 * f, f * N + n) = n % 2 ? -1.0 : 1.0;
            at(kPartConst, 4 * N + 2 * f + 1, f * N + n) = 1.0;
          }
        }
        at(kPartConst, 4 * N - 1, 4 * N + 4) = 1.0;
        if (mean) {
          at(kPartConst, 3 * N, 4 * N + 6) = 1.0;
          for (int n = 0; n < N; n += 2) at(kPartConst, 4 * N + 6, 3 * N + n) = 2.0 / (1.0 - (double)n * n);
        } else {
          at(kPartConst, 4 * N + 6, 4 * N + 6) = 1.0;
        }
        // columns psi_j = T_j - w T_{j+2} of the velocities (w = 1) and of the mean pencil's pressure (even j, zero mean)
        for (int t = 0; t < kBandParts; ++t)
          for (int f = 0; f < 4; ++f)
            for (int j = 0; j + 2 < N; ++j) {
              if (f == 3 && (!mean || j % 2)) continue;
              const double w = f < 3 ? 1.0 : (1.0 - (j + 2.0) * (j + 2.0)) / (1.0 - (double)j * j);
              for (int r = 0; r < nv; ++r) at(t, r, f * N + j) -= w * at(t, r, f * N + j + 2);
            }
        // order: by mode, velocities and pressure together; the gauge first (the mean pencil's gauge row last)
        std::vector<int> pr, pc;
        if (!mean) pr.push_back(4 * N + 6);
        pc.push_back(4 * N + 6);
        for (int n = 0; n < N; ++n)
          for (int f = 0; f < 4; ++f) { pr.push_back(f * N + n); pc.push_back(f * N + n); }
        for (int b = 0; b < 6; ++b) { pr.push_back(4 * N + b); pc.push_back(4 * N + b); }
        if (mean) pr.push_back(4 * N + 6);
        int kl = 0, ku = 0;
        double worst = 0.0;
        for (const BandEntry& e : band_parts(o, Um, UP, mean, kl, ku)) {
          if (e.i - e.k > kl || e.k - e.i > ku) std::abort();
          double& a = at(e.t, pr[e.i], pc[e.k]);
          worst = std::max(worst, std::fabs(a - e.v) / std::fabs(e.v));
          a = 0.0;
        }
        double left = 0.0;  // what no entry stands for
        for (const V& a : A)
          for (double v : a) left = std::max(left, std::fabs(v));
        std::printf("%d %d %d %d %d %g %g\n", N, base, mean, kl, ku, worst, left);
      }
  double ops = 1e9, parts = 1e9;
  for (int rep = 0; rep < 5; ++rep) {
    const double t0 = now();
    const auto o = rbhost::build_operators(96, 144, 1.0);
    V Um, UP;
    base_flow(o, 1, Um, UP);
    const double t1 = now();
    int kl, ku;
    for (int mean = 0; mean < 2; ++mean) if (band_parts(o, Um, UP, mean, kl, ku).empty()) std::abort();
    ops = std::min(ops, t1 - t0);
    parts = std::min(parts, now() - t1);
  }
  std::printf("%g %g\n", ops, parts);
  return 0;
}
'''


def test_parts_and_their_cost(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    src = tmp_path / "p.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "p")
    subprocess.run(["g++", "-std=c++17", "-O3", "-pthread", "-I", CSRC, "-o", exe, str(src), os.path.join(CSRC, "couette_setup.cpp"),
                    os.path.join(CSRC, "rb_setup.cpp")], check=True, capture_output=True)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.strip().splitlines()
    assert len(lines) == 13
    for line in lines[:-1]:
        worst, left = (float(v) for v in line.split()[5:])
        # one subtraction each (a contracted one differs in its last bit); the gauge row's recombined entries are a
        # rounding residue of at most 2 and are dropped
        assert worst <= 2.0 ** -50 and left <= 2.0 ** -50, line
    ops, parts = (float(v) for v in lines[-1].split())
    assert parts <= ops, (parts, ops)
