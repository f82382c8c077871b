"""Host-side check (no GPU) of the fixed-point transforms: the arithmetic that the CUDA kernels run
(conversion from FP64, scalings, butterflies, real packing and unpacking, conversion back) is compiled
for the host from the library's own header and compared with direct sums in extended precision, next to
the same transforms in FP64.

Bars, set before the first run: every value stays inside the 64-bit words (moduli < 2^63), and the
relative 2-norm error is no larger than that of FP64 butterflies of the same radices on the same input,
or 2^-52 where those happen to be exact (a result rounded once to FP64 carries up to 2^-53 by itself)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2506_14792_gb300", "csrc")
# every radix order, lengths that are and are not multiples of 8, both ends of the real range
LENGTHS = [3, 6, 9, 12, 18, 24, 27, 48, 54, 72, 96, 108, 192, 288, 384, 432, 576, 768, 1536]
KINDS = ["flat", "smooth", "single_mode", "one_large", "inverse_k", "low_pass", "signs", "coherent"]
# signs and coherent: components just below a power of two, so that butterflies meet their largest operands

PROGRAM = r'''
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "fxfft.cuh"
using namespace spadj;
typedef std::complex<double> cd;
typedef std::complex<long double> cl;
static long double g_mod = 0;
static void see(fx2 v) { g_mod = std::max(g_mod, hypotl(v.x, v.y)); }

// the passes with the kernel's own indexing (fx_pass_list)
static std::vector<fx2> passes(std::vector<fx2> a, const FFTPlan& p, int sch) {
  const int4* tw = p.fxt;
  const int n = p.n;
  const fx2 poison{1ll << 60, 1ll << 60};
  a.resize(n, poison);
  int ps = 0;
  for (const FxPass& q : fx_pass_list(n)) {
    std::vector<fx2> b(n, poison);
    const int sg = (sch >> (2 * ps)) & 3;
    for (int j = 0; j < q.nbf; ++j) {
      const int blk = q.mNs ? (int)(((unsigned long long)j * q.mNs) >> 32) : j, k = j - blk * q.Ns;
      if (blk != j / q.Ns) std::abort();
      fx2 v[6];
      for (int r = 0; r < q.R; ++r) v[r] = a.at(j + r * q.nbf);
      if (ps == 0) {
        for (int r = 0; r < q.R; ++r) v[r] = fx_shr(v[r], sg);
      } else {
        v[0] = fx_shr(v[0], sg);
        for (int r = 1; r < q.R; ++r) v[r] = fx_cmul(v[r], tw[q.tw + (q.R - 1) * k + r - 1], sg);
      }
      if (q.R == 6) fx_out6(v);
      else if (q.R == 4) fx_out4(v[0], v[1], v[2], v[3]);
      else if (q.R == 3) fx_out3(v[0], v[1], v[2]);
      else { const fx2 t = fx_add(v[0], v[1]); v[1] = fx_sub(v[0], v[1]); v[0] = t; }
      for (int r = 0; r < q.R; ++r) { see(v[r]); b.at(blk * q.Ns * q.R + k + r * q.Ns) = v[r]; }
    }
    a = b;
    ++ps;
  }
  return a;
}
static std::vector<cd> fp64(std::vector<cd> a, const FFTPlan& p, int sign) {
  const int n = p.n;
  std::vector<cd> b(n);
  for (int ps = 0, Ns = 1; ps < p.nrad; ++ps) {
    const int R = p.rad[ps], nbf = n / R;
    for (int j = 0; j < nbf; ++j) {
      const int k = j % Ns, base = (j - k) * R + k;
      cd v[4], y[4], I(0, sign);
      for (int r = 0; r < R; ++r) {
        const long double th = sign * 2 * M_PIl * r * k / (long double)(R * Ns);
        const cd x = a[j + r * nbf], w((double)cosl(th), (double)sinl(th));
        v[r] = r == 0 || k == 0 ? x : cd(fma(x.real(), w.real(), -x.imag() * w.imag()),
                                          fma(x.real(), w.imag(), x.imag() * w.real()));
      }
      if (R == 4) {
        const cd t0 = v[0] + v[2], t1 = v[0] - v[2], t2 = v[1] + v[3], t3 = I * (v[1] - v[3]);
        y[0] = t0 + t2; y[1] = t1 + t3; y[2] = t0 - t2; y[3] = t1 - t3;
      } else if (R == 3) {
        const cd t = v[1] + v[2], m = v[0] - 0.5 * t, r = I * (0.86602540378443864676 * (v[1] - v[2]));
        y[0] = v[0] + t; y[1] = m + r; y[2] = m - r;
      } else { y[0] = v[0] + v[1]; y[1] = v[0] - v[1]; }
      for (int r = 0; r < R; ++r) b[base + r * Ns] = y[r];
    }
    Ns *= R;
    std::swap(a, b);
  }
  return a;
}
struct Scale { int emax, pre; };
static Scale scale_of(const std::vector<cd>& x) {
  unsigned mx = 0;
  for (const cd& v : x)
    for (double q : {v.real(), v.imag()}) {
      unsigned long long b;
      std::memcpy(&b, &q, 8);
      mx = std::max(mx, (unsigned)(b >> 32) & 0x7fffffffu);
    }
  Scale s{(int)(mx >> 20), 0};
  if (s.emax < 128) { s.emax = std::max(s.emax, 1) + 512; s.pre = 512; }
  return s;
}
template <int B>
static fx2 conv(cd v, Scale s) {
  if (s.pre) v = cd(v.real() * 0x1p512, v.imag() * 0x1p512);
  return fx2{fx_from_double<B>(v.real(), s.emax), fx_from_double<B>(v.imag(), s.emax)};
}
static int l1_bits(const std::vector<fx2>& a) {
  unsigned l1 = 0;
  for (const fx2& v : a) { see(v); l1 += fx_l1(v); }
  return 42 + 32 - __builtin_clz(l1);
}
static double rel(long double e, long double n) { return n > 0 ? (double)sqrtl(e / n) : (double)sqrtl(e); }

int main(int argc, char** argv) {
  const double amp = std::atof(argv[1]);  // overall scale of the inputs
  std::mt19937_64 g(7);
  std::normal_distribution<double> N;
  for (int arg = 2; arg < argc; ++arg) {
    const int n = std::atoi(argv[arg]);
    FFTPlan p = make_plan(n);
    const std::vector<double2> tab = fft_tables(p, false);
    fft_bind(p, false, tab.data(), nullptr);
    FFTPlan pr = make_plan(n);
    std::vector<double2> tabr;
    if (fx_has_plan(n, true)) {
      tabr = fft_tables(pr, true);
      fft_bind(pr, true, tabr.data(), nullptr);
    }
    const unsigned long long radw = fx_radices(n);
    std::vector<cl> W(2 * n);
    for (int i = 0; i < 2 * n; ++i) W[i] = cl(cosl(M_PIl * i / n), sinl(M_PIl * i / n));
    for (int kind = 0; kind < 8; ++kind) {
      auto env = [&](int f, int top) {
        switch (kind) {
          case 0: return 1.0;
          case 1: return 1.0 / ((1.0 + f) * (1.0 + f));
          case 2: return f == top / 2 ? 1.0 : 0.0;
          case 3: return f == 1 % top ? 1.0 : 1e-6;
          case 4: return 1.0 / (1 + f);
          default: return f > top / 3 ? 0.0 : 1.0;
        }
      };
      auto full = [&](int i, int f) {  // entry i of the last two kinds, mode f
        const double s = 1.999 * amp;
        if (kind == 6) return cd(g() & 1 ? s : -s, g() & 1 ? s : -s);
        return cd(s * (double)(W[2ll * i * f % (2 * n)].real()), s * (double)(W[2ll * i * f % (2 * n)].imag()));
      };
      g_mod = 0;
      double e[3] = {0, 0, 0}, d[3] = {0, 0, 0};  // complex, inverse real, forward real: fixed point and FP64
      for (int rep = 0; rep < 3; ++rep) {
        std::vector<cd> x(n);
        for (int i = 0; i < n; ++i) x[i] = kind < 6 ? cd(N(g), N(g)) * (env(std::min(i, n - i), n / 2 + 1) * amp) : full(i, n / 3 + rep);
        for (int sign : {-1, 1}) {
          const Scale s = scale_of(x);
          std::vector<fx2> a(n);
          for (int i = 0; i < n; ++i) a[i] = conv<kFxB>(x[i], s);
          const int sch = fx_schedule(radw, kFxComplex, l1_bits(a)), se = s.emax + 1 - 1023 - kFxB + (sch >> 24) - s.pre;
          if (sign > 0) for (fx2& v : a) v = fx_swap(v);
          std::vector<fx2> r = passes(a, p, sch);
          if (sign > 0) for (fx2& v : r) v = fx_swap(v);
          const std::vector<cd> f = fp64(x, p, sign);
          long double e1 = 0, e2 = 0, nn = 0;
          for (int k = 0; k < n; ++k) {
            cl t = 0;
            for (int i = 0; i < n; ++i) {
              cl w = W[(2ll * i * k) % (2 * n)];
              if (sign < 0) w = conj(w);
              t += cl(x[i].real(), x[i].imag()) * w;
            }
            e1 += norm(cl(fx_to_double(r[k].x, se), fx_to_double(r[k].y, se)) - t);
            e2 += norm(cl(f[k].real(), f[k].imag()) - t);
            nn += norm(t);
          }
          e[0] = std::max(e[0], rel(e1, nn));
          d[0] = std::max(d[0], rel(e2, nn));
        }
        if (!fx_has_plan(n, true)) continue;
        const unsigned long long radr = fx_radices(n);
        // inverse real transform of K coefficients, then the forward one of its grid
        const int K = std::max(1, 2 * n / 3);
        std::vector<cd> c(K), A(n);
        for (int k = 0; k < K; ++k) c[k] = kind < 6 ? cd(N(g), k ? N(g) : 0.0) * (env(k, K) * amp) : full(k, n / 3 + rep);
        c[0].imag(0.0);
        Scale s = scale_of(c);
        std::vector<fx2> q(n + 1, fx2{0, 0}), a(n);
        for (int k = 0; k < K; ++k) q[k] = conv<kFxBReal>(c[k], s);
        for (int k = 0; k <= n / 2; ++k) {
          fx2 z0, z1;
          fx_pack(q[k], k ? q[n - k] : fx2{0, 0}, pr.fxr[k], z0, z1);
          a[k] = z0;
          if (k && n - k != k) a[n - k] = z1;
        }
        for (fx2& v : a) v = fx_swap(v);
        int sch = fx_schedule(radr, kFxInvReal, l1_bits(a)), se = s.emax + 1 - 1023 - kFxBReal + (sch >> 24) - s.pre;
        std::vector<fx2> r = passes(a, pr, sch);
        for (fx2& v : r) v = fx_swap(v);
        for (int k = 0; k < n; ++k) {
          const cd xk = k < K ? c[k] : cd(0), xc = k && n - k < K ? conj(c[n - k]) : cd(0);
          A[k] = xk + xc + cd(0, 1) * (xk - xc) * cd((double)W[k].real(), (double)W[k].imag());
        }
        std::vector<cd> f = fp64(A, p, 1);
        long double e1 = 0, e2 = 0, nn = 0;
        std::vector<cd> G(n);
        for (int j = 0; j < 2 * n; ++j) {
          long double t = c[0].real();
          for (int k = 1; k < K; ++k) {
            const cl w = W[((long long)j * k) % (2 * n)];
            t += 2 * (c[k].real() * w.real() - c[k].imag() * w.imag());
          }
          const double u = fx_to_double(j & 1 ? r[j / 2].y : r[j / 2].x, se), v = j & 1 ? f[j / 2].imag() : f[j / 2].real();
          if (j & 1) G[j / 2].imag((double)t); else G[j / 2].real((double)t);
          e1 += (u - t) * (u - t);
          e2 += (v - t) * (v - t);
          nn += t * t;
        }
        e[1] = std::max(e[1], rel(e1, nn));
        d[1] = std::max(d[1], rel(e2, nn));
        s = scale_of(G);
        a.resize(n);
        for (int j = 0; j < n; ++j) a[j] = conv<kFxB>(G[j], s);
        sch = fx_schedule(radr, kFxFwdReal, l1_bits(a));
        const int us = (sch >> 16) & 3;
        se = s.emax + 1 - 1023 - kFxB + (sch >> 24) - s.pre;
        r = passes(a, pr, sch);
        f = fp64(G, p, -1);
        e1 = e2 = nn = 0;
        for (int k = 0; k < K; ++k) {
          cl t = 0;
          for (int j = 0; j < 2 * n; ++j) t += (long double)(j & 1 ? G[j / 2].imag() : G[j / 2].real()) * conj(W[((long long)j * k) % (2 * n)]);
          const fx2 h = fx_unpack(r[k], r[k ? n - k : 0], pr.fxr[k], us);
          const cd zk = f[k], zc = conj(f[k ? n - k : 0]), w((double)W[k].real(), -(double)W[k].imag());
          const cd v = 0.5 * ((zk + zc) - cd(0, 1) * w * (zk - zc));
          e1 += norm(cl(fx_to_double(h.x, se + us - 1), fx_to_double(h.y, se + us - 1)) - t);
          e2 += norm(cl(v.real(), v.imag()) - t);
          nn += norm(t);
        }
        e[2] = std::max(e[2], rel(e1, nn));
        d[2] = std::max(d[2], rel(e2, nn));
      }
      std::printf("%d %d %g %g %g %g %g %g %g\n", n, kind, e[0], d[0], e[1], d[1], e[2], d[2],
                  g_mod > 0 ? (double)log2l(g_mod) : 0.0);
    }
  }
  return 0;
}
'''

CONVERT = r'''
#include <cstdio>
#include "fxfft.cuh"
using namespace spadj;
int main() {
  // one value alone in its sequence: to fixed point and back is exact
  for (double v : {1.0, -1.0, 0.0, 1e300, -3.5e-300, 4.9406564584124654e-324, 2.2250738585072014e-308, 1.7976931348623157e308, 0.1}) {
    unsigned long long b;
    std::memcpy(&b, &v, 8);
    int e = (int)(b >> 52) & 0x7ff, pre = 0;
    double w = v;
    if (e < 128) { w = v * 0x1p512; e = (e > 1 ? e : 1) + 512; pre = 512; }
    const double r59 = fx_to_double(fx_from_double<59>(w, e), e + 1 - 1023 - 59 - pre);
    const double r58 = fx_to_double(fx_from_double<58>(w, e), e + 1 - 1023 - 58 - pre);
    std::printf("%a %a %a\n", v, r59, r58);
  }
  // overflow, and a sequence marked as non-finite
  std::printf("%a %a %d\n", fx_to_double(1ll << 62, 1000), fx_to_double(-(1ll << 62), 1000), (int)std::isnan(fx_to_double(0, kFxNaN)));
  return 0;
}
'''


def _build(tmp, name, text):
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc not available")
    src = tmp / (name + ".cu")
    src.write_text(text)
    exe = tmp / name
    subprocess.run(["nvcc", "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-o", str(exe), str(src)],
                   check=True, capture_output=True)
    return str(exe)


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    return _build(tmp_path_factory.mktemp("fx_fft"), "fx", PROGRAM)


@pytest.mark.parametrize("amp", ["1.0", "1e-300", "1e290"])
def test_no_less_exact_than_fp64_and_inside_the_words(program, amp):
    out = subprocess.run([program, amp] + [str(n) for n in LENGTHS], check=True, capture_output=True, text=True).stdout
    rows = [[float(v) for v in line.split()] for line in out.strip().splitlines()]
    assert len(rows) == len(LENGTHS) * len(KINDS)
    bar = 2.0 ** -52
    for n, kind, ce, cd, ie, id_, fe, fd, mod in rows:
        where = (int(n), KINDS[int(kind)], amp)
        assert mod < 62.95, where
        assert ce <= max(cd, bar) and ie <= max(id_, bar) and fe <= max(fd, bar), (where, ce, cd, ie, id_, fe, fd)


def test_conversions_at_the_ends_of_the_range(tmp_path):
    exe = _build(tmp_path, "conv", CONVERT)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.strip().splitlines()
    for line in lines[:-1]:
        v, a, b = (float.fromhex(x) for x in line.split())
        assert a == v and b == v, line
    hi, lo, nan = lines[-1].split()
    assert float(hi) == float("inf") and float(lo) == float("-inf") and nan == "1"
