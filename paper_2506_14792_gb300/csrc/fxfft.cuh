// Collocation FFTs in 64-bit block fixed point: the transforms' FP64 inputs and outputs, with the
// butterflies between them on the integer pipes.
//
// Why: this chip issues 2 FP64 multiply-adds per clock and SM against 64 32-bit integer
// multiply-adds, about 32 of their 32 x 32 + 64 bit form and 128 additions (measured: 1.6, 59, 25
// and 110 a clock; a 64-bit addition costs 1/34 of an FP64 one).  A radix-4 butterfly with three
// twiddles is 22 FP64 instructions (14 clocks per thread and SM) or 36 wide multiply-adds and
// about 70 additions and shifts (2 clocks).
//
// Format.  One sequence of the transform shares one exponent: its largest input component, of
// biased exponent emax, is placed below 2^B (B = 59; 58 for the packed real spectra), and every value is a
// signed 64-bit integer from there on.  Twiddles are fixed point too (2^-61 resolution).  A product
// keeps the top 64 bits of the 128: with
//   x 2^-sg = 2^29 xh + xl / 8,   w = 2^-29 wh + 2^-61 wl     (signed 32-bit xh, xl, wh, wl)
//   x w 2^-sg = xh wh + (xh wl + xl wh) 2^-32 + O(1/4)
// which is three wide multiply-adds, and the cross products' high word is taken by register, not by a
// shift; sg in 0..3 is a free scaling by 2^-sg (it only moves the split).
//
// Overflow.  A product's scaled operand has a complex modulus <= 2^60 (then the sums of four products stay
// below 2^63), so a pass of radix R <= 4 leaves moduli <= 2^62, and the differences that radix 3 multiplies by
// sqrt(3)/2 stay below 2^62 (split at bit 31 there).  A pass multiplies the bound of the moduli by at most R,
// and no value ever exceeds the sum of the moduli of the pass-0 inputs times the scalings so far.  Each pass
// scales by the smallest 2^-sg that brings the smaller of the two bounds to 2^60: a peaked input (one mode, a
// smooth spectrum) is hardly scaled at all, a flat one by 2^-2 per radix-4 pass.
//
// Accuracy.  The rounding is about 0.7 units of 2^-59 of the largest value in each pass, against 2^-53 of each
// value in FP64, and the results are rounded to FP64 once: the relative 2-norm error of complex transforms
// (n = 3..1536; flat, smooth, single-mode, 1/k, low-pass and alternating inputs at scales 1e-300, 1 and 1e290) is at most
// 1.5e-16 against 3.3e-16 of FP64 butterflies, and that of the real ones up to 2 x 768 points at most 1.7e-16 against
// 3.3e-16; a single mode, where FP64 happens to be nearly exact, can be up to 8 % above it at 8e-17.  Longer real transforms
// (peaked spectra: 2.0e-16 against 2.0e-16) stay with the FP64 butterflies of fft.cuh.  Every output is a sum of all
// inputs with factors of modulus 1, so what counts is the error against the sequence's largest entries: entries 2^-6 and
// more below the largest are held with fewer than 53 bits, and below 2^-59 of it they vanish, as they all but do in an FP64
// sum with it.  Non-finite input gives NaN in every output of the sequence; sequences below 2^-895 are scaled up by
// 2^512 first, so subnormals keep their bits.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "fft.cuh"

namespace spadj {

constexpr int kFxMaxN = 2048;      // longest complex transform: 32-bit index and sum ranges
constexpr int kFxMaxReal = 768;    // longest packed real transform (2 x 768 grid points)
constexpr int kFxB = 59, kFxBReal = 58;  // log2 of the bound on the converted inputs' components
constexpr int kFxSeqMax = 8;       // sequences of one call
constexpr int kFxWarpsMax = 8;     // warps of a CTA that calls the transforms
constexpr int kFxNaN = 1 << 20;    // scale exponent of a sequence with non-finite input

struct alignas(16) fx2 {
  long long x, y;
};
struct FxLimb {
  int h, l;
};

// The 16-byte accesses of the kernels that run the fixed-point transforms are written out one by one (here and at
// fx_get / fx_put), each of exactly its own width.  A precaution: builds of Burgers' single calls in this form
// raised a misaligned-address error whose cause was not found (those calls run the FP64 butterflies).
__device__ __forceinline__ double2 ldg128(const double2* p) {
  double2 v;
  asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ void stg128(double2* p, double2 v) {
  asm volatile("st.global.v2.f64 [%0], {%1, %2};" ::"l"(p), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ double2 ldcg128(const double2* p) {  // from L2: written by other CTAs of the same launch
  double2 v;
  asm volatile("ld.global.cg.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ int4 ldtab(const int4* p) {  // read-only tables
  int4 v;
  asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// ---- arithmetic (host and device: the host side is the CPU check of the same code) ----------------

__host__ __device__ __forceinline__ FxLimb fx_split(long long v, int sg) {
  const unsigned lo = (unsigned)v, hi = (unsigned)(v >> 32);
  FxLimb r;
  r.l = (int)(lo << (3 - sg));
#ifdef __CUDA_ARCH__
  r.h = (int)(__funnelshift_rc(lo, hi, 29 + sg) + ((unsigned)r.l >> 31));
#else
  r.h = (int)((unsigned)(((unsigned long long)hi << 32 | lo) >> (29 + sg)) + ((unsigned)r.l >> 31));
#endif
  return r;
}
__host__ __device__ __forceinline__ long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }
// high word of a cross-product sum, sign-extended
__host__ __device__ __forceinline__ long long fx_hi(long long c) { return (long long)(int)(c >> 32); }
constexpr long long kFxRound = 1ll << 31;

// v w 2^-sg, w = (re.h, re.l, im.h, im.l)
__host__ __device__ __forceinline__ fx2 fx_cmul(fx2 v, int4 w, int sg) {
  const FxLimb a = fx_split(v.x, sg), b = fx_split(v.y, sg);
  const int nh = -w.z, nl = -w.w;
  const long long cr = fx_mad(b.h, nl, fx_mad(b.l, nh, fx_mad(a.h, w.y, fx_mad(a.l, w.x, kFxRound))));
  const long long ci = fx_mad(b.h, w.y, fx_mad(b.l, w.x, fx_mad(a.h, w.w, fx_mad(a.l, w.z, kFxRound))));
  fx2 r;
  r.x = fx_mad(a.h, w.x, fx_mad(b.h, nh, fx_hi(cr)));
  r.y = fx_mad(a.h, w.z, fx_mad(b.h, w.x, fx_hi(ci)));
  return r;
}
// v c for a real constant c = 2^-31 ch + 2^-63 cl, |v| < 2^62
__host__ __device__ __forceinline__ long long fx_rmul(long long v, int ch, int cl) {
  const FxLimb a = fx_split(v, 2);  // v = 2^31 h + l / 2
  return fx_mad(a.h, ch, fx_hi(fx_mad(a.h, cl, fx_mad(a.l, ch, kFxRound))));
}
__host__ __device__ __forceinline__ fx2 fx_add(fx2 a, fx2 b) { return fx2{a.x + b.x, a.y + b.y}; }
__host__ __device__ __forceinline__ fx2 fx_sub(fx2 a, fx2 b) { return fx2{a.x - b.x, a.y - b.y}; }
__host__ __device__ __forceinline__ fx2 fx_shr(fx2 a, int sg) { return fx2{a.x >> sg, a.y >> sg}; }
__host__ __device__ __forceinline__ fx2 fx_swap(fx2 a) { return fx2{a.y, a.x}; }

// Forward (exp(-)) butterflies in place, outputs in order.  Inverse transforms run the forward passes on swapped
// components: IDFT(x) = swap(DFT(swap(x))).
__host__ __device__ __forceinline__ void fx_out4(fx2& v0, fx2& v1, fx2& v2, fx2& v3) {
  const fx2 t0 = fx_add(v0, v2), t1 = fx_sub(v0, v2), t2 = fx_add(v1, v3), t3 = fx_sub(v1, v3);
  v0 = fx_add(t0, t2);
  v2 = fx_sub(t0, t2);
  v1 = fx2{t1.x + t3.y, t1.y - t3.x};  // t1 -+ i t3
  v3 = fx2{t1.x - t3.y, t1.y + t3.x};
}
constexpr int kFxS3h = 1859775393, kFxS3l = 1630710223;  // sqrt(3)/2 = 2^-31 h + 2^-63 l
__host__ __device__ __forceinline__ void fx_out3(fx2& v0, fx2& v1, fx2& v2) {
  const fx2 t = fx_add(v1, v2), d = fx_sub(v1, v2);
  const fx2 m = fx_sub(v0, fx_shr(t, 1));
  const fx2 r = fx2{fx_rmul(d.y, kFxS3h, kFxS3l), -fx_rmul(d.x, kFxS3h, kFxS3l)};  // -i (sqrt3/2) d
  v0 = fx_add(v0, t);
  v1 = fx_add(m, r);
  v2 = fx_sub(m, r);
}
// Radix 6 as 2 x 3 (prime factors: no twiddles)
__host__ __device__ __forceinline__ void fx_out6(fx2 (&v)[6]) {
  fx2 a0 = v[0], a1 = v[2], a2 = v[4], b0 = v[3], b1 = v[5], b2 = v[1];
  fx_out3(a0, a1, a2);
  fx_out3(b0, b1, b2);
  v[0] = fx_add(a0, b0);
  v[3] = fx_sub(a0, b0);
  v[4] = fx_add(a1, b1);
  v[1] = fx_sub(a1, b1);
  v[2] = fx_add(a2, b2);
  v[5] = fx_sub(a2, b2);
}

// Fixed-point value of the double x: x = v 2^(emax + 1 - 1023 - B) to the last unit (toward zero; to the nearest for
// the packed real spectra, whose many small entries would add up otherwise), |v| <= 2^B for biased exponents <= emax.  emax >= 128, so that whatever has a zero exponent field vanishes.
template <int B>
__host__ __device__ __forceinline__ long long fx_from_double(double x, int emax) {
#ifdef __CUDA_ARCH__
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
#else
  unsigned long long bits;
  std::memcpy(&bits, &x, 8);
  const unsigned hi = (unsigned)(bits >> 32), lo = (unsigned)bits;
#endif
  const int d = emax - (int)((hi >> 20) & 0x7ff);
  constexpr int kUp = B - 53 + (B == kFxBReal ? 1 : 0);
  const unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 | lo) << kUp;
  unsigned long long v;
#ifdef __CUDA_ARCH__
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"(d));  // shifts above 63 give 0
#else
  v = d > 63 ? 0 : m >> d;
#endif
  if (B == kFxBReal) v = (v + 1) >> 1;
  const long long s = (int)hi >> 31;
  return ((long long)v ^ s) - s;
}

// v 2^se rounded to FP64; se >= kFxNaN / 2 marks a sequence with non-finite input.
__host__ __device__ inline double fx_to_double_rare(long long v, int se) {
#ifdef __CUDA_ARCH__
  if (se >= kFxNaN / 2) return __longlong_as_double(0x7ff8000000000000ll);
#else
  if (se >= kFxNaN / 2) return std::nan("");
#endif
  return ldexp((double)v, se);  // overflow and subnormal results
}
__host__ __device__ __forceinline__ double fx_to_double(long long v, int se) {
  const long long s = v >> 63;
  const unsigned long long mag = (unsigned long long)((v ^ s) - s);
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)mag);
#else
  const int lz = mag ? __builtin_clzll(mag) : 64;
#endif
  const int e = se + 1086 - lz;  // biased exponent of the leading bit
  if ((unsigned)(e - 1) >= 2046u) return fx_to_double_rare(v, se);
  const unsigned long long m = mag << (lz & 63);
  // mantissa with the implicit bit at 52, rounded half up; a carry moves into the exponent
  unsigned long long bits = (m >> 11) + ((m >> 10) & 1) + ((unsigned long long)(e - 1) << 52);
  bits = mag ? bits : 0ull;
  bits |= (unsigned long long)s & 0x8000000000000000ull;
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)bits);
#else
  double r;
  std::memcpy(&r, &bits, 8);
  return r;
#endif
}

// Entries k and n - k of the packed spectrum of a half-length real transform, from x = c_k and y = c_{n-k}
// (0 where not stored), w = exp(-i pi k / n):
//   Z_k = e + t,  Z_{n-k} = conj(e - t),  e = x + conj(y),  t = i conj(w) (x - conj(y))
__host__ __device__ __forceinline__ void fx_pack(fx2 x, fx2 y, int4 w, fx2& z0, fx2& z1) {
  w.z = -w.z;
  w.w = -w.w;
  const fx2 t = fx_cmul(fx2{-x.y - y.y, x.x - y.x}, w, 0);
  z0 = fx2{x.x + y.x + t.x, x.y - y.y + t.y};
  z1 = fx2{x.x + y.x - t.x, y.y - x.y + t.y};
}
// Twice the spectrum entry ((u + conj(v)) - i w (u - conj(v))) / 2 of a real field, scaled by 2^-us, from the
// entries u = Z_k, v = Z_{n-k} of its packed transform.
__host__ __device__ __forceinline__ fx2 fx_unpack(fx2 u, fx2 v, int4 w, int us) {
  const fx2 t = fx_cmul(fx2{u.y + v.y, v.x - u.x}, w, us);
  return fx2{((u.x + v.x) >> us) + t.x, ((u.y - v.y) >> us) + t.y};
}
__host__ __device__ __forceinline__ unsigned fx_l1(fx2 v) {  // >= (|x| + |y|) / 2^42
  const int x = (int)(v.x >> 32), y = (int)(v.y >> 32);
  return ((unsigned)(x < 0 ? -x : x) >> 10) + ((unsigned)(y < 0 ? -y : y) >> 10) + 2u;
}

// The scalings sg of the passes, two bits each from the low end, and their sum in bits 24.., for inputs whose sum of
// moduli is below 2^l.  The bounds are followed in quarters of log2.  The values of a forward real transform
// stay <= 2^61.5, and bits 16 and 17 hold the scaling of its fx_unpack.
enum { kFxComplex = 0, kFxInvReal = 1, kFxFwdReal = 2 };
inline int fx_schedule(unsigned long long radw, int kind, int l) {
  // bound of the pass-0 moduli: sqrt(2) 2^B, and 4 sqrt(2) 2^B for the packed spectra
  int bits = 0, tot = 0, b = kind == kFxInvReal ? 4 * kFxBReal + 10 : 4 * kFxB + 2;
  l *= 4;
  for (int i = 0; radw; ++i, radw >>= 8) {
    const int R = (int)(radw & 0xff), grow = R == 6 ? 11 : R == 4 ? 8 : R == 3 ? 7 : 4;
    int lim = 240;  // of a scaled operand: the sums of four products fit the words
    if (kind == kFxFwdReal && lim > 246 - grow) lim = 246 - grow;
    // pass 0 has no products: only its results have to fit (six times a packed real spectrum's bound may not)
    const int sg = i > 0 ? (b > lim ? (b - lim + 3) / 4 : 0) : (b + grow < l ? b + grow : l) > 251 ? 1 : 0;
    bits |= sg << (2 * i);
    tot += sg;
    l -= 4 * sg;
    b += grow - 4 * sg;
    if (b > l) b = l;
  }
  if (kind == kFxFwdReal && b + 4 > 240) bits |= ((b + 4 - 240 + 3) / 4) << 16;
  return bits | tot << 24;
}

// ---- tables (host) ---------------------------------------------------------------------------------

inline void fx_const(long double w, int* h, int* l) {
  const long long W = llroundl(w * 2305843009213693952.0L);  // 2^61
  const long long hh = (W + (1ll << 31)) >> 32;
  long long ll = W - (hh << 32);
  if (ll == -(1ll << 31)) ll += 1;  // its negative stays a 32-bit number
  *h = (int)hh;
  *l = (int)ll;
}
// exp(i pi j / n), j < 2n, from the cosines and sines of the first octant (4 | n; else all of them)
inline std::vector<int4> fx_roots(int n) {
  std::vector<int4> r(2 * n);
  const long double pi = 3.14159265358979323846264338327950288L;
  auto at = [&](int j) {
    int4 w;
    fx_const(cosl(pi * j / n), &w.x, &w.y);
    fx_const(sinl(pi * j / n), &w.z, &w.w);
    return w;
  };
  if (n % 4 != 0) {
    for (int j = 0; j < 2 * n; ++j) r[j] = at(j);
    return r;
  }
  for (int j = 0; j <= n / 4; ++j) r[j] = at(j);
  for (int j = n / 4 + 1; j <= n / 2; ++j) {  // mirrored at 45 degrees
    const int4 a = r[n / 2 - j];
    r[j] = make_int4(a.z, a.w, a.x, a.y);
  }
  for (int j = n / 2 + 1; j < 2 * n; ++j) {  // quarter turns
    const int4 a = r[j - n / 2];
    r[j] = make_int4(-a.z, -a.w, a.x, a.y);
  }
  return r;
}
// Radices of the fixed-point passes, a byte each from the low end: a 6 (when the power of 2 is odd) or a 3 first,
// without twiddles and with the least growth of the moduli, which the packed real spectra need; then the other 3s,
// then 4s.  Radix 8 in place of the 4s needs fewer passes but leaves half the lanes idle at these lengths (24
// butterflies at n = 192): 16384 Burgers members of N = 256 take 18.9 ms with it and 17.8 ms without.  0: no such
// plan (n without a factor 3, or above kFxMaxN).
inline unsigned long long fx_radices(int n) {
  if (n < 3 || n > kFxMaxN) return 0;
  unsigned long long w = 0;
  int m = n, i = 0;
  auto push = [&](int r) {
    w |= (unsigned long long)r << (8 * i++);
    m /= r;
  };
  if (m % 3 != 0) return 0;
  int two = 0;
  for (int q = m; q % 2 == 0; q /= 2) ++two;
  if (two % 2 == 1 && n != 6) push(6);
  while (m % 3 == 0 && i < 8) push(3);
  while (m % 4 == 0 && i < 8) push(4);
  if (m % 2 == 0 && i < 8) push(2);  // n = 6: a single pass would leave too large values to unpack
  return m == 1 ? w : 0;
}
// One pass: butterfly j = q Ns + k of nbf reads entries j + r nbf of its input and writes q Ns R + k + r Ns;
// mNs: 2^32 / Ns rounded up (division by multiplication); tw: offset of its twiddles.
struct alignas(16) FxPass {
  int R, Ns, nbf, tw;
  unsigned mNs;
  int more;  // whether another pass follows
};
inline std::vector<FxPass> fx_pass_list(int n) {
  std::vector<FxPass> v;
  int Ns = 1, tw = 0;
  for (unsigned long long w = fx_radices(n); w; w >>= 8) {
    FxPass p{};
    p.R = (int)(w & 0xff);
    p.Ns = Ns;
    p.nbf = n / p.R;
    p.more = (w >> 8) != 0;
    p.mNs = Ns > 1 ? (unsigned)(((1ull << 32) + Ns - 1) / Ns) : 0u;
    p.tw = tw;
    if (Ns > 1) tw += Ns * (p.R - 1);
    Ns *= p.R;
    v.push_back(p);
  }
  return v;
}
// Tables of a plan, as 16-byte entries: the passes, exp(-) twiddles in pass order (R - 1 per k), exp(-pi i k / n),
// k < n (the real transforms' unpacking), the scalings of the passes by the leading zeros of the sum of
// the moduli (fx_schedule; 32 words for each kind of transform), and the FP64 records where needed.
// real: the plan is that of packed real transforms; both: the FP64 records in any case.
inline bool fx_has_plan(int n, bool real) { return !(real && n > kFxMaxReal) && fx_radices(n) != 0; }
inline std::vector<double2> fft_tables(const FFTPlan& p, bool real, bool both = false) {
  std::vector<int4> t;
  if (fx_has_plan(p.n, real)) {
    const unsigned long long radw = fx_radices(p.n);
    const std::vector<FxPass> ps = fx_pass_list(p.n);
    t.resize(ps.size() * (sizeof(FxPass) / sizeof(int4)));
    std::memcpy(t.data(), ps.data(), sizeof(FxPass) * ps.size());
    const std::vector<int4> root = fx_roots(p.n);
    const int period = 2 * p.n;
    for (const FxPass& q : ps)
      if (q.Ns > 1)
        for (int k = 0; k < q.Ns; ++k)
          for (int m = 1; m < q.R; ++m) t.push_back(root[(period - m * k * (period / (q.R * q.Ns)) % period) % period]);
    for (int k = 0; k < p.n; ++k) t.push_back(root[(period - k) % period]);
    for (int kind : {kFxComplex, kFxInvReal, kFxFwdReal})
      for (int z = 0; z < 32; z += 4) {
        int s[4];
        for (int q = 0; q < 4; ++q) s[q] = fx_schedule(radw, kind, 42 + 32 - (z + q));
        t.push_back(make_int4(s[0], s[1], s[2], s[3]));
      }
  }
  std::vector<double2> out(t.size());
  if (!t.empty()) std::memcpy(out.data(), t.data(), sizeof(int4) * t.size());
  if (both || !fx_has_plan(p.n, real)) {
    const std::vector<double2> s = scaled_twiddle_table(p);
    out.insert(out.end(), s.begin(), s.end());
  }
  return out;
}
// The plan's pointers into the device copy of its tables; wm: device table of exp(-2 pi i m / 2n), m < 2n (the FP64
// real transforms').
inline void fft_bind(FFTPlan& p, bool real, const double2* dev, const double2* wm, bool both = false) {
  p.fxp = nullptr;
  if (fx_has_plan(p.n, real)) {
    const std::vector<FxPass> ps = fx_pass_list(p.n);
    int tw = 0;
    for (const FxPass& q : ps) tw += q.Ns > 1 ? q.Ns * (q.R - 1) : 0;
    const int np = (int)(ps.size() * (sizeof(FxPass) / sizeof(int4)));
    const int4* t = reinterpret_cast<const int4*>(dev);
    p.fxp = t;
    p.fxt = t + np;
    p.fxr = p.fxt + tw;
    p.fxs = reinterpret_cast<const int*>(p.fxr + p.n);
    p.fxodd = (int)ps.size() & 1;
    p.fxr0 = ps[0].R;
    if (both) bind_scaled_twiddles(p, dev + np + tw + p.n + 3 * 32 / 4);
  } else {
    bind_scaled_twiddles(p, dev);
  }
  p.wm = wm;
}

// ---- device: the transform of the sequences of one CTA ------------------------------------------------
//
// Buffers are offsets (in 16-byte entries) into the CTA's dynamic shared memory.  Sequence s of a call holds its
// entries from a + s * stride (and the other buffer from b + s * stride); every buffer has n entries.  All
// threads of the CTA (a multiple of 32, <= 256, divisible by the call's sequences: 1, 2, 4 or 8) call.

__device__ __forceinline__ double2* fx_mem64() {
  extern __shared__ double2 fx_dyn[];
  return fx_dyn;
}
// One 16-byte shared-memory access each, to entry e of the buffers.
__device__ __forceinline__ unsigned fx_addr(int e) {
  return static_cast<unsigned>(__cvta_generic_to_shared(fx_mem64())) + 16u * (unsigned)e;
}
__device__ __forceinline__ fx2 fx_get(int e) {
  fx2 v;
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(fx_addr(e)) : "memory");
  return v;
}
__device__ __forceinline__ void fx_put(int e, fx2 v) {
  asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(fx_addr(e)), "l"(v.x), "l"(v.y) : "memory");
}
__device__ __forceinline__ double2 fx_get64(int e) {
  double2 v;
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(fx_addr(e)) : "memory");
  return v;
}
__device__ __forceinline__ void fx_put64(int e, double2 v) {
  asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(fx_addr(e)), "d"(v.x), "d"(v.y) : "memory");
}

// Per-warp slots: every warp reduces over its own entries, and all warps combine the slots after the
// barrier that the data needs anyway.
struct alignas(16) FxShared {
  unsigned mx[kFxWarpsMax][kFxSeqMax];  // largest |high word| of the sequence's components
  unsigned l1[kFxWarpsMax][kFxSeqMax];  // sum of the moduli, in units of 2^42
  unsigned se[kFxWarpsMax][kFxSeqMax];  // scale exponent of the results and scalings of the passes (each
  unsigned sch[kFxWarpsMax][kFxSeqMax]; // warp's copy)
};
__device__ __forceinline__ FxShared& fx_shared() {
  __shared__ FxShared s;
  return s;
}
__device__ __forceinline__ unsigned lds32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(static_cast<unsigned>(__cvta_generic_to_shared(p))) : "memory");
  return v;
}
__device__ __forceinline__ void sts32(unsigned* p, unsigned v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(p))), "r"(v) : "memory");
}

struct FxLay {
  int ns, stride;  // sequences of the call, entries between their buffers
  int s0;          // first of the ns slots for their scales (a later call on other slots leaves the earlier
                   // results readable)
};

__device__ __forceinline__ unsigned fx_absmax(unsigned m, double2 v) {
  return max(m, max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu));
}
// The threads of a CTA share out over the NS sequences of a call: thread l of the T threads of sequence s, so that
// whatever depends on the sequence (base, scale, scalings) is computed once per thread and call.  The T
// threads are consecutive, or (W > 1: W = NS) every W-th one, for callers whose sequences are adjacent in memory.
struct FxGroup {
  int s, l, T;
};
template <int NS, int W>
__device__ __forceinline__ FxGroup fx_group() {
  const int tid = threadIdx.x, nt = blockDim.x;
  if (W > 1) return FxGroup{tid & (W - 1), tid / W, nt / W};
  if (NS == 1) return FxGroup{0, tid, nt};
  const int T = nt / NS, s = tid >> (31 - __clz(T));
  return FxGroup{s, tid - s * T, T};
}
// warps that hold threads of sequence s: first and one past the last
template <int NS, int W>
__device__ __forceinline__ int2 fx_warps(int s) {
  const int nt = blockDim.x;
  if (W > 1 || NS == 1) return make_int2(0, nt >> 5);
  const int T = nt / NS, w = (s * T) >> 5;
  return make_int2(w, max(w + 1, ((s + 1) * T) >> 5));
}
// Reductions by shuffles over the lanes of a sequence; its first lane writes the warp's value to the slot
// (v[warp][s0 + s])
template <int W>
__device__ __forceinline__ void fx_reduce_max(FxGroup g, int s0, unsigned m) {
#pragma unroll
  for (int d = 16; d >= W; d >>= 1)
    if (W > 1 || d < g.T) m = max(m, __shfl_xor_sync(0xffffffffu, m, d));
  const int lane = threadIdx.x & 31;
  if (W > 1 ? lane < W : (g.l & 31) == 0) sts32(&fx_shared().mx[threadIdx.x >> 5][s0 + g.s], m);
}
template <int W>
__device__ __forceinline__ void fx_reduce_l1(FxGroup g, int s0, unsigned v) {
#pragma unroll
  for (int d = 16; d >= W; d >>= 1)
    if (W > 1 || d < g.T) v += __shfl_xor_sync(0xffffffffu, v, d);
  const int lane = threadIdx.x & 31;
  if (W > 1 ? lane < W : (g.l & 31) == 0) sts32(&fx_shared().l1[threadIdx.x >> 5][s0 + g.s], v);
}
// The warp's largest high word of the sequence of slot s, from each thread's m (all threads call)
__device__ __forceinline__ void fx_put_max(int s, unsigned m) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, d));
  if ((threadIdx.x & 31) == 0) sts32(&fx_shared().mx[threadIdx.x >> 5][s], m);
}
__device__ __forceinline__ unsigned fx_get_max(int s, int2 warps) {
  unsigned m = 0u;
  for (int w = warps.x; w < warps.y; ++w) m = max(m, lds32(&fx_shared().mx[w][s]));
  return m;
}
struct FxExp {
  int emax;  // biased exponent of the sequence's scale, >= 128
  bool pre;  // inputs are multiplied by 2^512 first (sequences of tiny values)
};
__device__ __forceinline__ FxExp fx_exponent(unsigned mx) {
  FxExp r;
  r.emax = (int)(mx >> 20);
  r.pre = r.emax < 128;
  if (r.pre) r.emax = max(r.emax, 1) + 512;
  return r;
}
template <int B>
__device__ __forceinline__ fx2 fx_load(double2 v, FxExp e) {
  if (e.pre) {
    v.x *= 0x1p512;
    v.y *= 0x1p512;
  }
  return fx2{fx_from_double<B>(v.x, e.emax), fx_from_double<B>(v.y, e.emax)};
}

// Each warp writes its copy of the sequences' scale exponents and scalings (after a barrier that makes mx and
// l1 final): results are v 2^exponent.  sched: the plan's table for this kind of input; EVERY: all warps hold
// maxima (fx_put_max).
template <int B, int NS, int W, bool EVERY>
__device__ __forceinline__ void fx_make_meta(FxLay lay, const int* __restrict__ sched) {
  FxShared& S = fx_shared();
  const int s = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (s < NS) {
    const int2 own = fx_warps<NS, W>(s);
    unsigned l1 = 0u;
    for (int v = own.x; v < own.y; ++v) l1 += lds32(&S.l1[v][lay.s0 + s]);
    const unsigned mx = fx_get_max(lay.s0 + s, EVERY ? make_int2(0, (int)(blockDim.x >> 5)) : own);
    const int sch = __ldg(sched + __clz((int)l1));
    const FxExp e = fx_exponent(mx);
    sts32(&S.se[w][lay.s0 + s], (unsigned)(mx >= 0x7ff00000u ? kFxNaN : e.emax + 1 - 1023 - B + (sch >> 24) - (e.pre ? 512 : 0)));
    sts32(&S.sch[w][lay.s0 + s], (unsigned)sch);
  }
  __syncwarp();
}
__device__ __forceinline__ int fx_se(int s) { return (int)lds32(&fx_shared().se[threadIdx.x >> 5][s]); }
__device__ __forceinline__ int fx_sch(int s) { return (int)lds32(&fx_shared().sch[threadIdx.x >> 5][s]); }

// Pass 0 of a sequence: butterfly j of n / R takes the entries j + r n / R through get and writes R j + r from b on.
template <class Get>
__device__ __forceinline__ void fx_first(int b, FxGroup g, int n, int R, Get get) {
  if (R == 6) {
    const int m = n / 6;
#pragma unroll 1
    for (int j = g.l; j < m; j += g.T) {
      fx2 v[6];
#pragma unroll
      for (int r = 0; r < 6; ++r) v[r] = get(j + r * m);
      fx_out6(v);
#pragma unroll
      for (int r = 0; r < 6; ++r) fx_put(b + 6 * j + r, v[r]);
    }
  } else {
    const int m = n / 3;
#pragma unroll 1
    for (int j = g.l; j < m; j += g.T) {
      fx2 v0 = get(j), v1 = get(j + m), v2 = get(j + 2 * m);
      fx_out3(v0, v1, v2);
      fx_put(b + 3 * j, v0);
      fx_put(b + 3 * j + 1, v1);
      fx_put(b + 3 * j + 2, v2);
    }
  }
}
// The other passes of this thread's sequence, from the results of pass 0 in a (b: the other buffer; sch: the
// scalings); the threads meet after each.
struct FxDesc {
  int4 d0, d1;
};
__device__ __forceinline__ FxDesc fx_desc(const int4* passes) { return FxDesc{ldtab(passes), ldtab(passes + 1)}; }
// AHEAD: next holds pass 1's parameters, and those of each later pass are loaded a pass ahead too: for kernels
// that run one transform and find the tables in L2 (the Rayleigh-Benard pieces at 64 x 32 take 178 us with
// it, 192 us without); the step loops find them in L1 and need the registers (16384 Burgers members: 16.8 and 15.7 ms).
template <bool AHEAD>
__device__ __forceinline__ void fx_rest(int a, int b, FxGroup g, int sch, FxDesc next, const int4* __restrict__ passes,
                                        const int4* __restrict__ twiddles) {
  const int tid = g.l, nt = g.T;
  for (;;) {
    sch >>= 2;
    if (!AHEAD) next = fx_desc(passes);
    const int R = next.d0.x, Ns = next.d0.y, nbf = next.d0.z, more = next.d1.y, sg = sch & 3;
    const int4* tw = twiddles + next.d0.w;
    const unsigned mNs = (unsigned)next.d1.x;
    passes += 2;
    if (AHEAD && more) next = fx_desc(passes);
#pragma unroll 1
    for (int j = tid; j < nbf; j += nt) {
      const int q = (int)__umulhi((unsigned)j, mNs), k = j - q * Ns;
      const int rd = a + j, wr = b + q * Ns * R + k;
      if (R == 4) {
        fx2 v0 = fx_get(rd), v1 = fx_get(rd + nbf), v2 = fx_get(rd + 2 * nbf), v3 = fx_get(rd + 3 * nbf);
        const int4* w = tw + 3 * k;
        v0 = fx_shr(v0, sg);
        v1 = fx_cmul(v1, ldtab(w), sg);
        v2 = fx_cmul(v2, ldtab(w + 1), sg);
        v3 = fx_cmul(v3, ldtab(w + 2), sg);
        fx_out4(v0, v1, v2, v3);
        fx_put(wr, v0);
        fx_put(wr + Ns, v1);
        fx_put(wr + 2 * Ns, v2);
        fx_put(wr + 3 * Ns, v3);
      } else if (R == 3) {
        const int4* w = tw + 2 * k;
        fx2 v0 = fx_shr(fx_get(rd), sg);
        fx2 v1 = fx_cmul(fx_get(rd + nbf), ldtab(w), sg);
        fx2 v2 = fx_cmul(fx_get(rd + 2 * nbf), ldtab(w + 1), sg);
        fx_out3(v0, v1, v2);
        fx_put(wr, v0);
        fx_put(wr + Ns, v1);
        fx_put(wr + 2 * Ns, v2);
      } else {
        const fx2 v0 = fx_shr(fx_get(rd), sg), v1 = fx_cmul(fx_get(rd + nbf), ldtab(tw + k), sg);
        fx_put(wr, fx_add(v0, v1));
        fx_put(wr + Ns, fx_sub(v0, v1));
      }
    }
    __syncthreads();
    if (!more) return;
    const int t = a;
    a = b;
    b = t;
  }
}

// ---- device: transforms ----------------------------------------------------------------------------------
//
// xf_c2c, xf_c2r and xf_r2c stage their input through load(s, e) (called once per entry of each of the NS
// sequences), run the passes and return the results where FxRes reads them; what load reads must not lie in the
// buffers.  The CTA synchronises before the buffers are used again.  Lengths without a fixed-point plan run the
// FP64 butterflies; PATH kFxOnly: the caller's lengths never do, kFp64: all do.  W: see FxGroup.

enum { kFxOnly = 0, kFxAny = 1, kFp64 = 2 };

template <bool INV>
struct FxRes {
  int z;  // buffer that holds the results
  FxLay lay;
  int n;
  const int4* fxr;
  const double2* wm;
  bool fixed;  // constant true where the FP64 path is not compiled in
  __device__ __forceinline__ double2 raw64(int s, int e) const { return fx_get64(z + s * lay.stride + e); }
  // entry e of a complex transform, or grid pair (g_2e, g_2e+1) of an inverse real one
  __device__ __forceinline__ double2 at(int s, int e) const {
    if (!fixed) return raw64(s, e);
    fx2 v = fx_get(z + s * lay.stride + e);
    if (INV) v = fx_swap(v);
    const int se = fx_se(lay.s0 + s);
    return make_double2(fx_to_double(v.x, se), fx_to_double(v.y, se));
  }
  // spectrum entry X_k = sum_j g_j exp(-2 pi i j k / 2n) of a forward real transform, times 2^e (e: 0 or 1)
  __device__ __forceinline__ double2 coef(int s, int k, int e = 0) const {
    const int kc = k == 0 ? 0 : n - k;
    if (!fixed) {
      const double2 x = r2c_combine(raw64(s, k), cconj(raw64(s, kc)), __ldg(&wm[k]));
      return e ? make_double2(2.0 * x.x, 2.0 * x.y) : x;
    }
    const int q = z + s * lay.stride;
    const int us = (fx_sch(lay.s0 + s) >> 16) & 3;
    const fx2 r = fx_unpack(fx_get(q + k), fx_get(q + kc), ldtab(fxr + k), us);
    const int se = fx_se(lay.s0 + s) + us - 1 + e;
    return make_double2(fx_to_double(r.x, se), fx_to_double(r.y, se));
  }
};

// Entry k of a real field's spectrum without Im c_0, which the inverse transforms do not use: it must not take part in the
// sequence's scale either (a large one would cost the other coefficients their bits, a non-finite one the row).
__device__ __forceinline__ double2 fx_c0(int k, double2 v) { return k == 0 ? make_double2(v.x, 0.0) : v; }

// FP64 values of cnt entries of every sequence into dst, and the sequences' largest high words
template <int NS, int W, class Load>
__device__ __forceinline__ void fx_stage(int dst, FxLay lay, int cnt, Load load) {
  const FxGroup g = fx_group<NS, W>();
  const int q = dst + g.s * lay.stride;
  unsigned m = 0u;
  for (int e = g.l; e < cnt; e += g.T) {
    const double2 v = load(g.s, e);
    fx_put64(q + e, v);
    m = fx_absmax(m, v);
  }
  fx_reduce_max<W>(g, lay.s0, m);
}

// The passes after pass 0 (whose results are in b)
template <bool INV, bool AHEAD>
__device__ __forceinline__ FxRes<INV> fx_run(int a, int b, FxLay lay, FxGroup g, const FFTPlan& p, FxDesc next) {
  if (p.fxr0 != p.n)
    fx_rest<AHEAD>(b + g.s * lay.stride, a + g.s * lay.stride, g, fx_sch(lay.s0 + g.s), next, p.fxp + 2, p.fxt);
  else
    __syncthreads();  // a single pass (n = 3): a later call writes the slots that fx_make_meta reads
  return FxRes<INV>{p.fxodd ? b : a, lay, p.n, p.fxr, p.wm, true};
}
template <bool INV>
__device__ __forceinline__ FxRes<INV> fx_run64(int a, int b, FxLay lay, const FFTPlan& p) {
  cfft_smem_sets<INV ? 1 : -1>(fx_mem64() + a, fx_mem64() + b, lay.stride, lay.ns, p);
  return FxRes<INV>{(p.nrad & 1) ? b : a, lay, p.n, p.fxr, p.wm, false};
}

// xf_c2c (below) with the entries of every sequence already in a as FP64 pairs and their largest high words given
// (EVERY: by fx_put_max in all warps); the call starts with a barrier.
template <bool INV, int NS, int W = 1, int PATH = kFxAny, bool REAL = false, bool EVERY = true>
__device__ __forceinline__ FxRes<INV> xf_c2c_staged(int a, int b, FxLay lay, const FFTPlan& p) {
  __syncthreads();
  if (PATH == kFp64 || (PATH == kFxAny && !p.fxp)) return fx_run64<INV>(a, b, lay, p);
  // pass 0 converts its inputs
  const FxGroup g = fx_group<NS, W>();
  FxDesc next{};
  if (PATH == kFxAny && p.fxr0 != p.n) next = fx_desc(p.fxp + 2);
  const FxExp ex = fx_exponent(fx_get_max(lay.s0 + g.s, EVERY ? make_int2(0, (int)(blockDim.x >> 5)) : fx_warps<NS, W>(g.s)));
  const int A = a + g.s * lay.stride;
  unsigned l1 = 0u;
  fx_first(b + g.s * lay.stride, g, p.n, p.fxr0, [&](int e) {
    const fx2 v = fx_load<kFxB>(fx_get64(A + e), ex);
    l1 += fx_l1(v);
    return INV ? fx_swap(v) : v;
  });
  fx_reduce_l1<W>(g, lay.s0, l1);
  __syncthreads();
  fx_make_meta<kFxB, NS, W, EVERY>(lay, p.fxs + 32 * (REAL ? kFxFwdReal : kFxComplex));
  return fx_run<INV, PATH == kFxAny>(a, b, lay, g, p, next);
}

// Complex transform of length p.n, unnormalised: exp(-), or exp(+) for INV.  REAL: the packed grid of a forward
// real transform.
template <bool INV, int NS, int W = 1, int PATH = kFxAny, bool REAL = false, class Load>
__device__ __forceinline__ FxRes<INV> xf_c2c(int a, int b, FxLay lay, const FFTPlan& p, Load load) {
  fx_stage<NS, W>(a, lay, p.n, load);
  return xf_c2c_staged<INV, NS, W, PATH, REAL, false>(a, b, lay, p);
}

// xf_c2r (below) with the c_k of every sequence already in b as FP64 pairs and their largest high words, of c_0 the real
// part's (fx_c0), given (EVERY: by fx_put_max in all warps); the call starts with a barrier.
template <int NS, int PATH = kFxAny, bool EVERY = true>
__device__ __forceinline__ FxRes<true> xf_c2r_staged(int a, int b, FxLay lay, const FFTPlan& p, int K) {
  const int n = p.n;
  __syncthreads();
  if (PATH == kFp64 || (PATH == kFxAny && !p.fxp)) {
    for (int s = 0; s < NS; ++s) {
      const double2* S = fx_mem64() + b + s * lay.stride;
      for (int i = threadIdx.x; i < n; i += blockDim.x)
        fx_mem64()[a + s * lay.stride + i] = c2r_entry<true>([&](int k) { return S[k]; }, i, K, n, p.wm, 1.0, 1.0);
    }
    __syncthreads();
    return fx_run64<true>(a, b, lay, p);
  }
  const FxGroup g = fx_group<NS, 1>();
  FxDesc next{};
  if (PATH == kFxAny && p.fxr0 != p.n) next = fx_desc(p.fxp + 2);
  const int half = n / 2 + 1, S = b + g.s * lay.stride, A = a + g.s * lay.stride;
  const FxExp ex = fx_exponent(fx_get_max(lay.s0 + g.s, EVERY ? make_int2(0, (int)(blockDim.x >> 5)) : fx_warps<NS, 1>(g.s)));
  unsigned l1 = 0u;
  for (int k = g.l; k < half; k += g.T) {
    const int kc = n - k;
    // c_k and c_{n-k} (0 where not stored), c_0's real part
    const bool hx = k < K, hy = k > 0 && kc < K;
    double2 sx = fx_get64(S + (hx ? k : 0)), sy = fx_get64(S + (hy ? kc : 0));
    if (!hx) sx.x = 0.0;
    if (!hx || k == 0) sx.y = 0.0;
    if (!hy) sy = make_double2(0.0, 0.0);
    const fx2 x = fx_load<kFxBReal>(sx, ex), y = fx_load<kFxBReal>(sy, ex);
    fx2 z0, z1;
    fx_pack(x, y, ldtab(p.fxr + k), z0, z1);
    fx_put(A + k, fx_swap(z0));
    l1 += fx_l1(z0);
    if (k > 0 && kc != k) {
      fx_put(A + kc, fx_swap(z1));
      l1 += fx_l1(z1);
    }
  }
  fx_reduce_l1<1>(g, lay.s0, l1);
  __syncthreads();
  fx_make_meta<kFxBReal, NS, 1, EVERY>(lay, p.fxs + 32 * kFxInvReal);
  const int sg = fx_sch(lay.s0 + g.s) & 3;
  fx_first(S, g, n, p.fxr0, [&](int e) { return fx_shr(fx_get(A + e), sg); });
  __syncthreads();
  return fx_run<true, PATH == kFxAny>(a, b, lay, g, p, next);
}

// Inverse real transform: the grid values g_j = Re c_0 + 2 Re sum_{1 <= k < K} c_k exp(2 pi i j k / 2n),
// j < 2n, from c_k = load(s, k) (the imaginary part of c_0 is not used).
template <int NS, int PATH = kFxAny, class Load>
__device__ __forceinline__ FxRes<true> xf_c2r(int a, int b, FxLay lay, const FFTPlan& p, int K, Load load) {
  fx_stage<NS, 1>(b, lay, K, [&](int s, int k) { return fx_c0(k, load(s, k)); });
  return xf_c2r_staged<NS, PATH, false>(a, b, lay, p, K);
}

// Forward real transform of the grid pairs (g_2j, g_2j+1) = load(s, j), j < n; results by FxRes::coef.
template <int NS, int PATH = kFxAny, class Load>
__device__ __forceinline__ FxRes<false> xf_r2c(int a, int b, FxLay lay, const FFTPlan& p, Load load) {
  return xf_c2c<false, NS, 1, PATH, true>(a, b, lay, p, load);
}

}  // namespace spadj
