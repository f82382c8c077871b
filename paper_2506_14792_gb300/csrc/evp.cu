// Linear stability eigenvalues of plane shear flows and their adjoint-based parameter
// sensitivities for a batch of pencils (Problem types, "Eigenvalue problems"; Parametric
// sensitivity example).
//
// Pencil p has wavenumbers (alpha_p, beta_p), Reynolds number Re_p and a complex shift
// sigma_p.  With A_p = sigma_p M + L_p, the prognostic block of Phi_p = A_p^-1 [S1S0 on the
// momentum rows] has eigenvalues mu = 1 / (sigma_p - lambda).  On the GPU, per pencil:
//
//   1. A_p and A_p^H in the banded form of couette_setup.h (recombined Chebyshev columns, ordered by mode),
//      from real parts tabled once per problem, and their band LU with partial pivoting;
//   2. shift-invert power iteration with the factors: x <- Phi_p x for the right eigenvector and
//      psi <- Phi_p^H psi (the adjoint eigenproblem) side by side; the two-sided Rayleigh quotient
//      mu = psi^H Phi x / psi^H x gives lambda = sigma - 1/mu;
//   3. the full eigenvectors X = A^-1 [S1S0 x] (velocity, pressure, tau variables) and
//      Y = A^-H [psi], which solve (lambda M + L) X = 0 and (conj(lambda) M^H + L^H) Y = 0;
//   4. eq. eigenvalue_sens, dlambda/dp = -<Y, dL/dp X> / <Y, M X> for p = Re, alpha, beta
//      (M does not depend on them), with dL/dp applied from the N x N ultraspherical blocks.
//
// Why banded: 96 pencils with 20 iterations at N = 48 took 22.7 ms with dense inverses (one LU and 6N solves of
// 4N + 7 unknowns per pencil on the host's 16 cores, 21 ms of it) and take 2.2 ms now; on the GPU the
// inverses would be 10 GFLOP, 10 ms at its FP64 rate.
#include <algorithm>
#include <cmath>
#include <complex>
#include <string>
#include <vector>

#include "couette_setup.h"
#include "pdl.cuh"
#include "problem.h"
#include "rb_setup.h"

namespace spadj {
namespace {

constexpr int kEvpThreads = 256;
constexpr int kEvpWarps = kEvpThreads / 32;
constexpr int kEvpMaxN = 128;      // largest N
constexpr int kEvpMaxLower = 31;   // lower band width: a warp holds the elimination front's rows
constexpr int kEvpMaxUpper = 64;   // width of U with its fill: two entries per lane of a warp
constexpr int kEvpOut = 10;        // lambda, dlambda/dRe, dlambda/dalpha, dlambda/dbeta, residuals

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Deterministic sum of NV values per thread over the CTA's NW warps (fixed warp-then-block order); every
// thread receives the totals.  red holds NW * NV doubles.
template <int NV, int NW>
__device__ __forceinline__ void block_sum(double (&v)[NV], double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = warp_sum(v[i]);
  __syncthreads();
  if (lane == 0)
#pragma unroll
    for (int i = 0; i < NV; ++i) red[warp * NV + i] = v[i];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    double s = 0.0;
    for (int w = 0; w < NW; ++w) s += red[w * NV + i];
    v[i] = s;
  }
}

// The banded systems of a call: system s = 2 p is A' of pencil p, s = 2 p + 1 is J A'^H J (the adjoint direction,
// see couette_setup.h), each of nv unknowns with kl entries below and ku above the diagonal.
struct EvpBand {
  int N, nv, nvp, kl, ku;    // nvp: nv rounded up to whole chunks of sweep steps
  const double *E0, *E1;     // [kBandParts][nv][kl + ku + 1] of the pencils with k != 0 and of the mean pencil
  const double* prm;         // [P][3]: alpha, beta, Re
  const double* shift;       // [P][2]
  double2* B;                // [2P][nv][kl + ku + 1] assembled
  double2* L;                // [2P][nvp][kl] multipliers by column (0 from nv on)
  double2* U;                // [2P][nvp][kl + ku]: U_{j-1-k,j} / U_{j-1-k,j-1-k}, 0 where there is none
  double2* dinv;             // [2P][nv]: 1 / U_jj
  unsigned char* piv;        // [2P][nv]: pivot row - j
  int* width;                // [2P]: largest k + 1 of a non-zero U entry
  int* bad;                  // [P + 1]: singular pencils, and whether there is one
  __device__ __forceinline__ bool mean(int p) const { return prm[3 * p] == 0.0 && prm[3 * p + 1] == 0.0; }
};

__global__ void __launch_bounds__(kEvpThreads) evp_assemble_kernel(const EvpBand S) {
  const int p = blockIdx.x >> 1, dir = blockIdx.x & 1, w = S.kl + S.ku + 1;
  const double al = S.prm[3 * p], be = S.prm[3 * p + 1], nu = 1.0 / S.prm[3 * p + 2];
  const double* E = S.mean(p) ? S.E1 : S.E0;
  const size_t part = (size_t)S.nv * w;
  const double sr = S.shift[2 * p] + nu * (al * al + be * be), si = S.shift[2 * p + 1];
  double2* B = S.B + (size_t)blockIdx.x * part;
  for (int i = threadIdx.x; i < S.nv * w; i += blockDim.x) {
    const int r = i / w, d = i - r * w, k = r - S.kl + d;
    double2 v = make_double2(0.0, 0.0);
    if (k >= 0 && k < S.nv) {
      // entry (r, k) of J A'^H J is the conjugate of A'_{nv-1-k, nv-1-r}, on the same diagonal
      const double* e = E + (size_t)(dir ? S.nv - 1 - k : r) * w + d;
      const double es = __ldg(e + couhost::kPartShift * part);
      v.x = fma(nu, __ldg(e + couhost::kPartVisc * part), fma(sr, es, __ldg(e)));
      v.y = fma(be, __ldg(e + couhost::kPartBeta * part), fma(al, __ldg(e + couhost::kPartAlpha * part), si * es));
      if (dir) v.y = -v.y;
    }
    B[i] = v;
  }
}

__device__ __forceinline__ bool is_zero(double2 v) {
  return (((unsigned)__double2hiint(v.x) << 1) | (unsigned)__double2loint(v.x) | ((unsigned)__double2hiint(v.y) << 1) |
          (unsigned)__double2loint(v.y)) == 0u;
}
__device__ __forceinline__ double2 cinverse(double2 v) {  // 1 / v, scaled where |v|^2 could leave the range
  double s = 1.0;
  const unsigned e = max((unsigned)__double2hiint(v.x) & 0x7ff00000u, (unsigned)__double2hiint(v.y) & 0x7ff00000u) >> 20;
  if (e - 600u > 800u && e != 0x7ffu && e != 0u) {
    s = __hiloint2double((int)((2046u - e) << 20), 0);
    v = make_double2(v.x * s, v.y * s);
  }
  const double q = s / fma(v.x, v.x, v.y * v.y);
  return make_double2(v.x * q, -v.y * q);
}
__device__ __forceinline__ double2 csub_mul(double2 y, double2 f, double2 x) {  // y - f x
  return make_double2(fma(-f.x, x.x, fma(f.y, x.y, y.x)), fma(-f.x, x.y, fma(-f.y, x.x, y.y)));
}

// Band LU of one system per CTA.  The kl + 1 rows of the elimination front and the next two rows sit in shared
// memory, addressed through slot numbers (an interchange swaps two slots) with the columns modulo Wc.  Step j is
// one barrier: warps 1.. update the columns beyond j + 1, scale and store row j of U and load a row, while warp 0
// updates column j + 1 alone, picks its pivot, divides and publishes the multipliers of step j + 1.
// Bound by FP64 issue: an FP64 instruction of a warp takes 64 clocks of its SM partition whatever its active
// lanes, so warp 0's chain (update, reciprocal, multipliers: about 20 of them) runs beside the update
// (4 per row and 32 columns, rows of zero multipliers and columns beyond the pivot row's extent skipped):
// 0.31 ms for the 192 systems of 96 pencils at N = 48.
__global__ void __launch_bounds__(kEvpThreads) evp_lu_kernel(const EvpBand S) {
  const int nv = S.nv, kl = S.kl, ku = S.ku, w = kl + ku + 1, Wc = w + 1, kuf = kl + ku;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
  const double2* B = S.B + (size_t)blockIdx.x * nv * w;
  double2* Lo = S.L + (size_t)blockIdx.x * S.nvp * kl;
  double2* Uo = S.U + (size_t)blockIdx.x * S.nvp * kuf;
  double2* Do = S.dinv + (size_t)blockIdx.x * nv;
  unsigned char* Po = S.piv + (size_t)blockIdx.x * nv;
  extern __shared__ double2 evsm[];
  double2* ring = evsm;                                       // [kl + 3][Wc]
  double2* mul = ring + (size_t)(kl + 3) * Wc;                // [2][32] multipliers of the step, [.][0] = 1 / pivot
  int* slot = reinterpret_cast<int*>(mul + 64);               // [2][34]: rows j..j+kl, row j+1+kl, the free slot
  int* ext = slot + 68;                                       // [kl + 3] last non-zero column of a slot's row
  const double2 zero = make_double2(0.0, 0.0);
  auto load_row = [&](int r, int s, int first, int step) {  // columns r - kl .. r + ku, and zero in the column after
    for (int d = first; d < Wc; d += step) {
      int c = (r - kl + d) % Wc;
      if (c < 0) c += Wc;
      ring[s * Wc + c] = d < w && r < nv ? __ldg(B + (size_t)r * w + d) : zero;
    }
    if (first == 0) ext[s] = r < nv ? min(nv - 1, r + ku) : -1;
  };
  // warp 0: pivot and multipliers of step j from lane k's entry a of row j + k (slot t), into buffer b
  auto panel = [&](int j, double2 a, int t, int b) {
    const unsigned hi = max((unsigned)__double2hiint(a.x) & 0x7fffffffu, (unsigned)__double2hiint(a.y) & 0x7fffffffu);
    unsigned key = lane <= kl ? (hi & ~31u) | (unsigned)(31 - lane) : 0u;  // the first of the largest
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
    const int p = 31 - (int)(key & 31u);
    const double2 ap = make_double2(__shfl_sync(0xffffffffu, a.x, p), __shfl_sync(0xffffffffu, a.y, p));
    const double2 a0 = make_double2(__shfl_sync(0xffffffffu, a.x, 0), __shfl_sync(0xffffffffu, a.y, 0));
    const int tp = __shfl_sync(0xffffffffu, t, p), t0 = __shfl_sync(0xffffffffu, t, 0);
    if (lane == p) { a = a0; t = t0; }
    if (lane == 0) { a = ap; t = tp; }
    const bool sing = is_zero(ap);
    const double2 inv = sing ? zero : cinverse(ap);
    const double2 l = make_double2(a.x * inv.x - a.y * inv.y, a.x * inv.y + a.y * inv.x);
    if (lane <= kl) {
      slot[b * 34 + lane] = t;
      mul[b * 32 + lane] = lane == 0 ? inv : l;
      if (lane > 0) Lo[(size_t)j * kl + lane - 1] = l;
    }
    if (lane == 0) {
      Do[j] = inv;
      Po[j] = (unsigned char)p;
      if (sing) S.bad[blockIdx.x >> 1] = S.bad[gridDim.x >> 1] = 1;
    }
  };
  for (int i = tid; i < (S.nvp - nv) * kl; i += blockDim.x) Lo[(size_t)nv * kl + i] = zero;
  for (int i = tid; i < (S.nvp - nv) * kuf; i += blockDim.x) Uo[(size_t)nv * kuf + i] = zero;
  for (int c = warp; c < min(kuf, nv); c += kEvpWarps)
    for (int q = c + lane; q < kuf; q += 32) Uo[(size_t)c * kuf + q] = zero;
  for (int r = warp; r < kl + 2; r += kEvpWarps) load_row(r, r, lane, 32);
  __syncthreads();
  if (warp == 0) {
    panel(0, lane <= kl ? ring[lane * Wc] : zero, lane, 0);
    if (lane == 0) { slot[kl + 1] = kl + 1; slot[kl + 2] = kl + 2; }
  }
  __syncthreads();
  int jc = 0, width = 0;  // jc = j mod Wc
  for (int j = 0; j < nv; ++j) {
    const int b = j & 1;
    const int* sl = slot + b * 34;
    const double2* m = mul + b * 32;
    const int s0 = sl[0], e0 = ext[s0];
    const double2* piv = ring + s0 * Wc;
    auto pos = [&](int q) { return jc + q < Wc ? jc + q : jc + q - Wc; };  // column j + q, q < Wc
    if (warp == 0) {
      if (j + 1 < nv) {
        const int t = lane <= kl ? sl[lane + 1] : 0;
        double2 a = lane <= kl ? ring[t * Wc + pos(1)] : zero;
        if (lane < kl) a = csub_mul(a, m[lane + 1], piv[pos(1)]);
        if (lane == 0) {
          slot[(b ^ 1) * 34 + kl + 1] = sl[kl + 2];
          slot[(b ^ 1) * 34 + kl + 2] = s0;
        }
        panel(j + 1, a, t, b ^ 1);
      }
    } else {
      if (warp == 1) load_row(j + 2 + kl, sl[kl + 2], lane, 32);
      if (warp == 2)
        for (int q = lane; q < kuf; q += 32) {
          const int c = j + 1 + q;
          if (c >= nv) break;
          double2 u = zero;
          if (c <= e0) {
            const double2 v = piv[pos(q + 1)], inv = m[0];
            u = make_double2(v.x * inv.x - v.y * inv.y, v.x * inv.y + v.y * inv.x);
          }
          Uo[(size_t)c * kuf + q] = u;
        }
      if (warp == 3 && lane >= 1 && lane <= kl) {
        const int s = sl[lane];
        ring[s * Wc + (jc == 0 ? Wc - 1 : jc - 1)] = zero;  // column j + w of the rows that stay
        if (!is_zero(m[lane])) ext[s] = max(ext[s], e0);
      }
      for (int k = warp; k <= kl; k += kEvpWarps - 1) {
        const double2 l = m[k];
        if (is_zero(l)) continue;
        double2* row = ring + sl[k] * Wc;
        for (int c = j + 2 + lane; c <= e0; c += 32) {
          const int q = pos(c - j);
          row[q] = csub_mul(row[q], l, piv[q]);
        }
      }
      width = max(width, e0 - j);
    }
    __syncthreads();
    jc = jc + 1 < Wc ? jc + 1 : 0;
  }
  if (tid == 32) S.width[blockIdx.x] = width;
}

struct EvpIterArgs {
  EvpBand S;
  const double* ssb;  // [N][5]: S1S0[n][n + d]
  const double* pw;   // [N]: the mean pencil's pressure recombination
  double2* x;         // [P][H] right iterate (in / out)
  double2* psi;       // [P][H] left iterate (in / out)
  double2* XY;        // [P][2][nv]: X, Y
  double* out;        // [P][kEvpOut]
  int n_iter;
};

constexpr int kIterThreads = 128, kIterWarps = 4;
constexpr int kChunk = 8;                 // sweep steps whose factors are copied together
constexpr int kPadLow = 64, kPadHigh = 32;  // entries around the unknowns that steps near the ends touch

// The two warps of a direction meet (one named barrier each)
__device__ __forceinline__ void pair_sync(int dir) {
  if (dir) asm volatile("bar.sync 2, 64;" ::: "memory");
  else asm volatile("bar.sync 1, 64;" ::: "memory");
}

// Dynamic shared memory of evp_iter_kernel: x, psi and their images, sums, unknowns, factors, 1 / U_jj, pivots
inline int evp_padded(int nv) { return (nv + kChunk - 1) / kChunk * kChunk; }
inline size_t iter_smem(int N, int kuf) {
  const size_t nvp = evp_padded(4 * N + 7);
  return sizeof(double2) * 12 * N + sizeof(double) * (kIterWarps * 6 + 4 * (kPadLow + nvp + kPadHigh)) +
         sizeof(double2) * (4 * (size_t)kChunk * kuf + 2 * nvp) + 2 * (nvp + kChunk);
}

// One CTA per pencil: n_iter steps of x <- Phi x / |Phi x|, psi <- Phi^H psi / |Phi^H psi|, then X and Y (n_iter = 0: of x
// and psi as they are, which another kernel has iterated).  Warps 0
// and 1 run the solves with A', warps 2 and 3 those with J A'^H J; of each pair one warp holds the real parts of
// the unknowns and one the imaginary ones, so a sweep step is two FP64 instructions deep (128 clocks of latency).
// Bound by that chain: 2 nv steps per solve.  The factors are copied to shared memory a chunk of steps ahead and
// the steps of a chunk are unrolled, with entries around the unknowns so that none needs a bounds check: 96 pencils,
// N = 48, 20 iterations 2.29 ms with factors loaded from L2 step by step, 2.08 ms copied ahead, 1.78 ms unrolled.
__global__ void __launch_bounds__(kIterThreads) evp_iter_kernel(const EvpIterArgs A) {
  const EvpBand& S = A.S;
  const int p = blockIdx.x, N = S.N, H = 3 * N, nv = S.nv, nvp = S.nvp, kl = S.kl, kuf = S.kl + S.ku;
  if (S.bad[gridDim.x]) return;  // the call fails: nothing is written
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, dir = warp >> 1, im = warp & 1, t64 = tid & 63;
  const bool mean = S.mean(p);
  const int orow = mean ? 0 : 1;  // position of mode 0's equations
  extern __shared__ double2 evsm[];
  double2* x = evsm;
  double2* ps = x + H;
  double2* y = ps + H;
  double2* z = y + H;
  double* red = reinterpret_cast<double*>(z + H);       // [kIterWarps * 6]
  const int ld = kPadLow + nvp + kPadHigh;
  double* sol = red + kIterWarps * 6 + dir * 2 * ld + kPadLow;    // this direction's unknowns: real parts,
  double* mine = sol + im * ld;                                   // imaginary parts ld later
  const double* other = sol + (im ^ 1) * ld;
  double2* after = reinterpret_cast<double2*>(red + kIterWarps * 6 + 4 * ld);
  double2* fac = after + dir * 2 * kChunk * kuf;                  // [2][kChunk][kuf] factors of two chunks of steps
  double2* dinv = after + 4 * kChunk * kuf + dir * nvp;           // [nv]
  unsigned char* pv = reinterpret_cast<unsigned char*>(after + 4 * kChunk * kuf + 2 * nvp) + dir * (nvp + kChunk);
  const size_t sys = 2 * (size_t)p + dir;
  const double2* Lp = S.L + sys * nvp * kl;
  const double2* Up = S.U + sys * nvp * kuf;
  const double2* Dp = S.dinv + sys * nv;
  const unsigned char* Pp = S.piv + sys * nv;
  const int wu = min(S.width[sys], kuf);
  const double2 zero = make_double2(0.0, 0.0);
  // right-hand side of this direction from v (H entries), by its 64 threads
  auto fill = [&](const double2* v) {
    for (int i = t64; i < 2 * ld; i += 64) sol[i - kPadLow] = 0.0;
    pair_sync(dir);
    for (int c = t64; c < H; c += 64) {
      const int f = c / N, n = c - f * N;
      double2 r = zero;
      int q;
      if (dir == 0) {
        for (int d = 0; d < 5 && n + d < N; ++d) {
          const double s = __ldg(A.ssb + n * 5 + d);
          r.x = fma(s, v[c + d].x, r.x);
          r.y = fma(s, v[c + d].y, r.y);
        }
        q = orow + 4 * n + f;
      } else {
        r = v[c];
        if (n + 2 < N) r = make_double2(r.x - v[c + 2].x, r.y - v[c + 2].y);
        q = nv - 1 - (1 + 4 * n + f);
      }
      sol[q] = r.x;
      sol[ld + q] = r.y;
    }
    pair_sync(dir);
  };
  // a factor as this warp uses it: f x has the parts f.x xr - f.y xi and f.x xi + f.y xr
  auto part = [&](double2 f) {
    return make_double2(f.x, __hiloint2double(__double2hiint(f.y) ^ (im ? (int)0x80000000 : 0), __double2loint(f.y)));
  };
  // v - f x: xa is x's part of this warp, xb the other one (two dependent FP64 instructions)
  auto sub = [&](double v, double2 f, double xa, double xb) { return fma(-f.x, xa, fma(f.y, xb, v)); };
  // rows r0 .. r0 + n - 1 of a factor with wd entries per row into buffer b, by this direction's threads
  auto copy = [&](const double2* src, int wd, int r0, int n, int b) {
    double2* to = fac + b * kChunk * kuf;
    for (int i = t64; i < n * wd; i += 64) cp_async16(to + i, src + (size_t)r0 * wd + i);
    cp_async_commit();
  };
  const int chunks = nvp / kChunk;
  auto solve = [&]() {
    // forward: the interchange of step j + 1 is made by where step j writes its results
    if (lane == 0 && pv[0]) {
      const double a = mine[0];
      mine[0] = mine[pv[0]];
      mine[pv[0]] = a;
    }
    copy(Lp, kl, 0, kChunk, 0);
    for (int c = 0; c < chunks; ++c) {
      cp_async_wait_all();
      pair_sync(dir);
      if (c + 1 < chunks) copy(Lp, kl, (c + 1) * kChunk, kChunk, (c + 1) & 1);
      const double2* F = fac + (c & 1) * kChunk * kuf + lane;
      double* m = mine + c * kChunk;
      const double* o = other + c * kChunk;
      double2 f[kChunk];
      int to[kChunk];
#pragma unroll
      for (int a = 0; a < kChunk; ++a) {
        f[a] = part(lane < kl ? F[a * kl] : zero);
        const int pc = pv[c * kChunk + a + 1];
        to[a] = lane == 0 ? pc : lane == pc ? 0 : lane;
      }
#pragma unroll
      for (int a = 0; a < kChunk; ++a) {
        if (a > 0) pair_sync(dir);
        const double v = sub(m[a + 1 + lane], f[a], m[a], o[a]);
        __syncwarp();
        m[a + 1 + to[a]] = v;
      }
    }
    pair_sync(dir);
    copy(Up, kuf, (chunks - 1) * kChunk, kChunk, 0);
    for (int i = t64; i < nv; i += 64) {
      const double2 d = dinv[i];
      const double a = sol[i], c = sol[ld + i];
      sol[i] = a * d.x - c * d.y;
      sol[ld + i] = a * d.y + c * d.x;
    }
    for (int c = chunks - 1, b = 0; c >= 0; --c, b ^= 1) {
      cp_async_wait_all();
      pair_sync(dir);
      if (c > 0) copy(Up, kuf, (c - 1) * kChunk, kChunk, b ^ 1);
      const double2* F = fac + b * kChunk * kuf + lane;
      double* m = mine + c * kChunk;
      const double* o = other + c * kChunk;
      double2 f[kChunk], g[kChunk];  // entries lane and lane + 32 (fill of the interchanges: few are non-zero)
      unsigned far = 0u;
#pragma unroll
      for (int a = 0; a < kChunk; ++a) {
        f[a] = part(lane < wu ? F[a * kuf] : zero);
        g[a] = lane + 32 < wu ? F[a * kuf + 32] : zero;
        if (!is_zero(g[a])) far |= 1u << a;
        g[a] = part(g[a]);
      }
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) far |= __shfl_xor_sync(0xffffffffu, far, s);
#pragma unroll
      for (int a = kChunk - 1; a >= 0; --a) {
        if (a < kChunk - 1) pair_sync(dir);
        const double xa = m[a], xb = o[a];
        double* e = m + a - 1 - lane;
        e[0] = sub(e[0], f[a], xa, xb);
        if (far >> a & 1u) e[-32] = sub(e[-32], g[a], xa, xb);
      }
    }
    pair_sync(dir);
  };
  auto at = [&](int i) { return make_double2(sol[i], sol[ld + i]); };
  for (int i = t64; i < nv; i += 64) dinv[i] = __ldg(Dp + i);
  for (int i = t64; i < nvp + kChunk; i += 64) pv[i] = i < nv ? __ldg(Pp + i) : 0;
  for (int k = tid; k < H; k += kIterThreads) {
    x[k] = A.x[(size_t)p * H + k];
    ps[k] = A.psi[(size_t)p * H + k];
  }
  double mur = 0.0, mui = 0.0, res_r = 1.0, res_l = 1.0;
  for (int it = 0; it < A.n_iter; ++it) {
    __syncthreads();
    fill(dir == 0 ? x : ps);
    solve();
    for (int c = t64; c < H; c += 64) {
      const int f = c / N, n = c - f * N;
      if (dir == 0) {
        double2 v = at(1 + 4 * n + f);
        if (n >= 2) v = make_double2(v.x - sol[1 + 4 * (n - 2) + f], v.y - sol[ld + 1 + 4 * (n - 2) + f]);
        y[c] = v;
      } else {
        double2 v = zero;
        for (int d = 0; d < 5 && n - d >= 0; ++d) {
          const double s = __ldg(A.ssb + (n - d) * 5 + d);
          const double2 q = at(nv - 1 - (orow + 4 * (n - d) + f));
          v.x = fma(s, q.x, v.x);
          v.y = fma(s, q.y, v.y);
        }
        z[c] = v;
      }
    }
    __syncthreads();
    // norms and the two-sided Rayleigh quotient
    double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int k = tid; k < H; k += kIterThreads) {
      const double2 yk = y[k], zk = z[k], xk = x[k], pk = ps[k];
      v[0] = fma(yk.x, yk.x, fma(yk.y, yk.y, v[0]));
      v[1] = fma(zk.x, zk.x, fma(zk.y, zk.y, v[1]));
      v[2] += pk.x * yk.x + pk.y * yk.y;  // psi^H y
      v[3] += pk.x * yk.y - pk.y * yk.x;
      v[4] += pk.x * xk.x + pk.y * xk.y;  // psi^H x
      v[5] += pk.x * xk.y - pk.y * xk.x;
    }
    block_sum<6, kIterWarps>(v, red);
    const double dd = v[4] * v[4] + v[5] * v[5];
    if (dd > 0.0) {
      mur = (v[2] * v[4] + v[3] * v[5]) / dd;
      mui = (v[3] * v[4] - v[2] * v[5]) / dd;
    }
    if (it + 1 == A.n_iter) {  // residuals |Phi x - mu x| / |Phi x|, |Phi^H psi - conj(mu) psi| / |Phi^H psi|
      double r2[2] = {0.0, 0.0};
      for (int k = tid; k < H; k += kIterThreads) {
        const double2 yk = y[k], xk = x[k], pk = ps[k], zk = z[k];
        const double ex = yk.x - (mur * xk.x - mui * xk.y), ey = yk.y - (mur * xk.y + mui * xk.x);
        const double fx = zk.x - (mur * pk.x + mui * pk.y), fy = zk.y - (mur * pk.y - mui * pk.x);
        r2[0] += ex * ex + ey * ey;
        r2[1] += fx * fx + fy * fy;
      }
      block_sum<2, kIterWarps>(r2, red);
      res_r = v[0] > 0.0 ? sqrt(r2[0] / v[0]) : 1.0;
      res_l = v[1] > 0.0 ? sqrt(r2[1] / v[1]) : 1.0;
    }
    const double sy = v[0] > 0.0 ? 1.0 / sqrt(v[0]) : 0.0, sz = v[1] > 0.0 ? 1.0 / sqrt(v[1]) : 0.0;
    for (int k = tid; k < H; k += kIterThreads) {
      const double2 yk = y[k], zk = z[k];
      x[k] = make_double2(yk.x * sy, yk.y * sy);
      ps[k] = make_double2(zk.x * sz, zk.y * sz);
    }
  }
  __syncthreads();
  for (int k = tid; k < H && A.n_iter > 0; k += kIterThreads) {
    A.x[(size_t)p * H + k] = x[k];
    A.psi[(size_t)p * H + k] = ps[k];
  }
  if (tid == 0 && A.n_iter > 0) {
    double* o = A.out + (size_t)p * kEvpOut;
    const double m2 = mur * mur + mui * mui;
    // lambda = sigma - 1/mu
    o[0] = m2 > 0.0 ? S.shift[2 * p] - mur / m2 : 0.0;
    o[1] = m2 > 0.0 ? S.shift[2 * p + 1] + mui / m2 : 0.0;
    o[8] = res_r;
    o[9] = res_l;
  }
  // X (unknowns u, v, w, p, tau_u1, ..., tau_w2, tau_p) and Y (equations u, v, w, continuity, boundary, gauge)
  fill(dir == 0 ? x : ps);
  solve();
  double2* o = A.XY + sys * nv;
  for (int i = t64; i < nv; i += 64) {
    const int f = i / N, n = i - f * N;
    double2 v;
    if (dir == 0) {
      if (f < 4) {
        v = at(1 + 4 * n + f);
        if (n >= 2 && (f < 3 || (mean && n % 2 == 0))) {
          const double s = f < 3 ? 1.0 : __ldg(A.pw + n - 2);
          const double2 u = at(1 + 4 * (n - 2) + f);
          v = make_double2(v.x - s * u.x, v.y - s * u.y);
        }
      } else {
        v = at(i == nv - 1 ? 0 : 1 + i);
      }
    } else {
      const int q = f < 4 ? orow + 4 * n + f : i < nv - 1 ? orow + i : mean ? nv - 1 : 0;
      v = at(nv - 1 - q);
    }
    o[i] = v;
  }
}

// ---- iterations with the dense Phi ------------------------------------------------------------------------
//
// A step of the banded iteration is a chain of 2 nv dependent sweep steps however few the pencils; with the 3N x 3N
// operator itself it is one matrix-vector product per direction.  Where enough steps pay for the operator's columns (3N
// banded solves per pencil), it is built and iterated with (ShearEvp::dense_iterations).

// Column c of Phi_p = (A_p^-1 [S1S0 e_c]) on u, v, w, one warp per column: a lane per row below the pivot (or above it, in
// the back substitution), factors loaded a chunk of steps ahead.  Bound by FP64 issue when all partitions have
// a warp (4 instructions a step), by the chain of 2 nv steps when there are fewer columns.
constexpr int kPhiWarps = 4;
inline size_t phi_smem(int nvp) { return sizeof(double) * 2 * kPhiWarps * (size_t)(kPadLow + nvp + kPadHigh); }
__global__ void __launch_bounds__(32 * kPhiWarps) evp_phi_kernel(const EvpBand S, int P, const double* __restrict__ ssb,
                                                                double2* __restrict__ phi) {
  const int N = S.N, H = 3 * N, nv = S.nv, nvp = S.nvp, kl = S.kl, kuf = S.kl + S.ku;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, blocks = (H + kPhiWarps - 1) / kPhiWarps;
  const int p = blockIdx.x / blocks, col = (blockIdx.x - p * blocks) * kPhiWarps + warp;
  if (S.bad[P] || col >= H) return;  // (the warps do not meet)
  extern __shared__ double2 evsm[];
  const int ld = kPadLow + nvp + kPadHigh;
  double* re = reinterpret_cast<double*>(evsm) + 2 * warp * ld + kPadLow;
  double* im = re + ld;
  const size_t sys = 2 * (size_t)p;
  const double2* Lp = S.L + sys * nvp * kl;
  const double2* Up = S.U + sys * nvp * kuf;
  const double2* Dp = S.dinv + sys * nv;
  const unsigned char* Pp = S.piv + sys * nv;
  const int wu = min(S.width[sys], kuf), orow = S.mean(p) ? 0 : 1;
  const double2 zero = make_double2(0.0, 0.0);
  for (int i = lane; i < 2 * ld; i += 32) re[i - kPadLow] = 0.0;
  __syncwarp();
  const int f0 = col / N, n0 = col - f0 * N;
  if (lane < 5 && n0 >= lane) re[orow + 4 * (n0 - lane) + f0] = __ldg(ssb + (n0 - lane) * 5 + lane);
  __syncwarp();
  if (lane == 0 && Pp[0]) {
    const int q = Pp[0];
    const double a = re[0], b = im[0];
    re[0] = re[q]; im[0] = im[q];
    re[q] = a; im[q] = b;
  }
  __syncwarp();
  // v - f x
  auto sub = [](double2 v, double2 f, double2 x) { return csub_mul(v, f, x); };
  double2 f[kChunk], g[kChunk];
  int to[kChunk];
  auto loadL = [&](int j0) {
#pragma unroll
    for (int a = 0; a < kChunk; ++a) {
      f[a] = lane < kl ? __ldg(Lp + (size_t)(j0 + a) * kl + lane) : zero;
      const int pc = j0 + a + 1 < nv ? __ldg(Pp + j0 + a + 1) : 0;
      to[a] = lane == 0 ? pc : lane == pc ? 0 : lane;  // the next step's interchange, made by where this one writes
    }
  };
  loadL(0);
  for (int j0 = 0; j0 < nvp; j0 += kChunk) {
    double2 h[kChunk];
    int th[kChunk];
#pragma unroll
    for (int a = 0; a < kChunk; ++a) { h[a] = f[a]; th[a] = to[a]; }
    if (j0 + kChunk < nvp) loadL(j0 + kChunk);
#pragma unroll
    for (int a = 0; a < kChunk; ++a) {
      const int j = j0 + a;
      const double2 v = sub(make_double2(re[j + 1 + lane], im[j + 1 + lane]), h[a], make_double2(re[j], im[j]));
      __syncwarp();
      re[j + 1 + th[a]] = v.x;
      im[j + 1 + th[a]] = v.y;
      __syncwarp();
    }
  }
  auto loadU = [&](int j0) {
#pragma unroll
    for (int a = 0; a < kChunk; ++a) {
      f[a] = lane < wu ? __ldg(Up + (size_t)(j0 + a) * kuf + lane) : zero;
      g[a] = lane + 32 < wu ? __ldg(Up + (size_t)(j0 + a) * kuf + lane + 32) : zero;
    }
  };
  loadU(nvp - kChunk);
  for (int i = lane; i < nv; i += 32) {
    const double2 d = __ldg(Dp + i);
    const double a = re[i], b = im[i];
    re[i] = a * d.x - b * d.y;
    im[i] = a * d.y + b * d.x;
  }
  __syncwarp();
  for (int j0 = nvp - kChunk; j0 >= 0; j0 -= kChunk) {
    double2 h[kChunk], w[kChunk];
    unsigned far = 0u;
#pragma unroll
    for (int a = 0; a < kChunk; ++a) {
      h[a] = f[a];
      w[a] = g[a];
      if (__any_sync(0xffffffffu, !is_zero(w[a]))) far |= 1u << a;
    }
    if (j0 > 0) loadU(j0 - kChunk);
#pragma unroll
    for (int a = kChunk - 1; a >= 0; --a) {
      const int j = j0 + a, e = j - 1 - lane;
      const double2 x = make_double2(re[j], im[j]);
      const double2 v = sub(make_double2(re[e], im[e]), h[a], x);
      re[e] = v.x;
      im[e] = v.y;
      if (far >> a & 1u) {
        const double2 u = sub(make_double2(re[e - 32], im[e - 32]), w[a], x);
        re[e - 32] = u.x;
        im[e - 32] = u.y;
      }
      __syncwarp();
    }
  }
  double2* o = phi + (size_t)p * H * H + col;
  for (int r = lane; r < H; r += 32) {
    const int q = r / N, n = r - q * N, i = 1 + 4 * n + q;
    o[(size_t)r * H] = n >= 2 ? make_double2(re[i] - re[i - 8], im[i] - im[i - 8]) : make_double2(re[i], im[i]);
  }
}

constexpr int kRows = 4;       // rows per warp block in evp_dense_kernel (2 kRows partial sums per lane)
constexpr int kRowsLog2V = 3;  // log2(2 kRows)

// Warp reduction of 2 kRows values per lane at once: a butterfly in which every exchange halves
// the values a lane carries (offsets 16, 8, ...; the lane keeps the half selected by that bit of
// its index) until one is left, then plain exchanges at the remaining offsets.  Every lane of the
// group l >> (5 - kRowsLog2V) = m ends with the total of value m.  2 kRows + 1 additions per lane
// for 2 kRows sums instead of 5 per sum; fixed order, so deterministic.
__device__ __forceinline__ double warp_reduce_rows(double (&v)[2 * kRows], int lane) {
  int off = 16;
#pragma unroll
  for (int half = kRows; half >= 1; half >>= 1, off >>= 1) {
    const bool hi = (lane & off) != 0;
#pragma unroll
    for (int j = 0; j < half; ++j) {
      const double send = hi ? v[j] : v[j + half];
      const double keep = hi ? v[j + half] : v[j];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  double t = v[0];
#pragma unroll
  for (int o = 16 >> kRowsLog2V; o >= 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

struct EvpDenseArgs {
  const double2* phi;    // [P][H][H]
  double2* x;            // [P][H] right iterate (in / out)
  double2* psi;          // [P][H] left iterate (in / out)
  const double* shift;   // [P][2]
  const int* bad;        // [P + 1]
  double* out;           // [P][kEvpOut]
  int H, n_iter;
};

// One CTA per pencil: n_iter steps of x <- Phi x / |Phi x|, psi <- Phi^H psi / |Phi^H psi| with
// each row of Phi read once per step for both products (warps over rows, lanes over columns,
// coalesced), all in shared memory between steps.
// NC = ceil(3N / 32) column chunks per lane, fixed at compile time so that only the last chunk
// carries a bounds predicate.
template <int NC>
__global__ void __launch_bounds__(kEvpThreads, 2) evp_dense_kernel(const EvpDenseArgs A) {
  const int p = blockIdx.x, H = A.H;
  if (A.bad[gridDim.x]) return;  // the call fails: nothing is written
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  extern __shared__ double2 evsm[];
  double2* x = evsm;
  double2* ps = x + H;
  double2* y = ps + H;
  double2* zp = y + H;                                    // [kEvpWarps][H] partial Phi^H psi
  double* red = reinterpret_cast<double*>(zp + (size_t)kEvpWarps * H);
  const double2* Tp = A.phi + (size_t)p * H * H;
  for (int k = threadIdx.x; k < H; k += blockDim.x) {
    x[k] = A.x[(size_t)p * H + k];
    ps[k] = A.psi[(size_t)p * H + k];
  }
  double mur = 0.0, mui = 0.0, res_r = 1.0, res_l = 1.0;
  for (int it = 0; it < A.n_iter; ++it) {
    __syncthreads();
    double2 zacc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) zacc[c] = make_double2(0.0, 0.0);
    // blocks of kRows rows per warp: each x chunk is read once per block, and the row sums of
    // the block are reduced together (warp_reduce_rows) instead of one butterfly per row
    for (int rb = warp * kRows; rb < H; rb += kRows * kEvpWarps) {
      double acc[2 * kRows];
      double2 pr[kRows];
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        acc[2 * i] = acc[2 * i + 1] = 0.0;
        pr[i] = rb + i < H ? ps[rb + i] : make_double2(0.0, 0.0);
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int k = c * 32 + lane;
        if (c < NC - 1 || k < H) {
          const double2 xv = x[k];
#pragma unroll
          for (int i = 0; i < kRows; ++i) {
            if (rb + i >= H) continue;
            const double2 t = __ldg(&Tp[(size_t)(rb + i) * H + k]);
            acc[2 * i] = fma(t.x, xv.x, acc[2 * i]);
            acc[2 * i] = fma(-t.y, xv.y, acc[2 * i]);
            acc[2 * i + 1] = fma(t.x, xv.y, acc[2 * i + 1]);
            acc[2 * i + 1] = fma(t.y, xv.x, acc[2 * i + 1]);
            zacc[c].x = fma(t.x, pr[i].x, zacc[c].x);  // conj(t) * psi_r
            zacc[c].x = fma(t.y, pr[i].y, zacc[c].x);
            zacc[c].y = fma(t.x, pr[i].y, zacc[c].y);
            zacc[c].y = fma(-t.y, pr[i].x, zacc[c].y);
          }
        }
      }
      const double tot = warp_reduce_rows(acc, lane);
      // lane group m = lane >> (5 - kRowsLog2V) holds value m = 2 (row - rb) + component
      const int m = lane >> (5 - kRowsLog2V), r = rb + (m >> 1);
      if ((lane & ((1 << (5 - kRowsLog2V)) - 1)) == 0 && r < H) reinterpret_cast<double*>(y)[2 * r + (m & 1)] = tot;
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int k = c * 32 + lane;
      if (c < NC - 1 || k < H) zp[(size_t)warp * H + k] = zacc[c];
    }
    __syncthreads();
    // z = sum of the warp partials (into zp row 0); norms and the two-sided Rayleigh quotient
    double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int k = threadIdx.x; k < H; k += blockDim.x) {
      double2 z = zp[k];
      for (int w = 1; w < kEvpWarps; ++w) {
        const double2 q = zp[(size_t)w * H + k];
        z.x += q.x;
        z.y += q.y;
      }
      zp[k] = z;
      const double2 yk = y[k], xk = x[k], pk = ps[k];
      v[0] = fma(yk.x, yk.x, fma(yk.y, yk.y, v[0]));
      v[1] = fma(z.x, z.x, fma(z.y, z.y, v[1]));
      v[2] += pk.x * yk.x + pk.y * yk.y;  // psi^H y
      v[3] += pk.x * yk.y - pk.y * yk.x;
      v[4] += pk.x * xk.x + pk.y * xk.y;  // psi^H x
      v[5] += pk.x * xk.y - pk.y * xk.x;
    }
    block_sum<6, kEvpWarps>(v, red);
    const double dd = v[4] * v[4] + v[5] * v[5];
    if (dd > 0.0) {
      mur = (v[2] * v[4] + v[3] * v[5]) / dd;
      mui = (v[3] * v[4] - v[2] * v[5]) / dd;
    }
    if (it + 1 == A.n_iter) {  // residuals |Phi x - mu x| / |Phi x|, |Phi^H psi - conj(mu) psi| / |Phi^H psi|
      double r2[2] = {0.0, 0.0};
      for (int k = threadIdx.x; k < H; k += blockDim.x) {
        const double2 yk = y[k], xk = x[k], pk = ps[k], z = zp[k];
        const double ex = yk.x - (mur * xk.x - mui * xk.y), ey = yk.y - (mur * xk.y + mui * xk.x);
        const double fx = z.x - (mur * pk.x + mui * pk.y), fy = z.y - (mur * pk.y - mui * pk.x);
        r2[0] += ex * ex + ey * ey;
        r2[1] += fx * fx + fy * fy;
      }
      block_sum<2, kEvpWarps>(r2, red);
      res_r = v[0] > 0.0 ? sqrt(r2[0] / v[0]) : 1.0;
      res_l = v[1] > 0.0 ? sqrt(r2[1] / v[1]) : 1.0;
    }
    const double sy = v[0] > 0.0 ? 1.0 / sqrt(v[0]) : 0.0, sz = v[1] > 0.0 ? 1.0 / sqrt(v[1]) : 0.0;
    for (int k = threadIdx.x; k < H; k += blockDim.x) {
      const double2 yk = y[k], z = zp[k];
      x[k] = make_double2(yk.x * sy, yk.y * sy);
      ps[k] = make_double2(z.x * sz, z.y * sz);
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < H; k += blockDim.x) {
    A.x[(size_t)p * H + k] = x[k];
    A.psi[(size_t)p * H + k] = ps[k];
  }
  if (threadIdx.x == 0) {
    double* o = A.out + (size_t)p * kEvpOut;
    const double m2 = mur * mur + mui * mui;
    // lambda = sigma - 1/mu
    o[0] = m2 > 0.0 ? A.shift[2 * p] - mur / m2 : 0.0;
    o[1] = m2 > 0.0 ? A.shift[2 * p + 1] + mui / m2 : 0.0;
    o[8] = res_r;
    o[9] = res_l;
  }
}

using EvpDenseFn = void (*)(const EvpDenseArgs);
constexpr int kDenseMaxN = 64;
const EvpDenseFn kEvpDense[3 * kDenseMaxN / 32] = {evp_dense_kernel<1>, evp_dense_kernel<2>, evp_dense_kernel<3>,
                                                   evp_dense_kernel<4>, evp_dense_kernel<5>, evp_dense_kernel<6>};

struct EvpSensArgs {
  const double2* XY;                 // [P][2][nv]: X, Y
  const double* prm;                 // [P][3]: alpha, beta, Re
  const double *SS, *DD, *Um, *S0;   // N x N row-major
  double* out;                       // [P][kEvpOut]
  const int* bad;                    // non-zero: the call fails, nothing is written
  int N, nv, lift_row;
  double lift_val;
};

// eq. eigenvalue_sens for p = Re, alpha, beta.  With lap = DD - k^2 SS on each velocity block:
//   dL/dRe    = lap / Re^2 on the u, v, w blocks, lift_val / Re^2 at the tau_q1 lifts;
//   dL/dalpha = 2 alpha nu SS + i Umat on the blocks, i SS at (u-eq, p), i S0 at (cont, u);
//   dL/dbeta  = 2 beta nu SS on the blocks, i SS at (v-eq, p), i S0 at (cont, v);
// <Y, M X> = sum over u, v, w of Y_q^H SS X_q.
__global__ void __launch_bounds__(kEvpThreads) evp_sens_kernel(const EvpSensArgs A) {
  const int p = blockIdx.x, N = A.N, nv = A.nv;
  if (*A.bad) return;
  extern __shared__ double2 essm[];
  double2* X = essm;
  double2* Y = X + nv;
  double* red = reinterpret_cast<double*>(Y + nv);
  for (int i = threadIdx.x; i < nv; i += blockDim.x) {
    X[i] = A.XY[((size_t)p * 2 + 0) * nv + i];
    Y[i] = A.XY[((size_t)p * 2 + 1) * nv + i];
  }
  __syncthreads();
  const double al = A.prm[3 * p], be = A.prm[3 * p + 1], Re = A.prm[3 * p + 2];
  const double nu = 1.0 / Re, k2 = al * al + be * be;
  // accumulators (re, im): den, nRe, nA, nB
  double v[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  auto cjmul_add = [](double* acc, double2 y, double2 z) {  // acc += conj(y) z
    acc[0] += y.x * z.x + y.y * z.y;
    acc[1] += y.x * z.y - y.y * z.x;
  };
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    double2 s[3], d[3], u[3], sp, s0u, s0v;
    for (int q = 0; q < 3; ++q) s[q] = d[q] = u[q] = make_double2(0.0, 0.0);
    sp = s0u = s0v = make_double2(0.0, 0.0);
    for (int j = 0; j < N; ++j) {
      const double ss = __ldg(&A.SS[(size_t)i * N + j]), dd = __ldg(&A.DD[(size_t)i * N + j]);
      const double um = __ldg(&A.Um[(size_t)i * N + j]), s0 = __ldg(&A.S0[(size_t)i * N + j]);
      for (int q = 0; q < 3; ++q) {
        const double2 xq = X[q * N + j];
        s[q].x = fma(ss, xq.x, s[q].x); s[q].y = fma(ss, xq.y, s[q].y);
        d[q].x = fma(dd, xq.x, d[q].x); d[q].y = fma(dd, xq.y, d[q].y);
        u[q].x = fma(um, xq.x, u[q].x); u[q].y = fma(um, xq.y, u[q].y);
      }
      const double2 xp = X[3 * N + j], xu = X[j], xv = X[N + j];
      sp.x = fma(ss, xp.x, sp.x); sp.y = fma(ss, xp.y, sp.y);
      s0u.x = fma(s0, xu.x, s0u.x); s0u.y = fma(s0, xu.y, s0u.y);
      s0v.x = fma(s0, xv.x, s0v.x); s0v.y = fma(s0, xv.y, s0v.y);
    }
    for (int q = 0; q < 3; ++q) {
      const double2 yq = Y[q * N + i];
      cjmul_add(&v[0], yq, s[q]);
      cjmul_add(&v[2], yq, make_double2(d[q].x - k2 * s[q].x, d[q].y - k2 * s[q].y));
      // 2 alpha nu s + i u
      cjmul_add(&v[4], yq, make_double2(2.0 * al * nu * s[q].x - u[q].y, 2.0 * al * nu * s[q].y + u[q].x));
      cjmul_add(&v[6], yq, make_double2(2.0 * be * nu * s[q].x, 2.0 * be * nu * s[q].y));
    }
    const double2 yu = Y[i], yv = Y[N + i], yp = Y[3 * N + i];
    cjmul_add(&v[4], yu, make_double2(-sp.y, sp.x));    // i SS p in the u-equation
    cjmul_add(&v[4], yp, make_double2(-s0u.y, s0u.x));  // i S0 u in continuity
    cjmul_add(&v[6], yv, make_double2(-sp.y, sp.x));
    cjmul_add(&v[6], yp, make_double2(-s0v.y, s0v.x));
  }
  if (threadIdx.x == 0)
    for (int q = 0; q < 3; ++q) {  // tau_q1 lift entries of -nu d/dz(lift)
      const double2 xt = X[4 * N + 2 * q];
      cjmul_add(&v[2], Y[q * N + A.lift_row], make_double2(A.lift_val * xt.x, A.lift_val * xt.y));
    }
  block_sum<8, kEvpWarps>(v, red);
  if (threadIdx.x == 0) {
    double* o = A.out + (size_t)p * kEvpOut;
    const double dr = v[0], di = v[1], dd = dr * dr + di * di;
    const double sc[3] = {1.0 / (Re * Re), 1.0, 1.0};
    for (int t = 0; t < 3; ++t) {
      const double nr = sc[t] * v[2 + 2 * t], ni = sc[t] * v[3 + 2 * t];
      // -num / den
      o[2 + 2 * t] = dd > 0.0 ? -(nr * dr + ni * di) / dd : 0.0;
      o[3 + 2 * t] = dd > 0.0 ? -(ni * dr - nr * di) / dd : 0.0;
    }
  }
}

struct ShearEvp : EqImpl {
  int N = 0, H = 0, nv = 0, base = 0, Pmax = 0;
  rbhost::Operators ops;
  int kl = 0, ku = 0;
  int sms = 0;
  DevBuf band, XY, args, mats, phi;

  ~ShearEvp() override {
    for (DevBuf* b : {&band, &XY, &args, &mats, &phi}) b->release();
  }

  size_t state_len(int which) const override { return which == 0 ? (size_t)Pmax * H * 2 : 0; }

  spadj_status init(Problem* p) {
    const spadj_desc& d = p->desc;
    N = d.n[2];
    base = (int)d.params[0];
    Pmax = d.batch;
    if (N < 8 || N > kEvpMaxN)
      return p->fail(SPADJ_ERR_INVALID, "shear evp: need 8 <= n[2] <= " + std::to_string(kEvpMaxN));
    if ((base != 0 && base != 1) || (double)base != d.params[0])
      return p->fail(SPADJ_ERR_INVALID, "shear evp: params[0] must be 0 (plane Couette) or 1 (plane Poiseuille)");
    H = 3 * N;
    nv = 4 * N + 7;
    ops = rbhost::build_operators(N, 3 * N / 2, 1.0);
    std::vector<double> Um, UP;
    couhost::base_flow(ops, base, Um, UP);
    int l[2], u[2];
    std::vector<couhost::BandEntry> E[2];
    for (int k = 0; k < 2; ++k) E[k] = couhost::band_parts(ops, Um, UP, k == 1, l[k], u[k]);
    kl = std::max(l[0], l[1]);
    ku = std::max(u[0], u[1]);
    if (kl > kEvpMaxLower || kl + ku > kEvpMaxUpper) return p->fail(SPADJ_ERR_UNSUPPORTED, "shear evp: the pencil's band is wider than supported");
    const int w = kl + ku + 1;
    const size_t part = (size_t)couhost::kBandParts * nv * w;
    std::vector<double> m;
    m.reserve(4 * (size_t)N * N + 6 * (size_t)N + 2 * part);
    m.insert(m.end(), ops.SS.begin(), ops.SS.end());
    m.insert(m.end(), ops.DD.begin(), ops.DD.end());
    m.insert(m.end(), Um.begin(), Um.end());
    m.insert(m.end(), ops.S0.begin(), ops.S0.end());
    // S1S0's band, the pressure recombination, and the parts of the banded pencil (both kinds of pencil at the same
    // widths)
    for (int n = 0; n < N; ++n)
      for (int d = 0; d < 5; ++d) m.push_back(n + d < N ? ops.SS[(size_t)n * N + n + d] : 0.0);
    for (int n = 0; n < N; ++n) m.push_back(n % 2 == 0 ? couhost::pressure_weight(n) : 0.0);
    for (int k = 0; k < 2; ++k) {  // entry (i, k) of part t at ((t nv) + i) w + k - i + kl
      const size_t at = m.size();
      m.resize(at + part, 0.0);
      for (const couhost::BandEntry& e : E[k]) m[at + ((size_t)e.t * nv + e.i) * w + (e.k - e.i + kl)] = e.v;
    }
    SPADJ_CUDA_TRY(p, mats.ensure(sizeof(double) * m.size()));
    SPADJ_CUDA_TRY(p, cudaMemcpy(mats.ptr, m.data(), sizeof(double) * m.size(), cudaMemcpyHostToDevice));
    int dev = 0;
    SPADJ_CUDA_TRY(p, cudaGetDevice(&dev));
    SPADJ_CUDA_TRY(p, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    SPADJ_CUDA_TRY(p, raise_smem(evp_iter_kernel, iter_smem(kEvpMaxN, kEvpMaxUpper)));
    return SPADJ_OK;
  }

  // Whether the iterations run with the dense Phi.  Measured (us): a step of up to 152 pencils takes 12.9, 18, 31, 60 and
  // 88 at N = 8, 16, 32, 48, 64 with it and 21.6, 34, 58, 85 and 107 banded (N = 96: 182 and 158), and it costs about
  // 1.8 N + 0.0054 P N^2 to build: one pencil of N = 16 with 30 steps 834 and 1247, 96 of N = 48 with 20 3067 and 2260, with
  // 60 5489 and 5653.  With more pencils than SMs the banded CTAs share an SM better: 200 pencils 34 and 43 a step at
  // N = 16, 61 and 74 at 32, 118 and 106 at 48; 400 of N = 24 78 and 81, for 1400 to build.
  bool dense_iterations(int P, int n_iter) const {
    if (P > sms) return N <= 32 && 4ll * n_iter >= 5ll * P;
    return N <= kDenseMaxN && n_iter >= 5.0 + 0.1 * N + 3e-4 * P * N * N;
  }

  spadj_status eigen(Problem* p, int P, const double* prm, const double* shift, int n_iter, double* x, double* psi,
                     double* out) {
    if (P < 1 || P > Pmax) return p->fail(SPADJ_ERR_INVALID, "eigen: n_pencils must be in 1..batch");
    if (n_iter < 1) return p->fail(SPADJ_ERR_INVALID, "eigen: n_iter < 1");
    for (int i = 0; i < P; ++i)
      if (!(prm[3 * i + 2] > 0.0) || !std::isfinite(prm[3 * i]) || !std::isfinite(prm[3 * i + 1]))
        return p->fail(SPADJ_ERR_INVALID, "eigen: need finite wavenumbers and Re > 0");
    EvpBand S{};
    S.N = N; S.nv = nv; S.nvp = evp_padded(nv); S.kl = kl; S.ku = ku;
    const int w = kl + ku + 1, kuf = kl + ku;
    const size_t nn = (size_t)N * N, part = (size_t)couhost::kBandParts * nv * w, ns = 2 * (size_t)P * S.nvp;
    // per call: the arguments and flags, and the systems
    SPADJ_CUDA_TRY(p, args.ensure(sizeof(double) * 5 * P + sizeof(int) * (3 * (size_t)P + 1)));
    SPADJ_CUDA_TRY(p, band.ensure((sizeof(double2) * (w + kl + kuf + 1) + 1) * ns));
    SPADJ_CUDA_TRY(p, XY.ensure(sizeof(double2) * (size_t)P * 2 * nv));
    double* prmd = args.as<double>();
    double* shiftd = prmd + 3 * P;
    int* flags = reinterpret_cast<int*>(shiftd + 2 * P);
    SPADJ_CUDA_TRY(p, cudaMemcpyAsync(prmd, prm, sizeof(double) * 3 * P, cudaMemcpyHostToDevice, p->stream));
    SPADJ_CUDA_TRY(p, cudaMemcpyAsync(shiftd, shift, sizeof(double) * 2 * P, cudaMemcpyHostToDevice, p->stream));
    SPADJ_CUDA_TRY(p, cudaMemsetAsync(flags, 0, sizeof(int) * (P + 1), p->stream));
    const double* ssb = mats.as<double>() + 4 * nn;
    S.E0 = ssb + 6 * N;
    S.E1 = S.E0 + part;
    S.prm = prmd;
    S.shift = shiftd;
    S.B = band.as<double2>();
    S.L = S.B + ns * w;
    S.U = S.L + ns * kl;
    S.dinv = S.U + ns * kuf;
    S.piv = reinterpret_cast<unsigned char*>(S.dinv + ns);
    S.bad = flags;
    S.width = flags + P + 1;
    spadj_status s;
    cudaEvent_t t0 = p->tic();
    evp_assemble_kernel<<<2 * P, kEvpThreads, 0, p->stream>>>(S);
    if ((s = check_launch(p, "evp assemble")) != SPADJ_OK) return s;
    const size_t lsmem = sizeof(double2) * ((size_t)(kl + 3) * (w + 1) + 64) + sizeof(int) * (68 + kl + 3);
    evp_lu_kernel<<<2 * P, kEvpThreads, lsmem, p->stream>>>(S);
    if ((s = check_launch(p, "evp factorise")) != SPADJ_OK) return s;
    EvpIterArgs ia{};
    ia.S = S;
    ia.ssb = ssb;
    ia.pw = ssb + 5 * N;
    ia.x = reinterpret_cast<double2*>(x);
    ia.psi = reinterpret_cast<double2*>(psi);
    ia.XY = XY.as<double2>();
    ia.out = out;
    ia.n_iter = n_iter;
    double dense_flops = 0.0;  // the operator's columns, and its two products per step (16 flops per entry)
    if (dense_iterations(P, n_iter)) {
      if (phi.ensure(sizeof(double2) * (size_t)P * H * H) == cudaSuccess) {
        const int blocks = (H + kPhiWarps - 1) / kPhiWarps;
        evp_phi_kernel<<<P * blocks, 32 * kPhiWarps, phi_smem(S.nvp), p->stream>>>(S, P, ssb, phi.as<double2>());
        if ((s = check_launch(p, "evp operator")) != SPADJ_OK) return s;
        EvpDenseArgs da{phi.as<double2>(), ia.x, ia.psi, shiftd, flags, out, H, n_iter};
        const size_t dsmem = sizeof(double2) * (size_t)(3 + kEvpWarps) * H + sizeof(double) * kEvpWarps * 6;
        kEvpDense[(H + 31) / 32 - 1]<<<P, kEvpThreads, dsmem, p->stream>>>(da);
        if ((s = check_launch(p, "evp dense iterate")) != SPADJ_OK) return s;
        ia.n_iter = 0;
        dense_flops = (8.0 * nv * (kl + ku + 1.0) + 16.0 * H * n_iter) * H * P;
      } else {
        cudaGetLastError();  // no memory for the operators: the banded iterations need none
      }
    }
    evp_iter_kernel<<<P, kIterThreads, iter_smem(N, kuf), p->stream>>>(ia);
    // two factorisations, and two banded solves per step and for the eigenvectors, 8 flops per factor entry
    p->toc(t0, KC_SOLVE, 16.0 * nv * ((double)kl * (kl + ku) + (kl + ku + 1.0) * (ia.n_iter + 1)) * P + dense_flops);
    if ((s = check_launch(p, "evp iterate")) != SPADJ_OK) return s;
    EvpSensArgs sa{};
    sa.XY = XY.as<double2>();
    sa.prm = prmd;
    sa.bad = flags + P;
    sa.SS = mats.as<double>();
    sa.DD = sa.SS + nn;
    sa.Um = sa.DD + nn;
    sa.S0 = sa.Um + nn;
    sa.out = out;
    sa.N = N;
    sa.nv = nv;
    sa.lift_row = ops.lift_row;
    sa.lift_val = ops.lift_val;
    const size_t ssmem = sizeof(double2) * 2 * nv + sizeof(double) * kEvpWarps * 8;
    cudaEvent_t t2 = p->tic();
    evp_sens_kernel<<<P, kEvpThreads, ssmem, p->stream>>>(sa);
    p->toc(t2, KC_OBJECTIVE, (12.0 * 4.0 * N * N + 64.0 * N) * P);
    if ((s = check_launch(p, "evp sensitivity")) != SPADJ_OK) return s;
    std::vector<int> bad(P + 1);
    SPADJ_CUDA_TRY(p, cudaMemcpyAsync(bad.data(), flags, sizeof(int) * (P + 1), cudaMemcpyDeviceToHost, p->stream));
    SPADJ_CUDA_TRY(p, cudaStreamSynchronize(p->stream));
    for (int i = 0; i < P; ++i)
      if (bad[i]) return p->fail(SPADJ_ERR_INVALID, "eigen: singular shifted pencil matrix at pencil " + std::to_string(i));
    return SPADJ_OK;
  }

  // ---- operations of the time-dependent problems are not defined here ------------------------
  spadj_status unsupported(Problem* p, const char* what) {
    return p->fail(SPADJ_ERR_UNSUPPORTED, std::string(what) + ": not defined for the shear-flow eigenproblem");
  }
  spadj_status transform(Problem* p, int, const double*, double*) override { return unsupported(p, "transform"); }
  spadj_status eval_F(Problem* p, int, const double*, const double*, double*) override {
    return unsupported(p, "eval_F");
  }
  spadj_status forward(Problem* p, int, const double*, double*, double*) override { return unsupported(p, "forward"); }
  spadj_status tangent(Problem* p, int, const double*, const double*, double*) override {
    return unsupported(p, "tangent");
  }
  spadj_status adjoint(Problem* p, int, const double*, const double*, double*, double*) override {
    return unsupported(p, "adjoint");
  }
  spadj_status objective(Problem* p, int, const double*, const double*, double*, double*) override {
    return unsupported(p, "objective");
  }
  spadj_status gradient(Problem* p, const double*, int, int, const double*, int, double*, double*, double*) override {
    return unsupported(p, "gradient");
  }
  spadj_status vjp(Problem* p, const double*, int, int, const std::vector<int>&, const double*, double*) override {
    return unsupported(p, "vjp");
  }
};

}  // namespace

EqImpl* make_shear_evp(Problem* p, spadj_status* st) {
  ShearEvp* e = new ShearEvp();
  *st = e->init(p);
  if (*st != SPADJ_OK) {
    delete e;
    return nullptr;
  }
  return e;
}

spadj_status evp_eigen(EqImpl* impl, Problem* p, int P, const double* prm, const double* shift, int n_iter, double* x,
                       double* psi, double* out) {
  ShearEvp* e = dynamic_cast<ShearEvp*>(impl);
  if (!e) return p->fail(SPADJ_ERR_UNSUPPORTED, "eigen: only defined for the shear-flow eigenproblem");
  return e->eigen(p, P, prm, shift, n_iter, x, psi, out);
}

}  // namespace spadj
