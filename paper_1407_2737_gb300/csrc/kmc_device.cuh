// kmc_device.cuh -- device building blocks of the kMC step (sm_103a): the
// Philox4x32-10 draw and the per-NP update of steps iii-vii of Sec. II.1
// (the bulk-copy staging is in kmc_stage.cuh).
#pragma once
#include <stdint.h>

#include <type_traits>

#include "kmc_pair.cuh"
#include "kmc_stage.cuh"
#include "kmc_types.h"

namespace kmc {

// Grid of step iv: theta_j = 2 pi (j + 1/2) / 200 and (sin, cos) of it,
// written once per device by init_device (kmc_step.cu, the only translation
// unit that includes this header).
// (16-byte aligned: the FP32 step kernels copy them to shared memory in bulk)
__device__ __align__(16) float g_theta_f[kGrid];
__device__ __align__(16) float2 g_sc_f[kGrid];
// The same sin and cos in two arrays of their own, node j at j mod kGrid for
// j < kGridPad, so that the FP32 scan reads two consecutive nodes as one
// packed pair, past the end of the grid too.
constexpr int kGridPad = kGrid + 16;
__device__ __align__(16) float g_ss_f[kGridPad];
__device__ __align__(16) float g_cc_f[kGridPad];
__device__ double g_theta_d[kGrid];
__device__ double2 g_sc_d[kGrid];

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): ten rounds of two
// 32x32->64 multiplications with the Philox multipliers; the key advances by
// the Weyl constants after every round.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    k.x += 0x9E3779B9u;
    k.y += 0xBB67AE85u;
  }
  return c;
}

// 53-bit uniform in [0,1) for (seed, global step, NP within lysosome, lysosome).
__device__ __forceinline__ double kmc_uniform(unsigned long long seed, long long step,
                                              int np, int lys) {
  const unsigned long long s = static_cast<unsigned long long>(step);
  const uint4 w = philox4x32_10(
      make_uint4(static_cast<uint32_t>(s), static_cast<uint32_t>(s >> 32),
                 static_cast<uint32_t>(np), static_cast<uint32_t>(lys)),
      make_uint2(static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32)));
  const unsigned long long bits =
      (static_cast<unsigned long long>(w.x) << 21) ^ static_cast<unsigned long long>(w.y >> 11);
  return static_cast<double>(bits) * 0x1.0p-53;
}

// ---------------------------------------------------------------------------
// Steps iii-vii for one NP, in reduced units (kmc_types.h).

template <typename R>
struct Prec;
template <>
struct Prec<float> {
  static constexpr float two_pi = 6.28318530717958647692f;
  static constexpr float plane_tol = 1e-6f;   // |b x a| below this: plane from m
  // Newton stops once a step is below newton_tol (absolute, on the offset in
  // a cell of 0.0314 rad). With de/dth and its derivative in FP32 the step
  // itself carries rounding noise of order 1e-8..1e-7 rad, so the tolerance
  // sits above it: a tighter one is never met and every root runs to
  // newton_max. From the secant start the convergence is quadratic, so the
  // root is then within rounding (~1e-7 rad) after 2-3 steps.
  static constexpr float newton_tol = 3e-7f;
  static constexpr int newton_max = 6;
  __device__ static float div(float a, float b) { return __fdividef(a, b); }
  __device__ static float theta(int j) { return g_theta_f[j]; }
  __device__ static float2 sc(int j) { return g_sc_f[j]; }
  // sin and cos of 0 <= d <= 2 pi / 200 by their Taylor series (error < 1e-11)
  __device__ static void sincos_small(float d, float &s, float &c) {
    const float d2 = d * d;
    s = d * fmaf(d2, fmaf(d2, 1.0f / 120.0f, -1.0f / 6.0f), 1.0f);
    c = fmaf(d2, fmaf(d2, 1.0f / 24.0f, -0.5f), 1.0f);
  }
};
template <>
struct Prec<double> {
  static constexpr double two_pi = 6.283185307179586476925286766559;
  static constexpr double plane_tol = 1e-12;
  static constexpr double newton_tol = 1e-14;
  static constexpr int newton_max = 100;
  __device__ static double div(double a, double b) { return a / b; }
  __device__ static double theta(int j) { return g_theta_d[j]; }
  __device__ static double2 sc(int j) { return g_sc_d[j]; }
  // Taylor series to d^7 / d^8: the next terms are below 8.3e-20 and 2.6e-22
  // for d <= 2 pi / 200, a thousandth of the rounding of the sums
  __device__ static void sincos_small(double d, double &s, double &c) {
    const double d2 = d * d;
    s = d * fma(d2, fma(d2, fma(d2, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), 1.0);
    c = fma(d2, fma(d2, fma(d2, fma(d2, 1.0 / 40320.0, -1.0 / 720.0), 1.0 / 24.0), -0.5), 1.0);
  }
};

// Copy of the grid of step iv in shared memory, filled by every block at its
// start (the pair loop hides the loads); the scan reads one node per warp
// (a broadcast), Newton one node per thread.
struct ScanPairs {
  float ss[kGridPad], cc[kGridPad];  // g_ss_f, g_cc_f (both precisions scan in FP32)
};
template <typename R>
struct GridTables : ScanPairs {
  typename std::conditional<std::is_same<R, float>::value, float2, double2>::type sc[kGrid];
  R th[kGrid];
  __device__ void load() {
    for (int j = threadIdx.x; j < kGrid; j += blockDim.x) {
      sc[j] = Prec<R>::sc(j);
      th[j] = Prec<R>::theta(j);
    }
    for (int j = threadIdx.x; j < kGridPad; j += blockDim.x) {
      ss[j] = g_ss_f[j];
      cc[j] = g_cc_f[j];
    }
  }
};
static_assert(sizeof(GridTables<float>::sc) % 16 == 0 && sizeof(GridTables<float>::th) % 16 == 0 &&
                  sizeof(ScanPairs::ss) % 16 == 0 && sizeof(ScanPairs) % 16 == 0,
              "the FP32 tables are copied in bulk");

// de/dth of Eq. 2 at (sin, cos) = (s, c): s (2k c + b cos phi) - b sin phi c,
// with its roundings spelled out so that every evaluation at a node gives the
// same bits wherever the compiler places it (the scan tests the sign of values
// that can sit within rounding of zero, and evaluates each node twice).
__device__ __forceinline__ float profile_d1(float k2, float bc, float bs, float s, float c) {
  return __fmaf_rn(s, __fmaf_rn(k2, c, bc), -__fmul_rn(bs, c));
}
__device__ __forceinline__ double profile_d1(double k2, double bc, double bs, double s,
                                             double c) {
  return __fma_rn(s, __fma_rn(k2, c, bc), -__dmul_rn(bs, c));
}

// Eq. 2 in a working plane: e = k sin^2 th - b cos(th - phi);
// de/dth = 2k s c + b (s cos phi - c sin phi); d2e = 2k (c^2 - s^2) + b (c cos phi + s sin phi).
template <typename R>
struct Profile {
  R k2;  // 2k
  R k;
  R bc;  // b cos phi
  R bs;  // b sin phi
  __device__ R d1(R s, R c) const { return profile_d1(k2, bc, bs, s, c); }
  __device__ R d2(R s, R c) const { return k2 * (c * c - s * s) + fma(bc, c, bs * s); }
  __device__ R e(R s, R c) const { return k * s * s - fma(bc, c, bs * s); }
};

// Newton's method with bisection fallback for the root of de/dth inside grid
// cell [theta_j, theta_j + h], as offset d from theta_j. dlo, dhi = de/dth at
// theta_j and theta_j + h (opposite signs); the first iterate is the secant
// point, so that two or three Newton steps reach the root.
template <typename R>
__device__ __forceinline__ R refine_in_cell(const Profile<R> &pf, R S0, R C0, R h, R dlo,
                                            R dhi, R &s_out, R &c_out) {
  R lo = R(0), hi = h;
  R x = (dlo != dhi) ? h * Prec<R>::div(dlo, dlo - dhi) : R(0.5) * h;
  if (!(x > lo && x < hi)) x = R(0.5) * h;
  for (int it = 0; it < Prec<R>::newton_max; ++it) {
    R sd, cd;
    Prec<R>::sincos_small(x, sd, cd);
    const R s = fma(S0, cd, C0 * sd), c = fma(C0, cd, -S0 * sd);
    const R d = pf.d1(s, c);
    if (d == R(0)) break;
    if ((d < R(0)) == (dlo < R(0))) {
      lo = x;
      dlo = d;
    } else {
      hi = x;
    }
    const R dd = pf.d2(s, c);
    R xn = (dd != R(0)) ? x - Prec<R>::div(d, dd) : R(0.5) * (lo + hi);
    // Converged: the step is below the tolerance. Tested before the bracket
    // safeguard, because a step that rounds to nothing leaves xn on the
    // bracket end that x itself just became, and the safeguard would then
    // bisect away from the root it has found.
    if (fabs(xn - x) < Prec<R>::newton_tol) {
      x = xn;
      break;
    }
    if (!(xn > lo && xn < hi)) xn = R(0.5) * (lo + hi);
    const bool done = hi - lo < Prec<R>::newton_tol;
    x = xn;
    if (done) break;
  }
  R sd, cd;
  Prec<R>::sincos_small(x, sd, cd);
  s_out = fma(S0, cd, C0 * sd);
  c_out = fma(C0, cd, -S0 * sd);
  return x;
}

// Start of 1/sqrt(x): the hardware's approximation, whose low word is zero.
__device__ __forceinline__ double rsqrt_seed(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}

// 1/sqrt(r2), and 0 for r2 = 0 (a self pair, or two NPs at one point) or an
// overflowed r2. The seed y has a short mantissa, so y y is exact and e = 1 -
// r2 y^2 is rounded once; the binomial series (1 - e)^(-1/2) = 1 + e/2 + 3/8 e^2
// + ..., cut there (Chebyshev's iteration for y^-2 = r2), leaves 5/16 e^3, far below the
// rounding for a seed good to 2^-20. Fields of single pairs come out as the
// oracle's do, 1e-15 off (sqrt and a division).
__device__ __forceinline__ double rsqrt_pair(double r2) {
  const int hi = __double2hiint(r2);
  const bool none = (hi | __double2loint(r2)) == 0 || hi >= 0x7ff00000;
  double y = rsqrt_seed(r2);
  if (none) {
    y = 0.0;
    r2 = 0.0;
  }
  const double e = fma(-r2, y * y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// sqrt(x) and 1/sqrt(x) to an ulp or two, for x >= 0: a chain of six dependent
// FP64 operations where sqrt and a division take about thirty. Outside the seed's
// comfortable range, the functions themselves.
__device__ __forceinline__ double sqrt_inv(double x, double &inv) {
  if (x > 1e-290 && x < 1e290) {
    inv = rsqrt_pair(x);
    return x * inv;
  }
  const double r = sqrt(x);
  inv = 1.0 / r;
  return r;
}

// FP64 root of de/dth inside grid cell [theta_j, theta_j + h] (left_neg: de/dth
// is negative at theta_j), as offset from theta_j; (S0, C0) = sin, cos of
// theta_j, (S0f, C0f) the same in FP32. FP64 instructions issue at 1/64 of the
// FP32 rate here, and a dependent one takes 60 cycles or so, so the search runs in
// FP32 until its rounding (about 1e-8 rad from the cell's middle in three Newton
// steps) and FP64 only finishes, in one evaluation: the step with its second-order
// term, d = D + C D^2 with D = f / f' and C = f'' / (2 f') (C in FP32: it scales a
// correction of 1e-15), leaves about C^2 D^3, below 1e-18 under the conditions
// tested. The divisor is an FP32 reciprocal with one FP64 Newton step (1e-14
// relative). sin and cos move with the step to second order (the next term is
// below 2e-19). Where that does not hold (a near-double root, profiles outside
// FP32's range) the safeguarded Newton iteration of refine_in_cell runs, with its
// bracket, tolerance and cap. With the FP32 sign pass (fp64_signs) it took the
// FP64 step from 49.2 to 38.6 us at 100 NPs and from 284 to 241 us at 2000, with
// two to three evaluations each; one evaluation took the mean mode's wells from
// 350 to 291 us (2000 NPs x 200 steps).
__device__ __forceinline__ double root_in_cell(const Profile<double> &pf, double S0, double C0,
                                               float S0f, float C0f, double h, bool left_neg,
                                               double &s_out, double &c_out) {
  double x;
  const float k2 = static_cast<float>(pf.k2);
  {
    const float bc = static_cast<float>(pf.bc), bs = static_cast<float>(pf.bs),
                hf = static_cast<float>(h);
    float xf = 0.5f * hf;
#pragma unroll
    for (int it = 0; it < 3; ++it) {
      float sd, cd;
      Prec<float>::sincos_small(xf, sd, cd);
      const float s = fmaf(S0f, cd, C0f * sd), c = fmaf(C0f, cd, -S0f * sd);
      const float d = profile_d1(k2, bc, bs, s, c);
      const float dd = k2 * (c * c - s * s) + fmaf(bc, c, bs * s);
      xf = fminf(fmaxf(xf - __fdividef(d, dd), 0.0f), hf);  // (a NaN becomes 0)
    }
    x = static_cast<double>(xf);
  }
  double lo = 0.0, hi = h;
  if (!(x > lo && x < hi)) x = 0.5 * h;
  for (int it = 0; it < Prec<double>::newton_max; ++it) {
    double sd, cd;
    Prec<double>::sincos_small(x, sd, cd);
    const double s = fma(S0, cd, C0 * sd), c = fma(C0, cd, -S0 * sd);
    const double d = pf.d1(s, c);
    if (d == 0.0) {
      s_out = s;
      c_out = c;
      return x;
    }
    const double dd = pf.d2(s, c);
    const float ddf = static_cast<float>(dd), df = static_cast<float>(d);
    const float r = __frcp_rn(ddf), stepf = df * r;
    // C D, with f'' = -3 (2k) sin cos at the root
    const float cstep = -1.5f * k2 * static_cast<float>(s) * static_cast<float>(c) * r * stepf;
    const bool range = fabsf(ddf) > 1e-30f && fabsf(ddf) < 1e30f;
    if (range && fabsf(stepf) < 1e-6f && fabsf(cstep) < 1e-6f && x > 2e-6 && x < h - 2e-6) {
      const double rd = static_cast<double>(r);
      const double step = d * fma(rd, fma(-dd, rd, 1.0), rd);
      const double full = fma(static_cast<double>(cstep), step, step);
      s_out = fma(-full, fma(0.5 * full, s, c), s);
      c_out = fma(full, fma(-0.5 * full, c, s), c);
      return x - full;
    }
    if ((d < 0.0) == left_neg)
      lo = x;
    else
      hi = x;
    const double step = range ? d * static_cast<double>(r) : d / dd;
    double xn = x - step;
    if (fabs(step) < Prec<double>::newton_tol) {
      s_out = fma(-step, c, s);
      c_out = fma(step, s, c);
      return xn;
    }
    if (!(xn > lo && xn < hi)) xn = 0.5 * (lo + hi);
    const bool done = hi - lo < Prec<double>::newton_tol;
    x = xn;
    if (done) break;
  }
  double sd, cd;
  Prec<double>::sincos_small(x, sd, cd);
  s_out = fma(S0, cd, C0 * sd);
  c_out = fma(C0, cd, -S0 * sd);
  return x;
}

// FP32 copy of a profile for the FP64 path's sign pass, with the bound on its
// error. With u = 2^-24, de/dth formed in FP32 from rounded coefficients and
// table entries errs by at most 6 u (|2k| + |b cos phi| + |b sin phi|) (one
// rounding each of the coefficient, the sine, the cosine and the operations);
// guard is 16.8 u times that sum. A value beyond the guard has the FP64 sign;
// the others are evaluated in FP64. Outside FP32's comfortable range (or not
// finite) the guard is infinite: every node is evaluated in FP64.
struct SignProfile {
  float k2, bc, nbs, guard;
  __device__ SignProfile(double k2d, double bcd, double bsd) {
    k2 = static_cast<float>(k2d);
    bc = static_cast<float>(bcd);
    nbs = static_cast<float>(-bsd);
    const float sum = fabsf(k2) + fabsf(bc) + fabsf(nbs);
    guard = (sum > 1e-25f && sum < 1e30f) ? 1e-6f * sum : INFINITY;
  }
};

// Nodes per segment of the scan at most.
constexpr int kMaxSeg = 50;

// FP32 sign pass over kPairBatch consecutive nodes j0 + q0 .. (j0 + q0 even):
// two nodes per packed instruction, read as pairs from the split sin and cos
// tables, each node with profile_d1's roundings (s (2k c + b cos phi) +
// (-b sin phi) c; a packed operation rounds each half as the scalar one), so
// the signs are those of the scalar pass. Bit q of the result: node q0 + q.
constexpr int kPairBatch = 14;
__device__ __forceinline__ unsigned long long pair_signs(const ScanPairs &tab, f2 K2, f2 BC,
                                                         f2 NBS, int j0, int q0) {
  unsigned bits = 0;
#pragma unroll
  for (int u = 0; u < kPairBatch; u += 2) {
    const int j = j0 + q0 + u;  // < kGridPad: the tables repeat the grid past its end
    const f2 s = *reinterpret_cast<const f2 *>(&tab.ss[j]);
    const f2 c = *reinterpret_cast<const f2 *>(&tab.cc[j]);
    const f2 d = fma2(s, fma2(K2, c, BC), mul2(NBS, c));
    float dl, dh;
    upk(d, dl, dh);
    bits |= (static_cast<unsigned>(dl < 0.f) << u) | (static_cast<unsigned>(dh < 0.f) << (u + 1));
  }
  return static_cast<unsigned long long>(bits) << q0;
}

// Signs of the FP64 de/dth at nodes j0 .. j0 + len (bit q: negative at node j0 +
// q, cyclically; len <= kMaxSeg): the FP32 pass, then FP64 at the nodes whose
// FP32 value lies within its error bound (SignProfile), so that every bit is
// that of the FP64 evaluation. Such nodes are rare (a root within about 1e-6 rad
// of one), and the FP64 pipe, at 1/64 of the FP32 rate, stays free.
__device__ __forceinline__ unsigned long long fp64_signs(const GridTables<double> &tab,
                                                         const Profile<double> &pf,
                                                         const SignProfile &sp, int j0, int len) {
  const f2 K2 = pk(sp.k2, sp.k2), BC = pk(sp.bc, sp.bc), NBS = pk(sp.nbs, sp.nbs);
  const int odd = j0 & 1, je = j0 - odd, le = len + odd;  // the packed pairs start on even nodes
  unsigned long long neg = 0, unsure = 0;
#pragma unroll 1
  for (int q0 = 0; q0 <= le; q0 += kPairBatch) {
    unsigned nb = 0, ub = 0;
#pragma unroll
    for (int u = 0; u < kPairBatch; u += 2) {
      const int j = je + q0 + u;  // < kGridPad: the tables repeat the grid past its end
      const f2 s = *reinterpret_cast<const f2 *>(&tab.ss[j]);
      const f2 c = *reinterpret_cast<const f2 *>(&tab.cc[j]);
      float dl, dh;
      upk(fma2(s, fma2(K2, c, BC), mul2(NBS, c)), dl, dh);
      nb |= (static_cast<unsigned>(dl < 0.f) << u) | (static_cast<unsigned>(dh < 0.f) << (u + 1));
      ub |= (static_cast<unsigned>(!(fabsf(dl) > sp.guard)) << u) |
            (static_cast<unsigned>(!(fabsf(dh) > sp.guard)) << (u + 1));
    }
    neg |= static_cast<unsigned long long>(nb) << q0;
    unsure |= static_cast<unsigned long long>(ub) << q0;
  }
  neg >>= odd;
  unsure = (unsure >> odd) & ((2ull << len) - 1);
  while (unsure) {
    const int q = __ffsll(static_cast<long long>(unsure)) - 1;
    unsure &= unsure - 1;
    const int j = j0 + q < kGrid ? j0 + q : j0 + q - kGrid;
    const bool n = pf.d1(tab.sc[j].x, tab.sc[j].y) < 0.0;
    neg = (neg & ~(1ull << q)) | (static_cast<unsigned long long>(n) << q);
  }
  return neg;
}

// 1 if x lies on the arc running counter-clockwise from just after `from` up
// to and including `to` (all angles in [0, 2 pi)).
template <typename R>
__device__ __forceinline__ bool on_arc(R x, R from, R to) {
  R dx = x - from, dt = to - from;
  if (dx < R(0)) dx += Prec<R>::two_pi;
  if (dt < R(0)) dt += Prec<R>::two_pi;
  return dx > R(0) && dx <= dt;
}

}  // namespace kmc
