// Broken-line refit of the fitted tracks (Sec. 2.2.1 and Fig. 2: a fit of each picked
// group of hits determines the track parameters; the broken-line form is V. Blobel,
// NIM A566 (2006) 14).  The track is its offsets from the circle + line fit at the n
// hits, joined by pieces of one common curvature; the direction changes at the hits are
// multiple-scattering kinks weighted by their expected variance.  The library's reading:
//   [B1] reference = the track's circle + line fit; for hit i, s_i = arc length from
//        the closest approach to the hit's radial projection on the reference circle,
//        eps_i = signed distance from that circle (positive to the left of the motion);
//   [B2] transverse unknowns u_1..u_n, dkappa; between hits u'' + kappa0^2 u = dkappa
//        (first-order departure of a circle from the reference circle), so a segment of
//        length h has end slopes a (u_b - c u_a) - a g dkappa and a (c u_b - u_a) +
//        a g dkappa, c = cos(kappa0 h), a = kappa0 / sin(kappa0 h), g = 2 sin^2(kappa0
//        h / 2) / kappa0^2; kink beta_i = slope after - slope before; chi2_T = sum
//        (eps_i - u_i)^2 / (10 um)^2 + sum beta_i^2 / vartheta_i^2;
//   [B3] z is linear in the arc length along the fitted transverse path, s'_i = s_i -
//        kappa0 int_0^{s_i} u (per segment the parabola through its end offsets with
//        second derivative dkappa); unknowns w_i = z offsets from z0 + cot s', kinks of
//        the straight pieces, errors 20 um (barrel z) and |cot| 20 um (disk r);
//   [B4] Highland theta0 = 13.6 MeV / p sqrt(t) (1 + 0.038 ln t), p and the incidence
//        from the reference, t = x/X0 / cos(incidence) (barrel: direction . radial
//        direction; disk: |cos theta|; floored at 1e-3); vartheta^2 = theta0^2 /
//        sin^2 theta, tau^2 = theta0^2 / sin^4 theta;
//   [B5] parameters at the closest approach continue the first segment backwards:
//        kappa0 + dkappa, phi0 + u'(0), d0 - u(0), cot0 + w'_1, z0 + w(0);
//   [B6] a reference with a non-finite value, |kappa0| < 1e-7 /cm or hits not strictly
//        ordered along s (a step <= 1e-6 cm) keeps its circle + line fit;
//   [B7] passes repeat with the previous result as the reference while a pass changes
//        the curvature by more than 1e-3 relative, at most four (one pass is linear in
//        the departures from its reference, and the first moves low-momentum forward
//        tracks by up to 13 % from the circle fit).
//
// One thread per track.  The residuals are micrometres on coordinates of tens of
// centimetres, and the normal equations mix weights of 1e6 (hits) and 1e4..1e8 (kinks):
// 24 bits are too few.  GB300 issues a float64 operation at 1/64 of the float32 rate, so the
// numbers are pairs of floats (F2, 48 bits: 7 float32 operations for a product, 11 for a
// sum); a track whose kinks outweigh its hits by more than 1e7 (so that too few of the 48
// bits are left for the hits: kStiffMax), or whose pass leaves the range of float32 anywhere
// (a result that is not finite), is done in float64 by the same template.  On 211k tracks, of
// events of 800 to 4400 particles, the errors against a 64-bit reference are the ones that a
// pass in float64 has (the results of the two differ by at most 6e-8 of a parameter's spread);
// they come from the turning angle below.  The geometry is written so that nothing cancels:
// with q = (sin phi0, -cos phi0), a hit p has eps = N / (1 + |kappa0| |p -
// c|), N = d0 (2 - kappa0 d0) - kappa0 p.p + 2 (kappa0 d0 - 1) p.q, and turning angle
// atan2(p.(cos phi0, sin phi0) / kappa0, (1 + kappa0 (p.q - d0)) / kappa0^2) (the cross and
// scalar products of the closest approach and p seen from c), c the circle's centre.  The
// kink variances only need a few significant digits and are formed in float32, and so is
// each hit's turning angle (relative error ~1e-7: under 0.1 um of arc on 30 cm).  The
// segment trigonometry (|kappa0 h| <= 0.5 on nearly every track) uses the Taylor series of
// cos x, sin x / x and (1 - cos x) / x^2, the terms from x^8 on in float32 (truncation and
// rounding below 1e-14), the library in float64 beyond.
// The two planes' least squares have the same form (a kink couples three neighbouring
// hits; the transverse one has the curvature correction besides), so one routine sets up
// and eliminates both, hit by hit, three rows and the curvature's at a time.  All loops over
// the hits stay loops, their arrays in shared memory: unrolled over the largest ntuplet the
// pass was 7400 instructions that every warp ran once, and 7 of 11 cycles per instruction
// went to instruction fetch.
// Each pass is its own launch over the tracks the previous pass listed as still moving (a
// warp-aggregated append), so a warp never waits for the slowest of its tracks; the
// reference of a later pass is the float32 track the previous pass wrote (the result
// depends on its reference only at second order).
//
// Bound by instruction issue where there are tracks enough (51 % of it active on 59k) and
// by the latency of one pass (20 us) in the later launches.  59k pileup-50 tracks, first
// pass and all four: 31 and 95 us; float64 in registers 297 us (all four); pairs of floats
// in registers, unrolled, 53 and 122 us.
#include <cooperative_groups.h>

#include "brokenline.cuh"

namespace ptca {

namespace {

constexpr int kN = kMaxHits;
constexpr double kSigmaT = 10e-4;  // cm
constexpr double kSigmaL = 20e-4;  // cm
constexpr double kCpt = 0.299792458;
constexpr double kPi = 3.141592653589793238462643383280;

constexpr float kPassTol = 1e-3f;
constexpr int kMaxPasses = 4;
static_assert(kMaxPasses <= kRefitCounters, "one counter per pass");

// ------------------------------------------------------------------ pairs of floats
// h + l with |l| <= ulp(h) / 2, after T. J. Dekker (Numer. Math. 18 (1971) 224).
struct F2 {
  float h, l;
};
__device__ __forceinline__ F2 two_quick(float a, float b) {  // a + b, |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ F2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ F2 operator-(F2 a) { return {-a.h, -a.l}; }
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
  const F2 s = two_sum(a.h, b.h);
  return two_quick(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return a + (-b); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
  const float p = __fmul_rn(a.h, b.h);
  return two_quick(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
// a * b + c
__device__ __forceinline__ F2 mad(F2 a, F2 b, F2 c) {
  const float p = __fmul_rn(a.h, b.h);
  const float e = __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)));
  const F2 s = two_sum(p, c.h);
  return two_quick(s.h, __fadd_rn(s.l, __fadd_rn(e, c.l)));
}
__device__ __forceinline__ F2 recip(F2 a) {
  const float r = __frcp_rn(a.h);
  const float e = __fmaf_rn(-a.l, r, __fmaf_rn(-a.h, r, 1.0f));
  return two_quick(r, __fmul_rn(r, e));
}
__device__ __forceinline__ F2 root(F2 a) {  // a > 0
  const float r = __fsqrt_rn(a.h);
  const float e = __fadd_rn(__fmaf_rn(-r, r, a.h), a.l);
  return two_quick(r, __fdividef(e, 2.0f * r));
}
__device__ __forceinline__ F2 absv(F2 a) { return a.h < 0.0f ? -a : a; }
__device__ __forceinline__ float lead(F2 a) { return a.h; }

__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double recip(double a) { return 1.0 / a; }
__device__ __forceinline__ double root(double a) { return sqrt(a); }
__device__ __forceinline__ double absv(double a) { return fabs(a); }
__device__ __forceinline__ float lead(double a) { return (float)a; }

// Constants and float32 values as T.
template <class T>
__device__ __forceinline__ T num(double c);
template <>
__device__ __forceinline__ F2 num<F2>(double c) {
  const float h = (float)c;
  return {h, (float)(c - (double)h)};
}
template <>
__device__ __forceinline__ double num<double>(double c) {
  return c;
}
template <class T>
__device__ __forceinline__ T val(float f);
template <>
__device__ __forceinline__ F2 val<F2>(float f) {
  return {f, 0.0f};
}
template <>
__device__ __forceinline__ double val<double>(float f) {
  return f;
}

template <class T>
constexpr bool kPairs = false;
template <>
constexpr bool kPairs<F2> = true;
// Largest weight of a kink in the normal equations that pairs of floats take: 1e7 times a hit's
// in the transverse plane (1e6 /cm^2) and 4e7 times a barrel hit's in the longitudinal one
// (2.5e5), less by |cot| / 2 for steep tracks, whose hit errors on a disk, and so the offsets'
// rounding, grow with it.  There the solved offsets are within 3e-9 cm of the exact ones, less
// than the float32 results resolve, and the results equal those of the float64 form to one unit
// in the last place; at 1e10 the offsets were up to 1e-3 of a hit's error away and z0 40 units.
// A track of 1 GeV through 2 % of a radiation length has a weight of 1e4, one of 10 TeV reaches
// the limit; the straight fakes that do make the refit of 64 pileup-200 events, 675k tracks, 458
// instead of 455 us (510 with a tenth of the limit).
constexpr float kStiffMax = 1e13f;

// sin and cos of a float32 angle within +-pi (a track's phi0).
__device__ __forceinline__ void sin_cos(float x, double& s, double& c) { sincos((double)x, &s, &c); }
__device__ __forceinline__ void sin_cos(float x, F2& s, F2& c) {
  // x = k pi/2 + y, |y| <= pi/4 (+ rounding); Taylor series of sin y and cos y, the terms
  // from y^9 / 9! on in float32 (below 3e-7, so their rounding stays below 1e-13 relative)
  const float k = rintf(x * (float)(2.0 / kPi));
  const F2 y = mad(num<F2>(-0.5 * kPi), val<F2>(k), val<F2>(x));
  const F2 t = y * y;
  const float ft = t.h;
  const float ts = (float)(1.0 / 362880) +
                   ft * ((float)(-1.0 / 39916800) + ft * (float)(1.0 / 6227020800.0));
  const float tc = (float)(1.0 / 40320) +
                   ft * ((float)(-1.0 / 3628800) +
                         ft * ((float)(1.0 / 479001600) + ft * (float)(-1.0 / 87178291200.0)));
  F2 a = mad(t, val<F2>(ts), num<F2>(-1.0 / 5040));
  a = mad(t, a, num<F2>(1.0 / 120));
  a = mad(t, a, num<F2>(-1.0 / 6));
  a = mad(t * y, a, y);
  F2 b = mad(t, val<F2>(tc), num<F2>(-1.0 / 720));
  b = mad(t, b, num<F2>(1.0 / 24));
  b = mad(t, b, num<F2>(-1.0 / 2));
  b = mad(t, b, val<F2>(1.0f));
  const int q = (int)k & 3;
  s = (q & 1) ? b : a;
  c = (q & 1) ? a : b;
  if (q & 2) s = -s;
  if (q == 1 || q == 2) c = -c;
}

// cos x, sin x / x and (1 - cos x) / x^2: Taylor series in x^2 for |x| <= 0.5 (the next
// terms are below 1e-15), the library beyond.
__device__ __forceinline__ void trig3_far(double x, double& c, double& sc, double& vc) {
  double sn;
  sincos(x, &sn, &c);
  sc = sn / x;
  vc = (1.0 - c) / (x * x);
}
__device__ __noinline__ void trig3_far(F2 x, F2& c, F2& sc, F2& vc) {
  double a, b, d;
  trig3_far((double)x.h + (double)x.l, a, b, d);
  c = num<F2>(a);
  sc = num<F2>(b);
  vc = num<F2>(d);
}
template <class T>
__device__ __forceinline__ void trig3(T x, T& c, T& sc, T& vc) {
  if (fabsf(lead(x)) <= 0.5f) {
    const T t = x * x;
    const float f = lead(t);
    // from t^4 on: below 1e-8 and 1e-9 of the sums
    const T hs = val<T>((float)(1.0 / 362880) +
                        f * ((float)(-1.0 / 39916800) + f * (float)(1.0 / 6227020800.0)));
    const T hv = val<T>((float)(1.0 / 3628800) +
                        f * ((float)(-1.0 / 479001600) + f * (float)(1.0 / 87178291200.0)));
    sc = mad(t, mad(t, mad(t, mad(t, hs, num<T>(-1.0 / 5040)), num<T>(1.0 / 120)),
                    num<T>(-1.0 / 6)), val<T>(1.0f));
    vc = mad(t, mad(t, mad(t, mad(t, hv, num<T>(-1.0 / 40320)), num<T>(1.0 / 720)),
                    num<T>(-1.0 / 24)), num<T>(1.0 / 2));
    c = mad(-t, vc, val<T>(1.0f));
  } else {
    trig3_far(x, c, sc, vc);
  }
}

// v brought into [-pi, pi].
template <class T>
__device__ __forceinline__ T wrap(T v) {
  T r = mad(num<T>(-2.0 * kPi), val<T>(rintf(lead(v) * (float)(0.5 / kPi))), v);
  const T over = r - num<T>(kPi), under = r + num<T>(kPi);
  if (lead(over) > 0.0f) r = r - num<T>(2.0 * kPi);
  else if (lead(under) < 0.0f) r = r + num<T>(2.0 * kPi);
  return r;
}

// Per-thread arrays of a pass, in shared memory (column threadIdx.x of each row), so that
// its loops over the hits stay loops.
constexpr int kThreads = 128;
constexpr int kBlocksPerSm = 3;  // 71 KB of shared memory each
template <class T>
struct Work {
  T s[kN][kThreads];       // arc lengths, then those along the fitted path
  T e[kN][kThreads];       // residuals of the plane
  T a[kN - 1][kThreads];   // segment coefficients of the plane's kinks: kink i is
  T b[kN - 1][kThreads];   //   a_{i-1} u_{i-1} - (b_i + b_{i-1}) u_i + a_i u_{i+1}
  T g[kN - 1][kThreads];   //   - (g_i + g_{i-1}) dkappa
  T u[kN][kThreads];       // solution
  T l1[kN][kThreads], l2[kN][kThreads], lb[kN][kThreads];  // factors
  float w[kN][kThreads];   // inverse variances of the kinks
};
static_assert(sizeof(F2) == sizeof(double), "either form in the same memory");

// Least squares of one plane: minimises the sum of wm_i (e_i - u_i)^2 over the n hits and of
// kf w_i kink_i^2 over the interior ones, wm_i = wb (barrel) or wd; the unknowns are the u_i
// (left in W.u) and, where `bend`, dkappa (returned; else 0).  A kink couples three
// neighbouring hits, so the normal equations have two subdiagonals and dkappa's row; they
// are set up and eliminated hit by hit, three rows at a time.
template <class T>
__device__ __noinline__ T solve_plane(Work<T>& W, int n, uint32_t barrel, T wb, T wd, T kf,
                                      bool bend, float* chi2) {
  const int t = threadIdx.x;
  const T zero = val<T>(0.0f);
  auto wm = [&](int i) { return (barrel >> i & 1u) ? wb : wd; };
  T d0 = wm(0), d1 = wm(1), d2 = wm(2);  // diagonal of rows j, j + 1, j + 2
  T e1 = zero, f1 = zero;                // (j + 1, j), (j + 2, j + 1)
  T e2 = zero;                           // (j + 2, j)
  T b0 = zero, b1 = zero, b2 = zero, bb = zero;  // dkappa's row
  T r0 = W.e[0][t] * d0, r1 = W.e[1][t] * d1, r2 = W.e[2][t] * d2, rb = zero;
#pragma unroll 1
  for (int j = 0; j < n; ++j) {
    if (j + 2 < n) {  // the kink at hit j + 1
      const T w = kf * val<T>(W.w[j + 1][t]);
      const T q0 = W.a[j][t], q1 = -(W.b[j][t] + W.b[j + 1][t]), q2 = W.a[j + 1][t];
      const T q3 = -(W.g[j][t] + W.g[j + 1][t]);
      const T w0 = w * q0, w1 = w * q1, w2 = w * q2, w3 = w * q3;
      d0 = mad(w0, q0, d0);
      e1 = mad(w0, q1, e1);
      e2 = w0 * q2;
      b0 = mad(w0, q3, b0);
      d1 = mad(w1, q1, d1);
      f1 = w1 * q2;
      b1 = mad(w1, q3, b1);
      d2 = mad(w2, q2, d2);
      b2 = w2 * q3;
      bb = mad(w3, q3, bb);
    }
    const T inv = recip(d0);
    const T l1 = e1 * inv, l2 = e2 * inv, lb = b0 * inv;
    W.l1[j][t] = l1;
    W.l2[j][t] = l2;
    W.lb[j][t] = lb;
    W.u[j][t] = r0 * inv;
    bb = mad(-lb, b0, bb);
    rb = mad(-lb, r0, rb);
    r0 = mad(-l1, r0, r1);
    r1 = mad(-l2, W.u[j][t] * d0, r2);
    b0 = mad(-lb, e1, b1);
    b1 = mad(-lb, e2, b2);
    d0 = mad(-l1, e1, d1);
    d1 = mad(-l2, e2, d2);
    e1 = mad(-l2, e1, f1);
    e2 = f1 = b2 = zero;
    const bool more = j + 3 < n;
    d2 = more ? wm(j + 3) : val<T>(1.0f);
    r2 = more ? W.e[j + 3][t] * d2 : zero;
  }
  const T dk = bend ? rb * recip(bb) : zero;
  T x1 = zero, x2 = zero;
#pragma unroll 1
  for (int j = n - 1; j >= 0; --j) {
    const T x = mad(-W.l1[j][t], x1, mad(-W.l2[j][t], x2, mad(-W.lb[j][t], dk, W.u[j][t])));
    W.u[j][t] = x;
    x2 = x1;
    x1 = x;
  }
  T c2 = zero;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const T d = W.e[i][t] - W.u[i][t];
    c2 = mad(d * d, wm(i), c2);
    if (i >= 1 && i + 1 < n) {
      T k = mad(W.a[i - 1][t], W.u[i - 1][t], W.a[i][t] * W.u[i + 1][t]);
      k = mad(-(W.b[i][t] + W.b[i - 1][t]), W.u[i][t], k);
      k = mad(-(W.g[i][t] + W.g[i - 1][t]), dk, k);
      c2 = mad(k * k, kf * val<T>(W.w[i][t]), c2);
    }
  }
  *chi2 = lead(c2);
  return dk;
}

// One refit pass of a track (float32 parameters in tr, n hits in xyz) in T.  false: the
// reference does not allow one ([B6]); otherwise tr holds the result, *more is set when the
// curvature moved by more than kPassTol.
template <class T>
__device__ __forceinline__ bool fit_pass(Work<T>& W, pt_track& tr, int n,
                                         const float (&xyz)[3][kN][kThreads], uint32_t barrel,
                                         float bfield, float x0b, float x0d, bool* more) {
  // [B6]
  if (!isfinite(tr.kappa) || !isfinite(tr.phi0) || !isfinite(tr.d0) || !isfinite(tr.cot_theta) ||
      !isfinite(tr.z0) || fabsf(tr.kappa) < 1e-7f)
    return false;
  const int t = threadIdx.x;
  const T one = val<T>(1.0f);
  const T k0 = val<T>(tr.kappa), d0 = val<T>(tr.d0), cot0 = val<T>(tr.cot_theta);
  // [B1] arc lengths and transverse residuals
  T sp0, cp0;
  sin_cos(tr.phi0, sp0, cp0);
  const T ik0 = recip(k0);
  const T ak0 = absv(k0), ik02 = ik0 * ik0;
  const T kd = mad(k0, d0, val<T>(-1.0f));              // kappa0 d0 - 1
  const T n0 = d0 * (one - kd);                         // d0 (2 - kappa0 d0)
  bool ordered = true;
  T before = one;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const T x = val<T>(xyz[0][i][t]), y = val<T>(xyz[1][i][t]);
    const T along = mad(x, cp0, y * sp0), across = mad(x, sp0, -(y * cp0));
    const T u = k0 * along, v = mad(k0, across, -kd);  // 1 + kappa0 (p.q - d0)
    const T s = val<T>(atan2f(lead(along * ik0), lead(v * ik02))) * ik0;
    const T N = mad(-k0, mad(x, x, y * y), n0) + (kd + kd) * across;
    W.s[i][t] = s;
    W.e[i][t] = N * recip(one + root(mad(u, u, v * v)));
    ordered = ordered && (i == 0 || lead(s - before) > 1e-6f);
    before = s;
  }
  if (!ordered) return false;
  // [B4] kink variances at the interior hits (float32)
  const T sth = recip(root(mad(cot0, cot0, one)));
  const float sthf = lead(sth), cthf = lead(cot0 * sth);
  const T cb = num<T>(kCpt / 100.0) * val<T>(bfield);
  const float pf = lead(cb * recip(ak0 * sth));
#pragma unroll 1
  for (int i = 1; i + 1 < n; ++i) {
    float tx;
    if (barrel >> i & 1u) {
      const float x = xyz[0][i][t], y = xyz[1][i][t];
      float sps, cps;
      sincosf(lead(val<T>(tr.phi0) + k0 * W.s[i][t]), &sps, &cps);
      const float cos_inc = fabsf(sthf * (cps * x + sps * y)) / sqrtf(x * x + y * y);
      tx = x0b / fmaxf(cos_inc, 1e-3f);
    } else {
      tx = x0d / fmaxf(fabsf(cthf), 1e-3f);
    }
    const float th0 = 0.0136f / pf * sqrtf(tx) * (1.0f + 0.038f * logf(tx));
    W.w[i][t] = (sthf * sthf) / (th0 * th0);
  }
  // [B2] segment coefficients a, a c and a g; the last turn is the way from the closest
  // approach to the first hit
  T cs, snk, gs;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const bool last = i == n - 1;
    const T h = last ? W.s[0][t] : W.s[i + 1][t] - W.s[i][t];
    T c, sc, vc;
    trig3(k0 * h, c, sc, vc);
    const T hs = h * sc, hv = h * h * vc;
    if (last) {
      cs = c;
      snk = hs;
      gs = hv;
    } else {
      const T a = recip(hs);
      W.a[i][t] = a;
      W.b[i][t] = a * c;
      W.g[i][t] = a * hv;
    }
  }
  if (kPairs<T>) {
    float stiff = 0.0f;
#pragma unroll 1
    for (int i = 1; i + 1 < n; ++i) {
      const float a = fmaxf(lead(W.a[i - 1][t]), lead(W.a[i][t]));
      stiff = fmaxf(stiff, W.w[i][t] * a * a);
    }
    if (!(stiff * fmaxf(1.0f, 0.5f * fabsf(tr.cot_theta)) <= kStiffMax)) {
      tr.chi2_circle = __int_as_float(0x7fffffff);  // not finite: float64
      return true;
    }
  }
  const T wm = num<T>(1.0 / (kSigmaT * kSigmaT));
  const T dk = solve_plane(W, n, barrel, wm, wm, one, true, &tr.chi2_circle);
  // [B5] transverse parameters at the closest approach
  const T u1 = W.u[0][t];
  const T du1 = mad(W.a[0][t], W.u[1][t], -mad(W.b[0][t], u1, W.g[0][t] * dk));
  const T u0 = mad(u1, cs, mad(gs, dk, -(du1 * snk)));
  const T du0 = mad(du1, cs, mad(k0 * k0 * u1, snk, -(dk * snk)));
  // [B3] arc lengths along the fitted transverse path, z residuals
  const T half = val<T>(0.5f), twelfth = num<T>(1.0 / 12.0);
  T acc = val<T>(0.0f), s_old = val<T>(0.0f), u_old = u0, sp_old = val<T>(0.0f), sp1 = acc;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const T s = W.s[i][t], u = W.u[i][t];
    const T h = s - s_old;
    acc = acc + mad(h * (u_old + u), half, -(dk * (h * h * h) * twelfth));
    const T sp = mad(-k0, acc, s);
    if (i == 0) {
      sp1 = sp;
    } else {
      const T ih = recip(sp - sp_old);
      W.a[i - 1][t] = ih;
      W.b[i - 1][t] = ih;
      W.g[i - 1][t] = val<T>(0.0f);
    }
    W.e[i][t] = val<T>(xyz[2][i][t]) - mad(cot0, sp, val<T>(tr.z0));
    s_old = s;
    u_old = u;
    sp_old = sp;
  }
  T sld = absv(cot0) * num<T>(kSigmaL);
  if (lead(sld) < 1e-12f) sld = num<T>(1e-12);
  const T isld = recip(sld);
  solve_plane(W, n, barrel, num<T>(1.0 / (kSigmaL * kSigmaL)), isld * isld,
              val<T>(sthf * sthf), false, &tr.chi2_line);
  const T w1 = W.u[0][t];
  const T dw1 = (W.u[1][t] - w1) * W.a[0][t];
  const T kappa = k0 + dk;
  tr.kappa = lead(kappa);
  tr.phi0 = lead(wrap(val<T>(tr.phi0) + du0));
  tr.d0 = lead(d0 - u0);
  tr.z0 = lead(val<T>(tr.z0) + mad(-sp1, dw1, w1));
  tr.cot_theta = lead(cot0 + dw1);
  tr.pt = lead(cb * recip(absv(kappa)));
  tr.charge = tr.kappa > 0.0f ? -1 : (tr.kappa < 0.0f ? 1 : 0);
  *more = lead(absv(dk) * recip(ak0)) > kPassTol;
  return true;
}

// The pass in float64, for a track that leaves the range of float32 on the way.
__device__ __noinline__ bool fit_pass_f64(Work<double>& W, pt_track& tr, int n,
                                          const float (&xyz)[3][kN][kThreads], uint32_t barrel,
                                          float bfield, float x0b, float x0d, bool* more) {
  return fit_pass<double>(W, tr, n, xyz, barrel, bfield, x0b, x0d, more);
}

struct RefitSmem {
  union {
    Work<F2> f;
    Work<double> d;
  } w;
  float xyz[3][kN][kThreads];
};

// One refit pass of track j from its current fit, written back; *more: it still moves.
__device__ __forceinline__ void refit_pass(const Buffers& b, RefitSmem& S, uint64_t j,
                                           float bfield, float x0b, float x0d, bool* more) {
  *more = false;
  const uint32_t t = b.sv[j];
  const int n = b.nt_n[t];
  if (n < 3 || n > kN) return;
  uint32_t barrel = 0;
#pragma unroll
  for (int i = 0; i < kN; ++i) {
    if (i < n) {
      const int32_t g = b.nt_hits[(uint64_t)t * kMaxHits + i];
      S.xyz[0][i][threadIdx.x] = b.in_x[g];
      S.xyz[1][i][threadIdx.x] = b.in_y[g];
      S.xyz[2][i][threadIdx.x] = b.in_z[g];
      barrel |= b.in_layer[g] < 4 ? 1u << i : 0u;
    }
  }
  pt_track tr = b.tracks[j];
  if (!fit_pass<F2>(S.w.f, tr, n, S.xyz, barrel, bfield, x0b, x0d, more)) return;
  if (!(isfinite(tr.kappa) && isfinite(tr.phi0) && isfinite(tr.d0) && isfinite(tr.cot_theta) &&
        isfinite(tr.z0) && isfinite(tr.pt) && isfinite(tr.chi2_circle) &&
        isfinite(tr.chi2_line))) {
    tr = b.tracks[j];
    if (!fit_pass_f64(S.w.d, tr, n, S.xyz, barrel, bfield, x0b, x0d, more)) return;
  }
  b.tracks[j] = tr;
}

// One pass over every cleaned track (in_list null) or over the in_n[0] tracks of
// in_list; tracks that keep moving are appended to out_list (when given).
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
    k_refit_bl(Buffers b, float bfield, float x0b, float x0d, const uint32_t* in_list,
               const unsigned long long* in_n, uint32_t* out_list, unsigned long long* out_n,
               uint64_t cap) {
  pdl_sync();
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char rsm[];
  RefitSmem& S = *(RefitSmem*)rsm;
  const uint64_t N = min(in_list ? *in_n : b.cnt[CNT_SV], (unsigned long long)cap);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += stride) {
    const uint64_t j = in_list ? in_list[i] : i;
    bool more;
    refit_pass(b, S, j, bfield, x0b, x0d, &more);
    if (more && out_list) {
      cg::coalesced_group g = cg::coalesced_threads();
      unsigned long long base = 0;
      if (g.thread_rank() == 0) base = atomicAdd(out_n, (unsigned long long)g.size());
      base = g.shfl(base, 0);
      out_list[base + g.thread_rank()] = (uint32_t)j;
    }
  }
}

}  // namespace

cudaError_t launch_refit_broken_line(const Buffers& b, const Params& p, float x0_barrel,
                                     float x0_disk, uint32_t* list, unsigned long long* counters,
                                     const Launch& l, cudaStream_t s) {
  const uint64_t cap = (uint64_t)p.max_ntuplets;
  uint32_t* lists[2] = {list, list + cap};
  cudaError_t e = cudaFuncSetAttribute(k_refit_bl, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(RefitSmem));
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(counters, 0, kMaxPasses * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  for (int pass = 0; pass < kMaxPasses; ++pass) {
    const uint32_t* in = pass == 0 ? nullptr : lists[(pass - 1) & 1];
    const unsigned long long* in_n = pass == 0 ? nullptr : &counters[pass - 1];
    uint32_t* out = pass + 1 < kMaxPasses ? lists[pass & 1] : nullptr;
    unsigned long long* out_n = pass + 1 < kMaxPasses ? &counters[pass] : nullptr;
    PT_TRACE(l, s, "k_refit_bl",
             launch_pdl(k_refit_bl, l.sms * kBlocksPerSm, kThreads, sizeof(RefitSmem), s, b,
                        p.bfield, x0_barrel, x0_disk, in, in_n, out, out_n, cap));
  }
  return cudaGetLastError();
}

}  // namespace ptca
