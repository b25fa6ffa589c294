// analytic_series.cuh -- the analytic push (constant E, B over the step) by the
// downward recurrence of the series of exp(L tau): the form of the FP64 and
// compensated particle kernels, and the pieces of the FP32-pair push
// (pair_push.cuh).  It takes two thirds of the FP64 operations of analytic_push
// (pushers.cuh), which the ensembles keep: 2D compensated fields, 1.5 M electrons,
// particle kernel 0.855 -> 0.69 ms per step.
#pragma once
#include "pushers.cuh"

namespace pic {

// ---------------------------------------------------------------------------
// Analytic pusher for E, B constant over the step (Sec. 1, Sec. 4.1): the
// four-velocity U = (gamma, u) obeys dU/dtau = L U with
//   L U = (e.u, gamma e + u x b),  e = qm E, b = qm B.
// L^4 = S1 L^2 + S2 with S1 = e^2 - b^2, S2 = (e.b)^2 (Cayley-Hamilton), so
// exp(L tau) = c0 + c1 L + c2 L^2 + c3 L^3.  With A = S1 tau^2, Q = S2 tau^4 and
// the numbers p_1 = 1, p_2 = A, p_{n+1} = A p_n + Q p_{n-1},
//   s_a = sum_{n>=1} p_n / (2n + a)!,
// the coefficients are c0 = 1 + Q s_2, c1 = tau (1 + Q s_3), c2 = tau^2 s_0,
// c3 = tau^3 s_1, and the lab time is t(tau) = [c1 U + tau^2 (s_0 - A s_2) LU +
// c3 L^2U + tau^4 s_2 L^3U]_0.  Summing by parts with the recurrence of p_n,
//   s_a = 1/(a + 2)! + A s_{a+2} + Q s_{a+4},
// a downward recurrence of two multiply-adds per term and series: no root, no
// division, nothing singular at null fields (the plane-wave case).  Where the
// roots lE^2 tau^2 = X, lB^2 tau^2 = Y of S1 = lE^2 - lB^2, S2 = lE^2 lB^2 add up to 2 or
// more the closed forms in X and Y take over: with the entire functions
//   h(X) = (cosh x - 1)/X,  f(X) = (sinh x - x)/(X x),
//   k(Y) = (1 - cos y)/Y,   g(Y) = (y - sin y)/(Y y),
// s_2 = (h - k)/(X + Y), s_3 = (f - g)/(X + Y), s_0 = h - Y s_2, s_1 = f - Y s_3.
// The proper time with t(tau) = dt is found by bracketed Newton (dt/dtau = gamma).
// ---------------------------------------------------------------------------

struct AsState {
  double S1, S2;
  double U[4], LU[4], L2U[4], L3U[4];
};

// Terms needed by the series: they stop once a term falls below `tol` of the
// leading ones.  With M = max(X, Y), term n of every series is at most
// B_n(M) = (M^n + n M^(n-1)) / (2n+2)! (|p_n| <= n M^(n-1)), increasing in M;
// m[K] is the largest M <= 2 (found by bisection at compile time, rounded down to
// FP32 with a 1e-6 margin) for which B_(K-1)(M) < tol, so K terms (n = 0 .. K-1)
// are enough for every M <= m[K].
constexpr AnTerms as_terms_table(double tol) {
  AnTerms t{};
  for (int K = 0; K < 22; ++K) {
    if (K < 1) {
      t.m[K] = -1.0f;
      continue;
    }
    double lo = 0.0, hi = 2.0;
    if (an_bound(K - 1, 0.0) >= tol) {
      t.m[K] = -1.0f;   // not enough terms even for M = 0
      continue;
    }
    for (int it = 0; it < 80; ++it) {
      const double mid = 0.5 * (lo + hi);
      if (an_bound(K - 1, mid) < tol) lo = mid; else hi = mid;
    }
    t.m[K] = (float)(lo * (1.0 - 1e-6));
  }
  return t;
}
// FP64 series (2^-60) and FP32 series (2^-27); the coefficients in FP64 and as FP32
// pairs
struct AsTables {
  AnCoef c;
  float h2[21], l2[21], h3[21], l3[21];
  AnTerms t64, t24;
};
constexpr AsTables as_tables() {
  AsTables t{};
  t.c = an_coef_table();
  for (int n = 0; n < 14; ++n) {   // later terms and low parts are below 1e-30
    t.h2[n] = (float)t.c.c2[n];
    t.h3[n] = (float)t.c.c3[n];
    if (n < 10) {
      t.l2[n] = (float)(t.c.c2[n] - (double)t.h2[n]);
      t.l3[n] = (float)(t.c.c3[n] - (double)t.h3[n]);
    }
  }
  t.t64 = as_terms_table(8.7e-19);
  t.t24 = as_terms_table(7.5e-9);
  return t;
}
#ifdef __CUDACC__
__constant__ constexpr AsTables kAs = as_tables();
#endif
constexpr AsTables kAsHost = as_tables();
#ifdef __CUDA_ARCH__
#define PIC_AS kAs
#else
#define PIC_AS kAsHost
#endif

// max(X, Y) of the roots from A = X - Y and Q = X Y, in FP32 and rounded up; a
// NaN (overflow) compares false with every limit
PIC_HD float as_root_max(float A, float Q) {
  return 0.5000005f * (fabsf(A) + sqrtf(fmaf(A, A, 4.0f * Q)));
}
// the series hold for X + Y < 2
PIC_HD bool as_series_ok(float A, float Q) { return fmaf(A, A, 4.0f * Q) < 4.0f; }

PIC_HD int as_terms(const AnTerms& t, float M) {
  int K = 1;
  while (K < 21 && !(M <= t.m[K])) ++K;
  return K;
}

// s_0, s_1, s_2, s_3 of A and Q (see above)
struct AsSums {
  double s0, s1, s2, s3;
};
PIC_HD AsSums as_sums(double A, double Q) {
  AsSums r;
  const float Af = narrow_sat(A), Qf = narrow_sat(Q);
  if (as_series_ok(Af, Qf)) {
    const int K = as_terms(PIC_AS.t64, as_root_max(Af, Qf));
    double e1 = 0.0, o1 = 0.0, e0 = PIC_AS.c.c2[K - 1], o0 = PIC_AS.c.c3[K - 1];
#pragma unroll 1
    for (int n = K - 2; n >= 0; --n) {
      const double en = fma(A, e0, fma(Q, e1, PIC_AS.c.c2[n]));
      const double on = fma(A, o0, fma(Q, o1, PIC_AS.c.c3[n]));
      e1 = e0;
      o1 = o0;
      e0 = en;
      o0 = on;
    }
    r.s0 = e0;
    r.s1 = o0;
    r.s2 = e1;
    r.s3 = o1;
  } else {
    const double root = sqrt(A * A + 4.0 * Q);
    double X, Y;
    if (A >= 0.0) {
      X = 0.5 * (A + root);
      Y = Q / X;
    } else {
      Y = 0.5 * (root - A);
      X = Q / Y;
    }
    const double h = an_h(X), f = an_f(X);
    r.s2 = (h - an_k(Y)) / (X + Y);
    r.s3 = (f - an_g(Y)) / (X + Y);
    r.s0 = h - Y * r.s2;
    r.s1 = f - Y * r.s3;
  }
  return r;
}

// gamma(tau) and t(tau); c[0..3] receive c0 - 1, c1, c2, c3, from which
// as_momentum forms the spatial part of U(tau)
PIC_HD void as_eval(const AsState& a, double tau, double* gam, double* tl, double c[4]) {
  const double t2 = tau * tau;
  const double A = a.S1 * t2, Q = a.S2 * t2 * t2;
  const AsSums F = as_sums(A, Q);
  const double q2 = Q * F.s2, c1 = fma(tau, Q * F.s3, tau);
  const double c2 = t2 * F.s0, t3 = t2 * tau;
  const double c3 = t3 * F.s1;
  const double d1 = t2 * fma(-A, F.s2, F.s0), d3 = t2 * t2 * F.s2;
  *gam = fma(c3, a.L3U[0], fma(c2, a.L2U[0], fma(c1, a.LU[0], fma(q2, a.U[0], a.U[0]))));
  *tl = fma(d3, a.L3U[0], fma(c3, a.L2U[0], fma(d1, a.LU[0], c1 * a.U[0])));
  c[0] = q2;
  c[1] = c1;
  c[2] = c2;
  c[3] = c3;
}
PIC_HD void as_momentum(const AsState& a, const double c[4], double* uo) {
#pragma unroll
  for (int m = 0; m < 3; ++m)
    uo[m] = a.U[m + 1] + fma(c[3], a.L3U[m + 1],
                             fma(c[2], a.L2U[m + 1], fma(c[1], a.LU[m + 1], c[0] * a.U[m + 1])));
}

// The equation F(s) = D of the proper time in FP32: F = t(s), dF/ds = gamma(s),
// with the time components V[k] of L^k U.  Newton from D/gamma0 inside the
// bracket (0, D]; the result only starts the accurate iterations, so it need
// not converge (the series limit or an overflow ends it early).  Fields and
// momenta scale the same way in every unit: with the raw fields and D = qm dt
// the variable is s = qm tau, of either sign.
PIC_HD float as_start(const float V[4], float S1, float S2, float D, float s) {
  float in = 0.0f, out = D;   // |F(in)| < |D| <= |F(out)|
#pragma unroll 1
  for (int it = 0; it < 8; ++it) {
    const float z = s * s, A = S1 * z, Q = S2 * z * z;
    if (!as_series_ok(A, Q)) return s;
    const int K = as_terms(PIC_AS.t24, as_root_max(A, Q));
    float e1 = 0.0f, o1 = 0.0f, e0 = PIC_AS.h2[K - 1], o0 = PIC_AS.h3[K - 1];
#pragma unroll 1
    for (int n = K - 2; n >= 0; --n) {
      const float en = fmaf(A, e0, fmaf(Q, e1, PIC_AS.h2[n]));
      const float on = fmaf(A, o0, fmaf(Q, o1, PIC_AS.h3[n]));
      e1 = e0;
      o1 = o0;
      e0 = en;
      o0 = on;
    }
    const float q2 = Q * e1, c1 = fmaf(s, Q * o1, s), c2 = z * e0, c3 = z * s * o0;
    const float gam = V[0] + fmaf(c3, V[3], fmaf(c2, V[2], fmaf(c1, V[1], q2 * V[0])));
    const float F = fmaf(z * z * e1, V[3], fmaf(c3, V[2], fmaf(z * fmaf(-A, e1, e0), V[1], c1 * V[0])));
    const float r = F - D;
    float sn = s - r / gam;
    if (fabsf(sn - s) <= 1e-6f * fabsf(s)) return sn;
    if ((r > 0.0f) == (D > 0.0f)) out = s; else in = s;
    if (!((sn > in) == (sn < out)) || sn == in || sn == out) sn = 0.5f * (in + out);
    s = sn;
  }
  return s;
}

// Returns the number of evaluations (> 0), or -1 if the proper-time iteration
// did not converge within its bound (u is then left unchanged).
// FP64-pipe operations, which bound the FP64 and compensated particle kernels:
// about 75 for the invariants and L^k U, 45 per evaluation (one to three).
PIC_HDI int analytic_push_series(double qm, double dt, const double eb[6], double u[3]) {
  AsState a;
  const double e[3] = {qm * eb[0], qm * eb[1], qm * eb[2]};
  const double b[3] = {qm * eb[3], qm * eb[4], qm * eb[5]};
  const double ee = e[0] * e[0] + e[1] * e[1] + e[2] * e[2];
  const double bb = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
  const double ebd = e[0] * b[0] + e[1] * b[1] + e[2] * b[2];
  a.S1 = ee - bb;
  a.S2 = ebd * ebd;
  // gamma0 = x / sqrt(x) from the Newton 1/sqrt (x >= 1), which also gives dt/gamma0
  const double x0 = 1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const double ig0 = rsqrt_nr(x0);
  const double g0 = x0 * ig0;
  a.U[0] = g0; a.U[1] = u[0]; a.U[2] = u[1]; a.U[3] = u[2];
  an_apply(e, b, a.U, a.LU);
  an_apply(e, b, a.LU, a.L2U);
  an_apply(e, b, a.L2U, a.L3U);
  // t(tau) >= tau (gamma >= 1): the root lies in (0, dt].  The FP32 root moves the
  // start dt/gamma0 (in FP64: a weak field then converges in one evaluation); Newton
  // goes on from there, keeping a bracket [lo, hi] (t increasing) for bisection.
  double lo = 0.0, hi = dt, tau = dt * ig0, gam, tl, cf[4];
  {
    const float V[4] = {narrow_sat(g0), narrow_sat(a.LU[0]), narrow_sat(a.L2U[0]),
                        narrow_sat(a.L3U[0])};
    const float s0 = narrow_signed(tau);
    const float d = as_start(V, narrow_sat(a.S1), narrow_sat(a.S2), narrow_signed(dt), s0) - s0;
    const double moved = tau + widen(d);
    if (moved > lo && moved < hi) tau = moved;
  }
  const double eps4 = 4.0 * 2.220446049250313e-16;
  int it = 1;
  for (; it <= 64; ++it) {
    as_eval(a, tau, &gam, &tl, cf);
    const double r = tl - dt;
    // gam >= 1; one Newton step of 1/gam suffices: its 1e-13 relative error only
    // scales the (then tiny) correction, the state is taken at the evaluated tau
    double tn = tau - r * rcp_nr<1>(gam);
    // converged: the Newton step is below rounding of tau (tested before the
    // bracket, whose strict bounds would turn a step that rounds to nothing,
    // or a zero residual, into a bisection step away from the root)
    if (fabs(tn - tau) <= eps4 * fabs(tau)) break;
    if (r > 0.0) hi = tau; else lo = tau;
    if (!(tn > lo && tn < hi)) tn = 0.5 * (lo + hi);
    if (hi - lo <= eps4 * hi) break;
    tau = tn;
  }
  if (it > 64) return -1;
  double uo[3];
  as_momentum(a, cf, uo);   // at the last evaluated tau
  u[0] = uo[0]; u[1] = uo[1]; u[2] = uo[2];
  return it;
}

}  // namespace pic
