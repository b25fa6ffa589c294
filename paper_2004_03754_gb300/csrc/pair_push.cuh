// pair_push.cuh -- the momentum advance of particles in FP32 fields, in FP32 pairs
// (dfloat.cuh: hi + lo, about 47 bits) added to the FP64 momentum and position.
//
// Why: FP64 instructions issue at 1/64 of the FP32 rate on this GPU, and the FP64
// Boris push of 49 of them kept that pipe 83 % busy and the rest of the SM idle.
// With FP32 fields (relative rounding 6e-8) a push needs far fewer than 53 bits in
// its *change* of u: u^{n+1/2} = u^{n-1/2} + du and x^{n+1} = x^n + dx are added in
// FP64, so nothing of the state is rounded to the pairs' width, and du, dx come
// from error-free FP32 transformations with a relative error near 2^-45 (the FP64
// form with one Newton step of its reciprocals had 2^-43).  An FP64 operation
// takes the issue slots of 64 FP32 ones here; its pair form takes 4 to 11.
// Measured (one step, particle kernel): 2D Boris, 29.4 M electrons 2.61 -> 2.02 ms;
// 2D Higuera-Cary, 1.4 M electrons 0.280 -> 0.118 ms; 3D analytic, 84 M electrons
// 29.2 -> 24.6 ms (there the windows' handling is half of what remains).
//
// Products feeding a TwoSum are rounded on their own (mul_rn); sums written
// plainly hold no product, so no contraction can break them.
#pragma once
#include "dfloat.cuh"
#include "analytic_series.cuh"
#include "pushers.cuh"

namespace pic {

// ---- pair arithmetic without renormalisation where the next operation allows it

// x = hi + lo: hi the FP32 value nearest to x, lo the rest rounded to FP32
// (relative error below 2^-49), on the integer pipe.  |x| < 2^-126 gives zero,
// |x| < 2^-74 no low part.
PIC_HD dfl pr_split(double x) {
  const uint64_t b = f64_bits(x);
  const uint64_t mag = b & 0x7fffffffffffffffull;
  const uint32_t sign = (uint32_t)(b >> 32) & 0x80000000u;
  const uint64_t r = mag + 0x0fffffffull + ((mag >> 29) & 1ull);
  const uint32_t r29 = (uint32_t)(r >> 29);
  const uint32_t h = mag < (897ull << 52) ? 0u : r29 - (896u << 23);
  // mag - hi in units of the FP64 mantissa's last place: within +-2^28
  const int32_t d = (int32_t)((uint32_t)mag - (r29 << 29));
  const uint32_t eh = (uint32_t)((mag >> 29) - ((uint64_t)896 << 23)) & 0x7f800000u;
  const uint32_t sc = h != 0u && eh > (52u << 23) ? eh - (52u << 23) : 0u;   // that unit in FP32
  const float l = mul_rn((float)d, f32_from_bits(sc));
  return dfl(f32_from_bits(h | sign), f32_from_bits(f32_bits(l) ^ sign));
}
// the pair in FP64 (exact unless a part is subnormal)
PIC_HD double pr_join(dfl a) { return widen_normal(a.hi) + widen_normal(a.lo); }

PIC_HD dfl pr_mul(dfl a, dfl b) {
  const float p = mul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return dfl(p, e);
}
PIC_HD dfl pr_mulf(dfl a, float b) {
  const float p = mul_rn(a.hi, b);
  float e = fmaf(a.hi, b, -p);
  e = fmaf(a.lo, b, e);
  return dfl(p, e);
}
PIC_HD dfl pr_mulff(float a, float b) {
  const float p = mul_rn(a, b);
  return dfl(p, fmaf(a, b, -p));
}
PIC_HD dfl pr_sqr(dfl a) {
  const float p = mul_rn(a.hi, a.hi);
  float e = fmaf(a.hi, a.hi, -p);
  e = fmaf(a.hi, 2.0f * a.lo, e);
  return dfl(p, e);
}
// a + b, the low part not renormalised
PIC_HD dfl pr_add_raw(dfl a, dfl b) {
  const dfl s = two_sum(a.hi, b.hi);
  return dfl(s.hi, s.lo + (a.lo + b.lo));
}
PIC_HD dfl pr_norm(dfl a) { return fast_two_sum(a.hi, a.lo); }
PIC_HD dfl pr_add(dfl a, dfl b) { return pr_norm(pr_add_raw(a, b)); }
PIC_HD dfl pr_neg(dfl a) { return dfl(-a.hi, -a.lo); }
// a b - c d
PIC_HD dfl pr_det(dfl a, dfl b, dfl c, dfl d) { return pr_add_raw(pr_mul(a, b), pr_neg(pr_mul(c, d))); }
// 1 + |v|^2 (all terms positive: each TwoSum may take the larger sum first)
PIC_HD dfl pr_one_plus_sqr(const dfl v[3]) {
  dfl s(1.0f, 0.0f);
#pragma unroll
  for (int d = 0; d < 3; ++d) s = pr_add_raw(s, pr_sqr(v[d]));
  return pr_norm(s);
}
// 1/sqrt(x), 1/x, x >= 1 (positive normal), x normalised: the FP32 seed and one
// Newton step whose residual is formed exactly, with the next term of its series
PIC_HD dfl pr_rsqrt(dfl x) {
  const float y = seed_rsqrt(x.hi);
  const dfl s = pr_mulff(y, y);
  const float p = mul_rn(x.hi, s.hi);
  float r = (1.0f - p) - fmaf(x.hi, s.hi, -p);       // 1 - x y^2
  r = fmaf(-x.hi, s.lo, r);
  r = fmaf(-x.lo, s.hi, r);
  return fast_two_sum(y, mul_rn(y, fmaf(mul_rn(0.375f, r), r, 0.5f * r)));
}
PIC_HD dfl pr_rcp(dfl x) {
  const float y = seed_rcp(x.hi);
  float r = fmaf(-x.hi, y, 1.0f);
  r = fmaf(-x.lo, y, r);
  return fast_two_sum(y, mul_rn(y, fmaf(r, r, r)));
}

// ---- Boris: du = (u- + u- x t) x s + 2 h E with u- = u + h E, h = q dt/2m
PIC_HD void boris_push_pair(dfl h, const float eb[6], const dfl u[3], dfl du[3]) {
  dfl k[3], m[3], t[3], v[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    k[d] = pr_mulf(h, eb[d]);
    m[d] = pr_add(u[d], k[d]);
  }
  const dfl hig = pr_norm(pr_mul(h, pr_rsqrt(pr_one_plus_sqr(m))));
#pragma unroll
  for (int d = 0; d < 3; ++d) t[d] = pr_mulf(hig, eb[3 + d]);
  dfl f = pr_rcp(pr_one_plus_sqr(t));
  f = dfl(2.0f * f.hi, 2.0f * f.lo);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int a = (d + 1) % 3, b = (d + 2) % 3;
    v[d] = pr_add(m[d], pr_det(m[a], t[b], m[b], t[a]));
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) t[d] = pr_mul(f, t[d]);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int a = (d + 1) % 3, b = (d + 2) % 3;
    du[d] = pr_add(pr_det(v[a], t[b], v[b], t[a]), dfl(2.0f * k[d].hi, 2.0f * k[d].lo));
  }
}

// ---- Higuera-Cary: t = h B / gbar, w = (u- + (u-.t) t + u- x t)/(1 + t^2), u+ = w + w x t.
// u+ - u- = 2 (w x t) (from w + t x w = u-, u+ = w + w x t), so du = 2 w x t + 2 h E.
PIC_HD void hc_push_pair(dfl h, const float eb[6], const dfl u[3], dfl du[3]) {
  dfl k[3], m[3], t[3], w[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    k[d] = pr_mulf(h, eb[d]);
    m[d] = pr_add(u[d], k[d]);
    t[d] = pr_norm(pr_mulf(h, eb[3 + d]));
  }
  // gbar^2 = (sigma + root)/2, root^2 = sigma^2 + 4 w4, sigma = gamma-^2 - b^2,
  // w4 = b^2 + (u-.b)^2; for sigma < 0 the same root as 2 w4 / (root - sigma)
  dfl b2 = pr_norm(pr_add_raw(pr_add_raw(pr_sqr(t[0]), pr_sqr(t[1])), pr_sqr(t[2])));
  const dfl us = pr_norm(pr_add_raw(pr_add_raw(pr_mul(m[0], t[0]), pr_mul(m[1], t[1])), pr_mul(m[2], t[2])));
  const dfl w4 = pr_add(b2, pr_sqr(us));
  const dfl sigma = pr_add(pr_one_plus_sqr(m), pr_neg(b2));
  const dfl q = pr_add(pr_sqr(sigma), dfl(4.0f * w4.hi, 4.0f * w4.lo));
  const dfl root = pr_norm(pr_mul(q, pr_rsqrt(q)));
  dfl g2;
  if (sigma.hi >= 0.0f) {
    g2 = pr_add(sigma, root);
    g2 = dfl(0.5f * g2.hi, 0.5f * g2.lo);
  } else {
    g2 = pr_norm(pr_mul(dfl(2.0f * w4.hi, 2.0f * w4.lo), pr_rcp(pr_add(root, pr_neg(sigma)))));
  }
  const dfl ig = pr_rsqrt(g2);
#pragma unroll
  for (int d = 0; d < 3; ++d) t[d] = pr_norm(pr_mul(t[d], ig));
  const dfl ut = pr_norm(pr_add_raw(pr_add_raw(pr_mul(m[0], t[0]), pr_mul(m[1], t[1])), pr_mul(m[2], t[2])));
  const dfl s2 = pr_rcp(pr_one_plus_sqr(t));
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int a = (d + 1) % 3, b = (d + 2) % 3;
    const dfl x = pr_add_raw(pr_mul(ut, t[d]), pr_det(m[a], t[b], m[b], t[a]));
    w[d] = pr_norm(pr_mul(s2, pr_add(m[d], x)));
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int a = (d + 1) % 3, b = (d + 2) % 3;
    const dfl x = pr_add(pr_det(w[a], t[b], w[b], t[a]), k[d]);
    du[d] = dfl(2.0f * x.hi, 2.0f * x.lo);
  }
}

// ---- analytic push (analytic_series.cuh) in s = (q/m) tau with the raw fields

// sum of three exact products plus their low parts, normalised
PIC_HD dfl pr_sum3(dfl a, dfl b, dfl c) {
  const dfl s = two_sum(a.hi, b.hi), r = two_sum(s.hi, c.hi);
  return fast_two_sum(r.hi, r.lo + (s.lo + ((a.lo + b.lo) + c.lo)));
}
PIC_HD void pr_apply(const float eb[6], const dfl V[4], dfl o[4]) {
  o[0] = pr_sum3(pr_mulf(V[1], eb[0]), pr_mulf(V[2], eb[1]), pr_mulf(V[3], eb[2]));
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int a = (d + 1) % 3, b = (d + 2) % 3;
    o[d + 1] = pr_sum3(pr_mulf(V[0], eb[d]), pr_mulf(V[a + 1], eb[3 + b]), pr_mulf(V[b + 1], -eb[3 + a]));
  }
}
// D = (q/m) dt; du = u^{n+1/2} - u^{n-1/2}.  The root of F(s) = D is found in FP32
// (as_start); one evaluation in pairs gives its residual delta, which then only
// shifts the state to first order (|delta| <= 2^-21 |s|, so the second order is below
// 2^-43 L s).  Returns false when the fields are beyond the series or the iteration
// does not settle; the caller then takes the FP64 push.
PIC_HD bool analytic_push_pair(dfl D, const float eb[6], const dfl u[3], dfl du[3]) {
  dfl V[4][4];
  const dfl x0 = pr_one_plus_sqr(u);
  const dfl ig0 = pr_rsqrt(x0);
  V[0][0] = pr_norm(pr_mul(x0, ig0));
#pragma unroll
  for (int d = 0; d < 3; ++d) V[0][d + 1] = u[d];
  pr_apply(eb, V[0], V[1]);
  pr_apply(eb, V[1], V[2]);
  pr_apply(eb, V[2], V[3]);
  const dfl ee = pr_sum3(pr_mulff(eb[0], eb[0]), pr_mulff(eb[1], eb[1]), pr_mulff(eb[2], eb[2]));
  const dfl bb = pr_sum3(pr_mulff(eb[3], eb[3]), pr_mulff(eb[4], eb[4]), pr_mulff(eb[5], eb[5]));
  const dfl dot = pr_sum3(pr_mulff(eb[0], eb[3]), pr_mulff(eb[1], eb[4]), pr_mulff(eb[2], eb[5]));
  const dfl S1 = pr_add(ee, pr_neg(bb)), S2 = pr_norm(pr_sqr(dot));
  dfl s = pr_norm(pr_mul(D, ig0));
  {
    const float Vf[4] = {V[0][0].hi, V[1][0].hi, V[2][0].hi, V[3][0].hi};
    const float s0 = s.hi;
    const float d = as_start(Vf, S1.hi, S2.hi, D.hi, s0) - s0;
    if (d != 0.0f) s = pr_add(s, dfl(d, 0.0f));
  }
#pragma unroll 1
  for (int it = 0; it < 6; ++it) {
    const dfl z = pr_norm(pr_sqr(s));
    const dfl A = pr_norm(pr_mul(S1, z)), Q = pr_norm(pr_mul(S2, pr_norm(pr_sqr(z))));
    if (!as_series_ok(A.hi, Q.hi)) return false;
    const int K = as_terms(PIC_AS.t48, as_root_max(A.hi, Q.hi));
    dfl e1(0.0f, 0.0f), o1(0.0f, 0.0f), e0(PIC_AS.h2[K - 1], PIC_AS.l2[K - 1]), o0(PIC_AS.h3[K - 1], PIC_AS.l3[K - 1]);
#pragma unroll 1
    for (int n = K - 2; n >= 0; --n) {
      const dfl en = pr_sum3(dfl(PIC_AS.h2[n], PIC_AS.l2[n]), pr_mul(A, e0), pr_mul(Q, e1));
      const dfl on = pr_sum3(dfl(PIC_AS.h3[n], PIC_AS.l3[n]), pr_mul(A, o0), pr_mul(Q, o1));
      e1 = e0;
      o1 = o0;
      e0 = en;
      o0 = on;
    }
    const dfl q2 = pr_norm(pr_mul(Q, e1));
    const dfl c1 = pr_add(s, pr_mul(s, pr_norm(pr_mul(Q, o1))));
    const dfl c2 = pr_norm(pr_mul(z, e0)), c3 = pr_norm(pr_mul(pr_norm(pr_mul(z, s)), o0));
    const dfl d1 = pr_norm(pr_mul(z, pr_add(e0, pr_neg(pr_mul(A, e1)))));
    const dfl d3 = pr_norm(pr_mul(pr_norm(pr_sqr(z)), e1));
    // residual F(s) - D and gamma(s) (FP32: it only scales the residual)
    const dfl F = pr_add(pr_add_raw(pr_mul(c1, V[0][0]), pr_mul(d1, V[1][0])),
                         pr_add_raw(pr_mul(c3, V[2][0]), pr_mul(d3, V[3][0])));
    const float gam = V[0][0].hi + fmaf(c3.hi, V[3][0].hi, fmaf(c2.hi, V[2][0].hi, fmaf(c1.hi, V[1][0].hi, q2.hi * V[0][0].hi)));
    const dfl r = pr_add_raw(F, pr_neg(D));
    const float delta = -(r.hi + r.lo) / gam;
    if (!(fabsf(delta) < fabsf(s.hi))) return false;   // also NaN
    if (fabsf(delta) <= 4.76837158203125e-7f * fabsf(s.hi)) {
      // u(s) - u(0), then delta du/ds = delta (gamma E + u(s) x B) in FP32
      float un[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        du[d] = pr_add(pr_add_raw(pr_mul(q2, u[d]), pr_mul(c1, V[1][d + 1])),
                       pr_add_raw(pr_mul(c2, V[2][d + 1]), pr_mul(c3, V[3][d + 1])));
        un[d] = u[d].hi + du[d].hi;
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int a = (d + 1) % 3, b = (d + 2) % 3;
        const float g = fmaf(gam, eb[d], fmaf(un[a], eb[3 + b], -(un[b] * eb[3 + a])));
        du[d] = pr_add(du[d], dfl(delta * g, 0.0f));
      }
      return true;
    }
    s = pr_add(s, dfl(delta, 0.0f));
  }
  return false;
}

// ---- one particle: u (FP64, in and out) and the pair dx[d] of its move over dt
// along the first ndim axes, 1/gamma and u^{n+1/2} in FP32.  Returns false when the
// analytic push did not converge (u unchanged).
struct PairMove {
  dfl dx[3];
  float dtig, ig, u[3];   // dt/gamma, 1/gamma, u^{n+1/2}
};

PIC_HDI bool push_wide(double qm, double dt, int kind, const float eb[6], double u[3]);

// max |v_d| below 2^e (e > 0), false for NaN; on the integer pipe
PIC_HD bool pr_below(const double v[3], int e) {
  const uint32_t m = 0x7fffffffu;
  const uint32_t a = (uint32_t)(f64_bits(v[0]) >> 32) & m, b = (uint32_t)(f64_bits(v[1]) >> 32) & m,
                 c = (uint32_t)(f64_bits(v[2]) >> 32) & m;
  const uint32_t ab = a > b ? a : b;
  return (ab > c ? ab : c) < (uint32_t)(1023 + e) << 20;
}

template <int PUSH, int NDIM>
PIC_HD bool push_pair(double qm, double dt, int pusher, const float eb[6], double u[3], PairMove& mv) {
  // The pairs hold |u| and |q/m dt E|, |q/m dt B| below 2^28 (gamma^4 within FP32 in the
  // Higuera-Cary root); anything else, infinities and NaN among it, takes the FP64
  // push, which either moves the particle or gives a non-finite dt/gamma.
  const int kind = PUSH < 0 ? pusher : PUSH;
  const float k = fabsf(narrow_sat(qm * dt));
  float em = 0.0f;
  bool inside = pr_below(u, 28);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    em = fmaxf(em, fabsf(eb[c]));
    inside = inside && eb[c] == eb[c];
  }
  inside = inside && k * em < 0x1p28f;
  double un[3] = {u[0], u[1], u[2]};
  if (inside) {
    dfl U[3], du[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) U[d] = pr_split(u[d]);
    if (kind == PIC_ANALYTIC) {
      inside = analytic_push_pair(pr_split(qm * dt), eb, U, du);
    } else if (kind == PIC_HC) {
      hc_push_pair(pr_split(0.5 * qm * dt), eb, U, du);
    } else {
      boris_push_pair(pr_split(0.5 * qm * dt), eb, U, du);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) un[d] += pr_join(du[d]);
    inside = inside && pr_below(un, 60);
    if (inside) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        u[d] = un[d];
        U[d] = pr_add(U[d], du[d]);
      }
      const dfl ig = pr_rsqrt(pr_one_plus_sqr(U));
      const dfl dtig = pr_norm(pr_mul(pr_split(dt), ig));
#pragma unroll
      for (int d = 0; d < NDIM; ++d) mv.dx[d] = pr_mul(dtig, U[d]);
      mv.dtig = dtig.hi;
      mv.ig = ig.hi;
#pragma unroll
      for (int d = 0; d < 3; ++d) mv.u[d] = U[d].hi;
      return true;
    }
  }
  if (!push_wide(qm, dt, kind, eb, u)) return false;
  const double ig = rsqrt_nr<1>(1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
  const double dtig = dt * ig;
  // (a non-finite dt/gamma must reach the caller's check as such)
  mv.dtig = isfinite(dtig) ? narrow_signed(dtig) : NAN;
  mv.ig = narrow_signed(ig);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (d < NDIM) mv.dx[d] = pr_split(dtig * u[d]);
    mv.u[d] = narrow_signed(u[d]);
  }
  return true;
}

// the FP64 push of a particle in FP32 fields (out of line)
#ifdef __CUDA_ARCH__
__noinline__
#endif
PIC_HDI bool push_wide(double qm, double dt, int kind, const float eb[6], double u[3]) {
  double e[6];
  for (int c = 0; c < 6; ++c) e[c] = (double)eb[c];
  double v[3] = {u[0], u[1], u[2]};
  if (kind == PIC_ANALYTIC) {
    if (analytic_push_series(qm, dt, e, v) < 0) return false;
  } else if (kind == PIC_HC) {
    hc_push<1>(qm, dt, e, v);
  } else {
    boris_push<1>(qm, dt, e, v);
  }
  for (int d = 0; d < 3; ++d) u[d] = v[d];
  return true;
}

}  // namespace pic
