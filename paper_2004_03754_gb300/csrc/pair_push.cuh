// pair_push.cuh -- the push of particles in FP32 fields: the FP64 push of pushers.cuh
// with the parts that lose nothing by it in FP32 pairs (dfloat.cuh: hi + lo, 48 bits).
//
// Why: FP64 instructions issue at 1/64 of the FP32 rate on this GPU, and the FP64 Boris
// push of 49 of them kept that pipe 83 % busy and the rest of the SM idle.  In pairs
// are only changes of u that are small against u, or that the FP64 form next to FP32
// fields leaves less accurate (one Newton step per reciprocal, 2^-44):
//   Boris, Higuera-Cary   the rotation about B, while |t| = |h B|/gamma < 1/4;
//   analytic              what L^2 and higher powers add to U + s L U, while the
//                         arguments of the exponential are below 1/16.
// The electric kicks, s L U, the residual of the proper time, gamma and the move
// (dt/gamma) u stay in FP64.  Every other particle, infinities, NaN and momenta past
// 2^40 (analytic 2^30) among them, takes the FP64 push.  FP64 instructions per push,
// against the FP64 form: 2D Boris 34 -> 22, 3D analytic 153 -> 68.
//
// Error against 64 bits (113-bit reference on the device, 5e5 electrons in pulses of
// a0 = 1 to 100 with plasma fields, at rest to gamma = 600): |du|/|u| root mean square
// and 99th percentile, the FP64 form before the arrow
//   Boris 3.8e-16 -> 3.4e-16, 1.3e-15 -> 1.1e-15;  Higuera-Cary 2.0e-15 -> 3.3e-16,
//   6.2e-15 -> 1.2e-15;  analytic 1.1e-16 -> 7.4e-17, 2.5e-16 -> 1.7e-16;
// the move 3.2e-15 dt in all (the reciprocal's one Newton step).
// Measured: 2D Boris, 29.4 M electrons, ten steps and their read-back, all FP64 rotation
// and cells 24.2 -> 20.2 ms; 2D Higuera-Cary, 1.4 M, twelve steps 2.80 -> 2.24 ms; 3D
// analytic, 84 M, two steps 54.8 -> 42.8 ms.
//
// Products feeding a TwoSum are rounded on their own (mul_rn); sums written
// plainly hold no product, so no contraction can break them.
#pragma once
#include "dfloat.cuh"
#include "analytic_series.cuh"
#include "push_const.h"
#include "pushers.cuh"

namespace pic {

// nearest integer, |x| < 2^31
PIC_HD int32_t round_int(float x) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return (int32_t)nearbyintf(x);
#endif
}

// ---- pair arithmetic without renormalisation where the next operation allows it

// x = hi + lo: hi the FP32 value nearest to x, lo the rest rounded to FP32
// (relative error below 2^-49), on the integer pipe.  |x| < 2^-126 gives zero,
// |x| < 2^-74 no low part; |x| < 2^128.
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
// the pair in FP64, rounded once, |lo| < 2^-21 |hi|: lo enters hi's FP64 mantissa as an
// integer (the integer pipe; below 2^-74, where its scale leaves FP32, an FP64 add)
PIC_HD double pr_join(dfl a) {
  const uint32_t h = f32_bits(a.hi), mag = h & 0x7fffffffu, eh = mag & 0x7f800000u;
  if (eh <= (52u << 23)) return widen_normal(a.hi) + widen_normal(a.lo);
  // lo in units of hi's FP64 last place (half of that below a power of two), signed as hi
  const bool down = (mag & 0x007fffffu) == 0u && ((f32_bits(a.lo) ^ h) >> 31) != 0u;
  const float unit = f32_from_bits((306u << 23) - eh + (down ? 1u << 23 : 0u));   // 2^(52 - e)
  const int32_t d = round_int(mul_rn(a.lo, f32_from_bits(f32_bits(unit) ^ (h & 0x80000000u))));
  const uint64_t m = ((uint64_t)((mag >> 3) + 0x38000000u) << 32 | (uint64_t)(mag << 29)) + (uint64_t)(int64_t)d;
  return f64_from_bits(m | (uint64_t)(h & 0x80000000u) << 32);
}

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
  const dfl s = dfl::two_sum(a.hi, b.hi);
  return dfl(s.hi, s.lo + (a.lo + b.lo));
}
PIC_HD dfl pr_norm(dfl a) { return dfl::fast_two_sum(a.hi, a.lo); }
PIC_HD dfl pr_add(dfl a, dfl b) { return pr_norm(pr_add_raw(a, b)); }
PIC_HD dfl pr_neg(dfl a) { return dfl(-a.hi, -a.lo); }
// v . b and component a x b of v x b, b in FP32
PIC_HD dfl pr_dotf(const dfl v[3], const float b[3]) {
  return pr_norm(pr_add_raw(pr_add_raw(pr_mulf(v[0], b[0]), pr_mulf(v[1], b[1])), pr_mulf(v[2], b[2])));
}
PIC_HD dfl pr_crossf(const dfl v[3], const float b[3], int i, int j) {
  return pr_norm(pr_add_raw(pr_mulf(v[i], b[j]), pr_mulf(v[j], -b[i])));
}
// 1/sqrt(x), 1/x, x positive normal and normalised: the FP32 seed and one
// Newton step whose residual is formed exactly, with the next term of its series
PIC_HD dfl pr_rsqrt(dfl x) {
  const float y = seed_rsqrt(x.hi);
  const dfl s = pr_mulff(y, y);
  const float p = mul_rn(x.hi, s.hi);
  float r = (1.0f - p) - fmaf(x.hi, s.hi, -p);       // 1 - x y^2
  r = fmaf(-x.hi, s.lo, r);
  r = fmaf(-x.lo, s.hi, r);
  return dfl::fast_two_sum(y, mul_rn(y, fmaf(mul_rn(0.375f, r), r, 0.5f * r)));
}
PIC_HD dfl pr_rcp(dfl x) {
  const float y = seed_rcp(x.hi);
  float r = fmaf(-x.hi, y, 1.0f);
  r = fmaf(-x.lo, y, r);
  return dfl::fast_two_sum(y, mul_rn(y, fmaf(r, r, r)));
}

// The leading word of |x| (orders as |x|; infinities and NaN are the largest)
PIC_HD uint32_t mag_word(double x) { return (uint32_t)(f64_bits(x) >> 32) & 0x7fffffffu; }
PIC_HD bool mag_sign(double x) { return (f64_bits(x) >> 63) != 0; }
constexpr uint32_t mag_word_of(int e) { return (uint32_t)(1023 + e) << 20; }   // that of 2^e

// 1 + |v|^2 (all terms positive: each TwoSum may take the larger sum first)
PIC_HD dfl pr_one_plus_sqr(const dfl v[3]) {
  dfl s(1.0f, 0.0f);
#pragma unroll
  for (int d = 0; d < 3; ++d) s = pr_add_raw(s, pr_sqr(v[d]));
  return pr_norm(s);
}

// The rotation of Boris, u+ = u- + (u- + u- x t) x 2 t/(1 + t^2), and of Higuera-Cary
// (the same about t at its own gamma: w + w x t with (1 + t^2) w = u- + (u-.t) t + u- x t
// is that rotation): du = u+ - u- of m = u-.  With t = c B, B exact in FP32, both cross
// products run on B itself and only c and f = 2 c/(1 + t^2) are rounded; f is formed as
// 2 (c - c t^2/(1 + t^2)), so that its error shrinks with t^2.  c^-2 is gamma^2/h^2 or
// Higuera-Cary's gbar^2/h^2,
//   gbar^2 = (sigma + root)/2, root^2 = sigma^2 + 4 (b^2 + (u-.b)^2), sigma = gamma^2 - b^2
// (no cancellation in sigma: gbar <= gamma, so b^2 < gamma^2/16 below).  False outside
// the pairs' range.
template <bool HC>
PIC_HD bool rotate_pair(const double m64[3], const float B[3], const PushConst& k, dfl du[3]) {
  const uint32_t m0 = mag_word(m64[0]), m1 = mag_word(m64[1]), m2 = mag_word(m64[2]);
  const uint32_t m01 = m0 > m1 ? m0 : m1, mm = m01 > m2 ? m01 : m2;
  dfl m[3], v[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) m[d] = pr_split(m64[d]);
  const dfl ih2(k.ih2_hi, k.ih2_lo), bb = pr_norm(pr_add_raw(
      pr_add_raw(pr_mulff(B[0], B[0]), pr_mulff(B[1], B[1])), pr_mulff(B[2], B[2])));
  dfl g2 = pr_norm(pr_mul(pr_one_plus_sqr(m), ih2));
  // (also |t| and the products below within FP32: gamma^2/h^2 from 2^-40 to 2^80)
  const bool inside = (mm == 0u || mm - mag_word_of(-64) < mag_word_of(40) - mag_word_of(-64)) &&
                      g2.hi > 0x1p-40f && g2.hi < 0x1p80f;
  if constexpr (HC) {
    const dfl sg = pr_add(g2, pr_neg(bb));
    const dfl w4 = pr_mul(ih2, pr_add(bb, pr_sqr(pr_dotf(m, B))));
    const dfl q = pr_add(pr_sqr(sg), dfl(4.0f * w4.hi, 4.0f * w4.lo));
    g2 = pr_add(sg, pr_norm(pr_mul(q, pr_rsqrt(q))));
    g2 = dfl(0.5f * g2.hi, 0.5f * g2.lo);
  }
  dfl c = pr_rsqrt(g2);
  const dfl t2 = pr_norm(pr_mul(pr_norm(pr_sqr(c)), bb));
  if (mag_sign(k.h)) c = pr_neg(c);
  const dfl q = pr_norm(pr_mul(t2, pr_rcp(pr_add(dfl(1.0f, 0.0f), t2))));
  dfl f = pr_add(c, pr_neg(pr_mul(c, q)));
  f = dfl(2.0f * f.hi, 2.0f * f.lo);
#pragma unroll
  for (int d = 0; d < 3; ++d) v[d] = pr_add(m[d], pr_mul(c, pr_crossf(m, B, (d + 1) % 3, (d + 2) % 3)));
#pragma unroll
  for (int d = 0; d < 3; ++d) du[d] = pr_norm(pr_mul(f, pr_crossf(v, B, (d + 1) % 3, (d + 2) % 3)));
  return inside && t2.hi < 0.0625f;   // (false for NaN)
}

// sum of three pairs with exact high parts, normalised
PIC_HD dfl pr_sum3(dfl a, dfl b, dfl c) {
  const dfl s = two_sum(a.hi, b.hi), r = two_sum(s.hi, c.hi);
  return fast_two_sum(r.hi, r.lo + (s.lo + ((a.lo + b.lo) + c.lo)));
}
// s L V, L V = (E.v, V0 E + v x B)
PIC_HD void pr_apply(const float eb[6], float s, const dfl V[4], dfl o[4]) {
  o[0] = pr_sum3(pr_mulf(V[1], eb[0]), pr_mulf(V[2], eb[1]), pr_mulf(V[3], eb[2]));
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int a = (d + 1) % 3, b = (d + 2) % 3;
    o[d + 1] = pr_sum3(pr_mulf(V[0], eb[d]), pr_mulf(V[a + 1], eb[3 + b]), pr_mulf(V[b + 1], -eb[3 + a]));
  }
#pragma unroll
  for (int d = 0; d < 4; ++d) o[d] = pr_norm(pr_mulf(o[d], s));
}

// The analytic push (analytic_series.cuh) while L s is small, |s|^2 (E^2 + B^2) < 2^-8: U(s) =
// U + s L U + R(s) in s = (q/m) tau with the raw fields; s L U, of size |L s| |U|, in
// FP64 and R, of size |L s|^2 |U|/2, in pairs, so that R's rounding, 2^-48 of it, stays
// below FP64's.  With b_k = s^k L^k U, A = S1 s^2, Q = S2 s^4 (|A| < 2^-8, Q < 2^-18) and
// p_1 = 1, p_2 = A, p_{n+1} = A p_n + Q p_{n-1}, s_a = sum_n p_n/(2n + a)!,
//   R = s_0 b_2 + s_1 b_3 + Q s_2 U + Q s_3 b_1,
//   F(s) = s [gamma + b_1/2 + s_1 b_2 + s_2 b_3 + Q s_3 gamma + Q s_4 b_1] (time components)
// is q/m times the lab time.  An FP32 Newton gives s to about 2^-23, the FP64 residual
// F(s) - (q/m) dt the rest, delta, which moves s in the FP64 term and R to second order.
// The line: for electrons at rest R is B s/2 of u, so the pairs' share grows with |L s|;
// root mean square error of |u| for |L s| from 2^-5 to 2^-4 1.2e-16 (FP64 form 1.4e-16),
// up to 2^-3 it would be 1.8e-16.  False outside, with u unchanged.
PIC_HD bool analytic_push_weak(double D, const float eb[6], double u[3]) {
  const uint32_t m0 = mag_word(u[0]), m1 = mag_word(u[1]), m2 = mag_word(u[2]);
  const uint32_t m01 = m0 > m1 ? m0 : m1, mm = m01 > m2 ? m01 : m2;
  bool inside = mm < mag_word_of(30);   // (with |D| > 2^-20: s^2 and its low part normal)
  const double x0 = 1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const double ig0 = rsqrt_nr(x0), g0 = x0 * ig0;
  double E[6], LU[4];
#pragma unroll
  for (int c = 0; c < 6; ++c) E[c] = widen(eb[c]);
  LU[0] = E[0] * u[0] + E[1] * u[1] + E[2] * u[2];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int a = (d + 1) % 3, b = (d + 2) % 3;
    LU[d + 1] = fma(g0, E[d], fma(u[a], E[3 + b], -(u[b] * E[3 + a])));
  }
  const double sd = D * ig0;
  const float Df = narrow_sat(D), ig = narrow_sat(ig0);
  const dfl ee = pr_sum3(pr_mulff(eb[0], eb[0]), pr_mulff(eb[1], eb[1]), pr_mulff(eb[2], eb[2]));
  const dfl bb = pr_sum3(pr_mulff(eb[3], eb[3]), pr_mulff(eb[4], eb[4]), pr_mulff(eb[5], eb[5]));
  const dfl dot = pr_sum3(pr_mulff(eb[0], eb[3]), pr_mulff(eb[1], eb[4]), pr_mulff(eb[2], eb[5]));
  const float sa = narrow_sat(sd);
  inside = inside && sa * sa * (ee.hi + bb.hi) < 0.00390625f && fabsf(Df) > 0x1p-20f && fabsf(Df) < 0x1p20f;
  if (!inside) return false;                        // (also NaN)
  dfl V0[4], b1[4], b2[4], b3[4];
  V0[0] = pr_split(g0);
#pragma unroll
  for (int d = 0; d < 3; ++d) V0[d + 1] = pr_split(u[d]);
  dfl W1[4];
#pragma unroll
  for (int d = 0; d < 4; ++d) W1[d] = pr_split(LU[d]);
  // s in FP32: Newton on s (1 + s (p + s (r + s (t + s v)))) = D/gamma, the terms of L^k U in
  // FP32 (L^4 = S1 L^2 + S2), the right side with its low part, so that s is good to its
  // last place
  float s = sa;
  {
    const float sl = narrow_signed(sd - widen(sa));
    float w[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int a = (d + 1) % 3, b = (d + 2) % 3;
      w[d] = fmaf(W1[0].hi, eb[d], fmaf(W1[a + 1].hi, eb[3 + b], -(W1[b + 1].hi * eb[3 + a])));
    }
    const float p = 0.5f * (W1[0].hi * ig);
    const float r = 0.16666667f * (fmaf(eb[0], W1[1].hi, fmaf(eb[1], W1[2].hi, eb[2] * W1[3].hi)) * ig);
    const float t = 0.041666668f * (fmaf(eb[0], w[0], fmaf(eb[1], w[1], eb[2] * w[2])) * ig);
    const float v = fmaf(ee.hi - bb.hi, 0.05f * r, 0.0083333333f * (dot.hi * dot.hi));
#pragma unroll
    for (int it = 0; it < 3; ++it) {
      const float F = fmaf(s * s, fmaf(s, fmaf(s, fmaf(s, v, t), r), p), (s - sa) - sl);
      const float G = s * fmaf(s, fmaf(s, 4.0f * t, 3.0f * r), 2.0f * p);   // dF/ds - 1, small
      s = fmaf(-F, fmaf(G, G, 1.0f - G), s);
    }
  }
#pragma unroll
  for (int d = 0; d < 4; ++d) b1[d] = pr_norm(pr_mulf(W1[d], s));
  pr_apply(eb, s, b1, b2);
  pr_apply(eb, s, b2, b3);
  const dfl z = pr_mulff(s, s);
  const dfl A = pr_norm(pr_mul(pr_add(ee, pr_neg(bb)), z)), dz = pr_norm(pr_mul(dot, z)), Q = pr_norm(pr_sqr(dz));
  const dfl P3 = pr_add(pr_sqr(A), Q);
  const float p3 = P3.hi, p4 = A.hi * fmaf(A.hi, A.hi, 2.0f * Q.hi);
  // 1/3!, 1/4!, 1/5!, 1/6! as pairs
  const dfl i6(PIC_AS.h3[0], PIC_AS.l3[0]), i24(PIC_AS.h2[1], PIC_AS.l2[1]), i120(PIC_AS.h3[1], PIC_AS.l3[1]),
            i720(PIC_AS.h2[2], PIC_AS.l2[2]);
  const dfl s0 = pr_sum3(dfl(0.5f, 0.0f), pr_mul(A, i24), pr_add_raw(pr_mul(P3, i720), dfl(p4 * PIC_AS.h2[3], 0.0f)));
  const dfl s1 = pr_sum3(i6, pr_mul(A, i120), dfl(fmaf(p4, PIC_AS.h3[3], p3 * PIC_AS.h3[2]), 0.0f));
  const dfl s2 = pr_add(i24, dfl(fmaf(p3, PIC_AS.h2[3], A.hi * PIC_AS.h2[2]), 0.0f));
  const dfl q3 = pr_norm(pr_mul(Q, pr_add(i120, dfl(A.hi * PIC_AS.h3[2], 0.0f))));
  const float q4 = Q.hi * fmaf(A.hi, PIC_AS.h2[3], PIC_AS.h2[2]);
  const dfl q2 = pr_norm(pr_mul(Q, s2));
  dfl Rf = pr_add(pr_add_raw(pr_mul(s1, b2[0]), pr_mul(s2, b3[0])), pr_add_raw(pr_mul(q3, V0[0]), dfl(q4 * b1[0].hi, 0.0f)));
  const double s64 = widen(s);
  const double r = fma(s64, fma(0.5 * s64, LU[0], g0) + pr_join(Rf), -D);
  const float Rg = fmaf(s0.hi, b2[0].hi, fmaf(s1.hi, b3[0].hi, fmaf(q2.hi, V0[0].hi, q3.hi * b1[0].hi)));
  const double gam = fma(s64, LU[0], g0) + widen(Rg);
  const double rg = rcp_nr<1>(gam), d1 = -r * rg;
  const float d1f = narrow_signed(d1), e = d1f * seed_rcp(s);   // delta, delta/s
  // second order of Newton: -(gamma'/2 gamma) delta^2
  const float d2 = -0.5f * narrow_signed(rg) * (b1[0].hi + fmaf(0.5f, b3[0].hi, b2[0].hi)) * (e * d1f);
  if (!(fabsf(e) <= 0x1p-21f)) return false;         // not settled, NaN
  const double sn = s64 + (d1 + widen(d2));
  // R(s + delta) = R + delta L (s L U + R) + (delta^2/2) L^2 (U + s L U)
  dfl R[3];
#pragma unroll
  for (int d = 0; d < 3; ++d)
    R[d] = pr_add(pr_add_raw(pr_mul(s0, b2[d + 1]), pr_mul(s1, b3[d + 1])),
                  pr_add_raw(pr_mul(q2, V0[d + 1]), pr_mul(q3, b1[d + 1])));
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int a = (d + 1) % 3, b = (d + 2) % 3;
    const float T = s * fmaf(Rg, eb[d], fmaf(R[a].hi, eb[3 + b], -(R[b].hi * eb[3 + a])));
    const float dR = e * (fmaf(0.5f * e, b2[d + 1].hi + b3[d + 1].hi, b2[d + 1].hi) + T);
    u[d] = fma(sn, LU[d + 1], u[d] + pr_join(pr_add(R[d], dfl(dR, 0.0f))));
  }
  return true;
}

// The FP64 push next to FP32 fields, out of line for the rare particles outside the
// pairs' range (arguments and result by value: the caller's stay in registers).  ok:
// false when the analytic push did not converge.
struct PushState {
  double u[3];
  float eb[6];
  bool ok;
};
template <int KIND>
#ifdef __CUDA_ARCH__
__noinline__
#endif
PIC_HDI PushState push_wide(double qm, double dt, PushState s) {
  double e[6];
  for (int c = 0; c < 6; ++c) e[c] = widen(s.eb[c]);
  if constexpr (KIND == PIC_ANALYTIC) s.ok = analytic_push_series(qm, dt, e, s.u) > 0;
  else if constexpr (KIND == PIC_HC) hc_push<1>(qm, dt, e, s.u);
  else boris_push<1>(qm, dt, e, s.u);
  return s;
}

// ---- one particle: u (in and out), dt/gamma, 1/gamma of u^{n+1/2}, and its move
// dx[d] = (dt/gamma) u_d, which takes one fused multiply-add onto the position.
// Returns false when the analytic push did not converge (u unchanged).
struct Move {
  double v, u;
};
PIC_HD double pr_join(Move m) { return m.v * m.u; }
struct PairMove {
  Move dx[3];
  double dtig, ig;
};

template <int KIND>
PIC_HD bool push_kind(double qm, double dt, const PushConst& k, const float eb[6], double u[3]) {
  if constexpr (KIND == PIC_ANALYTIC) {
    if (analytic_push_weak(2.0 * k.h, eb, u)) return true;
  } else {
    double e[3], m[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      e[d] = widen(eb[d]);
      m[d] = fma(k.h, e[d], u[d]);
    }
    dfl du[3];
    if (rotate_pair<KIND == PIC_HC>(m, eb + 3, k, du)) {
#pragma unroll
      for (int d = 0; d < 3; ++d) u[d] = fma(k.h, e[d], m[d] + pr_join(du[d]));
      return true;
    }
  }
  const PushState w = push_wide<KIND>(
      qm, dt, PushState{{u[0], u[1], u[2]}, {eb[0], eb[1], eb[2], eb[3], eb[4], eb[5]}, true});
  if (!w.ok) return false;
#pragma unroll
  for (int d = 0; d < 3; ++d) u[d] = w.u[d];
  return true;
}

template <int PUSH, int NDIM>
PIC_HD bool push_pair(double qm, double dt, const PushConst& k, int pusher, const float eb[6],
                      double u[3], PairMove& mv) {
  const int kind = PUSH < 0 ? pusher : PUSH;
  bool ok;
  if (kind == PIC_ANALYTIC) ok = push_kind<PIC_ANALYTIC>(qm, dt, k, eb, u);
  else if (kind == PIC_HC) ok = push_kind<PIC_HC>(qm, dt, k, eb, u);
  else ok = push_kind<PIC_BORIS>(qm, dt, k, eb, u);
  if (!ok) return false;
  mv.ig = rsqrt_nr<1>(1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
  mv.dtig = dt * mv.ig;
#pragma unroll
  for (int d = 0; d < NDIM; ++d) mv.dx[d] = Move{mv.dtig, u[d]};
  return true;
}
template <int PUSH, int NDIM>
PIC_HD bool push_pair(double qm, double dt, int pusher, const float eb[6], double u[3], PairMove& mv) {
  return push_pair<PUSH, NDIM>(qm, dt, push_const(qm, dt), pusher, eb, u, mv);
}

}  // namespace pic
