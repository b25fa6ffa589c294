// Errors of the push of particles in FP32 fields (pair_push.cuh) and of the FP64 push
// with one Newton step per reciprocal (pushers.cuh, the analytic one in its eigenvalue
// form), against the same push in long double, compiled for the host.  Reads cases from
// argv[1] -- int32 count, then per case int32 kind (pic.h), qm, dt, E1..E3, B1..B3,
// u1..u3 as FP64 -- and writes per case to argv[2]: |u error|/|u| of the former and the
// latter, |error of the move|/dt of both.  Also compares the cell and FP32 fraction of
// a coordinate (fpbits.cuh) with its FP64 form; exits 3 if they differ.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <vector>

#include "pic.h"

#include "pair_push.cuh"

typedef long double L;

static L dot(const L* a, const L* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }
static void cross(const L* a, const L* b, L* o) {
  for (int d = 0; d < 3; ++d) {
    const int i = (d + 1) % 3, j = (d + 2) % 3;
    o[d] = a[i] * b[j] - a[j] * b[i];
  }
}

static void reference(int kind, const double* v, L* u) {
  const L qm = v[0], dt = v[1], h = qm * dt / 2, E[3] = {v[2], v[3], v[4]}, B[3] = {v[5], v[6], v[7]};
  for (int d = 0; d < 3; ++d) u[d] = v[8 + d];
  if (kind != PIC_ANALYTIC) {   // the rotation about t = h B / gamma (gbar for Higuera-Cary)
    L m[3], b[3], t[3], w[3], c[3];
    for (int d = 0; d < 3; ++d) {
      m[d] = u[d] + h * E[d];
      b[d] = h * B[d];
    }
    L g2 = 1 + dot(m, m);
    if (kind == PIC_HC) {
      const L b2 = dot(b, b), us = dot(m, b), sg = g2 - b2, root = sqrtl(sg * sg + 4 * (b2 + us * us));
      g2 = sg >= 0 ? (sg + root) / 2 : 2 * (b2 + us * us) / (root - sg);
    }
    for (int d = 0; d < 3; ++d) t[d] = b[d] / sqrtl(g2);
    cross(m, t, c);
    for (int d = 0; d < 3; ++d) w[d] = m[d] + c[d];
    cross(w, t, c);
    for (int d = 0; d < 3; ++d) u[d] = m[d] + 2 * c[d] / (1 + dot(t, t)) + h * E[d];
    return;
  }
  // power series of exp(L tau) U, the proper time by bracketed Newton
  const int K = 60;
  static L V[K + 1][4];
  L e[3], b[3];
  for (int d = 0; d < 3; ++d) {
    e[d] = qm * E[d];
    b[d] = qm * B[d];
  }
  V[0][0] = sqrtl(1 + dot(u, u));
  for (int d = 0; d < 3; ++d) V[0][d + 1] = u[d];
  for (int n = 0; n < K; ++n) {
    L c[3];
    cross(V[n] + 1, b, c);
    V[n + 1][0] = dot(e, V[n] + 1);
    for (int d = 0; d < 3; ++d) V[n + 1][d + 1] = V[n][0] * e[d] + c[d];
  }
  L tau = dt / V[0][0], lo = 0, hi = dt;
  for (int it = 0; it < 60; ++it) {
    L c = 1, t = 0, g = 0;
    for (int n = 0; n <= K; ++n) {
      g += V[n][0] * c;
      c *= tau / (n + 1);
      t += V[n][0] * c;
    }
    (t > dt ? hi : lo) = tau;
    L tn = tau - (t - dt) / g;
    if (!(tn >= lo && tn <= hi)) tn = (lo + hi) / 2;
    tau = tn;
  }
  L c = 1;
  for (int d = 0; d < 3; ++d) u[d] = 0;
  for (int n = 0; n <= K; ++n) {
    for (int d = 0; d < 3; ++d) u[d] += V[n][d + 1] * c;
    c *= tau / (n + 1);
  }
}

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  FILE* in = std::fopen(argv[1], "rb");
  if (!in) return 2;
  int32_t n = 0;
  if (std::fread(&n, 4, 1, in) != 1 || n < 0) return 2;
  std::vector<double> out;
  for (int32_t q = 0; q < n; ++q) {
    int32_t kind = 0;
    double v[11];
    if (std::fread(&kind, 4, 1, in) != 1 || std::fread(v, 8, 11, in) != 11) return 2;
    float ef[6];
    double eb[6];
    for (int k = 0; k < 6; ++k) eb[k] = ef[k] = (float)v[2 + k];
    L r[3];
    reference(kind, v, r);
    const L rn = sqrtl(dot(r, r)), g = sqrtl(1 + dot(r, r));
    double u[2][3], dtig[2], e[4];
    for (int f = 0; f < 2; ++f) {
      for (int d = 0; d < 3; ++d) u[f][d] = v[8 + d];
      if (f == 0) {
        pic::PairMove mv;
        if (!pic::push_pair<-1, 3>(v[0], v[1], kind, ef, u[f], mv)) return 4;
        dtig[f] = mv.dtig;
      } else {
        if (kind == PIC_ANALYTIC) pic::analytic_push(v[0], v[1], eb, u[f]);
        else if (kind == PIC_HC) pic::hc_push<1>(v[0], v[1], eb, u[f]);
        else pic::boris_push<1>(v[0], v[1], eb, u[f]);
        dtig[f] = v[1] * pic::rsqrt_nr<1>(1.0 + u[f][0] * u[f][0] + u[f][1] * u[f][1] + u[f][2] * u[f][2]);
      }
      L s = 0, x = 0;
      for (int d = 0; d < 3; ++d) {
        const L a = u[f][d] - r[d], b = (L)dtig[f] * u[f][d] - (L)v[1] * r[d] / g;
        s += a * a;
        x += b * b;
      }
      e[f] = rn > 0 ? (double)(sqrtl(s) / rn) : (double)sqrtl(s);
      e[2 + f] = (double)(sqrtl(x) / v[1]);
    }
    out.insert(out.end(), e, e + 4);
    for (double c : {std::fabs(v[8]), std::fabs(v[9]) * 1e6, v[1], std::fabs(v[10]) * 1e-9, (double)q,
                     q + 1.0 - 1.2e-7, std::nextafter((double)q, 0.0)}) {
      if (!(c < 2147483648.0)) continue;
      float f32;
      double f64;
      if (pic::floor_split(c, f32) != pic::floor_split(c, f64)) return 3;
      if (f32 != (float)f64) return 3;
    }
  }
  std::fclose(in);
  FILE* o = std::fopen(argv[2], "wb");
  if (!o) return 2;
  std::fwrite(out.data(), 8, out.size(), o);
  std::fclose(o);
  return 0;
}
