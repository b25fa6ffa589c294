// The push of particles in FP32 fields (pair_push.cuh) beside the FP64 push it stands
// for (pushers.cuh, analytic_series.cuh), compiled for the host.  Reads cases from
// argv[1] -- int32 count, then per case int32 kind (pic.h), qm, dt, E1..E3, B1..B3,
// u1..u3 as FP64 -- and writes per case to argv[2], for each of the two pushes: u1..u3,
// the three moves, dt/gamma, and 1.0 for success.
#include <cstdint>
#include <cstdio>
#include <vector>

#include "pic.h"

#include "pair_push.cuh"

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  FILE* in = std::fopen(argv[1], "rb");
  if (!in) return 2;
  int32_t n = 0;
  if (std::fread(&n, 4, 1, in) != 1 || n < 0) return 2;
  std::vector<double> out;
  for (int32_t c = 0; c < n; ++c) {
    int32_t kind = 0;
    double v[11];
    if (std::fread(&kind, 4, 1, in) != 1 || std::fread(v, 8, 11, in) != 11) return 2;
    float ef[6];
    double eb[6];
    for (int k = 0; k < 6; ++k) eb[k] = ef[k] = (float)v[2 + k];
    {
      double u[3] = {v[8], v[9], v[10]};
      pic::PairMove mv{};
      const bool ok = pic::push_pair<-1, 3>(v[0], v[1], kind, ef, u, mv);
      out.insert(out.end(), {u[0], u[1], u[2], pic::pr_join(mv.dx[0]), pic::pr_join(mv.dx[1]),
                             pic::pr_join(mv.dx[2]), (double)mv.dtig, ok ? 1.0 : 0.0});
    }
    {
      double u[3] = {v[8], v[9], v[10]};
      int it = 1;
      if (kind == PIC_ANALYTIC) it = pic::analytic_push_series(v[0], v[1], eb, u);
      else if (kind == PIC_HC) pic::hc_push<1>(v[0], v[1], eb, u);
      else pic::boris_push<1>(v[0], v[1], eb, u);
      const double dtig = v[1] * pic::rsqrt_nr<1>(1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
      out.insert(out.end(), {u[0], u[1], u[2], dtig * u[0], dtig * u[1], dtig * u[2], dtig,
                             it > 0 ? 1.0 : 0.0});
    }
  }
  std::fclose(in);
  FILE* o = std::fopen(argv[2], "wb");
  if (!o) return 2;
  std::fwrite(out.data(), 8, out.size(), o);
  std::fclose(o);
  return 0;
}
