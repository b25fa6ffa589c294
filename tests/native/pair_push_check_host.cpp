// The FP32-pair pushers (pair_push.cuh) and the series form of the analytic push
// (analytic_series.cuh) compiled for the host.  Reads cases from argv[1] -- int32
// count, then per case int32 kind (0 Boris, 1 analytic, 2 Higuera-Cary: the pair
// pushers; 3: the FP64 series form of the analytic push), qm, dt, E1..E3, B1..B3
// (FP32 values), u1..u3 as FP64 -- and writes per case u1..u3 after the push, the
// three moves dx (pair pushers) and 1.0 for success as FP64 to argv[2].
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
    float eb[6];
    for (int k = 0; k < 6; ++k) eb[k] = (float)v[2 + k];
    double u[3] = {v[8], v[9], v[10]}, dx[3] = {0, 0, 0};
    bool ok;
    if (kind == 3) {
      ok = pic::analytic_push_series(v[0], v[1], v + 2, u) > 0;
    } else {
      pic::PairMove mv;
      ok = pic::push_pair<-1, 3>(v[0], v[1], kind, eb, u, mv);
      for (int d = 0; d < 3; ++d) dx[d] = pic::pr_join(mv.dx[d]);
    }
    out.insert(out.end(), {u[0], u[1], u[2], dx[0], dx[1], dx[2], ok ? 1.0 : 0.0});
  }
  std::fclose(in);
  FILE* o = std::fopen(argv[2], "wb");
  if (!o) return 2;
  std::fwrite(out.data(), 8, out.size(), o);
  std::fclose(o);
  return 0;
}
