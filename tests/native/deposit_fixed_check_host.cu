// The integer form of the FP64 deposit (deposit_fixed, particle_core.cuh) against the
// FP64 form (deposit) on the host.  Input (argv[1]): int32 count, then per case int32
// ndim, int32 l, FP64 bound (largest |w| of the tile), w, v3, and per axis f, delta,
// dx/dt.  Output (argv[2]): per case as FP64 the largest difference of the two currents
// over the nodes in units of the window's last limb, and relative to the largest value.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <map>
#include <vector>

#include "particle_core.cuh"

using namespace pic;

struct Nodes {
  std::map<int, double>* m;
  PIC_HD void add(int i, int j, int k, double v) const {
#ifndef __CUDA_ARCH__
    (*m)[(k * 16 + j) * 16 + i] += v;
#endif
  }
};
struct Units {
  std::map<int, int64_t>* m;
  int eS, l;
  PIC_HD void add_units(int i, int j, int k, int64_t y) const {
#ifndef __CUDA_ARCH__
    (*m)[(k * 16 + j) * 16 + i] += y;
#endif
  }
};

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  FILE* in = std::fopen(argv[1], "rb");
  FILE* out = std::fopen(argv[2], "wb");
  int32_t n = 0;
  if (!in || !out || std::fread(&n, 4, 1, in) != 1) return 2;
  for (int32_t c = 0; c < n; ++c) {
    int32_t h[2];
    double v[12];
    if (std::fread(h, 4, 2, in) != 2 || std::fread(v, 8, 12, in) != 12) return 2;
    const int nd = h[0];
    const double bound = v[0], w = v[1];
    const int li[3] = {5, 5, 5};
    double f[3], dl[3], cf[3];
    for (int d = 0; d < 3; ++d) {
      f[d] = v[3 + 3 * d];
      dl[d] = v[4 + 3 * d];
      cf[d] = -w * v[5 + 3 * d];
    }
    int eS, l;
    fix64_scales(1, bound, eS, l);
    l = h[1];
    std::map<int, double> a[3];
    std::map<int, int64_t> b[3];
    const Nodes na[3] = {{&a[0]}, {&a[1]}, {&a[2]}};
    const Units ub[3] = {{&b[0], eS, l}, {&b[1], eS, l}, {&b[2], eS, l}};
    if (nd == 2) {
      deposit<double, 2>(na, li, f, dl, cf, w * v[2]);
      deposit_fixed<2>(ub, li, f, dl, cf, w * v[2]);
    } else {
      deposit<double, 3>(na, li, f, dl, cf, 0.0);
      deposit_fixed<3>(ub, li, f, dl, cf, 0.0);
    }
    double worst = 0, big = 0;
    for (int k = 0; k < 3; ++k) {
      for (auto& e : b[k]) a[k][e.first] += 0.0;
      for (auto& e : a[k]) {
        const double y = std::ldexp((double)b[k][e.first], -(eS + 2 * l));
        worst = std::fmax(worst, std::fabs(y - e.second));
        big = std::fmax(big, std::fabs(e.second));
      }
    }
    const double res[2] = {worst, big};
    std::fwrite(res, 8, 2, out);
  }
  std::fclose(in);
  std::fclose(out);
  return 0;
}
