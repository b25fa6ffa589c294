// Addresses of field states kept one after another (common.cuh, FieldStates): prints
// for argv[1] cells the largest misalignment of a component against 16 bytes, the
// smallest distance between two components less the cells, and what the row passes
// answer for arrays off a 16-byte boundary (1: cudaErrorInvalidValue from both, before
// any launch).
#include <cstdio>
#include <cstdlib>

#include "field_halves.cu"

using namespace pic;

int main(int argc, char** argv) {
  if (argc != 2) return 2;
  const int64_t nc = std::atoll(argv[1]);
  const FieldStates<double> f{reinterpret_cast<double*>(4096), FieldStates<double>::pitch_of(nc)};
  uintptr_t off = 0;
  int64_t room = INT64_MAX;
  for (int64_t k = 0; k < 3; ++k)
    for (int m = 0; m < 6; ++m) {
      const uintptr_t a = reinterpret_cast<uintptr_t>(f.at(k, m));
      off = std::max<uintptr_t>(off, a & 15u);
      const uintptr_t b = reinterpret_cast<uintptr_t>(m < 5 ? f.at(k, m + 1) : f.at(k + 1, 0));
      room = std::min<int64_t>(room, (int64_t)(b - a) / (int64_t)sizeof(double) - nc);
    }
  // (addresses only: the check comes before any use of them)
  GridArgs g{};
  g.ndim = 2;
  StencilArgs<double> s{};
  s.M = 16;
  bool refused = true;
  for (int which = 0; which < 2; ++which) {
    FieldPtrs<double> a{}, o{};
    double* p = reinterpret_cast<double*>(4096);
    for (int c = 0; c < 3; ++c) a.e[c] = a.b[c] = o.e[c] = o.b[c] = p;
    (which ? o.b[2] : a.b[1]) = p + 1;
    refused = refused && launch_faraday<double>(a, o, nullptr, g, s, nullptr, nullptr) == cudaErrorInvalidValue;
    refused = refused && launch_ampere<double>(a, o, g, s, nullptr) == cudaErrorInvalidValue;
  }
  std::printf("%d %lld %d\n", (int)off, (long long)room, refused ? 1 : 0);
  return 0;
}
