// share_line (common.cuh) for each triple "particles occupied chunk" on stdin.
#include <cstdio>

#include "common.cuh"

int main() {
  long long n, occupied, chunk;
  while (std::scanf("%lld %lld %lld", &n, &occupied, &chunk) == 3)
    std::printf("%lld\n", (long long)pic::share_line(n, occupied, chunk));
  return 0;
}
