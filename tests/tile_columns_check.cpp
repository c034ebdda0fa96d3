// Prints tile_columns (mp_plan.cuh) for "n ncols fp64 shared nsm" lines.
#include <cstdio>

#include "mp_plan.cuh"

int main() {
  int n, fp64, shared, nsm;
  long long ncols;
  while (std::scanf("%d %lld %d %d %d", &n, &ncols, &fp64, &shared, &nsm) == 5)
    std::printf("%d\n", mp::tile_columns(n, ncols, fp64 != 0, shared != 0, nsm));
  return 0;
}
