// Host check of the kernels' tile count (layout.cuh): reads "rows B bt" and
// prints row_tiles(rows, B, bt).  Compiled with -ftrapv: an int overflow aborts.
#include <cstdio>

#include "layout.cuh"

int main() {
  int rows, B, bt;
  while (std::scanf("%d %d %d", &rows, &B, &bt) == 3) std::printf("%d\n", tsqr::row_tiles(rows, B, bt));
  return 0;
}
