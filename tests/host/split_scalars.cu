// Host check of the integer conversions of split.cuh and device.cuh (the same
// functions the kernels call, compiled for the host): reads "s P e", "d bits"
// or "f bits" (decimal) and prints the result's bits: split_to_double(P, e),
// f32_of(binary64), f64_of(binary32).
#include <cstdio>
#include <cstring>

#include "split.cuh"

int main() {
  char k;
  while (std::scanf(" %c", &k) == 1) {
    unsigned long long b = 0;
    if (k == 's') {
      long long P;
      int e;
      if (std::scanf("%lld %d", &P, &e) != 2) return 2;
      const double x = tsqr::split_to_double(P, e);
      std::memcpy(&b, &x, 8);
    } else if (std::scanf("%llu", &b) != 1) {
      return 2;
    } else if (k == 'd') {
      double x;
      std::memcpy(&x, &b, 8);
      const float y = tsqr::f32_of(x);
      b = 0;
      std::memcpy(&b, &y, 4);
    } else {
      const uint32_t w = static_cast<uint32_t>(b);
      float x;
      std::memcpy(&x, &w, 4);
      const double y = tsqr::f64_of(x);
      std::memcpy(&b, &y, 8);
    }
    std::printf("%llu\n", b);
  }
  return 0;
}
