// Reads pairs of FP64 bit patterns "a d" (signed decimals) from stdin; prints
// rs_quotient(a, d, 1 / d) and a / d as hex bit patterns.
#include <cstdio>
#include <cstring>

#include "fp64_rsqrt.cuh"

int main() {
  long long a, d;
  while (std::scanf("%lld %lld", &a, &d) == 2) {
    double x, y;
    memcpy(&x, &a, sizeof x);
    memcpy(&y, &d, sizeof y);
    const double q = cqr2::rs_quotient(x, y, 1.0 / y), t = x / y;
    unsigned long long u, v;
    memcpy(&u, &q, sizeof u);
    memcpy(&v, &t, sizeof v);
    std::printf("%016llx %016llx\n", u, v);
  }
  return 0;
}
