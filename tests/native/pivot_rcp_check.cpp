// Reads FP64 bit patterns (signed decimals) from stdin; prints, as hex bit
// patterns, pivot_rcp(d), and chol_rsqrt_tight's 1/sqrt(d) and sqrt(d).
#include <cstdio>
#include <cstring>

#include "fp64_rsqrt.cuh"

static unsigned long long bits_of(double x) {
  unsigned long long u;
  memcpy(&u, &x, sizeof u);
  return u;
}

int main() {
  long long b;
  while (std::scanf("%lld", &b) == 1) {
    double d, r, l;
    memcpy(&d, &b, sizeof d);
    cqr2::chol_rsqrt_tight(d, &r, &l);
    std::printf("%d %016llx %016llx %016llx\n", cqr2::pivot_rcp_ok(d) ? 1 : 0, bits_of(cqr2::pivot_rcp(d)), bits_of(r),
                bits_of(l));
  }
  return 0;
}
