// Reads "X Y H E" lines from stdin (H: the largest |X| of the group) and prints
// the group's shift and oz_xy_to_double_group's result as a hex bit pattern.
#include <cstdio>
#include <cstring>

#include "oz_fixed.cuh"

int main() {
  long long X, Y, H;
  int E;
  while (std::scanf("%lld %lld %lld %d", &X, &Y, &H, &E) == 4) {
    const int s = cqr2::oz_group_shift(cqr2::oz_high_bits(X) | cqr2::oz_high_bits(H));
    const double d = cqr2::oz_xy_to_double_group(X, Y, s, E);
    unsigned long long b;
    memcpy(&b, &d, sizeof b);
    std::printf("%d %016llx\n", s, b);
  }
  return 0;
}
