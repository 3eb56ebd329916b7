// Runs the library's rules for the memory of a map's box field (rmp_policy.h, host only) on
// commands read from stdin and prints one result line per command, for tests/test_map_memory.py:
//   fits BYTES ROOM FREE TOTAL -> 1 if a map gets a field of BYTES
//   keep LIVE LARGEST          -> bytes the pool keeps reserved
#include <cstdio>
#include <cstring>

#include "rmp_policy.h"

int main() {
  char op[16];
  while (std::scanf("%15s", op) == 1) {
    unsigned long long a, b, c, d;
    if (!std::strcmp(op, "fits")) {
      if (std::scanf("%llu %llu %llu %llu", &a, &b, &c, &d) != 4) return 2;
      std::printf("%d\n", rmp::box_field_fits(a, b, c, d) ? 1 : 0);
    } else if (!std::strcmp(op, "keep")) {
      if (std::scanf("%llu %llu", &a, &b) != 2) return 2;
      std::printf("%llu\n", (unsigned long long)rmp::pool_keep(a, b));
    } else {
      return 3;
    }
  }
  return 0;
}
