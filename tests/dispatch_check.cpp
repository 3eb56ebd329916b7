// Runs the library's choices between kernels (rmp_internal.h, host only) on lines read from stdin,
// for tests/test_dispatch_rules.py:
//   N RAYS SMS -> 1 if a batch of N states takes a CTA per state, 1 if a rollout of N robots does
#include <cstdio>

#include "rmp_internal.h"

int main() {
  unsigned n, rays, sms;
  while (std::scanf("%u %u %u", &n, &rays, &sms) == 3)
    std::printf("%d %d\n", rmp::state_per_cta(n, rays, sms) ? 1 : 0,
                rmp::rollout_resident(n, rays, sms) ? 1 : 0);
  return 0;
}
