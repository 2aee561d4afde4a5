// The polls of a grid barrier cover the slowest way through a row of any length:
// 64 cycles an entry in entry order, 250 cycles a poll.
#include "../../paper_2609_19557_gb300/csrc/common.cuh"

#include <cstdio>

int load_hook(const int *) { return 0; }
double load_hook(const double *) { return 0; }
float load_hook(const float *) { return 0; }

int main() {
  for (long long n : {0LL, 1000LL, 1000000LL, 20000000LL, 100000000LL, 2147483647LL}) {
    const unsigned polls = pdq::kSpinLimit + pdq::spin_more(n);
    if (polls < pdq::kSpinLimit || 250.0 * polls < 64.0 * n) {
      printf("%lld entries: %u polls\n", n, polls);
      return 1;
    }
  }
  return 0;
}
