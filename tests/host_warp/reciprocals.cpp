// Errors of recip and rsqrt_t in units in the last place of the result, over random
// mantissas and all exponents of FP32's range and beyond.
#include "../../paper_2609_19557_gb300/csrc/common.cuh"

#include <cfloat>
#include <cstdio>

int load_hook(const int *) { return 0; }
double load_hook(const double *) { return 0; }
float load_hook(const float *) { return 0; }

static uint64_t state = 1;
static uint64_t next() {  // splitmix64
  uint64_t z = state += 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
static double ulps(double got, long double want) {
  int e;
  frexpl(want, &e);
  return (double)(fabsl((long double)got - want) / ldexpl(1.0L, e - 53));
}

int main() {
  double worst[3] = {0, 0, 0};
  for (int i = 0; i < 4000000; ++i) {
    const double m = 1.0 + (double)(next() >> 12) * 0x1p-52, v = std::ldexp(m, (int)(next() % 241) - 120);
    worst[0] = max(worst[0], ulps(pdq::recip(v), 1.0L / (long double)v));
    const float f = (float)v;
    if (f > 0.0f && std::isfinite(f)) worst[1] = max(worst[1], ulps(pdq::recip(f), 1.0L / (long double)f));
    rsqrtf_off = (int)(next() % 5) - 2;
    worst[2] = max(worst[2], ulps(pdq::rsqrt_t(v), 1.0L / sqrtl((long double)v)));
  }
  printf("recip(double) %.4f, recip(float) %.4f, rsqrt_t(double) %.4f\n", worst[0], worst[1], worst[2]);
  return worst[0] > 0.51 || worst[1] > 0.51 || worst[2] > 1.01;
}
