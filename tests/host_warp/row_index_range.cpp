// Row sums of common.cuh over the last rows of a CSR matrix whose entries end
// just below 2^31 (the largest nnz the entry points accept).  The arrays are not
// there: every load is checked against [0, nnz) and answered by its position.
#include "../../paper_2609_19557_gb300/csrc/common.cuh"

#include <cstdio>
#include <cstdlib>

using namespace pdq;

static const long long kNnz = 2147483647LL;
static int *const kCol = (int *)0x100000000000;
static double *const kVal64 = (double *)0x200000000000;
static float *const kVal32 = (float *)0x300000000000;
static const double kVec[1] = {1.0};

template <typename T>
static long long position(const T *p, const T *base) {
  const long long k = ((long long)(uintptr_t)p - (long long)(uintptr_t)base) / (long long)sizeof(T);
  if (k < 0 || k >= kNnz) {
    printf("load at position %lld of %lld\n", k, kNnz);
    fflush(stdout);
    _Exit(1);
  }
  return k;
}
int load_hook(const int *p) {
  position(p, kCol);
  return 0;
}
double load_hook(const double *p) {
  if (p == kVec) return 1.0;
  position(p, kVal64);
  return 1.0;
}
float load_hook(const float *p) {
  position(p, kVal32);
  return 1.0f;
}

template <int Order>
struct One {
  static constexpr int kOrder = Order;
  template <typename I>
  double gather(I) const { return 1.0; }
  template <typename Acc>
  void add(Acc &a, Acc v, Acc x) const { a += v * x; }
};

static int fails = 0;
static void expect(const char *what, double got, double want) {
  if (got == want) return;
  printf("%s: %.17g entries summed, %.17g expected\n", what, got, want);
  ++fails;
}

// Entry ranges of 32 rows of the given lengths (in turn) that end at nnz.
template <typename Acc, typename T>
static void last_rows(const char *what, const T *val, const std::vector<int> &lens) {
  int rb[32], re[32];
  long long e = kNnz;
  for (int l = 31; l >= 0; --l) {
    re[l] = (int)e;
    e -= lens[l % lens.size()];
    rb[l] = (int)e;
  }
  static Slot<double> slots[kTileSlots];
  Slot<Acc> *buf = reinterpret_cast<Slot<Acc> *>(slots);
  double one[32], tile[32], lng[32];
  run_warp([&] {
    const int l = threadIdx.x;
    const One<0> f;
    tile[l] = tile_rows1<false, Acc>(kCol, val, rb[l], re[l], f, buf);
    // The last 8 rows, brought by lanes 0 .. 7.
    lng[l] = tile_long_rows<false, Acc>(kCol, val, l < 8 ? rb[24 + l] : 0, l < 8 ? re[24 + l] : 0, f, buf);
    one[l] = warp_row<false, Acc>(kCol, val, rb[31], re[31], f);
  });
  for (int l = 0; l < 32; ++l) {
    expect(what, tile[l], re[l] - rb[l]);
    expect(what, lng[l], re[24 + l % 8] - rb[24 + l % 8]);
    expect(what, one[l], re[31] - rb[31]);
  }
}

int main() {
  const std::vector<std::vector<int>> sets = {{1}, {3, 8, 0, 5}, {9, 31, 32}, {33, 100, 2}, {255, 256, 257}, {511, 513, 7}, {1025}};
  for (const auto &s : sets) {
    last_rows<double>("FP64", kVal64, s);
    last_rows<float>("FP32", kVal32, s);
  }
  for (int len : {1025, 1300}) {  // dense rows in entry order
    static Slot<double> buf[kTileSlots];
    double got[32];
    run_warp([&] { got[threadIdx.x] = one_row<false, double>(kCol, kVal64, (int)(kNnz - len), (int)kNnz, One<1>(), buf); });
    for (double g : got) expect("ordered", g, len);
  }
  return fails ? 1 : 0;
}
