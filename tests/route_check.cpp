// CPU check of csrc/route.h: where the lines between the solvers lie, and that
// every CTA size is one that the resident kernel takes.
#include <cstdint>
#include <cstdio>

#include "route.h"

int main() {
  using namespace pc;
  const int nsm = 152;
  auto cols = [](int W) { return 3 * W * (W + 1) + 1; };
  // measured on both sides (us per call, wavefront / resident)
  struct Case { int W, L; long long n; double p; bool resident; } cases[] = {
      {14, 14, 1, 0.95, true},        // 145 / 70
      {14, 14, 1, 0.15, false},       // 78 / 175
      {8, 8, 10000, 0.95, true},      // 917 / 539
      {8, 8, 10000, 0.25, false},     // 405 / 720
      {8, 64, 10000, 0.185, false},   // 500 / 7,200
      {8, 48, 10000, 0.95, false},    // 5,750 / 10,470
      {25, 1, 1500, 0.5, true},
      {16, 16, 16, 0.95, true},       // 182 / 119
      {6, 96, 1024, 0.3, false},      // 449 / 4,400
      {5, 100, 600, 0.95, false},     // 388 / 1,298
      {0, 64, 64, 0.95, false},       // 139 / 220
  };
  for (const Case& c : cases)
    if ((c.p >= resident_from(c.W, cols(c.W), c.L, c.n, nsm)) != c.resident) {
      std::printf("W=%d L=%d n=%lld p=%g\n", c.W, c.L, c.n, c.p);
      return 1;
    }
  for (int W = 0; W <= 104; W += W < 30 ? 1 : 7)  // the resident kernel's columns: below 2^15
    for (int L : {1, 2, 3, 5, 8, 16, 33, 64, 300, 4096, 50000, 1 << 20}) {
      const int A = cols(W);
      if ((int64_t)(A + 1) * (L + 2) >= (int64_t)1 << 31) continue;
      double last = 0.0;
      for (long long n : {1ll, 100ll, 153ll, 1000ll, 100000ll, 1ll << 32}) {
        const double from = resident_from(W, A, L, n, nsm);
        if (!(from >= last && from > 0.0)) { std::printf("line W=%d L=%d n=%lld\n", W, L, n); return 1; }
        last = from;
        for (size_t smem : {(size_t)2000, (size_t)30000, (size_t)110000, (size_t)232448}) {
          const int t = resident_cta(A, L, n, nsm, smem, 233472);
          if (t < 64 || t > 640 || t % 64) { std::printf("cta %d W=%d L=%d n=%lld\n", t, W, L, n); return 1; }
        }
      }
    }
  // near the threshold law's own points: wider fibres percolate earlier
  if (!(fibre_threshold(8, 48) > 0.19 && fibre_threshold(16, 48) < fibre_threshold(4, 48) && fibre_threshold(20, 20) < 0.19)) {
    std::printf("threshold\n");
    return 1;
  }
  auto few = [](int W, int L, double p, long long n) { return p < few_percolate_below(W, L, n); };
  if (!few(8, 48, 0.18, 100) || few(8, 48, 0.2, 100) || few(20, 301, 0.172, 500) || few(4, 12, 0.16, 300) || !few(6, 36, 0.19, 200)) {
    std::printf("few\n");
    return 1;
  }
  std::printf("ok\n");
  return 0;
}
