// Sums of products in three floats (tf_add_product) against the exact sum in
// 128-bit integers: n = 1 .. 160 terms, mixed signs and cancelling pairs, and the
// magnitudes that a track's gradients have in one map cell.  Prints the largest
// error in units of the bound 8 n^3 2^-72 S, and of FP64's n 2^-53 S.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <random>

#include "tpc_df.cuh"

static __int128 exact(float v) { return (__int128)std::ldexp((double)v, 62); }  // (a multiple of 2^-62)

int main() {
  std::mt19937_64 rng(7);
  std::uniform_real_distribution<double> u(-1.0, 1.0);
  double worst = 0.0, worst64 = 0.0;
  for (int it = 0; it < 200000; ++it) {
    const int n = 1 + (int)(rng() % 160);
    float hi = 0.0f, mid = 0.0f, lo = 0.0f;
    __int128 sum = 0;
    double S = 0.0;
    float a = 0.0f, b = 0.0f;
    for (int i = 0; i < n; ++i) {
      if (it % 3 == 1 && i % 2) {
        a = -a;  // cancels the term before, but for its last bits
        b = std::nextafterf(b, 2.0f * b);
      } else {
        a = (float)std::ldexp(u(rng), (int)(rng() % 16) - 8);
        b = (float)std::ldexp(it % 2 ? std::fabs(u(rng)) : u(rng), (int)(rng() % 16) - 8);
      }
      // multiples of 2^-31, so that every product is one of 2^-62
      a = (float)(std::nearbyint((double)a * 0x1p31) * 0x1p-31);
      b = (float)(std::nearbyint((double)b * 0x1p31) * 0x1p-31);
      tpc::tf_add_product(hi, mid, lo, a, b);
      const double p = (double)a * (double)b;  // exact: 48 bits
      const int64_t ia = (int64_t)((double)a * 0x1p31), ib = (int64_t)((double)b * 0x1p31);
      sum += (__int128)ia * ib;
      S += std::fabs(p);
    }
    __int128 d = exact(hi) + exact(mid) + exact(lo) - sum;
    if (d < 0) d = -d;
    const double err = (double)d * 0x1p-62;
    if (S == 0.0) continue;
    worst = std::fmax(worst, err / (8.0 * n * n * n * 0x1p-72 * S));
    worst64 = std::fmax(worst64, err / (n * 0x1p-53 * S));
  }
  std::printf("bound %.6f fp64 %.6f\n", worst, worst64);
  return 0;
}
