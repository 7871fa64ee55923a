// Strict mode's looper update: where the checked double-float update accepts,
// its results are the FP64 update's bit for bit (signed zeros among them).
// Inputs: (a) magnitudes over many binades with exact zeros, signed zeros, equal
// and cancelling terms, denormals, infinities and NaN; (b) covariances just reset
// to the seed's diagonal; (c) filter-like covariances of moderate correlation,
// as the fit meets them, for the share of updates accepted.  Prints
// "wrong <n> accepted_c <share>".
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>

#include "tpc_df.cuh"
#include "tpc_fp64.cuh"

namespace {

void update_fp64(float* p, float* c, float r0, float r1, float w00, float w01, float w11) {
  const int col0[5] = {0, 1, 3, 6, 10}, col1[5] = {1, 2, 4, 7, 11};
  double h0[5], h1[5], k0[5], k1[5];
  for (int i = 0; i < 5; ++i) {
    h0[i] = c[col0[i]];
    h1[i] = c[col1[i]];
    k0[i] = h0[i] * (double)w00 + h1[i] * (double)w01;
    k1[i] = h0[i] * (double)w01 + h1[i] * (double)w11;
  }
  for (int i = 0; i < 5; ++i) p[i] = (float)((double)p[i] + (k0[i] * (double)r0 + k1[i] * (double)r1));
  int idx = 0;
  for (int i = 0; i < 5; ++i)
    for (int j = 0; j <= i; ++j, ++idx)
      c[idx] = (float)((double)c[idx] - (k0[i] * h0[j] + k1[i] * h1[j]));
}

bool same(float a, float b) { return std::memcmp(&a, &b, 4) == 0; }

}  // namespace

int main() {
  std::mt19937_64 rng(42);
  std::uniform_real_distribution<double> u(-1.0, 1.0);
  auto wild = [&](int span) {
    const int k = (int)(rng() % 64);
    if (k < 6) return 0.0f;
    if (k < 8) return -0.0f;
    if (k == 8) return 1.0f;
    if (k == 9 && span > 60) return (float)std::ldexp(u(rng), -145);
    if (k == 10 && span > 60) return INFINITY;
    if (k == 11 && span > 60) return NAN;
    return (float)std::ldexp(u(rng), (int)(rng() % (2 * span)) - span);
  };
  long wrong = 0, acc_c = 0, n_c = 0;
  for (long it = 0; it < 3000000; ++it) {
    float p[5], c[15], r0, r1, w00, w01, w11;
    const int kind = (int)(it % 3);
    if (kind == 0) {
      const int span = it % 2 ? 12 : 100;
      for (float& v : p) v = wild(span);
      for (float& v : c) v = wild(span);
      r0 = wild(span); r1 = wild(span); w00 = wild(span); w01 = wild(span); w11 = wild(span);
      if (it % 5 == 0) { c[2] = c[0]; c[1] = -c[0]; w11 = w00; w01 = -w00; }
    } else {
      // a covariance A diag A^T (or the seed's diagonal) and its own weight
      double C[5][5] = {};
      const double sd[5] = {1.0, 1.0, 0.25, 0.25, 100.0};
      if (kind == 1) {
        for (int i = 0; i < 5; ++i) C[i][i] = sd[i];
      } else {
        double L[5][5] = {};
        const double s[5] = {0.05, 0.05, 0.01, 0.01, 0.3};
        for (int i = 0; i < 5; ++i)
          for (int j = 0; j <= i; ++j) L[i][j] = s[i] * (i == j ? 0.7 + 0.3 * u(rng) : 0.6 * u(rng));
        for (int i = 0; i < 5; ++i)
          for (int j = 0; j < 5; ++j)
            for (int l = 0; l < 5; ++l) C[i][j] += L[i][l] * L[j][l];
      }
      int idx = 0;
      for (int i = 0; i < 5; ++i)
        for (int j = 0; j <= i; ++j) c[idx++] = (float)C[i][j];
      p[0] = (float)(40 * u(rng)); p[1] = (float)(5000 * u(rng)); p[2] = (float)u(rng);
      p[3] = (float)u(rng); p[4] = (float)(20 * u(rng));
      const float s00 = c[0] + 0.01f, s01 = c[1], s11 = c[2] + 0.01f;
      const float idet = 1.0f / (s00 * s11 - s01 * s01);
      w00 = s11 * idet; w01 = -s01 * idet; w11 = s00 * idet;
      r0 = (float)(0.2 * u(rng)); r1 = (float)(0.2 * u(rng));
      if (it % 64 == 1) r0 = r1 = 0.0f;
    }
    float po[5], co[15];
    const bool ok = tpc::df_update_checked(p, c, r0, r1, w00, w01, w11, po, co);
    if (kind == 2) { ++n_c; acc_c += ok; }
    if (!ok) continue;
    update_fp64(p, c, r0, r1, w00, w01, w11);
    for (int i = 0; i < 5; ++i) wrong += !same(p[i], po[i]);
    for (int i = 0; i < 15; ++i) wrong += !same(c[i], co[i]);
  }
  std::printf("wrong %ld accepted_c %.6f\n", wrong, (double)acc_c / n_c);
  return 0;
}
