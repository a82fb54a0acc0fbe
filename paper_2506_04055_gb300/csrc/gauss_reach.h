// gauss_reach.h -- how far from an edge's distance a Gaussian of the radial basis has to be visited (host
// code only, no CUDA).
//
// The FP32 edge kernels contract filter weights w_ck with b_k(x) = exp(-(x - k)^2 / 2) (x: the distance in
// widths, centres k = 0 .. K - 1) and leave out whole groups of four centres far below x.  What that may
// cost depends on the weights, so the reach is worked out from them: the least X >= kLeastReach such
// that for every channel and every distance the centres left out, those of the groups that lie below
// x - X altogether, add up to at most 2^-26 of the largest term that is kept, in the filter (|w_k| b_k)
// and in its distance derivative (|w_k| |x - k| b_k).  FP32 rounds that one term to 2^-24.  Weights that do
// not allow it (a channel with nothing but far weights) end at kWholeReach, beyond which b_k is zero in
// FP32 (e^-105 is below half its smallest number).
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

namespace ctd {

constexpr float kLeastReach = 6.3246f;   // e^-20
constexpr float kWholeReach = 14.5f;
constexpr int kReachGroup = 4;           // centres are left out in groups of this many

// The first centre that an edge at x visits.
inline int first_centre(double x, double reach) {
  const int first = (int)std::ceil(x - reach);
  return first <= 0 ? 0 : first / kReachGroup * kReachGroup;
}

// w: [rows][stride], K weights in each row.
inline float gauss_reach(const float* w, int rows, int stride, int K) {
  constexpr int B = 32;   // rows at a time (compilers vectorise the fixed count)
  const double h = 0.125;
  const float most = 1.0f / 67108864.0f;   // 2^-26
  const int blocks = (rows + B - 1) / B;
  std::vector<float> t((size_t)blocks * K * B, 0.0f);   // |w| as [block][k][row]; rows of zeros lose nothing
  for (int r = 0; r < rows; ++r)
    for (int k = 0; k < K; ++k) t[((size_t)(r / B) * K + k) * B + r % B] = std::fabs(w[(size_t)r * stride + k]);
  std::vector<float> b(K), db(K), bm(K), dbm(K);
  float reach = kLeastReach;
  // Bounds over x0 <= x <= x0 + h: more than a width below x the left out terms fall with x, so their
  // largest value is that at x0; a kept term is least at an end (the derivative's: or zero inside).
  for (double x0 = std::floor((kLeastReach + 1.0 - h) / h) * h; x0 < K - 1; x0 += h) {
    for (int k = 0; k < K; ++k) {
      const double t0 = x0 - k, t1 = t0 + h, g0 = std::exp(-0.5 * t0 * t0), g1 = std::exp(-0.5 * t1 * t1);
      b[k] = (float)g0;
      db[k] = (float)(std::fabs(t0) * g0);
      bm[k] = (float)std::min(g0, g1);
      dbm[k] = t0 * t1 <= 0.0 ? 0.0f : (float)std::min(std::fabs(t0) * g0, std::fabs(t1) * g1);
    }
    for (int q = 0; q < blocks; ++q) {
      const float* v = &t[(size_t)q * K * B];
      for (int f = first_centre(x0 + h, reach); f > 0; f -= kReachGroup) {
        float lost[B] = {}, dlost[B] = {}, kept[B] = {}, dkept[B] = {};
        for (int k = 0; k < f; ++k)
          for (int r = 0; r < B; ++r) {
            lost[r] += v[k * B + r] * b[k];
            dlost[r] += v[k * B + r] * db[k];
          }
        for (int k = f; k < K; ++k)
          for (int r = 0; r < B; ++r) {
            const float x = v[k * B + r] * bm[k], y = v[k * B + r] * dbm[k];
            kept[r] = kept[r] > x ? kept[r] : x;
            dkept[r] = dkept[r] > y ? dkept[r] : y;
          }
        bool ok = true;
        for (int r = 0; r < B; ++r) ok = ok && lost[r] <= most * kept[r] && dlost[r] <= most * dkept[r];
        if (ok) break;
        // the last of these centres has to be within the reach up to x0 + h
        reach = std::min(kWholeReach, std::max(reach, (float)(x0 + h - f + 1.0) + 1e-3f));
        if (reach == kWholeReach) return reach;
      }
    }
  }
  return reach;
}

}  // namespace ctd
