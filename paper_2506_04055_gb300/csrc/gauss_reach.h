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

// Bounds of the terms over x0 <= x <= x0 + h: more than a width below x the left out ones fall with x, so
// their largest value is that at x0; a kept one is least at an end (the derivative's: or zero inside).
struct ReachBounds {
  float b[64], db[64], bm[64], dbm[64];
  ReachBounds(double x0, double h, int K) {
    for (int k = 0; k < K; ++k) {
      const double t0 = x0 - k, t1 = t0 + h, g0 = std::exp(-0.5 * t0 * t0), g1 = std::exp(-0.5 * t1 * t1);
      b[k] = (float)g0;
      db[k] = (float)(std::fabs(t0) * g0);
      bm[k] = (float)std::min(g0, g1);
      dbm[k] = t0 * t1 <= 0.0 ? 0.0f : (float)std::min(std::fabs(t0) * g0, std::fabs(t1) * g1);
    }
  }
};

constexpr int kReachRows = 32;   // rows checked at a time (compilers vectorise the fixed count)

// May the first f centres be left out of these rows?  v: |w| as [k][kReachRows].
inline bool may_leave_out(const float* v, int f, int K, const ReachBounds& q) {
  constexpr int B = kReachRows;
  const float most = 1.0f / 67108864.0f;   // 2^-26
  float lost[B] = {}, dlost[B] = {}, kept[B] = {}, dkept[B] = {};
  for (int k = 0; k < f; ++k)
    for (int r = 0; r < B; ++r) {
      lost[r] += v[k * B + r] * q.b[k];
      dlost[r] += v[k * B + r] * q.db[k];
    }
  for (int k = f; k < K; ++k)
    for (int r = 0; r < B; ++r) {
      const float x = v[k * B + r] * q.bm[k], y = v[k * B + r] * q.dbm[k];
      kept[r] = kept[r] > x ? kept[r] : x;
      dkept[r] = dkept[r] > y ? dkept[r] : y;
    }
  bool ok = true;
  for (int r = 0; r < B; ++r) ok = ok && lost[r] <= most * kept[r] && dlost[r] <= most * dkept[r];
  return ok;
}

// w: [rows][stride], K <= 64 weights in each row.  Distances are taken half a width at a time; rows that
// fail over such a piece are looked at again in quarters of it.
inline float gauss_reach(const float* w, int rows, int stride, int K) {
  constexpr int B = kReachRows;
  const double coarse = 0.5, fine = 0.125;
  const int blocks = (rows + B - 1) / B;
  std::vector<float> t((size_t)blocks * K * B, 0.0f);   // rows of zeros lose nothing
  for (int r = 0; r < rows; ++r)
    for (int k = 0; k < K; ++k) t[((size_t)(r / B) * K + k) * B + r % B] = std::fabs(w[(size_t)r * stride + k]);
  std::vector<const float*> failed;
  float reach = kLeastReach;
  for (double x0 = std::floor((kLeastReach + 1.0 - coarse) / coarse) * coarse; x0 < K - 1; x0 += coarse) {
    if (first_centre(x0 + coarse, reach) == 0) continue;
    const ReachBounds whole(x0, coarse, K);
    failed.clear();
    for (int q = 0; q < blocks; ++q) {
      const float* v = &t[(size_t)q * K * B];
      if (!may_leave_out(v, first_centre(x0 + coarse, reach), K, whole)) failed.push_back(v);
    }
    if (failed.empty()) continue;
    for (double x = x0; x < x0 + coarse && x < K - 1; x += fine) {
      const ReachBounds part(x, fine, K);
      for (const float* v : failed)
        for (int f = first_centre(x + fine, reach); f > 0; f -= kReachGroup) {
          if (may_leave_out(v, f, K, part)) break;
          // the last of these centres has to be within the reach up to x + fine
          reach = std::min(kWholeReach, std::max(reach, (float)(x + fine - f + 1.0) + 1e-3f));
          if (reach == kWholeReach) return reach;
        }
    }
  }
  return reach;
}

}  // namespace ctd
