// Operator entries as sums of two BF16 numbers, hi + lo, for the tensor-core products. Plain
// C++, shared by the library and a test program.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

namespace swe {

// bf16 round-to-nearest-even of a float, and its value
inline uint16_t bf16_bits(float f) {
  uint32_t u;
  std::memcpy(&u, &f, 4);
  return (uint16_t)((u + 0x7FFFu + ((u >> 16) & 1u)) >> 16);
}
inline float bf16_value(uint16_t b) {
  const uint32_t u = (uint32_t)b << 16;
  float f;
  std::memcpy(&f, &u, 4);
  return f;
}

// hi/lo bf16 split of a single-precision operator entry
inline void bf16_split(double v, uint16_t& hi, uint16_t& lo) {
  const float vf = (float)v;
  hi = bf16_bits(vf);
  lo = bf16_bits(vf - bf16_value(hi));
}

// The values hi + lo of a row of an operator, rounded for smooth data. A low part rounded to
// nearest leaves an error of up to 2^-17 of its entry, the same in every element and step: on
// a solution that is nearly linear in an element, the errors of a row add up to a fixed
// change of the operator, whose effect a run accumulates. So each low part is its nearest
// value or the one on the other side of the entry, whichever brings the row's sums over
// `modes` (functions at the points that the row multiplies) closest to the exact ones: one
// pass in order, then changes of one or two of them while that helps.
inline std::vector<double> smooth_row(const double* w, int n, const std::vector<std::vector<double>>& modes) {
  const size_t nm = modes.size();
  std::vector<double> val(n), step(n, 0.0), S(nm, 0.0);
  auto norm_with = [&](int j, double d) {   // |S + d modes_j|^2
    double c = 0.0;
    for (size_t q = 0; q < nm; ++q) {
      const double t = S[q] + d * modes[q][j];
      c += t * t;
    }
    return c;
  };
  auto add = [&](int j, double d) {
    for (size_t q = 0; q < nm; ++q) S[q] += d * modes[q][j];
  };
  auto change = [&](int j) {
    val[j] += step[j];
    step[j] = -step[j];
  };
  for (int j = 0; j < n; ++j) {
    uint16_t h, l;
    bf16_split(w[j], h, l);
    const float lo = bf16_value(l);
    val[j] = (double)bf16_value(h) + lo;
    if (lo != 0.f) {   // a step of the low part (or of the entry in single precision) past the entry
      int el = 0, ew = 0;
      std::frexp(lo, &el);
      std::frexp((float)w[j], &ew);
      step[j] = std::ldexp(val[j] < w[j] ? 1.0 : -1.0, el - 8 > ew - 24 ? el - 8 : ew - 24);
    }
    const double e = val[j] - w[j];
    if (norm_with(j, e + step[j]) < norm_with(j, e)) change(j);
    add(j, val[j] - w[j]);
  }
  for (int pass = 0; pass < 4 * n; ++pass) {   // the best single change or pair of changes
    double least = 0.0;
    for (double s : S) least += s * s;
    least *= 1.0 - 1e-12;
    int bj = -1, bk = -1;
    for (int j = 0; j < n; ++j) {
      if (step[j] == 0.0) continue;
      const std::vector<double> S0 = S;
      if (const double c = norm_with(j, step[j]); c < least) {
        least = c;
        bj = j;
        bk = -1;
      }
      add(j, step[j]);
      for (int k = j + 1; k < n; ++k) {
        if (step[k] == 0.0) continue;
        if (const double c = norm_with(k, step[k]); c < least) {
          least = c;
          bj = j;
          bk = k;
        }
      }
      S = S0;
    }
    if (bj < 0) break;
    for (int j : {bj, bk}) {
      if (j < 0) continue;
      add(j, step[j]);
      change(j);
    }
  }
  return val;
}

}  // namespace swe
