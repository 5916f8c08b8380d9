// tables.h -- host-side tables that the solver plans and the DS plans share.
#pragma once

#include <algorithm>
#include <cmath>
#include <vector>

namespace dsnu {

// FFT stage twiddles of a length-2^log2n transform in the order the device
// FFT reads them: stage s >= 1 (radix RAD, NS = product of the earlier
// radices), r = 1..RAD-1, k = 0..NS-1: e^{-2 pi i r k / (NS RAD)}.
// (lr: log2 of the full stages' radix)
inline void fft_stage_twiddles(int log2n, std::vector<double>& out, int lr = 4) {
  out.clear();
  for (int s = 1; s * lr < log2n; ++s) {
    const int rad = 1 << std::min(lr, log2n - s * lr), ns = 1 << (s * lr);
    for (int r = 1; r < rad; ++r)
      for (int k = 0; k < ns; ++k) {
        const double a = -2.0 * M_PI * double(r) * double(k) / double(ns * rad);
        out.push_back(std::cos(a));
        out.push_back(std::sin(a));
      }
  }
  if (out.empty()) out.assign(2, 0.0);
}

// A constant |v| <= 1 as v 2^bits = h + l 2^-32, h and l signed 32-bit (|l| < 2^31).
inline void fx_put(std::vector<int>& out, double v, int bits) {
  const double s = std::ldexp(v, bits), h = std::nearbyint(s);
  const double l = std::nearbyint((s - h) * 4294967296.0);
  out.push_back(int(h));
  out.push_back(int(std::min(std::max(l, -2147483647.0), 2147483647.0)));
}
inline std::vector<int> fx_table(const std::vector<double>& v, int bits) {
  std::vector<int> out;
  out.reserve(2 * v.size());
  for (double x : v) fx_put(out, x, bits);
  return out;
}

}  // namespace dsnu
