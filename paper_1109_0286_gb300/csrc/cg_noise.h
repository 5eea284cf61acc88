// Host side of the white-noise source (normal_pair in cg_common.cuh).
#pragma once
#include <cmath>
#include <vector>

#include "cg_types.h"

namespace cgf {

// The white-noise source's tables (kNoise*), each entry rounded once from
// extended precision.
inline std::vector<double> noise_tables() {
  std::vector<double> t(kNoiseEntries);
  for (int i = 0; i < 256; ++i) {
    long double c = 1.0L + (i + 0.5L) / 256.0L;
    if (i >= 128) c /= 2.0L;
    const double inv = i == 0 || i == 255 ? 1.0 : (double)(1.0L / c);
    t[kNoiseLog + 2 * i] = -2.0 * inv;
    t[kNoiseLog + 2 * i + 1] = (double)(2.0L * std::log((long double)inv));
    // cos, sin by octants (exact 0, 1 and equal magnitudes on the symmetries)
    const int o = i / 32, f = i % 32;
    const long double th = 3.14159265358979323846264338327950288L / 128.0L * (o & 1 ? 32 - f : f);
    const long double u = std::cos(th), v = std::sin(th);
    const bool swap = ((o + 1) / 2) % 2;   // octants 1, 2, 5, 6
    const long double c8 = (o >= 2 && o < 6 ? -1.0L : 1.0L) * (swap ? v : u);
    const long double s8 = (o >= 4 ? -1.0L : 1.0L) * (swap ? u : v);
    double* arc = &t[kNoiseArc + 4 * i];
    arc[0] = (double)c8;
    arc[1] = (double)s8;
    arc[2] = (double)(c8 - (long double)arc[0]);
    arc[3] = (double)(s8 - (long double)arc[1]);
  }
  for (int k = 0; k < 54; ++k) t[kNoiseExp + k] = (double)(2.0L * k * std::log(2.0L));
  return t;
}

}  // namespace cgf
