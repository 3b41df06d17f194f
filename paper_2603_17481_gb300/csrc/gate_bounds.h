// gate_bounds.h -- integer bounds on the fixed-point phi outside which the interfacial gate cannot pass.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace lbm {

// phi (1 - phi) >= q_th holds between the two roots 1/2 (1 -+ sqrt(1 - 4 q_th)). The gate takes it in
// binary32: phi is rounded once to 24 bits (half a unit is 2^-25 at most, and less than that times phi),
// 1 - phi once (2^-25 at most) and the product once (2^-27 at most, being below 1/4). Both factors are at
// most 1, so the q it compares exceeds the exact one by less than 2^-25 + 2^-25 + 2^-27 = 6.8e-8, and the
// roots of q_th - 1e-7 enclose every value that it passes. (The margin has to be one of q: towards
// q_th = 1/4 the slope of q vanishes, and one rounding moves the edge in phi by 1.5e-4.) With a q_th that
// is zero in binary32, or none that compares, phi outside [0, 1] passes too: no bound.
inline void gate_bounds(float q_th, int32_t &lo, uint32_t &span) {
  lo = INT32_MIN;
  span = UINT32_MAX;
  if (!(q_th > 0.0f)) return;
  const double q = std::max(0.0, (double)q_th - 1e-7);
  const double edge = 0.5 * (1.0 - std::sqrt(std::max(0.0, 1.0 - 4.0 * q)));
  lo = (int32_t)std::floor(edge * 1073741824.0);
  span = (uint32_t)(std::ceil((1.0 - edge) * 1073741824.0) - (double)lo);
}

}  // namespace lbm
