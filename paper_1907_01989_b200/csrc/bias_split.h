// An expansion's bias as four products in the K steps of a matrix instruction (block_ws_kernel): the A operand holds 1, 2^-11, 2^-22
// and 2^15 (frag::ones_word) in each of its rows, the B operand the bias in four fp16 parts of 11 bits each, the last one for biases
// beyond fp16's range.  A product of two fp16 values is exact in fp32, and the four add up to the bias itself from 2^-22 on;
// below, to within 2^-47, the resolution of the third part (a hidden value is stored in steps of 2^-24 and more).
#pragma once

#include <cmath>
#include <cstdint>

#include "gi_internal.h"

namespace gi {

// Biases for which every part and every rest is finite in fp16: up to 2^27 the rest behind the last part is at most 2^15 (half a
// step of fp16 below 2^12, times 2^15); from about 1.5e8 on it can pass 65504, and infinity times the zeros beside it would be NaN.
// Blocks with a larger bias, an infinite one (a masked channel) or NaN run on the kernel that starts its sums at the bias.
inline bool bias_splits(float b) { return std::fabs(b) <= 134217728.0f; }

inline double f16_value(uint16_t h) {
  const int e = (h >> 10) & 31, m = h & 1023;
  const double v = e == 0 ? std::ldexp(m, -24) : e == 31 ? (m ? NAN : INFINITY) : std::ldexp(1024 + m, e - 25);
  return h & 0x8000 ? -v : v;
}

inline void bias_parts(float b, uint16_t (&part)[4]) {
  static const double kScale[4] = {1.0, 2048.0, 4194304.0, 1.0 / 32768.0};  // reciprocals of what A holds
  double rest = b;
  auto take = [&](int i) {
    part[i] = f32_to_f16_rne(static_cast<float>(rest * kScale[i]));
    rest -= f16_value(part[i]) / kScale[i];
  };
  part[3] = 0;
  if (std::fabs(b) > 65504.0f) take(3);
  take(0);
  take(1);
  take(2);
}

}  // namespace gi
