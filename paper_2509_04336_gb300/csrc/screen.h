// screen.h -- the FP32 screen of a differential-evolution step: its scale s and the margin by which
// the screened point may leave the cube before the step is dropped.  Steps that pass are moved
// exactly, so the screen may keep too many but must never drop one that the exact test keeps.
//
// The error of the screened point x = u + s (u_a - u_b), 0 <= u, u_a, u_b <= 1, for
// s = c g, c = 2.38 / sqrt(2 D) <= 1.683, g = -(1/4) ln 2 sum_i log2 U_i:
//   U_i     two roundings to float, 2^-23 relative: 1.8e-7 in its logarithm;
//   log2    __log2f: 2^-22 for U_i in [1/2, 1), else 2 ulp, 2^-22 |log2 U_i|;
//   sum l2  three additions of values of one sign, 3 * 2^-24 |l2|
//           => |d l2| <= 4.2e-7 |l2| + 1.7e-6;
//   s       four more roundings => |ds| <= 6.6e-7 s + c (ln 2 / 4) 1.7e-6 <= 6.6e-7 s + 5.0e-7
//           (s = 1 exactly on a step without a scale draw);
//   x       the three coordinates and the difference rounded to float: 1.2e-7 s + 3e-8; product and
//           sum rounded: 6e-8 s + 6e-8
//           => |dx| <= 8.4e-7 s + 5.9e-7,
// a twelfth of the margin at most, in every dimension.  The logarithms are of U_i, not of the 52-bit
// integers 2^52 U_i: near 52 the 2 ulp of each and the roundings of the sum towards 208 left up to
// 5e-5 in l2 however small s, 1.5e-5 in s for one dimension, outside this margin for D <= 2.
#pragma once

#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define GWNS_HD __host__ __device__ __forceinline__
#else
#define GWNS_HD inline
#endif

namespace gwns {

// ((x >> 12) + 1/2) 2^-52, the uniform of a 64-bit draw, as a float in [2^-53, 1], from two 32-bit
// conversions: a 64-bit integer conversion runs on the FP64 pipe.
GWNS_HD float open_unit_f(uint64_t x) {
  const uint64_t v = x >> 12;
  return fmaf((float)(uint32_t)(v >> 20), 0x1p-32f, fmaf((float)(uint32_t)(v & 0xFFFFFull), 0x1p-52f, 0x1p-53f));
}

// s = de_scale * (-1/4 ln(U_0 U_1 U_2 U_3)); log2_: a base-2 logarithm of the accuracy above.
template <class Log2>
GWNS_HD float screen_scale(const uint64_t* v, float de_scale, Log2 log2_) {
  const float l2 = log2_(open_unit_f(v[0])) + log2_(open_unit_f(v[1])) + log2_(open_unit_f(v[2])) + log2_(open_unit_f(v[3]));
  return de_scale * (-0.25f * 0.6931471805599453f * l2);
}

GWNS_HD float screen_margin(float s) { return 1e-5f * (1.0f + fabsf(s)); }

}  // namespace gwns
