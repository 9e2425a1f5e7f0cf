// FP64 sin/cos from a 4096-entry table (method and error in rad_fp64.cu), shared by the FP64 kernels.
#pragma once
#include "rad_internal.cuh"

namespace rad {
namespace {

// 2 pi / kTabN = pi * 2^-11 split into the double nearest pi and its remainder, both
// scaled by 2^-11 (exact): C1 + C2 = 2 pi / 4096 to about 106 bits.
constexpr double kPiHi = 3.141592653589793116;        // nearest double to pi
constexpr double kPiLo = 1.2246467991473531772e-16;   // pi - kPiHi (rounded)
constexpr double kC1 = kPiHi / 2048.0;
constexpr double kC2 = kPiLo / 2048.0;
constexpr double kInvStep = 2048.0 / 3.141592653589793238462643383279502884;  // 4096/(2 pi)
constexpr double kMagic = 6755399441055744.0;  // 1.5 * 2^52: adding it rounds to an integer

// phi = j 2 pi / 4096 + r
__device__ __forceinline__ int reduce_table(double phi, double &r) {
  const double y = fma(phi, kInvStep, kMagic);  // round(phi * 4096/(2 pi)) + magic
  const double jd = y - kMagic;                 // exact
  r = fma(-jd, kC1, phi);
  r = fma(-jd, kC2, r);
  return __double2loint(y);                     // low word holds the integer (two's complement)
}

__device__ __forceinline__ void sincos_reduced(int j, double r, const double2 *__restrict__ tab, double &s, double &c) {
  const double2 t = tab[j & (kTabN - 1)];       // (cos, sin)(2 pi j / 4096)
  const double r2 = r * r;
  const double sr = fma(r2 * r, -1.0 / 6.0, r);           // sin r
  const double cm = r2 * fma(r2, 1.0 / 24.0, -0.5);       // cos r - 1
  s = fma(t.x, sr, fma(t.y, cm, t.y));                    // sin(a + r)
  c = fma(-t.y, sr, fma(t.x, cm, t.x));                   // cos(a + r)
}

__device__ __forceinline__ void sincos_table(double phi, const double2 *__restrict__ tab, double &s,
                                             double &c) {
  double r;
  const int j = reduce_table(phi, r);
  sincos_reduced(j, r, tab, s, c);
}

}  // namespace
}  // namespace rad
