// e^{i phi} in FP64 for the phase tables (Eq. ferm_op), by table lookup (Gal and
// Bachelis 1991; Tang 1991): phi = k 2 pi / K + rho with |rho| <= pi / K, the
// tabulated e^{i k 2 pi / K} as a sum of two doubles, and short series for
// sin rho and cos rho - 1. 16 FP64 instructions; the library function takes about
// 48, each of which holds the FP64 pipe for 16 cycles a warp.
//
// Error, K = 1024: rho^7/5040 and rho^6/720 are below 1.2e-18, the reduction's
// below 3e-20, and the table's low halves leave the last addition's rounding
// (half an ulp) plus that of the correction (|correction| <= 3.1e-3, 2^-53 of it).
#pragma once

#include "common.cuh"

namespace hmc {

constexpr int kPhaseTable = 1024;

// The table: kPhaseTable entries (cos, sin), then as many with what rounding them
// left over; filled by phase_table_host.
struct PhaseTable {
  const double2* e;
};
void phase_table_host(double2* out /* 2 kPhaseTable */);

// Out of line: fields beyond 1e5, infinities and NaN.
static __device__ __noinline__ double2 phase_rare(double x) {
  double s, c;
  sincos(x, &s, &c);
  return make_double2(c, s);
}
static __device__ __noinline__ float phi_to_f32_rare(double x) { return phi_to_f32(x); }

__device__ __forceinline__ double2 phase_of_field(const PhaseTable& t, double x) {
  // |x| < 1e5, by the high word (a comparison of doubles would take the pipe)
  if ((unsigned)(__double2hiint(x) & 0x7fffffff) >= 0x40f86a00u) return phase_rare(x);
  const double big = 6755399441055744.0;                   // 1.5 2^52: rounds to an integer in the low word
  const double kb = fma(x, 162.97466172610083, big);       // K / (2 pi)
  const int k = __double2loint(kb) & (kPhaseTable - 1);
  const double kd = kb - big;
  // 2 pi / K in two parts, the first of 27 bits: its product with kd (|kd| < 2^24) is exact
  double r = fma(-kd, 0x1.921fb54000000p-8, x);
  r = fma(-kd, 0x1.10b4611a62633p-38, r);
  const double r2 = r * r;
  const double sr = fma(r * r2, fma(r2, 1.0 / 120.0, -1.0 / 6.0), r);  // sin rho
  const double c1 = r2 * fma(r2, 1.0 / 24.0, -0.5);                     // cos rho - 1
  const double2 h = __ldg(t.e + k), l = __ldg(t.e + kPhaseTable + k);
  return make_double2(h.x + fma(h.x, c1, fma(-h.y, sr, l.x)), h.y + fma(h.y, c1, fma(h.x, sr, l.y)));
}

// phi reduced to [-pi, pi], as float (phi_to_f32): the reduction is needed
// beyond pi only, again by the high word.
__device__ __forceinline__ float field_to_f32(double x) {
  if ((unsigned)(__double2hiint(x) & 0x7fffffff) >= 0x400921fbu) return phi_to_f32_rare(x);
  return (float)x;
}

}  // namespace hmc
