// Pieces of the one-sided Jacobi kernels (setup.cu, arrowv.cu).  A float64 instruction of a warp holds
// its scheduler's pipe for 64 clocks on GB300 however few lanes need it, so the kernels count them.
#pragma once
#include <cstdint>

namespace esmp2 {

// Sums of three values over the warp, all lanes get them.  Lanes first trade values, so that each lane
// carries one sum through the remaining steps: 6 additions instead of 15.
__device__ __forceinline__ void warp_sum3(double &a, double &b, double &c) {
  const int lane = threadIdx.x & 31;
  const bool h = (lane & 16) != 0, q = (lane & 8) != 0;
  // lanes with bit 4: (c, -), without: (a, b)
  const double s0 = __shfl_xor_sync(0xffffffffu, h ? a : c, 16), s1 = __shfl_xor_sync(0xffffffffu, b, 16);
  double u = (h ? c : a) + s0, v = b + s1;   // v: the same sum in both halves
  // within the half: bit 3 keeps v, the others u
  const double t = __shfl_xor_sync(0xffffffffu, q ? u : v, 8);
  double w = (q ? v : u) + t;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
  a = __shfl_sync(0xffffffffu, w, 0);
  b = __shfl_sync(0xffffffffu, w, 8);
  c = __shfl_sync(0xffffffffu, w, 16);
}

// Rotation that makes two rows with squared norms al, be and product ga orthogonal: t = sign(d) g /
// (|d| + sqrt(d^2 + g^2)), d = be - al, g = 2 ga (the smaller root of t^2 + 2 zeta t - 1 = 0).  The angle
// in float32 (an error of 1e-7 of it is left to the next sweep); c = 1 / sqrt(1 + t^2) by Newton steps in
// float64 and s = c t, so that c^2 + s^2 = 1 to rounding whatever t is.
__device__ __forceinline__ void jacobi_rotation(double al, double be, double ga, double &c, double &s) {
  const double d0 = be - al, g0 = 2.0 * ga;
  // scaled by a power of two (exponent of the larger one) to the range of float32
  const int e = max(__double2hiint(d0) & 0x7FF00000, __double2hiint(g0) & 0x7FF00000);
  const double sc = __hiloint2double(0x7FE00000 - e, 0);   // e below the largest exponent field
  const float d = (float)(d0 * sc), g = (float)(g0 * sc);
  const float tf = (d >= 0.f ? g : -g) / (fabsf(d) + sqrtf(d * d + g * g));
  const double t = (double)tf, q = fma(t, t, 1.0);   // q in [1, 2]
  double y = (double)rsqrtf((float)q);
  const double hq = 0.5 * q;
  y = y * fma(-hq * y, y, 1.5);
  y = y * fma(-hq * y, y, 1.5);
  c = y;
  s = y * t;
}

}  // namespace esmp2
