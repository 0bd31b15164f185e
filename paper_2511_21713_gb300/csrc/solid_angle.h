// The solid angle of a triangle: one definition for the host's winding numbers (pbfb_check_charges) and the GPU's
// (pbfb_charges_set), so that both decide alike and in float64.  No CUDA types.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define PBFB_HD __host__ __device__ __forceinline__
#else
#define PBFB_HD inline
#endif

namespace pbfb {

// Half the signed solid angle that the triangle with corners a, b, c (relative to the point, of lengths la, lb, lc)
// takes up, Van Oosterom and Strackee (1983):
//   tan(Omega / 2) = a.(b x c) / (|a||b||c| + (a.b)|c| + (b.c)|a| + (c.a)|b|).
// *on: the point lies on the triangle (a corner, or coplanar to 1e-12 relative with the denominator not positive,
// i.e. within the triangle), where the sign of a rounded zero would make the angle +-2 pi.
PBFB_HD double half_solid_angle(double a0, double a1, double a2, double b0, double b1, double b2, double c0, double c1,
                                double c2, double la, double lb, double lc, bool* on) {
  const double s3 = la * lb * lc;
  const double det = a0 * (b1 * c2 - b2 * c1) - a1 * (b0 * c2 - b2 * c0) + a2 * (b0 * c1 - b1 * c0);
  const double den =
      s3 + (a0 * b0 + a1 * b1 + a2 * b2) * lc + (b0 * c0 + b1 * c1 + b2 * c2) * la + (c0 * a0 + c1 * a1 + c2 * a2) * lb;
  if (s3 == 0.0 || (std::fabs(det) <= 1e-12 * s3 && den <= 0.0)) *on = true;
  return std::atan2(det, den);
}

}  // namespace pbfb
