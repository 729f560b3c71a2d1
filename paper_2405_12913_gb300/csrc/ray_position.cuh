// Position of a line-of-sight node in mesh cells, shared by the ray step and its adjoint.
//
// The position r theta needs FP64 (1e-6 cells a thousand cells from the observer), but this part has only two FP64 lanes
// per SM and clock: the two FP64 divisions of the plain formulas, by the cell and by the mesh side, four times per ray,
// took most of a ray's FP64 time.  Both divisors are the step's own, so the quotient comes from the divisor's
// reciprocal with one residual correction (Markstein's method: the correctly rounded quotient), and the box index from the
// reciprocal alone, put right by a box where the product rounded across one.  Same bits as the divisions.
#pragma once

#include "mesh_kernels.h"

namespace hrt {

// (obs + r theta) / cell, unwrapped.
__device__ __forceinline__ double line_of_sight_cell(const RayStepParams& p, double obs, double r, double theta) {
  const double x = fma(r, theta, obs), q = x * p.inv_cell;
  return fma(fma(-q, p.cell, x), p.inv_cell, q);
}

// u wrapped into [0, n) as cell and fraction.
__device__ __forceinline__ void split_cell(const RayStepParams& p, double u, int& i0, float& f0) {
  const double n = p.n;
  u = fma(-n, floor(u * p.inv_n), u);
  if (u < 0.0) u += n;
  else if (u >= n) u -= n;
  const double fl = floor(u);
  i0 = static_cast<int>(fl);
  if (i0 >= p.n) i0 -= p.n;
  f0 = static_cast<float>(u - fl);
}

}  // namespace hrt
