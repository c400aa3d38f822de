// cfl_screen.cuh -- the flux pass's screen of the CFL maximum.  The maximum that blocks of a pass have
// already published is a lower bound of the pass's maximum; a grid point whose FP32 estimate of
// |u| + c_f lies below `screen` (that bound less 3e-6 relative and 1e-18 absolute, above the estimate's
// worst error: 3e-7 relative from FP32 sums and roots, and in FP64 1e-6 from the truncated operands)
// cannot raise it, so its exact speed (two FP64 square roots) is not formed.  The pass still yields the
// exact maximum, whichever blocks ran first; a NaN, an infinite estimate or a negative density always
// takes the exact path.
#pragma once

#include <math.h>

#include "fixed64.cuh"

namespace mhd {

FX_FN float cfl_screen(double published) { return (float)(published * (1.0 - 3e-6) - 1e-18); }

// |x| as an FP32 number from the high word alone, truncated (at most 2^-20 relative below |x|);
// infinite from 2^128 on and for a NaN.  Below 2^-126 it is 2^-126, not 0: a product of such a value
// with one as far from 1 the other way (|B|^2 / rho at a density of 1e-38 or 1e38) is then too large,
// never too small.  Integer instructions: a conversion costs as much as an FP64 multiplication.
FX_FN float float_near(double x) {
  int h = (int)(fx_hi(x) & 0x7fffffffu) - 0x38000000;
  h = h < 0x00100000 ? 0x00100000 : h > 0x0ff00000 ? 0x0ff00000 : h;
  const uint32_t bits = (uint32_t)h << 3;
  float f;
  memcpy(&f, &bits, 4);
  return f;
}

// Whether the point's speed |u| + sqrt(cs^2 + b2 ir), ir = 1 / rho, has to be formed.  FP64:
FX_FN bool cfl_may_raise(double ux, double uy, double uz, float cs2, double b2, double ir, float screen) {
  const float fx = float_near(ux), fy = float_near(uy), fz = float_near(uz);
  const float u2 = fx * fx + fy * fy + fz * fz, c2 = cs2 + float_near(b2) * float_near(ir);
  return !(sqrtf(u2) + sqrtf(c2) < screen) || (fx_hi(ir) >> 31) != 0u;
}
// Double-float, from the high parts (with a negative density the sum cs2 + b2 ir cancels):
FX_FN bool cfl_may_raise(float ux, float uy, float uz, float cs2, float b2, float ir, float screen) {
  const float u2 = ux * ux + uy * uy + uz * uz, c2 = cs2 + b2 * ir;
  return !(sqrtf(u2) + sqrtf(c2) < screen) || ir < 0.f;
}

}  // namespace mhd
