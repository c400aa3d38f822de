// The flux pass's CFL screen (csrc/cfl_screen.cuh) on the host.
#include "cfl_screen.cuh"

// need[i]: whether point i's speed has to be formed when `published[i]` is the maximum known so far;
// p[i] = (ux, uy, uz, cs^2, |B|^2, 1 / rho).
extern "C" void cfl_screen_points(int df, int count, const double *p, const double *published, int *need) {
  for (int i = 0; i < count; ++i, p += 6) {
    const float s = mhd::cfl_screen(published[i]);
    need[i] = df ? mhd::cfl_may_raise((float)p[0], (float)p[1], (float)p[2], (float)p[3], (float)p[4], (float)p[5], s)
                 : mhd::cfl_may_raise(p[0], p[1], p[2], (float)p[3], p[4], p[5], s);
  }
}
