// Device functions of the FP64 kernels compiled for the host (_host_cuda.h),
// for tests that need no GPU.
#include "_host_cuda.h"

#include "rough_speed.cuh"

using namespace hweno;

extern "C" {

// n states u[i][4] (M used): the FP32 speeds of direction x (and, 2D, y)
void host_rough_speeds(int eq, int dim, int n, const double* u, double gamma, float* sx,
                       float* sy) {
  for (int i = 0; i < n; ++i, u += 4) {
    const float g = (float)gamma;
    if (dim == 2) {
      if (eq == HWENO_EULER) rough_speeds2<HWENO_EULER>(u, g, sx[i], sy[i]);
      else rough_speeds2<HWENO_BURGERS>(u, g, sx[i], sy[i]);
    } else {
      sx[i] = eq == HWENO_EULER     ? rough_speed<HWENO_EULER>(u, g)
              : eq == HWENO_BUCKLEY ? rough_speed<HWENO_BUCKLEY>(u, g)
                                    : rough_speed<HWENO_BURGERS>(u, g);
    }
  }
}
}
