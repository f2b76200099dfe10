// Device functions of the FP64 kernels compiled for the host (_host_cuda.h),
// for tests that need no GPU.
#include "_host_cuda.h"

#include "hweno.h"
#include "hweno_adjoint.cuh"
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

// side_vjp (limiter = 0) or limiter_vjp of n stencils x[i][6] (5 used by the
// limiter) with cotangent 1: values v[i] and gradients g[i][6]
void host_vjp(int limiter, int n, const double* x, const double* w3, double eps, double* v,
              double* g) {
  Weights<double> w{};
  w.g0 = w.d0 = w3[0];
  w.g1 = w.d1 = w3[1];
  w.g2 = w.d2 = w3[2];
  w.eps = eps;
  for (int i = 0; i < n; ++i, x += 6, g += 6) {
    for (int k = 0; k < 6; ++k) g[k] = 0.0;
    v[i] = limiter ? limiter_vjp(x[0], x[1], x[2], x[3], x[4], 1.0, w, g)
                   : side_vjp(x[0], x[1], x[2], x[3], x[4], x[5], 1.0, w, g);
  }
}
}
