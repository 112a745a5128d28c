// Host build of the FP64 building blocks (gf_fp64.cuh): the device's FP32
// reciprocal and reciprocal-square-root seeds are replaced by exact ones with
// a relative error drawn from [-err, err].
#include <cmath>
#include <cstdint>

#include "gf_fp64.cuh"

namespace {
double g_err = 0.0;
uint64_t g_state = 1;
double draw() {
  g_state = g_state * 6364136223846793005ull + 1442695040888963407ull;
  return (double)(int64_t)g_state * 0x1p-63;
}
}  // namespace

namespace gfk {
float seed_rcp(float x) { return (float)((1.0 / (double)x) * (1.0 + g_err * draw())); }
float seed_rsqrt(float x) { return (float)((1.0 / std::sqrt((double)x)) * (1.0 + g_err * draw())); }
double native_sqrt(double x) { return std::sqrt(x); }
}  // namespace gfk

extern "C" void fp64_ops(int n, const double* a, const double* b, double err, double* quot,
                         double* root, double* halved, double* doubled, uint8_t* flags) {
  g_err = err;
  for (int k = 0; k < n; ++k) {
    quot[k] = gfk::div_rn(a[k], b[k]);
    root[k] = gfk::sqrt_rn(a[k]);
    halved[k] = gfk::half(a[k]);
    doubled[k] = gfk::twice(a[k]);
    flags[k] = (uint8_t)((gfk::dlt(a[k], b[k]) ? 1 : 0) | (gfk::neg(a[k]) ? 2 : 0) |
                         (gfk::pos(a[k]) ? 4 : 0) | (gfk::iszero(a[k]) ? 8 : 0) |
                         (gfk::above(a[k], 1e-3) ? 16 : 0));
  }
}
