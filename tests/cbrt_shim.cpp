// Host build of the FP64 cube root and the truncation to FP32 (gf_fp64.cuh):
// the device's FP32 estimates are replaced by exact ones with a relative error
// of err and -err in turn.
#include <cmath>
#include <cstdint>

#include "gf_fp64.cuh"

namespace {
double g_err = 0.0;
int g_native = 0;
}

namespace gfk {
float seed_rcp(float x) { return 1.0f / x; }
float seed_rsqrt(float x) { return 1.0f / std::sqrt(x); }
float seed_cbrt(float x) {
  g_err = -g_err;
  return (float)(std::cbrt((double)x) * (1.0 + g_err));
}
double native_sqrt(double x) { return std::sqrt(x); }
double native_cbrt(double x) {
  ++g_native;
  return std::cbrt(x);
}
}  // namespace gfk

extern "C" int cbrt_ops(int n, const double* x, double err, double* root) {
  g_err = err;
  g_native = 0;
  for (int k = 0; k < n; ++k) root[k] = gfk::cbrt_pos(x[k]);
  return g_native;
}

extern "C" void trunc_ops(int n, const double* x, uint32_t* bits) {
  for (int k = 0; k < n; ++k) bits[k] = gfk::fbits(gfk::trunc_f32(x[k]));
}
