// FP32 surface-deviation patch step with dimensional splitting (instantiation
// of gf_step_kernel.cuh).  Compiled with fused multiply-add allowed: checked
// against the FP64 oracle with absolute tolerances; one shape per patch size.
#include <cuda_runtime.h>

#include "gf_internal.h"
#include "gf_step_kernel.cuh"

namespace gf {

int launch_patch_step_f32_split(const GfGeom& g, const GfView& v, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (g.M == 32) return gfs::launch_step<gfs::PrecF32, 32, 32, 512, 2, true>(g, v, st);
  if (g.M == 16) return gfs::launch_step<gfs::PrecF32, 16, 16, 352, 2, true>(g, v, st);
  return -1;
}

}  // namespace gf
