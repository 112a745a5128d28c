// FP32 surface-deviation patch step, unsplit (instantiation of
// gf_step_kernel.cuh).  Compiled without contraction: the fused operations of
// this path are written out, so that every kernel shape rounds alike.  It is
// checked against the FP64 oracle with absolute depth and momentum tolerances.
#include <cuda_runtime.h>

#include "gf_internal.h"
#include "gf_step_kernel.cuh"

namespace gf {

// Shapes (variants of 32 x 32 patches): 0 = by the rule below; whole tiles
// with 3 = 320 threads, one CTA per SM, 7 = 384 threads, two, 2 = 640
// threads, one; 16 x 16 sub-tiles with 1 = 192 threads, four CTAs per SM, 4 =
// three, 6 = 96 threads, six; 5 = 8 x 8 sub-tiles with 96 threads.
//
// The rule for variant 0: whole tiles with 320 threads, two CTAs per SM (115
// KB of shared memory each), except where the sub-tiles of all patches are
// resident at once (152 SMs x 4 CTAs): a tile's chain of barriers, not the
// arithmetic, is then the launch's time, and smaller tiles have shorter ones.
// Measured, us per step with a front (a third wet) and with every cell wet,
// whole tiles / 16 x 16 / 8 x 8 (whole tiles of up to 152 patches in shape 3,
// one CTA per SM): 16 patches 20.5 / 14.7 / 13.7 and 18.0 / 13.3 / 13.4; 36
// patches 19.6 / 14.9 / 14.2 and 18.0 / 14.1 / 14.2; 64 patches 19.7 / 15.0 /
// 14.9 and 17.4 / 14.2 / 15.1; 144 patches 20.0 / 17.2 / 19.0 and 17.9 / 18.0 /
// 28.4; 256 patches 21.1 / 20.9 / 28.7 and 22.7 / 29.5 / 45.7; 1024 patches
// 39.3 / 45.3 / 71.7 and 68.0 / 89.6 / 146.
int launch_patch_step_f32(const GfGeom& g, const GfView& v, int variant,
                          void* stream) {
  if (v.npatch <= 0) return 0;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (g.dim_split) return launch_patch_step_f32_split(g, v, stream);
  if (g.M == 32) {
    // sub-tiles for small forests: see the rule above
    const int shape = variant != 0 ? variant
                      : v.npatch * 16 <= 152 * 4 ? 5
                      : v.npatch * 4 <= 152 * 4 ? 1 : 0;
    switch (shape) {
      case 1: return gfs::launch_step<gfs::PrecF32, 32, 16, 192, 4>(g, v, st);
      case 2: return gfs::launch_step<gfs::PrecF32, 32, 32, 640, 1>(g, v, st);
      case 3: return gfs::launch_step<gfs::PrecF32, 32, 32, 320, 1>(g, v, st);
      case 4: return gfs::launch_step<gfs::PrecF32, 32, 16, 192, 3>(g, v, st);
      case 5: return gfs::launch_step<gfs::PrecF32, 32, 8, 96, 8>(g, v, st);
      case 6: return gfs::launch_step<gfs::PrecF32, 32, 16, 96, 6>(g, v, st);
      case 7: return gfs::launch_step<gfs::PrecF32, 32, 32, 384, 2>(g, v, st);
      default: return gfs::launch_step<gfs::PrecF32, 32, 32, 320, 2>(g, v, st);
    }
  }
  if (g.M == 16) return gfs::launch_step<gfs::PrecF32, 16, 16, 192, 4>(g, v, st);
  return -1;
}

}  // namespace gf
