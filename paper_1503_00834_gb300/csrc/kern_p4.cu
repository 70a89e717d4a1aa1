// Residual kernels of order p = 4 (N = 5 solution points per direction).
// Elements per CTA: 2 (FP64 form); FP32 perturbation form: 5 (125 threads, four warps nearly full, three
// CTAs per SM; ten elements at two four-warp CTAs' registers ran 29 % slower).
// Tile 1 (two elements per CTA) is the other candidate of the batched-shell autotuner.
#include "kern_inst.cuh"

namespace chorus {
LaunchSet launchers_p4(int tile) {
  return tile == 1 ? Inst<5, 2, 2, 5>::set() : Inst<5, 2, 5, 5>::set();
}
}  // namespace chorus
