// Residual kernels of order p = 3 (N = 4 solution points per direction).
// Elements per CTA: 4 (FP64 form), 4 (FP32 perturbation form: 64-thread CTAs of two independent warps,
// six per SM; one-warp CTAs ran 4 % slower, eight-element ones 1 %); the update kernel takes 8.
// Tile 1 (eight elements per CTA) is the other candidate of the batched-shell autotuner.
// This translation unit is compiled with the approximate FP32 square root (build.py).
#include "kern_inst.cuh"

namespace chorus {
LaunchSet launchers_p3(int tile) {
  return tile == 1 ? Inst<4, 4, 8, 8>::set() : Inst<4, 4, 4, 8>::set();
}
}  // namespace chorus
