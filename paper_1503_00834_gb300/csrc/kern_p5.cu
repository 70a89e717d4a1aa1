// Residual kernels of order p = 5 (N = 6 solution points per direction).
// Elements per CTA: 2 (FP64 form), 4 (FP32 perturbation form: 144 threads, 4.5 of five warps full, two CTAs
// per SM; two-element CTAs leave a quarter of their three warps' lanes idle and ran 24 % slower).
// Tile 1 (two elements per CTA) is the other candidate of the batched-shell autotuner.
#include "kern_inst.cuh"

namespace chorus {
LaunchSet launchers_p5(int tile) {
  return tile == 1 ? Inst<6, 2, 2, 3>::set() : Inst<6, 2, 4, 3>::set();
}
}  // namespace chorus
