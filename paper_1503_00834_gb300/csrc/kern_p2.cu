// Residual kernels of order p = 2 (N = 3 solution points per direction).
// Elements per CTA: 6 (FP64 form); FP32 perturbation form: 14 (126 threads, four warps nearly full; seven
// elements measured the same), four CTAs per SM at 128 registers (4 % faster than three at 168).
// Tile 1 (six elements per CTA) is the other candidate of the batched-shell autotuner.
#include "kern_inst.cuh"

namespace chorus {
LaunchSet launchers_p2(int tile) {
  return tile == 1 ? Inst<3, 6, 6, 14>::set() : Inst<3, 6, 14, 14>::set();
}
}  // namespace chorus
