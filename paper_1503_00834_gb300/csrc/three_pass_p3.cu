// Three-pass kernels of order p = 3, four elements per CTA.  Compiled with the approximate
// FP32 square root (build.py).
#include "three_pass_inst.cuh"

namespace chorus {
ThreePassSet three_pass_p3() { return ThreePassInst<4, 4, 4, 4>::set(); }
}  // namespace chorus
