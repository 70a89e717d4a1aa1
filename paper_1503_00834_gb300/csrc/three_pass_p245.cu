// Three-pass kernels of the orders p = 2 (14 and 7 elements per CTA in FP32, 6 in FP64), 4 (5; 2) and 5
// (2; 2).
#include "three_pass_inst.cuh"

namespace chorus {
ThreePassSet three_pass_p2() { return ThreePassInst<3, 14, 7, 6>::set(); }
ThreePassSet three_pass_p4() { return ThreePassInst<5, 5, 5, 2>::set(); }
ThreePassSet three_pass_p5() { return ThreePassInst<6, 2, 2, 2>::set(); }
}  // namespace chorus
