// k_refine.cu -- instantiations of the FP32 refinement (tile code kScWC), without and with the
// best2 output (every pixel refines all D disparities, so the smallest E over d != d* is
// k_fused's value too).
#include "k_refine.cuh"

namespace sgb {

FusedKernel pick_refine(int rb, bool b2) { return b2 ? pick_refine_rb<true>(rb) : pick_refine_rb<false>(rb); }

}  // namespace sgb
