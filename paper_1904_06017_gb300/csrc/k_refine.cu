// k_refine.cu -- instantiations of the FP32 refinement (tile code kScWC), without and with the
// best2 output (every pixel refines all D disparities, so the smallest E over d != d* is
// k_fused's value too).
#include "k_refine.cuh"

namespace sgb {

FusedKernel pick_refine(int rb, bool b2, int rows, int ctas)
{
    if (rows == kRefineRows)
        return ctas == 2 ? pick_refine_rb<false, kRefineRows, 2>(rb) : pick_refine_rb<false, kRefineRows, 1>(rb);
    return b2 ? pick_refine_rb<true, tile_y(kScWC), 1>(rb) : pick_refine_rb<false, tile_y(kScWC), 1>(rb);
}

}  // namespace sgb
