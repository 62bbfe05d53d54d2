// k_march_64.cu -- instantiations of the tensor-core pass with 64 disparities per chunk.
#include "k_march.cuh"

namespace sgb {

MarchChoice pick_march_64(int cost_dtype, int rb, int rw)
{
    if (cost_dtype == STEREO_F32) return pick_march_rb<64, kMarchScreen, __half>(rb, rw);
    if (cost_dtype == STEREO_F16) return pick_march_rb<64, kMarchPlain, __half>(rb, rw);
    return pick_march_rb<64, kMarchPlain, __nv_bfloat16>(rb, rw);
}

}  // namespace sgb
