// k_march_32.cu -- instantiations of the tensor-core pass with 32 disparities per chunk.
#include "k_march.cuh"

namespace sgb {

MarchChoice pick_march_32(int cost_dtype, int rb, int rw)
{
    if (cost_dtype == STEREO_F32) return pick_march_rb<32, kMarchRefine, __half>(rb, rw);
    if (cost_dtype == STEREO_F16) return pick_march_rb<32, kMarchPlain, __half>(rb, rw);
    return pick_march_rb<32, kMarchPlain, __nv_bfloat16>(rb, rw);
}

// Screening alone: the second pass of a longer range (march_split).
MarchChoice pick_march_32_screen(int rb, int rw) { return pick_march_rb<32, kMarchScreen, __half>(rb, rw); }

}  // namespace sgb
