// k_fused_sc.cu -- instantiations of the screened FP32 tile kernel (tile code kScWC, ranges of at
// most 32 disparities).
#include "k_fused_sc.cuh"

namespace sgb {

FusedKernel pick_fused_sc(int rb) { return pick_sc_rb(rb); }
size_t sc_smem_bytes(const Geometry &g) { return sc_layout(g.rb, g.m, g.ref_box_w, g.tgt_box_w, g.box_h).total; }

}  // namespace sgb
