// k_diff.cuh -- what the translation units of the differentiable path share.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace sgb {

enum { AGG_FWD = 0, AGG_H = 1, AGG_GC = 2 };

// A value v of h as FP16 halves: hi = RN16(2^k v), lo = RN16(2^k v - hi), 22 bits and 32 bits of memory.
// Laid out as [B][ceil(D / 4)][H][W][8]: 4 hi, then 4 lo of the group's disparities (zero beyond D), so
// that a row of a group is one run of 16 bytes per pixel.
constexpr int kAggRange = 64;    // partial maxima of |dS/dl| per image

__device__ __forceinline__ uint32_t h2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// (x, y) as packed halves and what they leave.
__device__ __forceinline__ void split2(float x, float y, uint32_t &hi, uint32_t &lo)
{
    hi = h2(x, y);
    const float2 f = __ffma2_rn(__half22float2(*reinterpret_cast<const __half2 *>(&hi)), make_float2(-1.f, -1.f),
                                make_float2(x, y));
    lo = h2(f.x, f.y);
}
// hi + lo of two disparities; hi alone where it is not finite.
__device__ __forceinline__ float2 unsplit2(uint32_t hi, uint32_t lo)
{
    const float2 h = __half22float2(*reinterpret_cast<const __half2 *>(&hi));
    const float2 l = __half22float2(*reinterpret_cast<const __half2 *>(&lo));
    return make_float2(fabsf(h.x) < INFINITY ? h.x + l.x : h.x, fabsf(h.y) < INFINITY ? h.y + l.y : h.y);
}
// A scaled value that an FP16 pair cannot carry (infinite, NaN, or out of range).
__device__ __forceinline__ bool off_range(float x) { return !(fabsf(x) < 65504.f); }

__device__ __forceinline__ float pow2i(int k) { return __int_as_float((k + 127) << 23); }   // -126 <= k <= 127

struct AggArgs {
    const float *img;      // reference image [B][H][W]
    const float *vol;      // neighbour values: the cost (FWD, H) or h (GC; split up to kAggTcMaxRB) [B][D][H][W]
    const float *shift;    // FWD: row shifts
    float *disp;           // FWD: l
    float *lse, *lbar;     // FWD out, H in
    const float *gdisp;    // H: dS/dl
    float *h;              // H out (split up to kAggTcMaxRB)
    float *beta, *t1;      // H out, GC in
    float *gc;             // GC out
    const float *cost;     // GC: c(x, d) of the centre pixel
    float *gw;             // GC out: image gradient through the weights
    unsigned *range;       // split h: [B][kAggRange] partial maxima of |dS/dl|, bits
    int *hbad;             // split h: [B][H] rows of h that hold a value the split cannot carry
    int W, H, D;
    int warp_mode;         // FWD: the add-back is s_i (rounded) or s(v) (linear warp)
    float kappa;           // sqrt(log2 e) / sigma1: scaled intensities
    float k0;              // -log2 e / sigma0^2
    float kT;              // log2 e / T
    float invT;            // 1 / T
    float gw_scale;        // 2 / (sigma1^2 kappa)
};

// The exponent of h's scale in image b, called by a whole warp: |h| <= max|dS/dl| D / T, brought below 2^15.
__device__ __forceinline__ int h_shift(const AggArgs &a, int b, int lane)
{
    static_assert(kAggRange == 64, "two per lane");
    const unsigned m = __reduce_max_sync(0xffffffffu, max(a.range[b * 64 + lane], a.range[b * 64 + 32 + lane]));
    const int e = max((int)(m >> 23) - 127, -126) + 1 + min(ilogbf(a.invT * (float)a.D), 200) + 1;
    return max(-126, min(126, 15 - e));
}

constexpr int kAggTcMaxRB = 6;   // bil <= 13: a patch's window row fits the 16 k-slots of an mma

// k_dagg_tc.cu: the partial maxima that scale h and its row flags cleared (before H); GC on the tensor
// cores (rb <= kAggTcMaxRB).
cudaError_t launch_dabsmax(const AggArgs &a, int B, cudaStream_t st);
cudaError_t launch_gc_tc(const AggArgs &a, int rb, int B, cudaStream_t st);

}  // namespace sgb
