// k_refine.cuh -- the second half of the FP32 fused step: k_fused's FP32 arithmetic over the
// candidate ranges that k_march certified (k_march.cuh states the bound), so that the step's
// outputs are bit for bit those of k_fused, the plain FP32 kernel.
//
// A persistent CTA takes tiles of 32 columns and TY rows in turn (36, or kRefineRows with one or two CTAs
// per SM: refine_rows states where the line lies and what both sides measured).  Per tile it refines [dlo - 1, dhi + 1] of every
// pixel (sc_refine): FP32 costs of the tile's candidate disparities from the two-pass cost phase
// (the same integers and roundings as k_fused's), the weight ex2(fma(-t, t, K)), and the FMA
// chain in k_fused's order (window column outer, row inner), then k_fused's running WTA in
// increasing d.  The winner and its two neighbours (the parabola of eq. subpixel) are therefore
// k_fused's values exactly.  With the best2 output (B2) every pixel refines all D disparities (a
// diagnostic path, which needs no screening).
#pragma once
#include "k_sc_refine.cuh"

namespace sgb {

// Shared memory (offsets from the 128-byte aligned dynamic base):
//   sref, stgt  image tiles (TMA), as in k_fused
//   cbuf   planes of FP32 disparity pairs (float2 [QH][kScRPW], sc_psz(QH) entries apart)
//   vband  the cost phase's vertical window sums
//   sstr, sstt  window statistics of one band
//   sI     [QH][kScRPW] f32  the reference intensities times sqrt(log2 e) / sigma1 of the cost
//          positions (1e18 outside the image, as in k_fused)
//   sK     the spatial exponents as [2 RB + 1][sc_krw(RB)] f32
struct RefineLayout {
    size_t sref, stgt, cbuf, vband, sstr, sstt, sI, sK, total;
};

__host__ __device__ inline RefineLayout refine_layout(int rb, int m, int ref_box_w, int tgt_box_w, int box_h, int TY)
{
    RefineLayout L;
    const int TX = tile_x(kScWC);
    const int QH = TY + 2 * rb, QW = TX + 2 * rb, CW = TX + 2 * m;
    const size_t v8 = (size_t)kScRBand8 * CW * 8 * 4, v4 = (size_t)kScRBand4 * CW * 4 * 4;
    L.sref = 0;
    L.stgt = align_up((size_t)box_h * ref_box_w, 128);
    L.cbuf = align_up(L.stgt + (size_t)box_h * tgt_box_w, 128);
    L.vband = align_up(L.cbuf + (size_t)kScDCR * sc_psz(QH) * 4, 128);
    L.sstr = align_up(L.vband + (v8 > v4 ? v8 : v4), 16);
    L.sstt = align_up(L.sstr + (size_t)kScRBand4 * QW * 8, 16);
    L.sI = align_up(L.sstt + (size_t)kScRBand4 * (QW + kScDCR - 1) * 8, 16);
    L.sK = align_up(L.sI + (size_t)QH * kScRPW * 4, 16);
    L.total = align_up(L.sK + (size_t)(2 * rb + 1) * sc_krw(rb) * 4, 128);
    return L;
}

template <int RB, bool B2, int TY, int CTAS>
__global__ void __launch_bounds__(kThreads, CTAS)
k_refine(const __grid_constant__ PairDesc single, const PairDesc *__restrict__ pairs, const int2 *__restrict__ items,
         int nitems, int *__restrict__ counter)
{
    constexpr int TX = tile_x(kScWC);
    constexpr int KB = 2 * RB + 1;
    constexpr int QH = TY + 2 * RB, QW = TX + 2 * RB;
    static_assert(RB <= kScMaxRB && QW <= kScRPW, "a row of cost positions fits the planes' pitch");
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(16) FusedArgs s_args;
    __shared__ int s_item;
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ int s_flag;
    __shared__ int s_rlo, s_rhi;
    __shared__ int s_next, s_claimed, s_staged;   // the work item claimed ahead, its copies issued

    const int tid = threadIdx.x;
    const FusedArgs &a = s_args;
    if (tid == 0) {
        mbar_init(&s_bar, 1);
        s_staged = 0;
    }
    for (int iter = 0;; ++iter) {
        // the work item: the first one claimed here, every later one claimed ahead (the barrier
        // also orders the previous tile's last reads of s_args before it is overwritten)
        if (tid == 0) {
            s_item = iter == 0 ? (pairs ? atomicAdd(counter, 1) : (int)blockIdx.x) : s_next;
            s_claimed = 0;
        }
        __syncthreads();
        const int item = s_item;
        if (item >= nitems) return;
        const bool issued = iter > 0 && s_staged;
        int tx = 0, ty = 0;
        const PairDesc *pd = sc_decode(single, pairs, items, item, tx, ty);
        {
            const int *src = reinterpret_cast<const int *>(&pd->a);
            int *dst = reinterpret_cast<int *>(&s_args);
            for (int i = tid; i < (int)(sizeof(FusedArgs) / 4); i += kThreads) dst[i] = src[i];
        }
        __syncthreads();
        const int RP = a.ref_box_w;
        const RefineLayout L = refine_layout(RB, a.m, RP, a.tgt_box_w, a.box_h, TY);
        uint8_t *sref = smem + L.sref;
        uint8_t *stgt = smem + L.stgt;
        float *sIr = reinterpret_cast<float *>(smem + L.sI), *sKr = reinterpret_cast<float *>(smem + L.sK);
        const int x0 = tx * TX, y0 = ty * TY;
        if (tid == 0) {
            s_rlo = 0x7fffffff;
            s_rhi = -1;
        }
        if (!sc_stage(pd, a, sref, stgt, &s_bar, &s_flag, x0, y0, iter, tid, issued)) return;
        // called after a barrier that follows the tile's last read of sref / stgt
        auto images_free = [&]() {
            if (tid == 0)
                sc_claim_ahead(single, pairs, items, nitems, counter, item, a, sref, stgt, &s_bar, &s_next,
                               &s_claimed, &s_staged, TX, TY);
        };
        // scaled reference intensities of the cost positions, exactly as k_fused stages them;
        // positions outside the image and the row padding get 1e18 (weight 0)
        for (int i = tid; i < QH * kScRPW; i += kThreads) {
            const int yq = i / kScRPW, xq = i - yq * kScRPW;
            const int ix = x0 - RB + xq, iy = y0 - RB + yq;
            float v = 1e18f;
            if (xq < QW && ix >= 0 && ix < a.W && iy >= 0 && iy < a.H)
                v = (float)sref[(yq + a.rw) * RP + a.ref_e + xq + a.rw] * a.iscale;
            sIr[i] = v;
        }
        for (int i = tid; i < KB * sc_krw(RB); i += kThreads) {
            const int dx = i / sc_krw(RB), dy = i - dx * sc_krw(RB);
            sKr[i] = dy < KB ? a.K[dx * KB + dy] : 0.f;
        }
        sc_refine<RB, B2, kThreads, kScDCR, kScRSeg, TY>(
            a, sref, stgt, reinterpret_cast<float *>(smem + L.cbuf), reinterpret_cast<int *>(smem + L.vband),
            reinterpret_cast<int2 *>(smem + L.sstr), reinterpret_cast<int2 *>(smem + L.sstt), sIr, sKr, x0, y0, tid, &s_rlo,
            &s_rhi,
            [&](int py, int px) {
                const int r = a.cand[(size_t)(y0 + py) * a.W + x0 + px];
                return make_int2(r & 0xffff, r >> 16);
            },
            images_free);
        __syncthreads();
        images_free();   // (claimed already, unless the tile had no candidates to refine)
    }
}

template <bool B2, int TY, int CTAS>
FusedKernel pick_refine_rb(int rb)
{
    switch (rb) {
    case 0: return k_refine<0, B2, TY, CTAS>;
    case 1: return k_refine<1, B2, TY, CTAS>;
    case 2: return k_refine<2, B2, TY, CTAS>;
    case 3: return k_refine<3, B2, TY, CTAS>;
    case 4: return k_refine<4, B2, TY, CTAS>;
    case 5: return k_refine<5, B2, TY, CTAS>;
    case 6: return k_refine<6, B2, TY, CTAS>;
    }
    return nullptr;
}

}  // namespace sgb
