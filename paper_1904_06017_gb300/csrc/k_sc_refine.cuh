// k_sc_refine.cuh -- k_fused's FP32 arithmetic over the certified candidate ranges of one 32 x TY
// tile (sc_refine), and the persistent tiles' claiming and staging: shared by k_fused_sc (screening
// and refinement in one kernel) and k_refine (behind k_march).
#pragma once
#include <type_traits>

#include "k_cost.cuh"

namespace sgb {

constexpr int kScDCR = 8;       // disparities per FP32 refinement chunk
constexpr int kScRBand4 = 12;   // cost rows per band of a 4-disparity refinement chunk
constexpr int kScRBand8 = 8;    // cost rows per band of an 8-disparity refinement chunk
constexpr int kScRSeg = 3;      // cost columns per horizontal work item of the refinement chunks
// Refinement planes: rows of kScRPW entries and planes a multiple of 32 entries apart, so that
// a warp's 32 pixels of one row read 32 distinct banks whatever disparity each needs
constexpr int kScRPW = 44;
__host__ __device__ constexpr int sc_psz(int qh) { return (qh * kScRPW + 31) / 32 * 32; }
// Row length of the refinement's spatial-exponent table sKr: the 2 RB + 1 entries of a window
// column, padded to whole 16-byte rows
__host__ __device__ constexpr int sc_krw(int rb) { return (2 * rb + 1 + 3) / 4 * 4; }

// The screening's certificate (k_fused_sc.cuh, k_march.cuh)
constexpr int kScWSh = 12;      // weights scaled by 2^12 before rounding to 16 bits
constexpr int kScCSh = 8;       // costs scaled by 2^8
constexpr float kScEps = 1.1e-3f;
constexpr float kScAbs = 64.f;  // in the scaled units of E16 (2^20 x E32)
// (1 + eps) / (1 - eps), rounded up
constexpr float kScRho = (1.0f + kScEps) / (1.0f - kScEps) + 1e-6f;
__device__ __forceinline__ float sc_thr(float m) { return fmaf(m + kScAbs, kScRho, kScAbs); }

// ---- refinement of one tile (k_fused's FP32 arithmetic over each pixel's certified candidates)
//
// The range of pixel (u, v) is [dlo - 1, dhi + 1] (range_of(py, px) gives {dlo, dhi}; with B2
// every disparity), clipped at df + 1, df = max(0, u + m - L + 1), where L is the shortest run of
// target values equal to their row's column 0 over the rows v - m .. v + m (row table, .w).  For
// d >= df every target read behind the pixel falls at a column below L (or in the replicate
// padding left of column 0) and returns its row's column-0 value, so each block, its statistics
// and each cost c(q, d) are the same for all such d: E(p, d) = E(p, df) exactly (the same terms in
// the same order).  The lowest d wins ties, so d* <= df and d* + 1 stays inside the clipped range,
// and E(df) stands for the whole tail in the smallest E over d != d*: the cut changes none of the
// outputs.
//
// Each thread owns a column of RPY pixels (column lane, rows RPY warp ..), as the SIMT kernel's
// aggregation does: its loads serve every pixel of the column.  The tile's candidates are
// refined in chunks of DCR disparities (4 when they span at most 4) from the tile's lowest one;
// the FP32 costs come from the two-pass cost phase (the same integers and the same rounding as
// k_fused's costs), stored as planes of [QH][kScRPW] entries sc_psz(QH) apart.
//
// On entry: the tile's images are staged; sIr ([QH][kScRPW], the scaled reference intensities
// of the cost positions) and sKr ([KB][sc_krw(RB)], the spatial exponents K[dx][dy]) are written; *s_rlo
// = INT_MAX and *s_rhi = -1; and range_of's data are visible to every thread.  The function
// synchronises before it reads sIr and returns after the epilogue, without a final barrier.
// images_free() is called by every thread right after the barrier that ends the last chunk's
// cost phase: sref and stgt are not read after it.
template <int RB, bool B2, int NT, int DCR, int RKSEG, int TY, typename RangeOf, typename OnFree>
__device__ __forceinline__ void sc_refine(const FusedArgs &a, const uint8_t *sref, const uint8_t *stgt, float *cb32,
                                          int *vband, int2 *sstr, int2 *sstt, const float *sIr, const float *sKr,
                                          int x0, int y0, int tid, int *s_rlo, int *s_rhi, RangeOf range_of,
                                          OnFree images_free)
{
    constexpr int TX = tile_x(kScWC);
    constexpr int KB = 2 * RB + 1, QH = TY + 2 * RB;
    constexpr int RPW = kScRPW, PSZ = sc_psz(QH);
    constexpr int NW = NT / 32, RPY = TY / NW;
    constexpr int KRW = sc_krw(RB);
    static_assert(TX == 32 && TY % NW == 0, "one warp per strip of RPY rows");
    static_assert(DCR == 4 || DCR == 8, "refinement chunks of 4 or 8 disparities");
    const int lane = tid & 31, warp = tid >> 5;
    const int px = lane, py0 = warp * RPY;
    int rlo[RPY], rhi[RPY];
    {
        int ulo = 0x7fffffff, uhi = -1;
#pragma unroll
        for (int i = 0; i < RPY; ++i) {
            const int u = x0 + px, v = y0 + py0 + i;
            rlo[i] = 1;   // nothing to refine outside the image
            rhi[i] = 0;
            if (u < a.W && v < a.H) {
                const int lmin = __ldg(&a.row_tab[v].w);
                const int cap = min(a.D - 1, max(0, u + a.m - lmin + 1) + 1);
                const int2 rg = B2 ? make_int2(0, 0) : range_of(py0 + i, px);
                rlo[i] = B2 ? 0 : max(rg.x - 1, 0);
                rhi[i] = min(B2 ? a.D - 1 : rg.y + 1, cap);
                ulo = min(ulo, rlo[i]);
                uhi = max(uhi, rhi[i]);
            }
        }
        ulo = __reduce_min_sync(0xffffffffu, ulo);
        uhi = __reduce_max_sync(0xffffffffu, uhi);
        if (lane == 0 && uhi >= 0) {
            atomicMin(s_rlo, ulo);
            atomicMax(s_rhi, uhi);
        }
    }
    __syncthreads();
    const int ulo_t = *s_rlo, uhi_t = *s_rhi;
    const int rw = a.rw;

    float best[RPY], bm1[RPY], bp1[RPY], prev[RPY], sec[B2 ? RPY : 1];
    int bd[RPY];
    float ip[RPY];
    int tlo = 0x7fffffff, thi = -1;   // the union of this thread's ranges
#pragma unroll
    for (int i = 0; i < RPY; ++i) {
        best[i] = __int_as_float(0x7f800000);
        bm1[i] = bp1[i] = prev[i] = best[i];
        if constexpr (B2) sec[i] = best[i];
        bd[i] = -1;
        ip[i] = sIr[(py0 + i + RB) * RPW + px + RB];
        if (rlo[i] <= rhi[i]) {
            tlo = min(tlo, rlo[i]);
            thi = max(thi, rhi[i]);
        }
    }
    const int dcr = (DCR == 4 || uhi_t - ulo_t < 4) ? 4 : DCR;
    const float2 *cb2 = reinterpret_cast<const float2 *>(cb32);
    for (int cb = ulo_t; cb <= uhi_t; cb += dcr) {
        if (DCR == 4 || dcr == 4) {
            switch (rw) {
            case 1: cost_chunk<RB, 4, 1, float, TX, TY, NT, 0, kScRBand4, false, 0, RPW, PSZ, RKSEG, true>(a, sref, stgt, cb32, vband, sstr, sstt, x0, y0, cb, tid); break;
            case 2: cost_chunk<RB, 4, 2, float, TX, TY, NT, 0, kScRBand4, false, 0, RPW, PSZ, RKSEG, true>(a, sref, stgt, cb32, vband, sstr, sstt, x0, y0, cb, tid); break;
            case 3: cost_chunk<RB, 4, 3, float, TX, TY, NT, 0, kScRBand4, false, 0, RPW, PSZ, RKSEG, true>(a, sref, stgt, cb32, vband, sstr, sstt, x0, y0, cb, tid); break;
            case 4: cost_chunk<RB, 4, 4, float, TX, TY, NT, 0, kScRBand4, false, 0, RPW, PSZ, RKSEG, true>(a, sref, stgt, cb32, vband, sstr, sstt, x0, y0, cb, tid); break;
            default: cost_chunk<RB, 4, 5, float, TX, TY, NT, 0, kScRBand4, false, 0, RPW, PSZ, RKSEG, true>(a, sref, stgt, cb32, vband, sstr, sstt, x0, y0, cb, tid); break;
            }
        } else {
            constexpr int D8 = DCR == 4 ? 4 : 8;
            switch (rw) {
            case 1: cost_chunk<RB, D8, 1, float, TX, TY, NT, 0, kScRBand8, false, 0, RPW, PSZ, RKSEG, true>(a, sref, stgt, cb32, vband, sstr, sstt, x0, y0, cb, tid); break;
            case 2: cost_chunk<RB, D8, 2, float, TX, TY, NT, 0, kScRBand8, false, 0, RPW, PSZ, RKSEG, true>(a, sref, stgt, cb32, vband, sstr, sstt, x0, y0, cb, tid); break;
            case 3: cost_chunk<RB, D8, 3, float, TX, TY, NT, 0, kScRBand8, false, 0, RPW, PSZ, RKSEG, true>(a, sref, stgt, cb32, vband, sstr, sstt, x0, y0, cb, tid); break;
            case 4: cost_chunk<RB, D8, 4, float, TX, TY, NT, 0, kScRBand8, false, 0, RPW, PSZ, RKSEG, true>(a, sref, stgt, cb32, vband, sstr, sstt, x0, y0, cb, tid); break;
            default: cost_chunk<RB, D8, 5, float, TX, TY, NT, 0, kScRBand8, false, 0, RPW, PSZ, RKSEG, true>(a, sref, stgt, cb32, vband, sstr, sstt, x0, y0, cb, tid); break;
            }
        }
        if (cb + dcr > uhi_t) images_free();   // the last chunk's cost phase has read the images
        // One pass per thread and chunk: disparities dw .. dw + 2 NPP - 1 from the pair below
        // the thread's lowest candidate in the chunk, NPP pairs (the warp's largest need; 2 or
        // 4).  Pairs past the chunk read its last pair (their sums are discarded), and so do the
        // threads with nothing to refine in the chunk.
        const int lo = max(tlo, cb), hi = min(thi, cb + dcr - 1);
        const int dw = lo <= hi ? cb + ((lo - cb) & ~1) : cb;
        const int need = lo <= hi ? (hi - dw) / 2 + 1 : 0;
        const int wneed = __reduce_max_sync(0xffffffffu, need);
        auto pass = [&](auto npp_c) {
            constexpr int NPP = decltype(npp_c)::value;
            int o[NPP];
#pragma unroll
            for (int k = 0; k < NPP; ++k) o[k] = min((dw - cb) / 2 + k, dcr / 2 - 1) * PSZ;
            float2 e[RPY][NPP];
#pragma unroll
            for (int i = 0; i < RPY; ++i)
#pragma unroll
                for (int k = 0; k < NPP; ++k) e[i][k] = make_float2(0.f, 0.f);
            const float *ib = sIr + py0 * RPW + px;
            const float2 *cq = cb2 + py0 * RPW + px;
#pragma unroll 1
            for (int dx = 0; dx < KB; ++dx) {
                float kr[KRW];
#pragma unroll
                for (int k = 0; k < KRW / 4; ++k) {
                    const float4 q = *reinterpret_cast<const float4 *>(sKr + dx * KRW + 4 * k);
                    kr[4 * k] = q.x;
                    kr[4 * k + 1] = q.y;
                    kr[4 * k + 2] = q.z;
                    kr[4 * k + 3] = q.w;
                }
                // neighbour rows of the column, in increasing order: for every pixel the window
                // rows come in k_fused's order (row inner, column outer); each FMA of a pair is
                // the scalar FMA of k_fused (same operands, one rounding)
#pragma unroll
                for (int r = 0; r < RPY + 2 * RB; ++r) {
                    const float iq = ib[r * RPW + dx];
                    float2 c[NPP];
#pragma unroll
                    for (int k = 0; k < NPP; ++k) c[k] = cq[r * RPW + dx + o[k]];
#pragma unroll
                    for (int i = 0; i < RPY; ++i) {
                        const int dy = r - i;
                        if (dy < 0 || dy > 2 * RB) continue;
                        const float t = iq - ip[i];
                        const float w = ex2_approx(fmaf(-t, t, kr[dy]));
                        const float2 w2 = make_float2(w, w);
#pragma unroll
                        for (int k = 0; k < NPP; ++k) e[i][k] = __ffma2_rn(w2, c[k], e[i][k]);
                    }
                }
            }
            // k_fused's running WTA, in increasing d
#pragma unroll
            for (int i = 0; i < RPY; ++i)
#pragma unroll
                for (int j = 0; j < 2 * NPP; ++j) {
                    const int d = dw + j;
                    if (d < rlo[i] || d > rhi[i] || d > hi) continue;
                    const float v = (j & 1) ? e[i][j >> 1].y : e[i][j >> 1].x;
                    if (v < best[i]) {
                        if constexpr (B2) sec[i] = best[i];
                        best[i] = v;
                        bd[i] = d;
                        bm1[i] = prev[i];
                    } else {
                        if constexpr (B2) sec[i] = fminf(sec[i], v);
                        if (d == bd[i] + 1) bp1[i] = v;
                    }
                    prev[i] = v;
                }
        };
        if (wneed > 2) pass(std::integral_constant<int, 4>());
        else if (wneed > 0) pass(std::integral_constant<int, 2>());
        __syncthreads();
    }

    // ---- epilogue: eq. (subpixel), add back s_i(v), validity from the row table (k_fused's)
#pragma unroll
    for (int i = 0; i < RPY; ++i) {
        const int py = py0 + i;
        const int u = x0 + px, v = y0 + py;
        if (u >= a.W || v >= a.H) continue;
        const int4 rt = __ldg(a.row_tab + v);   // {s_i(v), max s_i, min s_i over v +- m, run}
        float delta = 0.f;
        if (bd[i] > 0 && bd[i] < a.D - 1) {
            const float den = 2.f * bm1[i] + 2.f * bp1[i] - 4.f * best[i];
            if (den > 0.f) delta = (bm1[i] - bp1[i]) / den;
        }
        const size_t o = (size_t)v * a.W + u;
        a.disp[o] = (float)bd[i] + delta + (float)rt.x;
        if (a.wta) a.wta[o] = bd[i];
        if (a.valid) {
            const int ulo = a.m + a.D - 1 + max(0, rt.y);
            const int uhi = a.W - 1 - a.m + min(0, rt.z);
            a.valid[o] = (uint8_t)(v >= a.m && v <= a.H - 1 - a.m && u >= ulo && u <= uhi);
        }
        if constexpr (B2) {
            // the skipped normaliser sum_q w(p,q), as k_fused sums it
            const float ipp = sIr[(py + RB) * RPW + px + RB];
            float ws = 0.f;
            for (int dx = 0; dx < KB; ++dx)
                for (int dy = 0; dy < KB; ++dy) {
                    const float t = sIr[(py + dy) * RPW + px + dx] - ipp;
                    ws += ex2_approx(fmaf(-t, t, a.K[dx * KB + dy]));
                }
            a.best2[2 * o] = best[i] / ws;
            a.best2[2 * o + 1] = sec[i] / ws;
        }
    }
}

// ---- persistent tiles: the next work item is claimed while the current tile is still being
// worked on, and its images are staged into sref / stgt as soon as the tile's last cost phase
// has read them, so that the copies land during the refinement's evaluation and the epilogue.

// The pair and tile of work item `item` (a batch's work list, or one pair's tiles in order).
__device__ __forceinline__ const PairDesc *sc_decode(const PairDesc &single, const PairDesc *pairs,
                                                     const int2 *items, int item, int &tx, int &ty)
{
    if (pairs) {
        const int2 it = items[item];
        tx = it.y & 0xffff;
        ty = it.y >> 16;
        return pairs + it.x;
    }
    tx = item % single.ntx;
    ty = item / single.ntx;
    return &single;
}

// Waits for the images of the tile at (x0, y0), issuing their copies first unless an earlier
// call of sc_claim_ahead did (issued).  The wait is bounded as in stage_images, with the same
// fail-safe: false, with the status word set, when the copies did not land.
__device__ __forceinline__ bool sc_stage(const PairDesc *pd, const FusedArgs &a, uint8_t *sref, uint8_t *stgt,
                                         uint64_t *bar, int *flag, int x0, int y0, int iter, int tid, bool issued)
{
    if (tid == 0) {
        const bool stall = a.stall_test != 0;
        if (!issued) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect_tx(bar, (uint32_t)(a.box_h * (a.ref_box_w + a.tgt_box_w)));
            if (!stall) {
                tma_load_3d(sref, &pd->tmap_ref, 0, (x0 + a.ref_box_x) / 16, y0, bar);
                tma_load_3d(stgt, &pd->tmap_tgt, 0, x0 / 16, y0, bar);
            }
        }
        const bool ok = mbar_wait_limited(bar, (uint32_t)(iter & 1), stall);
        *flag = ok ? 1 : 0;
        if (!ok) {
            atomicOr(a.status, 1);
            mbar_wait_limited(bar, (uint32_t)(iter & 1), stall);   // the CTA returns: no copy may land after it
        }
    }
    __syncthreads();
    return *flag != 0;
}

// Thread 0, once per tile, after a barrier that follows the tile's last read of sref / stgt:
// claims the next work item (*next) and, when its boxes fit the current ones (always within one
// pair), issues its image copies (*staged = 1).  Nothing is issued under the stall test hook.
__device__ __forceinline__ void sc_claim_ahead(const PairDesc &single, const PairDesc *pairs, const int2 *items,
                                               int nitems, int *counter, int item, const FusedArgs &a,
                                               uint8_t *sref, uint8_t *stgt, uint64_t *bar, int *next,
                                               int *claimed, int *staged, int tx_w, int ty_h)
{
    if (*claimed) return;
    *claimed = 1;
    *staged = 0;
    const int nx = pairs ? atomicAdd(counter, 1) : item + (int)gridDim.x;
    *next = nx;
    if (nx >= nitems || a.stall_test) return;
    int txn = 0, tyn = 0;
    const PairDesc *pn = sc_decode(single, pairs, items, nx, txn, tyn);
    const int bh = pn->a.box_h, rbw = pn->a.ref_box_w, tbw = pn->a.tgt_box_w;
    if (bh != a.box_h || rbw != a.ref_box_w || tbw > a.tgt_box_w || pn->a.stall_test) return;
    const int x0n = txn * tx_w, y0n = tyn * ty_h;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_expect_tx(bar, (uint32_t)(bh * (rbw + tbw)));
    tma_load_3d(sref, &pn->tmap_ref, 0, (x0n + pn->a.ref_box_x) / 16, y0n, bar);
    tma_load_3d(stgt, &pn->tmap_tgt, 0, x0n / 16, y0n, bar);
    *staged = 1;
}

}  // namespace sgb
