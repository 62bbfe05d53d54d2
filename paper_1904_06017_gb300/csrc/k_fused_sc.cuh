// k_fused_sc.cuh -- the FP32 fused step (eq. c, eq. omega_s, eq. fbs, WTA, eq. subpixel, §3.2)
// with certified tensor-core screening: its outputs are bit for bit those of k_fused, the plain
// FP32 kernel, at a fraction of the FP32 arithmetic.
//
// Screening.  Per chunk of 32 disparities the costs c32 of the tile plus its bilateral halo are
// computed in FP32 (cost_chunk, exact integer numerators) and stored as c16 = RN16(2^8 c32); the
// aggregation E(p, d) = sum_q w(p, q) c(q, d) runs on the tensor cores (mma.sync m16n8k16, FP16
// operands, FP32 accumulators) over 4 x 4 pixel patches, with the weights w16 = RN16(2^12 w32)
// formed in FP32 from k_fused's own exponent.  Every weight and cost is non-negative and each is
// rounded once to FP16 (relative error 2^-11 in the normal range), so for every (p, d)
//     |E16 - 2^20 E32| <= eps 2^20 E32 + a,
// where E32 is k_fused's FP32 sum: eps covers the two FP16 roundings of each product (2^-10),
// the tensor core's FP32 accumulation (at most 17 terms per k-step and 16 k-steps at bil = 13,
// each addition within 2^-23 of the running sum, truncating or rounding: 3.3e-5), k_fused's own
// chain of at most 169 FMAs (1.0e-5) and the ex2 / exponent roundings of the scaled weight
// (1e-5): 1.03e-3, taken as 1.1e-3; a (64, i.e. 6.1e-5 unscaled) covers FP16 subnormal weights
// and costs even if the tensor core flushed them.  Hence the FP32 argmin d* (lowest d on ties) satisfies
//     E16(d*) <= thr(min_d E16) = (min_d E16 + a) (1 + eps) / (1 - eps) + a,
// and so does every d that ties it.  Each pixel keeps the range [dlo, dhi] that holds every d
// with E16(d) <= thr(running minimum); a chunk whose minimum m makes thr(m) smaller than the
// previous minimum drops the earlier range (none of its disparities can satisfy the final test).
//
// Refinement.  After the last chunk the tile refines [dlo - 1, dhi + 1] of every pixel with
// k_fused's arithmetic (sc_refine): FP32 costs from the two-pass cost phase (the same integers
// and roundings as k_fused's), the weight ex2(fma(-t, t, K)), and the 121-term FMA chain in
// k_fused's order (window column outer, row inner), then k_fused's running WTA in increasing d.
// The winner and its two neighbours (the parabola of eq. subpixel) are therefore k_fused's
// values exactly.
//
// Taken for ranges of at most 32 disparities (sc_route, which gives both sides' times); k_march
// and k_refine share the bound and the refinement.
#pragma once
#include "k_fused_tc.cuh"
#include "k_sc_refine.cuh"

namespace sgb {

constexpr int kScBand = 6;      // cost rows per band of the screening chunk's cost phase
constexpr int kScSeg = 6;       // cost columns per horizontal work item (6 rows x 7 segments x 8 quads = 336 items)
// Row length of the staged FP32 intensities (>= QW + 2, >= 28 + 16): 44 up to bil = 11 (the
// measured layout), 48 at bil = 13
__host__ __device__ constexpr int sc_qwi(int rb) { return rb >= 6 ? 48 : 44; }
constexpr int kScRefOff = 16384;     // bytes into escr: past the refinement's window sums (<= 10 KB)

// Shared memory of the screened form (offsets from the 128-byte aligned dynamic base):
//   sref, stgt  image tiles (TMA), as in k_fused
//   cbuf   screening: [QH][QW][32] FP16 costs (16-byte units swizzled by bits 1..2 of the
//          column); refinement, in the same bytes: 4 planes of FP32 disparity pairs (float2
//          [QH][kScRPW], sc_psz(QH) entries apart), then the window statistics of a band
//   escr   the cost phase's vertical window sums ([band][CW][32] i32); after the screening the
//          refinement's vertical sums, and from kScRefOff on the intensities again as [QH][kScRPW] f32 and
//          the spatial exponents as [2 RB + 1][sc_krw(RB)] f32
//   sstr, sstt  window statistics of one band
//   sI     [QH][sc_qwi(RB)] f32  the reference intensities times sqrt(log2 e) / sigma1 of the cost
//          positions (1e18 outside the image, as in k_fused)
//   skxy   the row terms of the spatial exponent, (nKy(j), nKy(j - 2)) for j = -1 .. 3 + 2 RB
//          (float2)
//   sst    the screening state of every pixel of the tile ([TY][TX] float2: the running minimum
//          of E16, and the candidate range dlo | dhi << 16 as the bits of the second float)
struct ScLayout {
    size_t sref, stgt, cbuf, escr, sstr, sstt, sI, skxy, sst, total;
};

__host__ __device__ inline ScLayout sc_layout(int rb, int m, int ref_box_w, int tgt_box_w, int box_h)
{
    ScLayout L;
    const int TX = tile_x(kScWC), TY = tile_y(kScWC);
    const int QH = TY + 2 * rb, QW = TX + 2 * rb, CW = TX + 2 * m, NKS = 4 + 2 * rb, KB = 2 * rb + 1;
    const size_t vb = (size_t)kScBand * CW * kScDC * 4, eb = kScRefOff + ((size_t)QH * kScRPW + KB * sc_krw(rb)) * 4;
    const size_t c16 = (size_t)QH * QW * kScDC * 2, c32 = (size_t)kScDCR * sc_psz(QH) * 4;
    L.sref = 0;
    L.stgt = align_up((size_t)box_h * ref_box_w, 128);
    L.cbuf = align_up(L.stgt + (size_t)box_h * tgt_box_w, 128);
    L.escr = align_up(L.cbuf + (c16 > c32 ? c16 : c32), 128);
    L.sstr = align_up(L.escr + (vb > eb ? vb : eb), 16);
    L.sstt = align_up(L.sstr + (size_t)kScBand * QW * 8, 16);
    L.sI = align_up(L.sstt + (size_t)kScBand * (QW + kScDC - 1) * 8, 16);
    L.skxy = align_up(L.sI + (size_t)QH * sc_qwi(rb) * 4, 16);
    L.sst = align_up(L.skxy + (size_t)(NKS + 2) * 8, 16);
    L.total = align_up(L.sst + (size_t)TY * TX * 8, 128);
    return L;
}

// Two FP32 values as a packed FP16 pair (lo in the low half), each rounded to nearest.
__device__ __forceinline__ uint32_t h2_rn(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

template <int RB>
__global__ void __launch_bounds__(kThreads, 1)
k_fused_sc(const __grid_constant__ PairDesc single, const PairDesc *__restrict__ pairs,
           const int2 *__restrict__ items, int nitems, int *__restrict__ counter)
{
    using T = __half;
    using X = TcOps<T>;
    constexpr int DC = kScDC, DCR = kScDCR;
    constexpr int TX = tile_x(kScWC), TY = tile_y(kScWC);
    constexpr int KB = 2 * RB + 1;
    constexpr int QH = TY + 2 * RB, QW = TX + 2 * RB;
    constexpr int QWI = sc_qwi(RB);
    constexpr int NKS = 4 + 2 * RB;              // k-steps: the window rows of a patch
    constexpr int NPX = TX / 4, NPY = TY / 4;    // patches of the tile
    constexpr int NPW = NPX * NPY / kWarps;      // patches per warp
    static_assert(RB <= kScMaxRB && NKS <= 16 && QW + 2 <= QWI,
                  "a window row spans at most 16 columns");
    static_assert((NPX * NPY) % kWarps == 0 && NPW % 2 == 0, "patches must split evenly over the warps");
    static_assert(kScRBand8 * (TX + 2 * (RB + kMaxRW)) * kScDCR * 4 <= kScRefOff &&
                      kScRBand4 * (TX + 2 * (RB + kMaxRW)) * 4 * 4 <= kScRefOff, "refinement window sums");
    // the refinement's band statistics sit in the cost buffer, past its FP32 planes
    static_assert(kScRBand8 <= kScRBand4, "the refinement statistics are sized for the taller band");
    static_assert((size_t)kScDCR * sc_psz(QH) * 4 + (size_t)kScRBand4 * (2 * QW + kScDCR - 1) * 8 <=
                      (size_t)QH * QW * kScDC * 2, "refinement statistics");
    static_assert(kScRefOff + (QH * kScRPW + KB * sc_krw(RB)) * 4 <= kScBand * (TX + 2 * RB) * kScDC * 4,
                  "refinement tables");
    constexpr int RPW = kScRPW, PSZ = sc_psz(QH);
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(16) FusedArgs s_args;
    __shared__ int s_item;
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ int s_flag;
    __shared__ int s_rlo, s_rhi;
    __shared__ int s_next, s_claimed, s_staged;   // the work item claimed ahead, its copies issued
    __shared__ int s_dend;                        // the tile's screening chunks start below this

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t4 = lane & 3;      // fragment row group and column pair
    const int mx = g & 3, my0 = g >> 2;          // this lane's fragment pixels m0 = g, m1 = g + 8
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
        const ScLayout L = sc_layout(RB, a.m, RP, a.tgt_box_w, a.box_h);
        uint8_t *sref = smem + L.sref;
        uint8_t *stgt = smem + L.stgt;
        T *cb16 = reinterpret_cast<T *>(smem + L.cbuf);
        float *cb32 = reinterpret_cast<float *>(smem + L.cbuf);
        int *vband = reinterpret_cast<int *>(smem + L.escr);
        int2 *sstr = reinterpret_cast<int2 *>(smem + L.sstr);
        int2 *sstt = reinterpret_cast<int2 *>(smem + L.sstt);
        float *sI = reinterpret_cast<float *>(smem + L.sI);
        const int x0 = tx * TX, y0 = ty * TY;
        if (tid == 0) {
            s_rlo = 0x7fffffff;
            s_rhi = -1;
        }
        if (warp == 0) {
            // For d >= df = max(0, u + m - L + 1) every cost behind pixel (u, v) repeats its value at
            // df (L: the row table's shortest column-0 run over v +- m), so a chunk that starts past
            // the tile's largest df + 1 changes no candidate range (they are clipped at df + 1): the
            // screening stops before it.
            int lm = 0x7fffffff;
            for (int v = y0 + lane; v < min(y0 + TY, a.H); v += 32) lm = min(lm, __ldg(&a.row_tab[v].w));
            lm = __reduce_min_sync(0xffffffffu, lm);
            if (lane == 0) s_dend = min(a.D, max(0, min(x0 + TX, a.W) - 1 + a.m - lm + 1) + 2);
        }

        if (!sc_stage(pd, a, sref, stgt, &s_bar, &s_flag, x0, y0, iter, tid, issued)) return;
        // called after a barrier that follows the tile's last read of sref / stgt
        auto images_free = [&]() {
            if (tid == 0)
                sc_claim_ahead(single, pairs, items, nitems, counter, item, a, sref, stgt, &s_bar, &s_next,
                               &s_claimed, &s_staged, TX, TY);
        };

        const int rw = a.rw;
        // scaled reference intensities of the cost positions, exactly as k_fused stages them;
        // positions outside the image and the row padding get 1e18 (weight 0)
        for (int i = tid; i < QH * QWI; i += kThreads) {
            const int yq = i / QWI, xq = i - yq * QWI;
            const int ix = x0 - RB + xq, iy = y0 - RB + yq;
            float v = 1e18f;
            if (xq < QW && ix >= 0 && ix < a.W && iy >= 0 && iy < a.H)
                v = (float)sref[(yq + rw) * RP + a.ref_e + xq + rw] * a.iscale;
            sI[i] = v;
        }
        // spatial exponents, separable: -(K[dx][dy] + 12) = nKx(dx) + nKy(dy) with
        // nKx(i) = -(K[i][RB] + 12) and nKy(j) = -K[RB][j] (1e30 outside the window: weight 0).
        // The row terms as a table over j = r - my (the lane's first pixel row): (nKy(j), nKy(j - 2))
        float2 *sky = reinterpret_cast<float2 *>(smem + L.skxy);
        auto nky = [&](int j) { return (j >= 0 && j <= 2 * RB) ? -a.K[RB * KB + j] : 1e30f; };
        for (int j = tid; j < NKS + 2; j += kThreads) sky[j] = make_float2(nky(j - 1), nky(j - 3));
        float2 *sst0 = reinterpret_cast<float2 *>(smem + L.sst);
        for (int j = tid; j < TY * TX; j += kThreads) sst0[j] = make_float2(__int_as_float(0x7f800000), 0.f);
        // this lane's column terms: columns 2 t4 + {0, 1} and 2 t4 + {8, 9} of a window row
        auto nkx = [&](int col) {
            const int i = col - mx;
            return (i >= 0 && i <= 2 * RB) ? -(a.K[i * KB + RB] + (float)kScWSh) : 1e30f;
        };
        const float2 nkx_lo = make_float2(nkx(2 * t4), nkx(2 * t4 + 1));
        const float2 nkx_hi = make_float2(nkx(2 * t4 + 8), nkx(2 * t4 + 9));
        __syncthreads();

        // Screening work: vertical segments of three patches (8 patch columns x 3 segments of 3
        // patch rows), two per warp.  The patches of a segment share their window rows: each
        // row's costs (ldmatrix) and intensities are read once for every patch that uses it.
        constexpr int NSEGR = NPY / 3;                // segments per patch column
        constexpr int NR3 = 8 + NKS;                  // window rows of a segment
        static_assert(NPY % 3 == 0 && NPX * NSEGR == 2 * kWarps, "two segments of three patches per warp");
        // the screening state of each pixel lives in sst between chunks (set before the barrier
        // above); a quad reads its two pixels' entries and its first lane writes them back
        float2 *sst = reinterpret_cast<float2 *>(smem + L.sst);
        const int dend = s_dend;   // the bound (set before sc_stage's barrier)
        for (int d0 = 0; d0 < dend; d0 += DC) {
            // ---- costs of the chunk, 32 disparities, times 2^8, FP16, swizzled
            switch (rw) {
            case 1: cost_chunk<RB, DC, 1, T, TX, TY, kThreads, 0, kScBand, true, kScCSh, 0, 0, kScSeg>(a, sref, stgt, cb16, vband, sstr, sstt, x0, y0, d0, tid); break;
            case 2: cost_chunk<RB, DC, 2, T, TX, TY, kThreads, 0, kScBand, true, kScCSh, 0, 0, kScSeg>(a, sref, stgt, cb16, vband, sstr, sstt, x0, y0, d0, tid); break;
            case 3: cost_chunk<RB, DC, 3, T, TX, TY, kThreads, 0, kScBand, true, kScCSh, 0, 0, kScSeg>(a, sref, stgt, cb16, vband, sstr, sstt, x0, y0, d0, tid); break;
            case 4: cost_chunk<RB, DC, 4, T, TX, TY, kThreads, 0, kScBand, true, kScCSh, 0, 0, kScSeg>(a, sref, stgt, cb16, vband, sstr, sstt, x0, y0, d0, tid); break;
            default: cost_chunk<RB, DC, 5, T, TX, TY, kThreads, 0, kScBand, true, kScCSh, 0, 0, kScSeg>(a, sref, stgt, cb16, vband, sstr, sstt, x0, y0, d0, tid); break;
            }
            const int dn = min(DC, a.D - d0);
#pragma unroll 1
            for (int si = 0; si < 2; ++si) {
                const int sg = warp + kWarps * si;
                const int px0 = (sg % NPX) * 4, pys = (sg / NPX) * 12;
                float2 nip[3][2];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const float ip0 = sI[(pys + 4 * i + RB + my0) * QWI + px0 + RB + mx];
                    const float ip1 = sI[(pys + 4 * i + RB + my0 + 2) * QWI + px0 + RB + mx];
                    nip[i][0] = make_float2(-ip0, -ip0);
                    nip[i][1] = make_float2(-ip1, -ip1);
                }
                // ldmatrix rows: lanes 8i..8i+7 name matrix i = (k half, unit): k slots 0..7 /
                // 8..15 of the window row, 8-disparity units 2j + (lane >> 4)
                const int kk = ((lane >> 3) & 1) * 8 + (lane & 7);
                const int xq = min(px0 + kk, QW - 1);   // padding slots (zero weight) read a valid cost
                const uint32_t pos = smem_addr(cb16 + ((size_t)pys * QW + xq) * DC);
                uint32_t brow[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) brow[j] = pos + (uint32_t)(swz_unit<DC>(2 * j + (lane >> 4), xq) << 4);
                const float *irow = sI + pys * QWI + px0 + 2 * t4;
                float acc[3][4][4];
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int nb = 0; nb < 4; ++nb)
#pragma unroll
                        for (int k = 0; k < 4; ++k) acc[i][nb][k] = 0.f;
#pragma unroll
                for (int ra = 0; ra < NR3; ++ra) {
                    const float2 qlo = *reinterpret_cast<const float2 *>(irow + ra * QWI);
                    const float2 qhi = *reinterpret_cast<const float2 *>(irow + ra * QWI + 8);
                    uint32_t b[2][4];
                    const uint32_t roff = (uint32_t)(ra * QW * DC * (int)sizeof(__half));
#pragma unroll
                    for (int j = 0; j < 2; ++j) ldsm_x4_t(brow[j] + roff, b[j][0], b[j][1], b[j][2], b[j][3]);
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        const int r = ra - 4 * i;             // this patch's window row
                        if (r < 0 || r >= NKS) continue;
                        const float2 ky = sky[r - my0 + 1];   // (nKy(r - my0), nKy(r - my0 - 2))
                        // t = I_q - I_p; e' = t^2 - (K + 12); w16 = RN16(2^-e')
                        const float2 ta = __fadd2_rn(qlo, nip[i][0]), tb = __fadd2_rn(qlo, nip[i][1]);
                        const float2 tc = __fadd2_rn(qhi, nip[i][0]), td = __fadd2_rn(qhi, nip[i][1]);
                        const float2 ea = __fadd2_rn(__ffma2_rn(ta, ta, nkx_lo), make_float2(ky.x, ky.x));
                        const float2 eb = __fadd2_rn(__ffma2_rn(tb, tb, nkx_lo), make_float2(ky.y, ky.y));
                        const float2 ec = __fadd2_rn(__ffma2_rn(tc, tc, nkx_hi), make_float2(ky.x, ky.x));
                        const float2 ed = __fadd2_rn(__ffma2_rn(td, td, nkx_hi), make_float2(ky.y, ky.y));
                        uint32_t af[4];
                        af[0] = h2_rn(ex2_approx(-ea.x), ex2_approx(-ea.y));
                        af[1] = h2_rn(ex2_approx(-eb.x), ex2_approx(-eb.y));
                        af[2] = h2_rn(ex2_approx(-ec.x), ex2_approx(-ec.y));
                        af[3] = h2_rn(ex2_approx(-ed.x), ex2_approx(-ed.y));
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            X::mma(acc[i][2 * j], af, b[j][0], b[j][1]);
                            X::mma(acc[i][2 * j + 1], af, b[j][2], b[j][3]);
                        }
                    }
                }
                // the screening update, straight from the fragments: lane (g, t4) holds
                // disparities 8 nb + 2 t4 + {0, 1} (nb = 0..3) of pixels g and g + 8, and the
                // four lanes of a quad hold all 32 disparities of the same two pixels
#pragma unroll
                for (int i = 0; i < 3; ++i) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float v[8];
#pragma unroll
                        for (int nb = 0; nb < 4; ++nb) {
                            v[2 * nb] = acc[i][nb][2 * h];
                            v[2 * nb + 1] = acc[i][nb][2 * h + 1];
                        }
                        if (dn < DC) {   // the last chunk of a search range off the chunk grid
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                if (8 * (j >> 1) + 2 * t4 + (j & 1) >= dn) v[j] = __int_as_float(0x7f800000);
                        }
                        float cm = v[0];
#pragma unroll
                        for (int j = 1; j < 8; ++j) cm = fminf(cm, v[j]);
                        cm = fminf(cm, __shfl_xor_sync(0xffffffffu, cm, 1));
                        cm = fminf(cm, __shfl_xor_sync(0xffffffffu, cm, 2));
                        // the pixel's state.  A chunk whose minimum lies above thr(running
                        // minimum) changes neither (every E16 of it fails the test, and the
                        // minimum stays): a warp with no such pixel skips the update
                        const int pidx = ((sg / NPX) * 12 + 4 * i + my0 + 2 * h) * TX + px0 + mx;
                        const float2 sv = sst[pidx];
                        const float em = sv.x;
                        if (!__any_sync(0xffffffffu, cm <= sc_thr(em))) continue;
                        const float nm = fminf(em, cm);
                        const float tn = sc_thr(nm);
                        uint32_t mk = 0;
#pragma unroll
                        for (int j = 0; j < 8; ++j) mk |= (v[j] <= tn) ? (1u << (8 * (j >> 1) + (j & 1))) : 0u;
                        mk <<= 2 * t4;
                        mk |= __shfl_xor_sync(0xffffffffu, mk, 1);
                        mk |= __shfl_xor_sync(0xffffffffu, mk, 2);
                        const bool reset = mk && tn < em;   // the earlier range cannot hold d*
                        const int lo = d0 + __ffs(mk) - 1, hi = d0 + 31 - __clz(mk);
                        int r = __float_as_int(sv.y);
                        if (reset) r = (r & ~0xffff) | lo;
                        if (mk) r = (r & 0xffff) | (hi << 16);
                        if (t4 == 0) sst[pidx] = make_float2(nm, __int_as_float(r));
                    }
                }
            }
            // The aggregation reads nothing the next cost phase writes before its
            // first barrier (window sums, band statistics), so its fast warps go on to that
            // phase; the barrier there orders every read of this chunk's costs before the new
            // ones are stored.
        }
        __syncthreads();   // every pixel's screening state is final

        // ---- refinement of the candidates
        // the intensities on the refinement's row pitch: sI itself where the pitches agree
        float *sIc = reinterpret_cast<float *>(smem + L.escr + kScRefOff);   // [QH][RPW]
        float *sKr = sIc + QH * RPW;                                           // [KB][sc_krw(RB)]
        if constexpr (QWI != RPW) {
            for (int i = tid; i < QH * RPW; i += kThreads) {
                const int yq = i / RPW, xq = i - yq * RPW;
                sIc[i] = xq < QWI ? sI[yq * QWI + xq] : 1e18f;
            }
        }
        const float *sIr = QWI == RPW ? sI : sIc;
        for (int i = tid; i < KB * sc_krw(RB); i += kThreads) {
            const int dx = i / sc_krw(RB), dy = i - dx * sc_krw(RB);
            sKr[i] = dy < KB ? a.K[dx * KB + dy] : 0.f;
        }
        int2 *rstr = reinterpret_cast<int2 *>(cb32 + (size_t)DCR * PSZ);   // [kScRBand4][QW]
        int2 *rstt = rstr + kScRBand4 * QW;                                  // [kScRBand4][QW + DCR - 1]
        sc_refine<RB, false, kThreads, DCR, kScRSeg, TY>(a, sref, stgt, cb32, vband, rstr, rstt, sIr, sKr, x0, y0, tid, &s_rlo, &s_rhi,
                                         [&](int py, int px) {
                                             const int r = __float_as_int(sst[py * TX + px].y);
                                             return make_int2(r & 0xffff, r >> 16);
                                         },
                                         images_free);
        __syncthreads();
        images_free();   // (claimed already, unless the tile had no candidates to refine)
    }  // tile loop
}

inline FusedKernel pick_sc_rb(int rb)
{
    switch (rb) {
    case 0: return k_fused_sc<0>;
    case 1: return k_fused_sc<1>;
    case 2: return k_fused_sc<2>;
    case 3: return k_fused_sc<3>;
    case 4: return k_fused_sc<4>;
    case 5: return k_fused_sc<5>;
    case 6: return k_fused_sc<6>;   // bil = 13: a window row fills the 16 k-slots
    }
    return nullptr;
}

}  // namespace sgb
