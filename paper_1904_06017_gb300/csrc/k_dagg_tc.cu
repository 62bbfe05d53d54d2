// k_dagg_tc.cu -- the adjoint of the bilateral aggregation in its costs (k_diff.cu, GC) on the tensor
// cores, with FP32 accuracy from split operands.
//
// gc(q, d) = sum_p w(p, q) h(p, d), and with w (sI_p - sI_q) in place of w the weights' term, are banded
// matrix products.  A CTA marches down a strip of 32 pixel columns, four rows (a band) per iteration,
// and keeps the h of the rows its window spans in a shared-memory ring, a chunk of 32 disparities at a
// time; the four rows that the next band adds are copied (cp.async) while the band is worked on, one
// barrier per iteration.  A warp owns a 4 x 4 pixel patch: one k-step per window row (K = the 4 + 2 RB
// columns that the patch's windows span, padded to 16 with zero weights), four mma.sync m16n8k16 per
// product.
//
// Split.  A value x (scaled by a power of two into the FP16 range) is hi = RN16(x) and
// lo = RN16(x - hi): 22 bits.  w h is summed as w_hi h_hi + w_lo h_hi + w_hi h_lo in FP32 accumulators
// (the products are exact; w_lo h_lo is below 2^-22).  h comes split from the kernel that writes it
// (k_diff.cuh: the layout): no conversion on the way into the ring.  Weights are formed in FP32 as in
// k_dagg and scaled by 2^14; h, which has the range of the caller's dS/dl, by a power of two from the
// image's largest finite |dS/dl|.  Error of the gradients against 64 bits: below the FP32 form's on five
// seeds of 8 x 960 x 540 (reference 5.40e-6 -> 5.37e-6, target 4.19e-6 -> 4.07e-6 on the first).
//
// What is not finite, or out of the split's range, is flagged by row where it is written; a patch
// whose window rows hold a flagged row sums one value at a time instead, so that a NaN reaches the pixels
// whose windows hold it and no others.
//
// Bound: the tensor pipe at 45 % and the issue slots at 45 % (per window row and chunk 24 mma beside about
// 100 instructions that form and split 16 operands per lane); 54 % of the K slots carry a weight.  Two CTAs
// per SM, so that one's epilogue and barrier pass under the other's products, and the weights of the
// next window row are formed between the products of the current one.  8 x 960 x 540, D = 64, k = 11:
// FP32 form (FFMA, 65 % of the pipe) 3.11 ms, here 2.59 ms.  Slower and left out: producer warps that split
// an FP32 h (2.81 ms), 64 disparities a chunk in one CTA with pairs of warps sharing a patch (3.12), the
// same without pairs (3.37).  FWD and H in this form (1.73 -> 1.48 and 3.30 -> 2.53 ms) are left out too:
// their error against 64 bits is lower than the FP32 form's, but where a target window is nearly flat
// the FP32 form's rounding of E reaches 1.3e-3 of a gradient's root mean square, and the two forms
// differ by as much.
#include <math.h>

#include "internal.cuh"
#include "k_diff.cuh"
#include "k_fused_common.cuh"
#include "k_fused_tc.cuh"
#include "row_shift.cuh"
#include "stereo_diff.h"

namespace sgb {
namespace {

constexpr float kFar = 1e18f;        // scaled intensity of an out-of-image neighbour: weight 0
constexpr int kWSh = 14;             // weights are scaled by 2^kWSh
constexpr int kNT = 256;             // eight warps: the eight patches of a band
constexpr int kSIP = 48;             // row length of the intensity and beta rings
constexpr int N = 32;                // disparities of a chunk

template <int RB>
struct Shape {
    static constexpr int QW = 32 + 2 * RB, RR = 8 + 2 * RB, ROWB = QW * N * 2;
    static constexpr int PHI = (RB & 1) ? 2 : 0, LEAD = (2 * RB + PHI) / 4;
    static constexpr size_t lo = (size_t)RR * ROWB;              // the low parts' ring
    static constexpr size_t sI = 2 * lo;                         // [RR][kSIP] f32
    static constexpr size_t sB = sI + (size_t)RR * kSIP * 4;     // [RR][kSIP] f32: beta
    static constexpr size_t ky = sB + (size_t)RR * kSIP * 4;     // [NKS + 3] f32 pairs: see the kernel
    static constexpr size_t bad = ky + (size_t)(4 + 2 * RB + 3) * 8;   // [RR] int: tag of the row last found to hold
    static constexpr size_t total = bad + (size_t)RR * 4;        // a value that the split cannot carry
};

// The 16-byte unit of disparities [8 unit, 8 unit + 8) of column x sits at unit ^ swz(x): the eight
// rows of an ldmatrix (consecutive columns) meet distinct banks.
__device__ __forceinline__ int swz(int x) { return (x >> 1) & 3; }

__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src, bool valid)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(valid ? 8 : 0) : "memory");
}
__device__ __forceinline__ float quad_sum(float x)
{
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    return x + __shfl_xor_sync(0xffffffffu, x, 2);
}

// Of each image: the partial maxima of |dS/dl| that scale h, and the row flags of h cleared.
__global__ void __launch_bounds__(256) k_dabsmax(const float *__restrict__ g, int H, int W, unsigned *__restrict__ range,
                                                 int *__restrict__ hbad)
{
    const int b = blockIdx.y;
    const size_t n = (size_t)H * W;
    unsigned m = 0;
    for (size_t i = blockIdx.x * 256 + threadIdx.x; i < n; i += 256 * kAggRange) {
        const unsigned v = __float_as_uint(g[b * n + i]) & 0x7fffffffu;
        if (v < 0x7f800000u) m = max(m, v);
        if (i < H) hbad[b * H + i] = 0;
    }
    __shared__ unsigned s[8];
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) m = max(m, s[k]);
        range[b * kAggRange + blockIdx.x] = m;
    }
}

template <int RB>
__global__ void __launch_bounds__(kNT, 2) k_dagg_tc(const AggArgs a, int bands_per_item)
{
    using S = Shape<RB>;
    constexpr int QW = S::QW, RR = S::RR, NKS = 4 + 2 * RB;
    extern __shared__ __align__(128) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t4 = lane & 3;
    const int W = a.W, H = a.H, D = a.D;
    const size_t HW = (size_t)H * W;
    const int strips = (W + 31) / 32, b = blockIdx.y;
    const int x0 = 32 * (blockIdx.x % strips), band0 = (blockIdx.x / strips) * bands_per_item;
    const int nb = min(bands_per_item, (H + 3) / 4 - band0), Y0 = 4 * band0;
    const int nsteps = nb + S::LEAD;
    const int nchunks = (D + N - 1) / N;
    float *sI = reinterpret_cast<float *>(smem + S::sI);
    float *sB = reinterpret_cast<float *>(smem + S::sB);
    const int hs = h_shift(a, b, lane);
    const float *img = a.img + b * HW;
    int *bad = reinterpret_cast<int *>(smem + S::bad);
    for (int i = tid; i < RR; i += kNT) bad[i] = 0;
    // entry 3 + j, twice: the exponent -ky of window row j of a pixel (1e30 outside the window: weight 0)
    float2 *kyt = reinterpret_cast<float2 *>(smem + S::ky);
    for (int i = tid; i < NKS + 3; i += kNT) {
        const int j = i - 3 - RB;
        const float v = j >= -RB && j <= RB ? -(a.k0 * (float)(j * j)) : 1e30f;
        kyt[i] = make_float2(v, v);
    }
    __syncthreads();

    for (int ch = 0; ch < nchunks; ++ch) {
        const int d0 = ch * N, dn = min(N, D - d0);
        const int tag0 = 1 + ch * 4 * (nsteps + 1);      // ring row cr of this chunk has the tag tag0 + cr
        const int ng = (dn + 3) / 4;
        const __half *vol = reinterpret_cast<const __half *>(a.vol) + ((size_t)b * ((D + 3) / 4) + d0 / 4) * HW * 8;
        {
            const int px0 = 4 * warp, mx = g & 3, my0 = g >> 2;
            // spatial exponents -(kx + 14) of this lane's columns 2 t4 + {0, 1} and + {8, 9} of a window
            // row (1e30 outside the window: weight 0)
            auto nkx = [&](int col) {
                const int i = col - mx - RB;
                return (i >= -RB && i <= RB) ? -(a.k0 * (float)(i * i)) - (float)kWSh : 1e30f;
            };
            const float2 nkx_lo = make_float2(nkx(2 * t4), nkx(2 * t4 + 1));
            const float2 nkx_hi = make_float2(nkx(2 * t4 + 8), nkx(2 * t4 + 9));
            const int xq = min(px0 + ((lane >> 3) & 1) * 8 + (lane & 7), QW - 1);
            uint32_t bo[N / 16];
#pragma unroll
            for (int j = 0; j < N / 16; ++j)
                bo[j] = smem_addr(smem) + (uint32_t)(xq * N * 2 + (((2 * j + (lane >> 4)) ^ swz(xq)) << 4));
            const float2 *kyl = kyt + 3 - my0;
            int slot0 = 0, slot = 0;               // ring slots of the step's first row, of the band's
            for (int p = 0; p <= nsteps; ++p) {
                // the rows of the step after this iteration's: in flight while the band is worked on
                const int first = max(0, 4 * p - S::PHI);
                const int sr = tid / kSIP, sx = tid - sr * kSIP, scr = 4 * p - S::PHI + sr;
                float si = kFar, sbv = 0.f;
                int rowbad = 0;
                if (p < nsteps) {
                    if (sr < 4 && scr >= 0) {
                        const int y = Y0 - RB + scr, u = x0 - RB + sx;
                        if (sx < QW && y >= 0 && y < H && u >= 0 && u < W) {
                            si = img[(size_t)y * W + u];
                            sbv = a.beta[b * HW + (size_t)y * W + u];
                            rowbad = a.hbad[b * H + y];
                        }
                    }
                    // warp: row r, groups wq + 2 i; lane: 8 bytes (hi or lo) of positions (lane >> 1) + 16 k
                    const int r = warp & 3, wq = warp >> 2, cr = 4 * p - S::PHI + r, y = Y0 - RB + cr;
                    int sl = slot0 + cr - first;
                    if (sl >= RR) sl -= RR;
                    if (cr >= 0) {
                        const int x = lane >> 1, u = x0 - RB + x;
                        const uint32_t dst = smem_addr(smem) + (uint32_t)((lane & 1) * S::lo + sl * S::ROWB + x * N * 2 + wq * 8);
                        const bool yin = y >= 0 && y < H;
                        const __half *src = vol + ((size_t)wq * HW + (yin ? (size_t)y * W : 0)) * 8 + (lane & 1) * 4;
#pragma unroll
                        for (int i = 0; i < N / 8; ++i)
#pragma unroll
                            for (int k = 0; k < (QW + 15) / 16; ++k) {
                                if (x + 16 * k >= QW) continue;
                                const bool ok = yin && wq + 2 * i < ng && u + 16 * k >= 0 && u + 16 * k < W;
                                cp_async8(dst + (uint32_t)(16 * k * N * 2 + ((i ^ swz(x)) << 4)),
                                          ok ? src + (size_t)(2 * i) * HW * 8 + (ptrdiff_t)(u + 16 * k) * 8 : vol, ok);
                            }
                    }
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
                const int band = p - S::LEAD - 1;
                if (band >= 0) {
                    const int s0 = (slot + RB + my0) % RR, s2 = (slot + RB + my0 + 2) % RR;
                    const float ip0 = sI[s0 * kSIP + px0 + RB + mx], ip1 = sI[s2 * kSIP + px0 + RB + mx];
                    const float2 np0 = make_float2(-ip0, -ip0), np1 = make_float2(-ip1, -ip1);
                    float acc[N / 8][4], ac1[N / 8][4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
#pragma unroll
                        for (int n = 0; n < N / 8; ++n) {
                            acc[n][k] = ac1[n][k] = 0.f;
                        }
                    }
                    // the costs that the epilogue reads, into the caches ahead of the products (lane: a disparity)
                    if (lane < dn && x0 + px0 < W) {
                        const float *c = a.cost + ((size_t)b * D + d0 + lane) * HW + x0 + px0;
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (Y0 + 4 * band + k < H)
                                asm volatile("prefetch.global.L1 [%0];" ::"l"(c + (size_t)(Y0 + 4 * band + k) * W));
                    }
                    int rs = slot + lane;
                    if (rs >= RR) rs -= RR;
                    const bool slow = __any_sync(0xffffffffu, lane < NKS && bad[rs] == tag0 + 4 * band + lane);
                    float2 sb[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};   // GC: sum_q w (sI_q - sI_p) beta(q)
                    if (!slow) {
                        int sl = slot;
                        const float *il = sI + px0 + 2 * t4;
                        const float2 *kyr = kyl;
                        // the weights of window row r as A fragments (hi, lo; of w, and of w t with t = sI_q - sI_p):
                        // w 2^14 = 2^-(t^2 - (kx + ky) - 14)
                        struct Frag {
                            uint32_t ah[4], al[4], dh[4], dl[4];
                            uint32_t ro;          // the row's offset in the ring
                        };
                        auto weights = [&](Frag &f) {
                            const float *irow = il + sl * kSIP;
                            f.ro = (uint32_t)(sl * S::ROWB);
                            sl = sl == RR - 1 ? 0 : sl + 1;
                            const float2 qlo = *reinterpret_cast<const float2 *>(irow);
                            const float2 qhi = *reinterpret_cast<const float2 *>(irow + 8);
                            const float2 ky0 = kyr[0], ky1 = kyr[-2];
                            auto pairw = [&](float2 q, float2 np, float2 nk, float2 ky, int i) {
                                const float2 t = __fadd2_rn(q, np);
                                const float2 e = __ffma2_rn(t, t, __fadd2_rn(nk, ky));
                                const float2 w = make_float2(ex2_approx(-e.x), ex2_approx(-e.y));
                                split2(w.x, w.y, f.ah[i], f.al[i]);
                                const float2 d = __fmul2_rn(w, t);                 // w (sI_q - sI_p)
                                split2(d.x, d.y, f.dh[i], f.dl[i]);
                                sb[i & 1] = __ffma2_rn(d, *reinterpret_cast<const float2 *>(irow + (S::sB - S::sI) / 4 + (i & 2) * 4),
                                                       sb[i & 1]);
                            };
                            pairw(qlo, np0, nkx_lo, ky0, 0);
                            pairw(qlo, np1, nkx_lo, ky1, 1);
                            pairw(qhi, np0, nkx_hi, ky0, 2);
                            pairw(qhi, np1, nkx_hi, ky1, 3);
                            ++kyr;
                        };
                        // The products of a window row: 4 or 8 independent accumulators between two products into
                        // one of them.  next: the weights of the following row, formed while these are in flight.
                        auto products = [&](const Frag &f, auto next) {
                            uint32_t vh[2][4], vl[2][4];
#pragma unroll
                            for (int j = 0; j < 2; ++j) {
                                ldsm_x4_t(bo[j] + f.ro, vh[j][0], vh[j][1], vh[j][2], vh[j][3]);
                                ldsm_x4_t(bo[j] + f.ro + (uint32_t)S::lo, vl[j][0], vl[j][1], vl[j][2], vl[j][3]);
                            }
                            auto pass = [&](const uint32_t (&w)[4], const uint32_t (&v)[2][4], auto &c) {
#pragma unroll
                                for (int j = 0; j < 4; ++j) mma(c[j], w, v[j >> 1][2 * (j & 1)], v[j >> 1][2 * (j & 1) + 1]);
                            };
                            next();
                            pass(f.ah, vh, acc);
                            pass(f.dh, vh, ac1);
                            pass(f.al, vh, acc);
                            pass(f.dl, vh, ac1);
                            pass(f.ah, vl, acc);
                            pass(f.dh, vl, ac1);
                        };
                        Frag f0, f1;
                        weights(f0);
#pragma unroll 2
                        for (int r = 0; r < NKS / 2 - 1; ++r) {
                            products(f0, [&] { weights(f1); });
                            products(f1, [&] { weights(f0); });
                        }
                        products(f0, [&] { weights(f1); });
                        products(f1, [] {});
                    } else {
                        // the same sums one by one from the volume, so that what is not finite reaches the
                        // pixels whose windows hold it and no others
                        const int u0 = x0 + px0 + mx, v0 = Y0 + 4 * band + my0;
#pragma unroll 1
                        for (int i = 0; i < 2 * (2 * RB + 1) * (2 * RB + 1); ++i) {
                            const int h = i & 1, k = i >> 1, dy = k / (2 * RB + 1) - RB, dx = k % (2 * RB + 1) - RB;
                            const int y = v0 + 2 * h + dy, u = u0 + dx;
                            if (u0 >= W || v0 + 2 * h >= H || y < 0 || y >= H || u < 0 || u >= W) continue;
                            const float t = img[(size_t)y * W + u] * a.kappa - (h ? ip1 : ip0);
                            const float w = ex2_approx(fmaf(-t, t, a.k0 * (float)(dx * dx + dy * dy) + (float)kWSh));
                            const __half *q = vol + ((size_t)(t4 >> 1) * HW + (size_t)y * W + u) * 8 + 2 * (t4 & 1);
#pragma unroll
                            for (int hh = 0; hh < 2; ++hh) {
                                if (h != hh) continue;
                                if (t4 == 0) sb[hh].x = fmaf(w * t, a.beta[b * HW + (size_t)y * W + u], sb[hh].x);
#pragma unroll
                                for (int n = 0; n < N / 8; ++n) {
                                    if (2 * n + (t4 >> 1) >= ng) continue;
                                    const uint32_t *z = reinterpret_cast<const uint32_t *>(q + (size_t)n * HW * 16);
                                    const float2 v = unsplit2(z[0], z[2]);
                                    acc[n][2 * hh] = fmaf(w, v.x, acc[n][2 * hh]);
                                    acc[n][2 * hh + 1] = fmaf(w, v.y, acc[n][2 * hh + 1]);
                                    ac1[n][2 * hh] = fmaf(w * t, v.x, ac1[n][2 * hh]);
                                    ac1[n][2 * hh + 1] = fmaf(w * t, v.y, ac1[n][2 * hh + 1]);
                                }
                            }
                        }
                    }
                    // lane (g, t4) holds disparities d0 + 8 n + 2 t4 + {0, 1} of pixels g and g + 8; the four
                    // lanes of a quad hold all of the same two pixels
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int u = x0 + px0 + mx, y = Y0 + 4 * band + my0 + 2 * h;
                        const bool in = u < W && y < H;
                        const size_t pix = in ? (size_t)y * W + u : 0, o = b * HW + pix;
                        const bool last = ch + 1 == nchunks;
                        const float us = pow2i(-hs) * pow2i(-kWSh);
                        float tacc = 0.f;
                        const size_t vo = ((size_t)b * D + d0 + 2 * t4) * HW + pix;
                        const float *cp = a.cost + vo;
                        float cx[N / 8][2];
#pragma unroll
                        for (int n = 0; n < N / 8; ++n)
#pragma unroll
                            for (int e = 0; e < 2; ++e)
                                cx[n][e] = in && 8 * n + 2 * t4 + e < dn ? cp[(size_t)(8 * n + e) * HW] : 0.f;
#pragma unroll
                        for (int n = 0; n < N / 8; ++n)
#pragma unroll
                            for (int e = 0; e < 2; ++e)
                                if (in && 8 * n + 2 * t4 + e < dn) {
                                    a.gc[vo + (size_t)(8 * n + e) * HW] = acc[n][2 * h + e] * us;
                                    tacc = fmaf(cx[n][e], ac1[n][2 * h + e], tacc);
                                }
                        tacc = quad_sum(tacc) * us;
                        const float sbh = quad_sum(sb[h].x + sb[h].y) * pow2i(-kWSh);
                        if (ch == 0) tacc -= sbh;
                        else if (in) tacc += a.gw[o];
                        __syncwarp();
                        if (t4 == 0 && in) a.gw[o] = last ? a.gw_scale * (a.t1[o] + tacc) : tacc;
                    }
                }
                if (p < nsteps && sr < 4 && scr >= 0) {
                    int sl = slot0 + scr - first;
                    if (sl >= RR) sl -= RR;
                    if (si != kFar) si *= a.kappa;
                    sI[sl * kSIP + sx] = si;
                    sB[sl * kSIP + sx] = sbv;
                    if (rowbad || !(fabsf(si) <= kFar && fabsf(sbv) < INFINITY)) bad[sl] = tag0 + scr;
                }
                slot0 += 4 * p - S::PHI + 4 - first;
                if (slot0 >= RR) slot0 -= RR;
                if (band >= 0) {
                    slot += 4;
                    if (slot >= RR) slot -= RR;
                }
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                __syncthreads();
            }
        }
    }
}

template <int RB>
cudaError_t launch_rb(const AggArgs &a, int B, cudaStream_t st)
{
    using S = Shape<RB>;
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_dagg_tc<RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::total);
    if (e != cudaSuccess) return e;
    // bands per segment: of all equal splits, the one whose waves (one CTA per SM) take the fewest
    // iterations
    const int strips = (a.W + 31) / 32, bands = (a.H + 3) / 4;
    int best = bands;
    long best_t = 1l << 60;
    for (int s = 1; s <= bands; ++s) {
        const int nb = (bands + s - 1) / s, segs = (bands + nb - 1) / nb;
        const long waves = ((long)strips * segs * B + 2 * nsm - 1) / (2 * nsm), t = waves * (nb + S::LEAD + 1);
        if (t < best_t) {
            best_t = t;
            best = nb;
        }
    }
    k_dagg_tc<RB><<<dim3(strips * ((bands + best - 1) / best), B), kNT, S::total, st>>>(a, best);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_dabsmax(const AggArgs &a, int B, cudaStream_t st)
{
    k_dabsmax<<<dim3(kAggRange, B), 256, 0, st>>>(a.gdisp, a.H, a.W, a.range, a.hbad);
    return cudaGetLastError();
}

cudaError_t launch_gc_tc(const AggArgs &a, int rb, int B, cudaStream_t st)
{
    switch (rb) {
    case 0: return launch_rb<0>(a, B, st);
    case 1: return launch_rb<1>(a, B, st);
    case 2: return launch_rb<2>(a, B, st);
    case 3: return launch_rb<3>(a, B, st);
    case 4: return launch_rb<4>(a, B, st);
    case 5: return launch_rb<5>(a, B, st);
    default: return launch_rb<6>(a, B, st);
    }
}

}  // namespace sgb
