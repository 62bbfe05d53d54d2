// k_unfused.cu -- the stage-per-kernel form of §3.2 with FP32 volumes in device memory:
// cost volume (eq. c), bilateral aggregation (eq. fbs), WTA + eq. (subpixel).  The volumes are
// [H][W][D] (d fastest); the cost volume reads the staging buffers of k_prep.
#include <math.h>

#include "internal.cuh"

namespace sgb {

// ------------------------------------------------------------------ cost volume
// eq. (c) for every pixel and disparity: c = 1 - (n S - S_ref S_tar) r_ref r_tar, S the exact
// integer w x w correlation sum.
//
// A thread owns one column u and four disparities and walks down kCvRows rows: the horizontal
// sum of each image row is a few dp4a on packed bytes (the target's w + 3 bytes are extracted
// once per row; the four disparities meet them with the reference window shifted by 0..3
// bytes), and the vertical window is a running sum over a ring of the last w row sums (exact
// integers).  Eight disparity quads of 32 columns per block, so a warp writes whole 128-byte
// lines of the volume.  The bound is issue: about 45 instructions per row and four outputs,
// against 4 w^2 byte loads and products per four outputs with one thread per pixel and no
// reuse.  640 x 360, D = 32, w = 9: 17.3 us (300 us with one thread per pixel).
constexpr int kCvRows = 16;      // output rows per block
constexpr int kCvCols = 32;      // output columns per block
constexpr int kCvQuads = 8;      // disparity quads per block
constexpr int kCvRefB = 48, kCvTgtB = 96;   // staged bytes per row

template <int RW>
__global__ void __launch_bounds__(kCvCols *kCvQuads)
k_cost_volume(const uint8_t *__restrict__ ref_pad, const uint8_t *__restrict__ tgt_pad,
              const int2 *__restrict__ ref_stats, const int2 *__restrict__ tgt_stats, int W, int H, int D, int n,
              int pad_left, int pad_top, int pad_w, int pad_h, int pad_pitch, float *__restrict__ cost, int vec)
{
    constexpr int WS = 2 * RW + 1;
    constexpr int NWR = (WS + 3) / 4;          // words that hold the w reference bytes
    constexpr int NWT = (WS + 3 + 3) / 4;      // words that hold the w + 3 target bytes of four disparities
    constexpr int SR = kCvRows + 2 * RW;
    constexpr uint32_t TAIL = WS % 4 ? (1u << (8 * (WS % 4))) - 1u : 0xffffffffu;
    __shared__ uint32_t sr[SR][kCvRefB / 4];
    __shared__ uint32_t st[SR][kCvTgtB / 4];
    const int tid = threadIdx.x, dq = tid % kCvQuads, ul = tid / kCvQuads;
    const int u0 = blockIdx.x * kCvCols, y0 = blockIdx.y * kCvRows, db = blockIdx.z * 4 * kCvQuads;
    // staged columns: reference from u0 - 8, target from u0 - db - 40 (both multiples of 8 from
    // the padded origin, so the words are aligned); clamped words feed only outputs that are
    // not written
    const int wpr = pad_pitch / 4;
    for (int i = tid; i < SR * (kCvRefB / 4); i += kCvCols * kCvQuads) {
        const int r = i / (kCvRefB / 4), c = i - r * (kCvRefB / 4);
        const int py = min(y0 + r + pad_top - RW, pad_h - 1), wx = min((u0 - 8 + pad_left) / 4 + c, wpr - 1);
        sr[r][c] = __ldg(reinterpret_cast<const uint32_t *>(ref_pad) + (size_t)py * wpr + wx);
    }
    for (int i = tid; i < SR * (kCvTgtB / 4); i += kCvCols * kCvQuads) {
        const int r = i / (kCvTgtB / 4), c = i - r * (kCvTgtB / 4);
        const int x = u0 - db - 40 + pad_left;
        const int py = min(y0 + r + pad_top - RW, pad_h - 1), wx = min(max((x >> 2) + c, 0), wpr - 1);
        st[r][c] = __ldg(reinterpret_cast<const uint32_t *>(tgt_pad) + (size_t)py * wpr + wx);
    }
    __syncthreads();
    const int u = u0 + ul, d0 = db + 4 * dq;
    if (u >= W || d0 >= D) return;
    const int ri = ul + 8 - RW, ti = ul - 4 * dq + 37 - RW;   // first byte of each window in the staged rows
    const int rw0 = ri >> 2, rsh = (ri & 3) * 8, tw0 = ti >> 2, tsh = (ti & 3) * 8;
    // the four horizontal sums of staged row r (h[k]: disparity d0 + 3 - k)
    auto row_sums = [&](int r, int (&h)[4]) {
        uint32_t a[NWR], b[NWT];
        {
            uint32_t q = sr[r][rw0];
#pragma unroll
            for (int i = 0; i < NWR; ++i) {
                const uint32_t q1 = sr[r][rw0 + i + 1];
                a[i] = __funnelshift_r(q, q1, rsh);
                q = q1;
            }
            a[NWR - 1] &= TAIL;
            q = st[r][tw0];
#pragma unroll
            for (int i = 0; i < NWT; ++i) {
                const uint32_t q1 = st[r][tw0 + i + 1];
                b[i] = __funnelshift_r(q, q1, tsh);
                q = q1;
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t s = 0;
#pragma unroll
            for (int i = 0; i < NWT; ++i) {
                // the reference bytes moved up by k bytes
                const uint32_t lo = i > 0 && i - 1 < NWR ? a[i - 1] : 0u, hi = i < NWR ? a[i] : 0u;
                s = __dp4a(b[i], k == 0 ? hi : __funnelshift_l(lo, hi, 8 * k), s);
            }
            h[k] = (int)s;
        }
    };
    int ring[WS][4], V[4] = {0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < WS - 1; ++j) {
        row_sums(j, ring[j]);
#pragma unroll
        for (int k = 0; k < 4; ++k) V[k] += ring[j][k];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) ring[WS - 1][k] = 0;
    const int rows = min(kCvRows, H - y0);
    const int2 *rs = ref_stats + (size_t)(y0 + pad_top) * pad_w + u + pad_left;
    const int2 *ts = tgt_stats + (size_t)(y0 + pad_top) * pad_w + u + pad_left - d0;
    float *out = cost + ((size_t)y0 * W + u) * D + d0;
    const int nd = min(4, D - d0);
    for (int yb = 0; yb < rows; yb += WS) {
#pragma unroll
        for (int j = 0; j < WS; ++j) {
            const int y = yb + j;
            if (y >= rows) break;
            // the row entering the window replaces the one that left it in the ring
            int h[4];
            row_sums(y + WS - 1, h);
            const int2 r = __ldg(rs + (size_t)y * pad_w);
            float c[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                V[k] += h[k] - ring[(j + WS - 1) % WS][k];
                ring[(j + WS - 1) % WS][k] = h[k];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                c[q] = 0.f;
                if (q < nd) {
                    const int2 t = __ldg(ts + (size_t)y * pad_w - q);
                    const int num = n * V[3 - q] - r.x * t.x;
                    c[q] = fmaf(-(float)num, __int_as_float(r.y) * __int_as_float(t.y), 1.0f);
                }
            }
            float *o = out + (size_t)y * W * D;
            if (vec) {
                *reinterpret_cast<float4 *>(o) = make_float4(c[0], c[1], c[2], c[3]);
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (q < nd) o[q] = c[q];
            }
        }
    }
}

int launch_cost_volume(stereo_ctx *ctx, float *cost, cudaStream_t s)
{
    const Geometry &g = ctx->g;
    const dim3 grid((g.W + kCvCols - 1) / kCvCols, (g.H + kCvRows - 1) / kCvRows,
                    (g.D + 4 * kCvQuads - 1) / (4 * kCvQuads));
    const int vec = g.D % 4 == 0 && ((uintptr_t)cost & 15) == 0;   // every quad of d whole and aligned
#define SGB_CV(R)                                                                                                    \
    k_cost_volume<R><<<grid, kCvCols * kCvQuads, 0, s>>>(ctx->ref_pad, ctx->tgt_pad, ctx->ref_stats, ctx->tgt_stats, \
                                                         g.W, g.H, g.D, g.n, g.pad_left, g.pad_top, g.pad_w,         \
                                                         g.pad_h, g.pad_pitch, cost, vec)
    switch (g.rw) {
    case 1: SGB_CV(1); break;
    case 2: SGB_CV(2); break;
    case 3: SGB_CV(3); break;
    case 4: SGB_CV(4); break;
    default: SGB_CV(5); break;
    }
#undef SGB_CV
    return cuda_error(cudaGetLastError(), "k_cost_volume launch");
}

// ------------------------------------------------------------------ aggregation
// eq. (fbs): E(p,d) = sum_q w(p,q) c(q,d) / sum_q w(p,q), q over the in-image part of the
// k x k window, w per eq. (omega_s) in FP32.
//
// A block takes a 32 x 16 pixel tile and 16 disparities: the costs of the tile and its halo are
// staged as four planes of disparity quads (float4), the scaled intensities beside them; a
// thread owns four pixels of a column, so each staged cost serves four weights and each weight
// 16 disparities (eight packed FMAs).  Every pixel takes its neighbours row by row, left to
// right, as the definition's double loop does, and an out-of-image neighbour has a weight of
// exactly 0 and staged costs of 0, so the sums are those of that loop bit for bit.  The bound
// is the FMA pipe: 2 k^2 flops per (p, d); one thread per pixel read every cost k^2 times
// through L1 instead.  640 x 360, D = 32, k = 11: 93 us, 19 TFLOP/s (2.95 ms).
constexpr int kAvDC = 16, kAvTX = 32, kAvTY = 16, kAvPY = 4;
constexpr int kAvThreads = 32 * kAvTY / kAvPY;
// Intensity of an out-of-image neighbour: its exponent is -infinity for every 1 / sigma1^2 > 0, so its
// weight is 0 (the intensities are staged unscaled: a finite value would count once sigma1 is as large).
constexpr float kAvFar = INFINITY;

template <int RB>
__global__ void __launch_bounds__(kAvThreads)
k_aggregate_volume(const uint8_t *__restrict__ ref, int pitch, const float *__restrict__ cost, int W, int H, int D,
                   float inv_s0sq, float inv_s1sq, float *__restrict__ agg, int vec)
{
    constexpr int TW = kAvTX + 2 * RB, TH = kAvTY + 2 * RB, NQ = kAvDC / 4;
    extern __shared__ float4 av_smem[];
    float4 *V = av_smem;                                      // [NQ][TH][TW]
    float *sI = reinterpret_cast<float *>(V + NQ * TH * TW);  // [TH][TW]
    const int x0 = blockIdx.x * kAvTX, y0 = blockIdx.y * kAvTY, d0 = blockIdx.z * kAvDC;
    const int tid = threadIdx.x;
    // staged position by position, the NQ quads of a position on neighbouring lanes (one
    // position is 64 consecutive bytes of the volume)
    for (int i = tid; i < TH * TW * NQ; i += kAvThreads) {
        const int q = i % NQ, pos = i / NQ, r = pos / TW, c = pos - r * TW;
        const int y = y0 - RB + r, x = x0 - RB + c, d = d0 + 4 * q;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (y >= 0 && y < H && x >= 0 && x < W && d < D) {
            const float *src = cost + ((size_t)y * W + x) * D + d;
            if (vec) {
                v = __ldg(reinterpret_cast<const float4 *>(src));
            } else {
                v.x = __ldg(src);
                if (d + 1 < D) v.y = __ldg(src + 1);
                if (d + 2 < D) v.z = __ldg(src + 2);
                if (d + 3 < D) v.w = __ldg(src + 3);
            }
        }
        V[(q * TH + r) * TW + c] = v;
    }
    for (int i = tid; i < TH * TW; i += kAvThreads) {
        const int r = i / TW, c = i - r * TW, y = y0 - RB + r, x = x0 - RB + c;
        sI[i] = (y >= 0 && y < H && x >= 0 && x < W) ? (float)__ldg(ref + (size_t)y * pitch + x) : kAvFar;
    }
    __syncthreads();
    const int tx = tid & 31, py0 = kAvPY * (tid >> 5);
    float sIp[kAvPY], Z[kAvPY];
    float2 acc[kAvPY][kAvDC / 2];
#pragma unroll
    for (int i = 0; i < kAvPY; ++i) {
        sIp[i] = sI[(py0 + i + RB) * TW + tx + RB];
        Z[i] = 0.f;
#pragma unroll
        for (int k = 0; k < kAvDC / 2; ++k) acc[i][k] = make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int r = 0; r < kAvPY + 2 * RB; ++r) {
#pragma unroll 1
        for (int dx = -RB; dx <= RB; ++dx) {
            const int col = tx + RB + dx;
            const float sq = sI[(py0 + r) * TW + col];
            float4 v[NQ];
#pragma unroll
            for (int q = 0; q < NQ; ++q) v[q] = V[(q * TH + py0 + r) * TW + col];
#pragma unroll
            for (int i = 0; i < kAvPY; ++i) {
                const int dy = r - i - RB;
                if (dy < -RB || dy > RB) continue;
                const float di = sIp[i] - sq;
                const float w = expf(__fmaf_rn(-(float)(dx * dx + dy * dy), inv_s0sq, -__fmul_rn(__fmul_rn(di, di), inv_s1sq)));
                Z[i] += w;
                const float2 w2 = make_float2(w, w);
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    acc[i][2 * q] = __ffma2_rn(w2, make_float2(v[q].x, v[q].y), acc[i][2 * q]);
                    acc[i][2 * q + 1] = __ffma2_rn(w2, make_float2(v[q].z, v[q].w), acc[i][2 * q + 1]);
                }
            }
        }
    }
    const int u = x0 + tx;
    if (u >= W) return;
#pragma unroll
    for (int i = 0; i < kAvPY; ++i) {
        const int v = y0 + py0 + i;
        if (v >= H) break;
        const float iz = 1.0f / Z[i];
        float *out = agg + ((size_t)v * W + u) * D + d0;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float e[4] = {acc[i][2 * q].x * iz, acc[i][2 * q].y * iz, acc[i][2 * q + 1].x * iz,
                                acc[i][2 * q + 1].y * iz};
            if (vec) {
                if (d0 + 4 * q < D) *reinterpret_cast<float4 *>(out + 4 * q) = make_float4(e[0], e[1], e[2], e[3]);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (d0 + 4 * q + k < D) out[4 * q + k] = e[k];
            }
        }
    }
}

template <int RB>
static cudaError_t launch_av(const uint8_t *ref, const Geometry &g, const float *cost, float inv_s0sq, float inv_s1sq, float *agg,
                             int vec, cudaStream_t s)
{
    const size_t smem = (size_t)(kAvTX + 2 * RB) * (kAvTY + 2 * RB) * (kAvDC + 1) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(k_aggregate_volume<RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((g.W + kAvTX - 1) / kAvTX, (g.H + kAvTY - 1) / kAvTY, (g.D + kAvDC - 1) / kAvDC);
    k_aggregate_volume<RB><<<grid, kAvThreads, smem, s>>>(ref, g.pitch, cost, g.W, g.H, g.D, inv_s0sq, inv_s1sq, agg, vec);
    return cudaGetLastError();
}

int launch_aggregate_volume(stereo_ctx *ctx, const uint8_t *ref, const float *cost, float *agg, cudaStream_t s)
{
    const Geometry &g = ctx->g;
    const float s0 = ctx->p.sigma0, s1 = ctx->p.sigma1;
    // (1 / sigma1^2 at least the smallest positive float, which leaves every weight of two pixels as it
    // is and keeps the exponent of an out-of-image neighbour from becoming 0 x infinity)
    const float i0 = 1.0f / (s0 * s0), i1 = fmaxf(1.0f / (s1 * s1), 0x1p-149f);
    const int vec = g.D % 4 == 0 && (((uintptr_t)cost | (uintptr_t)agg) & 15) == 0;
    cudaError_t e;
    switch (g.rb) {
    case 0: e = launch_av<0>(ref, g, cost, i0, i1, agg, vec, s); break;
    case 1: e = launch_av<1>(ref, g, cost, i0, i1, agg, vec, s); break;
    case 2: e = launch_av<2>(ref, g, cost, i0, i1, agg, vec, s); break;
    case 3: e = launch_av<3>(ref, g, cost, i0, i1, agg, vec, s); break;
    case 4: e = launch_av<4>(ref, g, cost, i0, i1, agg, vec, s); break;
    case 5: e = launch_av<5>(ref, g, cost, i0, i1, agg, vec, s); break;
    case 6: e = launch_av<6>(ref, g, cost, i0, i1, agg, vec, s); break;
    default: e = launch_av<7>(ref, g, cost, i0, i1, agg, vec, s); break;
    }
    return cuda_error(e, "k_aggregate_volume launch");
}

// ------------------------------------------------------------------ WTA
// WTA (lowest d wins ties) + eq. (subpixel) on E, add back s_i(v) = floor(s(v) + 0.5).
//
// Eight lanes read one pixel's row of the volume together (consecutive words, so a warp reads
// four pixels' rows as whole lines: the kernel is bound by reading the volume once; one thread
// per pixel read words D apart).  640 x 360, D = 32: 14.3 us (73 us).  Each lane keeps the lowest value of its disparities, the
// lowest index on ties, and the second lowest; NaNs are never chosen, except that a NaN at
// d = 0 stays the winner (nothing compares below it), as in a scan that starts at d = 0.
constexpr int kWvThreads = 256, kWvLanes = 8;

__global__ void __launch_bounds__(kWvThreads)
k_wta_volume(const float *__restrict__ agg, const float *__restrict__ shift, int W, int H, int D,
             float *__restrict__ disp, int32_t *__restrict__ wta, float *__restrict__ best2)
{
    const float inf = __int_as_float(0x7f800000);
    const int l = threadIdx.x % kWvLanes, v = blockIdx.y;
    const int u = blockIdx.x * (kWvThreads / kWvLanes) + threadIdx.x / kWvLanes;
    const float *e = agg + ((size_t)v * W + min(u, W - 1)) * D;
    float m = inf, s = inf;     // lowest and second lowest of this lane
    int b = D;
    for (int d = l; d < D; d += kWvLanes) {
        const float x = __ldg(e + d);
        if (x < m) {
            s = m;
            m = x;
            b = d;
        } else if (x < s) {
            s = x;
        }
    }
#pragma unroll
    for (int o = 1; o < kWvLanes; o <<= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, m, o), s2 = __shfl_xor_sync(0xffffffffu, s, o);
        const int b2 = __shfl_xor_sync(0xffffffffu, b, o);
        const bool take = m2 < m || (m2 == m && b2 < b);
        // the loser's lowest value competes for the second place
        s = fminf(fminf(s, s2), take ? m : m2);
        if (take) {
            m = m2;
            b = b2;
        }
    }
    if (l != 0 || u >= W) return;
    const float e0 = __ldg(e);
    if (b >= D || isnan(e0)) {
        // no value below +inf (d = 0 stands, and a -inf or finite value never gets here), or a
        // NaN at d = 0: every other value competes for the second place
        s = b < D ? m : inf;
        b = 0;
    }
    float delta = 0.f;
    const float eb = __ldg(e + b);
    if (b > 0 && b < D - 1) {
        const float em = __ldg(e + b - 1), ep = __ldg(e + b + 1);
        const float den = 2.f * em + 2.f * ep - 4.f * eb;
        if (den > 0.f) delta = (em - ep) / den;
    }
    const int si = (int)floor((double)shift[v] + 0.5);
    const size_t o = (size_t)v * W + u;
    disp[o] = (float)b + delta + (float)si;
    if (wta) wta[o] = b;
    if (best2) {
        best2[2 * o] = eb;
        best2[2 * o + 1] = s;
    }
}

int launch_wta_volume(stereo_ctx *ctx, const float *agg, const float *shift, float *disp,
                      int32_t *wta, float *best2, cudaStream_t s)
{
    const Geometry &g = ctx->g;
    const int per = kWvThreads / kWvLanes;
    const dim3 grid((g.W + per - 1) / per, g.H);
    k_wta_volume<<<grid, kWvThreads, 0, s>>>(agg, shift, g.W, g.H, g.D, disp, wta, best2);
    return cuda_error(cudaGetLastError(), "k_wta_volume launch");
}

}  // namespace sgb
