// k_march.cuh -- the fused step's tensor-core pass (eq. c, eq. omega_s, eq. fbs; §3.2): costs,
// bilateral aggregation and, per pixel, either the certified candidate range of the FP32 form
// (k_refine then evaluates it) or the winner of the 16-bit form.
//
// A CTA marches down a strip of 32 pixel columns, four rows (a band) per iteration, and keeps
// the 16-bit costs of the rows its bilateral window spans in a shared-memory ring, all N
// disparities of a chunk at once (the whole search range up to 128).  Producer warps compute
// the costs of the next band's four new rows while consumer warps aggregate the current band;
// one barrier per iteration separates the two.  Against 32 x 36 tiles with every warp doing
// first one and then the other, 32 disparities at a time, this
//   - computes each cost 42 / 32 times (the strip's halo) instead of 1.7 times, and its vertical
//     window sums once, without a warm-up per tile and chunk;
//   - forms every weight once per pixel pair and chunk of N, not once per 32 disparities;
//   - overlaps the two phases, where 16 barriers per chunk separated their steps;
//   - has every disparity of a pixel in the registers of one quad, so the minimum, the candidate
//     range or the winner follow without running state (one chunk);
//   - splits into as many row segments as fill the SMs, whatever the frame size.
// It is bound by shared memory and issue (FP32 form at N = 128: shared-memory pipe 71 %, issue slots 55 %,
// tensor pipe 40 %; most stalls wait for a fixed latency or the math pipes).  1920 x 1080, D = 128, w = 9, k = 11: FP16 form 1.28 -> 0.69 ms; FP32 form
// with k_refine 1.34 -> 0.83 ms (0.60 + 0.23).  D = 192, k = 13, FP16 (two passes of 96): 1.80 ->
// 1.19 ms.
//
// Producers.  The cross term S(x, d) = sum of the block's I_ref(q) I_tar(q - d) runs on the
// tensor cores: 8-bit values are exact in FP16, every product and window sum is an integer
// below 2^23, so FP32 accumulators hold them exactly.  A warp owns 16 disparities and a run of
// 8-column blocks; for every image row entering the window one mma.m16n8k16 per block (two for
// w = 11) adds the products of that row: A = the target as a 16-disparity x 16-column Toeplitz
// matrix (A(m, k) = I_tar(x + k - d - m): every fragment register is one 4-byte load, and
// neighbouring blocks share all but one of them), B = the reference banded to each column's
// window.  The row that leaves is subtracted the same way.  Then c = 1 - (n S - S_r S_t) r_r r_t
// in the integers and roundings of cost_chunk, rounded once to the 16-bit type (times 2^8), and
// stmatrix transposes the fragments into the ring (d contiguous).
//
// Consumers.  A warp owns a 4 x 4 pixel patch: E(p, d) = sum_q w(p, q) c(q, d) as one k-step per
// window row (K = the 4 + 2 RB columns the patch's windows span, padded to 16 with zero weights),
// N / 8 mma per step, with w16 = RN16(2^12 w32) formed in FP32 from k_fused's own exponent.
// Patches, k-steps and roundings do not depend on N, the strip or the segment.
//
// Screening bound (FP32 form).  Every weight and cost is non-negative and each is rounded once
// to FP16 (relative error 2^-11 in the normal range), so for every (p, d)
//     |E16 - 2^20 E32| <= eps 2^20 E32 + a,
// where E32 is k_fused's FP32 sum: eps covers the two FP16 roundings of each product (2^-10),
// the tensor core's FP32 accumulation (at most 17 terms per k-step and 16 k-steps at bil = 13,
// each addition within 2^-23 of the running sum, truncating or rounding: 3.3e-5), k_fused's own
// chain of at most 169 FMAs (1.0e-5) and the ex2 / exponent roundings of the scaled weight
// (1e-5): 1.03e-3, taken as 1.1e-3; a (64, i.e. 6.1e-5 unscaled) covers FP16 subnormal weights
// and costs even if the tensor core flushed them.  Hence the FP32 argmin d* (lowest d on ties)
// satisfies E16(d*) <= thr(min_d E16) = (min_d E16 + a) (1 + eps) / (1 - eps) + a, and so does
// every d that ties it.  Each pixel's range [dlo, dhi] holds every d with E16(d) <= thr(minimum);
// over several chunks, a chunk whose minimum m makes thr(m) smaller than the previous minimum
// drops the earlier range (none of its disparities can satisfy the final test).
#pragma once
#include "k_fused_tc.cuh"
#include "k_sc_refine.cuh"

namespace sgb {

// MODE: kMarchScreen (FP32 storage: candidate ranges for k_refine), kMarchRefine (FP32 storage,
// ranges of at most 32 on small frames: screening and refinement, the step's outputs; the FP32 costs of the window
// stay in a second ring), kMarchPlain (FP16 / BF16 storage: the running WTA on the 16-bit sums and
// the step's outputs).
constexpr int kMarchScreen = 0, kMarchRefine = 1, kMarchPlain = 2;
constexpr int kMarchUnroll = 16;
constexpr int kMarchRows = 2;
constexpr int kMarchCW = 8;         // consumer warps: the eight patches of a band
constexpr int kMarchRW = 8;         // refiner warps: four for the rows of a band, four for its ambiguous pixels
constexpr int kMarchSI = 48;        // row length of the intensity ring (>= 28 + 16) and of the FP32 ring's planes
constexpr int kMarchRefB = 96;      // staged reference bytes per image row
constexpr int kMarchRefW = 40;      // words of FP16 pairs per reference row

template <int RB, int N>
struct MarchShape {
    static constexpr int QW = 32 + 2 * RB;              // cost columns
    static constexpr int XB = (QW + 7) / 8;             // 8-column blocks
    static constexpr int RR = 8 + 2 * RB;               // ring rows: a band's window and the four rows being produced
    static constexpr int XH = N >= 96 ? 1 : 2;          // column parts, one producer warp each
    static constexpr int XBW = (XB + XH - 1) / XH;      // blocks per producer warp
    static constexpr int PW = (N / 16) * XH;            // producer warps: 4, 8, 6, 8 for N = 32, 64, 96, 128
    static constexpr int PT = 32 * PW;
    static constexpr int RS = RR + 4;                   // rows of the intensity ring and of the FP32 ring
    __host__ __device__ static constexpr int threads(int mode)
    {
        return PT + 32 * (kMarchCW + (mode == kMarchRefine ? kMarchRW : 0));
    }
    static constexpr int ROWB = QW * N * 2;             // bytes of a ring row
    static constexpr int TW = N <= 64 ? 80 : 112;       // words per target copy (16 mod 32: the copies' banks differ)
    static constexpr int SR = 8 * XH * XBW;             // reference statistics per row
    static constexpr int ST = N + SR;                   // target statistics per row
    // words of a target row that the fragments of ks k-steps read
    __host__ __device__ static constexpr int tgt_words(int ks) { return 4 * (XH * XBW - 1) + 8 * ks + N / 2 + 3; }
    // staged target bytes per row (a start off 16 bytes included), a multiple of 16
    __host__ __device__ static constexpr int tgt_bytes(int ks) { return (15 + 2 * tgt_words(ks) + 1 + 15) / 16 * 16; }
};

__host__ __device__ constexpr int march_ks(int rw) { return rw <= 4 ? 1 : 2; }     // 8 + 2 rw columns in 16s

// Shared memory (offsets from the 128-byte aligned dynamic base):
//   ring   [RR][QW][N] 16-bit costs, 16-byte units swizzled by the column (march_swz)
//   sI     [RS][kMarchSI] f32 scaled reference intensities of the cost positions (1e18 outside)
//   tgt    [IR][2][TW] FP16 pairs of target rows: (2w, 2w+1) and (2w+1, 2w+2), so that a pair at
//          any column is one word; IR = 2 rw + 5 rows (a window, the row leaving it, three more)
//   ref    [IR][kMarchRefW] FP16 pairs of reference rows
//   raw    [2][4][kMarchRefB + tgt_bytes] staged bytes of four image rows (bulk copies)
//   srs, sts  window statistics of the four cost rows of a step (the reference's reciprocal times 2^8)
//   sky    [4 + 2 RB + 2] row terms of the spatial exponent, (nKy(j), nKy(j - 2))
//   dummy  16 bytes: where stmatrix puts the columns past QW
// and for the refinement (kMarchRefine):
//   sK     [2 RB + 1][march_kw(RB)] f32 the spatial exponents, one window column per row
//   cand   [2][4][32] the candidates of a band's pixels, double-buffered
//   amb    the band's ambiguous pixels: AmbList
//   r32    [RS][N][kMarchSI] f32 the costs times 2^8
struct AmbList {
    unsigned long long key[128];     // the winner so far: ordered bits of E, then d
    uint16_t first[129];             // the first evaluation unit of each listed pixel; the total at the end
    uint8_t pix[128], lo[128];       // the pixel, the lowest disparity to evaluate
    uint8_t hi[128], split[128];     // the highest; the other candidate where only two, far apart (or 255)
    int nw[4], uw[4];                // pixels and units of each row
};
struct MarchLayout {
    size_t ring, sI, tgt, ref, raw, srs, sts, sky, dummy, sK, cand, amb, r32, total;
};
__host__ __device__ constexpr int march_kw(int rb) { return (2 * rb + 1 + 3) / 4 * 4; }
template <int RB, int N>
__host__ __device__ inline MarchLayout march_layout(int rw, int mode)
{
    using S = MarchShape<RB, N>;
    const int ir = 2 * rw + 5;
    MarchLayout L;
    L.ring = 0;
    L.sI = align_up((size_t)S::RR * S::ROWB, 128);
    L.tgt = L.sI + (size_t)S::RS * kMarchSI * 4;
    L.ref = L.tgt + (size_t)ir * 2 * S::TW * 4;
    L.raw = align_up(L.ref + (size_t)ir * kMarchRefW * 4, 128);
    L.srs = align_up(L.raw + (size_t)8 * (kMarchRefB + S::tgt_bytes(march_ks(rw))), 16);
    L.sts = L.srs + (size_t)4 * S::SR * 8;
    L.sky = L.sts + (size_t)4 * S::ST * 8;
    L.dummy = align_up(L.sky + (size_t)(4 + 2 * RB + 2) * 8, 16);
    L.sK = L.cand = L.amb = L.r32 = L.dummy + 16;
    if (mode == kMarchRefine) {
        L.cand = L.sK + (size_t)(2 * RB + 1) * march_kw(RB) * 4;
        L.amb = align_up(L.cand + 2 * 128 * 4, 8);
        L.r32 = align_up(L.amb + sizeof(AmbList), 128);
        L.total = L.r32 + (size_t)S::RS * N * kMarchSI * 4;
    } else {
        L.total = align_up(L.r32, 128);
    }
    return L;
}

// The 16-byte unit of disparities [8 unit, 8 unit + 8) of column x sits at unit ^ swz(x): eight
// consecutive columns of one unit (a fragment's rows) then meet eight distinct bank groups.
template <int N>
__device__ __forceinline__ int march_swz(int x)
{
    return N % 64 == 0 ? (x & 7) : ((x >> 1) & 3);
}

template <typename T> __device__ __forceinline__ uint32_t pack_rn(float lo, float hi);
template <> __device__ __forceinline__ uint32_t pack_rn<__half>(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
template <> __device__ __forceinline__ uint32_t pack_rn<__nv_bfloat16>(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// (No memory clobber: only ldmatrix reads these bytes, behind a barrier, so the loads of other
// shared data may move across.)
__device__ __forceinline__ void stsm_x4_t(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r0), "r"(r1),
                 "r"(r2), "r"(r3));
}
__device__ __forceinline__ void stsm_x2_t(uint32_t addr, uint32_t r0, uint32_t r1)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1, %2};" ::"r"(addr), "r"(r0), "r"(r1));
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

// v[i] for a run-time i < M by a tree of selects (M values in registers).
template <int M>
__device__ __forceinline__ float pick_reg(const float (&v)[M], int i)
{
    if constexpr (M == 1) {
        return v[0];
    } else {
        float t[(M + 1) / 2];
#pragma unroll
        for (int k = 0; k < (M + 1) / 2; ++k) t[k] = 2 * k + 1 < M ? ((i & 1) ? v[2 * k + 1] : v[2 * k]) : v[2 * k];
        return pick_reg(t, i >> 1);
    }
}

// k_fused's FP32 sums of three disparities d, d + 1, d + 2 (past the range: the range's last) of one
// pixel: terms in k_fused's order, window column outer, row inner.  so[]: offsets of the window's
// rows in the intensity ring; ring32, sI, sK as in the layout; x the pixel's column in the strip.
// (The costs are k_fused's times 2^8, and so is every sum: the same bits but for the exponent.)
template <int RB, int N>
__device__ __forceinline__ void march_eval3(const float *ring32, const float *sI, const float *sK, const uint32_t (&so)[2 * RB + 1],
                                            int x, int d, float &e0, float &e1, float &e2)
{
    constexpr int KB = 2 * RB + 1, KW = march_kw(RB);
    const float ip = sI[so[RB] + x + RB];
    const float *p0 = ring32 + min(d, N - 1) * kMarchSI + x;
    const float *p1 = ring32 + min(d + 1, N - 1) * kMarchSI + x, *p2 = ring32 + min(d + 2, N - 1) * kMarchSI + x;
    e0 = e1 = e2 = 0.f;
#pragma unroll 1
    for (int dx = 0; dx < KB; ++dx) {
        float kr[KW];
#pragma unroll
        for (int k = 0; k < KW / 4; ++k) {
            const float4 q = *reinterpret_cast<const float4 *>(sK + dx * KW + 4 * k);
            kr[4 * k] = q.x;
            kr[4 * k + 1] = q.y;
            kr[4 * k + 2] = q.z;
            kr[4 * k + 3] = q.w;
        }
        float iq[KB], c0[KB], c1[KB], c2[KB];
#pragma unroll
        for (int j = 0; j < KB; ++j) {
            iq[j] = sI[so[j] + x + dx];
            c0[j] = p0[so[j] * N + dx];
            c1[j] = p1[so[j] * N + dx];
            c2[j] = p2[so[j] * N + dx];
        }
#pragma unroll
        for (int j = 0; j < KB; ++j) {
            const float t = iq[j] - ip;
            const float w = ex2_approx(fmaf(-t, t, kr[j]));
            e0 = fmaf(w, c0[j], e0);
            e1 = fmaf(w, c1[j], e1);
            e2 = fmaf(w, c2[j], e2);
        }
    }
}

// The end of a CTA that gave up on a copy: no copy may land after it, so the row groups g0 and g1 (of
// `end`) that it has in flight are waited for, with a limit too.  (A call: inlined, its registers cost
// the loop of some instantiations up to 3 %.)
static __device__ __noinline__ void march_drain(uint64_t *bar, int g0, int g1, int end, bool stall)
{
    if (g0 < end) mbar_wait_limited(bar + (g0 & 1), (uint32_t)(g0 >> 1) & 1u, stall);
    if (g1 < end) mbar_wait_limited(bar + (g1 & 1), (uint32_t)(g1 >> 1) & 1u, stall);
}

// One CTA per work item: item blockIdx.x of one frame's strips and segments, or of a batch's list.
template <int RB, int N, int MODE, typename T>
__global__ void __launch_bounds__((MarchShape<RB, N>::threads(MODE)), march_ctas(N, MODE != kMarchPlain))
k_march(const __grid_constant__ PairDesc single, const PairDesc *__restrict__ pairs,
        const MarchItem *__restrict__ items, int bands_per_item, int dlo, int dhi)
{
    using S = MarchShape<RB, N>;
    using X = TcOps<T>;
    constexpr int QW = S::QW, RR = S::RR, RS = S::RS, XBW = S::XBW, TW = S::TW, NKS = 4 + 2 * RB, KB = 2 * RB + 1;
    constexpr bool REF = MODE == kMarchRefine;
    constexpr int NT = S::threads(MODE);
    constexpr int TAIL = REF ? 2 : 1;              // iterations after the last step: the last band's aggregation, refinement
    static_assert(8 * S::XH * XBW <= kMarchSI, "the FP32 ring's planes hold every column block");
    static_assert(RB <= kScMaxRB && NKS <= 16, "a window row spans at most 16 columns");
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(16) FusedArgs s_args;
    __shared__ __align__(8) uint64_t s_bar[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t4 = lane & 3;
    MarchItem it0;
    if (items) {
        it0 = items[blockIdx.x];
    } else {
        const int strips = (single.a.W + 31) / 32;
        it0.pair = 0;
        it0.strip = blockIdx.x % strips;
        it0.b0 = (blockIdx.x / strips) * bands_per_item;
        it0.nb = min(bands_per_item, (single.a.H + 3) / 4 - it0.b0);
    }
    {
        const int *src = reinterpret_cast<const int *>(items ? &pairs[it0.pair].a : &single.a);
        int *dst = reinterpret_cast<int *>(&s_args);
        for (int i = tid; i < (int)(sizeof(FusedArgs) / 4); i += NT) dst[i] = src[i];
    }
    if (tid == 0) {
        mbar_init(&s_bar[0], 1);
        mbar_init(&s_bar[1], 1);
    }
    __syncthreads();
    const FusedArgs &a = s_args;
    const int rw = a.rw, m = RB + rw, IR = 2 * rw + 5, ks = march_ks(rw);
    const MarchLayout L = march_layout<RB, N>(rw, MODE);
    const int x0 = 32 * it0.strip, Y0 = 4 * it0.b0, nb = it0.nb;
    const int phi = march_phi(m), lead = march_lead(m), nsteps = nb + lead;
    const int KT = 4 * nb + 2 * m;                 // image rows of the segment, from image row Y0 - m
    float *sI = reinterpret_cast<float *>(smem + L.sI);
    float2 *sky = reinterpret_cast<float2 *>(smem + L.sky);
    float *sK = reinterpret_cast<float *>(smem + L.sK), *ring32 = reinterpret_cast<float *>(smem + L.r32);
    int *scand = reinterpret_cast<int *>(smem + L.cand);
    // spatial exponents, separable: -(K[dx][dy] + 12) = nKx(dx) + nKy(dy) with
    // nKx(i) = -(K[i][RB] + 12) and nKy(j) = -K[RB][j] (1e30 outside the window: weight 0).
    // The row terms as a table over j = r - my (the lane's first pixel row): (nKy(j), nKy(j - 2))
    auto nky = [&](int j) { return (j >= 0 && j <= 2 * RB) ? -a.K[RB * KB + j] : 1e30f; };
    for (int j = tid; j < NKS + 2; j += NT) sky[j] = make_float2(nky(j - 1), nky(j - 3));
    for (int i = tid; i < RS * kMarchSI; i += NT) sI[i] = 1e18f;   // (the columns past QW stay)
    if constexpr (REF)
        for (int i = tid; i < KB * march_kw(RB); i += NT) {
            const int dx = i / march_kw(RB), dy = i - dx * march_kw(RB);
            sK[i] = dy < KB ? a.K[dx * KB + dy] : 0.f;
        }
    const int nchunks = REF ? 1 : (min(a.D, dhi) - dlo + N - 1) / N;
    int gbase = 0;                                 // row groups staged by earlier chunks (barrier phases)
    __syncthreads();

    for (int ch = 0; ch < nchunks; ++ch, gbase += nsteps) {
        const int d0 = dlo + ch * N;
        if (warp < S::PW) {
            // ------------------------------------------------------------------ producers
            const int db = warp % (N / 16), xb0 = (warp / (N / 16)) * XBW;
            const int tbw = S::tgt_bytes(ks), rowb = kMarchRefB + tbw;
            uint8_t *raw = smem + L.raw;
            uint32_t *tw = reinterpret_cast<uint32_t *>(smem + L.tgt), *rfw = reinterpret_cast<uint32_t *>(smem + L.ref);
            int2 *srs = reinterpret_cast<int2 *>(smem + L.srs), *sts = reinterpret_cast<int2 *>(smem + L.sts);
            // staged columns: the reference from x0 - m, the target from x0 - m - (d0 + N - 1)
            const int rcol = x0 + a.pad_left - m, tcol = rcol - (d0 + N - 1);
            const int re = rcol & 15, te = tcol & 15;
            // the copies of row group gi (image rows 4 gi - phi + i inside the segment)
            auto issue = [&](int gi) {
                if (gi >= nsteps) return;
                const int k0 = max(0, 4 * gi - phi), k1 = min(KT, 4 * gi - phi + 4);
                uint64_t *bar = &s_bar[(gbase + gi) & 1];
                uint8_t *dst = raw + ((gbase + gi) & 1) * 4 * rowb;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_expect_tx(bar, (uint32_t)((k1 - k0) * rowb));
                if (a.stall_test) return;
                for (int k = k0; k < k1; ++k) {
                    const size_t row = (size_t)(Y0 - m + k + a.pad_top) * a.pad_pitch;
                    uint8_t *q = dst + (k - (4 * gi - phi)) * rowb;
                    bulk_load(q, a.ref_pad + row + (rcol - re), kMarchRefB, bar);
                    bulk_load(q + kMarchRefB, a.tgt_pad + row + (tcol - te), (uint32_t)tbw, bar);
                }
            };
            // The staging of a step's four rows: PT / 4 threads per row, thread lc of row lr.
            constexpr int LT = S::PT / 4;
            const int lr = tid / LT, lc = tid - lr * LT;
            // window statistics of the four cost rows of a step, one step ahead in registers
            constexpr int NST = (S::SR + S::ST + LT - 1) / LT;
            int2 stv[NST];
            auto load_stats = [&](int p) {
                const int cr = 4 * p - phi - 2 * rw + lr;
                const bool ok = cr >= 0 && p < nsteps;
                const size_t o = (size_t)(Y0 - RB + (ok ? cr : 0) + a.pad_top) * a.pad_w + x0 - RB + a.pad_left;
                const int2 *rs = a.ref_stats + o, *ts = a.tgt_stats + o - d0 - (N - 1) - S::SR;
#pragma unroll
                for (int k = 0; k < NST; ++k) {
                    const int c = lc + k * LT;
                    stv[k] = make_int2(0, 0);
                    if (ok && c < S::SR + S::ST) stv[k] = __ldg((c < S::SR ? rs : ts) + c);
                }
            };
            if (tid == 0) {
                issue(0);
                issue(1);
            }
            load_stats(0);
            // fragment constants: B's band masks (columns k = 2 t4 + {0, 1} + 8 j of output column
            // g: inside the window where 0 <= k - g <= 2 rw)
            uint32_t bm[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int k = 2 * t4 + 8 * j - g;
                bm[j] = ((k >= 0 && k <= 2 * rw) ? 0x0000ffffu : 0u) | ((k + 1 >= 0 && k + 1 <= 2 * rw) ? 0xffff0000u : 0u);
            }
            // the target pair of (disparity row g, column 2 t4) of block 0: column 2 t4 - 16 db - g + N - 1
            const int tq = N - 1 - g;
            const int tl = (tq & 1) * TW + 4 * xb0 - 8 * db + t4 + (tq >> 1) - 4;
            const int rl = 4 * xb0 + t4;
            float acc[XBW][4];
            // (from 2^23 up: the sums are whole numbers below 2^23, so the low mantissa bits of an
            // accumulator are the sum itself)
#pragma unroll
            for (int x = 0; x < XBW; ++x)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[x][k] = 8388608.f;
            auto add_part = [&](int slot, uint32_t sign, int q) {
                const uint32_t *ta = tw + slot * 2 * TW + tl + 8 * q, *rb = rfw + slot * kMarchRefW + rl + 8 * q;
                const uint32_t m0 = q ? bm[2] : bm[0], m1 = q ? bm[3] : bm[1];
                uint32_t A[XBW + 2], B[XBW + 1];
#pragma unroll
                for (int j = 0; j < XBW + 2; ++j) A[j] = ta[4 * j];
#pragma unroll
                for (int j = 0; j < XBW + 1; ++j) B[j] = rb[4 * j];
#pragma unroll
                for (int x = 0; x < XBW; ++x) {
                    const uint32_t af[4] = {A[x + 1], A[x], A[x + 2], A[x + 1]};
                    mma_f16_16816(acc[x], af, (B[x] & m0) ^ sign, (B[x + 1] & m1) ^ sign);
                }
            };
            auto add_row = [&](int slot, uint32_t sign) {
                add_part(slot, sign, 0);
                if (ks > 1) add_part(slot, sign, 1);
            };
            // stmatrix rows: lane (8 i + r) names column 8 (x + (i >> 1)) + r, unit 2 db + (i & 1)
            const uint32_t ringa = smem_addr(smem + L.ring), dummy = smem_addr(smem + L.dummy);
            constexpr int NP2 = (XBW + 1) / 2;
            uint32_t so[NP2];      // offset in a ring row, or ~0 for a column past QW
#pragma unroll
            for (int j = 0; j < NP2; ++j) {
                const int xq = 8 * (xb0 + 2 * j + (lane >> 4)) + (lane & 7);
                so[j] = xq < QW ? (uint32_t)(xq * N * 2 + (((2 * db + ((lane >> 3) & 1)) ^ march_swz<N>(xq)) << 4)) : 0xffffffffu;
            }
            float *r32 = ring32 + (16 * db + g) * kMarchSI + 8 * xb0 + 2 * t4;
            const int an = a.n, kn = -an * 0x4B000000;   // n (S + 2^23 as float bits) + kn = n S (mod 2^32)
            // image row k sits in slot k mod IR; cost row cr in ring slot cr mod RR
            int kslot = 0, cslot = 0, islot = 0;   // (islot: the intensity and FP32 rings' slot of cost row cr)
            for (int p = 0; p < nsteps + TAIL; ++p) {
                int bad = 0;
                if (p < nsteps) {
                    // ---- the step's rows: wait for their bytes, widen them, store the statistics
                    uint64_t *bar = &s_bar[(gbase + p) & 1];
                    const uint32_t parity = (uint32_t)((gbase + p) >> 1) & 1u;
                    if (!mbar_try_wait(bar, parity)) {
                        // bounded as in stage_images: a fail-safe that sets the status word
                        const long long limit = a.stall_test ? (1ll << 21) : (1ll << 31), t0 = clock64();
                        bool ok = false;
                        while (!(ok = mbar_try_wait(bar, parity)) && clock64() - t0 < limit) {
                        }
                        if (!ok) {
                            bad = 1;
                            atomicOr(a.status, 1);
                        }
                    }
                    {
                        const uint8_t *rp = raw + (((gbase + p) & 1) * 4 + lr) * rowb;
                        const int k = 4 * p - phi + lr, nwt = S::tgt_words(ks);
                        int slot = kslot + k - max(0, 4 * p - phi);
                        if (slot >= IR) slot -= IR;
                        constexpr int NW = (kMarchRefW + S::tgt_words(2) + LT - 1) / LT;
#pragma unroll
                        for (int j = 0; j < NW; ++j) {
                            const int c = lc + j * LT;
                            if (k < 0 || c >= kMarchRefW + nwt) break;
                            if (c < kMarchRefW) {
                                rfw[slot * kMarchRefW + c] = u8pair_h2(rp + re + 2 * c);
                            } else {
                                const uint8_t *b = rp + kMarchRefB + te + 2 * (c - kMarchRefW);
                                uint32_t *o = tw + slot * 2 * TW + c - kMarchRefW;
                                o[0] = u8pair_h2(b);
                                o[TW] = u8pair_h2(b + 1);
                            }
                        }
                    }
#pragma unroll
                    for (int k = 0; k < NST; ++k) {
                        const int c = lc + k * LT;
                        if (c < S::SR)
                            srs[lr * S::SR + c] = make_int2(stv[k].x, __float_as_int(__int_as_float(stv[k].y) * (float)(1 << kScCSh)));
                        else if (c < S::SR + S::ST)
                            sts[lr * S::ST + c - S::SR] = stv[k];
                    }
                    asm volatile("bar.sync 1, %0;" ::"n"(S::PT) : "memory");
                    // (the bytes of group p have been read; after an expired wait the barrier's phase is
                    // still open and must not be armed again: the CTA returns at the end of this step)
                    if (tid == 0 && !bad) issue(p + 2);
                    load_stats(p + 1);
                    // intensities of the step's cost rows: image row cr + rw of the segment
                    {
                        const int cr = 4 * p - phi - 2 * rw + lr;
                        int slot = islot + cr - max(0, 4 * p - phi - 2 * rw);
                        if (slot >= RS) slot -= RS;
                        int ksl = kslot + cr + rw - max(0, 4 * p - phi);
                        if (ksl < 0) ksl += IR;
                        if (ksl >= IR) ksl -= IR;
                        const int iy = Y0 - RB + cr;
#pragma unroll
                        for (int j = 0; j < (QW + LT - 1) / LT; ++j) {
                            const int c = lc + j * LT, ix = x0 - RB + c;
                            if (cr < 0 || c >= QW) break;
                            float v = 1e18f;
                            if (ix >= 0 && ix < a.W && iy >= 0 && iy < a.H)
                                v = __half2float(reinterpret_cast<const __half *>(rfw)[ksl * 2 * kMarchRefW + c + rw]) * a.iscale;
                            sI[slot * kMarchSI + c] = v;
                        }
                    }
                    // ---- the rows of the step
#pragma unroll kMarchRows
                    for (int i = 0; i < 4; ++i) {
                        const int k = 4 * p - phi + i, cr = k - 2 * rw;
                        if (k < 0) continue;
                        add_row(kslot, 0u);
                        if (k > 2 * rw) add_row(kslot + (kslot >= 2 * rw + 1 ? -(2 * rw + 1) : IR - (2 * rw + 1)), 0x80008000u);
                        if (++kslot == IR) kslot = 0;
                        if (cr < 0) continue;
                        const int2 *rsr = srs + i * S::SR + 8 * xb0 + 2 * t4;
                        const int2 *tsr = sts + i * S::ST + 8 * xb0 + 2 * t4 - 16 * db - g + N - 1 - 8;
                        int2 u0 = tsr[0], u1 = tsr[1];
                        const uint32_t rowa = ringa + (uint32_t)(cslot * S::ROWB);
                        uint32_t h[2 * NP2][2];
#pragma unroll
                        for (int x = 0; x < XBW; ++x) {
                            const int4 r = *reinterpret_cast<const int4 *>(rsr + 8 * x);   // columns 2 t4, 2 t4 + 1
                            const int2 v0 = tsr[8 * x + 8], v1 = tsr[8 * x + 9];
                            auto cost = [&](float s, int sr, float ir, int2 t) {
                                const int num = an * __float_as_int(s) + (kn - sr * t.x);
                                return fmaf(-(float)num, ir * __int_as_float(t.y), (float)(1 << kScCSh));
                            };
                            const float ir0 = __int_as_float(r.y), ir1 = __int_as_float(r.w);
                            const float c0 = cost(acc[x][0], r.x, ir0, v0), c1 = cost(acc[x][1], r.z, ir1, v1);
                            const float c2 = cost(acc[x][2], r.x, ir0, u0), c3 = cost(acc[x][3], r.z, ir1, u1);
                            h[x][0] = pack_rn<T>(c0, c1);
                            h[x][1] = pack_rn<T>(c2, c3);
                            if constexpr (REF) {
                                // columns 2 t4, 2 t4 + 1 of disparities g and g + 8
                                float *o = r32 + islot * (N * kMarchSI) + 8 * x;
                                *reinterpret_cast<float2 *>(o) = make_float2(c0, c1);
                                *reinterpret_cast<float2 *>(o + 8 * kMarchSI) = make_float2(c2, c3);
                            }
                            u0 = v0;
                            u1 = v1;
                        }
#pragma unroll
                        for (int j = 0; j < XBW / 2; ++j)
                            stsm_x4_t(so[j] == 0xffffffffu ? dummy : rowa + so[j], h[2 * j][0], h[2 * j][1], h[2 * j + 1][0],
                                      h[2 * j + 1][1]);
                        if constexpr (XBW % 2)
                            stsm_x2_t(so[NP2 - 1] == 0xffffffffu ? dummy : rowa + so[NP2 - 1], h[XBW - 1][0], h[XBW - 1][1]);
                        if (++cslot == RR) cslot = 0;
                        if (++islot == RS) islot = 0;
                    }
                }
                if (__syncthreads_or(bad)) {
                    // thread 0 has armed the next group, and this one or, had it landed, its successor
                    if (tid == 0) march_drain(s_bar, gbase + p + 1, gbase + p + (bad ? 0 : 2), gbase + nsteps, a.stall_test != 0);
                    return;
                }
            }
        } else if (!REF || warp < S::PW + kMarchCW) {
            // ------------------------------------------------------------------ consumers
            const int px0 = 4 * (warp - S::PW), mx = g & 3, my0 = g >> 2;
            auto nkx = [&](int col) {
                const int i = col - mx;
                return (i >= 0 && i <= 2 * RB) ? -(a.K[i * KB + RB] + (float)kScWSh) : 1e30f;
            };
            // this lane's column terms: columns 2 t4 + {0, 1} and 2 t4 + {8, 9} of a window row
            const float2 nkx_lo = make_float2(nkx(2 * t4), nkx(2 * t4 + 1));
            const float2 nkx_hi = make_float2(nkx(2 * t4 + 8), nkx(2 * t4 + 9));
            // ldmatrix rows: lanes 8i..8i+7 name matrix i = (k half, unit): k slots 0..7 / 8..15 of
            // the window row, 8-disparity units 2j + (lane >> 4); padding slots (zero weight) read a
            // valid cost
            constexpr int JP = N % 64 == 0 ? 4 : 2;       // the swizzle repeats every JP unit pairs
            const int xq = min(px0 + ((lane >> 3) & 1) * 8 + (lane & 7), QW - 1);
            uint32_t bo[JP];
#pragma unroll
            for (int j = 0; j < JP; ++j)
                bo[j] = smem_addr(smem + L.ring) + (uint32_t)(xq * N * 2 + (((2 * j + (lane >> 4)) ^ march_swz<N>(xq)) << 4));
            for (int p = 0; p < nsteps + TAIL; ++p) {
                const int b = p - lead - 1;
                if (b >= 0 && b < nb) {
                    int slot = (4 * b) % RR, isl = (4 * b) % RS;   // of the band's first window row
                    const int sc = (isl + RB + my0) % RS, sc2 = (isl + RB + my0 + 2) % RS;
                    const float ip0 = sI[sc * kMarchSI + px0 + RB + mx], ip1 = sI[sc2 * kMarchSI + px0 + RB + mx];
                    const float2 nip0 = make_float2(-ip0, -ip0), nip1 = make_float2(-ip1, -ip1);
                    float acc[N / 8][4];
#pragma unroll
                    for (int nbk = 0; nbk < N / 8; ++nbk)
#pragma unroll
                        for (int k = 0; k < 4; ++k) acc[nbk][k] = 0.f;
#pragma unroll kMarchUnroll
                    for (int r = 0; r < NKS; ++r) {
                        const float *irow = sI + isl * kMarchSI + px0 + 2 * t4;
                        const float2 qlo = *reinterpret_cast<const float2 *>(irow);
                        const float2 qhi = *reinterpret_cast<const float2 *>(irow + 8);
                        const float2 ky = sky[r - my0 + 1];   // (nKy(r - my0), nKy(r - my0 - 2))
                        const uint32_t ro = (uint32_t)(slot * S::ROWB);
                        if (++slot == RR) slot = 0;
                        if (++isl == RS) isl = 0;
                        // t = I_q - I_p; e' = t^2 - (K + 12); w16 = RN16(2^-e')
                        const float2 ta = __fadd2_rn(qlo, nip0), tb = __fadd2_rn(qlo, nip1);
                        const float2 tc = __fadd2_rn(qhi, nip0), td = __fadd2_rn(qhi, nip1);
                        const float2 ea = __fadd2_rn(__ffma2_rn(ta, ta, nkx_lo), make_float2(ky.x, ky.x));
                        const float2 eb = __fadd2_rn(__ffma2_rn(tb, tb, nkx_lo), make_float2(ky.y, ky.y));
                        const float2 ec = __fadd2_rn(__ffma2_rn(tc, tc, nkx_hi), make_float2(ky.x, ky.x));
                        const float2 ed = __fadd2_rn(__ffma2_rn(td, td, nkx_hi), make_float2(ky.y, ky.y));
                        uint32_t af[4];
                        af[0] = pack_rn<T>(ex2_approx(-ea.x), ex2_approx(-ea.y));
                        af[1] = pack_rn<T>(ex2_approx(-eb.x), ex2_approx(-eb.y));
                        af[2] = pack_rn<T>(ex2_approx(-ec.x), ex2_approx(-ec.y));
                        af[3] = pack_rn<T>(ex2_approx(-ed.x), ex2_approx(-ed.y));
#pragma unroll
                        for (int j = 0; j < N / 16; ++j) {
                            uint32_t b0, b1, b2, b3;
                            ldsm_x4_t(bo[j % JP] + ro + (uint32_t)((j / JP) * JP * 32), b0, b1, b2, b3);
                            X::mma(acc[2 * j], af, b0, b1);
                            X::mma(acc[2 * j + 1], af, b2, b3);
                        }
                    }
                    // lane (g, t4) holds disparities d0 + 8 nbk + 2 t4 + {0, 1} of pixels g and g + 8; the
                    // four lanes of a quad hold all N disparities of the same two pixels
                    const int dn = a.D - d0;              // valid disparities from d0 (may exceed N)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        constexpr int M = N / 4;
                        const float inf = __int_as_float(0x7f800000);
                        float v[M];
#pragma unroll
                        for (int nbk = 0; nbk < N / 8; ++nbk) {
                            v[2 * nbk] = acc[nbk][2 * h];
                            v[2 * nbk + 1] = acc[nbk][2 * h + 1];
                        }
                        if (dn < N) {                     // past the search range
#pragma unroll
                            for (int nbk = 0; nbk < N / 8; ++nbk) {
                                if (8 * nbk + 2 * t4 >= dn) v[2 * nbk] = inf;
                                if (8 * nbk + 2 * t4 + 1 >= dn) v[2 * nbk + 1] = inf;
                            }
                        }
                        float cm = v[0];
#pragma unroll
                        for (int j = 1; j < M; ++j) cm = fminf(cm, v[j]);
                        cm = fminf(cm, __shfl_xor_sync(0xffffffffu, cm, 1));
                        cm = fminf(cm, __shfl_xor_sync(0xffffffffu, cm, 2));
                        const int u = x0 + px0 + mx, vr = Y0 + 4 * b + my0 + 2 * h;
                        const bool in = u < a.W && vr < a.H;
                        const size_t o = in ? (size_t)vr * a.W + u : 0;
                        // the lowest and highest disparity of the quad (relative to d0) whose value is
                        // at most lim (0x7fff / -1 where there is none), and how many there are
                        auto range = [&](float lim, int &lo, int &hi, int &cnt) {
                            uint32_t mk = 0;
#pragma unroll
                            for (int j = 0; j < M; ++j) mk |= v[j] <= lim ? 1u << j : 0u;
                            const int jl = __ffs(mk) - 1, jh = 31 - __clz(mk);
                            lo = mk ? 8 * (jl >> 1) + 2 * t4 + (jl & 1) : 0x7fff;
                            hi = mk ? 8 * (jh >> 1) + 2 * t4 + (jh & 1) : -1;
                            lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, 1));
                            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, 1));
                            lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, 2));
                            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, 2));
                            cnt = 0;
                            if constexpr (REF) {
                                cnt = __popc(mk);
                                cnt += __shfl_xor_sync(0xffffffffu, cnt, 1);
                                cnt += __shfl_xor_sync(0xffffffffu, cnt, 2);
                            }
                        };
                        if constexpr (REF) {
                            // the pixel's certified candidates for the refiners: the lowest and the highest,
                            // and whether there are more than these two
                            const float tn = sc_thr(cm);
                            int lo, hi, cnt;
                            range(tn, lo, hi, cnt);
                            if (t4 == 0) scand[(b & 1) * 128 + (my0 + 2 * h) * 32 + px0 + mx] = lo | (hi << 8) | (cnt > 2 ? 1 << 16 : 0);
                        } else if constexpr (MODE == kMarchScreen) {
                            float em = inf;
                            int rg = 0;
                            if (d0 > 0 && in) {
                                em = a.emin[o];
                                rg = a.cand[o];
                            }
                            const float nm = fminf(em, cm), tn = sc_thr(nm);
                            int lo, hi, cnt;
                            range(tn, lo, hi, cnt);
                            if (hi >= 0) {
                                if (tn < em) rg = d0 + lo;         // the earlier range cannot hold d*
                                rg = (rg & 0xffff) | ((d0 + hi) << 16);
                            }
                            __syncwarp();                          // the quad has read the earlier state
                            if (t4 == 0 && in) {
                                a.cand[o] = rg;
                                if (d0 + N < a.D) a.emin[o] = nm;
                            }
                        } else {
                            // k_fused's running WTA over the chunks: {best, E(d* - 1), E(d* + 1), last value}
                            float best = inf, bm1 = inf, bp1 = inf, last = inf, sec = inf;
                            int bd = -1;
                            const bool b2 = a.best2 != nullptr;
                            const size_t HWs = (size_t)a.W * a.H;
                            if (d0 > 0 && in) {
                                best = a.wst[o];
                                bm1 = a.wst[HWs + o];
                                bp1 = a.wst[2 * HWs + o];
                                last = a.wst[3 * HWs + o];
                                bd = __float_as_int(a.wst[4 * HWs + o]);
                                if (b2) sec = a.wst[5 * HWs + o];
                            }
                            int lo, hi, cnt;
                            range(cm, lo, hi, cnt);
                            auto at = [&](int d) {                 // E(d0 + d) from the lane that holds it
                                const int j = 2 * (d >> 3) + (d & 1);
                                return __shfl_sync(0xffffffffu, pick_reg(v, j), (lane & ~3) | ((d >> 1) & 3));
                            };
                            const float em1 = at(max(lo - 1, 0)), ep1 = at(min(lo + 1, N - 1)), first = at(0), end = at(N - 1);
                            float m2 = inf;                        // the smallest value at another disparity
                            if (b2) {
#pragma unroll
                                for (int j = 0; j < M; ++j)
                                    if (8 * (j >> 1) + 2 * t4 + (j & 1) != lo) m2 = fminf(m2, v[j]);
                                m2 = fminf(m2, __shfl_xor_sync(0xffffffffu, m2, 1));
                                m2 = fminf(m2, __shfl_xor_sync(0xffffffffu, m2, 2));
                            }
                            if (cm < best) {
                                sec = fminf(best, m2);
                                best = cm;
                                bd = d0 + lo;
                                bm1 = lo > 0 ? em1 : last;
                                bp1 = lo + 1 < N ? ep1 : inf;
                            } else {
                                sec = fminf(sec, cm);
                                if (bd == d0 - 1) bp1 = first;
                            }
                            __syncwarp();                          // the quad has read the earlier state
                            if (t4 == 0 && in) {
                                if (d0 + N < a.D) {
                                    a.wst[o] = best;
                                    a.wst[HWs + o] = bm1;
                                    a.wst[2 * HWs + o] = bp1;
                                    a.wst[3 * HWs + o] = end;
                                    a.wst[4 * HWs + o] = __int_as_float(bd);
                                    if (b2) a.wst[5 * HWs + o] = sec;
                                } else {
                                    // eq. (subpixel), add back s_i(v), validity
                                    const int4 rt = __ldg(a.row_tab + vr);
                                    float delta = 0.f;
                                    if (bd > 0 && bd < a.D - 1) {
                                        const float den = 2.f * bm1 + 2.f * bp1 - 4.f * best;
                                        if (den > 0.f) delta = (bm1 - bp1) / den;
                                    }
                                    a.disp[o] = (float)bd + delta + (float)rt.x;
                                    if (a.wta) a.wta[o] = bd;
                                    if (a.valid) {
                                        const int ulo = a.m + a.D - 1 + max(0, rt.y);
                                        const int uhi = a.W - 1 - a.m + min(0, rt.z);
                                        a.valid[o] = (uint8_t)(vr >= a.m && vr <= a.H - 1 - a.m && u >= ulo && u <= uhi);
                                    }
                                    if (b2) {
                                        // the skipped normaliser in FP32 (the sums carry the factor 2^20)
                                        const float ipp = h ? ip1 : ip0;
                                        float wsum = 0.f;
                                        for (int dx = 0; dx < KB; ++dx)
                                            for (int dy = 0; dy < KB; ++dy) {
                                                const int sl = (4 * b + my0 + 2 * h + dy) % RS;
                                                const float t = sI[sl * kMarchSI + px0 + mx + dx] - ipp;
                                                wsum += ex2_approx(fmaf(-t, t, a.K[dx * KB + dy]));
                                            }
                                        const float sc = 1.f / (float)(1 << (kScWSh + kScCSh));
                                        a.best2[2 * o] = best * sc / wsum;
                                        a.best2[2 * o + 1] = sec * sc / wsum;
                                    }
                                }
                            }
                        }
                    }
                }
                if (__syncthreads_or(0)) return;
            }
        } else {
            // ------------------------------------------------------------------ refiners
            // k_fused's FP32 arithmetic on the previous band's certified candidates.  Most pixels have
            // one candidate: it wins, and E(d* - 1), E(d*), E(d* + 1) (eq. subpixel) are one evaluation
            // (warps 0-3, lane = pixel of one row).  The pixels with several are listed and their
            // evaluations dealt out to the lanes of warps 4-7 three disparities at a time (around each
            // of two candidates far apart, else over the whole range between), so that one wide range
            // does not hold up a warp; the winner's neighbours follow when it is known.
            const int rr = (warp - (S::PW + kMarchCW)) & 3;
            const bool listed = warp >= S::PW + kMarchCW + 4;
            AmbList &al = *reinterpret_cast<AmbList *>(smem + L.amb);
            for (int p = 0; p < nsteps + TAIL; ++p) {
                const int b = p - lead - 2;
                if (b >= 0) {
                    const int u = x0 + lane, v = Y0 + 4 * b + rr;
                    const bool in = u < a.W && v < a.H;
                    const int c = scand[(b & 1) * 128 + rr * 32 + lane];
                    // past df = u + m - run + 1 every target read behind the pixel repeats its row's
                    // column-0 value, so every cost and E(p, d) equals that at df: d* <= df
                    const int df = max(0, u + a.m - __ldg(&a.row_tab[min(v, a.H - 1)].w) + 1);
                    const int lo = c & 0xff, top = (c >> 8) & 0xff, hi = max(min(top, df), lo);
                    auto rows = [&](int row, uint32_t (&so)[KB]) {   // ring rows of a window
#pragma unroll
                        for (int j = 0; j < KB; ++j) so[j] = (uint32_t)((4 * b + row + j) % RS) * kMarchSI;
                    };
                    // the outputs of the pixel at column px of row `row` whose winner is bd
                    auto finish = [&](int row, int px, int bd, bool on) {
                        uint32_t so[KB];
                        rows(row, so);
                        float em, e, ep;
                        march_eval3<RB, N>(ring32, sI, sK, so, px, max(bd - 1, 0), em, e, ep);
                        if (bd == 0) {
                            ep = e;
                            e = em;
                        }
                        const int uu = x0 + px, vv = Y0 + 4 * b + row;
                        if (!on) return;
                        const int4 rt = __ldg(a.row_tab + vv);   // {s_i, max, min s_i over v +- m, run}
                        float delta = 0.f;
                        if (bd > 0 && bd < a.D - 1) {
                            const float den = 2.f * em + 2.f * ep - 4.f * e;
                            if (den > 0.f) delta = (em - ep) / den;
                        }
                        const size_t o = (size_t)vv * a.W + uu;
                        a.disp[o] = (float)bd + delta + (float)rt.x;
                        if (a.wta) a.wta[o] = bd;
                        if (a.valid) {
                            const int ulo = a.m + a.D - 1 + max(0, rt.y);
                            const int uhi = a.W - 1 - a.m + min(0, rt.z);
                            a.valid[o] = (uint8_t)(vv >= a.m && vv <= a.H - 1 - a.m && uu >= ulo && uu <= uhi);
                        }
                    };
                    if (!listed) {
                        if (__any_sync(0xffffffffu, in && lo == hi)) finish(rr, lane, lo, in && lo == hi);
                    } else {
                        // the list: each row's pixels, then the rows after one another
                        const bool amb = in && lo != hi, two = amb && !(c >> 16) && hi == top && hi - lo > 2;
                        const int nu = !amb ? 0 : two ? 2 : (hi - lo) / 3 + 1;
                        const unsigned bal = __ballot_sync(0xffffffffu, amb);
                        int us = nu;                       // inclusive sum of the units
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int t = __shfl_up_sync(0xffffffffu, us, o);
                            if (lane >= o) us += t;
                        }
                        if (lane == 31) {
                            al.nw[rr] = __popc(bal);
                            al.uw[rr] = us;
                        }
                        asm volatile("bar.sync 2, 128;" ::: "memory");
                        int n0 = 0, u0 = 0, nt = 0, ut = 0;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int nj = al.nw[j], uj = al.uw[j];
                            if (j < rr) {
                                n0 += nj;
                                u0 += uj;
                            }
                            nt += nj;
                            ut += uj;
                        }
                        if (amb) {
                            const int i = n0 + __popc(bal & ((1u << lane) - 1u));
                            al.key[i] = ~0ull;
                            al.first[i] = (uint16_t)(u0 + us - nu);
                            al.pix[i] = (uint8_t)(rr * 32 + lane);
                            al.lo[i] = (uint8_t)lo;
                            al.hi[i] = (uint8_t)hi;
                            al.split[i] = two ? (uint8_t)hi : 255;
                        }
                        if (lane == 0 && rr == 0) al.first[nt] = (uint16_t)ut;
                        asm volatile("bar.sync 2, 128;" ::: "memory");
                        for (int q = 32 * rr; q < ut; q += 128) {
                            const int unit = min(q + lane, ut - 1);
                            int i = 0;                     // the last listed pixel whose first unit is <= unit
#pragma unroll
                            for (int st = 64; st > 0; st >>= 1)
                                if (i + st < nt && al.first[i + st] <= unit) i += st;
                            const int px = al.pix[i], k = unit - al.first[i];
                            const bool sp = al.split[i] != 255;
                            const int d = sp ? (k ? al.split[i] : al.lo[i]) : al.lo[i] + 3 * k;
                            const int dend = sp ? d : al.hi[i];
                            uint32_t so[KB];
                            rows(px >> 5, so);
                            float e[3];
                            march_eval3<RB, N>(ring32, sI, sK, so, px & 31, d, e[0], e[1], e[2]);
                            unsigned long long key = ~0ull;
#pragma unroll
                            for (int j = 0; j < 3; ++j) {
                                unsigned x = __float_as_uint(e[j]);
                                x ^= (x >> 31) ? 0xffffffffu : 0x80000000u;
                                const unsigned long long kj = ((unsigned long long)x << 32) | (unsigned)(d + j);
                                if (d + j <= dend && kj < key) key = kj;
                            }
                            atomicMin(&al.key[i], key);
                        }
                        asm volatile("bar.sync 2, 128;" ::: "memory");
                        for (int q = 32 * rr; q < nt; q += 128) {
                            const int i = min(q + lane, nt - 1), px = al.pix[i];
                            finish(px >> 5, px & 31, (int)(unsigned)(al.key[i] & 0xffffffffu), q + lane < nt);
                        }
                    }
                }
                if (__syncthreads_or(0)) return;
            }
        }
    }
}

template <int RB, int N, int MODE, typename T>
MarchChoice march_choice(int rw)
{
    return MarchChoice{k_march<RB, N, MODE, T>, MarchShape<RB, N>::threads(MODE), march_layout<RB, N>(rw, MODE).total};
}

template <int N, int MODE, typename T>
MarchChoice pick_march_rb(int rb, int rw)
{
    switch (rb) {
    case 0: return march_choice<0, N, MODE, T>(rw);
    case 1: return march_choice<1, N, MODE, T>(rw);
    case 2: return march_choice<2, N, MODE, T>(rw);
    case 3: return march_choice<3, N, MODE, T>(rw);
    case 4: return march_choice<4, N, MODE, T>(rw);
    case 5: return march_choice<5, N, MODE, T>(rw);
    case 6:
        if constexpr (N <= 96) return march_choice<6, N, MODE, T>(rw);
    }
    return MarchChoice{nullptr, 0, 0};
}

}  // namespace sgb
