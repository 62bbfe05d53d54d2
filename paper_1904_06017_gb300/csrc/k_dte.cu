// k_dte.cu -- the disparity-transformation energy of eq. (E2), its adjoint, and roll
// refinement by gradient (include/stereo_diff.h).
//
// Every reduction runs in two fixed-order stages: kDteBlocks blocks per pair write FP64
// partial sums, one warp per pair adds them.  Per pixel the energy and its adjoint work in
// FP32; the refinement reduces the map once to ten moments in centred coordinates, and every
// step evaluates the sums it needs at its angle from them (exact algebra) and the line fit of
// eq. (alpha3) in FP64.
//
// An FP64 instruction of a warp occupies a GB300 SM about 16 times as long as an FP32 one and
// returns after about 65 cycles, so the per-pixel sums are kept out of FP64: a warp adds its
// pixels in three floats each (the rounding error of every addition and product is recovered
// exactly and summed in the second, that sum's own in the third, so that a sum carries more than
// 64 bits) and widens once at the end; sums over pixel coordinates are exact integers.
// (Two floats, 24 bits for the sum of the errors, left 3e-14 of sum l^2 on a constant map, 200 times
// the error of FP64 sums.)  A warp whose sum is not finite (an infinite or NaN disparity, or a sum
// beyond the FP32 range), or whose products leave errors below that range, adds its pixels again in
// FP64.  8 maps of 960 x 540: energy 15 us (24 us with FP64 sums and butterflies), adjoint 23 us
// (63), moments 32 us (152); bound by the FP64 tail of a block (the widened warp sums) and the
// two-sums more than by reading the map.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "dt_trig.cuh"
#include "internal.cuh"
#include "stereo_diff.h"

namespace sgb {
namespace {

constexpr int kDteBlocks = 64;     // partial-sum blocks per pair
constexpr int kDteSums = 10;       // the most sums one pass produces (the refinement)
constexpr int kDteThreads = 256;

enum { DTE_ENERGY = 0, DTE_BWD = 1 };

size_t dte_bytes(int B)
{
    const size_t part = (size_t)B * kDteBlocks * kDteSums * sizeof(double);
    return (part + 255) / 256 * 256;
}

// s + x, and what its rounding leaves.
__device__ __forceinline__ float two_sum(float &s, float x)
{
    const float t = __fadd_rn(s, x), b = __fsub_rn(t, s), e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b));
    s = t;
    return e;
}

// A sum of floats: hi, the rounding errors of its additions in mid, and those of mid's in lo.
struct TripleSum {
    float hi, mid, lo;
    __device__ __forceinline__ void add_error(float x) { lo = __fadd_rn(lo, two_sum(mid, x)); }
    __device__ __forceinline__ void add(float x) { add_error(two_sum(hi, x)); }
    // += the exact product x y (its error is exact unless it falls below the FP32 range)
    __device__ __forceinline__ void add_product(float x, float y)
    {
        const float p = __fmul_rn(x, y);
        add_error(__fmaf_rn(x, y, -p));
        add(p);
    }
    __device__ __forceinline__ bool finite() const { return isfinite(hi) && isfinite(mid) && isfinite(lo); }
    __device__ __forceinline__ double value() const { return (double)hi + ((double)mid + (double)lo); }
    // the total over the 32 lanes of a warp, the same bits on every lane (each step is symmetric in the
    // two lanes that meet)
    __device__ __forceinline__ void warp_add()
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float h = __shfl_xor_sync(0xffffffffu, hi, o), m = __shfl_xor_sync(0xffffffffu, mid, o),
                        l = __shfl_xor_sync(0xffffffffu, lo, o);
            const float eh = two_sum(hi, h), em = two_sum(mid, m), ee = two_sum(mid, eh);
            lo = __fadd_rn(__fadd_rn(lo, l), __fadd_rn(em, ee));
        }
    }
};

// The block's total of every warp's values (lane 0 of each warp holds them), in warp order.
template <int NS>
__device__ void block_sum_store(const double (&acc)[NS], double *out)
{
    __shared__ double red[kDteThreads / 32][NS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < NS; ++k) red[wid][k] = acc[k];
    }
    __syncthreads();
    if (threadIdx.x < NS) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < kDteThreads / 32; ++w) v += red[w][threadIdx.x];
        out[threadIdx.x] = v;
    }
}

__device__ __forceinline__ double warp_add(double x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

__device__ __forceinline__ long long warp_add(long long x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Per pixel r = l - alpha0 - alpha1 y(psi), y = v cos(psi) - u sin(psi) (eq. y).
// DTE_ENERGY: sum m r^2.  DTE_BWD: gl = 2 g m r, sums of m r x, m r, m r y.
template <int MODE>
__global__ void __launch_bounds__(kDteThreads) k_dte(const float *__restrict__ disp, const uint8_t *__restrict__ mask,
                                                     const double *__restrict__ theta, const double *__restrict__ gE,
                                                     float *__restrict__ gdisp, double *__restrict__ part, int W,
                                                     int H)
{
    constexpr int NS = MODE == DTE_ENERGY ? 1 : 3;
    __shared__ float sc[5];
    const int b = blockIdx.y;
    if (threadIdx.x == 0) {
        const double psi = theta[3 * b];
        sc[0] = (float)cos(psi);
        sc[1] = (float)sin(psi);
        sc[2] = (float)theta[3 * b + 1];
        sc[3] = (float)theta[3 * b + 2];
        sc[4] = MODE == DTE_BWD ? (float)(2.0 * gE[b]) : 0.f;
    }
    __syncthreads();
    const float c = sc[0], s = sc[1], a0 = sc[2], a1 = sc[3], g2 = sc[4];
    const int HW = W * H;
    const float *L = disp + (size_t)b * HW;
    const uint8_t *M = mask ? mask + (size_t)b * HW : nullptr;
    // the values of pixel i that are summed
    auto terms = [&](int i, float l, bool in, float (&t)[NS]) {
        const int v = i / W, u = i - v * W;
        const float m = in ? 1.f : 0.f;
        const float y = (float)v * c - (float)u * s;
        const float r = m * (l - a0 - a1 * y);
        if constexpr (MODE == DTE_ENERGY) {
            t[0] = __fmul_rn(r, r);
        } else {
            if (gdisp) gdisp[(size_t)b * HW + i] = g2 * r;
            const float x = (float)u * c + (float)v * s;
            t[0] = __fmul_rn(r, x);
            t[1] = r;
            t[2] = __fmul_rn(r, y);
        }
    };
    constexpr int kStep = kDteBlocks * kDteThreads, kAhead = 4;   // loads in flight per thread
    const int i0 = blockIdx.x * kDteThreads + threadIdx.x;
    TripleSum ps[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) ps[k] = TripleSum{0.f, 0.f, 0.f};
    for (int i = i0; i < HW; i += kAhead * kStep) {
        float l[kAhead];
        bool in[kAhead];
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int p = i + j * kStep;
            l[j] = p < HW ? L[p] : 0.f;
            in[j] = p < HW && (!M || M[p]);
        }
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int p = i + j * kStep;
            if (p >= HW) break;
            float t[NS];
            terms(p, l[j], in[j], t);
#pragma unroll
            for (int k = 0; k < NS; ++k) ps[k].add(t[k]);
        }
    }
    double acc[NS];
    bool finite = true;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        ps[k].warp_add();
        finite = finite && ps[k].finite();
        acc[k] = ps[k].value();
    }
    if (!__all_sync(0xffffffffu, finite)) {
#pragma unroll
        for (int k = 0; k < NS; ++k) acc[k] = 0.0;
        for (int i = i0; i < HW; i += kStep) {
            float t[NS];
            terms(i, L[i], !M || M[i], t);
#pragma unroll
            for (int k = 0; k < NS; ++k) acc[k] += (double)t[k];
        }
#pragma unroll
        for (int k = 0; k < NS; ++k) acc[k] = warp_add(acc[k]);
    }
    block_sum_store<NS>(acc, part + ((size_t)b * kDteBlocks + blockIdx.x) * kDteSums);
}

// The partials of pair b added by one warp: lane l takes partials l and l + 32, then a
// butterfly (every lane returns the total).
template <int NS>
__device__ __forceinline__ void sum_partials(const double *__restrict__ part, int b, double (&s)[NS])
{
    static_assert(kDteBlocks == 64, "two partials per lane");
    const double *p = part + ((size_t)b * kDteBlocks + (threadIdx.x & 31)) * kDteSums;
#pragma unroll
    for (int k = 0; k < NS; ++k) s[k] = p[k] + p[32 * kDteSums + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < NS; ++k) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
}

// One warp (block) per pair.
template <int MODE>
__global__ void __launch_bounds__(32) k_dte_finish(const double *__restrict__ part, const double *__restrict__ theta,
                                                   const double *__restrict__ gE, double *__restrict__ out)
{
    constexpr int NS = MODE == DTE_ENERGY ? 1 : 3;
    const int b = blockIdx.x;
    double s[NS];
    sum_partials<NS>(part, b, s);
    if (threadIdx.x != 0) return;
    if constexpr (MODE == DTE_ENERGY) {
        out[b] = s[0];
    } else {
        const double g = gE[b], a1 = theta[3 * b + 2];
        out[3 * b + 0] = 2.0 * g * a1 * s[0];      // dL/dpsi: dy/dpsi = -x
        out[3 * b + 1] = -2.0 * g * s[1];          // dL/dalpha0
        out[3 * b + 2] = -2.0 * g * s[2];          // dL/dalpha1
    }
}

// The ten moments of the fitted pixels in coordinates centred on the image:
// n, S_u, S_v, S_l, S_uu, S_uv, S_vv, S_ul, S_vl, S_ll with u' = u - (W-1)/2, v' = v - (H-1)/2.
// Every sum the refinement needs at an angle psi is a fixed combination of them.  The
// coordinates enter doubled (whole numbers); the sums with l are those of exact products.
__global__ void __launch_bounds__(kDteThreads) k_dref_moments(const float *__restrict__ disp,
                                                              const uint8_t *__restrict__ mask,
                                                              double *__restrict__ part, int W, int H)
{
    const int b = blockIdx.y;
    const int HW = W * H;
    const float *L = disp + (size_t)b * HW;
    const uint8_t *M = mask ? mask + (size_t)b * HW : nullptr;
    constexpr int kStep = kDteBlocks * kDteThreads, kAhead = 4;
    const int i0 = blockIdx.x * kDteThreads + threadIdx.x;
    int n = 0;
    long long su = 0, sv = 0, suu = 0, suv = 0, svv = 0;   // sums over 2u', 2v' and their products
    TripleSum sl{0.f, 0.f, 0.f}, sul{0.f, 0.f, 0.f}, svl{0.f, 0.f, 0.f}, sll{0.f, 0.f, 0.f};
    bool any = false;   // a disparity other than 0
    for (int i = i0; i < HW; i += kAhead * kStep) {
        float l[kAhead];
        bool in[kAhead];
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int p = i + j * kStep;
            l[j] = p < HW ? L[p] : 0.f;
            in[j] = p < HW && (!M || M[p]);
        }
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            if (!in[j]) continue;
            const int p = i + j * kStep, v = p / W, u = p - v * W;
            const int x = 2 * u - (W - 1), y = 2 * v - (H - 1);
            ++n;
            any = any || l[j] != 0.f;
            su += x;
            sv += y;
            suu += (long long)x * x;
            suv += (long long)x * y;
            svv += (long long)y * y;
            sl.add(l[j]);
            sul.add_product(0.5f * (float)x, l[j]);
            svl.add_product(0.5f * (float)y, l[j]);
            sll.add_product(l[j], l[j]);
        }
    }
    sl.warp_add();
    sul.warp_add();
    svl.warp_add();
    sll.warp_add();
    n = __reduce_add_sync(0xffffffffu, n);
    double acc[kDteSums] = {(double)n, 0.5 * (double)warp_add(su), 0.5 * (double)warp_add(sv), sl.value(),
                            0.25 * (double)warp_add(suu), 0.25 * (double)warp_add(suv), 0.25 * (double)warp_add(svv),
                            sul.value(), svl.value(), sll.value()};
    // below 2^-80 the errors of the products l^2 (and with them those of u l, v l) may have underflowed
    const bool small = __any_sync(0xffffffffu, any) && !(acc[9] >= 0x1p-80);
    if (__any_sync(0xffffffffu, small || !(sl.finite() && sul.finite() && svl.finite() && sll.finite()))) {
        double f[4] = {0.0, 0.0, 0.0, 0.0};
        for (int i = i0; i < HW; i += kStep) {
            if (M && !M[i]) continue;
            const int v = i / W, u = i - v * W;
            const double x = (double)u - 0.5 * (W - 1), y = (double)v - 0.5 * (H - 1), l = (double)L[i];
            f[0] += l;
            f[1] = fma(x, l, f[1]);
            f[2] = fma(y, l, f[2]);
            f[3] = fma(l, l, f[3]);
        }
        acc[3] = warp_add(f[0]);
        acc[7] = warp_add(f[1]);
        acc[8] = warp_add(f[2]);
        acc[9] = warp_add(f[3]);
    }
    block_sum_store<kDteSums>(acc, part + ((size_t)b * kDteBlocks + blockIdx.x) * kDteSums);
}

__device__ double wrap_half_pi_d(double psi)
{
    psi = fmod(psi, M_PI);
    if (psi > 0.5 * M_PI) psi -= M_PI;
    else if (psi <= -0.5 * M_PI) psi += M_PI;
    return psi;
}

// All refinement steps of one pair (one warp per pair).  The moments, per pixel and about the
// centroid of the fitted pixels, are taken once; at an angle, with x = u cos + v sin and
// y = v cos - u sin (eq. x, eq. y), the line fit of eq. (alpha3) is alpha1 = C_yl / C_yy and
// alpha0 = mean(l) - alpha1 mean(y), E = n (C_ll - alpha1 C_yl), g = dE/dpsi = 2 n alpha1
// (C_xl - alpha1 C_xy) (eq. d_e_min), and the Gauss-Newton curvature H = 2 n alpha1^2
// (C_xx - C_xy^2 / C_yy); the step is psi <- wrap(psi - g / H).
//
// The steps are one FP64 dependency chain, so only what the next angle needs is on it: with
// C_xx C_yy - C_xy^2 = det, the same at every angle, g / H = C_yy (C_xl C_yy - C_yl C_xy) /
// (C_yl det), one quotient: an FP32 reciprocal with one Newton step in FP64 (about 47 bits), then the
// quotient corrected by its own remainder (a rounding off; 7e-15 of the step without it), or the
// full division where FP32 cannot hold the divisor.  The angles go to shared memory, and the trajectory's
// entries are then evaluated with one step per lane.  50 steps: 106 us (289 us with the sums
// over raw coordinates and every quantity of a step evaluated on the chain).
constexpr int kDrefSteps = 1000;   // the most steps a call may ask for

__global__ void __launch_bounds__(32) k_dref_run(const double *__restrict__ part, double psi_init,
                                                 double *__restrict__ traj, int steps, int W, int H)
{
    __shared__ double sp[kDrefSteps + 1];
    const int b = blockIdx.x;
    double m[kDteSums];
    sum_partials<kDteSums>(part, b, m);
    // (divisions: the mean of equal coordinates is that coordinate exactly, and its spread 0)
    const double n = m[0], n1 = n > 0.0 ? n : 1.0;
    const double mu = m[1] / n1, mv = m[2] / n1, ml = m[3] / n1;
    const double Cuu = (m[4] - m[1] * mu) / n1, Cuv = (m[5] - m[1] * mv) / n1, Cvv = (m[6] - m[2] * mv) / n1;
    const double Cul = (m[7] - m[1] * ml) / n1, Cvl = (m[8] - m[2] * ml) / n1, Cll = (m[9] - m[3] * ml) / n1;
    const double Cdf = Cvv - Cuu, det = Cuu * Cvv - Cuv * Cuv;
    double psi = wrap_half_pi_d(psi_init);
    for (int k = 0; k < steps; ++k) {
        if (threadIdx.x == 0) sp[k] = psi;
        double s, c;
        sincos_half_pi(psi, &s, &c);
        const double cs = c * s, ss = s * s;
        const double Cyy = (Cvv - ss * Cdf) - 2.0 * cs * Cuv, Cxy = cs * Cdf + (Cuv - 2.0 * ss * Cuv);
        const double Cyl = c * Cvl - s * Cul, Cxl = c * Cul + s * Cvl;
        if (!(Cyy > 0.0)) continue;   // no line to fit: the angle stays
        const double num = Cyy * (Cxl * Cyy - Cyl * Cxy), den = Cyl * det;
        const float r0 = 1.0f / (float)den;
        double d;
        if (fabsf(r0) > 1e-30f && fabsf(r0) < 1e30f) {
            const double r = (double)r0, r1 = r * (2.0 - den * r);
            d = num * r1;
            d = fma(fma(-d, den, num), r1, d);
        } else {
            d = num / den;
        }
        // a step only where the curvature is positive (C_yl^2 det > 0) and the quotient finite
        if (den * Cyl > 0.0 && isfinite(d)) {
            psi -= d;
            if (psi > 0.5 * M_PI || psi <= -0.5 * M_PI) psi = wrap_half_pi_d(psi);
        }
    }
    if (threadIdx.x == 0) sp[steps] = psi;
    __syncwarp();
    const double uc = mu + 0.5 * (W - 1), vc = mv + 0.5 * (H - 1);   // the centroid in raw coordinates
    for (int k = threadIdx.x; k <= steps; k += 32) {
        const double p = sp[k];
        double s, c;
        sincos_half_pi(p, &s, &c);
        const double cs = c * s, ss = s * s;
        const double Cyy = (Cvv - ss * Cdf) - 2.0 * cs * Cuv, Cxy = cs * Cdf + (Cuv - 2.0 * ss * Cuv);
        const double Cyl = c * Cvl - s * Cul, Cxl = c * Cul + s * Cvl;
        double a0 = ml, a1 = 0.0, g = 0.0;
        if (n > 0.0 && Cyy > 0.0) {
            a1 = Cyl / Cyy;
            g = 2.0 * n * a1 * (Cxl - a1 * Cxy);
            a0 = ml - a1 * (vc * c - uc * s);
        }
        double *t = traj + ((size_t)b * (steps + 1) + k) * 5;
        t[0] = p;
        t[1] = a0;
        t[2] = a1;
        t[3] = g;
        t[4] = n * (Cll - a1 * Cyl);
    }
}

int check_sizes(int W, int H, int B, const char *who)
{
    if (W < 1 || H < 1 || W > 8192 || H > 8192)
        return set_error(STEREO_EINVAL, "%s: width/height %d x %d outside 1..8192", who, W, H);
    if (B < 1 || B > 64) return set_error(STEREO_EINVAL, "%s: batch %d outside 1..64", who, B);
    return STEREO_OK;
}

int check_dte_ws(int B, void *ws, size_t bytes, const char *who)
{
    if (!ws) return set_error(STEREO_EINVAL, "%s: null workspace", who);
    if ((uintptr_t)ws % 256) return set_error(STEREO_EINVAL, "%s: workspace not 256-byte aligned", who);
    if (bytes < dte_bytes(B))
        return set_error(STEREO_EINVAL, "%s: workspace of %zu bytes, %zu needed", who, bytes, dte_bytes(B));
    return STEREO_OK;
}

}  // namespace
}  // namespace sgb

using namespace sgb;

extern "C" int stereo_dt_energy_workspace_bytes(int32_t batch, size_t *bytes)
{
    if (batch < 1 || batch > 64 || !bytes)
        return set_error(STEREO_EINVAL, "stereo_dt_energy_workspace_bytes: batch outside 1..64 or null output");
    *bytes = dte_bytes(batch);
    return STEREO_OK;
}

extern "C" int stereo_dt_energy_fwd(int32_t W, int32_t H, int32_t B, const float *disp, const uint8_t *mask,
                                    const double *theta, double *energy, void *ws, size_t ws_bytes,
                                    stereo_stream_t stream)
{
    static const char *who = "stereo_dt_energy_fwd";
    int rc = check_sizes(W, H, B, who);
    if (rc) return rc;
    if (!disp || !theta || !energy) return set_error(STEREO_EINVAL, "%s: null pointer", who);
    if ((rc = check_dte_ws(B, ws, ws_bytes, who))) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    double *part = (double *)ws;
    k_dte<DTE_ENERGY><<<dim3(kDteBlocks, B), kDteThreads, 0, st>>>(disp, mask, theta, nullptr, nullptr, part,
                                                                    W, H);
    k_dte_finish<DTE_ENERGY><<<B, 32, 0, st>>>(part, theta, nullptr, energy);
    return cuda_error(cudaGetLastError(), who);
}

extern "C" int stereo_dt_energy_bwd(int32_t W, int32_t H, int32_t B, const float *disp, const uint8_t *mask,
                                    const double *theta, const double *gE, float *gdisp, double *gtheta,
                                    void *ws, size_t ws_bytes, stereo_stream_t stream)
{
    static const char *who = "stereo_dt_energy_bwd";
    int rc = check_sizes(W, H, B, who);
    if (rc) return rc;
    if (!disp || !theta || !gE) return set_error(STEREO_EINVAL, "%s: null pointer", who);
    if ((rc = check_dte_ws(B, ws, ws_bytes, who))) return rc;
    if (!gdisp && !gtheta) return STEREO_OK;
    cudaStream_t st = (cudaStream_t)stream;
    double *part = (double *)ws;
    k_dte<DTE_BWD><<<dim3(kDteBlocks, B), kDteThreads, 0, st>>>(disp, mask, theta, gE, gdisp, part, W, H);
    if (gtheta) k_dte_finish<DTE_BWD><<<B, 32, 0, st>>>(part, theta, gE, gtheta);
    return cuda_error(cudaGetLastError(), who);
}

extern "C" int stereo_dt_refine_roll(int32_t W, int32_t H, int32_t B, const float *disp, const uint8_t *mask,
                                     double psi_init, int32_t steps, double *traj, void *ws, size_t ws_bytes,
                                     stereo_stream_t stream)
{
    static const char *who = "stereo_dt_refine_roll";
    int rc = check_sizes(W, H, B, who);
    if (rc) return rc;
    if (!disp || !traj) return set_error(STEREO_EINVAL, "%s: null pointer", who);
    if (steps < 0 || steps > kDrefSteps) return set_error(STEREO_EINVAL, "%s: steps %d outside 0..%d", who, steps, kDrefSteps);
    if (!isfinite(psi_init)) return set_error(STEREO_EINVAL, "%s: psi_init not finite", who);
    if ((rc = check_dte_ws(B, ws, ws_bytes, who))) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    double *part = (double *)ws;
    k_dref_moments<<<dim3(kDteBlocks, B), kDteThreads, 0, st>>>(disp, mask, part, W, H);
    k_dref_run<<<B, 32, 0, st>>>(part, psi_init, traj, steps, W, H);
    return cuda_error(cudaGetLastError(), who);
}
