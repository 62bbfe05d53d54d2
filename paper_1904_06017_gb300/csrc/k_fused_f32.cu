// k_fused_f32.cu -- FP32 cost storage instantiations of the fused kernel, and the host
// side shared by all storage types (shared-memory sizing, kernel choice, launch).
#include <string.h>

#include <algorithm>

#include "k_fused.cuh"
#include "k_fused_tc.cuh"
#include "k_refine.cuh"

namespace sgb {

FusedKernel pick_fused_f32(int rb, int dc, int wc)
{
    if (wc != 2) return pick_fused_f32_tiles(rb, dc, wc);
    if (dc == 12) return pick_rb<12, float, 2>(rb);
    if (dc == 4) return pick_fused_f32_dc4(rb);
    return nullptr;
}

FusedKernel pick_fused(int cost_dtype, int rb, int dc, int wc)
{
    if (wc == kWsWC) return cost_dtype == STEREO_F32 && rb <= kWsMaxRB ? pick_fused_ws(rb, dc) : nullptr;
    if (wc == kTcWC) return dc == kTcDC && rb <= kTcMaxRB ? pick_fused_tc(cost_dtype, rb) : nullptr;
    switch (wc == kScWC ? -1 : cost_dtype) {
    case STEREO_F32: return pick_fused_f32(rb, dc, wc);
    case STEREO_F16: return pick_fused_f16(rb, dc, wc);
    case STEREO_BF16: return pick_fused_bf16(rb, dc, wc);
    }
    return nullptr;
}

bool fused_available(int cost_dtype, int rb, int dc, int wc)
{
    if (wc == kScWC) return dc == kScDC && rb <= kScMaxRB;
    return pick_fused(cost_dtype, rb, dc, wc) != nullptr;
}

size_t refine_smem_bytes(const Geometry &g, int rows)
{
    return refine_layout(g.rb, g.m, g.ref_box_w, g.tgt_box_w, g.box_h, rows).total;
}

size_t fused_smem_bytes(const Geometry &g)
{
    if (g.wc == kTcWC) return tc_layout(g.rb, g.m, g.ref_box_w, g.tgt_box_w, g.box_h, g.esize).total;
    if (g.wc == kScWC) {
        if (g.rb > kScMaxRB) return (size_t)1 << 30;
        if (g.esize != 4) return pick_march(STEREO_F16, g.rb, g.rw, g.D).smem;
        const size_t m = sc_route(g.W, g.H, g.D) == kRouteTile ? sc_smem_bytes(g) : pick_march(STEREO_F32, g.rb, g.rw, g.D).smem;
        return std::max(m, refine_smem_bytes(g));
    }
    // the warp-specialised form keeps the two-pass cost phase (vband, staged statistics); the
    // others compute costs on the tensor cores and need neither
    const bool ws = g.wc == kWsWC;
    return smem_layout(g.rb, g.m, g.dc, g.ref_box_w, g.tgt_box_w, g.box_h, g.esize, g.tx, g.ty, ws ? 2 : 1,
                       ws ? kWsBand : 0)
        .total;
}

static FusedKernel pick(const stereo_ctx *ctx)
{
    return pick_fused(ctx->p.cost_dtype, ctx->g.rb, ctx->g.dc, ctx->g.wc);
}

int fused_configure(stereo_ctx *ctx)
{
    const Geometry &g = ctx->g;
    if (g.wc == kScWC) {
        if (!fused_available(ctx->p.cost_dtype, g.rb, g.dc, g.wc))
            return set_error(STEREO_ENOTSUP, "no tensor-core form for bil=%d dc=%d", ctx->p.bil, g.dc);
        const bool f32 = ctx->p.cost_dtype == STEREO_F32;
        int rc;
        if (f32 && sc_route(g.W, g.H, g.D) == kRouteTile) {
            rc = allow_smem((const void *)pick_fused_sc(g.rb), sc_smem_bytes(g), "cudaFuncSetAttribute(tiles)");
        } else {
            const MarchChoice c = pick_march(ctx->p.cost_dtype, g.rb, g.rw, g.D);
            rc = allow_smem((const void *)c.kernel, c.smem, "cudaFuncSetAttribute(march)");
            if (!rc && march_split(g.rb, g.D)) {
                const MarchChoice m = pick_march(ctx->p.cost_dtype, g.rb, g.rw, march_split(g.rb, g.D)),
                                  r = pick_march_rest(ctx->p.cost_dtype, g.rb, g.rw, g.D);
                rc = allow_smem((const void *)m.kernel, m.smem, "cudaFuncSetAttribute(march)");
                if (!rc) rc = allow_smem((const void *)r.kernel, r.smem, "cudaFuncSetAttribute(march)");
            }
        }
        if (rc || !f32) return rc;
        const size_t rs = refine_smem_bytes(g);
        for (int ctas = 1; ctas <= 2; ++ctas)
            if ((rc = allow_smem((const void *)pick_refine(g.rb, false, kRefineRows, ctas), refine_smem_bytes(g, kRefineRows),
                                 "cudaFuncSetAttribute(refine)")))
                return rc;
        if ((rc = allow_smem((const void *)pick_refine(g.rb, false), rs, "cudaFuncSetAttribute(refine)"))) return rc;
        return allow_smem((const void *)pick_refine(g.rb, true), rs, "cudaFuncSetAttribute(refine, best2)");
    }
    FusedKernel k = pick(ctx);
    if (!k)
        return set_error(STEREO_ENOTSUP, "no fused kernel for bil=%d dc=%d cost_dtype=%d", ctx->p.bil, ctx->g.dc,
                         ctx->p.cost_dtype);
    int rc = allow_smem((const void *)k, ctx->g.smem_bytes, "cudaFuncSetAttribute(fused)");
    FusedKernel k2 = pick_fused_b2(ctx->p.cost_dtype, ctx->g.rb, ctx->g.dc, ctx->g.wc);
    if (!rc && k2) rc = allow_smem((const void *)k2, ctx->g.smem_bytes, "cudaFuncSetAttribute(fused, best2)");
    return rc;
}

// The pair descriptor of a context for one call (outputs are per call).
void fill_pair_desc(const stereo_ctx *ctx, float *disp, int32_t *wta, uint8_t *valid, PairDesc &d, float *best2)
{
    const Geometry &g = ctx->g;
    FusedArgs &a = d.a;
    memset(&d, 0, sizeof(d));
    d.tmap_ref = ctx->tmap_ref;
    d.tmap_tgt = ctx->tmap_tgt;
    d.ntx = g.ntx;
    d.nty = g.nty;
    a.ref_stats = ctx->ref_stats;
    a.tgt_stats = ctx->tgt_stats;
    a.row_tab = ctx->row_tab;
    a.disp = disp;
    a.wta = wta;
    a.valid = valid;
    a.best2 = best2;
    a.ref_pad = ctx->ref_pad;
    a.tgt_pad = ctx->tgt_pad;
    a.cand = ctx->cand;
    a.emin = ctx->emin;
    a.wst = ctx->wst;
    a.status = ctx->status_dev;
    a.stall_test = ctx->stall_test;
    a.W = g.W;
    a.H = g.H;
    a.D = g.D;
    a.Dp = g.Dp;
    a.rw = g.rw;
    a.m = g.m;
    a.n = g.n;
    a.pad_left = g.pad_left;
    a.pad_top = g.pad_top;
    a.pad_w = g.pad_w;
    a.pad_pitch = g.pad_pitch;
    a.ref_e = g.ref_e;
    a.tgt_e = g.tgt_e;
    a.ref_box_w = g.ref_box_w;
    a.tgt_box_w = g.tgt_box_w;
    a.box_h = g.box_h;
    a.ref_box_x = g.pad_left - (int)align_up(g.m, 16);
    a.iscale = ctx->iscale;
    const int kb = 2 * g.rb + 1;
    for (int i = 0; i < kb * kb; ++i) a.K[i] = ctx->kspatial[i];
}

int launch_fused(stereo_ctx *ctx, const float *shift, float *disp, int32_t *wta, uint8_t *valid,
                 cudaStream_t s, float *best2)
{
    (void)shift;   // the integer shifts come from the row table built by k_row_tables
    const Geometry &g = ctx->g;
    if (g.wc == kScWC) {
        PairDesc d;
        fill_pair_desc(ctx, disp, wta, valid, d, best2);
        const bool f32 = ctx->p.cost_dtype == STEREO_F32;
        const int route = !f32 ? kRouteMarch : best2 ? kRouteTile : sc_route(g.W, g.H, g.D);
        if (!(f32 && route == kRouteTile)) {
            const int split = march_split(g.rb, g.D);
            cudaError_t e = cudaSuccess;
            for (int lo = 0; lo < g.D && e == cudaSuccess; lo = split && !lo ? split : g.D) {
                const int hi = split && !lo ? split : g.D;
                const MarchChoice c = lo ? pick_march_rest(ctx->p.cost_dtype, g.rb, g.rw, g.D)
                                         : pick_march(ctx->p.cost_dtype, g.rb, g.rw, hi);
                const int nb = march_bands(g.W, g.H, g.m, ctx->nsm * march_ctas(march_n(g.rb, hi - lo), f32));
                c.kernel<<<march_items(g.W, g.H, nb), c.threads, c.smem, s>>>(d, nullptr, nullptr, nb, lo, hi);
                e = cudaGetLastError();
            }
            if (e != cudaSuccess || !f32 || route == kRouteRefine) return cuda_error(e, "k_march launch");
        }
        // persistent tiles: one CTA per SM (two of k_refine's low tiles), tiles in turn, the next tile's
        // images staged while the current one finishes.  (With best2 every disparity is refined: nothing
        // to screen.)
        const bool tile = route == kRouteTile && !best2;
        const int rows = tile || best2 ? g.ty : refine_rows(g.ntx * g.nty, ctx->nsm);
        const int ntiles = g.ntx * ((g.H + rows - 1) / rows);
        const int ctas = tile || best2 ? 1 : refine_ctas(g.ntx * g.nty, ctx->nsm, g.rb);
        const FusedKernel k = tile ? pick_fused_sc(g.rb) : pick_refine(g.rb, best2 != nullptr, rows, ctas);
        k<<<std::min(ntiles, ctas * ctx->nsm), kThreads, tile ? sc_smem_bytes(g) : refine_smem_bytes(g, rows), s>>>(d, nullptr, nullptr,
                                                                                                       ntiles, nullptr);
        return cuda_error(cudaGetLastError(), "k_fused_sc / k_refine launch");
    }
    FusedKernel k = best2 ? pick_fused_b2(ctx->p.cost_dtype, g.rb, g.dc, g.wc) : pick(ctx);
    if (!k)
        return set_error(STEREO_ENOTSUP, best2 ? "the best2 output needs FP32 storage (the screened form or 12 "
                                                 "disparities per chunk) or the tensor-core form (FP16 / BF16 with bil <= 13)"
                                               : "no fused kernel for bil=%d",
                         ctx->p.bil);
    PairDesc d;
    fill_pair_desc(ctx, disp, wta, valid, d, best2);
    const int ntiles = g.ntx * g.nty;
    k<<<ntiles, fused_threads(g.wc), g.smem_bytes, s>>>(d, nullptr, nullptr, ntiles, nullptr);
    return cuda_error(cudaGetLastError(), "k_fused launch");
}

}  // namespace sgb
