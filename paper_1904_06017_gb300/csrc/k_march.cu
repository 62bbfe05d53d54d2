// k_march.cu -- the choice of a k_march instantiation and of its row segments.
#include "k_fused_common.cuh"

namespace sgb {

MarchChoice pick_march(int cost_dtype, int rb, int rw, int D)
{
    if (rb > kScMaxRB || rw < 1 || rw > kMaxRW) return MarchChoice{nullptr, 0, 0};
    switch (march_n(rb, D)) {
    case 32: return pick_march_32(cost_dtype, rb, rw);
    case 64: return pick_march_64(cost_dtype, rb, rw);
    case 96: return pick_march_96(cost_dtype, rb, rw);
    case 128: return pick_march_128(cost_dtype, rb, rw);
    }
    return MarchChoice{nullptr, 0, 0};
}

MarchChoice pick_march_rest(int cost_dtype, int rb, int rw, int D)
{
    const int d = D - march_split(rb, D);
    return cost_dtype == STEREO_F32 && march_n(rb, d) == 32 ? pick_march_32_screen(rb, rw) : pick_march(cost_dtype, rb, rw, d);
}

// A segment of nb bands takes nb + march_lead + 1 iterations (the lead fills the window, the last
// band is aggregated behind the others), and
// one CTA runs per SM: of all splits of the strips into equal segments, the one whose waves
// take the fewest iterations.
int march_bands(int W, int H, int m, int nsm)
{
    const int strips = (W + 31) / 32, bands = (H + 3) / 4, extra = march_lead(m) + 1;
    int best = bands;
    long best_t = 1l << 60;
    for (int s = 1; s <= bands; ++s) {
        const int nb = (bands + s - 1) / s, segs = (bands + nb - 1) / nb;
        const long waves = ((long)strips * segs + nsm - 1) / nsm, t = waves * (nb + extra);
        if (t < best_t) {
            best_t = t;
            best = nb;
        }
    }
    return best;
}

int march_items(int W, int H, int bands) { return (W + 31) / 32 * (((H + 3) / 4 + bands - 1) / bands); }

}  // namespace sgb
