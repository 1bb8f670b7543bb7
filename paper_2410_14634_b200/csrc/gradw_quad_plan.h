// Launch geometry of the fp32 correlation kernel of gradw_quad.cuh (host side).
#pragma once

#include <stddef.h>

namespace invconv {

struct GradWQuadPlan {
    bool ok = false;
    int T = 0, RB = 0, nbands = 0, shares = 0, NCO = 0, cotiles = 0, tiles = 0, WPT = 0, gst = 0, xst = 0, gfloats = 0, stage = 0;
    int threads = 0, grid = 0;
    size_t smem = 0;
};

// Kernel sides with an instance, and the largest tile of each (T*T*K sums per thread).
inline int gradw_quad_max_tile(int K)
{
    switch (K) {
    case 1: case 2: case 3: case 4: case 5: return 4;
    case 7: return 3;
    case 9: case 11: return 3;
    default: return 0;
    }
}

inline GradWQuadPlan plan_gradw_quad(int B, int C, int H, int W, int K, size_t max_smem, int sms)
{
    GradWQuadPlan pl;
    const int tmax = gradw_quad_max_tile(K);
    if (tmax == 0 || B < 1) return pl;
    // the tile that wastes the fewest channels, the larger one among equals
    int best = 1 << 30;
    for (int t = C < tmax ? C : tmax; t >= 1; --t) {
        const int padded = (C + t - 1) / t * t;
        const int cost = padded * padded * (t >= 3 ? 2 : (t == 2 ? 3 : 6));
        if (cost < best) { best = cost; pl.T = t; }
    }
    const int T = pl.T, LP = (K - 1 + 3) / 4 * 4;
    pl.tiles = (C + T - 1) / T;
    pl.NCO = 12 / K > 0 ? 12 / K : 1;
    if (pl.NCO > pl.tiles) pl.NCO = pl.tiles;
    pl.cotiles = (pl.tiles + pl.NCO - 1) / pl.NCO;
    pl.NCO = (pl.tiles + pl.cotiles - 1) / pl.cotiles;
    pl.WPT = 12 / (pl.NCO * K);
    if (pl.WPT < 1) pl.WPT = 1;
    pl.threads = 32 * pl.NCO * K * pl.WPT;
    const int groups = pl.tiles * pl.cotiles;
    // shares that fill the SMs once: two CTAs per SM where the sums leave registers for them
    const bool two = T * T * K <= 32;
    int want = (two ? 2 : 1) * sms / groups;
    if (want < 1) want = 1;
    pl.gst = (W + 3) & ~3;
    pl.xst = pl.gst + LP;
    if (pl.xst % 32 == 0) pl.xst += 4;
    auto fit = [&](int bands) {
        pl.RB = (H + bands - 1) / bands;
        pl.gfloats = pl.NCO * T * pl.RB * pl.gst;
        pl.stage = (pl.gfloats + T * (pl.RB + K - 1) * pl.xst + 31) & ~31;
        pl.smem = sizeof(float) * 2 * (size_t)pl.stage;
        const size_t red = sizeof(float) * (size_t)(pl.threads / 32) * T * T * K;
        if (pl.smem < red) pl.smem = red;
        pl.nbands = (H + pl.RB - 1) / pl.RB;
        const int units = B * pl.nbands;
        const int slots = want < units ? want : units, per = (units + slots - 1) / slots;
        pl.shares = (units + per - 1) / per;           // even shares
        return (double)((groups * pl.shares + sms - 1) / sms) * per * (pl.RB + K - 1 + (two ? 2 : 8));
    };
    // rows per band: the busiest SM stages and walks (CTAs there) x (units of a share) x (rows of a unit with its halo, and a
    // few rows' worth of waiting, more where no second CTA fills it).  163x3x62x62: 2, 3, 4, 5 bands cost 132, 92, 108, 90 such rows and take 27.1, 22.8, 25.5, 23.9 us;
    // 32x3x128x128: 10 bands 60 and 17.1 us, 4 to 9 bands 34 and 13.9 us.
    double best_cost = 1e30;
    int best_bands = 0;
    for (int bands = 1; bands <= H; ++bands) {
        if (bands > (H + 3) / 4 && best_bands) break;
        const double cost = fit(bands);
        if (pl.smem > (two ? max_smem / 2 : max_smem) && pl.RB > 1) continue;
        if (cost < best_cost) { best_cost = cost; best_bands = bands; }
    }
    if (!best_bands) return pl;
    fit(best_bands);
    if (pl.smem > max_smem) return pl;
    pl.grid = groups * pl.shares;
    pl.ok = true;
    return pl;
}

}  // namespace invconv
