// How a packed fp32 product is tiled, and whether its slabs are split over CTAs
// (host code without CUDA, so that the rule can be tested by itself).
#pragma once

#include <math.h>

#include <algorithm>

namespace tdg {

// F32_TILE_BIG: 128 x 128, asymmetric W >= 3 64 x 128 (packed rows x columns);
// F32_TILE_MID (symmetric only): 128 x 64; F32_TILE_SMALL: 64 x 64
enum { F32_TILE_BIG = 0, F32_TILE_MID = 1, F32_TILE_SMALL = 2 };
struct F32Tile {
    int tile, groups;       // groups of slabs (1: not split)
};
struct F32Product {
    bool sym;
    int W, L;               // (a symmetric target's product: W = 2, whatever it asks for)
    long long mrows, ncols; // packed rows, columns
    int slabs;
    bool target;            // a distortion target's product
    bool may_split;
};

// One tile costs clocks of its SM: per k-row of a whole stage (1.5 times as many per
// row of a partial one) and at each slab's end, the latter in the asymmetric form per
// digit.  Fitted to products of 22 shapes (64 x 64 x 8192 to 3000 x 3000 x 1000), W =
// 1..4 and L = 64, 128, 256, within 10 % for nearly all; `one`: a tile alone on its SM,
// `more`: several.
struct F32Kernel {
    int tile, bm, bn, bk;
    double row_one, row_more, end_one, end_more, start_one, start_more;
};

// The SM with the most tiles sets the time.  CTAs alone on their SMs (spread_smem)
// start 1.5 to 2 us later, when the pack kernel has left the SM.  Where the tiles leave
// half of the SMs idle, groups of slabs may go to CTAs of their own (two to an SM, so
// that they all run at once); that stores every slab's packed results instead of
// unpacking them (2.9 TB/s) and, in a second kernel (6 us), reads and unpacks them
// (4 TB/s, less for asymmetric digits).  Over 476 calls in every tile (34 shapes) the
// rule's choice is 0.4 % slower than the best in the mean, 12 % at most.  Calls, us:
//   asymmetric W = 4, 2048 x 2048 x 1024, L = 256   64 x 64 102, 64 x 128 110, split 147
//   asymmetric W = 4, 1500 x 1300 x 3000, L = 128   64 x 64 147, 64 x 128 238, split 205
//   asymmetric W = 4,  512 x 512 x 4096, L = 128    64 x 64 176, 64 x 128 300, split 63
//   symmetric  W = 2, 1500 x 1500 x 1500, L = 128   128 x 128 95, 128 x 64 100, 64 x 64 110
//   symmetric  W = 2,  700 x 700 x 3000, L = 128    64 x 64 82, split 96, 128 x 64 106
inline F32Tile f32_tile_rule(const F32Product &p, int sms) {
    static const F32Kernel sym[] = {
        {F32_TILE_BIG, 128, 128, 32, 147, 134, 1600, 1220, 14000, 10000},
        {F32_TILE_MID, 128, 64, 32, 88, 80, 870, 695, 11000, 8000},
        {F32_TILE_SMALL, 64, 64, 32, 61, 50, 540, 250, 12000, 8000}};
    static const F32Kernel asym2[] = {
        {F32_TILE_BIG, 128, 128, 32, 153, 138, 1230, 1230, 14000, 10000},
        {F32_TILE_SMALL, 64, 64, 32, 59, 48, 310, 320, 12000, 8000}};
    static const F32Kernel asym4[] = {
        {F32_TILE_BIG, 64, 128, 16, 108, 85, 520, 600, 14000, 10000},
        {F32_TILE_SMALL, 64, 64, 32, 59, 48, 310, 320, 12000, 8000}};
    const F32Kernel *ks = p.sym ? sym : p.W <= 2 ? asym2 : asym4;
    const int n = p.sym ? 3 : 2;
    const double mhz = 1940.0;
    const int depth = p.sym ? (p.L + p.W - 1) / p.W : p.L;       // k-rows per slab
    const double digits = p.sym ? 1.0 : p.W;
    F32Tile best{F32_TILE_BIG, 1};
    double least = INFINITY;
    for (int i = 0; i < n; ++i) {
        const F32Kernel &k = ks[i];
        const double tiles = (double)((p.mrows + k.bm - 1) / k.bm) * (double)((p.ncols + k.bn - 1) / k.bn);
        const int rest = depth % k.bk;
        auto clocks = [&](double ctas, double slabs, double end_share) {
            const double r = ceil(ctas / sms);
            const double row = r <= 1 ? k.row_one : k.row_more;
            const double end = (r <= 1 ? k.end_one : k.end_more) * digits * end_share;
            return (r <= 1 ? k.start_one : k.start_more) +
                   r * slabs * ((depth - rest) * row + rest * 1.5 * row + end);
        };
        double t = clocks(tiles, p.slabs, 1.0);
        // where its product has 8 x 8 results a thread, a target's two other launches
        // cost 6.6 us
        if (p.target && k.bm * k.bn == 128 * 128) t += 6.6 * mhz;
        if (t < least) { least = t; best = {k.tile, 1}; }
        if (!p.may_split || k.tile == F32_TILE_MID || p.slabs < 4 || 2 * tiles > sms) continue;
        const double spg = ceil(p.slabs / std::min<double>(p.slabs, floor(2 * sms / tiles)));
        const double groups = ceil(p.slabs / spg);
        const double rbar = 4.0 * p.slabs * (double)p.mrows * (double)p.ncols;
        t = clocks(tiles * groups, spg, 1.5) +
            (rbar / 2.9e6 + rbar * (0.5 + 0.5 * digits) / 4e6 + 6.0) * mhz;
        if (groups > 1 && t < least) { least = t; best = {k.tile, (int)groups}; }
    }
    return best;
}

}  // namespace tdg
