// fp32 instantiations of the packed GEMM (sGEMM forms of Sec. 7).
#include <math.h>

#include <algorithm>

#include "tdg_gemm.cuh"
#include "tdg_gemm_tiles.h"

namespace tdg {

// Plain fp32 products with at most half as many 128 x 128 tiles as SMs run 64 x
// 64 tiles (the same fma chain per output).
static bool small_plain(long long M, long long N) {
    using S = TilesF32;
    return 2 * ((M + S::BM - 1) / S::BM) * ((N + S::BN - 1) / S::BN) <= device_sms();
}

// How a packed fp32 product over `slabs` slabs of `depth` k-rows is tiled.  A tile
// costs clocks per k-row of its SM, measured with the symmetric kernel (K = 1024
// to 4096; one tile on an SM / several): 128 x 128 202 / 177, 128 x 64 104 / 96,
// 64 x 64 70 / 61.  The SM with the most tiles sets the time.  Where even the
// smallest tiles leave SMs idle, groups of slabs go to CTAs of their own (two to
// an SM, so that they all run at once); that moves every slab's packed results out
// (2.9 TB/s) and, in a second kernel (5 us), in again (4 TB/s).
//   1024 x 1024 x 4096  split 187 us, 128 x 64 110, 64 x 64 128
//   1000 x 777 x 1531   split  71 us, 128 x 64  46, 64 x 64  52
//    700 x 700 x 3000   split  74 us, 128 x 64  84, 64 x 64  57
//    512 x 512 x 4096   split  50 us, 128 x 64 110, 64 x 64  74
F32Tile f32_tile(long long mrows, long long ncols, long long slabs, int depth, bool sym,
                 bool target, bool may_split) {
    const double sms = device_sms(), mhz = 1940.0;
    struct Shape { int tile; long long bm, bn; double one, more; };
    static const Shape shapes[] = {{F32_TILE_128, 128, 128, 202, 177},
                                   {F32_TILE_MID, 128, 64, 104, 96},
                                   {F32_TILE_SMALL, 64, 64, 70, 61}};
    F32Tile best{F32_TILE_128, 1};
    double least = INFINITY;
    for (const Shape &s : shapes) {
        if (s.tile == F32_TILE_MID && !sym) continue;
        const double tiles = (double)((mrows + s.bm - 1) / s.bm) * ((ncols + s.bn - 1) / s.bn);
        auto clocks = [&](double ctas, double rows) {
            const double r = ceil(ctas / sms);
            return rows * (r <= 1 ? s.one : r * s.more);
        };
        double t = clocks(tiles, (double)slabs * depth);
        // the default unless clearly slower; a target's two other launches cost 6.6 us
        if (s.tile == F32_TILE_128) t = 0.97 * t + (target ? 6.6 * mhz : 0.0);
        if (t < least) { least = t; best = {s.tile, 1}; }
        if (!may_split || s.tile == F32_TILE_MID || slabs < 4 || 2 * tiles > sms) continue;
        const double spg = ceil(slabs / std::min<double>((double)slabs, floor(2 * sms / tiles)));
        const double groups = ceil(slabs / spg), rbar = 4.0 * slabs * mrows * ncols;
        t = clocks(tiles * groups, spg * depth) +
            (rbar / 2.9e6 + rbar / 4e6 + 5.0) * mhz;
        if (groups > 1 && t < least) { least = t; best = {s.tile, (int)groups}; }
    }
    return best;
}

// C: the packed tile; the plain fallback's by its own rule, but for 64 x 64 tiles,
// whose registers (three CTAs per SM) hold no larger one
template <int FORM, int W, typename C>
static cudaError_t go(const GemmArgs<float> &g, const GemmOperands &ops, cudaStream_t st) {
    if constexpr (C::TM * C::TN > 16) {
        if (!(g.target && g.fallback && small_plain(g.M, g.N)))
            return launch_cfg<float, FORM, W, C, TilesF32>(g, ops, st);
    }
    return launch_cfg<float, FORM, W, C, TilesF32Small>(g, ops, st);
}

// Mixed tiles (Sec. 6) keep the tile that the tile order was made for, kept slab
// results the 128 x 128 ones.
static int tile_of(int form, int W, const GemmArgs<float> &g, bool target) {
    if (g.kmask || (g.Rbar && g.groups <= 1)) return F32_TILE_128;
    return f32_tile(g.Mrows, g.N, g.nK, form == G_SYM ? (g.L + W - 1) / W : g.L, form == G_SYM,
                    target, g.groups > 1)
        .tile;
}

bool f32_target_in_one_launch(int form, int W, const GemmArgs<float> &g) {
    return g.Rbar || tile_of(form, W, g, true) != F32_TILE_128;
}

bool fallback_keeps_tile(int form, int W, const GemmArgs<float> &g) {
    return tile_of(form, W, g, true) != F32_TILE_SMALL || small_plain(g.M, g.N);
}

template <int W, typename Big>
static cudaError_t go_asym(const GemmArgs<float> &g, const GemmOperands &ops, cudaStream_t st) {
    if (tile_of(G_ASYM, W, g, g.small_t < 0) == F32_TILE_SMALL) return go<G_ASYM, W, TilesF32Small>(g, ops, st);
    return go<G_ASYM, W, Big>(g, ops, st);
}

template <>
cudaError_t launch_packed_gemm<float>(int form, int W, const GemmArgs<float> &g0,
                                      const GemmOperands &ops, cudaStream_t st) {
    if (W < 1 || W > kMaxW) return cudaErrorNotSupported;
    GemmArgs<float> g = g0;
    g.W = W;
    if (form == G_PLAIN) {
        if (small_plain(g.M, g.N))
            return launch_cfg<float, G_PLAIN, 1, TilesF32Small, TilesF32Small>(g, ops, st);
        return launch_cfg<float, G_PLAIN, 1, TilesF32, TilesF32>(g, ops, st);
    }
    if (form == G_SYM) {
        // the symmetric kernel is the same for every W
        switch (tile_of(form, W, g, g.small_t < 0)) {
            case F32_TILE_MID: return go<G_SYM, 1, TilesF32Mid>(g, ops, st);
            case F32_TILE_SMALL: return go<G_SYM, 1, TilesF32Small>(g, ops, st);
            default: return go<G_SYM, 1, TilesF32>(g, ops, st);
        }
    }
    if (form == G_ASYM) {
        switch (W) {
            case 1: return go_asym<1, TilesF32AsymW2>(g, ops, st);
            case 2: return go_asym<2, TilesF32AsymW2>(g, ops, st);
            case 3: return go_asym<3, TilesF32Asym>(g, ops, st);
            case 4: return go_asym<4, TilesF32Asym>(g, ops, st);
        }
    }
    return cudaErrorNotSupported;
}

}  // namespace tdg
