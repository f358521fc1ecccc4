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
// 64 x 64 70 / 61.  The SM with the most tiles sets the time.  Splitting the slabs
// of 128 x 128 tiles over all SMs runs 85 fma per clock and SM and moves every
// slab's packed results out and in again (2.9 TB/s, and the second kernel's 8 us).
//   1024 x 1024 x 4096  split 187 us, 128 x 64 110, 64 x 64 128
//   1000 x 777 x 1531   split  71 us, 128 x 64  46, 64 x 64  52
//    700 x 700 x 3000   split  74 us, 128 x 64  84, 64 x 64  57
//    512 x 512 x 4096   split  50 us, 128 x 64 110, 64 x 64  74
F32Tile f32_tile(long long mrows, long long ncols, long long slabs, int depth, bool wide,
                 bool may_split) {
    const double sms = device_sms(), rows = (double)slabs * depth, mhz = 1940.0;
    auto count = [&](long long bm, long long bn) {
        return (double)(((mrows + bm - 1) / bm) * ((ncols + bn - 1) / bn));
    };
    auto cost = [&](long long bm, long long bn, double one, double more) {
        const double r = ceil(count(bm, bn) / sms);
        return rows * (r <= 1 ? one : r * more);
    };
    F32Tile best{F32_TILE_128, 1};
    double t = 0.97 * cost(128, 128, 202, 177);       // the default unless clearly slower
    const double mid = cost(128, 64, 104, 96), small = cost(64, 64, 70, 61);
    if (wide && mid < t) { best = {F32_TILE_MID, 1}; t = mid; }
    if (small < t) { best = {F32_TILE_SMALL, 1}; t = small; }
    const double tiles = count(128, 128);
    if (may_split && slabs >= 4 && 2 * tiles <= sms) {
        const double rbar = 4.0 * slabs * mrows * ncols;
        const double split = 8.0 * mhz + rows * tiles * 128 * 128 / (sms * 85) +
                             2 * rbar / 2.9e6 * mhz;
        if (split < t)
            best = {F32_TILE_128, (int)std::min<double>((double)slabs, (2 * sms + tiles - 1) / tiles)};
    }
    return best;
}

// C: the packed tile; the plain fallback's by its own rule
template <int FORM, int W, typename C>
static cudaError_t go(const GemmArgs<float> &g, const GemmOperands &ops, cudaStream_t st) {
    if (g.target && g.fallback && small_plain(g.M, g.N))
        return launch_cfg<float, FORM, W, C, TilesF32Small>(g, ops, st);
    return launch_cfg<float, FORM, W, C, TilesF32>(g, ops, st);
}

// Mixed tiles (Sec. 6) keep the tile that the tile order was made for, kept or
// split slab results the 128 x 128 ones.
static int tile_of(int form, int W, const GemmArgs<float> &g) {
    if (g.kmask || g.Rbar) return F32_TILE_128;
    return f32_tile(g.Mrows, g.N, g.nK, form == G_SYM ? (g.L + W - 1) / W : g.L, form == G_SYM, false)
        .tile;
}

bool f32_target_in_one_launch(int form, int W, const GemmArgs<float> &g) {
    return g.Rbar || tile_of(form, W, g) != F32_TILE_128;
}

template <int W, typename Big>
static cudaError_t go_asym(const GemmArgs<float> &g, const GemmOperands &ops, cudaStream_t st) {
    if (tile_of(G_ASYM, W, g) == F32_TILE_SMALL) return go<G_ASYM, W, TilesF32Small>(g, ops, st);
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
        switch (tile_of(form, W, g)) {
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
