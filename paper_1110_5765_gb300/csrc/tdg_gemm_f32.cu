// fp32 instantiations of the packed GEMM (sGEMM forms of Sec. 7).
#include "tdg_gemm.cuh"
#include "tdg_gemm_tiles.h"

namespace tdg {

// Plain fp32 products with at most half as many 128 x 128 tiles as SMs run 64 x
// 64 tiles (the same fma chain per output).
static bool small_plain(long long M, long long N) {
    using S = TilesF32;
    return 2 * ((M + S::BM - 1) / S::BM) * ((N + S::BN - 1) / S::BN) <= device_sms();
}

F32Tile f32_tile(const F32Product &p) { return f32_tile_rule(p, device_sms()); }

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

bool fallback_keeps_tile(const GemmArgs<float> &g) {
    return g.tile != F32_TILE_SMALL || small_plain(g.M, g.N);
}

template <int W, typename Big>
static cudaError_t go_asym(const GemmArgs<float> &g, const GemmOperands &ops, cudaStream_t st) {
    if (g.tile == F32_TILE_SMALL) return go<G_ASYM, W, TilesF32Small>(g, ops, st);
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
        switch (g.tile) {
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
