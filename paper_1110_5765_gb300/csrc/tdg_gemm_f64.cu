// fp64 instantiations of the packed GEMM (dGEMM forms of Sec. 7), and the TMA
// box shapes every packed-GEMM launch needs.
#include "tdg_gemm.cuh"
#include "tdg_gemm_tiles.h"

namespace tdg {

// Edge of the square CTA tile for an fp64 product with mrows x ncols outputs.
// The fp64 pipe (2 fma per clock and SM) bounds every size, and one CTA keeps
// it full, so the time is that of the SM with the most outputs:
// ceil(tiles / SMs) edge^2.  Smaller tiles leave fewer SMs idle and pad less
// (64-tiles on 256 x 256: 16 of 152 SMs busy); they pay more barriers and
// fragment loads per fma, so an edge is left only for a gain above 2 %.
// Measured with edges 64 / 32 / 16: 4096^3 W = 3 38.2 / 38.2 / 38.4 ms,
// 4096 x 400 x 10304 W = 3 11.2 / 10.3 / 10.06 ms, a 256^3 W = 2 call 71 / 54 /
// 50 us (64 and 32 split its slabs over CTAs, 16 need not).
int f64_tile_edge(long long mrows, long long ncols) {
    const long long sms = device_sms();
    auto cost = [&](long long e) {
        const long long tiles = ((mrows + e - 1) / e) * ((ncols + e - 1) / e);
        return (double)((tiles + sms - 1) / sms) * (double)(e * e);
    };
    int best = 64;
    for (int e : {32, 16})
        if (cost(e) < 0.98 * cost(best)) best = e;
    return best;
}

bool fallback_keeps_tile(const GemmArgs<double> &g) {
    return f64_tile_edge(g.Mrows, g.N) == f64_tile_edge(g.M, g.N);
}

template <int FORM, int W>
static cudaError_t go(const GemmArgs<double> &g, const GemmOperands &ops, cudaStream_t st) {
    // mixed tiles (Sec. 6) keep the tile that the tile order was made for
    const int edge = g.kmask ? 64 : f64_tile_edge(g.Mrows, g.N);
    if (edge == 64) return launch_cfg<double, FORM, W, TilesF64, TilesF64>(g, ops, st);
    if (edge == 32) return launch_cfg<double, FORM, W, TilesF64Mid, TilesF64Mid>(g, ops, st);
    return launch_cfg<double, FORM, W, TilesF64Small, TilesF64Small>(g, ops, st);
}

template <>
cudaError_t launch_packed_gemm<double>(int form, int W, const GemmArgs<double> &g0,
                                       const GemmOperands &ops, cudaStream_t st) {
    if (W < 1 || W > kMaxW) return cudaErrorNotSupported;
    GemmArgs<double> g = g0;
    g.W = W;
    if (form == G_PLAIN) return go<G_PLAIN, 1>(g, ops, st);
    // the symmetric kernel is the same for every W
    if (form == G_SYM) return go<G_SYM, 1>(g, ops, st);
    if (form == G_ASYM) {
        switch (W) {
            case 1: return go<G_ASYM, 1>(g, ops, st);
            case 2: return go<G_ASYM, 2>(g, ops, st);
            case 3: return go<G_ASYM, 3>(g, ops, st);
            case 4: return go<G_ASYM, 4>(g, ops, st);
        }
    }
    return cudaErrorNotSupported;
}

// TMA boxes {BM, BK} for A and {BN, BK} for B, from the same tile table the
// launches use
void packed_gemm_boxes(int dtype, int form, int W, int *box_x_a, int *box_x_b, int *bk) {
    if (dtype == TDG_F64) {
        *box_x_a = TilesF64::BM; *box_x_b = TilesF64::BN; *bk = TilesF64::BK;
    } else if (form == G_ASYM && W <= 2) {
        *box_x_a = TilesF32AsymW2::BM; *box_x_b = TilesF32AsymW2::BN; *bk = TilesF32AsymW2::BK;
    } else if (form == G_ASYM) {
        *box_x_a = TilesF32Asym::BM; *box_x_b = TilesF32Asym::BN; *bk = TilesF32Asym::BK;
    } else {
        *box_x_a = TilesF32::BM; *box_x_b = TilesF32::BN; *bk = TilesF32::BK;
    }
}

}  // namespace tdg
