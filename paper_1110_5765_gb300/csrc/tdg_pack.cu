// Steps (a) and (b) on the data: companding and rounding (eq. 3) fused with
// packing (eqs. 6, 7, 11), both operands and every packing the planner may have
// chosen in one launch, with the de-companding factors beside them.
//
// Every element is quantized as a~ = rint(fl_T(x * c_T)) with its block's
// compander c = gamma / max|x| and the packed number is built by Horner's rule,
//     acc = d_{W-1};  acc = fma(w, acc, d_i),  i = W-2 .. 0,
// with w = z for eqs. 6 and 11 and w = z^-1 for eq. 7.  Digits outside the
// L x L block or the matrix are zero (border clean-up, Sec. 2).  P = ceil(L / W)
// packed numbers per block.
//
//   along k  out[l P + j][x]  eq. 6 for A, eq. 7 for B; W = 1 for the unpacked
//                             operands and the plain copies
//   along x  out[k][i P + j]  eq. 11, the asymmetric A
// A thread packs G consecutive numbers from whole 16-byte vectors where the
// packing direction is the contiguous one, else one vector of numbers from W
// rows.  Results that lie across the output's rows go through shared memory
// (column c of a group's member g at g * groups + c: no bank conflicts either
// way); the others are stored as vectors.
//
// The kernel reads W from the device plan: one launch serves every candidate of
// a distortion target and the plain fallback, and takes c from the block maxima
// itself.  Launched apart (companders, factors, one pack and one plain copy per
// operand, each candidate's kernels returning at entry), this step was 6 to 9
// launches and 15 to 20 us of a small product.
#include <limits.h>

#include <algorithm>

#include "tdg_common.cuh"
#include "tdg_internal.h"
#include "tdg_pack.h"

namespace tdg {

namespace {

constexpr int NT = 256;
constexpr int KSPAN = 128;          // values along the packed dimension per tile (132 for W = 3)
constexpr int PAIR_TILE = 64;       // factors per tile and side

template <typename T>
struct VecT;
template <>
struct VecT<float> { static constexpr int n = 4; };
template <>
struct VecT<double> { static constexpr int n = 2; };

template <typename T>
__device__ inline void vload(const T *p, T *o) {
    if constexpr (sizeof(T) == 4) {
        float4 v = __ldg(reinterpret_cast<const float4 *>(p));
        o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
    } else {
        double2 v = __ldg(reinterpret_cast<const double2 *>(p));
        o[0] = v.x; o[1] = v.y;
    }
}
template <typename T>
__device__ inline void vstore(T *p, const T *o) {
    if constexpr (sizeof(T) == 4) *reinterpret_cast<float4 *>(p) = make_float4(o[0], o[1], o[2], o[3]);
    else *reinterpret_cast<double2 *>(p) = make_double2(o[0], o[1]);
}

// n <= N values from p (vec: n = N and 16-byte aligned), zeros after them
template <typename T, int N>
__device__ inline void load_run(const T *p, int n, bool vec, T (&d)[N]) {
    if (vec && n >= N) {
#pragma unroll
        for (int i = 0; i < N; i += VecT<T>::n) vload(p + i, d + i);
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) d[i] = i < n ? __ldg(p + i) : T(0);
    }
}

template <typename T>
__device__ inline T quant(T v, T c, bool compand) {
    if (!compand) return v;
    if constexpr (sizeof(T) == 4) return rintf(__fmul_rn(v, c));
    else return rint(__dmul_rn(v, c));
}
template <typename T>
__device__ inline T fma_t(T a, T b, T c) {
    if constexpr (sizeof(T) == 4) return __fmaf_rn(a, b, c);
    else return __fma_rn(a, b, c);
}
template <typename T>
__device__ inline T pow2_of(int e) {
    if constexpr (sizeof(T) == 4) return scalbnf(1.0f, e);
    else return scalbn(1.0, e);
}

// How one operand is packed in this launch
template <typename T>
struct Job {
    const PackOperand<T> *o;
    T *out;
    long long ldo;
    int L, P;                 // block length and packed numbers per block
    T w;                      // Horner's weight
    bool compand, vec, vec_out;
    bool manual;
    double gamma;             // of the plan, or the manual compander itself
    long long row_end;        // rows (along k) that the product reads
    // c of the block at (x, k): the fp64 quotient rounded to T (fp32: the fp32
    // quotient has the same bits, since 53 >= 2 * 24 + 2 and gamma is an fp32 number:
    // below 2^19 for fixed bits <= 20, at most R_max / L <= 2^24 / 16 for targets)
    __device__ inline T compander(long long x, long long k) const {
        if (!compand) return T(1);
        if (manual) return (T)gamma;
        const double m = __ldg(&o->mx[x / L * o->cx + k / L * o->cl]);
        if constexpr (sizeof(T) == 4)
            return m > 0.0 ? __fdiv_rn((float)gamma, (float)m) : 0.0f;
        else
            return m > 0.0 ? __ddiv_rn(gamma, m) : 0.0;
    }
};

// packed numbers per thread along the contiguous dimension: whole vectors
template <typename T, int W>
constexpr int group_of() {
    constexpr int V = VecT<T>::n;
    return W % V == 0 ? 1 : (2 * W) % V == 0 ? 2 : 4;
}
// packed numbers a tile spans
template <typename T, int W>
constexpr int jspan() { return W == 3 ? 44 : KSPAN / W; }

template <typename T, int W, int G>
__device__ inline void horner(const T *d, T c, bool compand, T w, int n, T (&acc)[G]) {
#pragma unroll
    for (int g = 0; g < G; ++g) {
        acc[g] = W * g + W - 1 < n ? quant(d[W * g + W - 1], c, compand) : T(0);
#pragma unroll
        for (int i = W - 2; i >= 0; --i)
            acc[g] = fma_t(w, acc[g], W * g + i < n ? quant(d[W * g + i], c, compand) : T(0));
    }
}

// Packing direction contiguous in the input.  Tile: R rows of the other
// dimension from r0, numbers [j0, j0 + jspan) of block b along the packed one.
// ACROSS: numbers of a row lie across output rows (along k), staged in shared
// memory; else along them (along x).
template <typename T, int W, bool ACROSS>
__device__ __forceinline__ void pack_contig(const Job<T> &jb, long long r0, long long rows,
                                            long long ld, int b, int j0, long long len, T *s,
                                            T *cs) {
    constexpr int G = group_of<T, W>(), GV = G * W, JT = jspan<T, W>(), UPR = JT / G;
    constexpr int R = ACROSS ? (sizeof(T) == 4 ? 64 : 32) : 32;
    // units per thread, and per batch of loads issued before any is used
    constexpr int NU = (R * UPR + NT - 1) / NT, UB = GV * sizeof(T) <= 16 ? 4 : 2;
    constexpr int PITCH = JT + 1;
    static_assert(JT % G == 0, "whole groups per tile");
    const int L = jb.L, P = jb.P;
    const long long v0 = (long long)b * L + (long long)W * j0;     // first value of the tile
    const long long vlim = min((long long)(b + 1) * L, len);
    __syncthreads();                      // the tile before is stored
    if (threadIdx.x < R) {
        const long long r = r0 + threadIdx.x;
        cs[threadIdx.x] = r < rows ? (ACROSS ? jb.compander(r, (long long)b * L)
                                             : jb.compander((long long)b * L, r))
                                   : T(0);
    }
    __syncthreads();
    for (int u0 = 0; u0 < NU; u0 += UB) {
        T d[UB][GV];
        int n[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int e = threadIdx.x + (u0 + u) * NT, r = e / UPR, q = e % UPR;
            const long long v = v0 + (long long)GV * q;
            const bool in = u0 + u < NU && r < R && r0 + r < rows && v < vlim;
            n[u] = in ? (int)min((long long)GV, vlim - v) : 0;
            load_run<T, GV>(jb.o->src + (r0 + r) * ld + v, n[u], jb.vec, d[u]);
        }
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int e = threadIdx.x + (u0 + u) * NT, r = e / UPR, q = e % UPR;
            if (u0 + u >= NU || r >= R) break;
            T acc[G];
            horner<T, W, G>(d[u], cs[r], jb.compand, jb.w, n[u], acc);
            if constexpr (ACROSS) {
#pragma unroll
                for (int g = 0; g < G; ++g) s[r * PITCH + g * UPR + q] = acc[g];
            } else {
                // numbers G q .. of row r0 + r: out[k][b P + j]
                T *dst = jb.out + (r0 + r) * jb.ldo + (long long)b * P + j0 + G * q;
                if (r0 + r < rows) {
#pragma unroll
                    for (int g = 0; g < G; ++g)
                        if (j0 + G * q + g < P) dst[g] = acc[g];
                }
            }
        }
    }
    if constexpr (ACROSS) {
        __syncthreads();
        // out[b P + j][r]: lanes along r
#pragma unroll 4
        for (int e = threadIdx.x; e < JT * R; e += NT) {
            const int j = e / R, r = e % R;
            const long long row = (long long)b * P + j0 + j;
            if (j0 + j >= P || r0 + r >= rows || row >= jb.row_end) continue;
            jb.out[row * jb.ldo + r0 + r] = s[r * PITCH + j % G * UPR + j / G];
        }
    }
}

// Packing direction across the input's rows: a thread takes VEC contiguous
// columns from W rows.  Tile: 32 VEC columns from c0, numbers [j0, j0 + JT).
// ACROSS: out[k][b P + j] with the columns k (along x), staged; else out[b P +
// j][x] with the columns x (along k).
template <typename T, int W, bool ACROSS>
__device__ __forceinline__ void pack_rows(const Job<T> &jb, long long c0, long long cols,
                                          long long ld, int b, int j0, long long len, T *s,
                                          T *cs) {
    constexpr int V = VecT<T>::n, CT = 32 * V, JT = ACROSS ? 32 : jspan<T, W>();
    constexpr int JW = (JT + 7) / 8;                 // numbers per warp
    constexpr int UB = W == 1 ? 8 : W == 2 ? 4 : 2;
    constexpr int PITCH = 33;
    const int L = jb.L, P = jb.P, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (threadIdx.x < CT / 16) {                     // blocks are multiples of 16 long
        const long long c = c0 + 16 * threadIdx.x;
        cs[threadIdx.x] = c < cols ? (ACROSS ? jb.compander((long long)b * L, c)
                                             : jb.compander(c, (long long)b * L))
                                   : T(0);
    }
    __syncthreads();
    const T c = cs[V * lane / 16];
    const long long col = c0 + V * lane;
    const int left = (int)max(0LL, min((long long)V, cols - col));
    const long long vbase = (long long)b * L, vlim = min(vbase + L, len);
    for (int u0 = 0; u0 < JW; u0 += UB) {
        T d[UB][W][V];
#pragma unroll
        for (int u = 0; u < UB; ++u)
#pragma unroll
            for (int i = 0; i < W; ++i) {
                const int j = j0 + warp + 8 * (u0 + u);
                const long long v = vbase + (long long)W * j + i;
                const bool in = u0 + u < JW && j < P && v < vlim;
                load_run<T, V>(jb.o->src + v * ld + col, in ? left : 0, jb.vec, d[u][i]);
            }
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int jt = warp + 8 * (u0 + u), j = j0 + jt;
            if (u0 + u >= JW || jt >= JT || j >= P) break;
            T acc[V];
#pragma unroll
            for (int e = 0; e < V; ++e) {
                // (a digit outside is zero, also where c is not finite)
                const long long v = vbase + (long long)W * j;
                acc[e] = v + W - 1 < vlim ? quant(d[u][W - 1][e], c, jb.compand) : T(0);
#pragma unroll
                for (int i = W - 2; i >= 0; --i)
                    acc[e] = fma_t(jb.w, acc[e],
                                   v + i < vlim ? quant(d[u][i][e], c, jb.compand) : T(0));
            }
            if constexpr (ACROSS) {
#pragma unroll
                for (int e = 0; e < V; ++e) s[(e * 32 + lane) * PITCH + jt] = acc[e];
            } else {
                const long long row = (long long)b * P + j;
                if (row >= jb.row_end) break;
                T *dst = jb.out + row * jb.ldo + col;
                if (jb.vec_out && left == V) {
                    vstore(dst, acc);
                } else {
#pragma unroll
                    for (int e = 0; e < V; ++e)
                        if (e < left) dst[e] = acc[e];
                }
            }
        }
    }
    if constexpr (ACROSS) {
        __syncthreads();
#pragma unroll 4
        for (int e = threadIdx.x; e < CT * JT; e += NT) {
            const int k = e / JT, j = e % JT;
            if (j0 + j >= P || c0 + k >= cols) continue;
            jb.out[(c0 + k) * jb.ldo + (long long)b * P + j0 + j] =
                s[(k % V * 32 + k / V) * PITCH + j];
        }
    }
}

// Tiles of one operand: t = (other-dimension tile) + count * (block chunk)
template <typename T>
struct TileGrid {
    unsigned int other, chunks, nblk;      // other-dimension tiles, chunks per block, blocks
    int jt, span;                          // numbers and other-dimension values per tile
    __device__ inline unsigned int tiles() const { return other * chunks * nblk; }
};
template <typename T, int W>
__device__ inline TileGrid<T> tile_grid(const PackOperand<T> &o, bool along_k, int L, int P) {
    const bool contig = along_k ? o.sk == 1 && o.sx != 1 : o.sx == 1;
    const bool across = along_k == contig;
    TileGrid<T> g;
    const long long oth = along_k ? o.X : o.K, len = along_k ? o.K : o.X;
    g.span = contig ? (across ? (sizeof(T) == 4 ? 64 : 32) : 32) : 32 * VecT<T>::n;
    g.jt = !contig && across ? 32 : jspan<T, W>();
    g.other = (unsigned int)((oth + g.span - 1) / g.span);
    g.chunks = (unsigned int)((P + g.jt - 1) / g.jt);
    g.nblk = (unsigned int)((len + L - 1) / L);
    return g;
}

template <typename T, int W, bool ALONG_K>
__device__ __forceinline__ void pack_tile(const Job<T> &jb, const TileGrid<T> &g, unsigned int t,
                                          T *s, T *cs) {
    const PackOperand<T> &o = *jb.o;
    const unsigned int r = t / g.other, b = r / g.chunks;
    const long long base = (long long)(t - r * g.other) * g.span;
    const int j0 = (int)(r - b * g.chunks) * g.jt;
    // contiguous dimension: k when sk = 1 (and x is not), else x
    if constexpr (ALONG_K) {
        if (o.sk == 1 && o.sx != 1) pack_contig<T, W, true>(jb, base, o.X, o.sx, (int)b, j0, o.K, s, cs);
        else pack_rows<T, W, false>(jb, base, o.X, o.sk, (int)b, j0, o.K, s, cs);
    } else {
        if (o.sx == 1) pack_contig<T, W, false>(jb, base, o.K, o.sk, (int)b, j0, o.X, s, cs);
        else pack_rows<T, W, true>(jb, base, o.K, o.sx, (int)b, j0, o.X, s, cs);
    }
}

// the de-companding factors (T)(s_A,il s_B,lj), s = 1/c in fp64, of one slab and
// a PAIR_TILE x PAIR_TILE tile of block pairs
template <typename T>
__device__ __forceinline__ void pair_tile(const PackArgs<T> &a, const DevPlan *plan, unsigned int t,
                                          double *s) {
    const unsigned int tn = (unsigned int)((a.nN + PAIR_TILE - 1) / PAIR_TILE);
    const unsigned int tm = (unsigned int)((a.nM + PAIR_TILE - 1) / PAIR_TILE);
    const unsigned int l = t / (tm * tn), r = t % (tm * tn);
    const int i0 = (int)(r / tn) * PAIR_TILE, j0 = (int)(r % tn) * PAIR_TILE;
    if (threadIdx.x < 2 * PAIR_TILE) {
        const bool isA = threadIdx.x < PAIR_TILE;
        const int e = isA ? i0 + threadIdx.x : j0 + threadIdx.x - PAIR_TILE;
        double v = 0.0;
        if (e < (isA ? a.nM : a.nN)) {
            const PackOperand<T> &o = isA ? a.A : a.B;
            double c;
            if (a.manual) {
                c = isA ? a.manual_cA : a.manual_cB;
            } else {
                const double m = __ldg(&o.mx[e * o.cx + l * o.cl]);
                c = m > 0.0 ? __ddiv_rn((double)(isA ? plan->gA : plan->gB), m) : 0.0;
            }
            v = c > 0.0 ? __ddiv_rn(1.0, c) : 0.0;
        }
        s[threadIdx.x] = v;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < PAIR_TILE * PAIR_TILE; e += NT) {
        const int i = e / PAIR_TILE, j = e % PAIR_TILE;
        if (i0 + i < a.nM && j0 + j < a.nN)
            a.pair[((long long)l * a.nM + i0 + i) * a.nN + j0 + j] =
                (T)__dmul_rn(s[i], s[PAIR_TILE + j]);
    }
    __syncthreads();
}

// The CTAs take the factor tiles first, then tiles of A and B in turn (A's
// transposing pack is bound by issue, B's by latency, in the row-major case),
// last tiles first: the statistics read op(A) and then op(B) front to back, so
// the ends are in L2.
template <typename T, int WA, int WB, bool A_ALONG_K>
__device__ __forceinline__ void pack_both(const PackArgs<T> &a, const DevPlan *plan, bool compand,
                                          T *s, T *cs) {
    const int q = plan->q;
    auto job = [&](const PackOperand<T> &o, T *out, long long ldo, int W, bool isA) {
        Job<T> j;
        j.o = &o;
        j.out = out;
        j.ldo = ldo;
        j.L = compand ? a.L : KSPAN;         // plain copies: any block length will do
        j.P = (j.L + W - 1) / W;
        j.w = W > 1 ? pow2_of<T>(isA ? -q : q) : T(1);
        j.compand = compand;
        j.manual = a.manual != 0;
        // unpacked rows end with k; packed slabs are read to their last number
        j.row_end = A_ALONG_K && compand ? LLONG_MAX : o.K;
        j.gamma = a.manual ? (isA ? a.manual_cA : a.manual_cB) : (double)(isA ? plan->gA : plan->gB);
        constexpr int V = VecT<T>::n;
        j.vec = (reinterpret_cast<uintptr_t>(o.src) & 15) == 0 && (o.sk == 1 ? o.sx : o.sk) % V == 0;
        j.vec_out = (reinterpret_cast<uintptr_t>(out) & 15) == 0 && ldo % V == 0;
        return j;
    };
    const Job<T> ja = job(a.A, a.outA, a.ldoA[compand ? WA : 0], WA, true);
    const Job<T> jbb = job(a.B, a.outB, a.ldoB, WB, false);
    TileGrid<T> ga = tile_grid<T, WA>(a.A, A_ALONG_K, ja.L, ja.P);
    TileGrid<T> gb = tile_grid<T, WB>(a.B, true, jbb.L, jbb.P);
    const bool skipA = a.skipA || (!compand && a.directA), skipB = a.skipB || (!compand && a.directB);
    const unsigned int nA = skipA ? 0u : ga.tiles(), nB = skipB ? 0u : gb.tiles();
    const unsigned int np = compand ? (unsigned int)a.pair_tiles : 0u, both = 2 * min(nA, nB);
    for (unsigned int t = blockIdx.x; t < np + nA + nB; t += a.log_cta) {
        if (t < np) {
            pair_tile(a, plan, t, reinterpret_cast<double *>(s));
            continue;
        }
        const unsigned int v = t - np;
        const bool isA = v < both ? (v & 1) != 0 : nA > nB;
        const unsigned int w = v < both ? v >> 1 : v - both / 2;
        if (isA) pack_tile<T, WA, A_ALONG_K>(ja, ga, nA - 1 - w, s, cs);
        else pack_tile<T, WB, true>(jbb, gb, nB - 1 - w, s, cs);
    }
}

template <typename T, bool ASYM>
__global__ void __launch_bounds__(NT, 4) pack_kernel(const __grid_constant__ PackArgs<T> a,
                                                     DevPlan *plan) {
    pdl_entry();
    // staging: the largest tile is 64 (fp32) or 32 (fp64) rows of KSPAN numbers
    __shared__ __align__(16) unsigned char raw[(sizeof(T) == 4 ? 64 : 32) * (KSPAN + 1) * sizeof(T)];
    __shared__ T cs[64];
    T *s = reinterpret_cast<T *>(raw);
    if (blockIdx.x == a.log_cta) {
        // the predicted SNR of a target's plan, which only the host reads
        if (threadIdx.x == 0 && plan->log_pending) plan->pred_snr = 10.0 * log10(plan->ratio);
        return;
    }
    const int W = a.plain ? 1 : plan->W;
    // W = 1 from the planner of a distortion target is the conventional product
    if (a.plain || (W == 1 && a.target)) {
        pack_both<T, 1, 1, true>(a, plan, false, s, cs);
        return;
    }
    if (a.plain_only) return;         // (pair-exact tiles are packed by the product itself)
    if constexpr (ASYM) {
        switch (W) {
            case 1: pack_both<T, 1, 1, false>(a, plan, true, s, cs); break;
            case 2: pack_both<T, 2, 1, false>(a, plan, true, s, cs); break;
            case 3: pack_both<T, 3, 1, false>(a, plan, true, s, cs); break;
            case 4: pack_both<T, 4, 1, false>(a, plan, true, s, cs); break;
        }
    } else {
        switch (W) {
            case 1: pack_both<T, 1, 1, true>(a, plan, true, s, cs); break;
            case 2: pack_both<T, 2, 2, true>(a, plan, true, s, cs); break;
            case 3: pack_both<T, 3, 3, true>(a, plan, true, s, cs); break;
            case 4: pack_both<T, 4, 4, true>(a, plan, true, s, cs); break;
        }
    }
}

}  // namespace

template <typename T>
cudaError_t launch_pack(bool asym, const PackArgs<T> &a0, DevPlan *plan, cudaStream_t st) {
    PackArgs<T> a = a0;
    const long long tm = (a.nM + PAIR_TILE - 1) / PAIR_TILE, tn = (a.nN + PAIR_TILE - 1) / PAIR_TILE;
    const long long np = a.pair ? tm * tn * a.nK : 0;
    // an upper bound of the tiles over every packing (32 values by 16 numbers)
    auto bound = [&](const PackOperand<T> &o) {
        return ((o.X + 31) / 32) * ((o.K + std::min(a.L, KSPAN) - 1) / std::min(a.L, KSPAN) + 1) +
               ((o.K + 31) / 32) * ((o.X + 31) / 32 + 1);
    };
    if (np > 0x3fffffffLL || bound(a.A) > 0x3fffffffLL || bound(a.B) > 0x3fffffffLL)
        return cudaErrorInvalidConfiguration;
    a.pair_tiles = (int)np;
    // a resident wave (four CTAs fit an SM), or less for small operands
    const long long want = np + (a.skipA ? 0 : bound(a.A)) + (a.skipB ? 0 : bound(a.B));
    a.log_cta = (unsigned int)std::max(1LL, std::min(want, 4LL * device_sms()));
    const unsigned int grid = a.log_cta + (a.target && !a.plain ? 1 : 0);
    return asym ? launch_pdl(pack_kernel<T, true>, dim3(grid), dim3(NT), 0, st, a, plan)
                : launch_pdl(pack_kernel<T, false>, dim3(grid), dim3(NT), 0, st, a, plan);
}

template cudaError_t launch_pack<float>(bool, const PackArgs<float> &, DevPlan *, cudaStream_t);
template cudaError_t launch_pack<double>(bool, const PackArgs<double> &, DevPlan *, cudaStream_t);

}  // namespace tdg
