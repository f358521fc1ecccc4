// Codes of the tensor-core forms: out[x][k], k contiguous, as integer-valued
// fp16 (rint(x c), eq. 3) or E4M3 (round to nearest even, saturating), with the
// companders c = gamma / max|x| of each L x L block of op(X).
//
// One CTA of 512 threads per SM (two for 64-tiles) walks its share of TS x TS
// tiles; three tiles are in flight to shared memory by cp.async (two between the
// wait for a tile and the refill of its stage), so the memory system sees 64 to 192
// KB of outstanding reads per SM whatever the phase.  HBM bounds the kernel: it reads 4
// bytes and writes 2 or 1 per value once.
//   FUSED   companders that depend on their own block only (fixed bits, E4M3)
//           with L = TS: the tile is a block; its maximum (and, for the integer
//           form, whose predicted SNR needs it, its sum of squares) is taken
//           from the same read.
//   else    the statistics pass has run (target mode, L > 128): c from the
//           block maxima and the plan's gammas.  Tiles are walked backwards: the
//           statistics read op(A) and then op(B), so the last ones are in L2.
// c is __fdiv_rn of two fp32 numbers (gamma <= 2048): the fp64 quotient rounded to
// fp32 has the same bits, since 53 >= 2 * 24 + 2.
// Shared-memory layout: rows of TS values as stored, 16-byte chunks permuted
// within the row so that the reads below have no bank conflicts.
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>

#include "tdg_common.cuh"
#include "tdg_internal.h"
#include "tdg_optin.h"
#include "tdg_planner.cuh"

namespace tdg {

namespace {

constexpr int STAGES = 3, THREADS = 512, WARPS = THREADS / 32;
constexpr int kMaxTiles = 1 << 30;      // per operand (2^42 values: 16 TB)

struct CodesOp {
    const float *p;
    long long sx, sk, X, K;
    int kt, tiles;                  // tiles along k, all tiles
    long long cx, cl;               // block (bx, bk) has index bx cx + bk cl in mx, var, s
    double *mx, *var, *s;
    unsigned char *out;
};

__device__ inline void cp_async16(uint32_t dst, const float *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ inline void cp_async4(uint32_t dst, const float *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ inline void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// 16 bytes of codes: 8 integer-valued fp16 (|v| <= 2049, so adding and
// subtracting 1.5 2^23 rounds to the nearest integer, ties to even) or 16 E4M3
__device__ inline uint4 encode(const float (&v)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float a = __fsub_rn(__fadd_rn(v[2 * i], 12582912.0f), 12582912.0f);
        const float b = __fsub_rn(__fadd_rn(v[2 * i + 1], 12582912.0f), 12582912.0f);
        const __half2 h = __floats2half2_rn(a, b);
        w[i] = *reinterpret_cast<const uint32_t *>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ inline uint4 encode(const float (&v)[16]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(v[4 * i], v[4 * i + 1]),
                                                     __NV_SATFINITE, __NV_E4M3);
        const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(v[4 * i + 2], v[4 * i + 3]),
                                                     __NV_SATFINITE, __NV_E4M3);
        w[i] = lo | (hi << 16);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// (hi, lo) += (bh, bl): TwoSum of the high parts, renormalised
__device__ inline void df_add(float &hi, float &lo, float bh, float bl) {
    const float s = __fadd_rn(hi, bh);
    const float v = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, v)), __fsub_rn(bh, v));
    const float t = __fadd_rn(e, __fadd_rn(lo, bl));
    hi = __fadd_rn(s, t);
    lo = __fsub_rn(t, __fsub_rn(hi, s));
}
// exact square as hi + err (TwoProduct), TwoSum into (hi, lo)
__device__ inline void df_add_sq(float &hi, float &lo, float x) {
    const float p = __fmul_rn(x, x);
    const float e = __fmaf_rn(x, x, -p);
    const float t = __fadd_rn(hi, p);
    const float bp = __fsub_rn(t, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bp)), __fsub_rn(p, bp));
    hi = t;
    lo = __fadd_rn(lo, __fadd_rn(err, e));
}

template <int FP8, int TS, bool FUSED>
__global__ void __launch_bounds__(THREADS, TS == 128 ? 1 : 2)
    codes_kernel(CodesOp A, CodesOp B, int L, double gamma, long long ldo, DevPlan *plan,
                 const __grid_constant__ SlabFinish fin) {
    pdl_entry();
    constexpr int KV = FP8 ? 16 : 8;                 // values per 16 bytes of codes
    constexpr int ES = FP8 ? 1 : 2;
    constexpr int NV = TS * TS / THREADS, NI = NV / KV;   // values and code items per thread
    constexpr int CH = TS / 4;                       // 16-byte chunks of a stored row
    constexpr int GP = TS / KV;                      // items per row of codes
    extern __shared__ __align__(128) unsigned char smem[];
    float *ring = reinterpret_cast<float *>(smem);
    __shared__ float red_h[2][WARPS], red_l[2][WARPS];
    __shared__ unsigned int red_m[2][WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned int total = (unsigned int)(A.tiles + B.tiles), step = gridDim.x;

    // tile i of the walk: its operand and origin.  (32-bit division, and only
    // one per tile: with 64-bit indices the divisions were half of the
    // kernel's instructions.)
    struct Tile {
        int xt, kt;                  // tile coordinates
        bool isA;
    };
    auto tile = [&](unsigned int i) {
        unsigned int t = FUSED ? i : total - 1 - i;
        Tile r;
        r.isA = t < (unsigned int)A.tiles;
        if (!r.isA) t -= (unsigned int)A.tiles;
        const unsigned int kt = (unsigned int)(r.isA ? A.kt : B.kt);
        r.xt = (int)(t / kt);
        r.kt = (int)(t - (unsigned int)r.xt * kt);
        return r;
    };
    // chunk permutations (see the reads): k-contiguous rows by the chunk
    // itself, x-contiguous rows by the row's k group
    auto phys_k = [](int ch) { return ch ^ ((ch >> 3) & (KV / 4 - 1)); };
    auto phys_x = [](int ch, int k) { return ch ^ (((k / KV) & 3) << 1); };
    auto fetch = [&](unsigned int i, const Tile &tl, int stage) {
        if (i < total) {
            const CodesOp &o = tl.isA ? A : B;
            const bool kc = o.sk == 1;
            const long long ld = kc ? o.sx : o.sk;
            const long long r0 = (long long)(kc ? tl.xt : tl.kt) * TS;
            const long long c0 = (long long)(kc ? tl.kt : tl.xt) * TS;
            const int rn = (int)min((long long)TS, (kc ? o.X : o.K) - r0);
            const int cn = (int)min((long long)TS, (kc ? o.K : o.X) - c0);
            const float *src = o.p + r0 * ld + c0;
            const uint32_t dst = smem_u32(ring + (size_t)stage * TS * TS);
            if (((reinterpret_cast<uintptr_t>(o.p) & 15) == 0) && (ld & 3) == 0) {
                constexpr int RS = THREADS / CH;         // rows between a thread's chunks
                const int r1 = tid / CH, ch = tid % CH;
                const float *q = src + r1 * ld + 4 * ch;
                const int cbytes = max(0, min(16, 4 * (cn - 4 * ch)));
                const uint32_t dk = dst + (uint32_t)(r1 * TS + 4 * phys_k(ch)) * 4;
#pragma unroll
                for (int u = 0; u < NV / 4; ++u) {
                    const int r = r1 + u * RS;
                    const int bytes = r < rn ? cbytes : 0;
                    const uint32_t d = kc ? dk + (uint32_t)(u * RS * TS) * 4
                                          : dst + (uint32_t)(r * TS + 4 * phys_x(ch, r)) * 4;
                    cp_async16(d, bytes ? q : o.p, bytes);
                    q += RS * ld;
                }
            } else {
#pragma unroll 4
                for (int u = 0; u < NV; ++u) {
                    const int e = tid + u * THREADS, r = e / TS, c = e % TS;
                    const int bytes = r < rn && c < cn ? 4 : 0;
                    const int pc = kc ? phys_k(c / 4) : phys_x(c / 4, r);
                    cp_async4(dst + (uint32_t)(r * TS + 4 * pc + c % 4) * 4,
                              bytes ? src + r * ld + c : o.p, bytes);
                }
            }
        }
        cp_async_commit();
    };

    const double gA = FUSED ? gamma : (double)plan->gA, gB = FUSED ? gamma : (double)plan->gB;
    const float gmA = (float)gA, gmB = (float)gB;
    const unsigned int ratio = (unsigned int)(L / TS);       // tiles per block along x and k
    Tile ahead[STAGES];                                      // the tiles in flight
#pragma unroll
    for (int s = 0; s < STAGES; ++s) {
        ahead[s] = tile(blockIdx.x + s * step);
        fetch(blockIdx.x + s * step, ahead[s], s);
    }
    int stage = 0;
    int it = 0;
    for (unsigned int i = blockIdx.x; i < total; i += step, ++it) {
        const Tile tl = ahead[0];
        const CodesOp &o = tl.isA ? A : B;
        const bool kc = o.sk == 1;
        const long long x0 = (long long)tl.xt * TS;
        const int k0 = tl.kt * TS;
        const long long idx = (FUSED ? tl.xt : (int)((unsigned int)tl.xt / ratio)) * o.cx +
                              (FUSED ? tl.kt : (int)((unsigned int)tl.kt / ratio)) * o.cl;
        float m = FUSED ? 0.f : (float)__ldg(&o.mx[idx]);
        cp_async_wait<STAGES - 1>();
        __syncthreads();
        const float *t = ring + (size_t)stage * TS * TS;
        // item u of this thread: KV consecutive k from kr of row xr
        float v[NI][KV];
        auto item = [&](int u, int &xr, int &kr) {
            const int e = tid + u * THREADS;
            if (kc) {
                xr = e / GP;
                kr = e % GP * KV;
            } else {                 // 8 rows x 4 k groups per warp
                const int g = e >> 5;
                xr = g % (TS / 8) * 8 + (lane & 7);
                kr = (g / (TS / 8) * 4 + (lane >> 3)) * KV;
            }
        };
#pragma unroll
        for (int u = 0; u < NI; ++u) {
            int xr, kr;
            item(u, xr, kr);
            if (kc) {
#pragma unroll
                for (int q = 0; q < KV / 4; ++q) {
                    const float4 a =
                        *reinterpret_cast<const float4 *>(t + xr * TS + 4 * phys_k(kr / 4 + q));
                    v[u][4 * q] = a.x; v[u][4 * q + 1] = a.y;
                    v[u][4 * q + 2] = a.z; v[u][4 * q + 3] = a.w;
                }
            } else {
                const float *col = t + kr * TS + 4 * phys_x(xr / 4, kr) + (xr & 3);
#pragma unroll
                for (int q = 0; q < KV; ++q) v[u][q] = col[q * TS];
            }
        }
        if constexpr (FUSED) {
            unsigned int mb = 0;
            float hi[2] = {0.f, 0.f}, lo[2] = {0.f, 0.f};
#pragma unroll
            for (int u = 0; u < NI; ++u)
#pragma unroll
                for (int q = 0; q < KV; ++q) {
                    mb = max(mb, __float_as_uint(v[u][q]) & 0x7fffffffu);
                    if constexpr (!FP8) df_add_sq(hi[q & 1], lo[q & 1], v[u][q]);
                }
            mb = __reduce_max_sync(0xffffffffu, mb);
            if constexpr (!FP8) {
                df_add(hi[0], lo[0], hi[1], lo[1]);
#pragma unroll
                for (int off = 16; off > 0; off >>= 1)
                    df_add(hi[0], lo[0], __shfl_xor_sync(0xffffffffu, hi[0], off),
                           __shfl_xor_sync(0xffffffffu, lo[0], off));
            }
            const int set = it & 1;
            if (lane == 0) {
                red_m[set][warp] = mb;
                red_h[set][warp] = hi[0];
                red_l[set][warp] = lo[0];
            }
            __syncthreads();         // the tile is read by all: its stage may be refilled
            mb = __reduce_max_sync(0xffffffffu, red_m[set][lane & (WARPS - 1)]);
            m = __uint_as_float(mb);
            if (warp == 0) {
                float h = 0.f, l = 0.f;
                if constexpr (!FP8) {
                    h = lane < WARPS ? red_h[set][lane] : 0.f;
                    l = lane < WARPS ? red_l[set][lane] : 0.f;
#pragma unroll
                    for (int off = WARPS / 2; off > 0; off >>= 1)
                        df_add(h, l, __shfl_xor_sync(0xffffffffu, h, off),
                               __shfl_xor_sync(0xffffffffu, l, off));
                }
                if (lane == 0) {
                    o.mx[idx] = (double)m;
                    if constexpr (!FP8) {
                        const int bxn = (int)min((long long)TS, o.X - x0);
                        const int bkn = (int)min((long long)TS, o.K - k0);
                        o.var[idx] = ((double)h + (double)l) / ((double)bxn * (double)bkn);
                    }
                    if (mb >= 0x7f800000u) atomicExch(fin.nonfinite, 1);
                }
            }
        } else {
            __syncthreads();
        }
#pragma unroll
        for (int s = 0; s + 1 < STAGES; ++s) ahead[s] = ahead[s + 1];
        ahead[STAGES - 1] = tile(i + STAGES * step);
        fetch(i + STAGES * step, ahead[STAGES - 1], stage);
        if (++stage == STAGES) stage = 0;
        const int xn = (int)min((long long)TS, o.X - x0);
        unsigned char *out = o.out + (x0 * ldo + k0) * ES;
        const float c = m > 0.f ? __fdiv_rn(tl.isA ? gmA : gmB, m) : 0.f;
#pragma unroll
        for (int u = 0; u < NI; ++u) {
            int xr, kr;
            item(u, xr, kr);
            if (xr >= xn) continue;
#pragma unroll
            for (int q = 0; q < KV; ++q) v[u][q] = __fmul_rn(v[u][q], c);
            *reinterpret_cast<uint4 *>(out + (xr * ldo + kr) * ES) = encode(v[u]);
        }
    }
    cp_async_wait<0>();
    __syncthreads();
    // s = 1/c in fp64 for the de-companding, one thread per block; then the
    // blocks are counted (slab_finish), one warp each
    for (unsigned int i = blockIdx.x + tid * step; i < total; i += THREADS * step) {
        const Tile tl = tile(i);
        if ((unsigned int)tl.xt % ratio || (unsigned int)tl.kt % ratio) continue;   // a block's first tile
        const CodesOp &o = tl.isA ? A : B;
        const long long idx = (tl.xt / (int)ratio) * o.cx + (tl.kt / (int)ratio) * o.cl;
        const double m = __ldcg(&o.mx[idx]);
        const double c = m > 0.0 ? __ddiv_rn(tl.isA ? gA : gB, m) : 0.0;
        o.s[idx] = c > 0.0 ? __ddiv_rn(1.0, c) : 0.0;
    }
    if constexpr (FUSED) {
        for (unsigned int i = blockIdx.x + warp * step; i < total; i += WARPS * step)
            slab_finish(fin, tile(i).kt, plan);
    }
}

template <int FP8, int TS, bool FUSED>
cudaError_t go(const CodesOp &A, const CodesOp &B, int L, double gamma, long long ldo,
               DevPlan *plan, const SlabFinish &fin, cudaStream_t st) {
    constexpr size_t smem = (size_t)STAGES * TS * TS * sizeof(float);
    auto kern = codes_kernel<FP8, TS, FUSED>;
    static SmemOptIn smem_ok;
    if (cudaError_t e = smem_ok.allow(kern, (int)smem)) return e;
    const long long total = (long long)A.tiles + B.tiles;
    const long long grid = std::min<long long>(total, (TS == 128 ? 1LL : 2LL) * device_sms());
    return launch_pdl(kern, dim3((unsigned)grid), dim3(THREADS), smem, st, A, B, L, gamma, ldo,
                      plan, fin);
}

}  // namespace

cudaError_t launch_codes(const PackOperand<float> &a, double *mxA, double *varA, double *sA,
                         void *outA, const PackOperand<float> *b, double *mxB, double *varB,
                         double *sB, void *outB, int fp8, bool fused, double gamma, long long ldo,
                         DevPlan *plan, const SlabFinish &fin, cudaStream_t st) {
    const int L = a.L;
    const int ts = L % 128 == 0 ? 128 : 64;
    if (L % ts || (fp8 && ts != 128) || (fused && L != ts)) return cudaErrorInvalidValue;
    auto op = [&](const PackOperand<float> &o, double *mx, double *var, double *s, void *out) {
        CodesOp c;
        c.p = o.src; c.sx = o.sx; c.sk = o.sk; c.X = o.X; c.K = o.K;
        c.kt = (int)((o.K + ts - 1) / ts);
        const long long tiles = (o.X + ts - 1) / ts * c.kt;
        c.tiles = (int)std::min<long long>(tiles, kMaxTiles + 1LL);
        c.cx = o.cx; c.cl = o.cl;
        c.mx = mx; c.var = var; c.s = s;
        c.out = reinterpret_cast<unsigned char *>(out);
        return c;
    };
    const CodesOp A = op(a, mxA, varA, sA, outA);
    CodesOp B = b ? op(*b, mxB, varB, sB, outB) : A;
    if (!b) B.tiles = 0;
    if (A.tiles > kMaxTiles || B.tiles > kMaxTiles) return cudaErrorInvalidConfiguration;
    if (fp8) return fused ? go<1, 128, true>(A, B, L, gamma, ldo, plan, fin, st)
                          : go<1, 128, false>(A, B, L, gamma, ldo, plan, fin, st);
    if (ts == 128) return fused ? go<0, 128, true>(A, B, L, gamma, ldo, plan, fin, st)
                                : go<0, 128, false>(A, B, L, gamma, ldo, plan, fin, st);
    return fused ? go<0, 64, true>(A, B, L, gamma, ldo, plan, fin, st)
                 : go<0, 64, false>(A, B, L, gamma, ldo, plan, fin, st);
}

}  // namespace tdg
