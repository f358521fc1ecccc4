// Step (a), first half: per-block statistics of op(A) and op(B).
//
// Sec. 3 gathers max/min of every L x L subblock during the block-major
// reorder; Sec. 5.B adds sigma.  Here one CTA reads one L x L tile of the
// stored matrix with 16-byte vector loads (one HBM pass) and produces
//   max|x|   exact,
//   sigma^2  sum x^2 / (valid elements), about zero (fp32 inputs:
//            double-float accumulation of exact squares per thread and a
//            double-float tree over the block; fp64 inputs: fp64 throughout).
// Non-finite inputs raise TDG_ENONFINITE in the plan's device status.
#include <algorithm>

#include "tdg_common.cuh"
#include "tdg_internal.h"
#include "tdg_planner.cuh"

namespace tdg {

namespace {

// max|x| is kept as the largest bit pattern of |x| (for non-negative IEEE
// values the integer order is the numeric order), which stays on the integer
// pipe, and NaN/Inf show in it.  Each thread keeps one running sum
// per vector lane so the dependent add chains run side by side.
struct Acc {
    float hi[4], lo[4];        // fp32 path: double-float sums of squares
    double d[2];               // fp64 path
    // bit pattern of the largest |x|; from the pattern of Inf on, an input is
    // NaN or Inf (32 bits for fp32: the per-element work stays at one and, one
    // max besides the sum)
    unsigned int m32;
    unsigned long long m64;
};

__device__ inline void add_sq(Acc &a, int lane, float x) {
    // exact square as hi + err (TwoProduct), then TwoSum into (hi, lo)
    float p = __fmul_rn(x, x);
    float e = __fmaf_rn(x, x, -p);
    float t = __fadd_rn(a.hi[lane], p);
    float bp = __fsub_rn(t, a.hi[lane]);
    float err = __fadd_rn(__fsub_rn(a.hi[lane], __fsub_rn(t, bp)), __fsub_rn(p, bp));
    a.hi[lane] = t;
    a.lo[lane] = __fadd_rn(a.lo[lane], __fadd_rn(err, e));
    a.m32 = max(a.m32, __float_as_uint(x) & 0x7fffffffu);
}

// (hi, lo) += (bh, bl) in double-float arithmetic (TwoSum of the high parts,
// low parts added to the error, then renormalised)
__device__ inline void df_add(float &hi, float &lo, float bh, float bl) {
    const float s = __fadd_rn(hi, bh);
    const float v = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, v)), __fsub_rn(bh, v));
    const float t = __fadd_rn(e, __fadd_rn(lo, bl));
    hi = __fadd_rn(s, t);
    lo = __fsub_rn(t, __fsub_rn(hi, s));
}

__device__ inline void add_sq(Acc &a, int lane, double x) {
    a.d[lane & 1] = __fma_rn(x, x, a.d[lane & 1]);
    a.m64 = max(a.m64, (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull);
}

__device__ inline void load_vec(const float *p, float *v) {
    const float4 q = __ldg(reinterpret_cast<const float4 *>(p));
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ inline void load_vec(const double *p, double *v) {
    const double2 q = __ldg(reinterpret_cast<const double2 *>(p));
    v[0] = q.x; v[1] = q.y;
}

// One operand: the stored matrix rows_s x cols_s (leading dimension ld),
// op() transposed when trans; block (bi, bj) of the stored matrix is block
// (bj, bi) of op() then.  nbc_op = block columns of op().
template <typename T>
struct StatsOp {
    const T *X;
    long long rows_s, cols_s, ld;
    int trans, nbc_op, nbc_s;       // nbc_s = block columns of the stored matrix
    unsigned int nblk;              // blocks of the stored matrix
    int slab_rows;                  // 1: a stored row of blocks is a slab, 0: a column
    double *mx, *var;
};

// Both operands in one launch: blocks [0, A.nblk) are A's, the rest B's, dealt
// out to a resident wave of CTAs.  A CTA counts its blocks for the planner's
// sums once, at its end (slab_finish): counted block by block, each CTA held
// its SM's registers for the 1.5 us of a fence and an atomic more.
template <typename T>
__global__ void __launch_bounds__(256, 3) block_stats_kernel(StatsOp<T> A, StatsOp<T> B, int L,
                                                          DevPlan *plan,
                                                          const __grid_constant__ SlabFinish fin) {
    pdl_entry();
    constexpr int VEC = 16 / sizeof(T);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    // two sets, so that the other warps may run on into the next block while
    // warp 0 finishes this one
    __shared__ float sh_h[2][32], sh_l[2][32];
    __shared__ double sh_d[2][32];
    __shared__ unsigned long long sh_m[2][32];
    const unsigned int total = A.nblk + B.nblk;
    int set = 0;
    for (unsigned int b = blockIdx.x; b < total; b += gridDim.x, set ^= 1) {
        const bool isA = b < A.nblk;
        const StatsOp<T> &o = isA ? A : B;
        const unsigned int blk = isA ? b : b - A.nblk;
        const int bi = (int)(blk / (unsigned int)o.nbc_s), bj = (int)blk - bi * o.nbc_s;
        const T *__restrict__ X = o.X;
        const long long ld = o.ld;
        const long long r0b = (long long)bi * L, c0 = (long long)bj * L;
        const int rn = (int)min((long long)L, o.rows_s - r0b);
        const int cn = (int)min((long long)L, o.cols_s - c0);
        Acc a{{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}, {0.0, 0.0}, 0u, 0ull};
        // rows in batches of eight per warp so eight 16-byte loads are in flight
        // before any of them is consumed
        constexpr int RB = 8;
        const bool vec_ok = (ld % VEC == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
        const long long step = (long long)nwarp * ld;
        for (int cb = 0; cb < cn; cb += 32 * VEC) {
            // 16 bytes per lane, or (ragged or unaligned rows) VEC times one
            // value with the lanes side by side
            if (vec_ok && cb + 32 * VEC <= cn) {
                const T *p = X + (r0b + warp) * ld + c0 + cb + lane * VEC;
                for (int r = warp; r < rn; r += RB * nwarp, p += RB * step) {
                    T v[RB][VEC];
#pragma unroll
                    for (int u = 0; u < RB; ++u) {
                        if (r + u * nwarp < rn) {
                            load_vec(p + u * step, v[u]);
                        } else {
#pragma unroll
                            for (int e = 0; e < VEC; ++e) v[u][e] = T(0);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < RB; ++u)
#pragma unroll
                        for (int e = 0; e < VEC; ++e) add_sq(a, e, v[u][e]);
                }
            } else {
                const T *p = X + (r0b + warp) * ld + c0 + cb + lane;
                const int left = cn - cb - lane;
                for (int r = warp; r < rn; r += RB * nwarp, p += RB * step) {
                    T v[RB][VEC];
#pragma unroll
                    for (int u = 0; u < RB; ++u)
#pragma unroll
                        for (int e = 0; e < VEC; ++e)
                            v[u][e] = (r + u * nwarp < rn && 32 * e < left) ? __ldg(p + u * step + 32 * e)
                                                                            : T(0);
#pragma unroll
                    for (int u = 0; u < RB; ++u)
#pragma unroll
                        for (int e = 0; e < VEC; ++e) add_sq(a, e, v[u][e]);
                }
            }
        }
        // block sum of squares and max|x|: fp32 inputs reduce (hi, lo) float pairs
        // with double-float additions and float bit patterns (GB300 runs fp64 at a
        // small fraction of the fp32 rate, so fp64 appears only once per block);
        // fp64 inputs reduce in fp64
        float hi = 0.f, lo = 0.f;
        double d = 0.0;
        if constexpr (sizeof(T) == 4) {
            hi = a.hi[0]; lo = a.lo[0];
#pragma unroll
            for (int q = 1; q < 4; ++q) df_add(hi, lo, a.hi[q], a.lo[q]);
        } else {
            d = a.d[0] + a.d[1];
        }
        unsigned int m32 = a.m32;
        unsigned long long m64 = a.m64;
        auto warp_reduce = [&]() {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                if constexpr (sizeof(T) == 4) {
                    const float oh = __shfl_xor_sync(0xffffffffu, hi, off);
                    const float ol = __shfl_xor_sync(0xffffffffu, lo, off);
                    df_add(hi, lo, oh, ol);
                } else {
                    d += __shfl_xor_sync(0xffffffffu, d, off);
                }
                if constexpr (sizeof(T) == 4)
                    m32 = max(m32, __shfl_xor_sync(0xffffffffu, m32, off));
                else
                    m64 = max(m64, (unsigned long long)__shfl_xor_sync(0xffffffffu, m64, off));
            }
        };
        warp_reduce();
        if (lane == 0) {
            sh_h[set][warp] = hi;
            sh_l[set][warp] = lo;
            sh_d[set][warp] = d;
            sh_m[set][warp] = sizeof(T) == 4 ? (unsigned long long)m32 : m64;
        }
        __syncthreads();
        if (warp == 0) {
            const bool in = lane < nwarp;
            hi = in ? sh_h[set][lane] : 0.f;
            lo = in ? sh_l[set][lane] : 0.f;
            d = in ? sh_d[set][lane] : 0.0;
            m64 = in ? sh_m[set][lane] : 0ull;
            m32 = (unsigned int)m64;
            warp_reduce();
            if (lane == 0) {
                const double ssum = sizeof(T) == 4 ? (double)hi + (double)lo : d;
                const double m = sizeof(T) == 4 ? (double)__uint_as_float(m32)
                                                : __longlong_as_double((long long)m64);
                const bool bad = sizeof(T) == 4 ? m32 >= 0x7f800000u : m64 >= 0x7ff0000000000000ull;
                const long long idx = o.trans ? (long long)bj * o.nbc_op + bi
                                              : (long long)bi * o.nbc_op + bj;
                o.mx[idx] = m;
                o.var[idx] = ssum / ((double)rn * (double)cn);   // sigma^2 about zero
                if (bad) atomicExch(fin.nonfinite, 1);
            }
        }
    }
    __syncthreads();
    for (unsigned int b = blockIdx.x + warp * gridDim.x; b < total; b += nwarp * gridDim.x) {
        const bool isA = b < A.nblk;
        const StatsOp<T> &o = isA ? A : B;
        const unsigned int blk = isA ? b : b - A.nblk, nbc = (unsigned int)o.nbc_s;
        slab_finish(fin, (int)(o.slab_rows ? blk / nbc : blk % nbc), plan);
    }
}

}  // namespace

template <typename T>
static StatsOp<T> stats_op(const T *X, long long rows_s, long long cols_s, long long ld, int L,
                           int trans, int nbc_op, int slab_rows, double *mx,
                           double *var) {
    StatsOp<T> o;
    o.X = X; o.rows_s = rows_s; o.cols_s = cols_s; o.ld = ld;
    o.trans = trans; o.nbc_op = nbc_op;
    o.nbc_s = cdiv_i(cols_s, L);
    o.nblk = (unsigned int)((long long)cdiv_i(rows_s, L) * o.nbc_s);
    o.slab_rows = slab_rows;
    o.mx = mx; o.var = var;
    return o;
}

template <typename T>
cudaError_t launch_block_stats(const T *A, long long rows_a, long long cols_a, long long lda,
                               int trans_a, int nbc_a, double *mxA, double *varA, const T *B,
                               long long rows_b, long long cols_b, long long ldb, int trans_b,
                               int nbc_b, double *mxB, double *varB, int L, DevPlan *plan,
                               const SlabFinish &fin, cudaStream_t st) {
    // slabs run along the columns of op(A) and the rows of op(B)
    StatsOp<T> oa = stats_op(A, rows_a, cols_a, lda, L, trans_a, nbc_a, trans_a, mxA, varA);
    StatsOp<T> ob = stats_op(B, rows_b, cols_b, ldb, L, trans_b, nbc_b, !trans_b, mxB, varB);
    const long long nb = (long long)cdiv_i(rows_a, L) * oa.nbc_s + (long long)cdiv_i(rows_b, L) * ob.nbc_s;
    if (nb > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    // 24 warps fit an SM.  With blocks for all of them, four warps a block: half
    // as many reductions per value read as with eight (8192^2 x 2 fp32: 110 us
    // against 127); fewer blocks are done sooner by eight warps each.
    const int nt = nb >= 6LL * device_sms() ? 128 : 256;
    const long long grid = std::min<long long>(nb, 768 / nt * device_sms());
    return launch_pdl(block_stats_kernel<T>, dim3((unsigned)grid), dim3(nt), 0, st, oa, ob, L,
                      plan, fin);
}

#define TDG_STATS_INST(T)                                                                     \
    template cudaError_t launch_block_stats<T>(const T *, long long, long long, long long, int, \
                                               int, double *, double *, const T *, long long, \
                                               long long, long long, int, int, double *,        \
                                               double *, int, DevPlan *, const SlabFinish &,    \
                                               cudaStream_t);
TDG_STATS_INST(float)
TDG_STATS_INST(double)

}  // namespace tdg
