// Steps (a) and (b) on the data: companding and rounding (eq. 3) fused with
// packing (eqs. 6, 7, 11) in one pass over each input.
//
// Every element is quantized as a~ = rint(fl_T(x * c_T)) with its block's
// compander and the packed number is built by Horner's rule,
//     acc = d_{W-1};  acc = fma(w, acc, d_i),  i = W-2 .. 0,
// with w = z for eqs. 6 and 11 and w = z^-1 for eq. 7.  Digits outside the
// L x L block or the matrix are zero (border clean-up, Sec. 2).
//
//   pack along k   out[l P + j][x]  (eq. 6 for A, eq. 7 for B, W = 1 for the
//                  unpacked operands and the plain copies):
//                    - x contiguous in the input: 16-byte vector loads of the
//                      W digit rows, vector stores, no shared memory;
//                    - k contiguous in the input: a TILE x TILE W tile (TILE =
//                      64 x-rows for fp32 with W <= 2, else 32) staged in
//                      shared memory with vector loads, then written along x.
//   pack along x   out[k][i P + j]  (eq. 11, asymmetric A), tile staged in
//                  shared memory.
// P = ceil(L / W) packed numbers per block.  Each kernel first reads the
// device plan and returns unless the planner chose its packing; the grids are
// capped and loop over tiles so that such early exits cost little.
#include <mutex>

#include "tdg_common.cuh"
#include "tdg_internal.h"
#include "tdg_pack.h"

namespace tdg {

namespace {

constexpr int TILE = 32;
constexpr int MAX_CTAS = 152 * 8;

template <typename T>
struct Src {
    const T *p;
    long long sx, sk;
    long long X, K;
    const T *c;       // nullptr: copy without companding
    long long cx, cl;
    int L;
};

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

// w = z = 2^-q (wsign < 0) or z^-1 = 2^q (wsign > 0), q from the device plan
template <typename T>
__device__ inline T pack_weight(const DevPlan *plan, int wsign) {
    int q = plan->q;
    if constexpr (sizeof(T) == 4) return scalbnf(1.0f, wsign < 0 ? -q : q);
    else return scalbn(1.0, wsign < 0 ? -q : q);
}

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

// ------------------------------------------------------------------ pack along k,
// x contiguous in the input: one item = VEC consecutive x of one packed row
// (the loop of CTA vb of vg working on this operand)
template <typename T, int W>
__device__ __forceinline__ void pack_k_xc_body(const Src<T> &S, int P, T w, T *out, long long ldo,
                                               long long rows_out, int vec_ok, long long vb,
                                               long long vg) {
    constexpr int VEC = VecT<T>::n;
    const bool compand = S.c != nullptr;
    const int L = S.L;
    const long long nx = (S.X + VEC - 1) / VEC;
    const long long items = rows_out * nx;
    for (long long it = vb * blockDim.x + threadIdx.x; it < items; it += vg * blockDim.x) {
        const long long row = it / nx;                 // l * P + j
        const long long x = (it - row * nx) * VEC;
        const int l = (int)(row / P), j = (int)(row - (long long)l * P);
        const long long kbase = (long long)l * L + (long long)W * j;
        const long long klim = min((long long)(l + 1) * L, S.K);
        const T c = compand ? S.c[(x / L) * S.cx + (long long)l * S.cl] : T(1);
        T acc[VEC];
        const bool full = vec_ok && x + VEC <= S.X;
#pragma unroll
        for (int i = W - 1; i >= 0; --i) {
            const long long k = kbase + i;
            T d[VEC];
            if (k < klim && W * j + i < L) {
                const T *src = S.p + k * S.sk + x;
                if (full) {
                    vload(src, d);
                } else {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) d[e] = (x + e < S.X) ? src[e] : T(0);
                }
#pragma unroll
                for (int e = 0; e < VEC; ++e) d[e] = quant(d[e], c, compand);
            } else {
#pragma unroll
                for (int e = 0; e < VEC; ++e) d[e] = T(0);
            }
#pragma unroll
            for (int e = 0; e < VEC; ++e) acc[e] = (i == W - 1) ? d[e] : fma_t(w, acc[e], d[e]);
        }
        T *dst = out + row * ldo + x;
        if (full) {
            vstore(dst, acc);
        } else {
#pragma unroll
            for (int e = 0; e < VEC; ++e)
                if (x + e < S.X) dst[e] = acc[e];
        }
    }
}

template <typename T, int W>
__global__ void __launch_bounds__(256) pack_k_xc_kernel(Src<T> S, int P, const DevPlan *plan,
                                                        int expectW, int wsign, T *out,
                                                        long long ldo, long long rows_out,
                                                        int vec_ok) {
    pdl_entry();
    if (expectW > 0 && plan->W != expectW) return;
    const T w = W > 1 ? pack_weight<T>(plan, wsign) : T(1);
    pack_k_xc_body<T, W>(S, P, w, out, ldo, rows_out, vec_ok, blockIdx.x, gridDim.x);
}

// ------------------------------------------------------------------ pack along k,
// k contiguous in the input: x-rows per tile of pack_k_kc_kernel (shared by
// the kernel and its launch), each tile TILE packed columns wide
template <typename T, int W>
constexpr int kc_tile() { return (sizeof(T) == 4 && W <= 2) ? 64 : 32; }

template <typename T, int W>
__device__ __forceinline__ void pack_k_kc_body(const Src<T> &S, int P, T w, T *out, long long ldo,
                                               long long rows_out, int vec_ok, long long vb,
                                               long long vg) {
    constexpr int VEC = VecT<T>::n;
    // fp32 with W <= 2: 64 x-rows per tile (a 33 KB tile, four times the
    // work per pass of the loop's fixed costs); else 32
    constexpr int TILE = kc_tile<T, W>();
    constexpr int NK = TILE * W;            // k values per tile row
    constexpr int PITCH = NK + 1;
    __shared__ T s[TILE * PITCH];
    __shared__ T crow[TILE];
    const bool compand = S.c != nullptr;
    const int L = S.L;
    const int jt = (P + TILE - 1) / TILE;
    const long long xt = (S.X + TILE - 1) / TILE;
    const int nK = (int)((S.K + L - 1) / L);
    const long long tiles = xt * nK * jt;
    for (long long t = vb; t < tiles; t += vg) {
        const long long xtile = t % xt;
        const long long r = t / xt;
        const int l = (int)(r / jt), j0 = (int)(r % jt) * TILE;
        const long long x0 = xtile * TILE;
        const long long kslab = (long long)l * L;
        const long long k0 = kslab + (long long)W * j0;
        const long long klim = min(kslab + L, S.K);
        __syncthreads();   // previous tile's readers are done with s / crow
        if (threadIdx.x < TILE) {
            const long long x = x0 + threadIdx.x;
            crow[threadIdx.x] = (compand && x < S.X) ? S.c[(x / L) * S.cx + (long long)l * S.cl] : T(1);
        }
        __syncthreads();
        constexpr int CH = NK / VEC;
        for (int e = threadIdx.x; e < TILE * CH; e += blockDim.x) {
            const int xr = e / CH, kc = (e % CH) * VEC;
            const long long x = x0 + xr, k = k0 + kc;
            T d[VEC];
            if (x < S.X && vec_ok && k + VEC <= klim) {
                vload(S.p + x * S.sx + k, d);
            } else {
#pragma unroll
                for (int q = 0; q < VEC; ++q)
                    d[q] = (x < S.X && k + q < klim) ? S.p[x * S.sx + k + q] : T(0);
            }
            const T c = crow[xr];
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                const bool valid = x < S.X && k + q < klim;
                s[xr * PITCH + kc + q] = valid ? quant(d[q], c, compand) : T(0);
            }
        }
        __syncthreads();
        for (int e = threadIdx.x; e < TILE * TILE; e += blockDim.x) {
            const int jr = e / TILE, xr = e % TILE;
            const int j = j0 + jr;
            const long long x = x0 + xr;
            const long long row = (long long)l * P + j;
            if (j >= P || x >= S.X || row >= rows_out) continue;
            const T *d = s + xr * PITCH + jr * W;
            T acc = d[W - 1];
#pragma unroll
            for (int i = W - 2; i >= 0; --i) acc = fma_t(w, acc, d[i]);
            out[row * ldo + x] = acc;
        }
    }
}

template <typename T, int W>
__global__ void __launch_bounds__(256) pack_k_kc_kernel(Src<T> S, int P, const DevPlan *plan,
                                                        int expectW, int wsign, T *out,
                                                        long long ldo, long long rows_out,
                                                        int vec_ok) {
    pdl_entry();
    if (expectW > 0 && plan->W != expectW) return;
    const T w = W > 1 ? pack_weight<T>(plan, wsign) : T(1);
    pack_k_kc_body<T, W>(S, P, w, out, ldo, rows_out, vec_ok, blockIdx.x, gridDim.x);
}

// Both operands of the symmetric form in one launch, A k-contiguous (eq. 6)
// and B x-contiguous (eq. 7), the layouts of C = A B with row-major A and B:
// the first 2 m CTAs alternate between the two (m = the smaller CTA count),
// the rest go to the operand with more, so every SM runs both kinds at once
// (the A pack is issue-bound, the B pack latency-bound).
template <typename T, int W>
__global__ void __launch_bounds__(256) pack_k_pair_kernel(Src<T> SA, Src<T> SB, int P,
                                                          const DevPlan *plan, int expectW,
                                                          T *outA, long long ldoA,
                                                          long long rowsA, int vecA, T *outB,
                                                          long long ldoB, long long rowsB,
                                                          int vecB, long long gA, long long gB) {
    pdl_entry();
    if (expectW > 0 && plan->W != expectW) return;
    const long long b = blockIdx.x, m = min(gA, gB);
    bool isA;
    long long vb;
    if (b < 2 * m) {
        isA = (b & 1) != 0;
        vb = b >> 1;
    } else {
        isA = gA > gB;
        vb = m + (b - 2 * m);
    }
    if (isA) {
        const T w = W > 1 ? pack_weight<T>(plan, -1) : T(1);
        pack_k_kc_body<T, W>(SA, P, w, outA, ldoA, rowsA, vecA, vb, gA);
    } else {
        const T w = W > 1 ? pack_weight<T>(plan, +1) : T(1);
        pack_k_xc_body<T, W>(SB, P, w, outB, ldoB, rowsB, vecB, vb, gB);
    }
}

// ------------------------------------------------------------------ plain k-major copy
// out[k][x] = in[x][k] of a k-contiguous operand without companding (the
// plain product's operands): 64 x 64 tiles through shared memory (s[x][k],
// pitch 65), 16-byte loads along k issued before any is used, 16-byte stores
// along x.  256 threads per CTA.
template <typename T>
__global__ void __launch_bounds__(256) transpose_copy_kernel(Src<T> S, const DevPlan *plan,
                                                             int expectW, T *out, long long ldo,
                                                             int vec_ok) {
    pdl_entry();
    if (expectW > 0 && plan->W != expectW) return;
    constexpr int VEC = VecT<T>::n;
    constexpr int TT = 64, PITCH = TT + 1;
    constexpr int NV = TT * TT / VEC / 256;     // vectors per thread and phase
    __shared__ T s[TT * PITCH];
    const long long xt = (S.X + TT - 1) / TT, kt = (S.K + TT - 1) / TT;
    for (long long t = blockIdx.x; t < xt * kt; t += gridDim.x) {
        const long long x0 = (t % xt) * TT, k0 = (t / xt) * TT;
        T v[NV][VEC];
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int e = threadIdx.x + u * 256;
            const int xr = e / (TT / VEC), kc = (e % (TT / VEC)) * VEC;
            const long long x = x0 + xr, k = k0 + kc;
            if (x < S.X && vec_ok && k + VEC <= S.K) {
                vload(S.p + x * S.sx + k, v[u]);
            } else {
#pragma unroll
                for (int q = 0; q < VEC; ++q)
                    v[u][q] = (x < S.X && k + q < S.K) ? S.p[x * S.sx + k + q] : T(0);
            }
        }
        __syncthreads();   // the previous tile's readers are done with s
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int e = threadIdx.x + u * 256;
            const int xr = e / (TT / VEC), kc = (e % (TT / VEC)) * VEC;
#pragma unroll
            for (int q = 0; q < VEC; ++q) s[xr * PITCH + kc + q] = v[u][q];
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int e = threadIdx.x + u * 256;
            const int kr = e / (TT / VEC), xc = (e % (TT / VEC)) * VEC;
            const long long k = k0 + kr, x = x0 + xc;
            if (k >= S.K || x >= S.X) continue;
            T w[VEC];
#pragma unroll
            for (int q = 0; q < VEC; ++q) w[q] = s[(xc + q) * PITCH + kr];
            T *dst = out + k * ldo + x;
            if (vec_ok && x + VEC <= S.X) {
                vstore(dst, w);
            } else {
#pragma unroll
                for (int q = 0; q < VEC; ++q)
                    if (x + q < S.X) dst[q] = w[q];
            }
        }
    }
}

// ------------------------------------------------------------------ pack along x
// out[k][i*P + j] for j in [j0, j0 + 32) of row block i, k in [k0, k0 + 32)
template <typename T, int W>
__global__ void __launch_bounds__(256) pack_x_kernel(Src<T> S, int P, const DevPlan *plan,
                                                     int expectW, int wsign, T *out,
                                                     long long ldo) {
    pdl_entry();
    if (expectW > 0 && plan->W != expectW) return;
    constexpr int NX = TILE * W;
    constexpr int PITCH = TILE + 1;
    __shared__ T s[NX * PITCH];
    __shared__ T ccol[TILE];
    const T w = W > 1 ? pack_weight<T>(plan, wsign) : T(1);
    const bool compand = S.c != nullptr;
    const int L = S.L;
    const int jt = (P + TILE - 1) / TILE;
    const int nM = (int)((S.X + L - 1) / L);
    const long long kt = (S.K + TILE - 1) / TILE;
    const long long tiles = (long long)nM * jt * kt;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const long long ktile = t % kt;
        const long long r = t / kt;
        const int i = (int)(r / jt), j0 = (int)(r % jt) * TILE;
        const long long k0 = ktile * TILE;
        const long long xblk0 = (long long)i * L;
        const long long xlim = min(xblk0 + L, S.X);
        const long long x0 = xblk0 + (long long)W * j0;
        __syncthreads();
        if (threadIdx.x < TILE) {
            const long long k = k0 + threadIdx.x;
            ccol[threadIdx.x] = (compand && k < S.K) ? S.c[(long long)i * S.cx + (k / L) * S.cl] : T(1);
        }
        __syncthreads();
        if (S.sk == 1) {
            for (int e = threadIdx.x; e < NX * TILE; e += blockDim.x) {
                const int xr = e / TILE, kc = e % TILE;
                const long long x = x0 + xr, k = k0 + kc;
                const bool valid = x < xlim && k < S.K;
                s[xr * PITCH + kc] = valid ? quant(S.p[x * S.sx + k], ccol[kc], compand) : T(0);
            }
        } else {
            for (int e = threadIdx.x; e < NX * TILE; e += blockDim.x) {
                const int kc = e / NX, xr = e % NX;
                const long long x = x0 + xr, k = k0 + kc;
                const bool valid = x < xlim && k < S.K;
                s[xr * PITCH + kc] = valid ? quant(S.p[x + k * S.sk], ccol[kc], compand) : T(0);
            }
        }
        __syncthreads();
        for (int e = threadIdx.x; e < TILE * TILE; e += blockDim.x) {
            const int kr = e / TILE, jr = e % TILE;
            const int j = j0 + jr;
            const long long k = k0 + kr;
            if (j >= P || k >= S.K) continue;
            const T *d = s + (jr * W) * PITCH + kr;
            T acc = d[(W - 1) * PITCH];
#pragma unroll
            for (int ii = W - 2; ii >= 0; --ii) acc = fma_t(w, acc, d[ii * PITCH]);
            out[k * ldo + (long long)i * P + j] = acc;
        }
    }
}

template <typename T>
Src<T> make_src(const PackOperand<T> &o) {
    Src<T> S;
    S.p = o.src; S.sx = o.sx; S.sk = o.sk; S.X = o.X; S.K = o.K;
    S.c = o.c; S.cx = o.cx; S.cl = o.cl; S.L = o.L;
    return S;
}

int capped(long long n) { return (int)max(1LL, min(n, (long long)MAX_CTAS)); }

// Grid of at most `waves` full waves of resident CTAs for `kern` (occupancy
// x SMs, cached per device and kernel under a lock, since host threads may
// launch concurrently), so a grid-stride kernel never ends on a partial wave
// of long-running CTAs and an early exit costs few CTAs.
int resident_grid(const void *kern, long long n, int waves) {
    struct Entry { const void *k; int dev, ctas; };
    static Entry cache[128];
    static int ncache = 0;
    static std::mutex mu;
    int dev = 0;
    cudaGetDevice(&dev);
    int ctas = 0;
    {
        std::lock_guard<std::mutex> lock(mu);
        for (int i = 0; i < ncache; ++i)
            if (cache[i].k == kern && cache[i].dev == dev) ctas = cache[i].ctas;
    }
    if (!ctas) {
        int sms = 0, per = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, 256, 0) != cudaSuccess || per < 1)
            per = 1;
        ctas = per * sms;
        std::lock_guard<std::mutex> lock(mu);
        if (ncache < 128) cache[ncache++] = {kern, dev, ctas};
    }
    return (int)max(1LL, min(n, (long long)ctas * waves));
}

template <typename T, int W>
cudaError_t launch_pack_k_w(const PackOperand<T> &o, const DevPlan *plan, int expectW, int wsign,
                            T *out, long long ldo, long long rows_out, cudaStream_t st) {
    constexpr int VEC = VecT<T>::n;
    Src<T> S = make_src(o);
    const int P = (o.L + W - 1) / W;
    const bool aligned_in = ((uintptr_t)o.src % 16 == 0);
    const bool aligned_out = ((uintptr_t)out % 16 == 0) && (ldo % VEC == 0);
    if (o.sx == 1) {
        const int vec_ok = aligned_in && aligned_out && (o.sk % VEC == 0);
        const long long items = rows_out * ((o.X + VEC - 1) / VEC);
        return launch_pdl(pack_k_xc_kernel<T, W>,
                          dim3(resident_grid((const void *)pack_k_xc_kernel<T, W>,
                                             (items + 255) / 256, 4)),
                          dim3(256), 0, st, S, P, plan, expectW, wsign, out, ldo, rows_out,
                          vec_ok);
    } else if (W == 1 && o.c == nullptr && o.sk == 1 && rows_out == o.K) {
        // plain copy: a straight transpose
        const int vec_ok = aligned_in && aligned_out && (o.sx % VEC == 0);
        const long long tiles = ((o.X + 63) / 64) * ((o.K + 63) / 64);
        return launch_pdl(transpose_copy_kernel<T>, dim3(capped(tiles)), dim3(256), 0, st, S, plan,
                          expectW, out, ldo, vec_ok);
    } else {
        const int vec_ok = aligned_in && (o.sx % VEC == 0) && o.sk == 1;
        constexpr int TK = kc_tile<T, W>();
        const long long tiles = ((o.X + TK - 1) / TK) * ((o.K + o.L - 1) / o.L) *
                                ((P + TK - 1) / TK);
        return launch_pdl(pack_k_kc_kernel<T, W>,
                          dim3(resident_grid((const void *)pack_k_kc_kernel<T, W>, tiles, 4)),
                          dim3(256), 0, st, S, P, plan, expectW, wsign, out, ldo, rows_out,
                          vec_ok);
    }
    return cudaGetLastError();
}

template <typename T, int W>
cudaError_t launch_pack_x_w(const PackOperand<T> &o, const DevPlan *plan, int expectW, int wsign,
                            T *out, long long ldo, cudaStream_t st) {
    Src<T> S = make_src(o);
    const int P = (o.L + W - 1) / W;
    const long long tiles = ((o.X + o.L - 1) / o.L) * ((P + TILE - 1) / TILE) *
                            ((o.K + TILE - 1) / TILE);
    return launch_pdl(pack_x_kernel<T, W>, dim3(capped(tiles)), dim3(256), 0, st, S, P, plan,
                      expectW, wsign, out, ldo);
    return cudaGetLastError();
}

}  // namespace

// The symmetric form's two packs (A with wsign -1, B with +1): one launch of
// pack_k_pair_kernel when A is k-contiguous and B x-contiguous, else B's pack
// and then A's.
template <typename T, int W>
cudaError_t launch_pack_k_pair_w(const PackOperand<T> &a, const PackOperand<T> &b,
                                 const DevPlan *plan, int expectW, T *outA, long long ldoA,
                                 long long rowsA, T *outB, long long ldoB, long long rowsB,
                                 cudaStream_t st) {
    constexpr int VEC = VecT<T>::n;
    const bool a_copy = W == 1 && a.c == nullptr && a.sk == 1 && rowsA == a.K;
    if (a.sx == 1 || a_copy || b.sx != 1) {
        cudaError_t e = launch_pack_k_w<T, W>(b, plan, expectW, +1, outB, ldoB, rowsB, st);
        if (e != cudaSuccess) return e;
        return launch_pack_k_w<T, W>(a, plan, expectW, -1, outA, ldoA, rowsA, st);
    }
    Src<T> SA = make_src(a), SB = make_src(b);
    const int P = (a.L + W - 1) / W;
    const int vecA = ((uintptr_t)a.src % 16 == 0) && (a.sx % VEC == 0) && a.sk == 1;
    const int vecB = ((uintptr_t)b.src % 16 == 0) && ((uintptr_t)outB % 16 == 0) &&
                     (ldoB % VEC == 0) && (b.sk % VEC == 0);
    constexpr int TK = kc_tile<T, W>();
    const long long tilesA = ((a.X + TK - 1) / TK) * ((a.K + a.L - 1) / a.L) * ((P + TK - 1) / TK);
    const long long blocksB = (rowsB * ((b.X + VEC - 1) / VEC) + 255) / 256;
    const void *kern = (const void *)pack_k_pair_kernel<T, W>;
    const long long gA = resident_grid(kern, tilesA, 2);
    const long long gB = resident_grid(kern, blocksB, 2);
    return launch_pdl(pack_k_pair_kernel<T, W>, dim3((unsigned)(gA + gB)), dim3(256), 0, st, SA,
                      SB, P, plan, expectW, outA, ldoA, rowsA, vecA, outB, ldoB, rowsB, vecB,
                      gA, gB);
}

template <typename T>
cudaError_t launch_pack_k_pair(const PackOperand<T> &a, const PackOperand<T> &b, int W,
                               const DevPlan *plan, int expectW, T *outA, long long ldoA,
                               long long rowsA, T *outB, long long ldoB, long long rowsB,
                               cudaStream_t st) {
    switch (W) {
        case 1: return launch_pack_k_pair_w<T, 1>(a, b, plan, expectW, outA, ldoA, rowsA, outB, ldoB, rowsB, st);
        case 2: return launch_pack_k_pair_w<T, 2>(a, b, plan, expectW, outA, ldoA, rowsA, outB, ldoB, rowsB, st);
        case 3: return launch_pack_k_pair_w<T, 3>(a, b, plan, expectW, outA, ldoA, rowsA, outB, ldoB, rowsB, st);
        case 4: return launch_pack_k_pair_w<T, 4>(a, b, plan, expectW, outA, ldoA, rowsA, outB, ldoB, rowsB, st);
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_pack_k(const PackOperand<T> &o, int W, const DevPlan *plan, int expectW,
                          int wsign, T *out, long long ldo, long long rows_out, cudaStream_t st) {
    switch (W) {
        case 1: return launch_pack_k_w<T, 1>(o, plan, expectW, wsign, out, ldo, rows_out, st);
        case 2: return launch_pack_k_w<T, 2>(o, plan, expectW, wsign, out, ldo, rows_out, st);
        case 3: return launch_pack_k_w<T, 3>(o, plan, expectW, wsign, out, ldo, rows_out, st);
        case 4: return launch_pack_k_w<T, 4>(o, plan, expectW, wsign, out, ldo, rows_out, st);
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_pack_x(const PackOperand<T> &o, int W, const DevPlan *plan, int expectW,
                          int wsign, T *out, long long ldo, cudaStream_t st) {
    switch (W) {
        case 1: return launch_pack_x_w<T, 1>(o, plan, expectW, wsign, out, ldo, st);
        case 2: return launch_pack_x_w<T, 2>(o, plan, expectW, wsign, out, ldo, st);
        case 3: return launch_pack_x_w<T, 3>(o, plan, expectW, wsign, out, ldo, st);
        case 4: return launch_pack_x_w<T, 4>(o, plan, expectW, wsign, out, ldo, st);
    }
    return cudaErrorInvalidValue;
}

template cudaError_t launch_pack_k_pair<float>(const PackOperand<float> &, const PackOperand<float> &,
                                               int, const DevPlan *, int, float *, long long,
                                               long long, float *, long long, long long,
                                               cudaStream_t);
template cudaError_t launch_pack_k_pair<double>(const PackOperand<double> &,
                                                const PackOperand<double> &, int,
                                                const DevPlan *, int, double *, long long,
                                                long long, double *, long long, long long,
                                                cudaStream_t);
template cudaError_t launch_pack_k<float>(const PackOperand<float> &, int, const DevPlan *, int, int,
                                          float *, long long, long long, cudaStream_t);
template cudaError_t launch_pack_k<double>(const PackOperand<double> &, int, const DevPlan *, int,
                                           int, double *, long long, long long, cudaStream_t);
template cudaError_t launch_pack_x<float>(const PackOperand<float> &, int, const DevPlan *, int, int,
                                          float *, long long, cudaStream_t);
template cudaError_t launch_pack_x<double>(const PackOperand<double> &, int, const DevPlan *, int,
                                           int, double *, long long, cudaStream_t);

}  // namespace tdg
