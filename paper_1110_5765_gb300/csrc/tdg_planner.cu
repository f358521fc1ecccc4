// Step (a), second half: choosing W, z and the companders on the device.
//
// * Fixed-bit mode: gamma_A = gamma_B = 2^(bits-1) - 1, R_max = L gamma^2
//   (eq. 17 with c = gamma / max|x|), z = 2^-q by eq. 15, W as requested.
// * Target mode (Prop. 4, eqs. 26-27, and Sec. 6 with one W per call): the
//   noise of eq. 21 summed over all subblock products (i, l, j) factorises
//   into four per-slab aggregates, so every candidate R_max level costs O(1):
//     N = L T1 / (12 gB^2) + L T2 / (12 gA^2) + T3 (L/144 + s^2) / (gA gB)^2,
//     S = L sum_l (sum_i sigma_A^2)(sum_j sigma_B^2).
//   One CTA evaluates every level for each W from the request down to 2, takes
//   the argmin of N (eq. 27's argmax of the SNR; ties go to the lower level) and
//   keeps the first W whose SNR meets the target.  Otherwise W = 1 (plain
//   product) with TDG_ALLOW_FALLBACK, else TDG_EUNREACHABLE.
// * Manual mode: given q and uniform companders (the Sec. 4.B protocol).
// The companders c and the de-companding factors (T)(s_A,il s_B,lj) follow in the
// pack launch.
#include "tdg_common.cuh"
#include "tdg_internal.h"
#include "tdg_planner.cuh"

namespace tdg {

namespace {

// Target mode, packed forms: for W from the request down to 2 the R_max level of
// least model noise (eq. 27's argmax of the SNR; ties to the lower level), the
// first W whose SNR meets the target; else the plain product (fallback) or
// TDG_EUNREACHABLE.
//
// An fp64 warp instruction takes 64 clocks of its SM sub-partition (2 lanes per
// clock and SM), and a candidate is some 170 of them, so what counts is how many
// follow one another.  One CTA: a warp per 32 levels forms the companders, which no
// W changes, then the quotients of eq. 21, those that the representation noise
// enters once per W, are dealt to the four sub-partitions side by side.  The
// logarithm of the SNR is left to the pack launch, where it delays nothing: the
// target is met where S / N exceeds 10^(target / 10), and only within 1e-9 of that
// the logarithm decides.  (A candidate per lane with every operation in sequence, 32
// per CTA, records in memory and the last CTA deciding, took 12 to 14 us; this kernel
// with 96 levels and one W at a time 10, but 19 where W = 4 was asked and 2 met the
// target, and 13 and 20 for the 145 levels of fp64.)
constexpr int kTermWarps = 12, kGroups = kMaxLevels / 32, kWs = kMaxW - 1;

__global__ void __launch_bounds__(32 * kTermWarps) level_kernel(PlanParams pp,
                                                                const double *__restrict__ stab,
                                                                DevPlan *plan) {
    pdl_entry();
    // [w]: of W = Wreq - w
    __shared__ double term[3][kMaxLevels], wterm[kWs][kMaxLevels], rep[kWs][kMaxLevels], uni[2];
    __shared__ int gam[2][kMaxLevels];
    __shared__ unsigned long long best_n[kWs][kGroups];
    __shared__ int best_t[kWs][kGroups], met[kWs];
    __shared__ DevPlan cand[kWs];
    const int L = pp.L, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the slab sums and rho that the statistics' last warp wrote
    const double S = (double)L * plan->tS, T1 = plan->tT1, T2 = plan->tT2, T3 = plan->tT3;
    const double rho = plan->trho;
    const int nf = plan->tnonfinite;
    int t_lo = 0;
    while (r_level(t_lo) < L) ++t_lo;
    const int t_hi = t_max_for(pp.p);
    const int ng = (t_hi - t_lo) / 32 + 1, nw = pp.Wreq - 1;      // groups of levels, packings

    // representation noise of level t for W with R = L gA gB (s < 0: not usable)
    auto rep_noise = [&](int W, int t, int gA, int gB) -> double {
        if (gA < 1) return -1.0;
        if (W <= w_ef((long long)L * gA * gB, q_for(r_level(t)), pp.p)) return 0.0;
        if (stab && t >= pp.t0 && t < pp.t0 + pp.nt) return __ldg(&stab[(W - 2) * pp.nt + (t - pp.t0)]);
        return -1.0;
    };
    if (warp < ng) {
        const int t = t_lo + 32 * warp + lane;
        if (t <= t_hi) {
            int gA, gB;
            split_gammas(r_level(t), L, rho, gA, gB);
            for (int w = 0; w < nw; ++w) rep[w][t] = rep_noise(pp.Wreq - w, t, gA, gB);
            gam[0][t] = max(gA, 1);
            gam[1][t] = max(gB, 1);
        }
    } else if (warp == ng) {
        const double l144 = __ddiv_rn((double)L, 144.0), sl = __ddiv_rn(S, (double)L);
        if (lane == 0) {
            uni[0] = l144;
            uni[1] = sl;
        }
    }
    __syncthreads();
    // the quotients of eq. 21 (model_noise), operation for operation: nb that no W
    // enters, then one per W.  (Warp i and i + 12 share a sub-partition.)
    const int nb = pp.noise_rms ? 3 : 2;
    for (int i = warp; i < (nb + nw) * ng; i += kTermWarps) {
        const int k = i / ng, t = t_lo + 32 * (i % ng) + lane;
        if (t > t_hi) continue;
        const double gA = (double)gam[0][t], gB = (double)gam[1][t];
        if (k == 0) {
            term[0][t] = __ddiv_rn(__dmul_rn((double)L, T1), __dmul_rn(__dmul_rn(12.0, gB), gB));
        } else if (k == 1) {
            term[1][t] = __ddiv_rn(__dmul_rn((double)L, T2), __dmul_rn(__dmul_rn(12.0, gA), gA));
        } else {
            const double g2 = __dmul_rn(__dmul_rn(__dmul_rn(gA, gA), gB), gB);
            if (k < nb) {
                term[2][t] = __ddiv_rn(__dmul_rn(T3, uni[0]), g2);
            } else {
                const double s = rep[k - nb][t];
                wterm[k - nb][t] =
                    __ddiv_rn(pp.noise_rms ? __dmul_rn(__dmul_rn(9.0, uni[1]), __dmul_rn(s, s))
                                           : __dmul_rn(T3, __dadd_rn(uni[0], __dmul_rn(s, s))),
                              g2);
            }
        }
    }
    __syncthreads();
    for (int i = warp; i < nw * ng; i += kTermWarps) {
        const int w = i / ng, g = i % ng, t = t_lo + 32 * g + lane;
        unsigned long long bn = ~0ull;
        int bt = -1;
        if (t <= t_hi && rep[w][t] >= 0.0) {
            double n = __dadd_rn(term[0][t], term[1][t]);
            if (pp.noise_rms) n = __dadd_rn(n, term[2][t]);
            // N >= 0: its bit pattern orders like its value
            bn = (unsigned long long)__double_as_longlong(__dadd_rn(n, wterm[w][t]));
            bt = t;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long n2 = __shfl_xor_sync(0xffffffffu, bn, off);
            const int t2 = __shfl_xor_sync(0xffffffffu, bt, off);
            if (t2 >= 0 && (bt < 0 || n2 < bn || (n2 == bn && t2 < bt))) { bn = n2; bt = t2; }
        }
        if (lane == 0) { best_n[w][g] = bn; best_t[w][g] = bt; }
    }
    __syncthreads();
    if (warp < nw) {                                   // W = Wreq - warp
        unsigned long long bn = ~0ull;
        int bt = -1;
        for (int g = 0; g < ng; ++g)                   // levels ascend
            if (best_t[warp][g] >= 0 && (bt < 0 || best_n[warp][g] < bn)) {
                bn = best_n[warp][g];
                bt = best_t[warp][g];
            }
        int ok = -1;                                   // no usable level
        if (bt >= 0) {
            const double N = __longlong_as_double((long long)bn);
            DevPlan c{};
            c.W = pp.Wreq - warp;
            c.level = bt;
            c.gA = gam[0][bt];
            c.gB = gam[1][bt];
            c.q = q_for(r_level(bt));
            c.R = (long long)L * c.gA * c.gB;
            c.Wef = w_ef(c.R, c.q, pp.p);
            c.s_rep = rep[warp][bt] > 0.0 ? rep[warp][bt] : 0.0;
            c.ratio = N <= 0.0 ? INFINITY : __ddiv_rn(S, N);
            c.log_pending = 1;
            ok = c.ratio > pp.target_ratio;
            if (!(fabs(c.ratio - pp.target_ratio) > 1e-9 * pp.target_ratio))
                ok = snr_db(S, N) >= pp.target_db;
            if (lane == 0) cand[warp] = c;
        }
        if (lane == 0) met[warp] = ok;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    int pick = -1, first = -1;
    for (int w = nw - 1; w >= 0; --w) {
        if (met[w] >= 0) first = w;
        if (met[w] > 0) pick = w;
    }
    DevPlan a{};
    if (pick >= 0) {
        a = cand[pick];
    } else if (pp.allow_fallback) {
        a.W = 1;
        a.level = -1;
        a.pred_snr = INFINITY;
    } else if (first >= 0) {
        a = cand[first];
        a.status = TDG_EUNREACHABLE;
    } else {
        a.W = pp.Wreq; a.q = q_for(L); a.gA = a.gB = 1; a.R = L;
        a.level = -1;
        a.pred_snr = NAN;
        a.status = TDG_EUNREACHABLE;
    }
    a.S = S;
    a.T1 = T1;
    a.T2 = T2;
    a.T3 = T3;
    write_plan(a, nf, plan);
}

// The plan of calls that take no statistics: the conventional product and
// manual companders (one warp).
__global__ void __launch_bounds__(32) planner_kernel(PlanParams pp, const double *__restrict__ stab,
                                                     DevPlan *plan) {
    pdl_entry();
    decide_plan(pp, stab, plan, 0.0, 0.0, 0.0, 0.0, rho_of(0.0, 0.0), 0);
}

// ---- Sec. 6: per inner kernel R_ij, predicted S_ij / N_ij with the call's
// companders.  One warp per inner kernel: lane u computes the terms of slab
// l0 + u, then every lane adds them in ascending l (the oracle's order), so
// the FP64 divisions spread over the warp while the sums keep their order.
__device__ inline void kernel_terms(const PlanParams &pp, const DevPlan &a, double va,
                                    double vb, double ma, double mb, double &s_out,
                                    double &n_out) {
    const double L = (double)pp.L;
    const double gA2 = __dmul_rn((double)a.gA, (double)a.gA), gB2 = __dmul_rn((double)a.gB, (double)a.gB);
    const double s = a.s_rep;
    const double ma2 = __dmul_rn(ma, ma), mb2 = __dmul_rn(mb, mb);
    s_out = __dmul_rn(__dmul_rn(L, va), vb);
    double n = __dadd_rn(__ddiv_rn(__dmul_rn(__dmul_rn(L, va), mb2), __dmul_rn(12.0, gB2)),
                         __ddiv_rn(__dmul_rn(__dmul_rn(L, vb), ma2), __dmul_rn(12.0, gA2)));
    if (pp.noise_rms) {
        n = __dadd_rn(n, __ddiv_rn(__dmul_rn(__dmul_rn(ma2, mb2), __ddiv_rn(L, 144.0)),
                                   __dmul_rn(gA2, gB2)));
        n = __dadd_rn(n, __ddiv_rn(__dmul_rn(__dmul_rn(__dmul_rn(9.0, va), vb), __dmul_rn(s, s)),
                                   __dmul_rn(gA2, gB2)));
    } else {
        n = __dadd_rn(n, __ddiv_rn(__dmul_rn(__dmul_rn(ma2, mb2),
                                             __dadd_rn(__ddiv_rn(L, 144.0), __dmul_rn(s, s))),
                                   __dmul_rn(gA2, gB2)));
    }
    n_out = n;
}

__global__ void kernel_ratio_kernel(PlanParams pp, const double *__restrict__ mA,
                                    const double *__restrict__ vA, const double *__restrict__ mB,
                                    const double *__restrict__ vB, const DevPlan *__restrict__ plan,
                                    double *ratio) {
    pdl_entry();
    const long long T = (long long)pp.nM * pp.nN;
    const long long t = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (t >= T) return;                      // uniform per warp
    const int i = (int)(t / pp.nN), j = (int)(t % pp.nN);
    const DevPlan a = *plan;
    if (a.W < 2) {
        if (lane == 0) ratio[t] = 0.0;
        return;
    }
    double S = 0.0, N = 0.0;
    for (int l0 = 0; l0 < pp.nK; l0 += 32) {
        const int l = l0 + lane;
        double sv = 0.0, nv = 0.0;
        if (l < pp.nK)
            kernel_terms(pp, a, vA[(long long)i * pp.nK + l], vB[(long long)l * pp.nN + j],
                         mA[(long long)i * pp.nK + l], mB[(long long)l * pp.nN + j], sv, nv);
        const int cnt = min(32, pp.nK - l0);
        for (int u = 0; u < cnt; ++u) {
            S = __dadd_rn(S, __shfl_sync(0xffffffffu, sv, u));
            N = __dadd_rn(N, __shfl_sync(0xffffffffu, nv, u));
        }
    }
    if (lane == 0) ratio[t] = N > 0.0 ? __ddiv_rn(S, N) : INFINITY;
}

// Sec. 6 (ii): the fewest of T inner kernels whose acceleration makes the
// product's predicted throughput T / ((T - k) + k / F_W) reach F, i.e.
// k = ceil(T (1 - 1/F) / (1 - 1/F_W)); none if F <= 1 or F_W <= 1, all if
// F >= F_W.  Every operation rounded as written (the oracle's order).
__device__ inline long long kernels_for_throughput(long long T, double F, double fw) {
    if (!(F > 1.0) || !(fw > 1.0)) return 0;
    if (F >= fw) return T;
    const double x = __ddiv_rn(__dmul_rn((double)T, __dsub_rn(1.0, __ddiv_rn(1.0, F))),
                               __dsub_rn(1.0, __ddiv_rn(1.0, fw)));
    const long long k = (long long)ceil(x);
    return k < 0 ? 0 : (k > T ? T : k);
}

// mode 1: ratio >= thr;  mode 2: rank (descending ratio, ties to the lower
// index) below k, counted against the ratios staged through shared memory;
// mode 3: as mode 2 with k from the throughput target.  Ratios are
// non-negative (or +inf), so their bit patterns order like the values and the
// O(T^2) rank count runs on the integer pipe.  A plan that fell back to W = 1
// accelerates nothing.
constexpr int kMaskThreads = 128, kMaskChunk = 2048;
__global__ void __launch_bounds__(kMaskThreads)
    kernel_mask_kernel(long long T, int mode, double thr, long long k, double F, Speedups fw,
                       const DevPlan *__restrict__ plan, const double *__restrict__ ratio,
                       unsigned char *mask) {
    pdl_entry();
    __shared__ unsigned long long chunk[kMaskChunk];
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int W = plan->W;
    const bool fell_back = W < 2;            // uniform
    if (mode == 3 && !fell_back) k = kernels_for_throughput(T, F, fw.fw[min(W, kMaxW)]);
    if (fell_back || mode == 1) {
        if (t < T) mask[t] = fell_back ? 0 : (ratio[t] >= thr ? 1 : 0);
        return;
    }
    const unsigned long long r =
        t < T ? (unsigned long long)__double_as_longlong(ratio[t]) : 0ull;
    long long rank = 0;
    for (long long c0 = 0; c0 < T; c0 += kMaskChunk) {
        const int n = (int)min((long long)kMaskChunk, T - c0);
        __syncthreads();
        for (int u = threadIdx.x; u < n; u += kMaskThreads)
            chunk[u] = (unsigned long long)__double_as_longlong(ratio[c0 + u]);
        __syncthreads();
        const long long tl = t - c0;         // ties count below this index
        for (int u = 0; u < n; ++u) {
            const unsigned long long ru = chunk[u];
            rank += (ru > r || (ru == r && u < tl)) ? 1 : 0;
        }
    }
    if (t < T) mask[t] = rank < k ? 1 : 0;
}

// One CTA: each thread counts the conventional tiles in its contiguous chunk
// of the row-major tile list, a block-wide exclusive scan gives every chunk
// its first position in both groups, and the chunk is written out.
constexpr int kOrderThreads = 1024;
__global__ void __launch_bounds__(kOrderThreads)
    tile_order_kernel(const unsigned char *__restrict__ mask, int nN, int L, int bm, int bn,
                      long long tiles_m, long long ntn, int *__restrict__ order) {
    pdl_entry();
    __shared__ long long scan[kOrderThreads];
    const long long n = tiles_m * ntn;
    const long long chunk = (n + kOrderThreads - 1) / kOrderThreads;
    const long long t0 = min(n, (long long)threadIdx.x * chunk), t1 = min(n, t0 + chunk);
    auto conventional = [&](long long t) {
        const long long tm = t / ntn, tn = t - tm * ntn;
        return mask[(tm * bm / L) * nN + (tn * bn / L)] == 0;
    };
    long long mine = 0;
    for (long long t = t0; t < t1; ++t) mine += conventional(t) ? 1 : 0;
    scan[threadIdx.x] = mine;
    __syncthreads();
    for (int off = 1; off < kOrderThreads; off <<= 1) {     // inclusive scan
        const long long v = threadIdx.x >= off ? scan[threadIdx.x - off] : 0;
        __syncthreads();
        scan[threadIdx.x] += v;
        __syncthreads();
    }
    const long long total_conv = scan[kOrderThreads - 1];
    long long pc = scan[threadIdx.x] - mine;                 // conventional tiles before t0
    long long pp = total_conv + (t0 - pc);                   // accelerated tiles before t0, offset
    for (long long t = t0; t < t1; ++t) {
        if (conventional(t)) order[pc++] = (int)t;
        else order[pp++] = (int)t;
    }
}

}  // namespace

cudaError_t launch_tile_order(const unsigned char *mask, int nN, int L, int bm, int bn,
                              long long tiles_m, long long ntn, int *order, cudaStream_t st) {
    return launch_pdl(tile_order_kernel, dim3(1), dim3(kOrderThreads), 0, st, mask, nN, L, bm,
                      bn, tiles_m, ntn, order);
}

cudaError_t launch_kernel_control(const PlanParams &pp, const double *mA, const double *vA,
                                  const double *mB, const double *vB, const DevPlan *plan,
                                  int mode, double thr, long long k, double F,
                                  const Speedups &fw, double *ratio, unsigned char *mask,
                                  cudaStream_t st) {
    const long long T = (long long)pp.nM * pp.nN, ctas = (T * 32 + 255) / 256;
    // Behind the statistics' full wave the few CTAs, launched early, pile up on the SMs
    // that are left first and share their fp64 pipes (fixed bits, 2048^3: the steps up to
    // the product took 73 us, with a plain launch 58).  A target's decision, one CTA,
    // leaves them all.  So few CTAs that no pile matters are launched early (1024^3,
    // eight of them: 131.0 us a call, with a plain launch 132.9).
    const bool pdl = pp.mode == MODE_TARGET || ctas <= 8 || pdl_for_grid(ctas);
    cudaError_t e = launch_pdl_if(pdl, kernel_ratio_kernel, dim3((unsigned)ctas), dim3(256), 0, st,
                                  pp, mA, vA, mB, vB, plan, ratio);
    if (e != cudaSuccess) return e;
    return launch_pdl(kernel_mask_kernel,
                      dim3((unsigned)((T + kMaskThreads - 1) / kMaskThreads)), dim3(kMaskThreads),
                      0, st, T, mode, thr, k, F, fw, plan, (const double *)ratio, mask);
}

cudaError_t launch_planner(const PlanParams &pp, const double *stab, DevPlan *plan,
                           cudaStream_t st) {
    if (pp.mode == MODE_TARGET && (pp.form == TDG_SYM || pp.form == TDG_ASYM))
        return launch_pdl(level_kernel, dim3(1), dim3(32 * kTermWarps), 0, st, pp, stab, plan);
    if (pp.form == TDG_PLAIN || pp.mode == MODE_MANUAL)
        return launch_pdl(planner_kernel, dim3(1), dim3(32), 0, st, pp, stab, plan);
    return cudaSuccess;      // decided by the statistics kernel
}

}  // namespace tdg
