// The planner's device code that both the statistics kernels (whose last warp
// takes the sums over slabs and, outside target mode, decides the plan) and the
// candidate kernel of target mode run.
#pragma once

#include <math.h>

#include "tdg_common.cuh"

namespace tdg {

__device__ inline int t_max_for(int p) { return p == 24 ? 4 * 24 : 4 * 40; }


// eq. 21 summed over (i, l, j); operation order as written above.  With rms
// the representation term is scaled by the blocks' crest factors (s measured
// on uniform integers, RMS = max / sqrt(3)): 9 s^2 sum(sigma_A^2 sigma_B^2).
__device__ inline double model_noise(const DevPlan &a, int L, double gA, double gB, double s,
                                     int rms) {
    double t1 = __ddiv_rn(__dmul_rn((double)L, a.T1), __dmul_rn(__dmul_rn(12.0, gB), gB));
    double t2 = __ddiv_rn(__dmul_rn((double)L, a.T2), __dmul_rn(__dmul_rn(12.0, gA), gA));
    const double g2 = __dmul_rn(__dmul_rn(__dmul_rn(gA, gA), gB), gB);
    if (!rms) {
        double t3 = __ddiv_rn(__dmul_rn(a.T3, __dadd_rn(__ddiv_rn((double)L, 144.0), __dmul_rn(s, s))), g2);
        return __dadd_rn(__dadd_rn(t1, t2), t3);
    }
    double t3 = __ddiv_rn(__dmul_rn(a.T3, __ddiv_rn((double)L, 144.0)), g2);
    double t4 = __ddiv_rn(__dmul_rn(__dmul_rn(9.0, __ddiv_rn(a.S, (double)L)), __dmul_rn(s, s)), g2);
    return __dadd_rn(__dadd_rn(__dadd_rn(t1, t2), t3), t4);
}

__device__ inline double snr_db(double S, double N) {
    return N <= 0.0 ? INFINITY : 10.0 * log10(S / N);
}

// S / L, T1, T2, T3: products of the per-slab aggregates summed over slabs by
// one warp (lanes over l, then a fixed xor tree); every caller gets the same
// bits.
__device__ inline void slab_totals(const double *__restrict__ agg, int nK, double &S, double &T1,
                                   double &T2, double &T3) {
    const int lane = threadIdx.x & 31;
    S = T1 = T2 = T3 = 0.0;
    for (int l = lane; l < nK; l += 32) {
        const double X = __ldcg(&agg[4 * (long long)l]), MA = __ldcg(&agg[4 * (long long)l + 1]);
        const double Y = __ldcg(&agg[4 * (long long)l + 2]), MB = __ldcg(&agg[4 * (long long)l + 3]);
        S += X * Y;
        T1 += X * MB;
        T2 += Y * MA;
        T3 += MA * MB;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        S += __shfl_xor_sync(0xffffffffu, S, off);
        T1 += __shfl_xor_sync(0xffffffffu, T1, off);
        T2 += __shfl_xor_sync(0xffffffffu, T2, off);
        T3 += __shfl_xor_sync(0xffffffffu, T3, off);
    }
}

__device__ inline double rho_of(double T1, double T2) {
    return (T1 <= 0.0 || T2 <= 0.0) ? 1.0 : sqrt(T2 / T1);
}

// The decided plan into the record (one thread); nf: NaN or Inf was seen.
__device__ inline void write_plan(DevPlan a, int nf, DevPlan *plan) {
    a.nonfinite = nf;
    if (nf && a.status == 0) a.status = TDG_ENONFINITE;
    *plan = a;
}

// The plan, decided by one full warp: fixed bits, manual parameters and the
// tensor-core forms (a distortion target's choice of packing: level_kernel).
static __device__ __forceinline__ void decide_plan(const PlanParams &pp,
                                                const double *__restrict__ stab, DevPlan *plan,
                                                double S, double T1, double T2, double T3,
                                                double rho, int nf) {
    const int lane = threadIdx.x & 31;
    const int L = pp.L;
    DevPlan a{};
    a.S = (double)L * S;
    a.T1 = T1;
    a.T2 = T2;
    a.T3 = T3;
    a.status = 0;
    a.level = -1;
    a.pred_snr = NAN;
    a.s_rep = 0.0;

    if (pp.form == TDG_PLAIN) {
        a.W = 1; a.q = 0; a.gA = a.gB = 0; a.R = 0; a.Wef = 0;
    } else if (pp.form == TDG_TC_FP8) {
        a.W = 1; a.q = 0; a.gA = a.gB = (int)kFp8Max; a.R = 0; a.Wef = 0;
    } else if (pp.form == TDG_TC_INT) {
        int gA, gB;
        if (pp.mode == MODE_FIXED) {
            gA = gB = (1 << (pp.bits - 1)) - 1;
        } else {
            split_gammas((long long)kTcIntExact, L, rho, gA, gB);
            gA = min(gA, kTcIntMaxGamma);
            gB = min(min(gB, kTcIntMaxGamma), (int)((long long)kTcIntExact / ((long long)L * gA)));
        }
        a.W = 1; a.gA = gA; a.gB = gB; a.R = (long long)L * gA * gB;
        a.q = q_for(a.R); a.Wef = w_ef(a.R, a.q, pp.p);
        a.pred_snr = snr_db(a.S, model_noise(a, L, gA, gB, 0.0, pp.noise_rms));
        if (pp.mode == MODE_TARGET && a.pred_snr < pp.target_db) a.status = TDG_EUNREACHABLE;
    } else if (pp.mode == MODE_MANUAL) {
        a.W = pp.Wreq; a.q = pp.manual_q; a.gA = a.gB = 0; a.R = 0; a.Wef = 0;
    } else if (pp.mode == MODE_FIXED) {
        int g = (1 << (pp.bits - 1)) - 1;
        a.W = pp.Wreq; a.gA = a.gB = g; a.R = (long long)L * g * g;
        a.q = q_for(a.R); a.Wef = w_ef(a.R, a.q, pp.p);
        double s = -1.0;
        if (a.W <= a.Wef) {
            s = 0.0;
        } else if (stab) {
            int tbest = -1;
            for (int t = 0; t <= t_max_for(pp.p); ++t)
                if (r_level(t) <= a.R) tbest = t;
            if (tbest >= pp.t0 && tbest < pp.t0 + pp.nt)
                s = stab[(pp.Wreq - 2) * pp.nt + (tbest - pp.t0)];
        }
        if (s >= 0.0) {
            a.pred_snr = snr_db(a.S, model_noise(a, L, g, g, s, pp.noise_rms));
            a.s_rep = s;
        }
    }
    if (lane == 0) write_plan(a, nf, plan);
}

// What the blocks of a call count up to, and what the last of them does.  The
// counters are modulo counters: each wraps to zero with its last arrival in the
// same atomic, so no store can drop an arrival, and after any number of complete
// calls they stand at zero, also when two calls overlapped by mistake (their
// results are then undefined, the next call's are not).  Calls that reuse B count
// to another number and have counters of their own.
struct SlabFinish {
    PlanParams pp;
    const double *mA, *vA, *mB, *vB;   // block maxima and variances of op(A), op(B)
    const double *stab;
    double *agg;
    unsigned int *count;               // [nK] blocks per slab, [nK]: slabs
    int *nonfinite;                    // set by the statistics, cleared with the decision
    unsigned int blocks;               // arrivals per slab
};

// bytes of the counters and the flag of a plan: a counter set for calls that
// process both operands, one for calls that reuse B
constexpr size_t slab_count_bytes(int nK) { return (2 * ((size_t)nK + 1) + 1) * sizeof(unsigned int); }
inline void set_slab_counters(SlabFinish &f, unsigned int *counters, bool reuse_b) {
    const size_t set = (size_t)f.pp.nK + 1;
    f.count = counters + (reuse_b ? set : 0);
    f.nonfinite = reinterpret_cast<int *>(counters + 2 * set);
    f.blocks = (unsigned int)(f.pp.nM + (reuse_b ? 0 : f.pp.nN));
}

// One arrival on a modulo-n counter, ordered after this thread's (and, behind a
// barrier, its CTA's) writes and before what it reads next; lighter than
// __threadfence() around a relaxed atomic, which orders sequentially consistently.
// True for the last of n.
__device__ inline bool last_arrival(unsigned int *p, unsigned int n) {
#ifdef __CUDA_ARCH__
    unsigned int v;
    asm volatile("atom.inc.acq_rel.gpu.global.u32 %0, [%1], %2;"
                 : "=r"(v)
                 : "l"(p), "r"(n - 1)
                 : "memory");
#else
    const unsigned int v = *p;
    *p = v + 1 < n ? v + 1 : 0;
#endif
    return v == n - 1;
}

// Called by one full warp of a statistics CTA once its block of slab l is
// written by lane 0: the last of the slab's blocks takes the slab's aggregates
// (lanes over the blocks, as slab_aggregate_warp orders them), the last slab
// the sums over slabs and rho -- and decides the plan, except for the packed
// forms' target mode, whose candidates need a kernel of their own.  Counters
// only, no waiting.  (A kernel of its own for the aggregates, and one for the
// decision, took 7-9 and 2.5-8 us of a call.  Inlined: as a call it cost the
// statistics and code kernels 1 to 3 us.  A target's candidates stay a kernel of
// their own: evaluated by this warp, three rounds of fp64 work, a 4096^3 fp32 call
// took 1217 us instead of 1204.)
static __device__ __forceinline__ void slab_finish(const SlabFinish &f, int l, DevPlan *plan) {
    const int lane = threadIdx.x & 31;
    int last = 0;
    if (lane == 0) last = last_arrival(&f.count[l], f.blocks);
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __syncwarp();
    const bool modelled = f.pp.form != TDG_TC_FP8;      // E4M3 has no noise model
    if (modelled) slab_aggregate_warp(l, f.pp.nM, f.pp.nK, f.pp.nN, f.mA, f.vA, f.mB, f.vB, f.agg);
    if (lane == 0) last = last_arrival(&f.count[f.pp.nK], (unsigned int)f.pp.nK);
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __syncwarp();
    // (on its way while the sums are taken)
    const int nf = lane == 0 ? atomicExch(f.nonfinite, 0) : 0;
    double S = 0.0, T1 = 0.0, T2 = 0.0, T3 = 0.0;
    if (modelled) slab_totals(f.agg, f.pp.nK, S, T1, T2, T3);
    const double rho = rho_of(T1, T2);
    if (f.pp.mode == MODE_TARGET && (f.pp.form == TDG_SYM || f.pp.form == TDG_ASYM)) {
        if (lane == 0) {
            plan->tS = S;
            plan->tT1 = T1;
            plan->tT2 = T2;
            plan->tT3 = T3;
            plan->trho = rho;
            plan->tnonfinite = nf;
        }
    } else {
        decide_plan(f.pp, f.stab, plan, S, T1, T2, T3, rho, nf);
    }
}

}  // namespace tdg
