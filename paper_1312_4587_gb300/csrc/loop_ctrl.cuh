// Placement-loop control scalars (Algorithm 1 with a Nesterov step; the
// parameter control of Section IV-A), kept in FP64 in device memory and
// updated by the last CTA of the kernel that produces their inputs (a CTA
// learns it is last from an atomic ticket after a memory fence; nothing
// waits, so no kernel can hang on it).
//
// The updates sit on the critical path of every iteration and the FP64 pipe
// is narrow, so a warp reads the 32 stripes of a sum with one load per lane,
// and what does not depend on an update's own input is formed beside it:
// lambda_k (for k >= 1 from the HPWL change alone) and the momentum weight by
// one block of the cell kernel, gamma_{k+1} by a second warp.  With one thread
// walking the stripes, pow() and every scalar in line, the three updates took
// 10 + 14 + 18 us of an iteration at 210K cells.
#pragma once

#include "fftpl_internal.cuh"

namespace fftpl {

enum {
    C_LAMBDA = 0, C_GAMMA, C_ALPHA, C_ALPHA_MAX, C_A, C_BETA, C_HP_PREV, C_K, C_DONE, C_A_NEXT,
    C_ALPHA_MAX0, C_DW_REF, C_GAMMA_FIXED, C_LAMBDA0_OPT, C_STOP_ON_TAU, C_TAU_STOP, C_WB,
    C_HALF_AB, C_MOV_AREA, C_REC_CAP, C_REC_BASE,
    // conjugate-gradient loop: |g_{k-1}|^2, f_k, slope along d/|d|_inf,
    // |d|_inf, restart flag, and the values recorded for iteration k
    C_GG_PREV, C_FK, C_SLOPE, C_DINF, C_RESTART, C_W_K, C_HP_K, C_N_K, C_TAU_K,
    C_ALPHA_CAP,   // ceiling of alpha_max in the Nesterov loop (0: none)
    // float32 copies of the values the per-element kernels read (F_*),
    // packed two to a slot
    C_FMIRROR, C_FMIRROR_LAST = C_FMIRROR + 4,
    C_COUNT
};

// The per-element kernels read their control values as float32 from this
// mirror, written by whichever thread last changed the FP64 scalars (the
// FP64 pipe of the GPU is narrow: a double compare, conversion or division
// per thread costs more than the kernel's own arithmetic).  The values are
// those the kernels computed before from the FP64 scalars.
enum {
    F_DONE = 0, F_FIRST, F_LAMBDA, F_ALPHA, F_BETA, F_RESTART, F_SCALE_TRIAL, F_SCALE_UPDATE,
    F_INV_G, F_L2G,   // 1/gamma and log2(e)/gamma (adjacent: one 8-byte load)
    F_COUNT
};
static_assert(F_COUNT <= 2 * (C_FMIRROR_LAST - C_FMIRROR + 1), "control mirror too small");
static_assert(F_INV_G % 2 == 0, "1/gamma and log2(e)/gamma share an 8-byte word");

__host__ __device__ inline float* ctrl_f(double* ctrl) {
    return reinterpret_cast<float*>(ctrl + C_FMIRROR);
}
__host__ __device__ inline const float* ctrl_f(const double* ctrl) {
    return reinterpret_cast<const float*>(ctrl + C_FMIRROR);
}

__host__ __device__ inline void ctrl_mirror(double* ctrl) {
    float* f = ctrl_f(ctrl);
    f[F_DONE] = ctrl[C_DONE] != 0.0 ? 1.0f : 0.0f;
    f[F_FIRST] = ctrl[C_K] == 0.0 ? 1.0f : 0.0f;
    f[F_LAMBDA] = (float)ctrl[C_LAMBDA];
    f[F_ALPHA] = (float)ctrl[C_ALPHA];
    f[F_BETA] = (float)ctrl[C_BETA];
    f[F_RESTART] = ctrl[C_RESTART] != 0.0 ? 1.0f : 0.0f;
    const double dinf = ctrl[C_DINF];
    f[F_SCALE_TRIAL] = dinf > 0.0 ? (float)(ctrl[C_ALPHA_MAX] / dinf) : 0.0f;
    f[F_SCALE_UPDATE] = dinf > 0.0 ? (float)(ctrl[C_ALPHA] / dinf) : 0.0f;
    const float g = (float)ctrl[C_GAMMA];
    if (g > 0.0f) wa_scale(g, &f[F_INV_G], &f[F_L2G]);
}
constexpr int kRecFields = 8;
// Doubles after the control scalars that are not part of a saved state: one
// ticket counter per loop kernel kind (32 bits each), then what one kernel of
// an iteration leaves for the next.
constexpr int kCounters = 8;
enum { S_GAMMA_NEXT = C_COUNT + 4, S_SCALE_NEXT /* 1/gamma, log2(e)/gamma as floats */ };
static_assert(S_SCALE_NEXT < C_COUNT + kCounters, "loop scratch too small");

// After a block barrier (which orders every thread's earlier reductions
// before thread 0's next operations), thread 0 fences at device scope and
// takes a ticket; the CTA that draws the last ticket resets the counter,
// fences again (its later reads see every CTA's reductions) and returns
// true.  One fence per block: a fence in every thread held each thread
// until its own stores had completed, which doubled the loop's vector
// kernels.
__device__ __forceinline__ bool last_cta(unsigned int* counter) {
    __shared__ bool is_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned int t = atomicAdd(counter, 1u);
        is_last = (t == gridDim.x - 1);
        if (is_last) {
            *counter = 0u;
            __threadfence();
        }
    }
    __syncthreads();
    return is_last;
}

// Totals of the striped accumulators (read past L1), one stripe per lane;
// called by a full warp, every lane gets the total.
__device__ __forceinline__ double acc_sum(const double* acc, int q) {
    static_assert(kAccStripes == 32, "one stripe per lane");
    double s = __ldcg(acc + (threadIdx.x & 31) * kAccStride + q);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}
// (non-negative values: ordered as their bit patterns)
__device__ __forceinline__ double acc_max(const double* acc, int q) {
    long long s = __double_as_longlong(__ldcg(acc + (threadIdx.x & 31) * kAccStride + q));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = max(s, __shfl_xor_sync(0xffffffffu, s, o));
    return __longlong_as_double(s);
}

// lambda_0 = ||grad W~||_1 / ||grad N||_1 unless given (a full warp).
__device__ __forceinline__ double lambda_start(const double* acc) {
    const double gn = acc_sum(acc, ACC_GN_L1), gw = acc_sum(acc, ACC_GW_L1);
    return gn > 0.0 ? gw / gn : 1.0;
}
// whether the first iteration forms lambda_0 itself
__device__ __forceinline__ bool lambda_from_norms(const double* ctrl) {
    return ctrl_f(ctrl)[F_FIRST] != 0.0f && !(ctrl[C_LAMBDA0_OPT] > 0.0);
}

// After the wirelength kernel (one warp): lambda_k for k >= 1, mu_k lambda_{k-1} with mu_k = 1.1^(-dW/dW_ref + 1) bounded to
// [0.75, 1.1], dW the HPWL change (1.1^z as exp(z ln 1.1)); and the momentum
// weight of iteration k, a_{k+1} = (1 + sqrt(1 + 4 a_k^2)) / 2,
// beta_k = (a_k - 1) / a_{k+1}.
__device__ __forceinline__ void ctrl_lambda(double* ctrl, const double* acc) {
    const double hp = acc_sum(acc, ACC_HPWL);
    if ((threadIdx.x & 31) != 0) return;
    float* f = ctrl_f(ctrl);
    if (ctrl[C_K] >= 1.0) {
        const double z = -(hp - ctrl[C_HP_PREV]) / ctrl[C_DW_REF] + 1.0;
        const double mu = z >= 1.0 ? 1.1 : exp(z * 0.095310179804324860044);
        const double lam = ctrl[C_LAMBDA] * fmin(1.1, fmax(0.75, mu));
        ctrl[C_LAMBDA] = lam;
        f[F_LAMBDA] = (float)lam;
    }
    ctrl[C_HP_PREV] = hp;
}
__device__ __forceinline__ void ctrl_momentum(double* ctrl) {
    const double a = ctrl[C_A];
    const double an = 0.5 * (1.0 + sqrt(1.0 + 4.0 * a * a)), beta = (a - 1.0) / an;
    ctrl[C_A_NEXT] = an;
    ctrl[C_BETA] = beta;
    ctrl_f(ctrl)[F_BETA] = (float)beta;
}

// gamma = 8.0 w_b 10^((20/9)(tau - 0.1) - 1) (Section IV-A).
__device__ __forceinline__ double gamma_schedule(double tau, double wb) {
    return 8.0 * wb * exp10((20.0 / 9.0) * (tau - 0.1) - 1.0);
}

// gamma_{k+1} and its float32 factors into the loop scratch (a full warp; the
// overflow of the evaluated point is known since the row pass).
__device__ __forceinline__ void ctrl_gamma_next(double* ctrl, const double* acc) {
    const double tau = acc_sum(acc, ACC_TAU) / ctrl[C_MOV_AREA];
    if ((threadIdx.x & 31) != 0 || ctrl[C_GAMMA_FIXED] > 0.0) return;
    const double g = gamma_schedule(tau, ctrl[C_WB]);
    float* sc = reinterpret_cast<float*>(ctrl + S_SCALE_NEXT);
    ctrl[S_GAMMA_NEXT] = g;
    wa_scale((float)g, sc, sc + 1);
}
// gamma_{k+1} in force (one thread).
__device__ __forceinline__ void ctrl_take_gamma(double* ctrl) {
    if (ctrl[C_GAMMA_FIXED] > 0.0) return;
    float* f = ctrl_f(ctrl);
    const double g = ctrl[S_GAMMA_NEXT];
    const float* sc = reinterpret_cast<const float*>(ctrl + S_SCALE_NEXT);
    ctrl[C_GAMMA] = g;
    if ((float)g > 0.0f) {
        f[F_INV_G] = sc[0];
        f[F_L2G] = sc[1];
    }
}

// After the combined gradient (a full warp): the step alpha_k.
// alpha_0 = alpha_max_0 / ||g||_inf; alpha_k = ||v_k - v_{k-1}|| / ||g_k - g_{k-1}||;
// alpha_k ||g||_inf is then kept within [0.01 alpha_max_k, alpha_max_k].
__device__ __forceinline__ void ctrl_alpha(double* ctrl, const double* acc) {
    // the scalars' loads go out with the stripes'
    double alpha = ctrl[C_ALPHA];
    const double amax = ctrl[C_ALPHA_MAX], amax0 = ctrl[C_ALPHA_MAX0], k = ctrl[C_K];
    const double ginf = acc_max(acc, ACC_GINF);
    const double dg2 = acc_sum(acc, ACC_DG2), dv2 = acc_sum(acc, ACC_DV2);
    if ((threadIdx.x & 31) != 0) return;
    if (k == 0.0) {
        alpha = ginf > 0.0 ? amax0 / ginf : 0.0;
    } else if (dg2 > 0.0) {
        alpha = sqrt(dv2) / sqrt(dg2);
    }
    if (ginf > 0.0) {
        if (alpha * ginf > amax) alpha = amax / ginf;
        if (alpha * ginf < 0.01 * amax) alpha = 0.01 * amax / ginf;
    }
    ctrl[C_ALPHA] = alpha;
    ctrl_f(ctrl)[F_ALPHA] = (float)alpha;
}

// Counts iteration k done: k + 1 and the stop test (one thread).
__device__ __forceinline__ void ctrl_advance(double* ctrl, int k, double tau) {
    float* f = ctrl_f(ctrl);
    ctrl[C_K] = (double)(k + 1);
    f[F_FIRST] = 0.0f;
    if (ctrl[C_STOP_ON_TAU] != 0.0 && tau <= ctrl[C_TAU_STOP]) {
        ctrl[C_DONE] = 1.0;
        f[F_DONE] = 1.0f;
    }
}

// After the position update (a full warp): record iteration k, then
// alpha_max_{k+1}, gamma_{k+1}, k+1 and the stop test tau <= tau_stop.
// Adaptive restart (the gradient test of O'Donoghue and Candes, 2015), one
// iteration late: when g_k . (u_{k+1} - u_k) > 0 the momentum sequence starts
// over, a_{k+1} = 1, so that the next momentum weight is 0.  alpha_max_{k+1}
// is kept at or below the handle's ceiling (alpha_max_cap_bins bin widths).
__device__ __forceinline__ void ctrl_record(double* ctrl, const double* acc, double* recs) {
    // the scalars' loads go out with the stripes'
    const double kd = ctrl[C_K], mov = ctrl[C_MOV_AREA], base = ctrl[C_REC_BASE],
                 cap = ctrl[C_REC_CAP], half_ab = ctrl[C_HALF_AB], lam = ctrl[C_LAMBDA],
                 gam = ctrl[C_GAMMA], alpha = ctrl[C_ALPHA], an = ctrl[C_A_NEXT],
                 amax0 = ctrl[C_ALPHA_MAX0], acap = ctrl[C_ALPHA_CAP];
    const double area = acc_sum(acc, ACC_TAU), step_max = acc_max(acc, ACC_STEPMAX);
    const double W = acc_sum(acc, ACC_W), hp = acc_sum(acc, ACC_HPWL), N = acc_sum(acc, ACC_N);
    const double gd = acc_sum(acc, ACC_GD);
    if ((threadIdx.x & 31) != 0) return;
    const int k = (int)kd;
    const double tau = area / mov;
    int slot = k - (int)base;
    if (slot >= 0 && slot < (int)cap) {
        double* r = recs + (size_t)slot * kRecFields;
        r[0] = W;
        r[1] = hp;
        r[2] = N * half_ab;
        r[3] = tau;
        r[4] = lam;
        r[5] = gam;
        r[6] = alpha;
        r[7] = step_max;
    }
    ctrl[C_A] = gd > 0.0 ? 1.0 : an;
    double amax = fmax(amax0, 2.0 * step_max);
    if (acap > 0.0) amax = fmin(amax, fmax(acap, amax0));
    ctrl[C_ALPHA_MAX] = amax;
    ctrl_take_gamma(ctrl);
    ctrl_advance(ctrl, k, tau);
}

// ------------------------------------------------ conjugate-gradient loop
// Algorithm 1's CGsolver with the search interval [0.01 a_max, a_max] of
// Section IV-A: Polak-Ribiere+ directions, the step measured as the farthest
// cell move (direction scaled by 1/|d|_inf), one quadratic-fit line search
// from f_k, the slope and one trial evaluation at a_max.

// After g_k (a full warp): beta_k (PR+), f_k and the values recorded for
// iteration k.
__device__ __forceinline__ void ctrl_cg_g(double* ctrl, const double* acc) {
    const double gg = acc_sum(acc, ACC_DG2), ggp = acc_sum(acc, ACC_DV2);
    const double W = acc_sum(acc, ACC_W), hp = acc_sum(acc, ACC_HPWL);
    const double N = acc_sum(acc, ACC_N) * ctrl[C_HALF_AB];
    const double tau = acc_sum(acc, ACC_TAU) / ctrl[C_MOV_AREA];
    if ((threadIdx.x & 31) != 0) return;
    const double prev = ctrl[C_GG_PREV];
    const double beta = (ctrl[C_K] > 0.0 && prev > 0.0) ? fmax(0.0, (gg - ggp) / prev) : 0.0;
    ctrl[C_BETA] = beta;
    ctrl_f(ctrl)[F_BETA] = (float)beta;
    ctrl[C_GG_PREV] = gg;
    ctrl[C_FK] = W + ctrl[C_LAMBDA] * N;
    ctrl[C_W_K] = W;
    ctrl[C_HP_K] = hp;
    ctrl[C_N_K] = N;
    ctrl[C_TAU_K] = tau;
}

// After d_k (a full warp): restart to -g_k unless g_k . d_k < 0; |d|_inf and
// the slope.
__device__ __forceinline__ void ctrl_cg_dir(double* ctrl, const double* acc) {
    double gd = acc_sum(acc, ACC_GD), dinf = acc_max(acc, ACC_DINF);
    const double ginf = acc_max(acc, ACC_GINF);
    if ((threadIdx.x & 31) != 0) return;
    float* f = ctrl_f(ctrl);
    const bool restart = !(gd < 0.0);
    if (restart) {
        dinf = ginf;
        gd = -ctrl[C_GG_PREV];
    }
    ctrl[C_RESTART] = restart ? 1.0 : 0.0;
    f[F_RESTART] = restart ? 1.0f : 0.0f;
    ctrl[C_DINF] = dinf;
    ctrl[C_SLOPE] = dinf > 0.0 ? gd / dinf : 0.0;
    f[F_SCALE_TRIAL] = dinf > 0.0 ? (float)(ctrl[C_ALPHA_MAX] / dinf) : 0.0f;
}

// After the trial evaluation at a_max (a full warp): the step a_k from the
// parabola through f_k (slope s) and f_t, kept in [0.01 a_max, a_max].
__device__ __forceinline__ void ctrl_cg_alpha(double* ctrl, const double* acc) {
    const double W = acc_sum(acc, ACC_W), N = acc_sum(acc, ACC_N);
    if ((threadIdx.x & 31) != 0) return;
    const double amax = ctrl[C_ALPHA_MAX], dinf = ctrl[C_DINF];
    double alpha = 0.0;
    if (dinf > 0.0) {
        double ft = W + ctrl[C_LAMBDA] * N * ctrl[C_HALF_AB];
        double s = ctrl[C_SLOPE];
        double c = (ft - ctrl[C_FK] - s * amax) / (amax * amax);
        double as = c > 0.0 ? -s / (2.0 * c) : amax;
        alpha = fmin(amax, fmax(0.01 * amax, as));
    }
    float* f = ctrl_f(ctrl);
    ctrl[C_ALPHA] = alpha;
    f[F_ALPHA] = (float)alpha;
    f[F_SCALE_UPDATE] = dinf > 0.0 ? (float)(alpha / dinf) : 0.0f;
}

// After the position update (one thread): record iteration k, then
// a_max_{k+1} = max(a_max_0, 2 a_k), gamma_{k+1}, k+1 and the stop test.
__device__ __forceinline__ void ctrl_record_cg(double* ctrl, double* recs) {
    int k = (int)ctrl[C_K];
    double tau = ctrl[C_TAU_K], alpha = ctrl[C_ALPHA];
    int slot = k - (int)ctrl[C_REC_BASE];
    if (slot >= 0 && slot < (int)ctrl[C_REC_CAP]) {
        double* r = recs + (size_t)slot * kRecFields;
        r[0] = ctrl[C_W_K];
        r[1] = ctrl[C_HP_K];
        r[2] = ctrl[C_N_K];
        r[3] = tau;
        r[4] = ctrl[C_LAMBDA];
        r[5] = ctrl[C_GAMMA];
        r[6] = alpha;
        r[7] = alpha;
    }
    ctrl[C_ALPHA_MAX] = fmax(ctrl[C_ALPHA_MAX0], 2.0 * alpha);
    ctrl_take_gamma(ctrl);
    ctrl_advance(ctrl, k, tau);
}

}  // namespace fftpl
