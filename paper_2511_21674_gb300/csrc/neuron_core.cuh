// One neuron's update and one readout's error signal, on values in
// registers: shared by the per-step kernels, the persistent step loop and
// the sample-resident step loop, so all of them compute the same bits.
#pragma once
#include "eprop_internal.cuh"

namespace eprop {

// State of one neuron between steps: v and a as FP32 pairs (hi + lo), the
// refractory count, the last spike and the filtered rate.
struct NeuronRegs {
    float v_hi, v_lo, a_hi, a_lo;
    int ref;
    float zp;                  // spike of the previous step, 0 or 1
    float rate;
};

// External drive of neuron j of sample b at absolute step t_abs: the number
// of thresholds at or below the hash's upper 32 bits (0 without drive).
__device__ __forceinline__ int drive_count(const Net &n, int b, int j, long long t_abs, const uint32_t *thr_s) {
    if (n.n_thr == 0) return 0;
    const uint64_t h = mix64(mix64(mix64(n.drive_seed ^ (uint64_t)j) ^ (uint64_t)t_abs) ^ (uint64_t)b);
    const uint32_t u = (uint32_t)(h >> 32);
    // thresholds are non-decreasing (checked at creation): the count of
    // thresholds <= u is the index of the first one above u
    int cnt = 0;
    while (cnt < n.n_thr && u >= thr_s[cnt]) ++cnt;
    return cnt;
}

// Update of neuron j at absolute step t_abs from its arrivals acc_q (fixed
// point) and its drive count (Eq. lif_update, Eq. binary-spike-state-variable, Eq.
// spike-threshold-adaptation, the surrogate).  forced_z >= 0 gives the spike.
// VAR: the e-prop+ variants (fixed reset, ignore-and-fire, exponential
// surrogate, rate regularisation) are compiled in; the plain method's
// instance carries none of their code.  DRIVE: the external drive is.
template <bool VAR, bool DRIVE = true>
__device__ __forceinline__ void neuron_core(const Net &n, int j, long long t_abs, int cnt, long long acc_q,
                                            int forced_z, NeuronRegs &s, float &psi, int &z) {
    // exact fixed-point input split into an FP32 pair
    float u_hi, u_lo;
    fixed_to_pair(acc_q, u_hi, u_lo);
    if (DRIVE && n.n_thr > 0) {
        const float dv = n.drive_weight * (float)cnt;
        const float de = fmaf(n.drive_weight, (float)cnt, -dv);
        float e;
        two_sum(u_hi, dv, u_hi, e);
        u_lo += e + de;
    }
    const float zp = s.zp;
    float vth = n.v_th, vth_lo = 0.0f;
    if (n.alif) {
        comp_step(n.rho, n.rho_lo, zp, 0.0f, s.a_hi, s.a_lo);
        vth = fmaf(n.beta_a, s.a_hi, n.v_th);
        vth_lo = fmaf(n.beta_a, s.a_hi, n.v_th - vth) + n.beta_a * s.a_lo;
    }
    if (VAR && n.reset_mode == 1 && zp != 0.0f) {
        // fixed reset: v' = v_reset + I (the decayed membrane is replaced)
        float sm, e;
        two_sum(n.v_reset, u_hi, sm, e);
        const float lo = e + u_lo;
        const float hi = sm + lo;
        s.v_lo = lo - (hi - sm);
        s.v_hi = hi;
    } else {
        // v' = alpha v + I - z_prev v_th (Eq. lif_update), input term as a pair
        if (!VAR || n.reset_mode == 0) {
            float e;
            two_sum(u_hi, -zp * vth, u_hi, e);
            u_lo += e - zp * vth_lo;
        }
        comp_step(n.alpha, n.alpha_lo, u_hi, u_lo, s.v_hi, s.v_lo);
    }
    const float m = (s.v_hi - vth) + (s.v_lo - vth_lo);
    const bool refractory = s.ref > 0;
    if (forced_z >= 0) {
        z = forced_z;
    } else if (VAR && n.if_period > 0) {
        // ignore-and-fire: a fixed schedule with the neuron's own phase
        const uint32_t ph = (uint32_t)(mix64(n.if_seed ^ (uint64_t)j) >> 32) % (uint32_t)n.if_period;
        z = ((t_abs + (long long)ph) % n.if_period) == 0 ? 1 : 0;
    } else {
        z = (!refractory && m > 0.0f) ? 1 : 0;
    }
    if (VAR && n.surrogate == 1) {      // Eq. exponential-surrogate-gradient
        psi = refractory ? 0.0f : n.gamma * expf(-n.beta_sg * fabsf(m));
    } else {                     // Eq. piecewise-linear-surrogate-gradient
        const float hh = 1.0f - n.beta_sg * fabsf(m);
        psi = refractory ? 0.0f : n.gamma * fmaxf(hh, 0.0f);
    }
    if (VAR && n.R_win) s.rate = n.beta_reg * s.rate + (1.0f - n.beta_reg) * (float)z;   // Eq. ema-rate
    if (refractory) s.ref -= 1;
    if (z) s.ref = n.t_ref;
    s.zp = (float)z;
}

// regularisation signal of Eq. ema-gradient with G_beta's factor (1 - beta)
__device__ __forceinline__ float rate_signal(const Net &n, float rate) {
    return n.c_reg * (1.0f - n.beta_reg) * (rate - n.f_target);
}

// Leaky readout (Eq. leaky_integrator): y' = kappa y + input, the input
// summed in fixed point
__device__ __forceinline__ float readout_step(const Net &n, float y, long long acc) {
    float in, rest;                      // in = the sum rounded to FP32
    fixed_to_pair(acc, in, rest);
    return __fadd_rn(in, __fmul_rn(n.kappa, y));
}

// Error signal E_k and this readout's share of the step's loss (Eq. mean-
// squared-error / Eq. softmax, Eq. cross-entropy-loss / Eq. temporal-mse);
// rmax and rsum reduce over the readouts.
template <class RMax, class RSum>
__device__ __forceinline__ float error_signal(const Net &n, float y, float tgt, float win, bool has_k, float &E,
                                              RMax rmax, RSum rsum) {
    if (n.loss == 0) {
        const float diff = y - tgt;
        E = win * diff;
        return has_k ? 0.5f * win * diff * diff : 0.0f;
    }
    if (n.loss == 2) {        // temporal MSE (Eq. temporal-mse)
        const float diff = y - tgt;
        const float invK = 1.0f / (float)n.n_out;
        E = win * (2.0f * invK) * diff;
        return has_k ? win * diff * diff * invK : 0.0f;
    }
    const float mx = rmax(has_k ? y : -INFINITY);
    const float ex = has_k ? expf(y - mx) : 0.0f;
    const float den = rsum(ex);
    E = win * (ex / den - tgt);
    return has_k ? -win * tgt * ((y - mx) - logf(den)) : 0.0f;
}

}  // namespace eprop
