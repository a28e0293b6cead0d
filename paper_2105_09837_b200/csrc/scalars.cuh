// The scalars of a layer that live on the device (so that an iteration of pdADMM-G needs no host round trip), and the steps that
// settle them from the sums over all nodes: tau, the acceptance of a quantised trial, theta.  A step is run by the kernel
// that completes its last sum.
#pragma once

#include "common.cuh"

namespace pd {

struct LayerScalars {
  double sum_g2;      // ||g||^2
  double sum_wg2;     // ||W g||^2
  double sum_d2;      // ||p+ - p||^2        (quantised trial)
  double sum_wd2;     // ||W (p+ - p)||^2    (quantised trial)
  double sum_G2;      // ||grad_W||^2
  double sum_Gp2;     // ||grad_W p+||^2
  double tau;         // tau_l
  double theta;       // theta_l (0 if grad_W = 0)
  float inv_tau;      // 1/tau
  float inv_theta;    // 1/theta, 0 if grad_W = 0
  int accepted;       // quantised trial: 1 if the stop condition held
  int trials;         // trials so far in this iteration
};

enum StepKind : int { STEP_NONE = 0, STEP_G2, STEP_TAU, STEP_TRIAL, STEP_THETA, STEP_SUM };
// What happens with the sum of squares of a product: it goes to its place in *sc (STEP_SUM: to *sum), and with `apply` (every
// other sum that the step needs is there already) the step itself follows.  Null words are skipped.
struct Step {
  int kind = STEP_NONE, apply = 0;
  LayerScalars *sc = nullptr;
  double *sum = nullptr;
  double rho = 0, nu = 0;
  int *nonfinite = nullptr;
  // Largest magnitudes (bit patterns) seen so far and exponents of planes that later kernels write before theirs are known.
  uint32_t *amax_p = nullptr, *amax_r = nullptr, *amax_W = nullptr;
  uint32_t *w_in = nullptr, *w_out = nullptr;      // STEP_TAU: max|g|, max|W g| (null: not kept); STEP_TRIAL: w_in = max|d|;
                                                   // STEP_THETA: w_in = max|G|; cleared here for the next iteration
  int *exp_p = nullptr, *exp_r = nullptr, *exp_W = nullptr, *exp_g = nullptr;
  volatile int *host_flag = nullptr;               // STEP_TRIAL: receives 1 or 0 (page-locked host memory)
};

__device__ __forceinline__ int tc_bound_exp(uint32_t a, uint32_t b, float factor) {       // of a + b * factor, a little up
  return tc_scale_exp(__float_as_uint((__uint_as_float(a) + __uint_as_float(b) * factor) * 1.0001f));
}

// One thread.
__device__ __forceinline__ void run_step(const Step &t) {
  LayerScalars *sc = t.sc;
  if (t.kind == STEP_TAU) {
    // tau = rho + nu ||W g||^2 / ||g||^2 : the smallest tau with phi(p - g/tau) <= U_l(p - g/tau; tau).
    // With max|W g| the p-step of pdADMM-G follows: |p+| <= max|p| + max|g|/tau and |r+| <= max|r| + max|W g|/tau are bounds.
    // Without, r after the trial is predicted from r before it.  g of the next iteration is predicted from this one's.
    const double gg = sc->sum_g2, wg = sc->sum_wg2;
    if (!(isfinite(gg) && isfinite(wg))) *t.nonfinite = 1;      // a NaN or Inf anywhere in the state reaches these sums
    const double tau = gg > 0.0 ? t.rho + t.nu * wg / gg : t.rho;
    const float inv_tau = (float)(1.0 / tau);
    sc->tau = tau;
    sc->inv_tau = inv_tau;
    sc->accepted = 0;
    sc->trials = 0;
    if (t.w_in == nullptr) return;
    if (t.exp_p != nullptr) *t.exp_p = tc_bound_exp(*t.amax_p, *t.w_in, inv_tau);
    *t.exp_r = t.w_out != nullptr ? tc_bound_exp(*t.amax_r, *t.w_out, inv_tau) : tc_predict_exp(*t.amax_r);
    *t.exp_g = tc_predict_exp(*t.w_in);
    *t.amax_p = 0u;                                             // max|p| of the layer restarts with the coming p-step
    *t.w_in = 0u;
    if (t.w_out != nullptr) *t.w_out = 0u;
  } else if (t.kind == STEP_TRIAL) {
    // Stop condition of the quantised step in its quadratic form: nu||W d||^2 + rho||d||^2 <= tau||d||^2 (1 + slack).
    // Not accepted: tau is doubled for the next trial.
    const bool ok = t.nu * sc->sum_wd2 + t.rho * sc->sum_d2 <= sc->tau * sc->sum_d2 * (1.0 + 1e-6);
    sc->trials += 1;
    sc->accepted = ok ? 1 : 0;
    if (!ok) {
      sc->tau *= 2.0;
      sc->inv_tau = (float)(1.0 / sc->tau);
    }
    if (t.w_in != nullptr) *t.w_in = 0u;
    if (t.host_flag != nullptr) { *t.host_flag = ok ? 1 : 0; __threadfence_system(); }
  } else if (t.kind == STEP_THETA) {
    // theta = nu ||grad_W p+||^2 / ||grad_W||^2 : the smallest theta with phi(W+) <= V_l(W+; theta).  W+ is bounded by
    // max|W| + max|G|/theta; the coming z-step's r and the next iteration's G are predicted from this iteration's.
    const double GG = sc->sum_G2, Gp = sc->sum_Gp2;
    if (!(isfinite(GG) && isfinite(Gp))) *t.nonfinite = 1;
    const double theta = GG > 0.0 ? t.nu * Gp / GG : 0.0;
    const float inv_theta = theta > 0.0 ? (float)(1.0 / theta) : 0.0f;
    sc->theta = theta;
    sc->inv_theta = inv_theta;
    if (t.w_in == nullptr) return;
    *t.exp_W = tc_bound_exp(*t.amax_W, *t.w_in, inv_theta);
    if (t.exp_r != nullptr) *t.exp_r = tc_predict_exp(*t.amax_r);
    *t.exp_g = tc_predict_exp(*t.w_in);
    *t.amax_r = 0u;                                             // max|r| restarts with the coming z-step, max|W| with the W-step
    *t.amax_W = 0u;
    *t.w_in = 0u;
  }
}
__device__ __forceinline__ void finish_step(const Step &t, double sum) {
  double *to = t.kind == STEP_G2 ? &t.sc->sum_g2 : t.kind == STEP_TAU ? &t.sc->sum_wg2 : t.kind == STEP_TRIAL ? &t.sc->sum_wd2
               : t.kind == STEP_THETA ? &t.sc->sum_Gp2 : t.sum;
  *to = sum;
  if (t.apply) run_step(t);
}

}  // namespace pd
