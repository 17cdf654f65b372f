// The FP32 arithmetic of one GD step per element (Eqs. 2, 5, 6; Sec. 2 RK4),
// shared by every step kernel: right-hand side, coupling scales, noise scale.
//
// Columns come in quads c0..c0+3 (c0 a multiple of 4): four Ising restarts, or
// two XY restarts as (re, im) pairs; one Philox call with counter (i, c0/4,
// step, 0) gives the quad's four normals, z_k for column c0+k (scaled by
// 1/sqrt 2 for complex amplitudes).
#pragma once
#include "gda_internal.h"
#include "philox.cuh"

namespace gda {

// Every rounding below is explicit (fused multiply-add, IEEE add / multiply /
// divide / square root), so each kernel that performs an update computes the
// same bits whatever code surrounds it.

// d beta / dt = eps_hat (1 - beta) (Eq. 6 with Delta = 1, K = beta J).
__device__ __forceinline__ float beta_rate(float eh, float b) { return __fmul_rn(eh, __fsub_rn(1.0f, b)); }

// Stage coupling scale beta_s of a restart for the launch's mode.
__device__ __forceinline__ float stage_beta(const StepArgs& a, float b) {
  const float eh = a.eps_hat, hdt = __fmul_rn(0.5f, a.dt);
  switch (a.mode) {
    case M_RK2: return __fmaf_rn(hdt, beta_rate(eh, b), b);
    case M_RK3: {
      const float b2 = __fmaf_rn(hdt, beta_rate(eh, b), b);
      return __fmaf_rn(hdt, beta_rate(eh, b2), b);
    }
    case M_RK4: {
      const float b2 = __fmaf_rn(hdt, beta_rate(eh, b), b);
      const float b3 = __fmaf_rn(hdt, beta_rate(eh, b2), b);
      return __fmaf_rn(a.dt, beta_rate(eh, b3), b);
    }
    case M_ENERGY: return 1.0f;
    default: return b;
  }
}

// beta^{n+1} from beta^n for a completed Euler or RK4 step.
__device__ __forceinline__ float next_beta(const StepArgs& a, float b) {
  const float eh = a.eps_hat, dt = a.dt, hdt = __fmul_rn(0.5f, a.dt);
  if (a.mode == M_EULER) return __fmaf_rn(dt, beta_rate(eh, b), b);
  const float k1 = beta_rate(eh, b);
  const float k2 = beta_rate(eh, __fmaf_rn(hdt, k1, b));
  const float k3 = beta_rate(eh, __fmaf_rn(hdt, k2, b));
  const float k4 = beta_rate(eh, __fmaf_rn(dt, k3, b));
  const float sum = __fadd_rn(__fadd_rn(__fadd_rn(k1, __fmul_rn(2.0f, k2)), __fmul_rn(2.0f, k3)), k4);
  return __fmaf_rn(__fdiv_rn(dt, 6.0f), sum, b);
}

__device__ __forceinline__ bool step_completes(int mode) { return mode == M_EULER || mode == M_RK4; }

// Noise amplitude sqrt(dt) D_r (times 1/sqrt 2 for complex amplitudes) of
// restart r; D_r = D max(0, 1 - mean_i rho_i / rho_th) under noise decay,
// with the mean over the N spins of psi^n from the per-tile partial sums.
__device__ __forceinline__ float noise_scale(const StepArgs& a, int r) {
  if (!step_completes(a.mode) || a.noise_D == 0.0f) return 0.0f;
  float D = a.noise_D;
  if (a.noise_decay) {
    float s = 0.0f;
    for (int t = 0; t < a.mt_count; ++t) s = __fadd_rn(s, a.rho_in[t * a.Rp + r]);
    const float ratio = __fdiv_rn(__fdiv_rn(s, float(a.N)), a.rho_th);
    D = __fmul_rn(D, fmaxf(0.0f, __fsub_rn(1.0f, ratio)));
  }
  return __fmul_rn(__fmul_rn(__fsqrt_rn(a.dt), D), a.cplx ? 0.70710678118654752f : 1.0f);
}

// Right-hand side of Eqs. (2) and (5) for one restart at one spin:
// k = x (gamma_s - |x|^2) + beta_s y + h,  k_gamma = eps (rho_th - |x|^2).
__device__ __forceinline__ void gd_rhs(float xr, float xi, float gs, float yr, float yi, float bs, float h, float eps,
                                       float rho_th, float& kr, float& ki, float& kg) {
  const float rho = density(xr, xi);
  const float t = __fsub_rn(gs, rho);
  kr = __fmaf_rn(xr, t, __fmaf_rn(bs, yr, h));
  ki = __fmaf_rn(xi, t, __fmul_rn(bs, yi));
  kg = __fmul_rn(eps, __fsub_rn(rho_th, rho));
}

// Resonant q:1 drive of Eq. (2) for complex amplitudes: (kr, ki) += h_q conj(x)^(q-1).
__device__ __forceinline__ void resonant_drive(float xr, float xi, int q, float hq, float& kr, float& ki) {
  float pr = 1.0f, pi = 0.0f;
  for (int k = 1; k < q; ++k) {  // p <- p conj(x)
    const float nr = __fmaf_rn(pr, xr, __fmul_rn(pi, xi));
    const float ni = __fmaf_rn(pi, xr, -__fmul_rn(pr, xi));
    pr = nr;
    pi = ni;
  }
  kr = __fmaf_rn(hq, pr, kr);
  ki = __fmaf_rn(hq, pi, ki);
}

// y + a x with one rounding.
__device__ __forceinline__ float axpy(float a, float x, float y) { return __fmaf_rn(a, x, y); }

}  // namespace gda
