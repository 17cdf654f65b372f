// Register-staged epilogue of the step kernels.
//
// Each epilogue thread walks columns of a spin row i in chunks of CW.  All inputs a chunk needs (amplitudes, gains, RK4 accumulators) are
// loaded into registers one chunk ahead of the arithmetic, and the first chunk
// is loaded while the MMAs are still running, so global-memory latency is
// paid about once per kernel instead of once per element.
#pragma once
#include <cuda_fp8.h>

#include "epilogue.cuh"

namespace gda {

template <int MODE>
struct ModeTraits {
  static constexpr bool rk_mid = MODE == M_RK2 || MODE == M_RK3 || MODE == M_RK4;
  static constexpr bool has_x = MODE != M_RAW;
  static constexpr bool has_g = MODE != M_RAW && MODE != M_ENERGY;
  // chunks whose inputs are loaded into registers ahead of the one computed
  // (a second chunk in registers spills at the 96 registers of a 576-thread
  // block and measured slower)
  static constexpr int prefetch = 1;
  // chunks whose state lines are pulled into L2 ahead of their register
  // loads (no registers: the loads of a chunk then find their lines in L2)
  static constexpr int l2_ahead = MODE == M_RAW ? 0 : 3;
};

// Loads and stores of the FP32 state.  (An evict-first L2 policy on them
// measured slower: the lines the L2 prefetch brings in were dropped before
// their loads.)
static __device__ __forceinline__ float ld_state(const float* p) { return *p; }
static __device__ __forceinline__ void st_state(float* p, float v) { *p = v; }

template <int MODE, bool CPLX, int CW>
struct EpiRegs {
  static constexpr int W = CPLX ? 2 : 1;
  static constexpr int NR = CW / W;
  using T = ModeTraits<MODE>;
  float x[T::has_x ? CW : 1];
  float pn[T::rk_mid ? CW : 1];
  float ac[T::rk_mid ? CW : 1];
  float gs[T::has_g ? NR : 1];
  float gn[T::rk_mid ? NR : 1];
  float ga[T::rk_mid ? NR : 1];
};

// Loads the inputs of columns c0 .. c0+CW-1 at row i.  A chunk lies inside the
// padded buffers (Cp and Rp are multiples of 256) or wholly beyond them, where
// its first column and restart are clamped so that every address is valid
// whatever the tile width; values of columns beyond C are discarded by
// epi_chunk.
template <int MODE, bool CPLX, int CW>
__device__ __forceinline__ void epi_load(const StepArgs& a, int i, int c0, EpiRegs<MODE, CPLX, CW>& R) {
  using Tr = ModeTraits<MODE>;
  constexpr int W = CPLX ? 2 : 1;
  const size_t Np = a.Np;
  const size_t o = size_t(min(c0, a.Cp - CW)) * Np + i;
  const size_t og = size_t(min(CPLX ? c0 / 2 : c0, a.Rp - CW / W)) * Np + i;
  const float* const x = (MODE == M_ENERGY ? a.psi_n : a.xs) + o;
#pragma unroll
  for (int k = 0; k < CW; ++k)
    if (Tr::has_x) R.x[k] = ld_state(x + k * Np);
  if (Tr::rk_mid) {
    const float *const pn = a.psi_n + o, *const ac = a.acc + o;
#pragma unroll
    for (int k = 0; k < CW; ++k) {
      R.pn[k] = ld_state(pn + k * Np);
      R.ac[k] = ld_state(ac + k * Np);
    }
  }
  if (Tr::has_g) {
    const float* const gs = ((MODE == M_EULER || MODE == M_RK1) ? a.gam : a.gstg) + og;
#pragma unroll
    for (int u = 0; u < CW / W; ++u) R.gs[u] = ld_state(gs + u * Np);
  }
  if (Tr::rk_mid) {
    const float *const gn = a.gam + og, *const ga = a.gacc + og;
#pragma unroll
    for (int u = 0; u < CW / W; ++u) {
      R.gn[u] = ld_state(gn + u * Np);
      R.ga[u] = ld_state(ga + u * Np);
    }
  }
}

static __device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Pulls into L2 the state lines that epi_load of columns c0 .. c0+CW-1 will
// read for the warp's 32 rows (i - lane .. i - lane + 31: one 128-byte line per
// column): lanes 0 .. CW-1 take the amplitude columns, the next CW / W lanes
// the gain rows.  Addresses are clamped as in epi_load.
template <int MODE, bool CPLX, int CW>
__device__ __forceinline__ void epi_prefetch_l2(const StepArgs& a, int i, int c0, int lane) {
  using Tr = ModeTraits<MODE>;
  constexpr int W = CPLX ? 2 : 1;
  constexpr int NR = CW / W;
  if (MODE == M_RAW) return;
  const size_t Np = a.Np;
  const int ib = i - lane;
  if (lane < CW) {
    const size_t o = size_t(min(c0 + lane, a.Cp - 1)) * Np + ib;
    prefetch_l2((MODE == M_ENERGY ? a.psi_n : a.xs) + o);
    if (Tr::rk_mid) {
      prefetch_l2(a.psi_n + o);
      prefetch_l2(a.acc + o);
    }
  } else if (Tr::has_g && lane < CW + NR) {
    const int r0 = CPLX ? c0 / 2 : c0;
    const size_t og = size_t(min(r0 + lane - CW, a.Rp - 1)) * Np + ib;
    prefetch_l2(((MODE == M_EULER || MODE == M_RK1) ? a.gam : a.gstg) + og);
    if (Tr::rk_mid) {
      prefetch_l2(a.gam + og);
      prefetch_l2(a.gacc + og);
    }
  }
}

// The drive h_1i of row i (0 beyond N).
__device__ __forceinline__ float epi_drive(const StepArgs& a, int i) { return i < a.N ? a.h1[i] : 0.0f; }

// Arithmetic and stores of one chunk.  y: the CW accumulator values of row i;
// h: the row's drive (epi_drive).
// beta_s / dsc: per-restart stage scale and noise amplitude, indexed by the
// chunk's local restart.  red[u]: per-restart contribution (density of the
// new amplitude, or Eq. (1) partial energy).  nxt (NXT only): receives the
// chunk's next operand values (the new amplitudes, or the next RK stage
// input), 0 for restarts beyond R.
template <int MODE, bool CPLX, int CW, bool NXT = false>
__device__ __forceinline__ void epi_chunk(const StepArgs& a, int i, int c0, const float* y,
                                          const EpiRegs<MODE, CPLX, CW>& R, float h, const float* beta_s,
                                          const float* dsc, float* red, int& bad, float* nxt = nullptr) {
  constexpr int W = CPLX ? 2 : 1;
  constexpr int NR = CW / W;
  // the arguments as values: where they live in shared memory, every store
  // below could otherwise change them
  const size_t Np = a.Np;
  const int r0 = CPLX ? c0 / 2 : c0;
  const int drive = CPLX ? a.q : 0;
  const float dt = a.dt, eps = a.eps, rho_th = a.rho_th, hq = a.hq, op8_inv = a.op8_inv;
  const bool row_ok = i < a.N;
  const int live = row_ok ? a.R - r0 : 0;  // restarts u < live exist; the others' values go nowhere
  const size_t o0 = size_t(c0) * Np + i, og = size_t(r0) * Np + i, p0 = size_t(c0) * a.op_pitch + i;
  if (MODE == M_RAW) {
    float* const out = a.psi_out + o0;
#pragma unroll
    for (int u = 0; u < NR; ++u) {
      red[u] = 0.0f;
      if (u < live)
#pragma unroll
        for (int w = 0; w < W; ++w) out[(u * W + w) * Np] = y[u * W + w];
    }
    return;
  }
  if (MODE == M_ENERGY) {
    const float gi = row_ok ? a.g[i] : 0.0f;
#pragma unroll
    for (int u = 0; u < NR; ++u) {
      const int k0 = u * W;
      const float yr = y[k0], yi = CPLX ? y[k0 + 1] : 0.0f;
      const float pr = R.x[k0], pi = CPLX ? R.x[k0 + 1] : 0.0f;
      float sr, si = 0.0f;
      if (CPLX && drive >= 2) {  // Potts: the nearest q-th root, as the operand's projection
        double dr, di;
        potts_project(pr, pi, drive, dr, di);
        sr = float(dr);
        si = float(di);
      } else if (CPLX) {
        const float m = sqrtf(pr * pr + pi * pi);
        sr = m > 0.0f ? pr / m : 1.0f;
        si = m > 0.0f ? pi / m : 0.0f;
      } else {
        sr = pr >= 0.0f ? 1.0f : -1.0f;
      }
      red[u] = u < live ? -(sr * yr + si * yi) + gi * sr : 0.0f;
    }
    return;
  }
  constexpr bool COMPLETES = MODE == M_EULER || MODE == M_RK4;
  // RK stages hold more values per element: they take one restart at a time
  // and read its scales where they are used; Euler runs a chunk as straight code
  constexpr bool MID = ModeTraits<MODE>::rk_mid, ONE = MODE != M_EULER;
  float bs[ONE ? 1 : NR], ds[ONE ? 1 : NR], z[CW];
  if (!ONE)
#pragma unroll
    for (int u = 0; u < NR; ++u) bs[ONE ? 0 : u] = beta_s[u];
  const bool noisy = a.noise_D != 0.0f;
  if (COMPLETES) {
    bool any = false;
    if (!ONE)
#pragma unroll
      for (int u = 0; u < NR; ++u) ds[ONE ? 0 : u] = 0.0f;
    if (noisy) {
#pragma unroll
      for (int u = 0; u < NR; ++u) {
        if (!ONE) ds[ONE ? 0 : u] = dsc[u];
        any |= dsc[u] != 0.0f;
      }
    }
#pragma unroll
    for (int q = 0; q < CW / 4; ++q) {
      if (any) {
        philox_normal4(uint32_t(i), uint32_t((c0 >> 2) + q), a.step, 0u, a.seed, &z[4 * q]);
      } else {
        z[4 * q] = z[4 * q + 1] = z[4 * q + 2] = z[4 * q + 3] = 0.0f;
      }
    }
  }
  float* const xo = (COMPLETES ? a.psi_out : a.xs_next) + o0;
  float* const go = (COMPLETES ? a.gam : a.gstg) + og;
  float *const ao = COMPLETES ? nullptr : a.acc + o0, *const gao = COMPLETES ? nullptr : a.gacc + og;
  __nv_bfloat16* const op = a.op_out;
  unsigned char* const op8 = a.op8_out;
  const size_t pitch = a.op_pitch;
  unsigned top = 0;  // largest density as bits: finite and below 1e30 where it is small
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int k0 = u * W;
    if (ONE) {
      if (u >= live) {
        red[u] = 0.0f;
        if (NXT) nxt[k0] = nxt[k0 + W - 1] = 0.0f;
        continue;
      }
      bs[0] = beta_s[u];
      ds[0] = noisy ? dsc[u] : 0.0f;
    }
    const float yr = y[k0], yi = CPLX ? y[k0 + 1] : 0.0f;
    const float xr = R.x[k0], xi = CPLX ? R.x[k0 + 1] : 0.0f;
    const float gs = R.gs[u];
    float kr, ki, kg;
    gd_rhs(xr, xi, gs, yr, yi, bs[ONE ? 0 : u], h, eps, rho_th, kr, ki, kg);
    if (CPLX && drive) resonant_drive(xr, xi, drive, hq, kr, ki);
    float nr, ni, ng;  // the next operand values and gain
    if (MODE == M_EULER) {
      nr = axpy(dt, kr, xr);
      ni = axpy(dt, ki, xi);
      ng = axpy(dt, kg, gs);
    } else {
      const float pr = MID ? R.pn[MID ? k0 : 0] : xr;
      const float pi = CPLX ? (MID ? R.pn[MID ? k0 + W - 1 : 0] : xi) : 0.0f;
      const float gn = MID ? R.gn[MID ? u : 0] : gs;
      if (MODE == M_RK4) {
        const float d6 = __fdiv_rn(dt, 6.0f);
        nr = axpy(d6, __fadd_rn(R.ac[MID ? k0 : 0], kr), pr);
        ni = CPLX ? axpy(d6, __fadd_rn(R.ac[MID ? k0 + W - 1 : 0], ki), pi) : 0.0f;
        ng = axpy(d6, __fadd_rn(R.ga[MID ? u : 0], kg), gn);
      } else {
        const float cf = (MODE == M_RK3) ? dt : __fmul_rn(0.5f, dt);
        if (u < live) {
          st_state(ao + k0 * Np, MID ? axpy(2.0f, kr, R.ac[MID ? k0 : 0]) : kr);
          if (CPLX) st_state(ao + (k0 + 1) * Np, MID ? axpy(2.0f, ki, R.ac[MID ? k0 + W - 1 : 0]) : ki);
          st_state(gao + u * Np, MID ? axpy(2.0f, kg, R.ga[MID ? u : 0]) : kg);
        }
        nr = axpy(cf, kr, pr);
        ni = axpy(cf, ki, pi);
        ng = axpy(cf, kg, gn);
      }
    }
    if (COMPLETES) {
      nr = axpy(ds[ONE ? 0 : u], z[k0], nr);
      if (CPLX) ni = axpy(ds[ONE ? 0 : u], z[CPLX ? k0 + 1 : 0], ni);
      const float rn = CPLX ? density(nr, ni) : __fmul_rn(nr, nr);  // density(nr, 0)
      red[u] = u < live ? rn : 0.0f;
      top = max(top, u < live ? __float_as_uint(rn) & 0x7fffffffu : 0u);
    } else {
      red[u] = 0.0f;
    }
    if (NXT) {
      nxt[k0] = u < live ? nr : 0.0f;
      if (CPLX) nxt[k0 + W - 1] = u < live ? ni : 0.0f;
    }
    if (u < live) {
      st_state(xo + k0 * Np, nr);
      if (CPLX) st_state(xo + (k0 + 1) * Np, ni);
      st_state(go + u * Np, ng);
      if (op) {
        op[p0 + k0 * pitch] = __float2bfloat16_rn(nr);
        if (CPLX) op[p0 + (k0 + 1) * pitch] = __float2bfloat16_rn(ni);
      }
      if (op8) {
        op8[o0 + k0 * Np] = __nv_cvt_float_to_fp8(nr * op8_inv, __NV_SATFINITE, __NV_E4M3);
        if (CPLX) op8[o0 + (k0 + 1) * Np] = __nv_cvt_float_to_fp8(ni * op8_inv, __NV_SATFINITE, __NV_E4M3);
      }
    }
  }
  bad |= top >= __float_as_uint(1e30f);
}

}  // namespace gda
