// FP32 GD steps over a dense J0 on CUDA cores: the plain FP32 path the
// tensor-core path is measured against, and the path whose amplitudes are
// compared with the FP64 oracle.  Two forms, same bits: every coupling sum is
// one FMA chain in ascending j, the update is the shared FP32 expression
// sequence, and density sums have one order.
//
//  * k_dense_step: one launch per step or RK4 stage, a tiled product
//    Y = J0 X over 64 x BN tiles of (spins i) x (columns c) fused with the
//    step epilogue (Eqs. 2, 5, 6).
//  * k_dense_seg: small N; one launch runs a whole tracking segment.
#include "epilogue.cuh"
#include "tc_epilogue.cuh"
#include "tc_ptx.cuh"

namespace gda {
namespace {

constexpr int BM = 64, BK = 32;
constexpr int LD = BK + 4;  // floats per staged row: 16-byte reads of 8 consecutive rows miss no bank
constexpr int STAGES = 3;

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ptx::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Thread (tx, ty) of 16 x TY computes rows tx + 16 q (q < 4) and columns
// CPT ty .. CPT ty + CPT - 1.  Both operands are staged as they lie in memory
// (K contiguous) by a 3-stage cp.async ring and read four K at a time: 3
// shared-memory loads per 32 FMAs at CPT = 8, so the FMA pipe bounds a full
// chip.  (The tile this replaced, 4 x 4 per thread with a transposing
// register-staged copy and no overlap, spent 5 loads per 16 FMAs and ~600
// cycles of exposed latency per 16 K.)
template <int TY, int CPT>
struct DenseCfg {
  static constexpr int BN = TY * CPT;
  static constexpr int THREADS = 16 * TY;
  // column groups of different ty are 4 floats apart modulo 32 banks
  static constexpr int B_FLOATS = BN * LD + TY * 4;
  static constexpr int STAGE_FLOATS = BM * LD + B_FLOATS;
  static constexpr size_t SMEM = size_t(STAGES) * STAGE_FLOATS * sizeof(float);
};

template <bool CPLX, int MODE, int TY, int CPT>
__global__ void __launch_bounds__(16 * TY, ModeTraits<MODE>::rk_mid ? 2 : (CPT == 8 ? 3 : 4))
    k_dense_step(StepArgs a, const float* __restrict__ J, const float* __restrict__ X) {
  using Cfg = DenseCfg<TY, CPT>;
  constexpr int BN = Cfg::BN, NT = Cfg::THREADS;
  extern __shared__ __align__(16) float sm[];
  __shared__ float s_beta[BN], s_dsc[BN];
  __shared__ int s_bad;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int Np = a.Np;
  constexpr int RPT = CPLX ? BN / 2 : BN;  // restarts per tile
  const int rbase = CPLX ? n0 / 2 : n0;

  const int KB = (a.N + BK - 1) / BK;  // Np is a multiple of 128: whole K blocks lie inside the padded rows
  auto stage = [&](int kb) {
    float* As = sm + (kb % STAGES) * Cfg::STAGE_FLOATS;
    float* Bs = As + BM * LD;
    for (int q = tid; q < BM * 8; q += NT)
      cp_async16(As + (q >> 3) * LD + (q & 7) * 4, J + size_t(m0 + (q >> 3)) * Np + kb * BK + (q & 7) * 4);
    for (int q = tid; q < BN * 8; q += NT) {
      const int c = q >> 3;
      cp_async16(Bs + c * LD + (c / CPT) * 4 + (q & 7) * 4, X + size_t(n0 + c) * Np + kb * BK + (q & 7) * 4);
    }
  };
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < KB) stage(s);
    cp_async_commit();
  }
  if (tid == 0) s_bad = 0;
  if (tid < RPT) {
    const int r = rbase + tid;
    const float b = r < a.R ? a.beta_in[r] : 1.0f;
    s_beta[tid] = stage_beta(a, b);
    s_dsc[tid] = r < a.R ? noise_scale(a, r) : 0.0f;
  }
  float acc[4][CPT] = {};
  for (int kb = 0; kb < KB; ++kb) {
    cp_async_wait<STAGES - 2>();
    __syncthreads();  // stage kb is in, and everyone is done with the stage refilled next
    if (kb + STAGES - 1 < KB) stage(kb + STAGES - 1);
    cp_async_commit();
    const float* As = sm + (kb % STAGES) * Cfg::STAGE_FLOATS + tx * LD;
    const float* Bs = sm + (kb % STAGES) * Cfg::STAGE_FLOATS + BM * LD + ty * (CPT * LD + 4);
#pragma unroll
    for (int k = 0; k < BK; k += 4) {
      float av[4][4], bv[CPT][4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4*>(av[q]) = *reinterpret_cast<const float4*>(As + 16 * q * LD + k);
#pragma unroll
      for (int v = 0; v < CPT; ++v)
        *reinterpret_cast<float4*>(bv[v]) = *reinterpret_cast<const float4*>(Bs + v * LD + k);
#pragma unroll
      for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int v = 0; v < CPT; ++v) acc[q][v] = __fmaf_rn(av[q][e], bv[v][e], acc[q][v]);
    }
  }
  __syncthreads();  // s_beta / s_dsc of a K loop without a block

  // Epilogue: rows m0 + tx + 16 q, a quad of columns at a time; every input of
  // a quad is loaded before its first store.
  constexpr int U = CPLX ? 2 : 4;
  float* out = (MODE == M_ENERGY) ? a.e_part : (step_completes(MODE) ? a.rho_out : nullptr);
  int bad = 0;
#pragma unroll
  for (int g = 0; g < CPT / 4; ++g) {
    const int lc = CPT * ty + 4 * g, c0 = n0 + lc;
    const int lr0 = CPLX ? lc / 2 : lc;  // first local restart of the quad
    float rsum[4] = {0.f, 0.f, 0.f, 0.f};
    EpiRegs<MODE, CPLX, 4> E[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) epi_load<MODE, CPLX, 4>(a, m0 + tx + 16 * q, c0, E[q]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = m0 + tx + 16 * q;
      if (i >= a.N) continue;
      float red[4] = {0.f, 0.f, 0.f, 0.f};
      epi_chunk<MODE, CPLX, 4>(a, i, c0, &acc[q][4 * g], E[q], &s_beta[lr0], &s_dsc[lr0], red, bad);
#pragma unroll
      for (int u = 0; u < U; ++u) rsum[u] += red[u];
    }
    // sum over the 16 row groups (lanes with the same ty are one half-warp)
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int off = 8; off; off >>= 1) rsum[u] += __shfl_xor_sync(0xffffffffu, rsum[u], off);
      const int r = rbase + lr0 + u;
      if (tx == 0 && out && r < a.R) out[size_t(blockIdx.y) * a.Rp + r] = rsum[u];
    }
  }
  if (bad) atomicOr(&s_bad, 1);
  __syncthreads();
  if (tid == 0 && s_bad) atomicOr(a.err, E_DIVERGED);
  if (blockIdx.y == 0 && step_completes(MODE) && tid < RPT) {
    const int r = rbase + tid;
    if (r < a.R) a.beta_out[r] = next_beta(a, a.beta_in[r]);
  }
}

template <bool CPLX, int MODE, int TY, int CPT>
cudaError_t launch_dense_cfg(const StepArgs& a, const float* J32, const float* operand, cudaStream_t s) {
  using Cfg = DenseCfg<TY, CPT>;
  auto kern = k_dense_step<CPLX, MODE, TY, CPT>;
  if (Cfg::SMEM > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(Cfg::SMEM));
    if (e != cudaSuccess) return e;
  }
  const dim3 grid((a.C + Cfg::BN - 1) / Cfg::BN, simt_mtiles(a.N));
  kern<<<grid, Cfg::THREADS, Cfg::SMEM, s>>>(a, J32, operand);
  return cudaGetLastError();
}

// Tile width: the busiest SM's columns, rounds x BN, the widest on a tie
// (64 x 64 tiles reuse a staged operand most; narrow tiles spread a product
// of few columns over more SMs).
int dense_bn(const StepArgs& a, int sms) {
  int best = 64;
  long long cost = -1;
  for (int bn : {64, 32, 16}) {
    const long long tiles = (long long)((a.C + bn - 1) / bn) * simt_mtiles(a.N);
    const long long c = (tiles + sms - 1) / sms * bn;
    if (cost < 0 || c < cost) {
      cost = c;
      best = bn;
    }
  }
  return best;
}

template <bool CPLX, int MODE>
cudaError_t launch_dense_mode(const StepArgs& a, const float* J32, const float* operand, int sms, cudaStream_t s) {
  switch (dense_bn(a, sms)) {
    case 64: return launch_dense_cfg<CPLX, MODE, 8, 8>(a, J32, operand, s);
    case 32: return launch_dense_cfg<CPLX, MODE, 8, 4>(a, J32, operand, s);
    default: return launch_dense_cfg<CPLX, MODE, 4, 4>(a, J32, operand, s);
  }
}

template <bool CPLX>
cudaError_t launch_dense(const StepArgs& a, const float* J32, const float* operand, int sms, cudaStream_t s) {
  switch (a.mode) {
    case M_EULER: return launch_dense_mode<CPLX, M_EULER>(a, J32, operand, sms, s);
    case M_RK1: return launch_dense_mode<CPLX, M_RK1>(a, J32, operand, sms, s);
    case M_RK2: return launch_dense_mode<CPLX, M_RK2>(a, J32, operand, sms, s);
    case M_RK3: return launch_dense_mode<CPLX, M_RK3>(a, J32, operand, sms, s);
    case M_RK4: return launch_dense_mode<CPLX, M_RK4>(a, J32, operand, sms, s);
    case M_ENERGY: return launch_dense_mode<CPLX, M_ENERGY>(a, J32, operand, sms, s);
    case M_RAW: return launch_dense_mode<CPLX, M_RAW>(a, J32, operand, sms, s);
    default: return cudaErrorInvalidValue;
  }
}

// A segment of steps of a small instance in one launch.  A column of the
// state only reads itself and J0, so a CTA that holds J0 in shared memory and
// owns NC columns runs all steps (forward Euler, or RK4) without meeting
// another CTA.  One thread per spin: its amplitudes, gains and RK4 sums stay
// in registers, and the NC stage inputs of every spin alternate between two
// shared-memory buffers, one barrier per stage.  J0 is symmetric, so thread i
// reads column i of row j: consecutive threads, consecutive words.
//
// Bound by the FMA chain of a coupling sum (N dependent FMAs, one load of J0
// and one of X for NC of them) and the barrier.
template <bool CPLX, bool RK, int NC>
__global__ void __launch_bounds__(256) k_dense_seg(StepArgs a, const float* __restrict__ J, int steps) {
  constexpr int W = CPLX ? 2 : 1;
  constexpr int U = NC / W;  // restarts
  extern __shared__ __align__(16) float sm[];
  __shared__ float s_dsc[U], s_rho[4 * U];
  __shared__ int s_bad;
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int N = a.N, Np = a.Np;
  const int c0 = NC * int(blockIdx.x);  // < Cp (a multiple of 256)
  const int r0 = c0 / W;
  const bool decay = a.rho_out != nullptr;
  float* xs = sm;                          // [2][N][NC]
  float* sJ = xs + 2 * N * NC;             // [N][N]
  float* s_den = sJ + size_t(N) * N;       // [N][U], noise decay only
  for (int k = tid; k < N * N; k += nthr) sJ[k] = J[size_t(k / N) * Np + k % N];
  if (decay)
    for (int k = tid; k < a.mt_count * U; k += nthr)
      s_rho[k] = r0 + k % U < a.R ? a.rho_in[size_t(k / U) * a.Rp + r0 + k % U] : 0.0f;
  if (tid == 0) s_bad = 0;
  const int i = tid;
  const bool row = i < N;
  const float h = row ? a.h1[i] : 0.0f;
  float p[NC], gam[U], beta[U];
#pragma unroll
  for (int c = 0; c < NC; ++c) p[c] = row ? a.psi_n[size_t(c0 + c) * Np + i] : 0.0f;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    gam[u] = row && r0 + u < a.R ? a.gam[size_t(r0 + u) * Np + i] : 0.0f;
    beta[u] = r0 + u < a.R ? a.beta_in[r0 + u] : 1.0f;
  }
  auto put = [&](float* x, const float* v) {
    if (!row) return;
    if (NC == 4)
      *reinterpret_cast<float4*>(x + size_t(i) * NC) = *reinterpret_cast<const float4*>(v);
    else
      *reinterpret_cast<float2*>(x + size_t(i) * NC) = *reinterpret_cast<const float2*>(v);
  };
  auto coupling = [&](const float* x, float (&y)[NC]) {
#pragma unroll
    for (int c = 0; c < NC; ++c) y[c] = 0.0f;
    if (!row) return;
#pragma unroll 8
    for (int j = 0; j < N; ++j) {
      const float v = sJ[j * N + i];
      float xj[NC];
      if (NC == 4)
        *reinterpret_cast<float4*>(xj) = *reinterpret_cast<const float4*>(x + j * NC);
      else
        *reinterpret_cast<float2*>(xj) = *reinterpret_cast<const float2*>(x + j * NC);
#pragma unroll
      for (int c = 0; c < NC; ++c) y[c] = __fmaf_rn(v, xj[c], y[c]);
    }
  };
  put(xs, p);
  __syncthreads();

  int bad = 0, b = 0;
  StepArgs na = a;  // the scales' view: this CTA's density sums, the stage as mode
  na.rho_in = s_rho;
  na.Rp = U;
  for (int n = 0; n < steps; ++n) {
    na.mode = RK ? M_RK4 : M_EULER;
    float dsc[U];
    if (decay) {
      if (tid < U) s_dsc[tid] = r0 + tid < a.R ? noise_scale(na, tid) : 0.0f;
      __syncthreads();
    }
    bool noise = false;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      dsc[u] = decay ? s_dsc[u] : (r0 + u < a.R ? noise_scale(na, u) : 0.0f);
      noise |= dsc[u] != 0.0f;
    }
    float np[NC], ng[U];
    if (!RK) {
      float y[NC];
      coupling(xs + b * N * NC, y);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float xr = p[u * W], xi = CPLX ? p[u * W + 1] : 0.0f;
        float kr, ki, kg;
        gd_rhs(xr, xi, gam[u], y[u * W], CPLX ? y[u * W + 1] : 0.0f, beta[u], h, a.eps, a.rho_th, kr, ki, kg);
        if (CPLX && a.q) resonant_drive(xr, xi, a.q, a.hq, kr, ki);
        np[u * W] = axpy(a.dt, kr, xr);
        if (CPLX) np[u * W + 1] = axpy(a.dt, ki, xi);
        ng[u] = axpy(a.dt, kg, gam[u]);
      }
    } else {
      float x[NC], gs[U], acc[NC], gacc[U];
#pragma unroll
      for (int c = 0; c < NC; ++c) x[c] = p[c];
#pragma unroll
      for (int u = 0; u < U; ++u) gs[u] = gam[u];
#pragma unroll
      for (int st = 0; st < 4; ++st) {
        na.mode = M_RK1 + st;
        float y[NC];
        coupling(xs + b * N * NC, y);
        const float cf = st == 2 ? a.dt : __fmul_rn(0.5f, a.dt);
        const float d6 = __fdiv_rn(a.dt, 6.0f);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int k0 = u * W;
          const float xr = x[k0], xi = CPLX ? x[k0 + 1] : 0.0f;
          float kr, ki, kg;
          gd_rhs(xr, xi, gs[u], y[k0], CPLX ? y[k0 + 1] : 0.0f, stage_beta(na, beta[u]), h, a.eps, a.rho_th, kr, ki,
                 kg);
          if (CPLX && a.q) resonant_drive(xr, xi, a.q, a.hq, kr, ki);
          if (st == 3) {
            np[k0] = axpy(d6, __fadd_rn(acc[k0], kr), p[k0]);
            if (CPLX) np[k0 + 1] = axpy(d6, __fadd_rn(acc[k0 + 1], ki), p[k0 + 1]);
            ng[u] = axpy(d6, __fadd_rn(gacc[u], kg), gam[u]);
          } else {
            acc[k0] = st == 0 ? kr : axpy(2.0f, kr, acc[k0]);
            if (CPLX) acc[k0 + 1] = st == 0 ? ki : axpy(2.0f, ki, acc[k0 + 1]);
            gacc[u] = st == 0 ? kg : axpy(2.0f, kg, gacc[u]);
            x[k0] = axpy(cf, kr, p[k0]);
            if (CPLX) x[k0 + 1] = axpy(cf, ki, p[k0 + 1]);
            gs[u] = axpy(cf, kg, gam[u]);
          }
        }
        if (st < 3) {
          b ^= 1;
          put(xs + b * N * NC, x);
          __syncthreads();
        }
      }
    }
    float z[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (noise) {
      philox_normal4(uint32_t(i), uint32_t(c0 >> 2), a.step + unsigned(n), 0u, a.seed, z);
      if (NC == 2 && (c0 & 2)) {  // the quad's second pair of columns
        z[0] = z[2];
        z[1] = z[3];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      p[u * W] = axpy(dsc[u], z[u * W], np[u * W]);
      if (CPLX) p[u * W + 1] = axpy(dsc[u], z[u * W + 1], np[u * W + 1]);
      gam[u] = ng[u];
      const float rn = density(p[u * W], CPLX ? p[u * W + 1] : 0.0f);
      bad |= row && r0 + u < a.R && !(rn < 1e30f);
      if (decay && row) s_den[i * U + u] = rn;
    }
    na.mode = RK ? M_RK4 : M_EULER;
#pragma unroll
    for (int u = 0; u < U; ++u) beta[u] = next_beta(na, beta[u]);
    b ^= 1;
    put(xs + b * N * NC, p);
    __syncthreads();
    if (decay) {  // density sums of the per-step kernel's 64-row tiles, in its order
      const unsigned half = (tid & 16) ? 0xffff0000u : 0x0000ffffu;
      for (int k = tid >> 4; k < a.mt_count * U; k += nthr >> 4) {
        const int t = k / U, u = k % U, tx = tid & 15;
        float v = 0.0f;
        for (int q = 0; q < 4; ++q) {
          const int j = t * 64 + tx + 16 * q;
          if (j < N) v += s_den[j * U + u];
        }
#pragma unroll
        for (int off = 8; off; off >>= 1) v += __shfl_xor_sync(half, v, off);
        if (tx == 0) s_rho[k] = v;
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c)
    if (row && c0 + c < a.C) a.psi_out[size_t(c0 + c) * Np + i] = p[c];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (row && r0 + u < a.R) a.gam[size_t(r0 + u) * Np + i] = gam[u];
    if (tid == u && r0 + u < a.R) a.beta_out[r0 + u] = beta[u];
  }
  if (decay)
    for (int k = tid; k < a.mt_count * U; k += nthr)
      if (r0 + k % U < a.R) a.rho_out[size_t(k / U) * a.Rp + r0 + k % U] = s_rho[k];
  if (bad) atomicOr(&s_bad, 1);
  __syncthreads();
  if (tid == 0 && s_bad) atomicOr(a.err, E_DIVERGED);
}

constexpr size_t kDenseSegSmemMax = 224 * 1024;

size_t dense_seg_smem(const StepArgs& a, int nc) {
  const size_t n = a.N;
  return (2 * n * nc + n * n + (a.rho_out ? n * (a.cplx ? nc / 2 : nc) : 0)) * sizeof(float);
}

template <bool CPLX, bool RK, int NC>
cudaError_t launch_dense_seg_cfg(const StepArgs& a, const float* J32, int steps, cudaStream_t s) {
  auto kern = k_dense_seg<CPLX, RK, NC>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kDenseSegSmemMax));
  if (e != cudaSuccess) return e;
  kern<<<(a.C + NC - 1) / NC, (a.N + 31) / 32 * 32, dense_seg_smem(a, NC), s>>>(a, J32, steps);
  return cudaGetLastError();
}

}  // namespace

int simt_mtiles(int N) { return (N + BM - 1) / BM; }

cudaError_t launch_step_dense(const StepArgs& a, const float* J32, const float* operand, int sms, cudaStream_t s) {
  return a.cplx ? launch_dense<true>(a, J32, operand, sms, s) : launch_dense<false>(a, J32, operand, sms, s);
}

// Columns per CTA of a segment launch, 0 where a launch per step is better:
// J0 must fit in shared memory (N <= ~235), and the busiest SM's coupling
// sums (rounds x warps x N x (NC FMAs + 2 loads) / 4 issue slots) stay below
// ~16 000 cycles a stage, about what a per-step launch takes at these sizes.
int dense_seg_columns(const StepArgs& a, int sms) {
  if (a.N > 256 || dense_seg_smem(a, 4) > kDenseSegSmemMax) return 0;
  auto rounds = [&](int nc) { return ((a.C + nc - 1) / nc + sms - 1) / sms; };
  const int nc = rounds(4) < rounds(2) ? 4 : 2;
  const long long cycles = (long long)rounds(nc) * ((a.N + 31) / 32) * a.N * (nc + 2) / 4;
  return cycles <= 16000 ? nc : 0;
}

cudaError_t launch_dense_seg(const StepArgs& a, const float* J32, bool rk4, int steps, int columns, cudaStream_t s) {
  if (columns == 4) {
    if (a.cplx) return rk4 ? launch_dense_seg_cfg<true, true, 4>(a, J32, steps, s)
                           : launch_dense_seg_cfg<true, false, 4>(a, J32, steps, s);
    return rk4 ? launch_dense_seg_cfg<false, true, 4>(a, J32, steps, s)
               : launch_dense_seg_cfg<false, false, 4>(a, J32, steps, s);
  }
  if (a.cplx) return rk4 ? launch_dense_seg_cfg<true, true, 2>(a, J32, steps, s)
                         : launch_dense_seg_cfg<true, false, 2>(a, J32, steps, s);
  return rk4 ? launch_dense_seg_cfg<false, true, 2>(a, J32, steps, s)
             : launch_dense_seg_cfg<false, false, 2>(a, J32, steps, s);
}

}  // namespace gda
