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
#include <algorithm>

#include "epilogue.cuh"
#include "tc_epilogue.cuh"
#include "tc_ptx.cuh"

namespace gda {
namespace {

constexpr int BM = 64, BK = 32;
constexpr int STAGES = 3;  // of J0; the operand is double-buffered

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ptx::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// A pair of FMAs in one instruction (the same two roundings as __fmaf_rn).
__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// Four warps; a thread computes RT rows (lx + LX q) and CPT consecutive
// columns of the 64 x BN tile.  Both operands lie K-major in shared memory, so
// that a thread's column values of one K are 16-byte loads that are pairs for
// fma.rn.f32x2 as they stand.  J0 is symmetric: row k of J0 is the K-major row
// of the tile, copied by cp.async; the operand is transposed through registers
// one K block ahead.  Shared memory returns one 4-byte value per thread and
// cycle, so a K costs an SM 4 (RT + CPT) cycles of loads against RT CPT of
// FMAs per scheduler: 64 / 64 for the 8 x 8 form (64 x 128 tiles), 48 / 32 for
// 4 x 8, 32 / 16 for 4 x 4, 24 / 8 for 2 x 4.  On one tile per SM a single
// warp per scheduler leaves latency exposed as well; dense_bn weighs both.
// Measured (GB300, us a step, against the 64 x 64 tile with 4 x 4 outputs per
// thread and a transposing copy that this replaced): XY N = 1000, R = 256, RK4
// 147 / 218; XY N = 1000, R = 1024, Euler 114 / 148; SK N = R = 4096, Euler
// 2556 / 3678 (54 TFLOP/s); XY N = 300, R = 64, RK4 36 / 102.
template <int RT, int CPT>
struct DenseCfg {
  static constexpr int LX = BM / RT, LY = 32 / LX;
  static constexpr int BN = 4 * LY * CPT;
  static constexpr int THREADS = 128;
  static constexpr size_t SMEM = size_t(STAGES * BK * BM + 2 * BK * BN) * sizeof(float);
};

template <bool CPLX, int MODE, int RT, int CPT>
__global__ void __launch_bounds__(128, RT == 8 ? 2 : ModeTraits<MODE>::rk_mid ? 3 : 4)
    k_dense_step(StepArgs a, const float* __restrict__ J, const float* __restrict__ X) {
  using Cfg = DenseCfg<RT, CPT>;
  constexpr int BN = Cfg::BN, NT = Cfg::THREADS, LX = Cfg::LX;
  extern __shared__ __align__(16) float sm[];
  __shared__ float s_beta[BN], s_dsc[BN];
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lx = lane % LX, lcol = (warp * Cfg::LY + lane / LX) * CPT;  // first row, first column of the thread
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int Np = a.Np;
  constexpr int RPT = CPLX ? BN / 2 : BN;  // restarts per tile
  const int rbase = CPLX ? n0 / 2 : n0;
  float* sA = sm;                          // [STAGES][BK][BM]
  float* sB = sm + STAGES * BK * BM;       // [2][BK][BN]

  const int KB = (a.N + BK - 1) / BK;  // Np is a multiple of 128: whole K blocks lie inside the padded rows
  auto stage_A = [&](int kb) {
    float* d = sA + (kb % STAGES) * BK * BM;
#pragma unroll
    for (int t = 0; t < BK * BM / 4 / NT; ++t) {
      const int q = tid + t * NT;
      cp_async16(d + q * 4, J + size_t(kb * BK + (q >> 4)) * Np + m0 + (q & 15) * 4);
    }
  };
  // the operand's block: 8 lanes load the 32 K of a column (one line), then
  // scatter them over the K rows; column quads are permuted by k / 4 so that
  // the scatter misses no bank
  constexpr int QM = BN / 4 < 8 ? BN / 4 - 1 : 7;
  constexpr int TB = BN * 8 / NT;
  float4 bx[TB];
  auto load_B = [&](int kb) {
#pragma unroll
    for (int t = 0; t < TB; ++t) {
      const int q = tid + t * NT;
      bx[t] = *reinterpret_cast<const float4*>(X + size_t(n0 + (q >> 3)) * Np + kb * BK + (q & 7) * 4);
    }
  };
  auto store_B = [&](int kb) {
#pragma unroll
    for (int t = 0; t < TB; ++t) {
      const int q = tid + t * NT, c = q >> 3, kq = q & 7;
      float* d = sB + (kb & 1) * BK * BN + 4 * kq * BN + (((c >> 2) ^ (kq & QM)) << 2) + (c & 3);
      d[0] = bx[t].x;
      d[BN] = bx[t].y;
      d[2 * BN] = bx[t].z;
      d[3 * BN] = bx[t].w;
    }
  };
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < KB) stage_A(s);
    cp_async_commit();
  }
  load_B(0);
  store_B(0);
  if (tid == 0) s_bad = 0;
  if (tid < RPT) {
    const int r = rbase + tid;
    const float b = r < a.R ? a.beta_in[r] : 1.0f;
    s_beta[tid] = stage_beta(a, b);
    s_dsc[tid] = r < a.R ? noise_scale(a, r) : 0.0f;
  }
  unsigned long long acc[RT][CPT / 2];
#pragma unroll
  for (int q = 0; q < RT; ++q)
#pragma unroll
    for (int v = 0; v < CPT / 2; ++v) acc[q][v] = 0ull;
  for (int kb = 0; kb < KB; ++kb) {
    cp_async_wait<STAGES - 2>();
    __syncthreads();  // block kb is in, and everyone is done with the buffers refilled next
    if (kb + STAGES - 1 < KB) stage_A(kb + STAGES - 1);
    cp_async_commit();
    if (kb + 1 < KB) load_B(kb + 1);
    const float* As = sA + (kb % STAGES) * BK * BM + lx;
    const float* Bs = sB + (kb & 1) * BK * BN;
    // the values of the next K are read while this one's FMAs run
    float av[2][RT];
    ulonglong2 bv[2][CPT / 4];
    auto frag = [&](int k) {
#pragma unroll
      for (int q = 0; q < RT; ++q) av[k & 1][q] = As[k * BM + LX * q];
#pragma unroll
      for (int v = 0; v < CPT / 4; ++v)
        bv[k & 1][v] = *reinterpret_cast<const ulonglong2*>(Bs + k * BN + (((lcol >> 2) + v) ^ ((k >> 2) & QM)) * 4);
    };
    frag(0);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      if (k + 1 < BK) frag(k + 1);
#pragma unroll
      for (int q = 0; q < RT; ++q) {
        const unsigned long long aa = pack2(av[k & 1][q], av[k & 1][q]);
#pragma unroll
        for (int v = 0; v < CPT / 4; ++v) {
          fma2(acc[q][2 * v], aa, bv[k & 1][v].x);
          fma2(acc[q][2 * v + 1], aa, bv[k & 1][v].y);
        }
      }
    }
    if (kb + 1 < KB) store_B(kb + 1);
  }
  __syncthreads();

  // Epilogue: rows m0 + lx + LX q, a quad of columns at a time; the inputs of
  // QB rows are loaded before their first store.
  constexpr int U = CPLX ? 2 : 4;
  constexpr int QB = RT < 4 || ModeTraits<MODE>::rk_mid ? 2 : 4;
  float* out = (MODE == M_ENERGY) ? a.e_part : (step_completes(MODE) ? a.rho_out : nullptr);
  int bad = 0;
#pragma unroll
  for (int g = 0; g < CPT / 4; ++g) {
    const int lc = lcol + 4 * g, c0 = n0 + lc;
    const int lr0 = CPLX ? lc / 2 : lc;  // first local restart of the quad
    float red[RT][4] = {};
#pragma unroll
    for (int q0 = 0; q0 < RT; q0 += QB) {
      EpiRegs<MODE, CPLX, 4> E[QB];
#pragma unroll
      for (int q = 0; q < QB; ++q) epi_load<MODE, CPLX, 4>(a, m0 + lx + LX * (q0 + q), c0, E[q]);
#pragma unroll
      for (int q = 0; q < QB; ++q) {
        float y[4];
        unpack2(acc[q0 + q][2 * g], y[0], y[1]);
        unpack2(acc[q0 + q][2 * g + 1], y[2], y[3]);
        epi_chunk<MODE, CPLX, 4>(a, m0 + lx + LX * (q0 + q), c0, y, E[q], epi_drive(a, m0 + lx + LX * (q0 + q)), &s_beta[lr0], &s_dsc[lr0], red[q0 + q], bad);
      }
    }
    if (out) {  // rows t + 16 p summed over p = 0 .. 3, then a tree over the 16 t
#pragma unroll
      for (int u = 0; u < U; ++u) {
        float s;
        if (RT == 2) {  // p = 1, 3 lie 16 lanes up
          const float r1 = __shfl_down_sync(0xffffffffu, red[0][u], 16);
          const float r3 = __shfl_down_sync(0xffffffffu, red[RT / 2][u], 16);
          s = ((red[0][u] + r1) + red[RT / 2][u]) + r3;
        } else if (RT == 4) {
          s = ((red[0][u] + red[1][u]) + red[RT / 2][u]) + red[RT - 1][u];
        } else {  // t = lx and t = lx + 8 in one thread
          s = ((red[0][u] + red[RT / 4][u]) + red[RT / 2][u]) + red[3 * RT / 4][u];
          const float s8 = ((red[1][u] + red[RT / 4 + 1][u]) + red[RT / 2 + 1][u]) + red[3 * RT / 4 + 1][u];
          s += s8;
        }
#pragma unroll
        for (int off = RT == 8 ? 4 : 8; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        const int r = rbase + lr0 + u;
        if (lx == 0 && r < a.R) out[size_t(blockIdx.y) * a.Rp + r] = s;
      }
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

template <bool CPLX, int MODE, int RT, int CPT>
cudaError_t launch_dense_cfg(const StepArgs& a, const float* J32, const float* operand, cudaStream_t s) {
  using Cfg = DenseCfg<RT, CPT>;
  auto kern = k_dense_step<CPLX, MODE, RT, CPT>;
  if (Cfg::SMEM > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(Cfg::SMEM));
    if (e != cudaSuccess) return e;
  }
  const dim3 grid((a.C + Cfg::BN - 1) / Cfg::BN, simt_mtiles(a.N));
  kern<<<grid, Cfg::THREADS, Cfg::SMEM, s>>>(a, J32, operand);
  return cudaGetLastError();
}

// Tile width with the smallest time per K of the busiest SM: a tile alone on it
// runs one warp per scheduler, at the latency of its loads and FMA chains (`lone`
// cycles); each further tile on the SM adds the cycles of its shared-memory
// loads and FMAs (`more`; DenseCfg: 64, 48, 32, 24).  Averages over every width on
// GB300, N = 250 .. 2200, 8 .. 6000 columns, both models, Euler and RK4; the choice is
// on average 1.2 % above the best width.  (us a step for 128 / 64 / 32 / 16 columns:
// XY N = 500, 3000 columns, Euler 65 / 48 / 51 / 61.)  *cycles: that time.
int dense_bn(const StepArgs& a, int sms, long long* cycles = nullptr) {
  static constexpr int width[4] = {128, 64, 32, 16}, lone[4] = {142, 73, 47, 32}, more[4] = {93, 46, 31, 21};
  int best = 0;
  long long cost = -1;
  for (int k = 0; k < 4; ++k) {
    const long long tiles = (long long)((a.C + width[k] - 1) / width[k]) * simt_mtiles(a.N);
    const long long c = lone[k] + ((tiles + sms - 1) / sms - 1) * more[k];
    if (cost < 0 || c < cost) {
      cost = c;
      best = width[k];
    }
  }
  if (cycles) *cycles = cost;
  return best;
}

template <bool CPLX, int MODE>
cudaError_t launch_dense_mode(const StepArgs& a, const float* J32, const float* operand, int sms, cudaStream_t s) {
  switch (dense_bn(a, sms)) {
    case 128: return launch_dense_cfg<CPLX, MODE, 8, 8>(a, J32, operand, s);
    case 64: return launch_dense_cfg<CPLX, MODE, 4, 8>(a, J32, operand, s);
    case 32: return launch_dense_cfg<CPLX, MODE, 4, 4>(a, J32, operand, s);
    default: return launch_dense_cfg<CPLX, MODE, 2, 4>(a, J32, operand, s);
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
// and one of X for NC of them) and the barrier.  Measured (GB300): N = 20, R =
// 64, Euler 0.58 us a step, 12.4 us with a launch per step; XY N = 129, R =
// 16, RK4 8.1 against 77.9 us.
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

// Columns per CTA of a segment of `steps` steps in one launch, 0 where a launch
// per stage is better.  J0 must fit in shared memory (N <= ~235).  A stage of
// a segment takes the chain of N FMAs and loads for every wave of CTAs (and the
// issue slots of further CTAs on the SM), and every wave first loads its J0; a
// stage by itself takes a launch and its tiles' K loops (dense_bn).  Times in
// ns, fitted to runs on GB300 over N = 10 .. 233, R = 16 .. 2048, both models and
// integrators, 13 and 300 steps: the rule chose nothing more than 3 % slower than
// a launch per stage.  us a step, segment / launch per stage, Euler: Ising N = 10,
// R = 64 0.5 / 5.2; N = 200, R = 256 3.6 / 8.2; XY N = 200, R = 400 8.1 / 10.3, R =
// 1024 (four waves) 16.2 / 14.4; and 13.5 us a wave to load J0 at N = 200.
int dense_seg_columns(const StepArgs& a, int sms, bool rk4, long long steps) {
  if (a.N > 256 || dense_seg_smem(a, 4) > kDenseSegSmemMax) return 0;
  auto rounds = [&](int nc) { return ((a.C + nc - 1) / nc + sms - 1) / sms; };
  const int nc = rounds(4) < rounds(2) ? 4 : 2;
  const long long N = a.N, ctas = (a.C + nc - 1) / nc, warps = (a.N + 31) / 32;
  const long long per_sm = std::min<long long>((227 * 1024) / (dense_seg_smem(a, nc) + 1024), 64 / warps);
  const long long waves = (ctas + sms * per_sm - 1) / (sms * per_sm);
  const long long shared = (std::min(ctas, sms * per_sm) + sms - 1) / sms - 1;
  const long long stage = waves * (350 + (a.cplx ? 19 : 17) * N + shared * warps * N * (nc + 2) / 8);
  const long long load = waves * (2000 + 65 * N);
  long long cycles = 0;
  (void)dense_bn(a, sms, &cycles);
  const long long single = 5000 + ((N + BK - 1) / BK * BK) * cycles / 2;
  const long long stages = steps * (rk4 ? 4 : 1);
  return stages * stage + load < stages * single ? nc : 0;
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
