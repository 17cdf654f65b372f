// Spin projection, Eq. (1) energies and the argmin over restarts.
//
//  * tracking: the projected spins are written as the operand of one more
//    coupling product (FP32 or BF16, the run's path) whose epilogue forms the
//    per-restart partial energies; k_track_reduce sums them, adds -sum_i J_ii
//    and records the best restart;
//  * final: FP64 energies of the full J with the projected spins (energy_tc.cu).
#include <cfloat>

#include "gda_internal.h"
#include "kernels.h"

namespace gda {


// ---------------------------------------------------------------- init
__global__ void k_init_state(float* psi, float* gam, float* beta, int N, int Np, int R, int cplx, int mode,
                             float amp, float gamma0, float beta0, unsigned long long seed, const float* base) {
  const size_t total = size_t(R) * N;
  for (size_t idx = blockIdx.x * size_t(blockDim.x) + threadIdx.x; idx < total; idx += size_t(gridDim.x) * blockDim.x) {
    const int r = int(idx / N), i = int(idx % N);
    float re = 0.0f, im = 0.0f;
    if (mode == 1 || mode == 3) {
      const U4 o = philox4x32_10(U4{uint32_t(i), uint32_t(r), 0u, 1u}, uint32_t(seed), uint32_t(seed >> 32));
      re = amp * (2.0f * philox_u01(o.x) - 1.0f);
      im = amp * (2.0f * philox_u01(o.y) - 1.0f);
      if (mode == 3) {  // per-spin base amplitude plus the seeded perturbation
        re = __fadd_rn(base[2 * i], re);
        im = __fadd_rn(base[2 * i + 1], im);
      }
    }
    if (cplx) {
      psi[size_t(2 * r) * Np + i] = re;
      psi[size_t(2 * r + 1) * Np + i] = im;
    } else {
      psi[size_t(r) * Np + i] = re;
    }
    gam[size_t(r) * Np + i] = gamma0;
    if (i == 0) beta[r] = beta0;
  }
}

__global__ void k_fill_h1(const double* g, float* h1, int N, float sq) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) h1[i] = float(-g[i]) * sq;
}

__global__ void k_to_bf16(const float* x, __nv_bfloat16* y, size_t n) {
  for (size_t k = blockIdx.x * size_t(blockDim.x) + threadIdx.x; k < n; k += size_t(gridDim.x) * blockDim.x)
    y[k] = __float2bfloat16_rn(x[k]);
}

// Partial sums of |psi|^2 over the spin tiles of one path, in the same order
// as that path's step epilogue, so a resumed run draws the same noise scale.
// TC order: rows of a 128-row tile reduced per 32-row quarter by an xor tree,
// quarters added in order.  SIMT order: rows tx + 16q summed over q, then an
// xor tree over the 16 tx.
__global__ void k_rho_partials_tc(const float* psi, int N, int Np, int R, int Rp, int cplx, float* out) {
  const int t = blockIdx.x, r = blockIdx.y;  // blockDim = 128
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ float part[4];
  const int i = t * 128 + 32 * q + lane;
  float x = 0.0f;
  if (i < N) {
    const float re = psi[size_t(cplx ? 2 * r : r) * Np + i];
    const float im = cplx ? psi[size_t(2 * r + 1) * Np + i] : 0.0f;
    x = density(re, im);
  }
  for (int off = 16; off; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  if (lane == 0) part[q] = x;
  __syncthreads();
  if (threadIdx.x == 0) out[size_t(t) * Rp + r] = part[0] + part[1] + part[2] + part[3];
}

__global__ void k_rho_partials_simt(const float* psi, int N, int Np, int R, int Rp, int cplx, float* out) {
  const int t = blockIdx.x, r = blockIdx.y;  // blockDim = 16
  const int tx = threadIdx.x;
  float s = 0.0f;
  for (int q = 0; q < 4; ++q) {
    const int i = t * 64 + tx + 16 * q;
    if (i >= N) continue;
    const float re = psi[size_t(cplx ? 2 * r : r) * Np + i];
    const float im = cplx ? psi[size_t(2 * r + 1) * Np + i] : 0.0f;
    s += density(re, im);
  }
  for (int off = 8; off; off >>= 1) s += __shfl_xor_sync(0x0000ffffu, s, off);
  if (tx == 0) out[size_t(t) * Rp + r] = s;
}

// ---------------------------------------------------------------- projection
template <typename T>
__device__ __forceinline__ T conv(float v);
template <>
__device__ __forceinline__ float conv<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 conv<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// Projected spins s of psi as a coupling-product operand [Cp][Np].
template <typename T>
__global__ void k_project_op(const float* psi, T* S, int N, int Np, int R, int cplx) {
  const size_t total = size_t(R) * N;
  for (size_t idx = blockIdx.x * size_t(blockDim.x) + threadIdx.x; idx < total; idx += size_t(gridDim.x) * blockDim.x) {
    const int r = int(idx / N), i = int(idx % N);
    if (cplx >= 2) {
      double sr, si;
      potts_project(psi[size_t(2 * r) * Np + i], psi[size_t(2 * r + 1) * Np + i], cplx, sr, si);
      S[size_t(2 * r) * Np + i] = conv<T>(float(sr));
      S[size_t(2 * r + 1) * Np + i] = conv<T>(float(si));
    } else if (cplx) {
      const float re = psi[size_t(2 * r) * Np + i], im = psi[size_t(2 * r + 1) * Np + i];
      const float m = sqrtf(re * re + im * im);
      S[size_t(2 * r) * Np + i] = conv<T>(m > 0.0f ? re / m : 1.0f);
      S[size_t(2 * r + 1) * Np + i] = conv<T>(m > 0.0f ? im / m : 0.0f);
    } else {
      S[size_t(r) * Np + i] = conv<T>(psi[size_t(r) * Np + i] >= 0.0f ? 1.0f : -1.0f);
    }
  }
}

// ---------------------------------------------------------------- tracking
// One block.  E_r = sum_t e_part[t][r] - sum_i J_ii; records (step, E, r) of
// the lowest E (ties: lowest r) at trace slot *count when it fits.
__global__ void k_track_reduce(const float* e_part, int mt, int R, int Rp, double diag, long long step,
                               long long* t_step, double* t_E, int* t_r, int cap, int* count, double* lastE,
                               int* lastR) {
  __shared__ double sE[32];
  __shared__ int sR[32];
  double best = DBL_MAX;
  int br = 0x7fffffff;
  for (int r = threadIdx.x; r < R; r += blockDim.x) {
    float s = 0.0f;
    for (int t = 0; t < mt; ++t) s += e_part[size_t(t) * Rp + r];
    const double E = double(s) + diag;
    if (E < best || (E == best && r < br)) { best = E; br = r; }
  }
  for (int off = 16; off; off >>= 1) {
    const double oE = __shfl_xor_sync(0xffffffffu, best, off);
    const int oR = __shfl_xor_sync(0xffffffffu, br, off);
    if (oE < best || (oE == best && oR < br)) { best = oE; br = oR; }
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { sE[w] = best; sR[w] = br; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < int(blockDim.x >> 5); ++k)
      if (sE[k] < best || (sE[k] == best && sR[k] < br)) { best = sE[k]; br = sR[k]; }
    const int c = *count;
    if (c < cap) { t_step[c] = step; t_E[c] = best; t_r[c] = br; }
    *count = c + 1;
    *lastE = best;
    *lastR = br;
  }
}

// ---------------------------------------------------------------- final energy
// Energies of real spins, g = 0 and a small instance of integer couplings whose
// sums all stay below 2^24: exact in FP32.  One CTA per restart, a warp per
// row of J.  A tile of the digit products costs a single small instance its
// fixed 19 us (prologue, pipeline, tile-wide sums); this kernel takes 8 for N =
// 100, R = 256 and reads N^2 doubles per restart from L2, so it is used up to
// 2^25 of them.
constexpr int ES_MAXN = 256, ES_WARPS = 16;

// An integer of at most 24 bits from double to float by its bits (the
// conversion instruction runs at the FP64 pipe's rate: 16 us instead of 8).
__device__ __forceinline__ float small_float(double v) {
  const unsigned hi = unsigned(__double2hiint(v)), lo = unsigned(__double2loint(v));
  if (!(hi & 0x7fffffffu)) return 0.0f;
  return __uint_as_float((hi & 0x80000000u) | (((hi & 0x7fffffffu) - (896u << 20)) << 3) | (lo >> 29));
}

__global__ void __launch_bounds__(32 * ES_WARPS) k_energy_small(const double* __restrict__ J,
                                                                const float* __restrict__ psi, int N, int Np,
                                                                double* __restrict__ E) {
  __shared__ float s[ES_MAXN], part[ES_WARPS];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < ES_MAXN) s[tid] = tid >= N ? 0.0f : psi[size_t(blockIdx.x) * Np + tid] >= 0.0f ? 1.0f : -1.0f;
  __syncthreads();
  float t = 0.0f;
#pragma unroll 2
  for (int i = warp; i < N; i += ES_WARPS) {
    float y = 0.0f;
#pragma unroll
    for (int k = 0; k < ES_MAXN / 32; ++k)
      if (k * 32 + lane < N) y = fmaf(small_float(J[size_t(i) * Np + k * 32 + lane]), s[k * 32 + lane], y);
    t = fmaf(s[i], y, t);
  }
  for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) part[warp] = t;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < ES_WARPS; ++w) t += part[w];
    E[blockIdx.x] = -double(t);
  }
}

// Lowest energy over restarts (ties: lowest index) -> best[0] = E, best_r.
__global__ void k_argmin(const double* E, int R, double* bestE, int* bestR) {
  __shared__ double sE[32];
  __shared__ int sR[32];
  double best = DBL_MAX;
  int br = 0x7fffffff;
  for (int r = threadIdx.x; r < R; r += blockDim.x) {
    const double e = E[r];
    if (e < best || (e == best && r < br)) { best = e; br = r; }
  }
  for (int off = 16; off; off >>= 1) {
    const double oE = __shfl_xor_sync(0xffffffffu, best, off);
    const int oR = __shfl_xor_sync(0xffffffffu, br, off);
    if (oE < best || (oE == best && oR < br)) { best = oE; br = oR; }
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { sE[w] = best; sR[w] = br; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < int(blockDim.x >> 5); ++k)
      if (sE[k] < best || (sE[k] == best && sR[k] < br)) { best = sE[k]; br = sR[k]; }
    *bestE = best;
    *bestR = br;
  }
}

// Configuration of the best restart: int8 spins (Ising) or theta (XY).
__global__ void k_best_cfg(const float* psi, const int* bestR, int N, int Np, int cplx, signed char* s8, double* th) {
  const int r = *bestR;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    if (cplx >= 2) {
      double sr, si;
      potts_project(psi[size_t(2 * r) * Np + i], psi[size_t(2 * r + 1) * Np + i], cplx, sr, si);
      th[i] = atan2(si, sr);
    } else if (cplx) {
      const double re = psi[size_t(2 * r) * Np + i], im = psi[size_t(2 * r + 1) * Np + i];
      th[i] = (re == 0.0 && im == 0.0) ? 0.0 : atan2(im, re);
    } else {
      s8[i] = psi[size_t(r) * Np + i] >= 0.0f ? 1 : -1;
    }
  }
}

// ---------------------------------------------------------------- launchers
static int grid_for(size_t n) {
  size_t b = (n + 255) / 256;
  return int(b > 4096 ? 4096 : (b ? b : 1));
}

cudaError_t launch_init_state(float* psi, float* gam, float* beta, int N, int Np, int R, int cplx, int mode,
                              float amp, float gamma0, float beta0, unsigned long long seed, const float* base,
                              cudaStream_t s) {
  k_init_state<<<grid_for(size_t(R) * N), 256, 0, s>>>(psi, gam, beta, N, Np, R, cplx, mode, amp, gamma0, beta0,
                                                        seed, base);
  return cudaGetLastError();
}

cudaError_t launch_fill_h1(const double* g, float* h1, int N, float sq, cudaStream_t s) {
  k_fill_h1<<<grid_for(N), 256, 0, s>>>(g, h1, N, sq);
  return cudaGetLastError();
}

cudaError_t launch_to_bf16(const float* x, __nv_bfloat16* y, size_t n, cudaStream_t s) {
  k_to_bf16<<<grid_for(n), 256, 0, s>>>(x, y, n);
  return cudaGetLastError();
}

cudaError_t launch_rho_partials(bool tc, const float* psi, int N, int Np, int R, int Rp, int cplx, float* out,
                                cudaStream_t s) {
  if (tc) {
    k_rho_partials_tc<<<dim3((N + 127) / 128, R), 128, 0, s>>>(psi, N, Np, R, Rp, cplx, out);
  } else {
    k_rho_partials_simt<<<dim3((N + 63) / 64, R), 16, 0, s>>>(psi, N, Np, R, Rp, cplx, out);
  }
  return cudaGetLastError();
}

cudaError_t launch_project_f32(const float* psi, float* S, int N, int Np, int R, int cplx, cudaStream_t s) {
  k_project_op<float><<<grid_for(size_t(R) * N), 256, 0, s>>>(psi, S, N, Np, R, cplx);
  return cudaGetLastError();
}

cudaError_t launch_project_bf16(const float* psi, __nv_bfloat16* S, int N, int Np, int R, int cplx, cudaStream_t s) {
  k_project_op<__nv_bfloat16><<<grid_for(size_t(R) * N), 256, 0, s>>>(psi, S, N, Np, R, cplx);
  return cudaGetLastError();
}

cudaError_t launch_track_reduce(const float* e_part, int mt, int R, int Rp, double diag, long long step,
                                long long* t_step, double* t_E, int* t_r, int cap, int* count, double* lastE,
                                int* lastR, cudaStream_t s) {
  k_track_reduce<<<1, 1024, 0, s>>>(e_part, mt, R, Rp, diag, step, t_step, t_E, t_r, cap, count, lastE, lastR);
  return cudaGetLastError();
}

namespace {

// Running best of the energy trace: when this evaluation's lowest tracking
// energy (*lastE, restart *lastR) is below the best so far, the restart's
// amplitudes (W columns of Np) are copied to snap and (E, r, step) recorded.
// Also keeps that restart's amplitudes in hist[entry] for the trace entry just
// recorded (entry = *count - 1) when entry < hist_cap.
__global__ void k_snapshot(const float* psi, int Np, int W, const double* lastE, const int* lastR, long long step,
                           double* snapE, int* snapR, long long* snapStep, float* snap, float* hist, int hist_cap,
                           const int* count) {
  __shared__ int take;
  if (threadIdx.x == 0) {
    take = *lastE < *snapE;
    if (take) {
      *snapE = *lastE;
      *snapR = *lastR;
      *snapStep = step;
    }
  }
  __syncthreads();
  const float* src = psi + size_t(*lastR) * W * Np;
  const int entry = *count - 1;
  if (hist && entry >= 0 && entry < hist_cap) {
    float* dst = hist + size_t(entry) * W * Np;
    for (int k = threadIdx.x; k < W * Np; k += blockDim.x) dst[k] = src[k];
  }
  if (!take) return;
  for (int k = threadIdx.x; k < W * Np; k += blockDim.x) snap[k] = src[k];
}

__global__ void k_snapshot_reset(double* snapE, int* snapR, long long* snapStep) {
  *snapE = DBL_MAX;
  *snapR = -1;
  *snapStep = -1;
}

}  // namespace

cudaError_t launch_snapshot(const float* psi, int Np, int W, const double* lastE, const int* lastR, long long step,
                            double* snapE, int* snapR, long long* snapStep, float* snap, float* hist, int hist_cap,
                            const int* count, cudaStream_t s) {
  k_snapshot<<<1, 1024, 0, s>>>(psi, Np, W, lastE, lastR, step, snapE, snapR, snapStep, snap, hist, hist_cap, count);
  return cudaGetLastError();
}

cudaError_t launch_snapshot_reset(double* snapE, int* snapR, long long* snapStep, cudaStream_t s) {
  k_snapshot_reset<<<1, 1, 0, s>>>(snapE, snapR, snapStep);
  return cudaGetLastError();
}

bool energy_small_fits(int N, double jmax) { return N <= ES_MAXN && double(N) * N * jmax <= double(1 << 24); }

cudaError_t launch_energy_small(const double* J64, const float* psi, int N, int Np, int R, double* E,
                                cudaStream_t s) {
  k_energy_small<<<R, 32 * ES_WARPS, 0, s>>>(J64, psi, N, Np, E);
  return cudaGetLastError();
}

cudaError_t launch_argmin(const double* E, int R, double* bestE, int* bestR, cudaStream_t s) {
  k_argmin<<<1, 1024, 0, s>>>(E, R, bestE, bestR);
  return cudaGetLastError();
}

cudaError_t launch_best_cfg(const float* psi, const int* bestR, int N, int Np, int cplx, signed char* s8, double* th,
                            cudaStream_t s) {
  k_best_cfg<<<grid_for(N), 256, 0, s>>>(psi, bestR, N, Np, cplx, s8, th);
  return cudaGetLastError();
}

}  // namespace gda

namespace gda {

// Host layout <-> device layout of the state.  Host psi: restart-major,
// (re, im) interleaved for XY; gamma: [R][N]; beta: [R].
__global__ void k_pack_state(const float* psi, const float* gam, const float* beta, int N, int Np, int R, int cplx,
                             float* hpsi, float* hgam, float* hbeta) {
  const size_t total = size_t(R) * N;
  const int W = cplx ? 2 : 1;
  for (size_t idx = blockIdx.x * size_t(blockDim.x) + threadIdx.x; idx < total; idx += size_t(gridDim.x) * blockDim.x) {
    const int r = int(idx / N), i = int(idx % N);
    if (hpsi)
      for (int p = 0; p < W; ++p) hpsi[idx * W + p] = psi[size_t(W * r + p) * Np + i];
    if (hgam) hgam[idx] = gam[size_t(r) * Np + i];
    if (hbeta && i == 0) hbeta[r] = beta[r];
  }
}

__global__ void k_unpack_state(float* psi, float* gam, float* beta, int N, int Np, int R, int cplx, const float* hpsi,
                               const float* hgam, const float* hbeta) {
  const size_t total = size_t(R) * N;
  const int W = cplx ? 2 : 1;
  for (size_t idx = blockIdx.x * size_t(blockDim.x) + threadIdx.x; idx < total; idx += size_t(gridDim.x) * blockDim.x) {
    const int r = int(idx / N), i = int(idx % N);
    for (int p = 0; p < W; ++p) psi[size_t(W * r + p) * Np + i] = hpsi[idx * W + p];
    gam[size_t(r) * Np + i] = hgam ? hgam[idx] : 0.0f;
    if (i == 0) beta[r] = hbeta ? hbeta[r] : 1.0f;
  }
}

// Instance checks and operand preparation.  J64 is [Np][Np] (zero padded,
// diagonal kept).  flags: bit0 non-finite, bit1 asymmetric, bit2 non-integer;
// maxabs: |J| maximum as the bits of a non-negative double.  One CTA per pair of
// mirrored 32 x 32 tiles: both are read along their rows and compared through
// shared memory, and the CTA's findings go out in one atomic each.  (Reading
// the mirrored element from global memory, a line per element, and a 64-bit
// atomic per thread took 0.68 ms at N = 2000; this takes 0.05.)
constexpr int CK = 32;
__global__ void __launch_bounds__(256) k_check_J(const double* J64, int N, int Np, int* flags,
                                                 unsigned long long* maxabs) {
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj < bi) return;
  __shared__ double t[CK][CK + 1];
  __shared__ double sm[8];
  __shared__ int sf[8];
  const int x = threadIdx.x & 31, y0 = threadIdx.x >> 5;
  int f = 0;
  double m = 0.0;
  auto look = [&](double v) {
    if (!isfinite(v)) {
      f |= 1;
    } else {
      if (v != rint(v)) f |= 4;
      m = fmax(m, fabs(v));
    }
  };
  for (int y = y0; y < CK; y += 8) {  // tile (bj, bi): element (row bj + y, column bi + x)
    const int i = bj * CK + y, j = bi * CK + x;
    const double v = i < N && j < N ? J64[size_t(i) * Np + j] : 0.0;
    look(v);
    t[y][x] = v;
  }
  __syncthreads();
  for (int y = y0; y < CK; y += 8) {  // tile (bi, bj), against its mirror
    const int i = bi * CK + y, j = bj * CK + x;
    const double v = i < N && j < N ? J64[size_t(i) * Np + j] : 0.0;
    look(v);
    const double w = t[x][y];
    if (isfinite(v) && v != w) f |= 2;
    if (isfinite(w) && v != w) f |= 2;
  }
  for (int o = 16; o; o >>= 1) {
    f |= __shfl_xor_sync(0xffffffffu, f, o);
    m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  }
  if (x == 0) {
    sf[y0] = f;
    sm[y0] = m;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) {
      f |= sf[k];
      m = fmax(m, sm[k]);
    }
    if (f) atomicOr(flags, f);
    if (m > 0.0) atomicMax(maxabs, static_cast<unsigned long long>(__double_as_longlong(m)));
  }
}

__global__ void k_check_g(const double* g, int N, int* flags) {
  int f = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    if (!isfinite(g[i])) f |= 8;
    if (g[i] != 0.0) f |= 16;
  }
  if (f) atomicOr(flags, f);
}

// diag = -sum_i J_ii in a fixed order (one block, a tree over its threads).
__global__ void __launch_bounds__(256) k_diag(const double* J64, int N, int Np, double* diag) {
  __shared__ double red[256];
  const int t = threadIdx.x;
  double s = 0.0;
  for (int i = t; i < N; i += 256) s += J64[size_t(i) * Np + i];
  red[t] = s;
  __syncthreads();
  for (int w = 128; w; w >>= 1) {
    if (t < w) red[t] += red[t + w];
    __syncthreads();
  }
  if (t == 0) *diag = -red[0];
}

// Coupling operands: J0 (diagonal removed) in FP32 and BF16.
__global__ void k_prepare_J(const double* J64, int Np, float* J32, __nv_bfloat16* J16) {
  const size_t total = size_t(Np) * Np;
  for (size_t idx = blockIdx.x * size_t(blockDim.x) + threadIdx.x; idx < total; idx += size_t(gridDim.x) * blockDim.x) {
    const int i = int(idx / Np), j = int(idx % Np);
    const double v = J64[idx];
    const float f = (i == j) ? 0.0f : float(v);
    J32[idx] = f;
    if (J16) J16[idx] = __float2bfloat16_rn(f);
  }
}

cudaError_t launch_pack_state(const float* psi, const float* gam, const float* beta, int N, int Np, int R, int cplx,
                              float* hpsi, float* hgam, float* hbeta, cudaStream_t s) {
  k_pack_state<<<grid_for(size_t(R) * N), 256, 0, s>>>(psi, gam, beta, N, Np, R, cplx, hpsi, hgam, hbeta);
  return cudaGetLastError();
}

cudaError_t launch_unpack_state(float* psi, float* gam, float* beta, int N, int Np, int R, int cplx, const float* hpsi,
                                const float* hgam, const float* hbeta, cudaStream_t s) {
  k_unpack_state<<<grid_for(size_t(R) * N), 256, 0, s>>>(psi, gam, beta, N, Np, R, cplx, hpsi, hgam, hbeta);
  return cudaGetLastError();
}

cudaError_t launch_check_instance(const double* J64, const double* g, int N, int Np, int* flags,
                                  unsigned long long* maxabs, double* diag, cudaStream_t s) {
  const int nb = (N + CK - 1) / CK;
  k_check_J<<<dim3(nb, nb), 256, 0, s>>>(J64, N, Np, flags, maxabs);
  k_check_g<<<grid_for(N), 256, 0, s>>>(g, N, flags);
  k_diag<<<1, 256, 0, s>>>(J64, N, Np, diag);
  return cudaGetLastError();
}

cudaError_t launch_prepare_J(const double* J64, int Np, float* J32, __nv_bfloat16* J16, cudaStream_t s) {
  k_prepare_J<<<grid_for(size_t(Np) * Np), 256, 0, s>>>(J64, Np, J32, J16);
  return cudaGetLastError();
}

}  // namespace gda
