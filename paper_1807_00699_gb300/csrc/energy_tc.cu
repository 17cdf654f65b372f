// Eq. (1) energies in FP64 through BF16 tensor-core products.
//
// E_r = -sum_i s_i (J s)_i + sum_i g_i s_i needs T = J S in FP64 (2 N^2 C
// FLOP), and GB300's FP64 pipe runs at ~1.2 TFLOP/s.  Here both factors are
// cut into 8-bit digits and the products run on tcgen05 tensor cores, exactly
// (the error-free splitting of Ozaki, Ogita, Oishi & Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 59, 2012):
//   J_ij = 2^(e_i - 55) sum_k d_ijk 2^(8 (6 - k)),  s_j = 2^-55 sum_l c_jl 2^(8 (6 - l)),
// |d|, |c| <= 128, e_i the exponent of row i's largest |J_ij|, the digits of
// -x the negated digits of x.  A digit is a BF16 number; a product of digits
// is an integer <= 2^14, so FP32 accumulation over at most 512 of them (sums
// <= 2^23) is exact.  Each accumulator is added, shifted to its weight, into
// an int64 whose unit is 2^-61 of sum_j |J_ij| (the largest of 32 rows), or
// the weight of the last digit where that is coarser: the sum over j cannot
// overflow, and its error (the digit pairs below the unit, k + l > 6, are left
// out) stays below the rounding errors of the same sum in FP64, for rows of a
// few nonzeros as well (a bound of N times the largest |J_ij| in place of the
// sum loses 6 bits on 3-regular rows at N = 4096).  Real spins are +-1: one digit, 7 products.  Integer J takes
// as many digits as its largest entry needs and no scaling, so those energies
// are exact integers.
//
// Digit tiles (128 rows x 64 k) are stored in global memory in the 128-byte
// swizzled K-major form that tcgen05.mma reads, so a stage of the ring is two
// plain 16 KB bulk copies.  Warp 0 loads, warp 1 issues MMAs into two
// tensor-memory accumulators in turn, 16 warps drain them.  What bounds it is
// that read-out into the int64 sums: ~3.5 us per accumulation, whether of 2 K
// blocks (XY N = 100, R = 64: 28 in 98 us) or of 8 (N = 1000, R = 1024: 56 in 206).
// Measured (GB300): every restart's energy at XY N = 1000, R = 1024 takes 206
// us here plus 86 us for the spins' digits (and 38 us more for J's in the first
// call after a load), where the FP64 pipe took 4.10 ms; those of SK N = R = 4096
// take 0.87 ms (1.21 after a load), where ranking in compensated FP32 and
// evaluating the candidates in FP64 took 11.1 ms.  Against sums in extended
// precision the energies are 2-5 times closer than the FP64 pipe's
// (relative error, N = 150 / 777 / 1000: 1.4e-16 / 1.4e-16 / 1.8e-16, before
// 3.0e-16 / 7.2e-16 / 7.5e-16).
#include "energy_tc.h"

#include <algorithm>
#include <cmath>

#include "gda_internal.h"
#include "tc_ptx.cuh"

namespace gda {
namespace {

using namespace ptx;
constexpr int TILE = 128;
constexpr int STAGES = 6;
constexpr int EWARPS = 16;
constexpr int ETHREADS = 64 + 32 * EWARPS;
constexpr uint32_t TBYTES = uint32_t(kEnergyTileBytes);
constexpr uint32_t ESMEM = 1024 + STAGES * 2 * TBYTES;
// A complex spin is a square root and two divisions in FP64: one CTA takes 47 us
// for the 64 x 64 spins of a block, four take 13 (XY N = 100, R = 64).
constexpr int SPLIT = 4;
constexpr int KCHUNK = 8;  // K blocks of 64 per accumulation of digit products up to 2^14

// Unit k of a list (problem, row or column block, column block of a tile).
__device__ __forceinline__ int4 unit_of(const int4* u, int k, int rows) {
  return u ? u[k] : make_int4(0, k % rows, k / rows, 0);
}

// Exponent of a row with a non-finite entry (a J that gda_load_dev refused): its
// energies are NaN.
constexpr int kRowBad = 1 << 24;
__device__ __forceinline__ double scaled(double a, int ex) {  // a 2^ex for any ex
  return ex > kRowBad / 2 ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(a, ex);
}

// Digits of J, and whether they are J's own (EnergyProb::fmt).
__device__ __forceinline__ int2 format_of(const EnergyProb& P) { return P.fmt ? *P.fmt : make_int2(P.nsJ, P.jint); }

// Integers up to 2^(8 n - 1) are their own n digits; 0: J takes scaled digits.
__host__ __device__ inline int integer_digits(double jmax) {
  for (int n = 1; n <= 4; ++n)
    if (jmax >= 0.0 && jmax <= double(1ll << (8 * n - 1))) return n;
  return 0;
}

__global__ void k_energy_format(const int* flags, const unsigned long long* maxabs, int2* fmt) {
  const int n = (*flags & 5) ? 0 : integer_digits(__longlong_as_double((long long)*maxabs));
  *fmt = n ? make_int2(n, 1) : make_int2(kEnergySlices, 0);
}

// Byte offset of the 16-byte group k8 (8 values) of row r inside a digit tile.
__device__ __forceinline__ uint32_t tile_off(int r, int k8) { return uint32_t(r) * 128u + uint32_t((k8 ^ (r & 7)) << 4); }

// 8-bit signed digits of x (|x| <= 2^(8 ns - 1)), most significant first, as
// BF16 bits; digits of -x are the negated digits of x.
template <int NS>
__device__ __forceinline__ void digits(long long x, int ns, unsigned short (&d)[NS]) {
  const int sg = x < 0 ? -1 : 1;
  unsigned long long a = x < 0 ? 0ull - (unsigned long long)x : (unsigned long long)x;
#pragma unroll
  for (int k = NS - 1; k >= 0; --k) {
    if (k >= ns) continue;
    int v;
    if (k > 0) {
      v = int(a & 255u);
      if (v >= 128) v -= 256;
      a = (a - (unsigned long long)(long long)v) >> 8;
    } else {
      v = int(a);
    }
    d[k] = __bfloat16_as_ushort(__float2bfloat16_rn(float(sg * v)));
  }
}

// (e_i, l_i) with |J_ij| <= 2^e_i for every j and sum_j |J_ij| < 2^(e_i + l_i), a
// factor 2 of rounding aside (one warp per row; integers: e_i the scale of the
// digits of J itself).
__global__ void __launch_bounds__(256) k_energy_rexp(EnergyProb p0, const EnergyProb* probs, const int4* units) {
  const int4 U = unit_of(units, blockIdx.x, p0.mtn);
  const EnergyProb& P = probs ? probs[U.x] : p0;
  const int lane = threadIdx.x & 31;
  const int i = (P.mt0 + U.y) * TILE + int(blockIdx.y) * 8 + int(threadIdx.x >> 5);
  if (i >= P.N) return;
  const int2 F = format_of(P);
  double m = 0.0, a = 0.0;
  bool bad = false;
  for (int j = lane; j < P.N; j += 32) {
    const double v = fabs(P.J[size_t(i) * P.ld + j]);
    bad |= !isfinite(v);
    m = fmax(m, v);
    a += v;
  }
  bad = __any_sync(0xffffffffu, bad);
  for (int o = 16; o; o >>= 1) {
    m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    a += __shfl_xor_sync(0xffffffffu, a, o);
  }
  const int e = bad ? kRowBad : F.y ? 8 * F.x - 1 : m > 0.0 ? ilogb(m) + 1 : 0;
  const int lgN = P.N > 1 ? 32 - __clz(P.N - 1) : 0;
  const int l = bad || !(m > 0.0) ? 0 : isfinite(a) ? ilogb(a) + 1 - e : lgN;
  if (lane == 0) P.rexp[i] = make_int2(e, l);
}

// Digit tiles of J: one CTA per (row block, K block).
__global__ void __launch_bounds__(256) k_energy_slice_J(EnergyProb p0, const EnergyProb* probs, const int4* units) {
  const int4 U = unit_of(units, blockIdx.x, p0.mtn);
  const EnergyProb& P = probs ? probs[U.x] : p0;
  const int kb = blockIdx.y;
  if (kb >= P.KB) return;
  const int ns = format_of(P).x;
  unsigned char* out = P.Jd + (size_t(U.y) * ns * P.KB + kb) * TBYTES;
  for (int q = threadIdx.x; q < TILE * 8; q += 256) {
    const int r = q >> 3, k8 = q & 7;
    const int i = (P.mt0 + U.y) * TILE + r, j0 = kb * 64 + k8 * 8;
    unsigned short d[8][kEnergySlices] = {};
    if (i < P.N) {
      const int sh = 8 * ns - 1 - P.rexp[i].x;
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const double v = j0 + t < P.N ? P.J[size_t(i) * P.ld + j0 + t] : 0.0;
        digits(llrint(scalbn(v, sh)), ns, d[t]);
      }
    }
#pragma unroll
    for (int k = 0; k < kEnergySlices; ++k) {
      if (k >= ns) break;
      uint4 w;
      w.x = d[0][k] | (uint32_t(d[1][k]) << 16);
      w.y = d[2][k] | (uint32_t(d[3][k]) << 16);
      w.z = d[4][k] | (uint32_t(d[5][k]) << 16);
      w.w = d[6][k] | (uint32_t(d[7][k]) << 16);
      *reinterpret_cast<uint4*>(out + size_t(k) * P.KB * TBYTES + tile_off(r, k8)) = w;
    }
  }
}

// Projected spins of one column block and K block, SPLIT CTAs to each: digit
// tiles, and (complex spins) s itself in double for the reduction.  A row of a tile is a column
// of the state; complex spins are handled as the pair of columns 2r, 2r + 1.
__global__ void __launch_bounds__(256) k_energy_slice_S(EnergyProb p0, const EnergyProb* probs, const int4* units) {
  const int4 U = unit_of(units, blockIdx.x, p0.ntn);
  const EnergyProb& P = probs ? probs[U.x] : p0;
  const int kb = blockIdx.y;
  if (kb >= P.KB) return;
  const int ns = P.nsS;
  unsigned char* out = P.Sd + (size_t(U.y) * ns * P.KB + kb) * TBYTES;
  const size_t slice = size_t(P.KB) * TBYTES;
  if (!P.pmode) {
    for (int q = blockIdx.z * 256 + threadIdx.x; q < TILE * 8; q += SPLIT * 256) {
      const int cr = q >> 3, k8 = q & 7;
      const int c = (P.nt0 + U.y) * TILE + cr, i0 = kb * 64 + k8 * 8;
      uint32_t w[4] = {0u, 0u, 0u, 0u};
      if (c < P.C) {
        const float* src = P.psi + size_t(c) * P.Np + i0;  // Np is a multiple of 128: inside the column
#pragma unroll
        for (int t = 0; t < 8; ++t)
          if (i0 + t < P.N) w[t >> 1] |= (src[t] >= 0.0f ? 0x3F80u : 0xBF80u) << (16 * (t & 1));  // +-1
      }
      *reinterpret_cast<uint4*>(out + tile_off(cr, k8)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    return;
  }
  // complex: a thread takes 4 spins of a restart (half a 16-byte group of both of its rows)
  for (int q = blockIdx.z * 256 + threadIdx.x; q < (TILE / 2) * 16; q += SPLIT * 256) {
    const int rr = q >> 4, k4 = q & 15;
    const int c = (P.nt0 + U.y) * TILE + 2 * rr, i0 = kb * 64 + k4 * 4;
    unsigned short d[2][4][kEnergySlices] = {};
    if (c < P.C) {
      const float4 re = *reinterpret_cast<const float4*>(P.psi + size_t(c) * P.Np + i0);
      const float4 im = *reinterpret_cast<const float4*>(P.psi + size_t(c + 1) * P.Np + i0);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (i0 + t >= P.N) continue;
        const double x = (&re.x)[t], y = (&im.x)[t];
        double sr, si;
        if (P.pmode >= 2) {
          potts_project(x, y, P.pmode, sr, si);
        } else {
          const double m = sqrt(x * x + y * y);
          sr = m > 0.0 ? x / m : 1.0;
          si = m > 0.0 ? y / m : 0.0;
        }
        P.S64[size_t(c) * P.Np + i0 + t] = sr;
        P.S64[size_t(c + 1) * P.Np + i0 + t] = si;
        // a non-finite spin keeps zero digits: its own s makes the energy non-finite
        digits(isfinite(sr) ? llrint(sr * 36028797018963968.0) : 0ll, ns, d[0][t]);  // 2^55
        digits(isfinite(si) ? llrint(si * 36028797018963968.0) : 0ll, ns, d[1][t]);
      }
    }
#pragma unroll
    for (int w = 0; w < 2; ++w)
#pragma unroll
      for (int k = 0; k < kEnergySlices; ++k) {
        if (k >= ns) break;
        uint2 v;
        v.x = d[w][0][k] | (uint32_t(d[w][1][k]) << 16);
        v.y = d[w][2][k] | (uint32_t(d[w][3][k]) << 16);
        *reinterpret_cast<uint2*>(out + k * slice + tile_off(2 * rr + w, k4 >> 1) + 8 * (k4 & 1)) = v;
      }
  }
}

// The digit pairs of a problem in one order for all warp roles.
struct PairIter {
  int nsJ, nsS, lim, i, j;
  __device__ PairIter(int J, int S) : nsJ(J), nsS(S), lim(J > S ? J : S), i(0), j(0) {}
  __device__ bool done() const { return i >= nsJ; }
  __device__ void next() {
    ++j;
    if (j >= nsS || i + j >= lim) {
      j = 0;
      ++i;
    }
  }
  __device__ int weight() const { return 8 * ((nsJ - 1 - i) + (nsS - 1 - j)); }
};

__device__ __forceinline__ int chunk_kb(const EnergyProb& P) { return P.nsS > 1 ? KCHUNK : P.KB; }

// acc += v 2^sh, rounded half away from zero for sh < 0 (so that the sum of -v is minus the sum of v).
__device__ __forceinline__ void add_shifted(long long& acc, int v, int sh) {
  if (sh < 0) {
    const int m = ((v < 0 ? -v : v) + (1 << (-sh - 1))) >> -sh;
    acc += v < 0 ? -m : m;
  } else if (sh <= 30) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(v), "r"(1 << sh));
  } else {
    acc += (long long)v << sh;
  }
}

__global__ void __launch_bounds__(ETHREADS, 1) k_energy_product(const __grid_constant__ EnergyProb p0,
                                                               const EnergyProb* probs, const int4* units,
                                                               int n_tile, int* err, long long lim) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * STAGES + 4];
  __shared__ double s_red[4][TILE];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto full_bar = [&](int s) { return smem_u32(bars + s); };
  auto empty_bar = [&](int s) { return smem_u32(bars + STAGES + s); };
  auto acc_full = [&](int b) { return smem_u32(bars + 2 * STAGES + b); };
  auto acc_empty = [&](int b) { return smem_u32(bars + 2 * STAGES + 2 + b); };
  auto aborted = [&]() { return *(volatile int*)&s_abort != 0; };
  const int2 f0 = probs ? make_int2(0, 0) : format_of(p0);  // problems of a list carry their own
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full(b), 1);
      mbar_init(acc_empty(b), EWARPS);
    }
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(smem_u32(&s_tmem), 256);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = warp_uniform(s_tmem);

  if (warp == 0) {
    if (elect_one()) {
      int it = 0;
      bool stop = false;
      for (int t = blockIdx.x; t < n_tile && !stop; t += gridDim.x) {
        const int4 U = unit_of(units, t, p0.mtn);
        const EnergyProb& P = probs ? probs[U.x] : p0;
        const int nsJ = probs ? P.nsJ : f0.x;
        for (PairIter q(nsJ, P.nsS); !q.done() && !stop; q.next()) {
          const unsigned char* A = P.Jd + (size_t(U.y) * nsJ + q.i) * P.KB * TBYTES;
          const unsigned char* B = P.Sd + (size_t(U.z) * P.nsS + q.j) * P.KB * TBYTES;
          for (int kb = 0; kb < P.KB; ++kb, ++it) {
            const int s = it % STAGES;
            if (!mbar_wait(empty_bar(s), ((it / STAGES) & 1) ^ 1, lim) || aborted()) {
              stop = true;
              break;
            }
            const uint32_t dst = base + s * 2 * TBYTES;
            mbar_arrive_expect_tx(full_bar(s), 2 * TBYTES);
            bulk_load(dst, A + size_t(kb) * TBYTES, TBYTES, full_bar(s));
            bulk_load(dst + TBYTES, B + size_t(kb) * TBYTES, TBYTES, full_bar(s));
          }
        }
      }
      if (stop) {
        atomicOr(&s_abort, 1);
        for (int k = it - 1; k >= 0 && k >= it - STAGES; --k)  // copies still in flight
          (void)mbar_wait(full_bar(k % STAGES), (k / STAGES) & 1, lim);
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      constexpr uint32_t idesc = idesc_bf16<TILE>();
      const uint64_t d0 = sdesc_sw128(base);
      int it = 0, use = 0;
      bool stop = false;
      for (int t = blockIdx.x; t < n_tile && !stop; t += gridDim.x) {
        const int4 U = unit_of(units, t, p0.mtn);
        const EnergyProb& P = probs ? probs[U.x] : p0;
        const int nsJ = probs ? P.nsJ : f0.x;
        const int ck = chunk_kb(P);
        for (PairIter q(nsJ, P.nsS); !q.done() && !stop; q.next()) {
          for (int k0 = 0; k0 < P.KB && !stop; k0 += ck, ++use) {
            const int b = use & 1;
            if (!mbar_wait(acc_empty(b), ((use >> 1) & 1) ^ 1, lim) || aborted()) {
              stop = true;
              break;
            }
            tc_fence_after();
            const int kend = k0 + ck < P.KB ? k0 + ck : P.KB;
            for (int kb = k0; kb < kend; ++kb, ++it) {
              const int s = it % STAGES;
              if (!mbar_wait(full_bar(s), (it / STAGES) & 1, lim) || aborted()) {
                stop = true;
                break;
              }
              tc_fence_after();
#pragma unroll
              for (int k = 0; k < 4; ++k)
                mma_bf16(tmem + b * TILE, sdesc_at(d0, s * 2 * TBYTES + k * 32), sdesc_at(d0, s * 2 * TBYTES + TBYTES + k * 32), idesc,
                         (kb > k0) || k);
              mma_commit(empty_bar(s));
            }
            mma_commit(acc_full(b));  // also after an abort: tracks every MMA issued
          }
        }
      }
      if (stop) {
        atomicOr(&s_abort, 1);
        // the MMAs in flight finish before tensor memory is freed
        if (use > 0) (void)mbar_wait(acc_full((use - 1) & 1), ((use - 1) >> 1) & 1, lim);
      }
    }
  } else {
    const int e = threadIdx.x - 64;
    const int q4 = warp & 3;           // tensor-memory lane quarter
    const int cpart = (warp - 2) >> 2;  // 32 of the tile's 128 columns
    int use = 0;
    for (int t = blockIdx.x; t < n_tile; t += gridDim.x) {
      const int4 U = unit_of(units, t, p0.mtn);
      const EnergyProb& P = probs ? probs[U.x] : p0;
      const int nsJ = probs ? P.nsJ : f0.x;
      const int ck = chunk_kb(P);
      const int i = (P.mt0 + U.y) * TILE + 32 * q4 + lane;
      const int2 re = i < P.N ? P.rexp[i] : make_int2(0, -(1 << 20));
      // unit of the int64 sums of the warp's rows: 2^unit of digit weight one, so that |sum| < 2^62
      const int fb = 8 * nsJ - 1 + (P.nsS > 1 ? 8 * P.nsS - 1 : 0);
      const int unit = max(0, fb + __reduce_max_sync(0xffffffffu, re.y) + 1 - 62);
      long long acc[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) acc[k] = 0;
      bool ok = true;
      for (PairIter q(nsJ, P.nsS); !q.done() && ok; q.next()) {
        const int sh = q.weight() - unit;
        for (int k0 = 0; k0 < P.KB; k0 += ck, ++use) {
          const int b = use & 1;
          ok = __all_sync(0xffffffffu, mbar_wait(acc_full(b), (use >> 1) & 1, lim) && !aborted());
          if (!ok) break;
          tc_fence_after();
          const uint32_t ta = tmem + b * TILE + (uint32_t(32 * q4) << 16) + cpart * 32;
          uint32_t v0[16], v1[16];
          tmem_ld16_nowait(ta, v0);
          tmem_ld16_nowait(ta + 16, v1);
          tmem_wait_ld16(v0);
          tmem_regs_after_wait16(v1);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty(b));
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            add_shifted(acc[k], __float2int_rn(__uint_as_float(v0[k])), sh);
            add_shifted(acc[16 + k], __float2int_rn(__uint_as_float(v1[k])), sh);
          }
        }
      }
      // Eq. (1) terms of row i and their sum over the rows, per restart; one
      // tree over the rows for every column, whatever its place
      const int c0 = (P.nt0 + U.z) * TILE + cpart * 32;
      const bool row = ok && i < P.N;
      const double gi = row && P.g ? P.g[i] : 0.0;
      const int ex = row ? unit - fb + re.x : 0;
      const bool wide = ex < -1000 || ex > 900;  // couplings near the ends of the double range
      const double f = __longlong_as_double((long long)((wide ? 0 : ex) + 1023) << 52);
      double v[32];
      if (P.pmode) {
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int c = c0 + 2 * u;
          v[u] = 0.0;
          if (row && c < P.C) {
            const double sr = P.S64[size_t(c) * P.Np + i], si = P.S64[size_t(c + 1) * P.Np + i];
            const double a = fma(sr, double(acc[2 * u]), si * double(acc[2 * u + 1]));
            v[u] = fma(gi, sr, -(wide ? scaled(a, ex) : a * f));
          }
        }
#pragma unroll
        for (int o = 16, n = 8; n; o >>= 1, n >>= 1)
#pragma unroll
          for (int u = 0; u < n; ++u) {
            const bool up = lane & o;
            const double give = up ? v[u] : v[u + n];
            v[u] = (up ? v[u + n] : v[u]) + __shfl_xor_sync(0xffffffffu, give, o);
          }
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        if (!(lane & 1))  // lane bits 4..1 are the restart's bits 3..0
          s_red[q4][cpart * 16 + (lane >> 1)] = v[0];
      } else if (probs ? P.jint : f0.y) {
        // integers: acc is (J s)_i itself (unit 0); 32 rows of them stay below
        // 2^52, summed as integers (in FP64, at a 64th of the rate, a tile's
        // sums took 30 of the kernel's 49 us at N = 100, R = 256)
        unsigned neg = 0;  // columns of spin -1
#pragma unroll 4
        for (int u = 0; u < 32; ++u)
          if (row && c0 + u < P.C && !(P.psi[size_t(c0 + u) * P.Np + i] >= 0.0f)) neg |= 1u << u;
#pragma unroll
        for (int u = 0; u < 32; ++u) acc[u] = !row || c0 + u >= P.C ? 0 : (neg >> u & 1) ? -acc[u] : acc[u];
#pragma unroll
        for (int o = 16, n = 16; n; o >>= 1, n >>= 1)
#pragma unroll
          for (int u = 0; u < n; ++u) {
            const bool up = lane & o;
            const long long give = up ? acc[u] : acc[u + n];
            acc[u] = (up ? acc[u + n] : acc[u]) + __shfl_xor_sync(0xffffffffu, give, o);
          }
        double e0 = -double(acc[0]);
        if (__any_sync(0xffffffffu, gi != 0.0)) {
          double v[32];
#pragma unroll
          for (int u = 0; u < 32; ++u) {
            v[u] = !row || c0 + u >= P.C ? 0.0 : (neg >> u & 1) ? -gi : gi;
          }
#pragma unroll
          for (int o = 16, n = 16; n; o >>= 1, n >>= 1)
#pragma unroll
            for (int u = 0; u < n; ++u) {
              const bool up = lane & o;
              const double give = up ? v[u] : v[u + n];
              v[u] = (up ? v[u + n] : v[u]) + __shfl_xor_sync(0xffffffffu, give, o);
            }
          e0 += v[0];
        }
        s_red[q4][cpart * 32 + lane] = e0;
      } else {
#pragma unroll
        for (int u = 0; u < 32; ++u) {
          const int c = c0 + u;
          v[u] = 0.0;
          if (row && c < P.C) {
            const double s = P.psi[size_t(c) * P.Np + i] >= 0.0f ? 1.0 : -1.0;
            const double a = double(acc[u]);
            v[u] = s * (gi - (wide ? scaled(a, ex) : a * f));
          }
        }
#pragma unroll
        for (int o = 16, n = 16; n; o >>= 1, n >>= 1)
#pragma unroll
          for (int u = 0; u < n; ++u) {
            const bool up = lane & o;
            const double give = up ? v[u] : v[u + n];
            v[u] = (up ? v[u + n] : v[u]) + __shfl_xor_sync(0xffffffffu, give, o);
          }
        s_red[q4][cpart * 32 + lane] = v[0];
      }
      // one decision for all warps; the vote also publishes s_red
      if (!epi_vote_all<32 * EWARPS>(ok)) {
        atomicOr(&s_abort, 1);
        break;
      }
      const int W = P.pmode ? 2 : 1;
      if (e < TILE / W) {
        const int r = (P.nt0 + U.z) * TILE / W + e;
        if (r < P.R)
          P.part[size_t(P.mt0 + U.y) * P.ldp + r] = ((s_red[0][e] + s_red[1][e]) + s_red[2][e]) + s_red[3][e];
      }
      epi_bar_sync_n<32 * EWARPS>();  // s_red is free for the next tile
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && s_abort) atomicOr(err, E_TIMEOUT);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
}

__global__ void k_energy_sum(const double* part, int mt, int R, int ldp, double* E) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= R) return;
  double s = 0.0;
  for (int t = 0; t < mt; ++t) s += part[size_t(t) * ldp + r];
  E[r] = s;
}

}  // namespace

EnergyProb energy_prob(int N, int Np, int ld, int R, int C, int pmode, double jmax) {
  EnergyProb p{};
  p.N = N; p.Np = Np; p.ld = ld; p.R = R; p.C = C;
  p.pmode = pmode;
  p.KB = (N + 63) / 64;
  p.nsJ = kEnergySlices;
  p.nsS = pmode ? kEnergySlices : 1;
  if (const int n = integer_digits(jmax)) {
    p.nsJ = n;
    p.jint = 1;
  }
  p.mtn = (N + TILE - 1) / TILE;
  p.ntn = (C + TILE - 1) / TILE;
  return p;
}

size_t energy_J_bytes(const EnergyProb& p) { return size_t(p.mtn) * p.nsJ * p.KB * kEnergyTileBytes; }
size_t energy_S_bytes(const EnergyProb& p) { return size_t(p.ntn) * p.nsS * p.KB * kEnergyTileBytes; }

cudaError_t launch_energy_format(const int* flags, const unsigned long long* maxabs, int2* fmt, cudaStream_t s) {
  k_energy_format<<<1, 1, 0, s>>>(flags, maxabs, fmt);
  return cudaGetLastError();
}

cudaError_t launch_energy_slice_J(const EnergyProb& p0, const EnergyUnits& u, cudaStream_t s) {
  k_energy_rexp<<<dim3(u.n_row, TILE / 8), 256, 0, s>>>(p0, u.probs, u.row);
  k_energy_slice_J<<<dim3(u.n_row, u.KBmax), 256, 0, s>>>(p0, u.probs, u.row);
  return cudaGetLastError();
}

cudaError_t launch_energy_slice_S(const EnergyProb& p0, const EnergyUnits& u, cudaStream_t s) {
  k_energy_slice_S<<<dim3(u.n_col, u.KBmax, SPLIT), 256, 0, s>>>(p0, u.probs, u.col);
  return cudaGetLastError();
}

cudaError_t energy_init() {
  return cudaFuncSetAttribute(k_energy_product, cudaFuncAttributeMaxDynamicSharedMemorySize, ESMEM);
}

cudaError_t launch_energy_product(const EnergyProb& p0, const EnergyUnits& u, int sms, int* err, cudaStream_t s) {
  k_energy_product<<<std::min(u.n_tile, sms), ETHREADS, ESMEM, s>>>(p0, u.probs, u.tile, u.n_tile, err, kWaitCycles);
  return cudaGetLastError();
}

cudaError_t launch_energy_sum(const double* part, int mt, int R, int ldp, double* E, cudaStream_t s) {
  k_energy_sum<<<(R + 255) / 256, 256, 0, s>>>(part, mt, R, ldp, E);
  return cudaGetLastError();
}

}  // namespace gda
