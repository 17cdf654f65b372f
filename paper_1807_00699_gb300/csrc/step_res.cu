// Resident persistent GD kernel (forward Euler, BF16 coupling product).
//
// One cooperative launch runs many steps.  Each CTA owns 128 rows (spins i) and
// one 128-column block, or one or two 64-column blocks, for the whole launch
// and keeps their FP32 state in tensor memory: the accumulators (columns
// 0..127), the amplitudes psi (128..255) and the gains gamma (256..), so per
// step the only global traffic is the BF16 operand X = bf16(psi) that every
// CTA reads and writes.  Steps are ordered by dataflow flags, one per row block
// and column block: the epilogue of block (m, c) writes its slice of X^{n+1}
// and then releases flag[c][m] = step + 1; the operand producer of column block
// c acquires flag[c][kb / 2] before loading K-block kb of X^{n+1}.  Column
// blocks never wait on each other.  Every wait is bounded.
//
// A step of one block is a serial chain: K loop, epilogue, flags, first operand
// tile.  64-column blocks shorten it and take more SMs, so they are used where
// each gets an SM of its own; two per CTA (one's K loop under the other's
// epilogue) pay only where the coupling tiles stay in shared memory (at most 9
// K-blocks).  Measured (GB300, us a step, against one 128 x 128 tile per CTA
// with MMAs issued from an `if (lane == 0)` branch): XY N = 1000, R = 1024 9.0 /
// 10.2; XY N = 2000, R = 256 12.0 / 15.6; XY N = 500, R = 300 5.1 / 7.4; XY N =
// 1024, R = 64 6.7 / 9.4; Ising N = 300, R = 4000 6.8 / 7.8.
//
// Roles: warp 0 operand (B) producer; warp 1 TMEM allocator + MMA issuer;
// warps 2..17 epilogue (warp w reads TMEM lane quarter w % 4 and a quarter of
// a block's columns); warp 18 coupling (A) producer.
// Per-element arithmetic is the Euler update of Eqs. (2), (5), (6) with the
// same FP32 expression sequence as the per-step kernels.
#include "tc_epilogue.cuh"
#include "tc_ptx.cuh"
#include "res.h"

namespace gda {
namespace {

using namespace ptx;
constexpr int EPI_WARPS = 16;                 // 4 per tensor-memory lane quarter
constexpr int RES_THREADS = 96 + 32 * EPI_WARPS;
constexpr int COLS = 128;                     // columns per CTA at most
constexpr uint32_t A_BYTES = BM * BK * 2;
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t T_PSI = 128;  // tensor-memory column of psi
constexpr uint32_t T_GAM = 256;  // tensor-memory column of gamma
// Two 64-column blocks per CTA up to this N (9 K-blocks: coupling tiles kept).
// Measured (us a step, two 64-column blocks / one of 128 columns): Ising N =
// 300, R = 4000 6.8 / 8.0; XY N = 1000, R = 1024 11.7 / 9.0; XY N = 2000, R =
// 500 21.3 / 13.5: where tiles are not kept, the two blocks load them twice.
// With noise decay each block also waits for the density sums of its column
// block: Ising N = 130, R = 6000 10.5 / 9.2; N = 300, R = 4096 10.6 / 10.3, R =
// 6000 10.9 / 11.6; N = 450, R = 4096 10.4 / 11.8, so one block up to N = 256.
constexpr int kResPairedMaxN = 576, kResPairedMinNDecay = 257;
// Rings of a CTA whose blocks have BN columns.
template <int BN>
struct ResCfg {
  static constexpr uint32_t B_BYTES = BN * BK * 2;
  static constexpr int A_SLOTS = BN == 64 ? 9 : 6;  // coupling tiles
  static constexpr int B_STAGES = A_SLOTS;          // operand tiles
  static constexpr int NBARS = 2 * A_SLOTS + 2 * B_STAGES + 4;
  static constexpr uint32_t TAIL = NBARS * 8 + (3 * COLS + 4 * BN) * 4 + 16;
  static constexpr uint32_t SMEM = 1024 + A_SLOTS * A_BYTES + B_STAGES * B_BYTES + TAIL;
  static_assert(SMEM <= 227 * 1024, "shared memory of one CTA");
};

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * EPI_WARPS) : "memory"); }

// Bounded wait until a block flag reaches target (acquire).
__device__ __forceinline__ bool flag_wait(const unsigned* f, unsigned target, long long limit) {
  if (ld_acquire_gpu(f) >= target) return true;
  const long long t0 = clock64();
  while (ld_acquire_gpu(f) < target) {
    if (clock64() - t0 > limit) return false;
  }
  return true;
}

// SUBS blocks of BN columns per CTA.
template <bool CPLX, int BN, int SUBS>
__global__ void __launch_bounds__(RES_THREADS, 1)
    step_res_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, ResArgs ra,
                    StepArgs a) {
  using Cfg = ResCfg<BN>;
  constexpr int A_SLOTS = Cfg::A_SLOTS, B_STAGES = Cfg::B_STAGES, NBARS = Cfg::NBARS;
  constexpr uint32_t B_BYTES = Cfg::B_BYTES;
  constexpr int CPT = BN / (EPI_WARPS / 4);  // columns per epilogue thread and block
  static_assert(SUBS * BN <= COLS, "tensor memory of one CTA");
  constexpr int W = CPLX ? 2 : 1;
  constexpr int RPT = BN / W;           // restarts per block
  constexpr int CW = 8;                 // columns per epilogue chunk
  constexpr int GR = CW / W;            // restarts per chunk
  constexpr int NCH = CPT / CW;
  static_assert(NCH % 2 == 0, "chunks are processed in pairs");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);
  const uint32_t sA = base;
  const uint32_t sB = base + A_SLOTS * A_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + A_SLOTS * A_BYTES + B_STAGES * B_BYTES);
  float* s_beta = reinterpret_cast<float*>(bars + NBARS);  // beta^n per local restart [SUBS][RPT]
  float* s_bstage = s_beta + COLS;                         // beta used in this step
  float* s_dsc = s_bstage + COLS;
  float* s_red = s_dsc + COLS;  // [4][BN]
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(s_red + 4 * BN);
  int* s_flag = reinterpret_cast<int*>(s_tmem + 1);  // [0] abort, [1] diverged

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int MT = int(gridDim.y);
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * (SUBS * BN);
  const int nsub = SUBS == 1 || a.C - n0 <= BN ? 1 : 2;  // blocks of this CTA that hold columns
  const int KB = (a.N + BK - 1) / BK;
  const bool kept = KB <= A_SLOTS;  // the CTA's coupling tiles stay in shared memory for the whole launch
  const long long lim = a.wait_cycles;
  auto a_full = [&](int s) { return smem_u32(bars + s); };
  auto a_empty = [&](int s) { return smem_u32(bars + A_SLOTS + s); };
  auto b_full = [&](int s) { return smem_u32(bars + 2 * A_SLOTS + s); };
  auto b_empty = [&](int s) { return smem_u32(bars + 2 * A_SLOTS + B_STAGES + s); };
  auto acc_full = [&](int h) { return smem_u32(bars + 2 * A_SLOTS + 2 * B_STAGES + h); };
  auto acc_free = [&](int h) { return smem_u32(bars + 2 * A_SLOTS + 2 * B_STAGES + 2 + h); };
  auto aborted = [&]() { return *(volatile int*)&s_flag[0] != 0; };

  if (threadIdx.x == 0) {
    stamp(a, 0);
    for (int s = 0; s < NBARS; ++s) mbar_init(smem_u32(bars + s), 1);
    s_flag[0] = 0;
    s_flag[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(smem_u32(s_tmem), TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = warp_uniform(*s_tmem);
  if (threadIdx.x == 0) stamp(a, 1);

  if (warp == 0) {
    // ---------------- operand producer ----------------
    if (elect_one()) {
      int it = 0;
      bool stop = false;
      for (int n = 0; n < ra.steps && !stop; ++n) {
        for (int h = 0; h < nsub && !stop; ++h) {
          const int brow = ((ra.buf0 + n) & 1) * ra.Cp + n0 + h * BN;
          const unsigned* fl = ra.flags + size_t(blockIdx.x * SUBS + h) * MT;
          int ready_m = -1;
          for (int kb = 0; kb < KB; ++kb, ++it) {
            const int s = it % B_STAGES;
            const int mb = (kb * BK) / BM;  // row block that produced these spins
            if (n > 0 && mb != ready_m) {
              if (!flag_wait(fl + mb, unsigned(n), lim)) {
                stop = true;
                break;
              }
              fence_proxy_async_global();
              ready_m = mb;
            }
            if (!mbar_wait(b_empty(s), ((it / B_STAGES) & 1) ^ 1, lim) || aborted()) {
              stop = true;
              break;
            }
            mbar_arrive_expect_tx(b_full(s), B_BYTES);
            tma_load_2d(sB + s * B_BYTES, &tmB, kb * BK, brow, b_full(s));
          }
        }
      }
      if (stop) {
        atomicOr(&s_flag[0], 1);
        for (int k = it - 1; k >= 0 && k >= it - B_STAGES; --k)  // copies still in flight
          (void)mbar_wait(b_full(k % B_STAGES), (k / B_STAGES) & 1, lim);
      }
    }
  } else if (warp == 2 + EPI_WARPS) {
    // ---------------- coupling producer ----------------
    if (elect_one()) {
      int it = 0;
      bool stop = false;
      const int rounds = kept ? 1 : ra.steps * nsub;
      for (int g = 0; g < rounds && !stop; ++g) {
        for (int kb = 0; kb < KB; ++kb, ++it) {
          const int s = it % A_SLOTS;
          if (!mbar_wait(a_empty(s), ((it / A_SLOTS) & 1) ^ 1, lim) || aborted()) {
            stop = true;
            break;
          }
          mbar_arrive_expect_tx(a_full(s), A_BYTES);
          tma_load_2d(sA + s * A_BYTES, &tmA, kb * BK, m0, a_full(s));
        }
      }
      if (stop) atomicOr(&s_flag[0], 1);
      if (stop || kept)  // copies still in flight (kept tiles: of a launch that stopped before it used them)
        for (int k = it - 1; k >= 0 && k >= it - A_SLOTS; --k)
          (void)mbar_wait(a_full(k % A_SLOTS), (k / A_SLOTS) & 1, lim);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (elect_one()) {
      constexpr uint32_t idesc = idesc_bf16<BN>();
      const uint64_t dA = sdesc_sw128(sA), dB = sdesc_sw128(sB);
      int ia = 0, ib = 0;
      bool stop = false;
      int last_h = -1, last_n = 0;  // block and step of the last commit to acc_full
      for (int n = 0; n < ra.steps && !stop; ++n) {
        for (int h = 0; h < nsub && !stop; ++h) {
          if ((n > 0 && !mbar_wait(acc_free(h), (n - 1) & 1, lim)) || aborted()) {
            stop = true;
            break;
          }
          tc_fence_after();
          for (int kb = 0; kb < KB; ++kb, ++ib) {
            const int s = ib % B_STAGES;
            const int sa = kept ? kb : ia % A_SLOTS;
            const bool a_ok = kept ? n + h > 0 || mbar_wait(a_full(sa), 0, lim)
                                   : mbar_wait(a_full(sa), (ia / A_SLOTS) & 1, lim);
            if (!a_ok || !mbar_wait(b_full(s), (ib / B_STAGES) & 1, lim) || aborted()) {
              stop = true;
              break;
            }
            tc_fence_after();
            if (n + h == 0 && kb == 0) stamp(a, 2);
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
              mma_bf16(tmem + h * BN, sdesc_at(dA, sa * A_BYTES + k * 32), sdesc_at(dB, s * B_BYTES + k * 32),
                       idesc, (kb | k) != 0);
            mma_commit(b_empty(s));
            if (!kept) {
              mma_commit(a_empty(sa));
              ++ia;
            }
          }
          if (n + h == 0) stamp(a, 3);
          mma_commit(acc_full(h));  // also after an abort: tracks every MMA issued
          last_h = h;
          last_n = n;
        }
      }
      if (stop) {
        atomicOr(&s_flag[0], 1);
        // the MMAs in flight finish before the CTA frees its tensor memory (the
        // epilogue may have stopped waiting for them)
        if (last_h >= 0) (void)mbar_wait(acc_full(last_h), last_n & 1, lim);
      }
    }
  } else {
    // ---------------- epilogue ----------------
    const int e = threadIdx.x - 64;
    const int q = warp & 3;
    const int part = (warp - 2) >> 2;
    const int i = m0 + 32 * q + lane;
    const bool row_ok = i < a.N;
    const size_t Np = a.Np;
    const uint32_t tb = tmem + (static_cast<uint32_t>(32 * q) << 16);
    const int cb = part * CPT;  // first column of this thread inside a block
    const float hd = row_ok ? a.h1[i] : 0.0f;
    const bool need_red = a.noise_decay && a.noise_D != 0.0f;

    // state -> tensor memory
    for (int h = 0; h < nsub; ++h) {
#pragma unroll 1
      for (int j = 0; j < CPT; j += 16) {
        const int lc = h * BN + cb + j, c = n0 + lc;
        float v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = a.psi_n[size_t(c + k) * Np + i];
        tmem_st16(tb + T_PSI + lc, v);
#pragma unroll
        for (int k = 0; k < 16 / W; ++k) v[k] = a.gam[size_t(c / W + k) * Np + i];
        if (CPLX)
          tmem_st8(tb + T_GAM + lc / W, v);
        else
          tmem_st16(tb + T_GAM + lc / W, v);
      }
      if (e < RPT) {
        const int r = (n0 + h * BN) / W + e;
        s_beta[h * BN + e] = r < a.R ? a.beta_in[r] : 1.0f;
      }
    }
    tmem_st_wait();

    StepArgs sa = a;
    sa.mode = M_EULER;
    int bad = 0;
    bool run = true;

    // one chunk of CW columns: accumulator, amplitudes, gains
    struct Chunk {
      uint32_t y[CW], p[CW], g[GR];
    };
    auto issue = [&](int lc, Chunk& t) {
      tmem_ld8_nowait(tb + lc, t.y);
      tmem_ld8_nowait(tb + T_PSI + lc, t.p);
      if (GR == 8)
        tmem_ld8_nowait(tb + T_GAM + lc / W, t.g);
      else
        tmem_ld4_nowait(tb + T_GAM + lc / W, t.g);
    };
    auto settle = [&](Chunk& t) {  // wait, then pin every register of t after it
      if (GR == 8)
        tmem_wait_ld8(t.g);
      else
        tmem_wait_ld4(t.g);
      tmem_regs_after_wait8(t.y);
      tmem_regs_after_wait8(t.p);
    };

#pragma unroll 1
    for (int n = 0; n < ra.steps && run; ++n) {
#pragma unroll 1
      for (int h = 0; h < nsub; ++h) {
        const int block = int(blockIdx.x) * SUBS + h;
        const int rbase = (n0 + h * BN) / W;
        unsigned* fl = ra.flags + size_t(block) * MT;
        sa.step = a.step + unsigned(n);
        sa.rho_in = (n & 1) ? ra.rho[1] : ra.rho[0];
        bool flags_ok = true;
        if (e < RPT) {
          const int r = rbase + e;
          s_bstage[h * BN + e] = s_beta[h * BN + e];
          if (need_red && n > 0) {  // partial sums of step n-1 from every row block of this column block, a lane per flag
            for (int mb = lane; mb < MT && flags_ok; mb += 32) flags_ok = flag_wait(fl + mb, unsigned(n), lim);
            flags_ok = __all_sync(0xffffffffu, flags_ok);
            __syncwarp();
          }
          s_dsc[h * BN + e] = r < a.R ? noise_scale(sa, r) : 0.0f;
        }
        // one decision for all epilogue warps (the vote is also the barrier that
        // publishes s_bstage / s_dsc)
        const bool ok = epi_vote_all<32 * EPI_WARPS>(flags_ok && mbar_wait(acc_full(h), n & 1, lim) && !aborted());
        tc_fence_after();
        if (!ok) {
          if (lane == 0) atomicOr(a.err, E_TIMEOUT);
          atomicOr(&s_flag[0], 1);
          run = false;
          break;
        }
        if (n + h == 0 && e == 0) stamp(a, 4);
        __nv_bfloat16* op = ra.ops + size_t((ra.buf0 + n + 1) & 1) * ra.Cp * Np;

        auto body = [&](int lc, const Chunk& t) {
          const int lr = h * BN + (lc - h * BN) / W;  // index into the per-restart arrays
          const int c0 = n0 + lc;
          float z[CW];
          bool any = false;
          if (a.noise_D != 0.0f)
#pragma unroll
            for (int u = 0; u < GR; ++u) any |= s_dsc[lr + u] != 0.0f;
#pragma unroll
          for (int qd = 0; qd < CW / 4; ++qd) {
            if (any) {
              philox_normal4(uint32_t(i), uint32_t((c0 >> 2) + qd), sa.step, 0u, a.seed, &z[4 * qd]);
            } else {
              z[4 * qd] = z[4 * qd + 1] = z[4 * qd + 2] = z[4 * qd + 3] = 0.0f;
            }
          }
          const int live = row_ok ? a.R - c0 / W : 0;  // restarts u < live exist
          __nv_bfloat16* const opc = op + size_t(c0) * Np + i;
          float npsi[CW], ngam[GR], red[GR];
#pragma unroll
          for (int u = 0; u < GR; ++u) {
            const int k0 = u * W;
            const float xr = __uint_as_float(t.p[k0]), xi = CPLX ? __uint_as_float(t.p[k0 + W - 1]) : 0.0f;
            const float yr = __uint_as_float(t.y[k0]), yi = CPLX ? __uint_as_float(t.y[k0 + W - 1]) : 0.0f;
            const float gs = __uint_as_float(t.g[u]);
            const float ds = any ? s_dsc[lr + u] : 0.0f;
            float kr, ki, kg;
            gd_rhs(xr, xi, gs, yr, yi, s_bstage[lr + u], hd, a.eps, a.rho_th, kr, ki, kg);
            float nr = axpy(a.dt, kr, xr);
            float ni = axpy(a.dt, ki, xi);
            const float ng = axpy(a.dt, kg, gs);
            nr = axpy(ds, z[k0], nr);
            if (CPLX) ni = axpy(ds, z[k0 + W - 1], ni);
            npsi[k0] = u < live ? nr : 0.0f;
            if (CPLX) npsi[k0 + W - 1] = u < live ? ni : 0.0f;
            ngam[u] = u < live ? ng : gs;
            const float rn = density(nr, ni);
            red[u] = u < live ? rn : 0.0f;
            bad |= u < live && !(rn < 1e30f);
            if (u < live) {
              opc[k0 * Np] = __float2bfloat16_rn(nr);
              if (CPLX) opc[(k0 + 1) * Np] = __float2bfloat16_rn(ni);
            }
          }
          tmem_st8(tb + T_PSI + lc, npsi);
          if (GR == 8)
            tmem_st8(tb + T_GAM + lc / W, ngam);
          else
            tmem_st4(tb + T_GAM + lc / W, ngam);
          if (need_red) {
#pragma unroll
            for (int u = 0; u < GR; ++u) {
              float x = red[u];
#pragma unroll
              for (int off = 16; off; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
              if (lane == 0) s_red[q * BN + (lr - h * BN) + u] = x;
            }
          }
        };
#pragma unroll 1
        for (int ch = 0; ch < NCH; ch += 2) {
          const int lc0 = h * BN + cb + ch * CW;
          Chunk t0, t1;
          issue(lc0, t0);
          issue(lc0 + CW, t1);
          settle(t0);  // a wait covers every load in flight
          tmem_regs_after_wait8(t1.y);
          tmem_regs_after_wait8(t1.p);
          if (GR == 8)
            tmem_regs_after_wait8(t1.g);
          else
            asm volatile("" : "+r"(t1.g[0]), "+r"(t1.g[1]), "+r"(t1.g[2]), "+r"(t1.g[3]));
          body(lc0, t0);
          body(lc0 + CW, t1);
        }
        tmem_st_wait();
        tc_fence_before();
        fence_proxy_async_global();
        if (e < RPT) s_beta[h * BN + e] = next_beta(sa, s_beta[h * BN + e]);  // read by this thread only
        epi_sync();
        if (e == 0) {
          mbar_arrive(acc_free(h));
          if (n + h == 0) stamp(a, 5);
        }
        if (need_red) {
          const int r = rbase + e;
          if (e < RPT && r < a.R)
            ((n & 1) ? ra.rho[0] : ra.rho[1])[size_t(blockIdx.y) * a.Rp + r] =
                s_red[e] + s_red[BN + e] + s_red[2 * BN + e] + s_red[3 * BN + e];
          epi_sync();
        }
        // a release store: ordered after every epilogue thread's writes (seen through the barrier)
        const bool withheld = ra.withhold_step == n + 1 && blockIdx.x + 1 == gridDim.x && blockIdx.y + 1 == gridDim.y;
        if (e == 0 && n + 1 < ra.steps && !withheld) st_release_gpu(fl + blockIdx.y, unsigned(n + 1));
      }
    }
    // tensor memory -> state
    if (!aborted()) {
      for (int h = 0; h < nsub; ++h) {
#pragma unroll 1
        for (int j = 0; j < CPT; j += 16) {
          const int lc = h * BN + cb + j, c = n0 + lc;
          float v[16];
          tmem_ld16(tb + T_PSI + lc, v);
          if (row_ok)
#pragma unroll
            for (int k = 0; k < 16; ++k)
              if (c + k < a.C) ra.psi_final[size_t(c + k) * Np + i] = v[k];
          if (CPLX)
            tmem_ld8(tb + T_GAM + lc / W, v);
          else
            tmem_ld16(tb + T_GAM + lc / W, v);
          if (row_ok)
#pragma unroll
            for (int k = 0; k < 16 / W; ++k)
              if (c / W + k < a.R) a.gam[size_t(c / W + k) * Np + i] = v[k];
        }
        const int r = (n0 + h * BN) / W + e;
        if (blockIdx.y == 0 && e < RPT && r < a.R) ra.beta_final[r] = s_beta[h * BN + e];
      }
    }
    if (bad) s_flag[1] = 1;
    epi_sync();
    if (e == 0 && s_flag[1]) atomicOr(a.err, E_DIVERGED);
    if (e == 0) stamp(a, 6);
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && s_flag[0]) atomicOr(a.err, E_TIMEOUT);
  if (threadIdx.x == 0) stamp(a, 7);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

template <bool CPLX, int BN, int SUBS>
cudaError_t launch_res_impl(const CUtensorMap& A, const CUtensorMap& B, const ResArgs& ra, const StepArgs& a,
                            cudaStream_t s) {
  auto kern = step_res_kernel<CPLX, BN, SUBS>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ResCfg<BN>::SMEM);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((a.C + SUBS * BN - 1) / (SUBS * BN), (a.N + BM - 1) / BM);
  cfg.blockDim = dim3(RES_THREADS);
  cfg.dynamicSmemBytes = ResCfg<BN>::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // every CTA resident: the block flags need it
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, A, B, ra, a);
}

template <bool CPLX>
cudaError_t launch_res(const TcPlan* plan, const ResArgs& ra, const StepArgs& a, int sms, cudaStream_t s) {
  const long long mt = (a.N + BM - 1) / BM;
  const CUtensorMap& A = *tc_plan_A(plan);
  // 64-column blocks where each gets an SM of its own; else two of them per CTA
  // while the chain they hide outweighs the coupling tiles they load twice, and
  // one 128-column block for larger N
  if ((a.C + 63) / 64 * mt <= sms) return launch_res_impl<CPLX, 64, 1>(A, *tc_plan_B64(plan), ra, a, s);
  const bool decay = a.noise_decay && a.noise_D != 0.0f;
  if (a.N <= kResPairedMaxN && !(decay && a.N < kResPairedMinNDecay))
    return launch_res_impl<CPLX, 64, 2>(A, *tc_plan_B64(plan), ra, a, s);
  return launch_res_impl<CPLX, 128, 1>(A, *tc_plan_B(plan), ra, a, s);
}

}  // namespace

bool res_fits(int N, int C, int device) {
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return false;
  int per_sm = 0;
  auto kern = step_res_kernel<true, 128, 1>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ResCfg<128>::SMEM) != cudaSuccess)
    return false;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, RES_THREADS, ResCfg<128>::SMEM) != cudaSuccess)
    return false;
  const long long grid = (long long)((C + COLS - 1) / COLS) * ((N + BM - 1) / BM);
  return per_sm >= 1 && grid <= (long long)per_sm * sms;
}

cudaError_t launch_step_res(const TcPlan* plan, const ResArgs& ra, const StepArgs& a, int sms, cudaStream_t s) {
  return a.cplx ? launch_res<true>(plan, ra, a, sms, s) : launch_res<false>(plan, ra, a, sms, s);
}

}  // namespace gda
