// FP64 energies of projected spins on the tensor cores (energy_tc.cu).
#pragma once
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace gda {

constexpr int kEnergySlices = 7;                     // 8-bit digits of a 55-bit fixed-point value
constexpr size_t kEnergyTileBytes = 128 * 64 * 2;    // one digit tile: 128 rows x 64 BF16, swizzled
// Bounds on the digit workspaces (a batch puts both kinds into their sum):
// larger products are cut into panels.
constexpr size_t kEnergyJBytes = size_t(2) << 30;
constexpr size_t kEnergySBytes = size_t(512) << 20;

// One product T = J S with its Eq. (1) reduction: row blocks [mt0, mt0 + mtn)
// of an N-spin instance against column blocks [nt0, nt0 + ntn) of its state.
struct EnergyProb {
  const double* J;      // [N][ld], diagonal kept
  const double* g;      // [N] or nullptr
  const float* psi;     // amplitudes [C][Np], column-major
  double* S64;          // complex spins s in double [C][Np]; nullptr for real spins
  int2* rexp;           // [N] (e, l) of every row: |J_ij| <= 2^e, sum_j |J_ij| < 2^(e + l)
  unsigned char* Jd;    // digit tiles [mtn][nsJ][KB]
  unsigned char* Sd;    // digit tiles [ntn][nsS][KB]
  double* part;         // [row blocks of 128][ldp] partial energies
  int N, Np, ld, R, C, ldp;
  int pmode;            // 0 real spins, 1 XY, q >= 2 Potts roots
  int nsJ, nsS, KB;     // digits of J and of s; K blocks of 64 spins
  int jint;             // J holds integers with |J_ij| <= 2^(8 nsJ - 1): digits of J itself
  int mt0, mtn, nt0, ntn;
  // nsJ and jint of the J loaded when the kernels run, on the device, or
  // nullptr: those above.  Work recorded into a graph outlives the J it was
  // recorded with.
  const int2* fmt;
};

// Digits, K blocks and tile counts of an N-spin instance with C columns
// (pointers and panel ranges are the caller's; the panel covers everything).
// jmax: the largest |J_ij| when every J_ij is an integer, else a negative value.
// (A caller with fmt passes -1 and gets sizes that hold any J.)
EnergyProb energy_prob(int N, int Np, int ld, int R, int C, int pmode, double jmax);
size_t energy_J_bytes(const EnergyProb& p);  // digit bytes of the panel's rows
size_t energy_S_bytes(const EnergyProb& p);  // digit bytes of the panel's columns

// *fmt = (nsJ, jint) of the checked J: flags and maxabs of launch_check_instance.
cudaError_t launch_energy_format(const int* flags, const unsigned long long* maxabs, int2* fmt, cudaStream_t s);

// units (device, or nullptr with probs = nullptr: the one problem p0): n_row
// entries (problem, row block), n_col entries (problem, column block) and
// n_tile entries (problem, row block, column block), blocks counted from the
// panel's start; KBmax the largest KB of the problems.
struct EnergyUnits {
  const EnergyProb* probs;
  const int4* row;
  const int4* col;
  const int4* tile;
  int n_row, n_col, n_tile, KBmax;
};
cudaError_t launch_energy_slice_J(const EnergyProb& p0, const EnergyUnits& u, cudaStream_t s);
cudaError_t launch_energy_slice_S(const EnergyProb& p0, const EnergyUnits& u, cudaStream_t s);
cudaError_t energy_init();  // once per device, before its first product
cudaError_t launch_energy_product(const EnergyProb& p0, const EnergyUnits& u, int sms, int* err, cudaStream_t s);

// E[r] = sum over the row blocks of part (mt rows of ldp), r < R.
cudaError_t launch_energy_sum(const double* part, int mt, int R, int ldp, double* E, cudaStream_t s);

}  // namespace gda
