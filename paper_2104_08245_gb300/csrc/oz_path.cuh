// The FP64 sign iteration on the tensor cores (oz_path.cu): declarations shared with the FP64 path's host side.
#pragma once
#include "nolsm_internal.cuh"

namespace nolsm {

// Seven digits of 9 bits up to this dimension, eight of 8 bits above. The FP32 accumulators hold sums of K products
// of digits that add up coherently on the diagonal of X X (near convergence X is nearly symmetric): K 2^(2 kB - 2) / 3
// for uniform digits, 4.2e6 at 9 bits and K = 192 and 1.1e7 at 512, below 2^24 = 1.7e7; 10-bit digits reach it at
// K = 190 (seen on the 168-row water submatrices), although six of them would need a quarter fewer products.
constexpr int kOzNineBits = 512;

// What the fixed point takes: how many exponents of X are tried (each 3 above the last; what it drops and rounds grows
// with their square), and the ||I - T_J(S) X||_F of the FP32 inverse, a measure of the overlap's condition, from which the
// Cholesky factorisation prepares A_J instead (solving with the factor loses less than a product with the inverse).
// kFixedFp64, the FP64 class: no more than what is as accurate as FP64 arithmetic. Distance of A_J, Q and D from
// extended precision, relative to their largest entry, at n = 60 and 170, conditions 2 to 10: 1e-16 to 7e-16, with the
// FP64 kernels 6e-16 to 4e-15; at 250 to 1,000, which these limits leave to the FP64 kernels: up to 4e-13, 2e-14, 8e-13
// against 2e-13, 8e-14, 3e-13. The norm is 1e-5 to 5e-5 on water of any density, 1e-4 to 3e-4 at condition 50.
// kFixedLoose, the submatrices that a tensor-core mode hands over: what keeps some twelve digits, for the six of the mode
// (28 of 64 submatrices at condition 1,200: 14.5 ms a solve, 118 with the FP64 limits).
struct Fixed { int tries; float far; };
constexpr Fixed kFixedFp64{1, 2e-4f}, kFixedLoose{4, 0.5f};

struct OzSolve {
  const int32_t* order; int32_t count;         // submatrices, largest first
  int32_t max_n;                               // largest dimension among them
  const int32_t* sub_n; const int32_t* nbf; const int64_t* a_off; const int64_t* c_off;
  const double* A; const double* Q; const double* Sc; const double* Hc; const double* lam; const double* lam_g;
  const int32_t* prep_status;
  bool loose;                                  // kFixedLoose
  double mu, tol;
  int32_t max_iter; const int32_t* budget;
  uint16_t* planes; double* xd; int32_t R, LD, clusters;   // scratch: oz_planes(mode) planes of R x LD per cluster, R x LD
  double* Dc; double* tS; double* tH; int32_t* iters; int32_t* status; int32_t* rsteps; int32_t* nbelow;
  // launch_inverse_oz: the chunk's T_J(S), T_J(H0) (FP64, at a_off[J] - a_base and chunk_n2 further) and T_J(S)^-1 in
  // FP32 (at a_off[J] - a_base), where prep_out[J] is kSubOk
  const double* ws; int64_t a_base, chunk_n2; const float* X32; const int32_t* sub_c0;
  double* Aout; double* Qout; int32_t* prep_out;
};
int oz_planes(int mode);
// Whether the kernels for this dimension came out of the compiler with the registers that their split needs.
bool oz_ready(int max_n);
// how many clusters run at once (the scratch is sized for them)
int oz_clusters(int max_n, int dev, int sms);
// Leaves status[J] = kSubRefine for the submatrices k_ns_fp64 has to take.
nolsm_status launch_ns_oz(const OzSolve& a, cudaStream_t st);
// Leaves all of them.
nolsm_status leave_ns_oz(const OzSolve& a, cudaStream_t st);
// A_J in FP64 to Aout + a_off[J] and the centre columns of T_J(S)^-1 to Qout + c_off[J], prep_out[J] = kSubOk; kSubRefine
// or kSubPending where k_prepare has to take the submatrix.
nolsm_status launch_inverse_oz(const OzSolve& a, cudaStream_t st);

}  // namespace nolsm
