// The FP64 sign iteration on the tensor cores (oz_path.cu): declarations shared with the FP64 path's host side.
#pragma once
#include "nolsm_internal.cuh"

namespace nolsm {

// Seven digits of 9 bits up to this dimension, eight of 8 bits above. The FP32 accumulators hold sums of K products
// of digits that add up coherently on the diagonal of X X (near convergence X is nearly symmetric): K 2^(2 kB - 2) / 3
// for uniform digits, 4.2e6 at 9 bits and K = 192 and 1.1e7 at 512, below 2^24 = 1.7e7; 10-bit digits reach it at
// K = 190 (seen on the 168-row water submatrices), although six of them would need a quarter fewer products.
constexpr int kOzNineBits = 512;

struct OzSolve {
  const int32_t* order; int32_t count;         // submatrices, largest first
  int32_t max_n;                               // largest dimension among them
  const int32_t* sub_n; const int32_t* nbf; const int64_t* a_off; const int64_t* c_off;
  const double* A; const double* Q; const double* Sc; const double* Hc; const double* lam; const double* lam_g;
  const int32_t* prep_status;
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
// how many clusters run at once (the scratch is sized for them)
int oz_clusters(int max_n, int dev, int sms);
// Leaves status[J] = kSubRefine for the submatrices k_ns_fp64 has to take.
nolsm_status launch_ns_oz(const OzSolve& a, cudaStream_t st);
// A_J in FP64 to Aout + a_off[J] and the centre columns of T_J(S)^-1 to Qout + c_off[J], prep_out[J] = kSubOk; kSubRefine
// or kSubPending where k_prepare has to take the submatrix.
nolsm_status launch_inverse_oz(const OzSolve& a, cudaStream_t st);

}  // namespace nolsm
