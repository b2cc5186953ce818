// The sign iteration with its operands on the SM (res_path.cu): declarations shared with the tensor-core host side.
#pragma once
#include "nolsm_internal.cuh"
#include "tc_split.cuh"

namespace nolsm {

// Largest submatrix: hi and lo planes of X in shared memory (147 KB), T and two Z accumulators in tensor memory
constexpr int kResMaxN = 192;

struct ResSolve {
  const int32_t* order; int32_t count;   // the work; submatrices above kResMaxN rows are passed over
  const int32_t* sub_n; const int32_t* nbf; const int64_t* a_off; const int64_t* c_off;
  const float* A; const double* Q; const double* Sc; const double* Hc; const double* lam; const double* lam_g;
  const int32_t* prep_status;
  double mu;
  float tol_ns, tol_accept;
  int32_t max_iter, refine_steps; const int32_t* budget;
  Fmt main_fmt;                          // a 2-byte format; the refinement's is FP16 in three terms
  bool exact_xq;                         // some submatrix of the work sums X Q exactly (exact_xq)
  int32_t* next; int32_t* err;           // work counter (reset by the launch), timeout flag
  double* Dc; double* tS; double* tH; int32_t* iters; int32_t* status; int32_t* rsteps; int32_t* nbelow;
  uint64_t wait_ns;                      // limit of a wait of one role on another, 0: 2 s
  const float* cond; float cond_max; int32_t ill_max_n;   // as for k_ns_tc
};
// Every status of the work has been set to kSubTimeout before.
nolsm_status launch_ns_res(const ResSolve& a, int sms, cudaStream_t st);

// a2-a3 the same way, every submatrix of at most kResMaxN rows (see launch_ns_inverse for the fields): prep_out[J] =
// kSubOk, kSubRefine, or kSubAgain where k_ns_tc has to take the submatrix (more than two steps); *again counts those, again_list names them.
constexpr int32_t kSubAgain = 66;
struct InvSolve {
  const int32_t* order; int32_t count;
  const int32_t* sub_n; const int64_t* a_off;
  const double* ws; int64_t a_base, chunk_n2;
  float* Aout; float* Xout;
  int32_t* prep_out;
  float tol_inv; int32_t max_inv;
  int32_t* next; int32_t* err; int32_t* again; int32_t* again_list;
  double* flops;
  uint64_t wait_ns;
};
nolsm_status launch_inv_res(const InvSolve& a, int sms, cudaStream_t st);
bool inv_res_ready();

}  // namespace nolsm
