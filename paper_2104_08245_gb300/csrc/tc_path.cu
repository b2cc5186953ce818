// a4-a7 on the 5th-generation tensor cores (tcgen05) for the low-precision modes.
//
// Newton-Schulz sign iteration (Eq. NS1): X_{k+1} = 1/2 X_k (3I - X_k^2), two products per step:
//   GEMM0: Y = X X      -> epilogue writes T = 3I - Y and sums the defect ||I - X^2||_F^2
//   GEMM1: Z = X T      -> epilogue writes X_{k+1} = Z / 2 (the last one feeds the centre columns)
// Each product is either one tensor-core product of the rounded operands (BF16 or FP16) or the
// three-term split hi*hi + hi*lo + lo*hi with x = hi + lo (hi = round(x), lo = round(x - hi)),
// accumulated in FP32 in tensor memory.
//
// Submatrices of more than 192 rows (and all of them in E4M3) run here; the others keep their operands on the SM
// (res_path.cu). One persistent CTA per SM; a group of 1, 2, 4 or 8 CTAs (group_size) shares two submatrices in flight
// ("slots", taken largest first from a work counter) and deals their products' tiles, and the rows of a start or a
// finish, among its CTAs. While the tensor cores run a product of one slot, the epilogues drain, round and store the
// previous product of the other, and the group meets. Operands live in per-slot scratch in global memory as 2-byte
// planes [X0 hi, X0 lo, X1 hi, X1 lo, T hi, T lo], each R x LD (R = n rounded up to 128 rows, LD = n rounded up to 64
// columns, zero padded). What bounds it: with two submatrices on every SM the planes (4 MB a submatrix at n = 650) miss
// L2, and each product's operands come from DRAM several times over; the groups keep the planes in flight within L2
// (512 submatrices of n = 600-713: 233 GB through DRAM before, 41 GB since; 40 -> 12.4 ms, 13.2 with the compensated
// X Q of large submatrices, exact_xq). What is left at 2.4 times
// the MMAs' own time is the phases' latency (first slices, last tile's epilogue, the group's meeting) and, below
// n = 256, the start and finish of a submatrix.
// Output tiles are 128 rows x up to 256 columns; the K dimension streams in slices of 32 through a four-stage TMA
// pipeline; the epilogue writes the rounded planes back with TMA stores.
// Warp roles: warp 0 (one thread) schedules the phases of the slots, decides convergence and publishes one descriptor
// per phase in a small ring; warp 2 issues the loads and warp 1 tcgen05.mma, both converged with one elected lane;
// warps 4-11 (two groups of four, even and odd 32-column chunks) drain the double-buffered TMEM accumulators
// (2 x 256 columns) and start and finish the submatrices. All waits are bounded by the global timer; a wait that runs
// out marks the submatrices in flight as timed out.
//
// The same kernel, instantiated in its second mode, prepares A_J = T_J(S)^-1 T_J(H0) on the tensor cores
// by the coupled Newton-Schulz iteration for the inverse square root (Eqs. inv1-inv3): with Y_0 = T_J(S)/c
// and Z_0 = I, V_k = Z_k Y_k, Y_{k+1} = 1/2 Y_k (3I - V_k), Z_{k+1} = 1/2 (3I - V_k) Z_k, Z_k tends to
// (T_J(S)/c)^-1/2, so T_J(S)^-1 = Z^2 / c (Eq. inv3) and A_J = (Z^2 / c) T_J(H0). Every product is a
// three-term FP16 split. The step whose V_k has ||I - V_k||_F / sqrt(n) <= tol_inv is the last (its Y
// update is skipped, Z alone is needed); c = Tr T_J(S) / n, the mean eigenvalue, so that the eigenvalues
// of Y_0 average 1 and lie in (0, 2), where the iteration converges, unless the largest eigenvalue of
// T_J(S) exceeds twice the mean (then the defect grows, and the submatrix, like any whose iteration does
// not reach tol_inv within max_inv steps, is flagged for the FP64 preparation). X = T_J(S)^-1 is also
// written in FP32 for the refinement of the centre columns of T_J(S)^-1.
// Submatrices of up to 192 rows come here only for what k_inv_res leaves (more than two steps).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <mutex>
#include <type_traits>

#include "nolsm_internal.cuh"
#include "prep.cuh"
#include "res_path.cuh"
#include "tc_path.cuh"
#include "tc_split.cuh"
#include "tcgen05.cuh"
#include "tmap.cuh"

namespace nolsm {

namespace {

constexpr int kStages = 4;                        // K slices of 32 in flight
constexpr uint32_t kABytes = 128 * 32 * 2;        // one A plane slice: 128 rows x 32 K
constexpr uint32_t kBBlock = 32 * 64 * 2;         // one B plane slice of a column block: 32 K x 64 columns
constexpr int kMaxEpiWarps = 12;

// The two launch shapes. The epilogue warps from warp 4 on come in groups of four (each group covers the 128 TMEM lanes)
// and deal a tile's 32-column chunks round robin. Shape 0: 384 threads, two groups, tiles of 128 x up to 256 columns.
// Shape 1: 512 threads, three groups, tiles of 128 x up to 192 columns (so that the twelve 4 KB staging buffers fit
// beside the operand stages). Which one runs a bucket of submatrices is measured (bucket_shape).
template <int kShape>
struct Shape {
  static constexpr int kThreads = kShape == 0 ? 384 : 512;
  static constexpr int kEpiWarps = kThreads / 32 - 4;
  static constexpr int kEpiThreads = 32 * kEpiWarps;
  static constexpr int kGroups = kEpiWarps / 4;
  static constexpr int kTileN = kShape == 0 ? 256 : 192;       // N of one MMA
  static constexpr uint32_t kStageBytes = 2 * kABytes + 2 * kBBlock * (kTileN / 64);   // hi and lo
  static constexpr uint32_t kStgTotal = 4096 * kEpiWarps;    // a 4 KB hi/lo staging buffer per epilogue warp
  static constexpr int kSmemBytes = kStages * kStageBytes + kStgTotal + 1024;
  // registers per thread: of the launch, of the first warpgroup, of the epilogue
  static constexpr int kRegsLaunch = kShape == 0 ? 168 : 128, kRegsLow = kShape == 0 ? 72 : 56, kRegsEpi = kShape == 0 ? 216 : 152;
};
static_assert(Shape<1>::kEpiWarps <= kMaxEpiWarps && Shape<0>::kEpiWarps <= kMaxEpiWarps, "epilogue warps");
static_assert(Shape<0>::kSmemBytes <= 227 * 1024 && Shape<1>::kSmemBytes <= 227 * 1024, "shared memory");
// The first warpgroup (TMA and MMA threads) releases registers down to kRegsLow and the epilogue warpgroups take
// kRegsEpi, within what the launch gives the block, so the increase never waits on registers that do not exist.
template <int kShape>
constexpr bool split_fits = 128 * Shape<kShape>::kRegsLow + Shape<kShape>::kEpiThreads * Shape<kShape>::kRegsEpi <=
                            Shape<kShape>::kThreads * Shape<kShape>::kRegsLaunch;
static_assert(split_fits<0> && split_fits<1>, "register split above the launch");
constexpr int kPlanes = 6;
constexpr uint64_t kWaitNs = 2000000000ull;        // default limit per wait (2 s); one product takes < 1 ms

// E4M3 operands carry a fixed power-of-two scale: the symmetric iterates have |x_ij| <= rho <= 1.7 (the
// scale guard), so x * 2^7 stays below 218 of E4M3's 448 and values down to 2^-16 keep a subnormal; a
// product of two scaled operands is scaled back by 2^-14.
constexpr float kF8Up = 128.0f;
constexpr float kF8Down = 1.0f / 16384.0f;
constexpr float kF8Switch = 0.1f;   // defect at which the E4M3 phase hands over to the refinement format
// K extent of an E4M3 operand row: whole 128-byte slices
__host__ __device__ inline int k8_extent(int n64) { return (n64 + 127) & ~127; }

struct TcArgs {
  int32_t j0, j1;
  const int32_t* order;       // submatrices of [j0, j1), largest first
  const int32_t* sub_n; const int32_t* nbf;
  const int64_t* a_off; const int64_t* c_off;
  const float* A;             // FP32 A_J
  const double* Q; const double* Sc; const double* Hc; const double* lam;
  const double* lam_g;        // Gershgorin interval (the scale never drops below its alpha / 1.7)
  const int32_t* prep_status;
  double mu;
  float tol_ns, tol_accept;
  int32_t max_iter, refine_steps;
  const int32_t* budget;      // per-submatrix step cap (nullable)
  Fmt main_fmt, refine_fmt;
  uint16_t* planes;           // [slots*6][R][LD]
  int32_t R, LD;
  int32_t* next;              // work counter
  int32_t* err;               // global error flag (timeouts)
  double* Dc; double* tS; double* tH; int32_t* iters; int32_t* status; int32_t* rsteps;
  int32_t* nbelow;            // eigenvalues below mu, (n - Tr X) / 2 (nullable)
  uint64_t wait_ns;           // limit of every wait on another role (the teardown's own waits: 50 ms)
  const float* cond;          // preparation's cond(T_J(S)) estimate (nullable): above cond_max the submatrix
  float cond_max;             // is left to the FP64 path (its status stays as it is) when it has at most
  int32_t ill_max_n;          // ill_max_n rows (what the FP64 preparation takes)
  int32_t above_n;            // sign mode: submatrices of at most this many rows are passed over (k_ns_res takes them)
  // inverse-square-root mode: the chunk's gathered T_J(S), T_J(H0) (FP64, at a_off[J] - a_base and
  // chunk_n2 further), the outputs and the iteration's stopping rule
  const double* ws;
  int64_t a_base, chunk_n2;
  float* Aout;                // FP32 A_J at a_off[J]; null: T_J(S)^-1 alone
  float* Xout;                // FP32 T_J(S)^-1 at a_off[J] - a_base
  int32_t* prep_out;          // kSubOk, or kSubRefine when the iteration failed (FP64 preparation next)
  float tol_inv;
  int32_t max_inv;
  double* flops;              // [2]: 2 n^3 per product (method count) and the split's issued flops, summed
  int32_t group;              // CTAs that share a submatrix (the grid is a multiple of it)
  struct GroupSlot* groups;   // [grid / group * kSlots], zeroed before the launch
};

// Views of the operand planes: A slices of 128 rows x 32 K, B slices of 32 K x 64 or 128 columns, of one plane or of hi
// and lo; the epilogue's stores; E4M3's slices of 128 bytes.
struct TcMaps { CUtensorMap A, A2, B, B2, Bx2, B2x2, S, S2, A8, B8; };

// Epilogue of a product: what is done with the accumulator P
enum : int {
  kEpiT = 0,      // T = 3I - P to the planes, and the defect ||I - P||_F^2
  kEpiScale = 1,  // scale * P to the planes
  kEpiX = 2,      // scale * P to the planes and in FP32 to Xout
  kEpiA = 3       // P in FP32 to Aout (no planes)
};
constexpr int kPlanesInv = 10;   // inverse mode: plane pairs Y (then T_J(H0)), Z, T (then X), Y', Z'

constexpr int kSlots = 2;   // submatrices in flight per CTA (their products interleave)
constexpr int kRing = 4;    // product descriptors between the scheduler and the MMA / epilogue warps

// The CTAs of a group run the same sequence of phases in each of the group's slots: a phase (a fetch, a turn, a fill or
// a product) ends when every CTA of the group has arrived on count, and then every scheduler derives the next one from
// the same numbers. Per (group, slot) in global memory:
constexpr int kMaxGroup = 16;
struct alignas(128) GroupSlot {
  uint32_t count;                // arrivals so far
  int32_t next;                  // fetch: the next submatrix, or -1
  float part[2][kMaxGroup];      // the CTAs' shares of the defect, by the phase's parity
  double tr[3][kMaxGroup];       // turn: their shares of the traces
};

// What a descriptor asks for
enum : int {
  kOpFetch = 0,   // (no descriptor) the first CTA of the group draws the next submatrix
  kOpTurn = 1,    // finish the slot's submatrix and start the next
  kOpFill = 2,    // inverse mode: T_J(H0) into Y's pair
  kOpProd = 3     // a product
};

// Iteration state of one in-flight submatrix: the scheduler's.
struct SlotState {
  int job, fin;                  // submatrix index, -1 for none; the one that a turn finishes
  int next;                      // fetch: the next one, as drawn by this CTA
  int op, rot;                   // phase under way; the CTA of tile 0 of the next product
  uint32_t seq, epar;            // phases begun; parity of this CTA's next epi_done
  bool alive, local;             // not retired; this CTA's epilogue is still to report
  int n, n64, R, nrb, ncb;       // dimension and tiling
  int kind;                      // next product: 0 (X X) or 1 (X T)
  int cur;                       // which X plane pair holds the current iterate
  int phase, refine_left, steps, rsteps, status, last;
  float dprev;                   // defect of the previous step (E4M3 stagnation test)
  Fmt fcur, fnxt;
  int yc, zc;                    // inverse mode: plane pairs of the current Y and Z
  int zdone;                     // inverse mode: this step's Z update was made at the start (step 0)
  float cinv;                    // inverse mode: 1 / c
  float zs;                      // inverse mode: Z = zs x (Z's planes); 1/2 until the first Z update, whose
                                 // planes hold T_0 = 2 Z_1
};

// One product as scheduled by the producer: read in order by the MMA issuer and the epilogue.
struct Desc {
  int term;                      // 1: no more products, exit
  int op, slot, kind, par;       // kOp*; parity of the phase
  int job, fin;                  // the submatrix (turn: to start), the one that a turn finishes
  int t0;                        // this CTA's first tile (then every group-th)
  int fill;                      // inverse mode: plane that T_J(H0) goes to at the product's end, -1: none
  Fmt f, fo;                     // format of the operands; of the operand the epilogue writes
  int n, n64, nrb, ncb;
  int za, zb, zo;                // plane indices (hi planes) of A, B and the output
  int epi;                       // kEpi*
  float scale;                   // kEpiScale, kEpiX
  float pscale;                  // kEpiT: the product is pscale P
};

struct Shared {
  uint64_t full[kStages], empty[kStages], accf[2], acce[2], idle;
  uint64_t epi_done[kSlots], desc_full[kRing], desc_free[kRing];
  uint32_t tmem;
  int err;
  SlotState slot[kSlots];
  float part[kSlots];            // a group of one: its GroupSlot's part and tr
  double tr[kSlots][3];
  float cinv[kSlots];            // inverse mode: 1 / c of the submatrix just started
  Desc ring[kRing];
  float red[2][kMaxEpiWarps];    // defect partial sums, by product parity
  double dred[3][kMaxEpiWarps];
};

// Eight rows of X a warp (2-byte hi and, with kLo, lo planes, columns k0 .. k0 + kn - 1, kn a multiple of 32) times 8
// columns of Q in FP32 (staged from row k0 on): four lanes a row, each 8 adjacent columns of every 32, so that a load
// reads 64 consecutive bytes of a row. FP32 sums of 8 products, each added to s + e with TwoSum, or with kExact (exact_xq)
// every product with its own rounding error; then the four lanes' sums together, the same in each of them.
__device__ __forceinline__ int qs_at(int k) { return 8 * k + 4 * (k >> 3); }   // four lanes' rows in different banks
template <int kFmt, bool kLo, bool kExact>
__device__ __forceinline__ void xq_rows(const uint16_t* __restrict__ xh, const uint16_t* __restrict__ xl, int kn,
                                        const float* __restrict__ Qs, int part, uint64_t (&s)[4], uint64_t (&e)[4]) {
  const uint64_t neg = pair2(-1.0f, -1.0f);
#pragma unroll
  for (int c = 0; c < 4; ++c) s[c] = e[c] = 0;
  auto add = [&](int c, uint64_t p) {   // TwoSum in pairs
    const uint64_t t = add2(s[c], p), z = fma2(s[c], neg, t);
    e[c] = add2(e[c], add2(fma2(fma2(z, neg, t), neg, s[c]), fma2(z, neg, p)));
    s[c] = t;
  };
  auto load = [&](int k, uint4& h, uint4& l) {   // (past the end the last piece again)
    k = min(k, kn - 32 + 8 * part);
    h = *reinterpret_cast<const uint4*>(xh + k);
    l = kLo ? *reinterpret_cast<const uint4*>(xl + k) : make_uint4(0, 0, 0, 0);
  };
  auto piece = [&](int k, const uint4& h4, const uint4& l4) {   // eight columns
    uint64_t p[4] = {0, 0, 0, 0};
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t h = u < 2 ? h4.x : u < 4 ? h4.y : u < 6 ? h4.z : h4.w;
      const uint32_t l = u < 2 ? l4.x : u < 4 ? l4.y : u < 6 ? l4.z : l4.w;
      float x = from_bits((uint16_t)(h >> (16 * (u & 1))), kFmt);
      if (kLo) x += from_bits((uint16_t)(l >> (16 * (u & 1))), kFmt);
      const ulonglong2 qa = *reinterpret_cast<const ulonglong2*>(Qs + qs_at(k) + 8 * u);
      const ulonglong2 qb = *reinterpret_cast<const ulonglong2*>(Qs + qs_at(k) + 8 * u + 4);
      const uint64_t xx = pair2(x, x), xn = pair2(-x, -x), q[4] = {qa.x, qa.y, qb.x, qb.y};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (kExact) add_product2(s[c], e[c], xx, xn, q[c]);
        else p[c] = fma2(xx, q[c], p[c]);
      }
    }
#pragma unroll
    for (int c = 0; c < 4 && !kExact; ++c) add(c, p[c]);
  };
  if constexpr (kExact) {   // 320 packed operations a piece: the next one's loads are in flight meanwhile (13.65 -> 13.2 ms)
    uint4 h, l, hn, ln;
    load(8 * part, h, l);
#pragma unroll 1
    for (int k = 8 * part; k < kn; k += 32) {
      load(k + 32, hn, ln);
      piece(k, h, l);
      h = hn;
      l = ln;
    }
  } else {
#pragma unroll 1
    for (int k0 = 8 * part; k0 < kn; k0 += 128) {
      uint4 hv[4], lv[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) load(k0 + 32 * t, hv[t], lv[t]);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (k0 + 32 * t >= kn) break;
        piece(k0 + 32 * t, hv[t], lv[t]);
      }
    }
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const uint64_t so = __shfl_xor_sync(0xffffffffu, (unsigned long long)s[c], o);
      const uint64_t eo = __shfl_xor_sync(0xffffffffu, (unsigned long long)e[c], o);
      add(c, so);
      e[c] = add2(e[c], eo);
    }
  }
}

// named barrier 3 for the N epilogue threads
template <int N>
__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 3, %0;" ::"n"(N) : "memory"); }
// barrier 3 with an OR over the N epilogue threads' predicates
template <int N>
__device__ __forceinline__ bool epi_bar_or(bool p) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred P, Q;\n\tsetp.ne.u32 P, %1, 0;\n\tbar.red.or.pred Q, 3, %2, P;\n\tselp.u32 %0, 1, 0, Q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)p), "n"(N)
      : "memory");
  return r != 0;
}

// kMode 0: the sign iteration (a4-a7); kMode 1: the inverse square root of T_J(S) and A_J (a2-a3); kShape:
// the launch shape (Shape)
template <int kMode, int kShape>
__global__ void __launch_bounds__(Shape<kShape>::kThreads, 1)
    k_ns_tc(const __grid_constant__ TcMaps maps, TcArgs g) {
  constexpr int kPps = kMode == 0 ? kPlanes : kPlanesInv;   // planes per slot
  constexpr int kEpiWarps = Shape<kShape>::kEpiWarps, kEpiThreads = Shape<kShape>::kEpiThreads;
  constexpr int kGroups = Shape<kShape>::kGroups, kTileN = Shape<kShape>::kTileN;
  constexpr uint32_t kStageBytes = Shape<kShape>::kStageBytes;
  constexpr uint32_t kStgTotal = Shape<kShape>::kStgTotal;
  extern __shared__ uint8_t smraw[];
  uint8_t* stage_mem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  __shared__ Shared sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      tc::mbar_init(&sh.full[s], 1);
      tc::mbar_init(&sh.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&sh.accf[b], 1);
      tc::mbar_init(&sh.acce[b], kEpiThreads);
    }
    for (int s = 0; s < kSlots; ++s) tc::mbar_init(&sh.epi_done[s], kEpiThreads);
    for (int r = 0; r < kRing; ++r) {
      tc::mbar_init(&sh.desc_full[r], 1);
      tc::mbar_init(&sh.desc_free[r], 3);   // loader, MMA issuer, epilogue
    }
    tc::mbar_init(&sh.idle, 1);
    tc::fence_mbar_init();
    sh.err = 0;
  }
  if (warp == 0) {
    tc::tmem_alloc(&sh.tmem, 512);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = sh.tmem;
  const size_t plane_elems = (size_t)g.R * g.LD;
  uint8_t* const stg = stage_mem + kStages * kStageBytes;   // epilogue staging: 4 KB per epilogue warp
  // the group's CTAs share its slots: rank 0 draws the submatrices, tiles and rows are dealt in turn
  const int G = g.group, gid = blockIdx.x / G, rank = blockIdx.x - gid * G;
  GroupSlot* const gs = g.groups + (size_t)gid * kSlots;
  const int sub0 = gid * kSlots;                             // scratch sub-slot of the group's slot 0
  uint32_t loads = 0;                                        // loader: K slices armed so far

  if (warp < 4) {
  tc::setmaxnreg_dec<Shape<kShape>::kRegsLow>();   // the TMA / MMA warpgroup gives registers up
  if (warp == 0 && lane == 0) {
    // ------------------------------------------------ producer: schedules the phases of the slots
    // a slot's next phase is issued once the previous one has ended in every CTA of the group; the live slots are
    // polled round robin from the one after the last pick, and the first that is ready goes (no slot waits behind
    // another's epilogue)
    auto fetch = [&]() -> int {
      for (;;) {
        const int k = atomicAdd(g.next, 1);
        if (k >= g.j1 - g.j0 || sh.err) return -1;
        const int J = g.order[k];
        if constexpr (kMode == 1) return J;
        if (g.sub_n[J] <= g.above_n) continue;
        if (g.cond && g.prep_status[J] == kSubOk && g.cond[J] > g.cond_max && g.sub_n[J] <= g.ill_max_n) continue;
        if (g.prep_status[J] == kSubOk) return J;
        g.status[J] = g.prep_status[J];
        g.iters[J] = 0;
        g.rsteps[J] = 0;
        g.tS[J] = 0.0;
        g.tH[J] = 0.0;
      }
    };
    auto begin_fetch = [&](int c) {
      SlotState& st = sh.slot[c];
      st.op = kOpFetch;
      ++st.seq;
      st.local = false;
      if (rank == 0) {
        st.next = fetch();
        if (G > 1) __stcg(&gs[c].next, st.next);
      }
      if (G > 1) tc::red_release_gpu(&gs[c].count, 1u);
    };
    auto ready = [&](int c) -> bool {
      SlotState& st = sh.slot[c];
      if (st.local) {
        if (!tc::mbar_test_wait(&sh.epi_done[c], st.epar)) return false;
        st.epar ^= 1;
        st.local = false;
      }
      return G == 1 || tc::reached_gpu(&gs[c].count, (uint32_t)G * st.seq);
    };
    auto defect = [&](int c) -> float {   // the phase's sum over the group, in an order that the slot does not change
      if (G == 1) return sh.part[c];
      float d = 0.0f;
      for (int r = 0; r < G; ++r) d += __ldcg(&gs[c].part[sh.slot[c].seq & 1][r]);
      return d;
    };
    // the phase under way in slot c has ended: its results, and the next phase's descriptor; false when that phase
    // needs none (a fetch) or the slot has retired
    auto advance = [&](int c, Desc& d) -> bool {
      SlotState& st = sh.slot[c];
      const int zb = (sub0 + c) * kPps;
      d.term = 0;
      d.slot = c;
      d.fill = -1;
      bool fill = false;
      if (st.op == kOpFetch) {
        const int J = rank == 0 ? st.next : __ldcg(&gs[c].next);
        if (J < 0 && st.job < 0) {
          st.alive = false;
          return false;
        }
        d.op = st.op = kOpTurn;
        d.fin = st.fin = kMode == 0 ? st.job : -1;
        d.n = st.n; d.n64 = st.n64;
        d.za = zb + 2 * st.cur;
        d.f = st.fcur;
        d.job = st.job = J;
        // X_0 goes into the other pair: other CTAs of the group may still read the finished X. (E4M3 runs in groups of one.)
        if (g.main_fmt.fmt == FMT_E4M3) st.cur = 0;
        else st.cur ^= 1;
        d.zo = zb + 2 * st.cur;
        st.rot = c * (G / 2);
      } else {
        if (st.op == kOpTurn) {
          if (kMode == 0 && st.fin >= 0) {
            if (rank == 0) {
              double t[3] = {0.0, 0.0, 0.0};
              for (int r = 0; r < G; ++r)
                for (int k = 0; k < 3; ++k) t[k] += G == 1 ? sh.tr[c][k] : __ldcg(&gs[c].tr[k][r]);
              const int J = st.fin;
              if (g.nbelow) g.nbelow[J] = (int32_t)lrint(0.5 * (st.n - t[2]));
              int stt = st.status;
              if (stt == kSubOk && !(isfinite(t[0]) && isfinite(t[1]))) stt = kSubNonFinite;
              g.tS[J] = t[0];
              g.tH[J] = t[1];
              g.iters[J] = st.steps;
              g.rsteps[J] = st.rsteps;
              g.status[J] = stt;
            }
            st.fin = -1;
          }
          if (st.job < 0) {
            st.alive = false;
            return false;
          }
          st.n = g.sub_n[st.job];
          st.n64 = (st.n + 63) & ~63;
          st.R = (st.n + 127) & ~127;
          st.nrb = st.R / 128; st.ncb = (st.n64 + kTileN - 1) / kTileN;
          st.dprev = INFINITY;
          st.last = 0;
          st.rsteps = 0;
          if constexpr (kMode == 0) {
            st.kind = 0;
            st.phase = 0; st.refine_left = g.refine_steps; st.steps = 0;
            st.status = kSubNotConv;
            st.fcur = g.main_fmt; st.fnxt = g.main_fmt;
          } else {
            st.yc = 0; st.zc = 1; st.cinv = sh.cinv[c]; st.zs = 0.5f;
            st.steps = 1; st.status = kSubOk;
            st.fcur = Fmt{FMT_F16, 3}; st.fnxt = st.fcur;
            const float d0 = sqrtf(defect(c) / (float)st.n);   // not finite when c was not positive
            st.zdone = 1;
            st.last = d0 <= g.tol_inv ? 1 : 0;
            st.kind = st.last ? 3 : 1;     // step 0 the last: X = Z_1 Z_1 / c next; else Y_1 = Y_0 T_0 / 2
            fill = st.last && g.Aout;      // Y_0 is not needed: T_J(H0) takes its pair (else after the last Z update)
            if (!isfinite(d0)) {           // the FP64 preparation takes it
              st.status = kSubRefine;
              st.kind = 5;
            }
          }
        } else if (st.op == kOpProd) {
          if constexpr (kMode == 1) {
            switch (st.kind) {
              case 0: {
                const float dd = sqrtf(defect(c) / (float)st.n);
                st.steps += 1;
                if (!isfinite(dd) || (dd > g.tol_inv && st.steps >= g.max_inv)) {
                  st.status = kSubRefine;   // diverged or too slow: the FP64 preparation takes it
                  st.last = 1;
                } else if (dd <= g.tol_inv) {
                  st.last = 1;                // this step's Z update is the last product of the iteration
                }
                st.kind = st.last ? 2 : 1;
                break;
              }
              case 1:   // after Y's update: Z's, unless the step's Z update was made at the start
                if (st.ncb != 1) st.yc = st.yc == 0 ? 3 : 0;
                st.kind = st.zdone ? 0 : 2;
                st.zdone = 0;
                break;
              case 2: st.zc = st.zc == 1 ? 4 : 1; st.zs = 1.0f; st.kind = st.last ? 3 : 0; break;
              case 3: st.kind = g.Aout ? 4 : 5; break;
              default: st.kind = 5; break;
            }
          } else if (st.kind == 0) {
            // defect of X_step and the decision about the following steps
            const float dd = sqrtf(defect(c) / (float)st.n);
            const int steps = st.steps + 1;
            if (st.phase == 1) st.rsteps += 1;   // this step ran in the refinement format
            int last_ = 0, status = kSubNotConv;
            Fmt nxt = st.fcur;
            if (!isfinite(dd)) {
              last_ = 1;
              status = kSubNonFinite;
            } else if (st.phase == 0) {
              // E4M3 iterates carry a rounding error of up to 2^-4 relative, which holds the defect at a floor
              // near 0.05, well above tol_ns: their phase ends at twice that floor, or when the defect has
              // stopped falling (below 0.25, where the exact iteration would at least halve it every step)
              const bool f8_end = st.fcur.fmt == FMT_E4M3 && (dd <= kF8Switch || (dd < 0.25f && dd > 0.5f * st.dprev));
              if (dd <= g.tol_ns || f8_end) {
                if (g.refine_steps == 0) {
                  last_ = 1;
                  status = dd <= g.tol_accept ? kSubOk : kSubNotConv;
                } else {
                  st.phase = 1;
                  st.refine_left = g.refine_steps;
                  nxt = g.refine_fmt;
                }
              }
            } else if (--st.refine_left <= 0) {
              if (dd <= g.tol_accept) {
                last_ = 1;
                status = kSubOk;
              } else if (dd < st.dprev) {
                st.refine_left = 1;   // still converging: one more step (bounded by the step cap below)
              } else {
                last_ = 1;
                status = kSubNotConv;
              }
            }
            const int cap = g.budget ? min(g.max_iter, g.budget[st.job]) : g.max_iter;
            if (!last_ && steps >= cap) {
              last_ = 1;
              status = kSubNotConv;
            }
            st.dprev = dd;
            st.steps = steps;
            st.last = last_;
            st.status = status;
            st.fnxt = nxt;
            st.kind = 1;
          } else {
            // after X T: X_{k+1} is the current X (ping-pong unless written in place), in the next format
            if (st.ncb != 1) st.cur ^= 1;
            st.fcur = st.fnxt;
            st.kind = st.last ? 5 : 0;
          }
        }
        if (st.kind == 5) {   // the submatrix is done
          if (kMode == 1) {
            if (rank == 0) {
              g.prep_out[st.job] = st.status;
              const double n3 = (double)st.n * st.n * st.n;
              // step 0 needs one product (Y_1), every further step three but the last two (no Y update); then X, A
              const double prods = 3.0 * st.steps - (g.Aout ? 1.0 : 2.0);
              atomicAdd(&g.flops[0], 2.0 * n3 * prods);
              atomicAdd(&g.flops[1], 6.0 * n3 * prods);
            }
            st.job = -1;
          }
          begin_fetch(c);
          return false;
        }
        d.job = st.job;
        d.n = st.n; d.n64 = st.n64; d.nrb = st.nrb; d.ncb = st.ncb;
        d.f = st.fcur;
        d.kind = st.kind;
        if (fill) {
          d.op = st.op = kOpFill;
          d.fill = zb;
        } else {
          d.op = st.op = kOpProd;
          d.t0 = (rank - st.rot + G) % G;
          st.rot = (st.rot + st.nrb * st.ncb) % G;
          d.pscale = 1.0f;
          if constexpr (kMode == 0) {   // the epilogue derives epi and scale from the kind
            d.fo = st.kind == 0 ? st.fcur : st.fnxt;
            d.za = zb + 2 * st.cur;
            d.zb = st.kind == 0 ? d.za : zb + 4;
            // X_{k+1} overwrites X_k when one column tile covers the matrix: row block mb of X_k is read
            // (as the A operand) only by tile (mb, 0), whose loads have completed before its epilogue writes
            d.zo = st.kind == 0 ? zb + 4 : (st.ncb == 1 ? d.za : zb + 2 * (st.cur ^ 1));
          } else {
            // pairs: Y in 0 (updated in place when one column tile covers the matrix, else ping-pong with 3),
            // Z in 1 or 4 (ping-pong: every row tile of T Z reads all of Z; until the first Z update the pair
            // holds T_0 = 2 Z_1, hence the factor zs), T and then X in 2; T_J(H0) goes into Y's pair once Y is
            // no longer needed
            d.scale = 0.5f;
            d.fo = st.fcur;
            switch (st.kind) {
              case 0:  // V = Z Y -> T = 3I - V
                d.za = zb + 2 * st.zc; d.zb = zb + 2 * st.yc; d.zo = zb + 4; d.epi = kEpiT; d.pscale = st.zs; break;
              case 1:  // Y' = 1/2 Y T (row block mb of Y is read only by tile (mb, 0), as for X X T); at step 0
                       // T_0 is in Z's pair
                d.za = zb + 2 * st.yc; d.zb = st.zdone ? zb + 2 * st.zc : zb + 4;
                d.zo = st.ncb == 1 ? d.za : zb + 2 * (st.yc == 0 ? 3 : 0);
                d.epi = kEpiScale; break;
              case 2:  // Z' = 1/2 T Z; after the last one Y (last read by this step's V = Z Y) makes room for T_J(H0)
                d.za = zb + 4; d.zb = zb + 2 * st.zc; d.zo = zb + 2 * (st.zc == 1 ? 4 : 1); d.epi = kEpiScale;
                d.scale = 0.5f * st.zs;
                if (st.last && g.Aout) d.fill = zb + 2 * st.yc;
                break;
              case 3:  // X = Z Z / c = T_J(S)^-1
                d.za = zb + 2 * st.zc; d.zb = d.za; d.zo = zb + 4; d.epi = kEpiX; d.scale = st.cinv * st.zs * st.zs;
                break;
              default:  // A_J = X T_J(H0)
                d.za = zb + 4; d.zb = zb + 2 * st.yc; d.zo = zb + 4; d.epi = kEpiA; break;
            }
          }
        }
      }
      ++st.seq;
      st.local = true;
      d.par = st.seq & 1;
      return true;
    };

    for (int c = 0; c < kSlots; ++c) {
      sh.slot[c].job = sh.slot[c].fin = -1;
      sh.slot[c].alive = true;
      sh.slot[c].seq = sh.slot[c].epar = 0;
      sh.slot[c].cur = 0;
      begin_fetch(c);
    }
    uint32_t i = 0;
    int s = 0;
    for (;;) {
      int pick = -1;
      const uint64_t deadline = tc::globaltimer() + 4 * g.wait_ns;
      for (;;) {
        bool any = false;
        for (int t = 0; t < kSlots && pick < 0; ++t) {
          const int c = (s + t) % kSlots;
          if (!sh.slot[c].alive) continue;
          any = true;
          if (ready(c)) pick = c;
        }
        if (pick >= 0 || !any || sh.err) break;
        if (tc::globaltimer() > deadline) {
          sh.err = 1;
          break;
        }
      }
      Desc d;
      d.term = 1;
      if (pick >= 0) {
        s = (pick + 1) % kSlots;
        if (!advance(pick, d)) continue;
      }
      if (i >= kRing && !tc::mbar_wait_ns(&sh.desc_free[i % kRing], ((i / kRing) & 1) ^ 1, 8 * g.wait_ns)) {
        sh.err = 1;
        break;
      }
      sh.ring[i % kRing] = d;
      tc::mbar_arrive(&sh.desc_full[i % kRing]);
      ++i;
      if (d.term) break;
    }
  } else if (warp == 2) {
    // ------------------------------------------------ loader: the K slices of the products, in the scheduler's order.
    // (The whole warp runs the loop and one elected lane issues: from one lane's branch a TMA instruction took some 140
    // cycles and an MMA 85, together more than the MMAs of a slice.)
    auto wait = [&](uint64_t* b, uint32_t parity, int more) {
      return (bool)__all_sync(0xffffffffu, tc::mbar_wait_ns(b, parity, more * g.wait_ns));
    };
    bool ok = true;
    for (uint32_t i = 0; ok && !sh.err; ++i) {
      if (!(ok = wait(&sh.desc_full[i % kRing], (i / kRing) & 1, 8))) break;
      const Desc& d = sh.ring[i % kRing];
      if (d.term) break;
      if (d.op == kOpProd) {
        tc::fence_proxy_async_global();   // the epilogues' plane writes, before TMA reads them
        const bool f8 = d.f.fmt == FMT_E4M3, two = d.f.terms > 1;
        const int nks = f8 ? k8_extent(d.n64) / 128 : (d.n + 31) / 32, tiles = d.nrb * d.ncb, ncb = d.ncb, za = d.za, zb = d.zb;
        const CUtensorMap* const ma = two ? &maps.A2 : &maps.A;
        const CUtensorMap* const mb1 = two ? &maps.B2 : &maps.B;
        const CUtensorMap* const mb2 = two ? &maps.B2x2 : &maps.Bx2;
        const uint32_t aoff = two ? 2 * kABytes : kABytes, boff = two ? 2 * kBBlock : kBBlock;
        for (int ti = d.t0; ti < tiles && ok; ti += G) {
          const int mb = ti / ncb, cb = ti - mb * ncb;
          const int nb = min(kTileN, d.n64 - kTileN * cb) / 64, c0 = kTileN / 64 * cb;
          // E4M3: both operands K-major (the symmetric iterate is its own transpose), 128-byte K slices; the B box is
          // always kTileN rows (rows past R are zero-filled by the copy)
          const uint32_t bytes = f8 ? 128 * 128 + (uint32_t)kTileN * 128u : aoff + nb * boff;
          for (int ks = 0; ks < nks; ++ks, ++loads) {
            const uint32_t st = loads % kStages;
            if (!(ok = wait(&sh.empty[st], ((loads / kStages) & 1) ^ 1, 1))) break;
            if (tc::elect_one()) {
              uint8_t* const sm = stage_mem + st * kStageBytes;
              uint64_t* const bar = &sh.full[st];
              tc::mbar_arrive_expect_tx(bar, bytes);
              if (f8) {
                tc::tma_load_3d(sm, &maps.A8, bar, 128 * ks, 128 * mb, za);
                tc::tma_load_3d(sm + 128 * 128, &maps.B8, bar, 128 * ks, kTileN * cb, zb);
              } else {
                tc::tma_load_3d(sm, ma, bar, 32 * ks, 128 * mb, za);
                if (nb >= 2) tc::tma_load_4d(sm + aoff, mb2, bar, 0, 32 * ks, zb, c0);
                if (nb == 4) tc::tma_load_4d(sm + aoff + 2 * boff, mb2, bar, 0, 32 * ks, zb, c0 + 2);
                if (nb & 1) tc::tma_load_4d(sm + aoff + (nb - 1) * boff, mb1, bar, 0, 32 * ks, zb, c0 + nb - 1);
              }
            }
            __syncwarp();
          }
        }
      }
      if (lane == 0) tc::mbar_arrive(&sh.desc_free[i % kRing]);
    }
    if (!ok) sh.err = 1;
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer: the products in the scheduler's order
    auto wait = [&](uint64_t* b, uint32_t parity, int more) {
      return (bool)__all_sync(0xffffffffu, tc::mbar_wait_ns(b, parity, more * g.wait_ns));
    };
    const uint32_t sm0 = __shfl_sync(0xffffffffu, tc::smem_u32(stage_mem), 0);
    uint32_t kcount = 0, tcount = 0;
    bool ok = true;
    for (uint32_t i = 0; ok && !sh.err; ++i) {
      if (!(ok = wait(&sh.desc_full[i % kRing], (i / kRing) & 1, 8))) break;
      const Desc& d = sh.ring[i % kRing];
      if (d.term) break;
      if (d.op == kOpProd) {
        const bool f8 = d.f.fmt == FMT_E4M3, two = d.f.terms > 1;
        // kind::f16 products run over n16 = n rounded up to 16 in N and K (the loads are whole slices of 32 and blocks of
        // 64): the operands' rows and columns past n are zero, so the entries the trimmed product leaves out are 0
        const int n16 = (d.n + 15) & ~15, n64 = d.n64, tiles = d.nrb * d.ncb, ncb = d.ncb;
        const int nks = f8 ? k8_extent(n64) / 128 : (d.n + 31) / 32;
        const uint32_t aoff = two ? 2 * kABytes : kABytes, boff = two ? 2 * kBBlock : kBBlock;
        const uint64_t ad0 = f8 ? tc::sdesc_sw128(sm0, 16, 1024) : tc::sdesc_sw64(sm0, 16, 512);
        const uint64_t bd0 = f8 ? tc::sdesc_sw128(sm0 + 128 * 128, 16, 1024) : tc::sdesc_sw128(sm0 + aoff, boff, 1024);
        for (int ti = d.t0; ti < tiles && ok; ti += G, ++tcount) {
          const int mb = ti / ncb, cb = ti - mb * ncb;
          const int nt = min(kTileN, n64 - kTileN * cb);
          // kind::f16: A K-major, B MN-major; kind::f8f6f4 (E4M3 = 0): both K-major
          const uint32_t id = f8 ? tc::idesc(0, 0, 0, 0, 128, nt)
                                 : tc::idesc(d.f.fmt, d.f.fmt, 0, 1, 128, min(nt, n16 - kTileN * cb));
          const int buf = tcount & 1;
          if (!(ok = wait(&sh.acce[buf], ((tcount >> 1) & 1) ^ 1, 1))) break;
          tc::tc_fence_after();
          const uint32_t dt = tmem + (uint32_t)buf * 256;
          for (int ks = 0; ks < nks; ++ks, ++kcount) {
            const uint32_t st = kcount % kStages;
            if (!(ok = wait(&sh.full[st], (kcount / kStages) & 1, 1))) break;
            tc::tc_fence_after();
            if (tc::elect_one()) {
              const uint64_t ad = ad0 + ((st * kStageBytes) >> 4), bd = bd0 + ((st * kStageBytes) >> 4);
              if (f8) {   // four K = 32 steps of 32 bytes through the 128-byte slice
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc::mma_f8(dt, ad + 2 * kk, bd + 2 * kk, id, (ks > 0 || kk > 0) ? 1u : 0u);
              } else {
#pragma unroll
                for (int kk = 0; kk < 2; ++kk) {   // K = 16 steps below n16 (at least one)
                  if (kk == 1 && 32 * ks + 16 >= n16) break;
                  const uint64_t ah = ad + 2 * kk, bh = bd + 128 * kk;
                  tc::mma_f16(dt, ah, bh, id, (ks > 0 || kk > 0) ? 1u : 0u);
                  if (two) {
                    tc::mma_f16(dt, ah, bh + (kBBlock >> 4), id, 1u);
                    tc::mma_f16(dt, ah + (kABytes >> 4), bh, id, 1u);
                  }
                }
              }
              tc::mma_commit(&sh.empty[st]);
              if (ks == nks - 1) tc::mma_commit(&sh.accf[buf]);
            }
            __syncwarp();
          }
        }
      }
      if (lane == 0) tc::mbar_arrive(&sh.desc_free[i % kRing]);
    }
    if (!ok) sh.err = 1;
  }
  } else {
  tc::setmaxnreg_inc<Shape<kShape>::kRegsEpi>();   // to the epilogue groups
  {
    // ------------------------------------------------ epilogue: drains products, decides, finishes and starts slots
    const int etid = tid - 128;              // 0..255
    const int q = warp & 3;                  // TMEM lane quarter of this warp
    const int grp = (warp - 4) >> 2;         // epilogue group: chunks grp, grp + 3, ... of a tile
    uint32_t tcount = 0;
    int share = 0;   // this CTA's place in the group for the slot at hand: its rows and sums

    // One FP64 n x n matrix M (row-major) as an n64 x n64 operand (zero padded) into the 3-term FP16 planes
    // hi, lo (hi + plane_elems): four rows per warp pass, 8 consecutive columns per lane, the pass's 32 loads
    // all issued before its first store, then 16-byte stores.
    auto fill_pair = [&](uint16_t* hi, int n, int n64, const double* __restrict__ M) {
      uint16_t* lo = hi + plane_elems;
      for (int i0 = 4 * (kEpiWarps * share + warp - 4); i0 < n64; i0 += 4 * kEpiWarps * G) {
        for (int j0 = 8 * lane; j0 < n64; j0 += 256) {
          float vv[4][8];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int i = i0 + r;
#pragma unroll
            for (int u = 0; u < 8; ++u) vv[r][u] = (i < n && j0 + u < n) ? (float)__ldg(M + (size_t)i * n + j0 + u) : 0.0f;
          }
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int i = i0 + r;
            if (i >= n64) break;
            const float (&v)[8] = vv[r];
            uint32_t h[4], l[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) split2(v[2 * u], v[2 * u + 1], FMT_F16, h[u], l[u]);
            *reinterpret_cast<uint4*>(hi + (size_t)i * g.LD + j0) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(lo + (size_t)i * g.LD + j0) = make_uint4(l[0], l[1], l[2], l[3]);
          }
        }
      }
    };

    // inverse mode, a new submatrix J in slot s: c = Tr T_J(S) / n and step 0 without products, since Z_0 = I:
    // V_0 = Y_0 = T_J(S) / c and T_0 = 3I - Y_0 are written directly (pairs 0 and 1, Z's pair: Z_1 = T_0 / 2,
    // the factor 1/2 applied by the products that read Z until its first update), with the defect
    // ||I - Y_0||_F / sqrt(n); only Y_1 = Y_0 T_0 / 2 needs the tensor cores.
    auto start_inverse = [&](int s, int J) -> float {
      const int n = g.sub_n[J], n64 = (n + 63) & ~63;
      const double* S = g.ws + (g.a_off[J] - g.a_base);
      // the trace of T_J(S) (every warp sums it alike, lanes along the diagonal)
      double tr = 0.0;
      for (int i = lane; i < n; i += 32) tr += S[(size_t)i * n + i];
      for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
      const double c = tr / n;
      const float inv = (float)(1.0 / c);
      uint16_t* base = g.planes + (size_t)(sub0 + s) * kPps * plane_elems;
      float dpart = 0.0f;   // this thread's share of ||I - Y_0||_F^2
      // Y_0 and T_0 from one read of T_J(S): the same pass pattern as fill_pair, two pairs out
      for (int i0 = 4 * (kEpiWarps * share + warp - 4); i0 < n64; i0 += 4 * kEpiWarps * G) {
        for (int j0 = 8 * lane; j0 < n64; j0 += 256) {
          float sv[4][8];   // the pass's 32 loads, all issued before its first store
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int i = i0 + r;
#pragma unroll
            for (int u = 0; u < 8; ++u) sv[r][u] = (i < n && j0 + u < n) ? (float)__ldg(S + (size_t)i * n + j0 + u) : 0.0f;
          }
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int i = i0 + r;
            if (i >= n64) break;
            float y[8], t[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int j = j0 + u;
              const bool in = i < n && j < n;
              y[u] = sv[r][u] * inv;
              const float e = (i == j && in ? 1.0f : 0.0f) - y[u];
              dpart += e * e;
              t[u] = in ? (i == j ? 3.0f : 0.0f) - y[u] : 0.0f;
            }
            uint32_t h[4], l[4];
            const size_t off = (size_t)i * g.LD + j0;
#pragma unroll
            for (int u = 0; u < 4; ++u) split2(y[2 * u], y[2 * u + 1], FMT_F16, h[u], l[u]);
            *reinterpret_cast<uint4*>(base + off) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(base + plane_elems + off) = make_uint4(l[0], l[1], l[2], l[3]);
#pragma unroll
            for (int u = 0; u < 4; ++u) split2(t[2 * u], t[2 * u + 1], FMT_F16, h[u], l[u]);
            *reinterpret_cast<uint4*>(base + 2 * plane_elems + off) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(base + 3 * plane_elems + off) = make_uint4(l[0], l[1], l[2], l[3]);
          }
        }
      }
      if (!(c > 0.0) || !isfinite(c)) dpart = INFINITY;   // the scheduler leaves it to the FP64 preparation
      if (tid == 128) sh.cinv[s] = inv;
      return dpart;
    };

    // a4 for a new submatrix of slot s: X_0 = (A - mu I) / alpha in the main format, zero padded
    auto start_sign = [&](int zo, int J) {
        const int n = g.sub_n[J], n64 = (n + 63) & ~63, R = (n + 127) & ~127;
        const float* A = g.A + g.a_off[J];
        const double alpha = scale_alpha(g.lam, g.lam_g, J, g.mu);
        const float inv = (float)(1.0 / alpha), fmu = (float)g.mu;
        uint16_t* hi = g.planes + (size_t)zo * plane_elems;
        uint16_t* lo = hi + plane_elems;
        const Fmt f = g.main_fmt;
        if (f.fmt == FMT_E4M3) {
          // one-byte view: X_0 * 2^7 in E4M3 over whole 128-byte K slices, and zeros in the K padding of
          // the other X plane and of T (their products write only the first n64 columns)
          const int k8 = k8_extent(n64);
          uint8_t* p8 = reinterpret_cast<uint8_t*>(hi);
          for (int e = etid + kEpiThreads * share; e < R * k8; e += kEpiThreads * G) {
            const int i = e / k8, j = e - i * k8;
            float x = 0.0f;
            if (i < n && j < n) x = (A[(size_t)i * n + j] - (i == j ? fmu : 0.0f)) * inv;
            p8[(size_t)i * 2 * g.LD + j] = (uint8_t)__nv_cvt_float_to_fp8(kF8Up * x, __NV_SATFINITE, __NV_E4M3);
            if (j >= n64) {
              p8[2 * 2 * plane_elems + (size_t)i * 2 * g.LD + j] = 0;   // X_1
              p8[4 * 2 * plane_elems + (size_t)i * 2 * g.LD + j] = 0;   // T
            }
          }
        } else {
          // four rows per warp pass, 8 consecutive columns per lane (all 32 loads in flight together, then
          // 16-byte stores of hi and lo); rows and columns n..n64 are the zero padding; rows from n64 on
          // only feed product rows that are never read back
          for (int i0 = 4 * (kEpiWarps * share + warp - 4); i0 < n64; i0 += 4 * kEpiWarps * G) {
            for (int j0 = 8 * lane; j0 < n64; j0 += 256) {
              float v[4][8];
#pragma unroll
              for (int r = 0; r < 4; ++r) {
                const float* row = A + (size_t)min(i0 + r, n - 1) * n;   // (no condition holds a load back)
#pragma unroll
                for (int u = 0; u < 8; ++u) v[r][u] = __ldg(row + min(j0 + u, n - 1));
              }
#pragma unroll
              for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                  const int i = i0 + r, j = j0 + u;
                  v[r][u] = i < n && j < n ? (v[r][u] - (i == j ? fmu : 0.0f)) * inv : 0.0f;
                }
#pragma unroll
              for (int r = 0; r < 4; ++r) {
                const int i = i0 + r;
                if (i >= n64) break;
                uint32_t h[4], l[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) split2(v[r][2 * u], v[r][2 * u + 1], f.fmt, h[u], l[u]);
                *reinterpret_cast<uint4*>(hi + (size_t)i * g.LD + j0) = make_uint4(h[0], h[1], h[2], h[3]);
                if (f.terms > 1)
                  *reinterpret_cast<uint4*>(lo + (size_t)i * g.LD + j0) = make_uint4(l[0], l[1], l[2], l[3]);
              }
            }
          }
        }
    };

    // a7 for the finished submatrix of slot s: centre columns of T_J(D) = 1/2 (I - X) T_J(S)^-1 and the
    // FP64 partial traces
    auto finish_sign = [&](const Desc& d) {
      const int J = d.fin, n = d.n, b = g.nbf[J];
      // this CTA's rows
      const int rows = 32 * (((n + 31) / 32 + G - 1) / G), r0 = min(n, rows * share), r1 = min(n, r0 + rows);
      // the final X_k, hi (+ lo) in the last product's output format
      const uint16_t* xh = g.planes + (size_t)d.za * plane_elems;
      const uint16_t* xl = xh + plane_elems;
      const Fmt xfmt = d.f;
      const double* Q = g.Q + g.c_off[J];
      const double* Sc = g.Sc + g.c_off[J];
      const double* Hc = g.Hc + g.c_off[J];
      double* Dc = g.Dc + g.c_off[J];
      // X Q eight columns at a time, Q in FP32 in the staging buffers (idle between products; in pieces of kRowsQ rows
      // when there are more), zero padded; the sums (hi, lo) of up to kRowsP rows of X then go through shared memory to
      // the FP64 step, which runs entry by entry
      constexpr int kRowsP = 128, kRowsQ = (int)((kStgTotal - 64 * kRowsP) / 34) & ~31;
      static_assert(4 * (8 * kRowsQ + 4 * (kRowsQ / 8)) + 64 * kRowsP <= kStgTotal, "staging");
      const int n64 = d.n64;
      const bool exact = exact_xq(n, b);
      float* const Qs = reinterpret_cast<float*>(stg);
      float2* const Ps = reinterpret_cast<float2*>(stg + kStgTotal - 64 * kRowsP);
      double ps = 0.0, ph = 0.0;
      for (int cg = 0; cg < b; cg += 8) {
        const int cn = min(8, b - cg);
        for (int rr = r0; rr < r1; rr += kRowsP) {
          const int rn = min(kRowsP, r1 - rr);
          for (int k0 = 0; k0 < n64; k0 += kRowsQ) {
            const int kn = min(kRowsQ, n64 - k0);
            if (rr == r0 || n64 > kRowsQ) {
              epi_bar<kEpiThreads>();   // the last piece has been used
              for (int e0 = etid; e0 < kn * 8; e0 += 8 * kEpiThreads) {   // eight loads in flight
                double v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                  const int e = e0 + u * kEpiThreads;
                  v[u] = __ldg(Q + (size_t)min(k0 + (e >> 3), n - 1) * b + cg + min(e & 7, cn - 1));
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                  const int e = e0 + u * kEpiThreads, k = e >> 3;
                  if (k < kn) Qs[qs_at(k) + (e & 7)] = k0 + k < n && (e & 7) < cn ? (float)v[u] : 0.0f;
                }
              }
              epi_bar<kEpiThreads>();
            }
            for (int it = warp - 4; 8 * it < rn; it += kEpiWarps) {
              const int row = 8 * it + (lane >> 2), part = lane & 3;
              const size_t ro = (size_t)min(rr + row, n - 1) * g.LD + k0;
              uint64_t s[4], e[4];
              auto sums = [&](auto sum) {
                if (exact) sum(std::true_type{});
                else sum(std::false_type{});
              };
              const uint16_t *h = xh + ro, *l = xl + ro;
              if (xfmt.fmt == FMT_BF16) {
                if (xfmt.terms > 1) sums([&](auto x) { xq_rows<FMT_BF16, true, x.value>(h, l, kn, Qs, part, s, e); });
                else sums([&](auto x) { xq_rows<FMT_BF16, false, x.value>(h, l, kn, Qs, part, s, e); });
              } else {
                if (xfmt.terms > 1) sums([&](auto x) { xq_rows<FMT_F16, true, x.value>(h, l, kn, Qs, part, s, e); });
                else sums([&](auto x) { xq_rows<FMT_F16, false, x.value>(h, l, kn, Qs, part, s, e); });
              }
              if (part == 0) {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                  const float2 sv = unpair2(s[c >> 1]), ev = unpair2(e[c >> 1]);
                  float2 p = c & 1 ? make_float2(sv.y, ev.y) : make_float2(sv.x, ev.x);
                  if (k0 > 0) {
                    const float2 o = Ps[row * 8 + c];
                    two_sum(p.x, p.y, o.x);
                    p.y += o.y;
                  }
                  Ps[row * 8 + c] = p;
                }
              }
            }
          }
          epi_bar<kEpiThreads>();
          for (int e = etid; e < rn * cn; e += kEpiThreads) {
            const int i = e / cn, c = e - i * cn;
            const float2 p = Ps[i * 8 + c];
            const size_t at = (size_t)(rr + i) * b + cg + c;
            const double dv = 0.5 * (Q[at] - ((double)p.x + (double)p.y));
            Dc[at] = dv;
            ps += dv * Sc[at];
            ph += dv * Hc[at];
          }
          epi_bar<kEpiThreads>();
        }
      }
      double px = 0.0;   // the trace of the final X: (n - Tr X) / 2 eigenvalues lie below mu
      for (int i = r0 + etid; i < r1; i += kEpiThreads) {
        float x = from_bits(xh[(size_t)i * g.LD + i], xfmt.fmt);
        if (xfmt.terms > 1) x += from_bits(xl[(size_t)i * g.LD + i], xfmt.fmt);
        px += x;
      }
      for (int o = 16; o > 0; o >>= 1) {
        ps += __shfl_xor_sync(0xffffffffu, ps, o);
        ph += __shfl_xor_sync(0xffffffffu, ph, o);
        px += __shfl_xor_sync(0xffffffffu, px, o);
      }
      if (lane == 0) {
        sh.dred[0][warp - 4] = ps;
        sh.dred[1][warp - 4] = ph;
        sh.dred[2][warp - 4] = px;
      }
      epi_bar<kEpiThreads>();
      if (tid < 131 && tid >= 128) {
        double t = 0.0;
        for (int w = 0; w < kEpiWarps; ++w) t += sh.dred[tid - 128][w];
        if (G > 1) __stcg(&gs[d.slot].tr[tid - 128][share], t);
        else sh.tr[d.slot][tid - 128] = t;
      }
      epi_bar<kEpiThreads>();   // staging and dred free again
    };

    // this CTA's part of a phase is done: its share of the defect (thread 128), and the arrival. Every thread's writes
    // precede the barrier.
    auto arrive = [&](const Desc& d, float part) {
      if (tid == 128) {
        if (G > 1) {
          __stcg(&gs[d.slot].part[d.par][share], part);
          tc::red_release_gpu(&gs[d.slot].count, 1u);
        } else {
          sh.part[d.slot] = part;
        }
      }
      tc::mbar_arrive(&sh.epi_done[d.slot]);
    };

    for (uint32_t i = 0;; ++i) {
      // every epilogue thread waits for the descriptor; a wait that ran out in any of them ends all
      const bool got = tc::mbar_wait_ns(&sh.desc_full[i % kRing], (i / kRing) & 1, 8 * g.wait_ns);
      if (epi_bar_or<kEpiThreads>(!got || sh.err)) {
        if (tid == 128) sh.err = 1;
        break;
      }
      const Desc d = sh.ring[i % kRing];
      if (d.term) break;
      const int n = d.n, n64 = d.n64, n16 = (n + 15) & ~15;
      share = (rank - d.slot * (G / 2) + G) % G;
      if (d.op != kOpProd) {
        float dpart = 0.0f;
        if (d.op == kOpFill) {
          fill_pair(g.planes + (size_t)d.fill * plane_elems, n, n64, g.ws + (g.a_off[d.job] - g.a_base) + g.chunk_n2);
        } else {
          if constexpr (kMode == 0) {
            if (d.fin >= 0) finish_sign(d);
            if (d.job >= 0) start_sign(d.zo, d.job);
          } else {
            dpart = start_inverse(d.slot, d.job);
          }
        }
        tc::fence_proxy_async_global();
        for (int o = 16; o > 0; o >>= 1) dpart += __shfl_xor_sync(0xffffffffu, dpart, o);
        if (lane == 0) sh.red[i & 1][warp - 4] = dpart;
        epi_bar<kEpiThreads>();
        float dsum = 0.0f;
        if (tid == 128)
          for (int w = 0; w < kEpiWarps; ++w) dsum += sh.red[i & 1][w];
        arrive(d, dsum);
        if (tid == 128) tc::mbar_arrive(&sh.desc_free[i % kRing]);
        continue;
      }
      // the sign iteration's epilogues are fixed by the product kind (no descriptor fields needed)
      const int epi = kMode == 0 ? (d.kind == 0 ? kEpiT : kEpiScale) : d.epi;
      const float escale = kMode == 0 ? 0.5f : (epi == kEpiA ? 1.0f : d.scale);
      float part = 0.0f;
      bool bad = false;   // a wait of this warp ran out: keep the barrier schedule, skip the work
      for (int ti = d.t0; ti < d.nrb * d.ncb; ti += G) {
          const int mb = ti / d.ncb, cb = ti - mb * d.ncb;
          const int nt = min(kTileN, n64 - kTileN * cb);
          const int buf = tcount & 1;
          if (!bad) bad = !tc::mbar_wait_ns(&sh.accf[buf], (tcount >> 1) & 1, g.wait_ns);
          bad = __any_sync(0xffffffffu, bad);   // tcgen05.ld needs the whole warp
          tc::tc_fence_after();
          const int rbase = 128 * mb + 32 * q;
          const int row = rbase + lane;
          const bool live = rbase < n64 && !bad;   // rows >= n64 are never read back
          const int nch = nt / 32;
          const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)buf * 256;
          uint32_t r[32];
          if (live && grp < nch) tc::tmem_ld32(taddr + 32 * grp, r);
          // E4M3 operand scales; and the factor of the inverse mode's Z before its first update
          const float sc = (d.f.fmt == FMT_E4M3 ? kF8Down : 1.0f) * (kMode == 1 && epi == kEpiT ? d.pscale : 1.0f);
          for (int c0 = grp; c0 < nch; c0 += kGroups) {
            const int col0 = kTileN * cb + 32 * c0;
            if (!live) continue;
            tc::tmem_wait_ld();
            // Zeros from column n16 on, where the trimmed product left the accumulator as it was: the next products'
            // K and N reach to n64. Rows and columns from n to n16 are zeros already, the operands' being zeros.
            if (col0 + 16 >= n16) {
              const bool none = col0 >= n16;
#pragma unroll
              for (int u = 0; u < 32; ++u) r[u] = u >= 16 || none ? 0u : r[u];
            }
            const bool rin = row < n;
            if (kMode == 1 && epi >= kEpiX) {
              // inverse mode: X or A_J in FP32, row-major n x n. The chunk goes through the warp's staging
              // buffer (row = lane, entry j at j ^ lane: no bank conflicts either way) so that each store
              // instruction writes 32 consecutive entries of one row
              float* dst = epi == kEpiX ? g.Xout + (g.a_off[d.job] - g.a_base) : g.Aout + g.a_off[d.job];
              float* wf = reinterpret_cast<float*>(stg + (size_t)(warp - 4) * 4096);
              if (lane == 0) tc::bulk_wait_read<0>();   // this warp's previous store has read the buffer
              __syncwarp();
#pragma unroll
              for (int j = 0; j < 32; ++j) wf[lane * 32 + (j ^ lane)] = escale * __uint_as_float(r[j]);
              __syncwarp();
              const int nr = min(32, n - rbase);
              float* at = dst + (size_t)rbase * n + col0 + lane;
              if (col0 + lane < n) {
#pragma unroll 8
                for (int rr = 0; rr < nr; ++rr, at += n) *at = wf[rr * 32 + (lane ^ rr)];
              }
              __syncwarp();   // the staging is free again
              if (epi == kEpiA) {   // no operand to write
                if (c0 + kGroups < nch) tc::tmem_ld32(taddr + 32 * (c0 + kGroups), r);
                continue;
              }
            }
            // T: (3I - P)_ij = (I - P)_ij = -P_ij off the diagonal. On it (rows below n): P - 1 first, whose negative
            // counts for the defect, then 2 more. sc is a power of two, so that P - 1 / sc is as exact as sc P - 1.
            const int du = epi == kEpiT && col0 == (rbase & ~31) && rin ? row - col0 : -1;   // this row's diagonal entry
            float m = escale * sc;
            if (epi == kEpiT) {
              m = -sc;
              if (col0 == (rbase & ~31)) {
                const float one = 1.0f / sc;
#pragma unroll
                for (int u = 0; u < 32; ++u) r[u] = pick(u, du, __float_as_uint(__uint_as_float(r[u]) - one), r[u]);
              }
            }
            if (kMode == 0 && kShape == 0 && d.fo.fmt == FMT_E4M3) {
              // E4M3 output (scaled by 2^7): this thread's 32 bytes of the row, two 16-byte stores into the
              // one-byte view of the plane (rows of 2 LD bytes)
              float q4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
              uint32_t w8[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                float v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  v[u] = m * __uint_as_float(r[4 * j + u]);
                  q4[u] = fmaf(v[u], v[u], q4[u]);
                  v[u] = kF8Up * __uint_as_float(pick(4 * j + u, du, __float_as_uint(v[u] + 2.0f), __float_as_uint(v[u])));
                }
                const uint32_t p0 = __nv_cvt_float2_to_fp8x2(make_float2(v[0], v[1]), __NV_SATFINITE, __NV_E4M3);
                const uint32_t p1 = __nv_cvt_float2_to_fp8x2(make_float2(v[2], v[3]), __NV_SATFINITE, __NV_E4M3);
                w8[j] = p0 | (p1 << 16);
              }
              if (rin) part += (q4[0] + q4[1]) + (q4[2] + q4[3]);
              if (c0 + kGroups < nch) tc::tmem_ld32(taddr + 32 * (c0 + kGroups), r);
              uint8_t* dst = reinterpret_cast<uint8_t*>(g.planes) + (size_t)d.zo * plane_elems * 2 +
                             (size_t)row * (2 * g.LD) + col0;
              reinterpret_cast<uint4*>(dst)[0] = make_uint4(w8[0], w8[1], w8[2], w8[3]);
              reinterpret_cast<uint4*>(dst)[1] = make_uint4(w8[4], w8[5], w8[6], w8[7]);
              continue;
            }
            uint32_t h[16], l[16];
            float sq = 0.0f;
            if constexpr (kMode == 1) scale_split_t<FMT_F16, true, true>(r, m, h, l, sq);
            else scale_split<true>(r, m, d.fo, h, l, sq);
            if (rin) part += sq;   // (lanes without a row hold anything; used after T alone)
            if (epi == kEpiT && col0 == (rbase & ~31)) {
              uint32_t e = 0;
#pragma unroll
              for (int u = 0; u < 32; ++u) e = pick(u, du, r[u], e);
              uint32_t th, tl;
              split2(fmaf(m, __uint_as_float(e), 2.0f), 0.0f, kMode == 1 ? (int)FMT_F16 : d.fo.fmt, th, tl);
              const uint32_t sel = du & 1 ? 0x5410u : 0x3254u;
              const int dw = du >> 1;   // (-1 for none)
#pragma unroll
              for (int u = 0; u < 16; ++u) {
                h[u] = pick(u, dw, __byte_perm(h[u], th, sel), h[u]);
                l[u] = pick(u, dw, __byte_perm(l[u], tl, sel), l[u]);
              }
            }
            if (c0 + kGroups < nch) tc::tmem_ld32(taddr + 32 * (c0 + kGroups), r);   // overlaps the stores
            // each warp stores its own 32 rows x 32 columns through its own 4 KB staging buffer (hi rows, then
            // lo rows; 64-byte swizzle: 16-byte unit c of row r at unit c ^ ((r >> 1) & 3)), with one TMA
            // tensor store issued by its lane 0 for both planes (a box two planes deep): no barrier between
            // warps, one store per chunk
            uint8_t* wb = stg + (size_t)(warp - 4) * 4096;
            if (lane == 0) tc::bulk_wait_read<0>();   // this warp's previous store has read the buffer
            __syncwarp();
            uint4* dh = reinterpret_cast<uint4*>(wb + lane * 64);
#pragma unroll
            for (int c = 0; c < 4; ++c)
              dh[c ^ ((lane >> 1) & 3)] = make_uint4(h[4 * c], h[4 * c + 1], h[4 * c + 2], h[4 * c + 3]);
            if (kMode == 1 || d.fo.terms > 1) {
              uint4* dl = reinterpret_cast<uint4*>(wb + 2048 + lane * 64);
#pragma unroll
              for (int c = 0; c < 4; ++c)
                dl[c ^ ((lane >> 1) & 3)] = make_uint4(l[4 * c], l[4 * c + 1], l[4 * c + 2], l[4 * c + 3]);
            }
            tc::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
              tc::tma_store_3d(kMode == 1 || d.fo.terms > 1 ? &maps.S2 : &maps.S, wb, col0, rbase, d.zo);
              tc::bulk_commit();
            }
          }
          tc::tc_fence_before();
          if (!bad) tc::mbar_arrive(&sh.acce[buf]);
          ++tcount;
        }
      if (lane == 0) tc::bulk_wait<0>();   // this warp's stores are written before anyone reads them
      tc::fence_proxy_async_global();
      // ---- end of the product: one uniform error decision, then the slot's next state
      for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      if (lane == 0) sh.red[i & 1][warp - 4] = part;
      if (epi_bar_or<kEpiThreads>(bad)) {
        if (tid == 128) sh.err = 1;
        break;
      }
      if (kMode == 1 && d.fill >= 0) {
        fill_pair(g.planes + (size_t)d.fill * plane_elems, n, n64, g.ws + (g.a_off[d.job] - g.a_base) + g.chunk_n2);
        tc::fence_proxy_async_global();
        epi_bar<kEpiThreads>();
      }
      float dsum = 0.0f;
      if (tid == 128)
        for (int w = 0; w < kEpiWarps; ++w) dsum += sh.red[i & 1][w];
      arrive(d, dsum);
      if (tid == 128) tc::mbar_arrive(&sh.desc_free[i % kRing]);
    }
    if (sh.err && tid == 128) {
      // a wait ran out: the submatrices in flight are reported as timed out
      for (int s = 0; s < 2 * kSlots; ++s) {
        const int J = s & 1 ? sh.slot[s >> 1].fin : sh.slot[s >> 1].job;
        if (J >= 0 && kMode == 1) {
          g.prep_out[J] = kSubTimeout;
        } else if (J >= 0) {
          g.status[J] = kSubTimeout;
          g.iters[J] = sh.slot[s >> 1].steps;
          g.rsteps[J] = sh.slot[s >> 1].rsteps;
          g.tS[J] = 0.0;
          g.tH[J] = 0.0;
        }
      }
      atomicExch(g.err, 1);
    }
  }
  }

  // every role has left its loop, so sh.err is final; after a timeout wait (bounded) for this CTA's
  // TMA loads and MMAs still in flight before the shared and tensor memory are released
  __syncthreads();
  if (sh.err) {
    if (warp == 2 && lane == 0)
      for (uint32_t k = loads > kStages ? loads - kStages : 0; k < loads; ++k)
        tc::mbar_wait_ns(&sh.full[k % kStages], (k / kStages) & 1, 50000000ull);
    if (warp == 1 && lane == 0) {
      tc::mma_commit(&sh.idle);
      tc::mbar_wait_ns(&sh.idle, 0, 50000000ull);
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// Every submatrix of the launch starts as "timed out": the sign kernel overwrites the status of each one it
// takes, so a submatrix that no block reached (every block gave up on a bounded wait) is reported as such
// instead of keeping the status of an earlier solve.
__global__ void k_status_pending(int32_t j0, int32_t count, const int32_t* __restrict__ list,
                                 int32_t* __restrict__ status) {
  for (int32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < count; e += gridDim.x * blockDim.x)
    status[list ? list[e] : j0 + e] = kSubTimeout;
}

}  // namespace

// ==================================================================================== host side

struct TcState {
  DevBuf planes, order, err, groups, again;
  int R = 0, LD = 0, slots = 0;
  int64_t ord_j0 = -1, ord_j1 = -1;
  int32_t ord_large = 0;          // how many of the cached order (a prefix) have n above 192
  int32_t ord_mean = 0;           // their mean dimension
  bool ord_exact = false;         // some of the others sum X Q exactly
  DevBuf inv_planes, inv_flops;   // inverse mode: its own plane layout (kPlanesInv per slot), flop sums
  int iR = 0, iLD = 0, islots = 0;
};

static TcState* state(nolsm_plan* plan) {
  if (!plan->tc) plan->tc = new TcState();
  return static_cast<TcState*>(plan->tc);
}

void tc_release(nolsm_plan* plan) {
  if (!plan->tc) return;
  TcState* s = static_cast<TcState*>(plan->tc);
  dev_free(plan, s->planes);
  dev_free(plan, s->order);
  dev_free(plan, s->err);
  dev_free(plan, s->groups);
  dev_free(plan, s->again);
  dev_free(plan, s->inv_planes);
  dev_free(plan, s->inv_flops);
  delete s;
  plan->tc = nullptr;
}

int main_terms(int precision) {
  return precision == NOLSM_FP32 || precision == NOLSM_BF16X3 ? 3 : 1;
}

static bool formats(int precision, Fmt* main_fmt, Fmt* refine_fmt) {
  *refine_fmt = Fmt{FMT_F16, 3};
  switch (precision) {
    case NOLSM_FP32: *main_fmt = Fmt{FMT_F16, 3}; return true;
    case NOLSM_BF16X3: *main_fmt = Fmt{FMT_BF16, 3}; return true;
    case NOLSM_BF16: *main_fmt = Fmt{FMT_BF16, 1}; return true;
    case NOLSM_FP8E4M3: *main_fmt = Fmt{FMT_E4M3, 1}; return true;
    case NOLSM_FP16: *main_fmt = Fmt{FMT_F16, 1}; return true;
    default: return false;
  }
}

// The register split (setmaxnreg) assumes that the launch gives each thread regs registers; with fewer, the epilogue
// warpgroups' increase could never be granted, so the launch is refused.
static bool split_ok(const void* fn, int regs) {
  cudaFuncAttributes at{};
  const bool ok = cudaFuncGetAttributes(&at, fn) == cudaSuccess;
  if (!ok) cudaGetLastError();
  return ok && at.numRegs == regs;
}
static nolsm_status check_register_split(const void* fn, int regs) {
  if (!split_ok(fn, regs)) {
    set_error("k_ns_tc was not built with the %d registers per thread that its register split needs", regs);
    return NOLSM_ERR_UNSUPPORTED;
  }
  return NOLSM_OK;
}

// ------------------------------------------------------------------ launch shapes and their tuner

// The maps of [planes][R][LD] 2-byte planes; one_byte: also as rows of 2 LD bytes for E4M3 (which runs in shape 0)
static nolsm_status make_maps(TcMaps* m, void* base, int R, int LD, int planes, bool one_byte) {
  const uint64_t r = (uint64_t)R, ld = (uint64_t)LD, z = (uint64_t)planes;
  const CUtensorMapSwizzle sw64 = CU_TENSOR_MAP_SWIZZLE_64B;
  bool ok = tmap::make_3d(&m->A, base, 2, ld, r, z, 32, 128, sw64) && tmap::make_3d(&m->A2, base, 2, ld, r, z, 32, 128, sw64, 2) &&
            tmap::make_blocks(&m->B, base, ld, r, z, 32, 1, 1) && tmap::make_blocks(&m->B2, base, ld, r, z, 32, 2, 1) &&
            tmap::make_blocks(&m->Bx2, base, ld, r, z, 32, 1, 2) && tmap::make_blocks(&m->B2x2, base, ld, r, z, 32, 2, 2) &&
            tmap::make_3d(&m->S, base, 2, ld, r, z, 32, 32, sw64) && tmap::make_3d(&m->S2, base, 2, ld, r, z, 32, 32, sw64, 2);
  m->A8 = m->A;
  m->B8 = m->B;
  if (one_byte)
    ok = ok && tmap::make_3d(&m->A8, base, 1, 2 * ld, r, z, 128, 128) &&
         tmap::make_3d(&m->B8, base, 1, 2 * ld, r, z, 128, Shape<0>::kTileN);
  if (ok) return NOLSM_OK;
  set_error("cuTensorMapEncodeTiled rejected the scratch layout (R %d, LD %d, planes %d)", R, LD, planes);
  return NOLSM_ERR_CUDA;
}

using TcKernel = decltype(&k_ns_tc<0, 0>);

static TcKernel tc_kernel(int mode, int shape) {
  if (mode == 0) return shape == 0 ? &k_ns_tc<0, 0> : &k_ns_tc<0, 1>;
  return shape == 0 ? &k_ns_tc<1, 0> : &k_ns_tc<1, 1>;
}

// How many CTAs share a submatrix, by the mean dimension of a launch's submatrices above 192 rows: enough for the planes
// of the submatrices in flight to stay in L2, few enough for a product's tiles (2 at n = 256, 18 at n = 650) to give
// each CTA some. Measured, sign + inverse, ms, with 1 / 2 / 4 / 8 CTAs: 5,000 of n = 193-310 (mean 222) 24.4 / 23.0 /
// 32.2 / 59.5; 512 merged sites of n = 200-400 13.6 / 7.4 / 6.8 / 8.4; 343 of n = 200-500 10.9 / 7.5 / 6.7 / 6.9; 512 of
// n = 598-713 35.5 / 30.0 / 24.3 / 20.9, with 16 38.3.
static int group_size(int mean_n) {
  return mean_n <= 192 ? 1 : mean_n <= 256 ? 2 : mean_n <= 512 ? 4 : 8;
}
static int group_slots(int G, int64_t count, int sms) {
  return (int)std::min<int64_t>(sms / G, (count + kSlots - 1) / kSlots) * kSlots;
}

// One launch of kernel (mode, shape) over the submatrices g.order[0, g.j1) (g.j0 = 0): one CTA per SM at most,
// kSlots submatrices in flight in each group of them; the work counter and the groups' are reset first. CTAs that wait
// on one another have to run at the same time: a cooperative launch.
static nolsm_status launch_shape(int mode, int shape, const TcMaps& m, TcArgs g, int sms, cudaStream_t st) {
  const TcKernel k = tc_kernel(mode, shape);
  const int threads = shape == 0 ? Shape<0>::kThreads : Shape<1>::kThreads;
  const int smem = shape == 0 ? Shape<0>::kSmemBytes : Shape<1>::kSmemBytes;
  NOLSM_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  NOLSM_TRY(check_register_split(reinterpret_cast<const void*>(k), shape == 0 ? Shape<0>::kRegsLaunch : Shape<1>::kRegsLaunch));
  NOLSM_CUDA_TRY(cudaMemsetAsync(g.next, 0, sizeof(int32_t), st));
  const int slots = group_slots(g.group, g.j1, sms);
  if (g.group > 1) NOLSM_CUDA_TRY(cudaMemsetAsync(g.groups, 0, sizeof(GroupSlot) * slots, st));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(slots / kSlots * g.group));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.attrs = &at;
  cfg.numAttrs = g.group > 1 ? 1 : 0;
  NOLSM_CUDA_TRY(cudaLaunchKernelEx(&cfg, k, m, g));
  return NOLSM_OK;
}

// The launch shapes of a (mode, precision) as measured in this process (-1: not yet): by the CTAs that share a submatrix
// (1, 2, 4, 8), which decide how tiles are dealt and so which shape is the faster; the last one taken; and bucket 0's. The
// environment variable NOLSM_TC_SHAPE ("0" or "1") fixes the shape instead.
struct Shapes { int of_group[4] = {-1, -1, -1, -1}, last = -1, small = -1; };
static std::mutex g_shape_mu;
static Shapes g_shape[2][8];
static int group_index(int G) { return G >= 8 ? 3 : G >= 4 ? 2 : G >= 2 ? 1 : 0; }

static int env_shape() {
  const char* e = std::getenv("NOLSM_TC_SHAPE");
  if (e && (e[0] == '0' || e[0] == '1') && e[1] == 0) return e[0] - '0';
  return -1;
}

// The launch shape of the submatrices order[0, count), all with n above 192 (bucket 1): the one NOLSM_TC_SHAPE
// fixes, else the one measured faster for (mode, precision, g.group) in this process. The
// first time, both shapes run on the largest of them (32 per slot of every SM: with fewer, the
// start and the tail of the launch decide; the shapes differ by 3-40 % in steady state), timed with CUDA
// events on the stream, and the faster is kept (not when a bounded wait ran out in the measurement); the
// results of those runs are computed again by the launches that follow. pending(order, count) resets the
// statuses of the submatrices a launch takes.
template <typename Pending>
static nolsm_status bucket_shape(int mode, int precision, const TcMaps& m, TcArgs g, const int32_t* order, int32_t count,
                                 int sms, cudaStream_t st, Pending pending, int* out) {
  int shape = env_shape();
  Shapes& known = g_shape[mode][precision & 7];
  const int gi = group_index(g.group);
  if (shape < 0) {
    std::lock_guard<std::mutex> lk(g_shape_mu);
    shape = known.of_group[gi];
    if (shape >= 0) known.last = shape;
  }
  if (shape < 0) {
    g.j0 = 0;
    g.order = order;
    const int32_t sample = std::min<int32_t>(count, 32 * kSlots * sms);
    struct Events {   // destroyed on every way out
      cudaEvent_t e[2] = {nullptr, nullptr};
      ~Events() {
        for (cudaEvent_t x : e)
          if (x) cudaEventDestroy(x);
      }
    } ev;
    float ms[2] = {0.0f, 0.0f};
    NOLSM_CUDA_TRY(cudaEventCreate(&ev.e[0]));
    NOLSM_CUDA_TRY(cudaEventCreate(&ev.e[1]));
    for (int sh = 0; sh < 2; ++sh) {
      g.j1 = sample;
      NOLSM_TRY(pending(order, sample));
      NOLSM_CUDA_TRY(cudaEventRecord(ev.e[0], st));
      NOLSM_TRY(launch_shape(mode, sh, m, g, sms, st));
      NOLSM_CUDA_TRY(cudaEventRecord(ev.e[1], st));
      NOLSM_CUDA_TRY(cudaEventSynchronize(ev.e[1]));
      NOLSM_CUDA_TRY(cudaEventElapsedTime(&ms[sh], ev.e[0], ev.e[1]));
    }
    int32_t errf = 0;
    NOLSM_CUDA_TRY(cudaMemcpyAsync(&errf, g.err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    NOLSM_CUDA_TRY(cudaStreamSynchronize(st));
    if (errf != 0) {
      shape = 0;
    } else {
      shape = ms[1] < ms[0] ? 1 : 0;
      std::lock_guard<std::mutex> lk(g_shape_mu);
      known.of_group[gi] = known.last = shape;
    }
  }
  *out = shape;
  return NOLSM_OK;
}

// Runs the submatrices order[0, count), largest first, as one launch: those of more than 192 rows in the shape that
// bucket_shape gives; E4M3 (fixed0: all dimensions) in shape 0 and groups of one.
template <typename Pending>
static nolsm_status run_largest_first(int mode, int precision, bool fixed0, const TcMaps& m, TcArgs g, const int32_t* order,
                                      int32_t count, int mean_n, int sms, cudaStream_t st, Pending pending) {
  if (count <= 0) return NOLSM_OK;
  int shape = 0;
  g.group = fixed0 ? 1 : group_size(mean_n);
  if (!fixed0) NOLSM_TRY(bucket_shape(mode, precision, m, g, order, count, sms, st, pending, &shape));
  g.j0 = 0;
  g.j1 = count;
  g.order = order;
  NOLSM_TRY(pending(order, count));
  return launch_shape(mode, shape, m, g, sms, st);
}

// Bucket 0 (n <= 192) has no shape to choose (res_path.cu): the query reports 0 once it has run.
static void resident_shape(int mode, int precision) {
  std::lock_guard<std::mutex> lk(g_shape_mu);
  g_shape[mode][precision & 7].small = 0;
}

int tc_shape_choice(int mode, int precision, int bucket) {
  if (mode < 0 || mode > 1 || bucket < 0 || bucket > 1) return -1;
  std::lock_guard<std::mutex> lk(g_shape_mu);
  const Shapes& known = g_shape[mode][precision & 7];
  return bucket == 0 ? known.small : known.last;
}

nolsm_status solve_tc(nolsm_plan* plan, double mu, const nolsm_options& o, int64_t j0, int64_t j1, const SolveSpec& spec,
                      cudaStream_t st) {
  Fmt mf, rf;
  if (!formats(o.precision, &mf, &rf)) {
    set_error("precision %d is not available on the tensor-core path in this build", o.precision);
    return NOLSM_ERR_UNSUPPORTED;
  }
  if (mf.fmt == FMT_E4M3 && o.refine_steps < 1) {
    set_error("E4M3 needs at least one refinement step (the centre-column phase reads a 2-byte X)");
    return NOLSM_ERR_UNSUPPORTED;
  }
  NOLSM_TRY(ensure_results(plan));
  TcState* S = state(plan);
  int dev = 0, sms = 0;
  NOLSM_CUDA_TRY(cudaGetDevice(&dev));
  NOLSM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  int32_t maxn = 0, minn = INT32_MAX;
  for (int64_t J = j0; J < j1; ++J) {
    maxn = std::max(maxn, plan->h_sub_n[J]);
    minn = std::min(minn, plan->h_sub_n[J]);
  }
  const int LD = (maxn + 63) & ~63, R = (maxn + 127) & ~127;
  const int64_t work = spec.list ? spec.count : j1 - j0;
  if (work <= 0) return NOLSM_OK;
  // submatrices of up to kResMaxN rows run with their operands on the SM (res_path.cu), the others, and E4M3, with
  // operands in scratch
  const bool f8 = mf.fmt == FMT_E4M3;
  const int32_t above = f8 ? 0 : kResMaxN;
  const bool streamed = maxn > above, resident = !f8 && minn <= kResMaxN;
  if (!S->err.p) NOLSM_TRY(dev_alloc(plan, S->err, sizeof(int32_t) * 4));
  if (!S->groups.p) NOLSM_TRY(dev_alloc(plan, S->groups, sizeof(GroupSlot) * kSlots * sms));
  if (S->ord_j0 != j0 || S->ord_j1 != j1) {
    std::vector<int32_t> ord;
    largest_first(plan->h_sub_n, j0, j1 - j0, ord);
    if (S->order.bytes < sizeof(int32_t) * ord.size()) {
      dev_free(plan, S->order);
      NOLSM_TRY(dev_alloc(plan, S->order, sizeof(int32_t) * (size_t)plan->n_mol));
    }
    NOLSM_CUDA_TRY(cudaMemcpyAsync(S->order.p, ord.data(), sizeof(int32_t) * ord.size(), cudaMemcpyHostToDevice, st));
    NOLSM_CUDA_TRY(cudaStreamSynchronize(st));
    S->ord_j0 = j0;
    S->ord_j1 = j1;
    S->ord_large = 0;
    int64_t sum = 0;
    while (S->ord_large < (int32_t)ord.size() && plan->h_sub_n[ord[(size_t)S->ord_large]] > 192)
      sum += plan->h_sub_n[ord[(size_t)S->ord_large++]];
    S->ord_mean = S->ord_large > 0 ? (int32_t)(sum / S->ord_large) : 0;
    S->ord_exact = false;
    for (size_t k = (size_t)S->ord_large; k < ord.size(); ++k)
      S->ord_exact = S->ord_exact || exact_xq(plan->h_sub_n[(size_t)ord[k]], plan->h_sub_b[(size_t)ord[k]]);
  }
  // one CTA per SM at most, each group of them with kSlots submatrices in flight (one scratch sub-slot each)
  const int group = f8 ? 1 : group_size(S->ord_mean);   // (E4M3: a turn writes the pair that it finishes)
  const int slots = group_slots(group, work, sms);
  if (streamed && (!S->planes.p || S->R < R || S->LD < LD || S->slots < slots)) {
    const int nR = std::max(R, S->R), nLD = std::max(LD, S->LD), nS = std::max(slots, S->slots);
    dev_free(plan, S->planes);
    NOLSM_TRY(dev_alloc(plan, S->planes, sizeof(uint16_t) * (size_t)kPlanes * nS * nR * nLD));
    S->R = nR;
    S->LD = nLD;
    S->slots = nS;
  }
  NOLSM_CUDA_TRY(cudaMemsetAsync(plan->counter.p, 0, sizeof(int32_t), st));
  NOLSM_CUDA_TRY(cudaMemsetAsync(S->err.p, 0, sizeof(int32_t), st));
  TcArgs g{};
  if (spec.list) {   // an explicit work list (reruns): in list order
    g.j0 = 0; g.j1 = spec.count;
    g.order = spec.list;
  } else {
    g.j0 = (int32_t)j0; g.j1 = (int32_t)j1;
    g.order = S->order.as<int32_t>();
  }
  g.sub_n = plan->sub_n.as<int32_t>(); g.nbf = plan->sub_b.as<int32_t>();
  g.a_off = plan->a_off.as<int64_t>(); g.c_off = plan->c_off.as<int64_t>();
  // the symmetric form iterates on M and its centre-column phase uses W_c = L^-1 E_c in place of Q
  const bool sym = prep_class(o) == kPrepSym;
  g.A = prepared(plan, prep_class(o)).A.as<float>();
  g.Q = sym ? plan->Wc.as<double>() : plan->Q.as<double>();
  g.Sc = plan->Sc.as<double>(); g.Hc = plan->Hc.as<double>();
  g.lam = spec.lam ? spec.lam : plan->lam.as<double>();
  g.lam_g = plan->lam.as<double>();
  g.prep_status = plan->prep_status.as<int32_t>();
  g.mu = mu;
  g.tol_ns = (float)o.tol_ns; g.tol_accept = (float)o.tol_accept;
  g.max_iter = o.max_iter; g.refine_steps = o.refine_steps;
  g.budget = spec.budget;
  g.main_fmt = mf; g.refine_fmt = rf;
  g.planes = S->planes.as<uint16_t>();
  g.R = S->R; g.LD = S->LD;
  g.next = plan->counter.as<int32_t>();
  g.err = S->err.as<int32_t>();
  g.Dc = plan->Dc.as<double>(); g.tS = plan->t_S.as<double>(); g.tH = plan->t_H.as<double>();
  g.iters = plan->iters.as<int32_t>(); g.status = plan->status.as<int32_t>();
  g.rsteps = plan->rsteps.as<int32_t>();
  g.nbelow = plan->nbelow.as<int32_t>();
  g.wait_ns = o.wait_ns > 0 ? (uint64_t)o.wait_ns : kWaitNs;
  g.cond = sym ? nullptr : prepared(plan, prep_class(o)).cond.as<float>();
  g.cond_max = cond_max(o.precision);
  g.ill_max_n = prepare_fp64_max_n();
  g.above_n = above;
  g.group = group;
  g.groups = S->groups.as<GroupSlot>();
  // every submatrix of a launch starts as "timed out" (k_status_pending), the kernel overwrites what it takes
  int32_t* status = plan->status.as<int32_t>();
  auto pending = [&](const int32_t* list, int32_t count) -> nolsm_status {
    k_status_pending<<<(unsigned)std::min<int64_t>(1024, ((int64_t)count + 255) / 256), 256, 0, st>>>(0, count, list,
                                                                                                        status);
    NOLSM_LAUNCH_CHECK();
    return NOLSM_OK;
  };
  const int32_t* order = spec.list ? spec.list : S->order.as<int32_t>();
  NOLSM_TRY(pending(order, (int32_t)work));
  if (streamed) {
    TcMaps m;
    NOLSM_TRY(make_maps(&m, S->planes.p, S->R, S->LD, S->slots * kPlanes, f8));
    if (spec.list) {   // reruns and a bisection's later points: one launch in list order, shape 0
      NOLSM_TRY(launch_shape(0, 0, m, g, sms, st));
    } else {           // E4M3: all of the order; else those above 192 rows
      NOLSM_TRY(run_largest_first(0, o.precision, f8, m, g, S->order.as<int32_t>(), f8 ? (int32_t)work : S->ord_large,
                                  S->ord_mean, sms, st, pending));
    }
  }
  if (resident) {
    ResSolve r{};
    r.order = spec.list ? spec.list : S->order.as<int32_t>() + S->ord_large;
    r.count = spec.list ? spec.count : (int32_t)work - S->ord_large;
    r.sub_n = g.sub_n; r.nbf = g.nbf; r.a_off = g.a_off; r.c_off = g.c_off;
    r.A = g.A; r.Q = g.Q; r.Sc = g.Sc; r.Hc = g.Hc; r.lam = g.lam; r.lam_g = g.lam_g;
    r.prep_status = g.prep_status;
    r.mu = mu;
    r.tol_ns = g.tol_ns; r.tol_accept = g.tol_accept;
    r.max_iter = g.max_iter; r.refine_steps = g.refine_steps; r.budget = g.budget;
    r.main_fmt = mf;
    r.exact_xq = S->ord_exact;
    r.next = plan->counter.as<int32_t>() + 1; r.err = g.err;
    r.Dc = g.Dc; r.tS = g.tS; r.tH = g.tH; r.iters = g.iters; r.status = g.status; r.rsteps = g.rsteps;
    r.nbelow = g.nbelow;
    r.wait_ns = g.wait_ns;
    r.cond = g.cond; r.cond_max = g.cond_max; r.ill_max_n = g.ill_max_n;
    NOLSM_TRY(launch_ns_res(r, sms, st));
    resident_shape(0, o.precision);
    plan->stats.launches += 1;
  }
  plan->stats.launches += 2;
  if (sym) {   // D_c = L^-T U and the traces
    SymArgs a;
    a.j0 = (int32_t)j0;
    a.list = spec.list;
    a.sub_n = plan->sub_n.as<int32_t>(); a.nbf = plan->sub_b.as<int32_t>();
    a.a_off = plan->a_off.as<int64_t>(); a.c_off = plan->c_off.as<int64_t>();
    a.prep_status = plan->prep_status.as<int32_t>();
    a.L = plan->Lsym.as<float>();
    a.Sc = plan->Sc.as<double>(); a.Hc = plan->Hc.as<double>();
    a.Dc = plan->Dc.as<double>(); a.tS = plan->t_S.as<double>(); a.tH = plan->t_H.as<double>();
    a.status = plan->status.as<int32_t>();
    NOLSM_TRY(launch_sym_finish(a, (int)work, maxn, plan->max_b, st));
    plan->stats.launches += 1;
  }
  return NOLSM_OK;
}

bool ns_inverse_ready() {
  return inv_res_ready() && split_ok(reinterpret_cast<const void*>(&k_ns_tc<1, 0>), Shape<0>::kRegsLaunch) &&
         split_ok(reinterpret_cast<const void*>(&k_ns_tc<1, 1>), Shape<1>::kRegsLaunch);
}

// a2-a3 on the tensor cores for the chunk's submatrices order[0, count) (gathered into args.ws): A_J into
// Aout, T_J(S)^-1 into Xout, prep_out[J] = kSubOk or kSubRefine. Adds the products' flops to the stats.
nolsm_status launch_ns_inverse(nolsm_plan* plan, const NsInvArgs& a, cudaStream_t st) {
  if (a.count <= 0) return NOLSM_OK;
  TcState* S = state(plan);
  int dev = 0, sms = 0;
  NOLSM_CUDA_TRY(cudaGetDevice(&dev));
  NOLSM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (!S->err.p) NOLSM_TRY(dev_alloc(plan, S->err, sizeof(int32_t) * 4));
  if (!S->groups.p) NOLSM_TRY(dev_alloc(plan, S->groups, sizeof(GroupSlot) * kSlots * sms));
  if (!S->inv_flops.p) NOLSM_TRY(dev_alloc(plan, S->inv_flops, sizeof(double) * 2));
  NOLSM_CUDA_TRY(cudaMemsetAsync(plan->counter.p, 0, sizeof(int32_t), st));
  NOLSM_CUDA_TRY(cudaMemsetAsync(S->err.p, 0, sizeof(int32_t) * 4, st));
  NOLSM_CUDA_TRY(cudaMemsetAsync(S->inv_flops.p, 0, sizeof(double) * 2, st));
  // every submatrix of a launch starts as "timed out" and the kernel overwrites what it takes. (The first call in a
  // process also counts the flops of the shape measurements.)
  auto pending = [&](const int32_t* list, int32_t count) -> nolsm_status {
    k_status_pending<<<(unsigned)std::min(1024, (count + 255) / 256), 256, 0, st>>>(0, count, list, a.prep_out);
    NOLSM_LAUNCH_CHECK();
    return NOLSM_OK;
  };
  auto read_back = [&](int32_t* again) -> nolsm_status {   // adds up the flops; how many k_inv_res has left
    double fl[2];
    NOLSM_CUDA_TRY(cudaMemcpyAsync(fl, S->inv_flops.p, sizeof(fl), cudaMemcpyDeviceToHost, st));
    NOLSM_CUDA_TRY(cudaMemcpyAsync(again, S->err.as<int32_t>() + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    NOLSM_CUDA_TRY(cudaStreamSynchronize(st));
    plan->stats.flops_prep_tensor += fl[0];
    plan->stats.flops_prep_tensor_issued += fl[1];
    return NOLSM_OK;
  };
  // n of at most kResMaxN: operands on the SM (res_path.cu)
  const int32_t n_small = a.count - a.n_large;
  if (n_small > 0) {
    InvSolve r{};
    r.order = a.order + a.n_large; r.count = n_small;
    r.sub_n = plan->sub_n.as<int32_t>(); r.a_off = plan->a_off.as<int64_t>();
    r.ws = a.ws; r.a_base = a.a_base; r.chunk_n2 = a.chunk_n2;
    r.Aout = a.Aout; r.Xout = a.Xout; r.prep_out = a.prep_out;
    r.tol_inv = a.tol_inv; r.max_inv = a.max_inv;
    r.next = plan->counter.as<int32_t>() + 1;
    if (S->again.bytes < sizeof(int32_t) * (size_t)n_small) {
      dev_free(plan, S->again);
      NOLSM_TRY(dev_alloc(plan, S->again, sizeof(int32_t) * (size_t)n_small));
    }
    r.err = S->err.as<int32_t>(); r.again = S->err.as<int32_t>() + 1;
    r.again_list = S->again.as<int32_t>();
    r.flops = S->inv_flops.as<double>();
    NOLSM_TRY(pending(r.order, n_small));
    NOLSM_TRY(launch_inv_res(r, sms, st));
    resident_shape(1, NOLSM_FP16);
    plan->stats.launches += 2;
  }
  // the others, and those that need more than two steps, with operands in scratch
  auto streamed = [&](const int32_t* order, int32_t count, bool again) -> nolsm_status {
    const int max_n = again ? std::min(a.max_n, kResMaxN) : a.max_n;
    const int LD = (max_n + 63) & ~63, R = (max_n + 127) & ~127;
    // the few that k_inv_res left: several CTAs each while there are enough, as the start of one dominates
    const int group = !again ? group_size(a.mean_n) : 2 * count <= sms ? 4 : count <= sms ? 2 : 1;
    const int slots = group_slots(group, count, sms);
    if (!S->inv_planes.p || S->iR < R || S->iLD < LD || S->islots < slots) {
      const int nR = std::max(R, S->iR), nLD = std::max(LD, S->iLD), nS = std::max(slots, S->islots);
      dev_free(plan, S->inv_planes);
      NOLSM_TRY(dev_alloc(plan, S->inv_planes, sizeof(uint16_t) * (size_t)kPlanesInv * nS * nR * nLD));
      S->iR = nR;
      S->iLD = nLD;
      S->islots = nS;
    }
    TcMaps m;
    NOLSM_TRY(make_maps(&m, S->inv_planes.p, S->iR, S->iLD, S->islots * kPlanesInv, false));
    TcArgs g{};
    g.j0 = 0; g.j1 = count;
    g.order = order;
    g.sub_n = plan->sub_n.as<int32_t>(); g.nbf = plan->sub_b.as<int32_t>();
    g.a_off = plan->a_off.as<int64_t>(); g.c_off = plan->c_off.as<int64_t>();
    g.main_fmt = Fmt{FMT_F16, 3}; g.refine_fmt = g.main_fmt;
    g.planes = S->inv_planes.as<uint16_t>();
    g.R = S->iR; g.LD = S->iLD;
    g.next = plan->counter.as<int32_t>();
    g.err = S->err.as<int32_t>();
    g.ws = a.ws; g.a_base = a.a_base; g.chunk_n2 = a.chunk_n2;
    g.Aout = a.Aout; g.Xout = a.Xout; g.prep_out = a.prep_out;
    g.tol_inv = a.tol_inv; g.max_inv = a.max_inv;
    g.group = group;
    g.groups = S->groups.as<GroupSlot>();
    g.wait_ns = kWaitNs;
    g.flops = S->inv_flops.as<double>();
    plan->stats.launches += 2;
    if (again) {
      NOLSM_TRY(pending(order, count));
      return launch_shape(1, 0, m, g, sms, st);
    }
    return run_largest_first(1, NOLSM_FP16, false, m, g, order, count, a.mean_n, sms, st, pending);
  };
  if (a.n_large > 0) NOLSM_TRY(streamed(a.order, a.n_large, false));
  int32_t again = 0;
  NOLSM_TRY(read_back(&again));
  if (again > 0) {
    NOLSM_CUDA_TRY(cudaMemsetAsync(S->inv_flops.p, 0, sizeof(double) * 2, st));
    NOLSM_TRY(streamed(S->again.as<int32_t>(), again, true));
    NOLSM_TRY(read_back(&again));
  }
  return NOLSM_OK;
}

// ==================================================================================== no-allocation entry point
// Some callers cannot call cudaMalloc at the moment they need a sign iteration: an MD engine or other
// host framework that owns every byte of device memory through its own pool, or code that must not
// allocate while it runs (fixed memory budgets, allocation-free inner loops). For them the tensor-core
// kernel above can also run on scratch that lives in this file's static device array instead of a
// plan's workspaces. Every GPU that loads the library holds the array until the process exits.

namespace {

constexpr int kNaMaxN = 192;                  // largest submatrix dimension accepted
constexpr int kNaR = 256, kNaLD = 192;        // scratch plane shape: rows rounded to 128, columns to 64
constexpr int kNaSlots = 4 * kSlots;          // scratch sub-slots: 4 CTAs with kSlots each
constexpr int kNaMaxSub = 4096;               // submatrices per call
constexpr size_t kNaPlaneElems = (size_t)kNaR * kNaLD;
constexpr size_t kNaPlanesBytes = sizeof(uint16_t) * kPlanes * kNaSlots * kNaPlaneElems;
constexpr size_t kNaIntBytes = sizeof(int32_t) * (3 * (size_t)kNaMaxSub + 64);
constexpr size_t kNaBytes = kNaPlanesBytes + kNaIntBytes;   // about 4.8 MB

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaBytes];

// Identity work order, zero factorisation status, zero counters: what the kernel expects to find. Every
// caller status starts as "timed out": the kernel overwrites it for each submatrix it takes, so one that
// no block reached (all of them gave up on a wait) cannot keep a stale OK from an earlier call.
__global__ void k_noalloc_reset(unsigned char* base, int count, int32_t* status) {
  int32_t* ints = reinterpret_cast<int32_t*>(base + kNaPlanesBytes);
  int32_t* order = ints;
  int32_t* prep = ints + kNaMaxSub;
  int32_t* rst = ints + 2 * kNaMaxSub;
  int32_t* ctr = ints + 3 * kNaMaxSub;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    order[i] = i;
    prep[i] = kSubOk;
    rst[i] = 0;
    status[i] = kSubTimeout;
  }
  if (blockIdx.x == 0 && threadIdx.x < 64) ctr[threadIdx.x] = 0;
}

// device address of the static array per device ordinal, looked up by the first call on that device
std::atomic<void*> g_na_addr[64];

}  // namespace

}  // namespace nolsm

extern "C" nolsm_status nolsm_sign_noalloc(int32_t count, const int32_t* sub_n, const int32_t* nbf,
                                           const int64_t* a_off, const int64_t* c_off, const float* A, const double* Q,
                                           const double* Sc, const double* Hc, const double* lam, double mu,
                                           const nolsm_options* opts, nolsm_stream_t stream, double* Dc,
                                           double* t_S, double* t_H, int32_t* iters, int32_t* status) {
  using namespace nolsm;
  cudaStream_t st = (cudaStream_t)stream;
  if (!opts || !sub_n || !nbf || !a_off || !c_off || !A || !Q || !Sc || !Hc || !lam || !Dc || !t_S || !t_H ||
      !iters || !status || !std::isfinite(mu)) {
    set_error("nolsm_sign_noalloc: NULL argument or non-finite mu");
    return NOLSM_ERR_ARG;
  }
  if (count < 1 || count > kNaMaxSub) {
    set_error("nolsm_sign_noalloc: %d submatrices requested; this entry point takes 1..%d per call", count,
              kNaMaxSub);
    return NOLSM_ERR_UNSUPPORTED;
  }
  Fmt mf, rf;
  if (!formats(opts->precision, &mf, &rf) || mf.fmt == FMT_E4M3) {
    set_error("nolsm_sign_noalloc: precision %d is not available here (E4M3 needs the symmetric form)",
              opts->precision);
    return NOLSM_ERR_UNSUPPORTED;
  }
  if (opts->max_iter < 1 || opts->refine_steps < 0 || !(opts->tol_ns > 0) || !(opts->tol_accept > 0)) {
    set_error("nolsm_sign_noalloc: invalid options");
    return NOLSM_ERR_ARG;
  }
  // sizes are checked against the static scratch before anything is launched
  int32_t h_n[kNaMaxSub];
  NOLSM_CUDA_TRY(cudaMemcpyAsync(h_n, sub_n, sizeof(int32_t) * count, cudaMemcpyDeviceToHost, st));
  NOLSM_CUDA_TRY(cudaStreamSynchronize(st));
  for (int i = 0; i < count; ++i) {
    if (h_n[i] < 1 || h_n[i] > kNaMaxN) {
      set_error("nolsm_sign_noalloc: submatrix %d has dimension %d; this entry point takes 1..%d", i, h_n[i],
                kNaMaxN);
      return NOLSM_ERR_UNSUPPORTED;
    }
  }
  // once per device: the device address of this file's static scratch array
  int dev = 0;
  NOLSM_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    set_error("nolsm_sign_noalloc: device ordinal %d out of range", dev);
    return NOLSM_ERR_UNSUPPORTED;
  }
  void* addr = g_na_addr[dev].load(std::memory_order_acquire);
  if (!addr) {   // threads that race here look up the same address
    NOLSM_CUDA_TRY(cudaGetSymbolAddress(&addr, g_noalloc_scratch));
    g_na_addr[dev].store(addr, std::memory_order_release);
  }
  unsigned char* base = static_cast<unsigned char*>(addr);
  int32_t* ints = reinterpret_cast<int32_t*>(base + kNaPlanesBytes);

  TcMaps m;
  NOLSM_TRY(make_maps(&m, base, kNaR, kNaLD, kNaSlots * kPlanes, false));
  k_noalloc_reset<<<(count + 255) / 256, 256, 0, st>>>(base, count, status);
  NOLSM_LAUNCH_CHECK();
  TcArgs g{};
  g.j0 = 0; g.j1 = count;
  g.order = ints;
  g.sub_n = sub_n; g.nbf = nbf; g.a_off = a_off; g.c_off = c_off;
  g.A = A; g.Q = Q; g.Sc = Sc; g.Hc = Hc; g.lam = lam; g.lam_g = lam;
  g.prep_status = ints + kNaMaxSub;
  g.mu = mu;
  g.tol_ns = (float)opts->tol_ns; g.tol_accept = (float)opts->tol_accept;
  g.max_iter = opts->max_iter; g.refine_steps = opts->refine_steps;
  g.budget = nullptr;
  g.main_fmt = mf; g.refine_fmt = rf;
  g.planes = reinterpret_cast<uint16_t*>(base);
  g.R = kNaR; g.LD = kNaLD;
  g.next = ints + 3 * kNaMaxSub;
  g.err = ints + 3 * kNaMaxSub + 32;
  g.Dc = Dc; g.tS = t_S; g.tH = t_H; g.iters = iters; g.status = status;
  g.rsteps = ints + 2 * kNaMaxSub;
  g.group = 1;
  g.nbelow = nullptr;
  g.wait_ns = opts->wait_ns > 0 ? (uint64_t)opts->wait_ns : kWaitNs;
  NOLSM_CUDA_TRY(cudaFuncSetAttribute((k_ns_tc<0, 0>), cudaFuncAttributeMaxDynamicSharedMemorySize, Shape<0>::kSmemBytes));
  NOLSM_TRY(check_register_split(reinterpret_cast<const void*>(&k_ns_tc<0, 0>), Shape<0>::kRegsLaunch));
  k_ns_tc<0, 0><<<std::min(kNaSlots / kSlots, (count + kSlots - 1) / kSlots), Shape<0>::kThreads, Shape<0>::kSmemBytes, st>>>(m, g);
  NOLSM_LAUNCH_CHECK();
  return NOLSM_OK;
}
