// The FP64 sign iteration (a4-a7) on the tensor cores, by error-free splitting of its products.
//
// A matrix is held in fixed point with one exponent E for all its entries, x = m 2^E with |m| < 1, and m as kD
// signed digits of kB bits (balanced, so that a digit is at most 2^(kB-1) in magnitude):
//   m = sum_p d_p 2^-(kB - 1 + kB p).
// A digit is a small integer, exact in FP16, and a product of two matrices is the sum over digit pairs (p, q) of
// integer matrix products D_p E_q. Pairs of equal p + q = l share one FP32 accumulator in tensor memory; as long
// as its integers stay below 2^24 every FP32 addition is exact (the splitting of Ozaki, Ogita, Oishi and Rump,
// Numer. Algorithms 59 (2012), on tensor cores as in Mukunoki, Ozaki, Ogita and Imamura, ISC 2020). The pairs with
// l < kD are kept, kD (kD + 1) / 2 products; what is left out is about (K kD)^1/2 2^-kB kD of the scale, 5e-18 for 9
// bits and 7 digits at K = 200. The epilogue adds the accumulators in 64-bit integers,
// so 3I - P, the halving of X T and the next operands' digits are integer work, and the FP64 pipe (two lanes per
// clock and SM on this GPU) only scales X_0 and forms the centre columns.
//
// Two CTAs (a cluster) share one submatrix: the 128 x 64 output tiles of every product are dealt to them
// alternately, all kD accumulators of a tile in tensor memory together, so that each operand digit that TMA
// brings in is used by every pair it belongs to (kD (kD + 1) / 2 MMAs per 2 kD tiles). Roles: warp 0 (one thread)
// TMA loads, warp 1 (one thread) MMAs, warps 4-11 the epilogue. The CTAs meet on a barrier in each other's shared
// memory after every product, which also carries the parts of the defect and the overflow flags; every role then
// takes the same decision by itself. All three roles of both CTAs arrive, loader and MMA warp when they begin to wait:
// so none is more than one meeting behind (the records are kept for two), also where nothing else holds it, as in a
// CTA that has no tile (n up to 64), between a finish and the next start, or after a start that gave up; and every role
// has looked a submatrix's status up before an epilogue writes it. All waits are bounded.
//
// The second mode prepares A_J = T_J(S)^-1 T_J(H0) and the centre columns of T_J(S)^-1 for the same path, from the FP32
// inverse X of the inverse-square-root kernel (good to about 1e-6): R = I - T_J(S) X, V = I + R (I + R), X <- X V, whose
// error is about R^3 (again from R when ||R||_F was above kOzLast), then A_J = X T_J(H0).
//
// What the fixed point does not hold, or not as accurately (Fixed), is left to the FP64 kernels (k_ns_fp64; in the second
// mode k_prepare), which run afterwards on the submatrices still marked kSubRefine: non-finite input, entries that outgrow
// every exponent tried, an accumulator at 2^24, an FP32 inverse too far off, or a wait that ran out.
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

#include "nolsm_internal.cuh"
#include "oz_path.cuh"
#include "prep.cuh"
#include "tcgen05.cuh"
#include "tmap.cuh"

namespace nolsm {

namespace {

constexpr int kOzThreads = 384;
constexpr int kOzEpi = 256;                  // epilogue threads (warps 4-11)
constexpr int kRegsLaunch = 168, kRegsLow = 56, kRegsEpi = 224;
static_assert(128 * kRegsLow + kOzEpi * kRegsEpi <= kOzThreads * kRegsLaunch, "register split above the launch");
constexpr uint64_t kOzWaitNs = 2000000000ull;
// Inverse mode: after an update from ||R||_F at most kOzLast the inverse is done: its cube is below 3.4e-15, and of that a
// direction gets its share of some sqrt(n) (an X whose ||R||_F is that small has rounding errors in all of them; the
// centre columns were 1.3e-16 off behind 1.35e-5). ||R||_F at or above Fixed::far, or no end after kOzRounds updates:
// the FP64 Cholesky takes the submatrix
constexpr float kOzLast = 1.5e-5f;
constexpr int kOzRounds = 4;
// operands in scratch: X, X', T; in inverse mode X, X', two that hold S (then V), R, H in turn, and I + R
constexpr int sets(int mode) { return mode == 0 ? 3 : 5; }

template <int kB_, int kD_>
struct Digits {
  static constexpr int kB = kB_, kD = kD_;
  static constexpr int F = (kB - 1) + kB * (kD - 1);        // fraction bits of the digits,
  static constexpr int U = 59;                              // and of m as a 64-bit integer: four bits above |m| < 1
  static constexpr int G = 2 * (kB - 1) + kB * (kD - 2);    // fraction bits of the last accumulator but one
  static_assert(F >= U && F <= 63 && G <= 62, "digits");
  static constexpr uint32_t kABytes = kD * 128 * 64;        // a stage: 128 rows x 32 k of every digit of A,
  static constexpr uint32_t kBBytes = kD * 32 * 128;        // 32 k x 64 columns of every digit of B
  static constexpr uint32_t kStage = kABytes + kBBytes;
  static constexpr int kStages = 3 * kStage <= 220 * 1024 ? 3 : 2;
  static constexpr int kSmem = kStages * kStage + 1024;
  static_assert(kD * 64 <= 512, "accumulators in tensor memory");
};

struct OzArgs {
  int32_t count;
  const int32_t* order;
  const int32_t* sub_n; const int32_t* nbf;
  const int64_t* a_off; const int64_t* c_off;
  const double* A; const double* Q; const double* Sc; const double* Hc; const double* lam; const double* lam_g;
  const int32_t* prep_status;
  double mu, tol;
  int32_t max_iter;
  const int32_t* budget;
  uint16_t* planes;            // per cluster 3 operands (X, X', T) of kD planes, each R x LD
  double* xd;                  // per cluster R x LD: the final X
  int32_t R, LD;
  double* Dc; double* tS; double* tH; int32_t* iters; int32_t* status; int32_t* rsteps; int32_t* nbelow;
  uint64_t wait_ns;
  Fixed lim;
  // inverse mode: the chunk's T_J(S), T_J(H0) (FP64, at a_off[J] - a_base and chunk_n2 further), X (FP32, at
  // a_off[J] - a_base), and the outputs
  const double* ws; int64_t a_base, chunk_n2;
  const float* X32;
  const int32_t* sub_c0;
  double* Aout; double* Qout;
  int32_t* prep_out;
};

// What the two CTAs tell each other at the end of a product (double buffered by its parity)
struct Record {
  float part[2];               // ||I - P||_F^2 of the CTA's tiles
  uint32_t bad[2];             // 1: an entry outgrew the exponent; 2: an accumulator may have rounded; 4: error
  double sum[2][3];            // t_S, t_H, Tr X of the CTA's rows (finish)
};

struct OzShared {
  uint64_t full[3], empty[3], accf, acce, done, idle;
  uint32_t tmem;
  int err;
  Record rec[2];
  float red[8];
  double dred[3][8];
  uint32_t ored;
};

__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool wait_cluster(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  const uint64_t deadline = tc::globaltimer() + limit_ns;
  for (;;) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(tc::smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (tc::globaltimer() > deadline) return false;
  }
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void oz_bar() { asm volatile("bar.sync 3, %0;" ::"n"(kOzEpi) : "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void st_global_256(void* p, const uint32_t (&v)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
               "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

// The balanced digits of two entries as packed FP16 pairs, out[p] for digit p. The bias makes every digit non-negative
// (u <= 2^kB below 1024), and 1024 + u is the FP16 number with bits 0x6400 | u.
template <class Dg>
__device__ __forceinline__ void digits2(long long a, long long b, uint32_t (&out)[Dg::kD]) {
  constexpr int kB = Dg::kB, kD = Dg::kD;
  constexpr uint32_t half = 1u << (kB - 1), mask = (1u << kB) - 1;
  long long bias = 0;
#pragma unroll
  for (int p = 0; p < kD; ++p) bias += (long long)half << (kB * (kD - 1 - p));
  const unsigned long long x = (unsigned long long)(a << (Dg::F - Dg::U)) + (unsigned long long)bias;
  const unsigned long long y = (unsigned long long)(b << (Dg::F - Dg::U)) + (unsigned long long)bias;
  const __half2 sub = __half2half2(__ushort_as_half((unsigned short)(0x6400u + half)));
#pragma unroll
  for (int p = 0; p < kD; ++p) {
    const int sh = kB * (kD - 1 - p);
    const uint32_t m = p == 0 ? 0x03FF03FFu : mask * 0x00010001u;
    const uint32_t pk = (__byte_perm((uint32_t)(x >> sh), (uint32_t)(y >> sh), 0x5410) & m) | 0x64006400u;
    const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&pk), sub);
    out[p] = *reinterpret_cast<const uint32_t*>(&d);
  }
}

// x 2^k rounded to the nearest integer (halves away from zero), by integer operations; |x| 2^k below 2^62.
__device__ __forceinline__ long long to_fixed(double x, int k) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7FF), sh = e - 1075 + k;
  unsigned long long m = ((unsigned long long)b & 0xFFFFFFFFFFFFFull) | (e ? 1ull << 52 : 0ull);
  if (sh >= 0) m <<= sh & 15;
  else m = sh < -60 ? 0ull : ((m >> (-sh - 1)) + 1) >> 1;
  return b < 0 ? -(long long)m : (long long)m;
}
__device__ __forceinline__ long long to_fixed(float x, int k) {
  const int b = __float_as_int(x), e = (b >> 23) & 0xFF, sh = e - 150 + k;
  unsigned long long m = ((uint32_t)b & 0x7FFFFFu) | (e ? 1u << 23 : 0u);
  if (sh >= 0) m <<= sh & 63;
  else m = sh < -30 ? 0ull : ((m >> (-sh - 1)) + 1) >> 1;
  return b < 0 ? -(long long)m : (long long)m;
}

// The MMAs of one 16-wide k step of a tile with kRows rows: every digit pair (p, q) with p + q < kD into accumulator
// p + q. The descriptors differ by constants alone: a thread that computes them at run time issues an MMA every 85
// cycles, and one of 128 x 64 takes 48 (32 with 64 rows).
template <class Dg, int kRows>
__device__ __forceinline__ void digit_pairs(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t id, bool first) {
  constexpr int kD = Dg::kD;
#pragma unroll
  for (int p = 0; p < kD; ++p)
#pragma unroll
    for (int q = 0; q + p < kD; ++q)
      tc::mma_f16(tmem + 64 * (p + q), ad + ((p * kRows * 64) >> 4), bd + ((q * 4096) >> 4), id, p > 0 || !first ? 1u : 0u);
}

__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

// kMode 0: the sign iteration; 1: the inverse of T_J(S) and A_J
template <class Dg, int kMode>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kOzThreads, 1)
    k_ns_oz(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapA64,
            const __grid_constant__ CUtensorMap mapB, OzArgs g) {
  constexpr int kB = Dg::kB, kD = Dg::kD, U = Dg::U, kStages = Dg::kStages;
  extern __shared__ uint8_t smraw[];
  uint8_t* stage_mem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  __shared__ OzShared sh;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int rank = (int)cta_rank(), cid = blockIdx.x >> 1, ncl = gridDim.x >> 1;
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      tc::mbar_init(&sh.full[s], 1);
      tc::mbar_init(&sh.empty[s], 1);
    }
    tc::mbar_init(&sh.accf, 1);
    tc::mbar_init(&sh.acce, kOzEpi);
    tc::mbar_init(&sh.done, 6);                // loader, MMA warp and epilogue of both CTAs
    tc::mbar_init(&sh.idle, 1);
    tc::fence_mbar_init();
    sh.err = 0;
    tc::prefetch_tmap(&mapA);
    tc::prefetch_tmap(&mapA64);
    tc::prefetch_tmap(&mapB);
  }
  if (warp == 0) {
    tc::tmem_alloc(&sh.tmem, 512);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  cluster_sync();   // the peer's barriers are initialised before anything arrives on them
  const uint32_t tmem = sh.tmem;
  const size_t plane_elems = (size_t)g.R * g.LD;
  const int zc = cid * sets(kMode) * kD;       // first plane of this cluster
  bool armed[3] = {false, false, false};
  uint32_t arm_phase[3] = {0, 0, 0};
  uint32_t kcount = 0, tcount = 0, ev = 0;     // stages, tiles and meetings so far (per role)

  // Every role follows the same course: per submatrix the start, then products, a meeting after each (mode 0: and the
  // end); after a meeting each takes the next step from the records.
  struct Course { int n, n16, nrb, ncb, cur, sp, steps, cap, tries, status; bool last, gave_up; };
  Course c;
  const bool mma_warp = warp == 1;
  auto arrive = [&]() {                        // one thread of a role
    const uint32_t done0 = tc::smem_u32(&sh.done);
    for (uint32_t to = 0; to < 2; ++to) arrive_cluster(mapa(done0, to));
  };
  auto meet = [&](Record& r) -> bool {         // waits for the meeting's end; false: give up
    if (warp < 4 && lane == 0) arrive();       // (the epilogue has arrived in tell)
    bool ok = !sh.err && wait_cluster(&sh.done, ev & 1, 8 * g.wait_ns);
    if (mma_warp) ok = __all_sync(0xffffffffu, ok);
    r = sh.rec[ev & 1];
    ++ev;
    return ok && !((r.bad[0] | r.bad[1]) & 4);
  };
  auto begin = [&](int J) -> bool {            // false: not taken here
    if (g.prep_status[J] != (kMode == 0 ? kSubOk : kSubPending)) return false;
    c.n = g.sub_n[J];
    c.n16 = (c.n + 15) & ~15;
    c.nrb = (c.n16 + 127) / 128;
    c.ncb = (c.n16 + 63) / 64;
    c.cap = kMode == 0 && g.budget ? min(g.max_iter, g.budget[J]) : g.max_iter;
    c.tries = 0;
    c.gave_up = false;
    return c.cap > 0;
  };
  // cur: which of the two X operands; sp: the operand that holds S (inverse mode: 2, R in 3, or the reverse)
  auto reset = [&]() { c.cur = 0; c.sp = 2; c.steps = 0; c.last = false; c.status = kSubNotConv; };
  // after the start or a new X. 0: go on, 1: start again (larger exponents), 2: finish
  auto after_x = [&](const Record& r) -> int {
    const uint32_t bad = r.bad[0] | r.bad[1];
    if (bad & 2) c.gave_up = true;
    else if (bad & 1) {
      if (++c.tries < g.lim.tries) return 1;
      c.gave_up = true;
    }
    return (c.gave_up || c.last) ? 2 : 0;
  };
  auto after_p = [&](const Record& r) {        // after X X (mode 0): the stopping rule; after S X: how far X is off
    const float sum = r.part[0] + r.part[1];
    c.steps += 1;
    if constexpr (kMode == 0) {
      if ((double)sqrtf(sum / (float)c.n) <= g.tol) {   // (the sum is good to 1e-6: a step more or less at that distance)
        c.last = true;
        c.status = kSubOk;
      } else if (c.steps >= c.cap) {
        c.last = true;
      }
    } else {
      const float far = sqrtf(sum);
      if (!(far < g.lim.far) || (far > kOzLast && c.steps >= kOzRounds)) c.gave_up = true;
      else if (far <= kOzLast) c.last = true;
    }
  };
  auto tail64 = [&](int mb) { return c.n16 - 128 * mb <= 64; };

  if (warp < 4) {
    tc::setmaxnreg_dec<kRegsLow>();
    if ((warp == 0 && lane == 0) || warp == 1) {   // one thread loads; the MMA warp runs converged, one lane issues
      // one product: A in operand set za, B in zb
      auto tiles = [&](int sa, int sb) -> bool {
        const int n32 = (c.n16 + 31) / 32;
        for (int t = rank; t < c.nrb * c.ncb; t += 2) {
          const int mb = t / c.ncb, cb = t - mb * c.ncb;
          const bool m64 = tail64(mb);
          const uint32_t rows = m64 ? 64 : 128;
          if (warp == 0) {
            for (int ks = 0; ks < n32; ++ks, ++kcount) {
              const int st = kcount % kStages;
              const uint32_t ph = (kcount / kStages) & 1;
              if (!tc::mbar_wait_ns(&sh.empty[st], ph ^ 1, g.wait_ns)) return false;
              uint8_t* sm = stage_mem + st * Dg::kStage;
              tc::mbar_arrive_expect_tx(&sh.full[st], kD * rows * 64 + Dg::kBBytes);
              armed[st] = true;
              arm_phase[st] = ph;
              tc::tma_load_3d(sm, m64 ? &mapA64 : &mapA, &sh.full[st], 32 * ks, 128 * mb, zc + sa * kD);
              tc::tma_load_3d(sm + Dg::kABytes, &mapB, &sh.full[st], 64 * cb, 32 * ks, zc + sb * kD);
            }
          } else {
            const uint32_t id = tc::idesc(0, 0, 0, 1, rows, min(64, c.n16 - 64 * cb));
            if (!__all_sync(0xffffffffu, tc::mbar_wait_ns(&sh.acce, (tcount & 1) ^ 1, g.wait_ns)))
              return false;
            tc::tc_fence_after();
            for (int ks = 0; ks < n32; ++ks, ++kcount) {
              const int st = kcount % kStages;
              if (!__all_sync(0xffffffffu, tc::mbar_wait_ns(&sh.full[st], (kcount / kStages) & 1, g.wait_ns)))
                return false;
              tc::tc_fence_after();
              const uint32_t a0 = __shfl_sync(0xffffffffu, tc::smem_u32(stage_mem + st * Dg::kStage), 0);
              const uint64_t ad = tc::sdesc_sw64(a0, 16, 512), bd = tc::sdesc_sw128(a0 + Dg::kABytes, 4096, 1024);
              if (tc::elect_one()) {
                for (int kk = 0; kk < 2 && 32 * ks + 16 * kk < c.n16; ++kk) {
                  const uint64_t ak = ad + ((kk * 32) >> 4), bk = bd + ((kk * 2048) >> 4);
                  if (m64) digit_pairs<Dg, 64>(tmem, ak, bk, id, ks == 0 && kk == 0);
                  else digit_pairs<Dg, 128>(tmem, ak, bk, id, ks == 0 && kk == 0);
                }
                tc::mma_commit(&sh.empty[st]);
              }
              __syncwarp();
            }
            if (tc::elect_one()) tc::mma_commit(&sh.accf);
            __syncwarp();
            ++tcount;
          }
        }
        return true;
      };
      auto product = [&](int sa, int sb) -> bool {
        if (tiles(sa, sb)) return true;
        sh.err = 1;                            // a wait ran out: the others meet once more without this role, and leave
        if (lane == 0) arrive();
        return false;
      };
      Record r;
      for (int k = cid; k < g.count; k += ncl) {
        if (!begin(g.order[k])) continue;
        reset();
        bool ok = true;
        for (;;) {
          if (!(ok = meet(r))) break;
          tc::fence_proxy_async_global();      // the epilogues' operand writes, before TMA reads them
          const int go = after_x(r);
          if (go == 1) {
            reset();
            continue;
          }
          if (go == 2) break;
          if constexpr (kMode == 0) {
            if (!(ok = product(c.cur, c.cur) && meet(r))) break;
            tc::fence_proxy_async_global();
            after_p(r);
            if (!(ok = product(c.cur, 2))) break;
            c.cur ^= 1;
          } else {
            if (!(ok = product(c.sp, c.cur) && meet(r))) break;      // R = I - S X
            tc::fence_proxy_async_global();
            after_p(r);
            if (c.gave_up) break;
            if (!(ok = product(5 - c.sp, 4) && meet(r))) break;      // V = I + R (I + R)
            tc::fence_proxy_async_global();
            if (!(ok = product(c.cur, c.sp))) break;                 // X' = X V
            c.cur ^= 1;
            c.sp = 5 - c.sp;                                         // S again (or H) in R's place
          }
        }
        if (kMode == 1 && ok && !c.gave_up) ok = product(c.cur, c.sp);   // A_J = X H
        if (!ok || ((kMode == 0 || !c.gave_up) && !meet(r))) {
          sh.err = 1;
          break;
        }
      }
    }
  } else {
    tc::setmaxnreg_inc<kRegsEpi>();
    const int etid = tid - 128, ew = warp - 4, q = warp & 3, grp = ew >> 2;
    uint16_t* const planes = g.planes + (size_t)zc * plane_elems;
    double* const xd = g.xd + (size_t)cid * plane_elems;
    const uint32_t rec0 = tc::smem_u32(&sh.rec[0]);
    int ex = 1, et = 2, es = 1, eh = 1;          // exponents of X, T (mode 0), S and H (inverse mode)

    // the CTA's part of the meeting: sums over its threads to both CTAs' records, then the arrivals
    auto tell = [&](float part, uint32_t bad, double s0, double s1, double s2, bool sums) {
      for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      bad = __reduce_or_sync(0xffffffffu, bad);
      if (sums) {
        for (int o = 16; o > 0; o >>= 1) {
          s0 += __shfl_xor_sync(0xffffffffu, s0, o);
          s1 += __shfl_xor_sync(0xffffffffu, s1, o);
          s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
      }
      if (lane == 0) {
        sh.red[ew] = part;
        if (bad) atomicOr(&sh.ored, bad);
        sh.dred[0][ew] = s0;
        sh.dred[1][ew] = s1;
        sh.dred[2][ew] = s2;
      }
      tc::fence_proxy_async_global();
      oz_bar();
      if (etid == 0) {
        float p = 0.0f;
        double t[3] = {0.0, 0.0, 0.0};
        for (int w = 0; w < 8; ++w) {
          p += sh.red[w];
          for (int u = 0; u < 3; ++u) t[u] += sh.dred[u][w];
        }
        const uint32_t b = sh.ored | (sh.err ? 4u : 0u);
        sh.ored = 0;
        for (uint32_t to = 0; to < 2; ++to) {
          const uint32_t at = mapa(rec0 + (ev & 1) * (uint32_t)sizeof(Record), to);
          st_cluster(at + 4 * rank, __float_as_uint(p));
          st_cluster(at + 8 + 4 * rank, b);
          for (int u = 0; u < 3; ++u) st_cluster(at + 16 + 24 * rank + 8 * u, t[u]);
        }
        arrive();
      }
    };

    // the largest |M_ij|, rounded up, of n x n entries (or, step n + 1, of the diagonal): by its leading bits
    auto largest = [&](const auto* M, int n, int step) -> double {
      uint32_t mx = 0;
#pragma unroll 8
      for (int e = etid * step; e < n * n; e += kOzEpi * step) {
        if constexpr (sizeof(*M) == 8) mx = max(mx, (uint32_t)__double2hiint(__ldg(M + e)) & 0x7FFFFFFFu);
        else mx = max(mx, __float_as_uint(__ldg(M + e)) & 0x7FFFFFFFu);
      }
      mx = __reduce_max_sync(0xffffffffu, mx);
      if (lane == 0) sh.red[ew] = __uint_as_float(mx);
      oz_bar();
      for (int w = 0; w < 8; ++w) mx = max(mx, __float_as_uint(sh.red[w]));
      oz_bar();
      return sizeof(*M) == 8 ? __hiloint2double((int)mx, -1) : (double)__uint_as_float(mx);
    };
    auto exponent = [](double big) {             // big < 2^e
      int e = 0;
      frexp(big, &e);
      return e;
    };
    // (M - mu I) inv (n x n, row-major) as the digits of operand `set` with exponent e, zero up to n16 rows and
    // columns: this CTA's half of the rows
    auto fill = [&](const auto* __restrict__ M, double mu, double inv, int set, int e) {
      const int n = c.n, n16 = c.n16;
      uint16_t* dst = planes + (size_t)set * kD * plane_elems;
      const int half = (n16 / 16 + 1) / 2 * 16;
      const int r0 = rank ? half : 0, r1 = rank ? n16 : half, w2 = n16 / 2;
      // four rows of a warp together: eight loads in flight per lane (no condition holds one back)
      for (int i0 = r0 + 4 * ew; i0 < r1; i0 += 32)
        for (int j = lane; j < w2; j += 32) {
          long long v[4][2];
          std::remove_cv_t<std::remove_reference_t<decltype(*M)>> x[4][2];
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int u = 0; u < 2; ++u) x[a][u] = __ldg(M + (size_t)min(i0 + a, n - 1) * n + min(2 * j + u, n - 1));
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int i = i0 + a, col = 2 * j + u;
              if constexpr (kMode == 0) x[a][u] = (x[a][u] - (i == col ? mu : 0.0)) * inv;
              v[a][u] = i < n && col < n ? to_fixed(x[a][u], U - e) : 0;
            }
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            if (i0 + a >= r1) break;
            uint32_t d[kD];
            digits2<Dg>(v[a][0], v[a][1], d);
#pragma unroll
            for (int p = 0; p < kD; ++p)
              *reinterpret_cast<uint32_t*>(dst + p * plane_elems + (size_t)(i0 + a) * g.LD + 2 * j) = d[p];
          }
        }
    };
    // The operands of a new submatrix (or of another attempt with larger exponents). Mode 0, a4: X_0 = (A - mu I) / alpha.
    // Inverse mode: X and S. Returns 2 when they cannot be represented.
    auto start = [&](int J) -> uint32_t {
      if constexpr (kMode == 0) {
        const double* A = g.A + g.a_off[J];
        const double inv = 1.0 / scale_alpha(g.lam, g.lam_g, J, g.mu);
        // the Gershgorin interval bounds every entry of A - mu I by its alpha, and alpha is at least 1/1.7 of that
        if (!isfinite(inv) || !isfinite(g.lam_g[2 * J]) || !isfinite(g.lam_g[2 * J + 1])) return 2;
        ex = 1 + 3 * c.tries;
        et = ex + 1;
        fill(A, g.mu, inv, 0, ex);
      } else {
        const int64_t at = g.a_off[J] - g.a_base;
        if (c.tries == 0) {
          // positive definite matrices have their largest entry on the diagonal (with anything else R gets large)
          const double bx = largest(g.X32 + at, c.n, c.n + 1), bs = largest(g.ws + at, c.n, c.n + 1);
          if (!isfinite(bx) || !isfinite(bs) || bx > 1e6 || bs > 1e6) return 2;
          ex = max(1, exponent(bx) + 1);
          es = max(-8, exponent(bs) + 1);
        } else {
          ex += 3;
        }
        fill(g.X32 + at, 0.0, 1.0, 0, ex);
        fill(g.ws + at, 0.0, 1.0, 2, es);
      }
      return 0;
    };

    // Drains this CTA's tiles of one product P into operand `so` (digits) or an FP64 array. Mode 0: kT (T = 3I - P and
    // the defect's sum), kX (P / 2), kXd (P / 2 in FP64: the last). Inverse mode: kR (R = I - P and I + R, the sum of
    // R^2), kV (I + P), kX (P; with last_q its centre columns in FP64 too), kA (P in FP64).
    enum : int { kT, kX, kXd, kR, kV, kA };
    auto drain = [&](int kind, int so, int J, bool last_q, float& part, uint32_t& bad) -> bool {
      const int n = c.n, n16 = c.n16;
      // exponents of the product's two operands together, and of the output
      const int ein = kMode == 0 ? (kind == kT ? 2 * ex : ex + et) : (kind == kR ? es + ex : kind == kX ? ex + 1 : kind == kA ? ex + eh : 1);
      const int eo = kMode == 0 ? (kind == kT ? et : ex + 1) : (kind == kR ? 0 : kind == kX ? ex : kind == kA ? ex + eh : 1);
      const int s = ein - eo;
      const long long one = 1ll << (U - eo);
      const float down = pow2f(eo - U);
      // the first accumulator (2^(2 kB - 2) times the product) below this: no wrap in 64 bits
      const float most0 = fminf(pow2f(62 - kB * (kD - 2)), pow2f(3 - s + 2 * (kB - 1)));
      const int shl = U + s - Dg::G;           // from the last accumulator but one to the output's units
      for (int t = rank; t < c.nrb * c.ncb; t += 2, ++tcount) {
        const int mb = t / c.ncb, cb = t - mb * c.ncb;
        bool ok = tc::mbar_wait_ns(&sh.accf, tcount & 1, g.wait_ns);
        if (!__all_sync(0xffffffffu, ok)) return false;
        tc::tc_fence_after();
        const bool m64 = tail64(mb);
        const int rbase = 128 * mb + (m64 ? 16 : 32) * q, row = rbase + lane;
        const bool rok = (!m64 || lane < 16) && row < n16;
        const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + 32 * grp;
        const int colg = 64 * cb + 32 * grp;
        long long v[32];
        uint32_t ov = 0;
        float big0 = 0.0f, big = 0.0f;         // the largest first accumulator, and of the next (all but the last two)
        if (rbase < n16 && colg < n16) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (colg + 16 * h >= n16) {        // columns the MMAs left out hold anything
#pragma unroll
              for (int j = 0; j < 16; ++j) v[16 * h + j] = 0;
              break;
            }
            uint32_t r[kD][16];
#pragma unroll
            for (int l = 0; l < kD; ++l) tmem_ld16(ta + 64 * l + 16 * h, r[l]);
            tc::tmem_wait_ld();
            // sum of the accumulators in units of the last but one: those up to 30 bits above it as 32 x 32 -> 64 bit
            // multiply-adds, the rest into the high word
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              int a[kD];
#pragma unroll
              for (int l = 0; l < kD; ++l) {
                const float f = __uint_as_float(r[l][j]);
                if (l == 0) big0 = fmaxf(big0, fabsf(f));
                else if (l < kD - 2) big = fmaxf(big, fabsf(f));
                a[l] = __float2int_rn(f);
              }
              long long w = (long long)a[kD - 2] + ((a[kD - 1] + (1 << (kB - 1))) >> kB);
              int hi = 0;
#pragma unroll
              for (int l = kD - 3; l >= 0; --l) {
                const int up = kB * (kD - 2 - l);
                if (up <= 30) w += (long long)a[l] * (1 << (up & 31));
                else hi += (int)((uint32_t)a[l] << ((up - 32) & 31));
              }
              w += (long long)hi << 32;
              v[16 * h + j] = shl >= 0 ? w << shl : (w + (1ll << (-shl - 1))) >> -shl;
            }
          }
        }
        tc::tc_fence_before();
        tc::mbar_arrive(&sh.acce);
        if (rbase < n16 && colg < n16) {
          const bool rin = rok && row < n;
          if (rin && !(big < 16777216.0f)) bad |= 2;
          if (rin && !(big0 < most0)) bad |= 1;
          // rows and columns from n to n16 are zeros of themselves, their operands' being zeros
          const bool dia = rin && row >= colg && row < colg + 32 && kind != kX && kind != kXd && kind != kA;
          float sq = 0.0f;
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            long long a = v[j];
            if (kind == kT || kind == kR) {
              a = -a;
              if (dia) a += row == colg + j ? one : 0;               // (I - P)_ij
              const float ef = down * (float)a;
              sq = fmaf(ef, ef, sq);
              if (dia && kind == kT) a += row == colg + j ? 2 * one : 0;
            } else if (kind == kV) {
              if (dia) a += row == colg + j ? one : 0;
            }
            const int hi = (int)(a >> 32);
            ov |= (uint32_t)(hi ^ (hi >> 31));
            v[j] = a;
          }
          if (rin) part += sq;
          if (rin && (ov >> (U - 32)) != 0 && kind != kXd && kind != kA) bad |= 1;
          if (rok) {
            if (kMode == 0 && kind == kXd) {
              const double to = pow2(ex - U);
              double* dst = xd + (size_t)row * g.LD + colg;
#pragma unroll
              for (int j = 0; j < 32; j += 2)
                *reinterpret_cast<double2*>(dst + j) = make_double2((double)v[j] * to, (double)v[j + 1] * to);
            } else if (kMode == 1 && kind == kA) {
              if (rin) {
                const double to = pow2(eo - U);
                double* dst = g.Aout + g.a_off[J] + (size_t)row * n + colg;
#pragma unroll
                for (int j = 0; j < 32; ++j)
                  if (colg + j < n) dst[j] = (double)v[j] * to;
              }
            } else {
              // the digits; after R also those of I + R (exponent 1)
              int set = so;
#pragma unroll 1
              for (int again = kMode == 1 && kind == kR ? 1 : 0; again >= 0; --again) {
                uint16_t* dst = planes + (size_t)set * kD * plane_elems + (size_t)row * g.LD + colg;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  uint32_t o[kD][8];
#pragma unroll
                  for (int j = 0; j < 8; ++j) {
                    uint32_t d[kD];
                    digits2<Dg>(v[16 * h + 2 * j], v[16 * h + 2 * j + 1], d);
#pragma unroll
                    for (int p = 0; p < kD; ++p) o[p][j] = d[p];
                  }
#pragma unroll
                  for (int p = 0; p < kD; ++p) st_global_256(dst + p * plane_elems + 16 * h, o[p]);
                }
                if (kMode == 1 && again) {
                  set = 4;
#pragma unroll
                  for (int j = 0; j < 32; ++j) v[j] = (v[j] + (dia && row == colg + j ? 1ll << U : 0) + 1) >> 1;
                }
              }
            }
            if (kMode == 1 && kind == kX && last_q && rin) {
              const int c0 = g.sub_c0[J], b = g.nbf[J];
              const double to = pow2(ex - U);
              double* Q = g.Qout + g.c_off[J] + (size_t)row * b;
              if (colg < c0 + b && colg + 32 > c0) {
#pragma unroll
                for (int j = 0; j < 32; ++j)
                  if (colg + j >= c0 && colg + j < c0 + b) Q[colg + j - c0] = (double)v[j] * to;
              }
            }
          }
        }
      }
      return true;
    };

    Record r;
    if (etid == 0) sh.ored = 0;
    oz_bar();
    for (int k = cid; k < g.count; k += ncl) {
      const int J = g.order[k];
      if (!begin(J)) continue;
      reset();
      bool ok = true;
      uint32_t bad = start(J);
      tell(0.0f, bad, 0.0, 0.0, 0.0, false);
      for (;;) {
        if (!(ok = meet(r))) break;
        const int go = after_x(r);
        if (go == 1) {
          reset();
          bad = start(J);
          tell(0.0f, bad, 0.0, 0.0, 0.0, false);
          continue;
        }
        if (go == 2) break;
        float part = 0.0f;
        bad = 0;
        if constexpr (kMode == 0) {
          ok = drain(kT, 2, J, false, part, bad);
          tell(part, bad | (ok ? 0u : 4u), 0.0, 0.0, 0.0, false);
          if (!(ok = meet(r) && ok)) break;
          bad = (r.bad[0] | r.bad[1]) & 3;     // an overflow in T counts with X T's
          after_p(r);
          ok = drain(c.last ? kXd : kX, c.cur ^ 1, J, false, part, bad);
          tell(0.0f, bad | (ok ? 0u : 4u), 0.0, 0.0, 0.0, false);
          if (!ok) break;
          c.cur ^= 1;
        } else {
          if (c.steps == 0 && c.tries == 0) {  // while the MMAs form S X
            const double bh = largest(g.ws + g.chunk_n2 + g.a_off[J] - g.a_base, c.n, 1);
            if (!isfinite(bh) || bh > 1e6) bad = 2;
            eh = max(-8, exponent(bh));
          }
          ok = drain(kR, 5 - c.sp, J, false, part, bad);
          tell(part, bad | (ok ? 0u : 4u), 0.0, 0.0, 0.0, false);
          if (!(ok = meet(r) && ok)) break;
          uint32_t all = (r.bad[0] | r.bad[1]) & 3;
          after_p(r);
          if (c.gave_up) break;
          bad = all;
          ok = drain(kV, c.sp, J, false, part, bad);
          tell(0.0f, bad | (ok ? 0u : 4u), 0.0, 0.0, 0.0, false);
          if (!(ok = meet(r) && ok)) break;
          bad = (r.bad[0] | r.bad[1]) & 3;
          const int64_t at = g.a_off[J] - g.a_base;
          // into R's place, while the MMAs form X V: S for another round, or H for A_J
          fill(g.ws + at + (c.last ? g.chunk_n2 : 0), 0.0, 1.0, 5 - c.sp, c.last ? eh : es);
          ok = drain(kX, c.cur ^ 1, J, c.last, part, bad);
          tell(0.0f, bad | (ok ? 0u : 4u), 0.0, 0.0, 0.0, false);
          if (!ok) break;
          c.cur ^= 1;
          c.sp = 5 - c.sp;
        }
      }
      if constexpr (kMode == 1) {
        float part = 0.0f;
        bad = 0;
        if (ok && !c.gave_up) {
          ok = drain(kA, 0, J, false, part, bad);
          tell(0.0f, bad | (ok ? 0u : 4u), 0.0, 0.0, 0.0, false);
          ok = meet(r) && ok;
        }
        if (!ok) {
          if (etid == 0) sh.err = 1;
          break;
        }
        if (rank == 0 && etid == 0) g.prep_out[J] = c.gave_up || (r.bad[0] | r.bad[1]) ? kSubRefine : kSubOk;
        continue;
      }
      if (!ok) {
        // the peer waits for this CTA's part of a meeting at most for its own limit
        if (etid == 0) sh.err = 1;
        break;
      }
      // a7: this CTA's half of the rows of the centre columns of T_J(D) = 1/2 (I - X) T_J(S)^-1, the partial traces
      double ps = 0.0, ph = 0.0, px = 0.0;
      if (!c.gave_up) {
        const int n = c.n, b = g.nbf[J];
        const int i0 = rank ? (n + 1) / 2 : 0, i1 = rank ? n : (n + 1) / 2;
        const double* Q = g.Q + g.c_off[J];
        const double* Sc = g.Sc + g.c_off[J];
        const double* Hc = g.Hc + g.c_off[J];
        double* Dc = g.Dc + g.c_off[J];
        for (int e = i0 * b + etid; e < i1 * b; e += kOzEpi) {
          const int i = e / b, col = e - i * b;
          const double* xi = xd + (size_t)i * g.LD;
          double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
          int kk = 0;
#pragma unroll 4
          for (; kk + 4 <= n; kk += 4) {   // 24 loads in flight: their latency is what a row of X costs
            const double2 xa = __ldcg(reinterpret_cast<const double2*>(xi + kk));
            const double2 xb = __ldcg(reinterpret_cast<const double2*>(xi + kk + 2));
            s0 = fma(xa.x, Q[(size_t)kk * b + col], s0);
            s1 = fma(xa.y, Q[(size_t)(kk + 1) * b + col], s1);
            s2 = fma(xb.x, Q[(size_t)(kk + 2) * b + col], s2);
            s3 = fma(xb.y, Q[(size_t)(kk + 3) * b + col], s3);
          }
          for (; kk < n; ++kk) s0 = fma(__ldcg(xi + kk), Q[(size_t)kk * b + col], s0);
          const double d = 0.5 * (Q[e] - ((s0 + s1) + (s2 + s3)));
          Dc[e] = d;
          ps += d * Sc[e];
          ph += d * Hc[e];
        }
        for (int i = i0 + etid; i < i1; i += kOzEpi) px += __ldcg(xd + (size_t)i * g.LD + i);
      }
      tell(0.0f, 0, ps, ph, px, true);
      if (!meet(r)) {
        if (etid == 0) sh.err = 1;
        break;
      }
      if (rank == 0 && etid == 0 && !c.gave_up) {
        const double ts = r.sum[0][0] + r.sum[1][0], th = r.sum[0][1] + r.sum[1][1], tx = r.sum[0][2] + r.sum[1][2];
        g.tS[J] = ts;
        g.tH[J] = th;
        g.iters[J] = c.steps;
        g.rsteps[J] = 0;
        g.nbelow[J] = (int32_t)lrint(0.5 * (c.n - tx));
        g.status[J] = c.status == kSubOk && !(isfinite(ts) && isfinite(th)) ? (int32_t)kSubNonFinite : c.status;
      }
    }
  }

  // every role has left its loop; after a wait that ran out, wait (bounded) for what is in flight
  __syncthreads();
  if (sh.err) {
    if (warp == 0 && lane == 0)
      for (int s = 0; s < kStages; ++s)
        if (armed[s]) tc::mbar_wait_ns(&sh.full[s], arm_phase[s], 50000000ull);
    if (warp == 1 && lane == 0) {
      tc::mma_commit(&sh.idle);
      tc::mbar_wait_ns(&sh.idle, 0, 50000000ull);
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
  cluster_sync();   // no CTA leaves while its peer may still write to its shared memory
}

// Mode 0: every submatrix of the work starts as kSubRefine, and what k_ns_oz does not finish k_ns_fp64 takes. Inverse
// mode: those whose FP32 inverse is there start as kSubPending, the others as kSubRefine (k_prepare takes both).
template <int kMode>
__global__ void k_oz_pending(int32_t count, const int32_t* __restrict__ order, int32_t* __restrict__ status) {
  for (int32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < count; e += gridDim.x * blockDim.x)
    status[order[e]] = kMode == 1 && status[order[e]] == kSubOk ? kSubPending : kSubRefine;
}

// How many two-CTA clusters of the kernel run at once on the device (asked once per device).
template <class Dg>
int active_clusters(int dev, int sms) {
  static std::atomic<int> known[64];
  if (dev >= 0 && dev < 64 && known[dev].load(std::memory_order_relaxed) > 0) return known[dev].load(std::memory_order_relaxed);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(2 * (sms / 2)));
  cfg.blockDim = dim3(kOzThreads);
  cfg.dynamicSmemBytes = Dg::kSmem;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 2;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(&k_ns_oz<Dg, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, Dg::kSmem) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, &k_ns_oz<Dg, 0>, &cfg) != cudaSuccess || n < 1) {
    cudaGetLastError();
    n = std::max(1, sms / 2);
  }
  if (dev >= 0 && dev < 64) known[dev].store(n, std::memory_order_relaxed);
  return n;
}

template <class Dg, int kMode>
bool split_fits() {
  cudaFuncAttributes at{};
  const bool ok = cudaFuncGetAttributes(&at, reinterpret_cast<const void*>(&k_ns_oz<Dg, kMode>)) == cudaSuccess;
  if (!ok) cudaGetLastError();
  return ok && at.numRegs == kRegsLaunch;
}

template <int kMode>
nolsm_status pending(const OzSolve& a, cudaStream_t st) {
  k_oz_pending<kMode><<<std::min(256, (a.count + 255) / 256), 256, 0, st>>>(a.count, a.order,
                                                                            kMode == 0 ? a.status : a.prep_out);
  NOLSM_LAUNCH_CHECK();
  return NOLSM_OK;
}

template <class Dg, int kMode>
nolsm_status launch(const OzSolve& a, cudaStream_t st) {
  const auto kernel = &k_ns_oz<Dg, kMode>;
  if (!split_fits<Dg, kMode>()) {
    set_error("k_ns_oz was not built with the %d registers per thread that its register split needs", kRegsLaunch);
    return NOLSM_ERR_UNSUPPORTED;
  }
  NOLSM_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Dg::kSmem));
  const uint64_t depth = (uint64_t)a.clusters * sets(kMode) * Dg::kD;
  CUtensorMap mA, mA64, mB;
  if (!tmap::make_3d(&mA, a.planes, 2, (uint64_t)a.LD, (uint64_t)a.R, depth, 32, 128, CU_TENSOR_MAP_SWIZZLE_64B, Dg::kD) ||
      !tmap::make_3d(&mA64, a.planes, 2, (uint64_t)a.LD, (uint64_t)a.R, depth, 32, 64, CU_TENSOR_MAP_SWIZZLE_64B, Dg::kD) ||
      !tmap::make_3d(&mB, a.planes, 2, (uint64_t)a.LD, (uint64_t)a.R, depth, 64, 32, CU_TENSOR_MAP_SWIZZLE_128B, Dg::kD)) {
    set_error("cuTensorMapEncodeTiled rejected the digit planes (R %d, LD %d, clusters %d)", a.R, a.LD, a.clusters);
    return NOLSM_ERR_CUDA;
  }
  OzArgs g{};
  g.count = a.count; g.order = a.order;
  g.sub_n = a.sub_n; g.nbf = a.nbf; g.a_off = a.a_off; g.c_off = a.c_off;
  g.A = a.A; g.Q = a.Q; g.Sc = a.Sc; g.Hc = a.Hc; g.lam = a.lam; g.lam_g = a.lam_g;
  g.prep_status = a.prep_status;
  g.mu = a.mu; g.tol = a.tol; g.max_iter = a.max_iter; g.budget = a.budget;
  g.planes = a.planes; g.xd = a.xd; g.R = a.R; g.LD = a.LD;
  g.Dc = a.Dc; g.tS = a.tS; g.tH = a.tH; g.iters = a.iters; g.status = a.status; g.rsteps = a.rsteps;
  g.nbelow = a.nbelow;
  g.wait_ns = kOzWaitNs;
  g.lim = a.loose ? kFixedLoose : kFixedFp64;
  g.ws = a.ws; g.a_base = a.a_base; g.chunk_n2 = a.chunk_n2; g.X32 = a.X32; g.sub_c0 = a.sub_c0;
  g.Aout = a.Aout; g.Qout = a.Qout; g.prep_out = a.prep_out;
  if (kMode == 1) g.max_iter = 1;
  NOLSM_TRY(pending<kMode>(a, st));
  kernel<<<2 * std::min(a.clusters, a.count), kOzThreads, Dg::kSmem, st>>>(mA, mA64, mB, g);
  NOLSM_LAUNCH_CHECK();
  return NOLSM_OK;
}

}  // namespace

int oz_planes(int mode) { return sets(mode) * Digits<8, 8>::kD; }

int oz_clusters(int max_n, int dev, int sms) {
  return max_n <= kOzNineBits ? active_clusters<Digits<9, 7>>(dev, sms) : active_clusters<Digits<8, 8>>(dev, sms);
}

bool oz_ready(int max_n) {
  return max_n <= kOzNineBits ? split_fits<Digits<9, 7>, 0>() && split_fits<Digits<9, 7>, 1>()
                              : split_fits<Digits<8, 8>, 0>() && split_fits<Digits<8, 8>, 1>();
}

nolsm_status leave_ns_oz(const OzSolve& a, cudaStream_t st) { return pending<0>(a, st); }

nolsm_status launch_ns_oz(const OzSolve& a, cudaStream_t st) {
  return a.max_n <= kOzNineBits ? launch<Digits<9, 7>, 0>(a, st) : launch<Digits<8, 8>, 0>(a, st);
}

nolsm_status launch_inverse_oz(const OzSolve& a, cudaStream_t st) {
  return a.max_n <= kOzNineBits ? launch<Digits<9, 7>, 1>(a, st) : launch<Digits<8, 8>, 1>(a, st);
}

}  // namespace nolsm
