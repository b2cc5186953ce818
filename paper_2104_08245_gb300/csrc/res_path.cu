// a4-a7 on the tensor cores for submatrices of up to 192 rows: the sign iteration with its operands on the SM.
//
// One CTA per SM runs one submatrix at a time, and nothing of an iterate leaves the SM: X lives in shared memory as
// hi and lo planes (192 x 192 in three blocks of 64 columns with 128-byte swizzle), which serve as the K-major A and
// as the MN-major B of the first product alike, and T = 3I - X X lives in tensor memory, written by the epilogue over
// the accumulators that it came from, as the A operand of the second. T commutes with X, so that product is T X:
//   P = X X      tile t (128 rows) over all n columns      -> T tile t in place
//   Z = T X      column block c (64) of every row tile     -> X' = Z / 2 over column block c of X
// Z's column block c needs nothing of X but its column block c, so X' can overwrite it as soon as the block's products
// are done. Tensor memory: T's two tiles take 2 x 192 columns, two Z accumulators 2 x 64.
// With one term T commutes with X only to the rounding of T, and the product keeps the order X T of the streaming kernel
// (T X differs from it as much as either does from the exact sign): T goes into the second plane as the B operand, Z over
// the accumulators of P, and X' over tile t's rows of X once tile t's products are done.
//
// The streaming kernel (k_ns_tc), which these submatrices used before and larger ones still use, keeps the operands of
// two submatrices per SM in global memory: 0.6 MB of TMA traffic a product at n = 172, more than the L2 holds over 152
// SMs (14.6 GB of DRAM traffic on 4,096 submatrices). Here a step takes some 17,000 cycles at n = 174 in the three-term
// split, 12,100 of them the MMAs' own, the rest where the epilogue waits for them or they for it; with one term the
// epilogue's (11,000 of 14,600 at n = 162), whose arithmetic on the two SM quarters that hold the second row tile counts.
// 27,000 submatrices: 18.2 ms, some 31 with the streaming kernel. Twelve or sixteen epilogue warps instead of eight: 18.6 and
// 26 ms (their registers spill); the MMAs unrolled over K: 19.0.
//
// Roles: warp 1 issues the MMAs (converged, one elected lane), warps 4-11 are the epilogue (two groups of four, even
// and odd 32-column chunks), which also starts and finishes the submatrices. All waits are bounded.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "nolsm_internal.cuh"
#include "prep.cuh"
#include "res_path.cuh"
#include "tcgen05.cuh"

namespace nolsm {

namespace {

constexpr int kThreadsR = 384, kEpiR = 256;
// the launch's 384 x 168 registers: 128 x 56 + 256 x 224
constexpr int kRegsLaunchR = 168, kRegsLowR = 56, kRegsEpiR = 224;
static_assert(128 * kRegsLowR + kEpiR * kRegsEpiR <= kThreadsR * kRegsLaunchR, "register split above the launch");
constexpr uint32_t kBlk = kResMaxN * 128;         // one column block of X: 192 rows of 128 bytes
constexpr uint32_t kPlane = 3 * kBlk;             // one plane
constexpr uint32_t kXBytes = 2 * kPlane;
constexpr int kQs = kResMaxN * 8;                 // staged columns of Q, FP32 [k][8]
constexpr int kSplit = 4;                         // shares of the k range in X Q
constexpr uint32_t kExtra = 4 * kQs + 8 * kSplit * kResMaxN * 8;   // Q, then the sums (hi, lo) of every share
constexpr uint32_t kSmemR = kXBytes + kExtra + 1024;
constexpr uint32_t kSmemI = kXBytes + 32 * 1024 + 2 * (16 * kResMaxN * 8 + 128) + 1024;   // inverse: FP32 staging of eight warps, the feed
static_assert(kExtra >= 64 * 128, "the second row tile's A reads up to 64 rows past the last block");
static_assert(kSmemR <= 227 * 1024 && kSmemI <= 227 * 1024 - 512, "shared memory");
static_assert(kExtra >= 2 * (16 * kResMaxN * 8 + 128), "the feed's buffers share it");
constexpr uint32_t kRing = 2 * kResMaxN;          // tensor memory column of the first Z accumulator
constexpr uint64_t kWaitNsR = 2000000000ull;

struct StepInfo { int term, n16, nrb, nch; Fmt f; };   // what the MMA warp needs of a step

struct SharedR {
  uint64_t xr, pf[2], tr[2], zf[2], ze[2], zp[2], ld[2], idle;
  uint32_t tmem;
  int err, fetch;
  StepInfo mm;
  float red[8];
  double dred[3][8];
};

__device__ __forceinline__ void bar_epi() { asm volatile("bar.sync 3, %0;" ::"n"(kEpiR) : "memory"); }
__device__ __forceinline__ bool bar_epi_or(bool p) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred P, Q;\n\tsetp.ne.u32 P, %1, 0;\n\tbar.red.or.pred Q, 3, %2, P;\n\tselp.u32 %0, 1, 0, Q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)p), "n"(kEpiR)
      : "memory");
  return r != 0;
}

// byte offset of the 16-byte unit u (eight columns) of row i in column block c of a plane
__device__ __forceinline__ uint32_t unit_at(int c, int i, int u) { return c * kBlk + i * 128 + ((u ^ (i & 7)) << 4); }

// The MMAs of one product: tile rows from A (descriptors in shared memory, or tensor memory for Z), all k.
template <bool kTs>
__device__ __forceinline__ void product(uint32_t dt, uint32_t x0, int row0, uint32_t at, uint32_t b0, int n16, uint32_t id,
                                        bool three) {
  const uint64_t bh0 = tc::sdesc_sw128(x0 + b0, kBlk, 1024);
  const uint64_t ah0 = tc::sdesc_sw128(x0 + row0 * 128, 16, 1024);
#pragma unroll 1
  for (int k = 0; k < n16 / 16; ++k) {
    const uint64_t bh = bh0 + ((k * 2048) >> 4), bl = bh + (kPlane >> 4);
    if constexpr (kTs) {
      const uint32_t ah = at + 32 * (k >> 1) + 8 * (k & 1), al = ah + 16;
      tc::mma_f16_ts(dt, ah, bh, id, k > 0 ? 1u : 0u);
      if (three) {
        tc::mma_f16_ts(dt, ah, bl, id, 1u);
        tc::mma_f16_ts(dt, al, bh, id, 1u);
      }
    } else {
      const uint64_t ah = ah0 + (((k >> 2) * kBlk + (k & 3) * 32) >> 4), al = ah + (kPlane >> 4);
      tc::mma_f16(dt, ah, bh, id, k > 0 ? 1u : 0u);
      if (three) {
        tc::mma_f16(dt, ah, bl, id, 1u);
        tc::mma_f16(dt, al, bh, id, 1u);
      }
    }
  }
}

// An n x n matrix (row-major, contiguous) from global into the operand in shared memory, by way of two staging buffers
// that bulk copies fill: the shared memory of these kernels leaves the L1 some 20 KB, so that loads which count on
// finding their lines there again fetch them several times over (45,000 cycles for the FP64 matrix at n = 172).
// A row a warp, two adjacent columns a lane in up to three blocks of 64: every access to shared memory is free of bank
// conflicts (with a 16-byte unit a lane the FP64 loads took 64 wavefronts a row, and 32,768 submatrices 12.2 ms in
// k_inv_res instead of 9.8).
// see(x, y, i, j): the entries (i, j) and (i, j + 1) in FP32, to be changed in place; zeros past the last column.
constexpr uint32_t kFeed = 16 * kResMaxN * 8 + 128;   // a staging buffer: 16 rows in FP64, and what the widening adds
__device__ __forceinline__ float narrow(float x, uint32_t&) { return x; }
// x in FP32, halves away from zero, by integer operations (the conversion instruction runs on the FP64 pipe); below
// 2^-126 a zero. big: the largest leading word; with an entry of kBeyond or more (out of FP32's range, infinite or not a
// number, for which this returns anything) the caller has to make the matrix non-finite itself. (A range check of every
// entry here instead: 374.2 ms for 262,144 submatrices, 372.9 this way.)
constexpr uint32_t kBeyond = 1151u << 20;
__device__ __forceinline__ float narrow(double x, uint32_t& big) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x), a = hi & 0x7FFFFFFFu;
  big = max(big, a);
  const uint32_t b = __funnelshift_l(lo, a, 3) + ((lo >> 28) & 1u) - (896u << 23);
  return __uint_as_float(a < (897u << 20) ? 0u : (b | (hi & 0x80000000u)));
}
template <typename T, typename See>
__device__ __forceinline__ uint32_t feed(uint8_t* X, const T* __restrict__ M, int n, int n64, Fmt f, uint8_t* stage,
                                         uint64_t (&ld)[2], uint32_t& nld, uint64_t wait_ns, bool& bad, int etid, See&& see) {
  const int ew = etid >> 5, lane = etid & 31;
  const int R = (int)((kFeed - 128) / (n * sizeof(T))) & ~7, nc = (n + R - 1) / R;   // rows a buffer, the same for every warp
  const bool even = (n & 1) == 0 && (reinterpret_cast<uintptr_t>(M) & (2 * sizeof(T) - 1)) == 0;
  uint32_t big = 0;
  auto issue = [&](int c) {   // one thread: rows [c R, ...) widened to whole 16-byte units
    const uintptr_t a = reinterpret_cast<uintptr_t>(M + (size_t)c * R * n), e = a + sizeof(T) * (size_t)min(R, n - c * R) * n;
    const uint32_t bytes = (uint32_t)(((e + 15) & ~uintptr_t(15)) - (a & ~uintptr_t(15)));
    uint64_t* bar = &ld[(nld + c) & 1];
    tc::mbar_arrive_expect_tx(bar, bytes);
    tc::bulk_load(stage + ((nld + c) & 1) * kFeed, reinterpret_cast<const void*>(a & ~uintptr_t(15)), bytes, bar);
  };
  if (etid == 0) {
    issue(0);
    if (nc > 1) issue(1);
  }
  const uint32_t unit = (lane >> 2) & 7, part = 4 * (lane & 3);
  auto put = [&](int t, int i, uint32_t h, uint32_t l) {
    uint8_t* at = X + t * kBlk + i * 128 + ((unit ^ (i & 7)) << 4) + part;
    *reinterpret_cast<uint32_t*>(at) = h;
    if (f.terms > 1) *reinterpret_cast<uint32_t*>(at + kPlane) = l;
  };
  for (int i = n + ew; i < n64; i += 8) {   // the rows of zeros
    for (int t = 0; 64 * t < n64; ++t) put(t, i, 0, 0);
  }
#pragma unroll 1
  for (int c = 0; c < nc; ++c) {
    const uint32_t b = (nld + c) & 1;
    if (!bad) bad = !tc::mbar_wait_ns(&ld[b], ((nld + c) >> 1) & 1, wait_ns);
    if (bad && etid == 0) tc::mbar_wait_ns(&ld[b], ((nld + c) >> 1) & 1, 50000000ull);   // none left in flight
    const T* rows = reinterpret_cast<const T*>(stage + b * kFeed + (reinterpret_cast<uintptr_t>(M + (size_t)c * R * n) & 15));
    const int count = min(R, n - c * R);
#pragma unroll 1
    for (int r = ew; r < count; r += 8) {
      const int i = c * R + r;
      T x[3], y[3];
#pragma unroll
      for (int t = 0; t < 3; ++t) {   // past the row's end the last column again
        const int j = 64 * t + 2 * lane;
        if (even) {
          struct alignas(2 * sizeof(T)) Pair { T x, y; };
          const Pair v = *reinterpret_cast<const Pair*>(rows + r * n + min(j, n - 2));
          x[t] = v.x;
          y[t] = v.y;
        } else {
          x[t] = rows[r * n + min(j, n - 1)];
          y[t] = rows[r * n + min(j + 1, n - 1)];
        }
      }
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        const int j = 64 * t + 2 * lane;
        if (t > 0 && 64 * t >= n64) break;
        float xf = narrow(x[t], big), yf = narrow(y[t], big);
        if (j >= n) xf = 0.0f;
        if (j + 1 >= n) yf = 0.0f;
        see(xf, yf, i, j);
        uint32_t h, l;
        split2(xf, yf, f.fmt, h, l);
        put(t, i, h, l);
      }
    }
    bar_epi();   // the buffer has been read
    if (etid == 0 && c + 2 < nc) issue(c + 2);
  }
  nld += nc;
  return big;
}

// This lane's row of X (hi, with kLo lo) times eight columns of Q over k0 <= k < k1 (multiples of 16): FP32 sums of 16
// products, each added to s + e with TwoSum.
template <int kFmt, bool kLo>
__device__ __forceinline__ void xq_part(const uint8_t* __restrict__ X, int i, int k0, int k1, const float* __restrict__ Qs,
                                        uint64_t (&s)[4], uint64_t (&e)[4]) {
  const uint64_t neg = pair2(-1.0f, -1.0f);
#pragma unroll
  for (int c = 0; c < 4; ++c) s[c] = e[c] = 0;
  for (int k = k0; k < k1; k += 16) {
    uint4 hv[2], lv[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const uint32_t at = unit_at(k >> 6, i, ((k >> 3) & 7) + t);
      hv[t] = *reinterpret_cast<const uint4*>(X + at);
      lv[t] = kLo ? *reinterpret_cast<const uint4*>(X + kPlane + at) : make_uint4(0, 0, 0, 0);
    }
    uint64_t p[4] = {0, 0, 0, 0};
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      const uint4 h4 = hv[w >> 2], l4 = lv[w >> 2];
      const uint32_t h = (w & 3) == 0 ? h4.x : (w & 3) == 1 ? h4.y : (w & 3) == 2 ? h4.z : h4.w;
      const uint32_t l = (w & 3) == 0 ? l4.x : (w & 3) == 1 ? l4.y : (w & 3) == 2 ? l4.z : l4.w;
      float2 x;
      if (kFmt == FMT_BF16) {
        x = make_float2(__uint_as_float(h << 16), __uint_as_float(h & 0xFFFF0000u));
        if (kLo) {
          x.x += __uint_as_float(l << 16);
          x.y += __uint_as_float(l & 0xFFFF0000u);
        }
      } else {
        x = __half22float2(*reinterpret_cast<const __half2*>(&h));
        if (kLo) {
          const float2 y = __half22float2(*reinterpret_cast<const __half2*>(&l));
          x.x += y.x;
          x.y += y.y;
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const ulonglong2 qa = *reinterpret_cast<const ulonglong2*>(Qs + (k + 2 * w + u) * 8);
        const ulonglong2 qb = *reinterpret_cast<const ulonglong2*>(Qs + (k + 2 * w + u) * 8 + 4);
        const uint64_t xx = u == 0 ? pair2(x.x, x.x) : pair2(x.y, x.y);
        p[0] = fma2(xx, qa.x, p[0]);
        p[1] = fma2(xx, qa.y, p[1]);
        p[2] = fma2(xx, qb.x, p[2]);
        p[3] = fma2(xx, qb.y, p[3]);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {   // TwoSum in pairs
      const uint64_t t = add2(s[c], p[c]), z = fma2(s[c], neg, t);
      e[c] = add2(e[c], add2(fma2(fma2(z, neg, t), neg, s[c]), fma2(z, neg, p[c])));
      s[c] = t;
    }
  }
}

// The same with every product's rounding error (exact_xq): two products a step, as short in code as it can be.
template <int kFmt, bool kLo>
__device__ __forceinline__ void xq_exact(const uint8_t* __restrict__ X, int i, int k0, int k1, const float* __restrict__ Qs,
                                         uint64_t (&s)[4], uint64_t (&e)[4]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) s[c] = e[c] = 0;
#pragma unroll 1
  for (int k = k0; k < k1; k += 2) {
    const uint32_t at = unit_at(k >> 6, i, (k >> 3) & 7) + 2 * (k & 7);
    const uint32_t h = *reinterpret_cast<const uint32_t*>(X + at), l = kLo ? *reinterpret_cast<const uint32_t*>(X + kPlane + at) : 0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      float x = from_bits((uint16_t)(h >> (16 * u)), kFmt);
      if (kLo) x += from_bits((uint16_t)(l >> (16 * u)), kFmt);
      const ulonglong2 qa = *reinterpret_cast<const ulonglong2*>(Qs + (k + u) * 8);
      const ulonglong2 qb = *reinterpret_cast<const ulonglong2*>(Qs + (k + u) * 8 + 4);
      const uint64_t xx = pair2(x, x), xn = pair2(-x, -x), q[4] = {qa.x, qa.y, qb.x, qb.y};
#pragma unroll
      for (int c = 0; c < 4; ++c) add_product2(s[c], e[c], xx, xn, q[c]);
    }
  }
}

// kFmt, kTerms: the main phase's operand format (the refinement's is FP16 in three terms). A template of it, and one site
// each of T and of the Z blocks, because the epilogue's code has to stay in the instruction cache: with all four formats
// at every site the code is 84 KB, against 62-74 KB. kExact: some submatrix takes xq_exact (1 % more time on 262,144 that
// do not, with its code there).
template <int kFmt, int kTerms, bool kExact>
__global__ void __launch_bounds__(kThreadsR, 1) k_ns_res(ResSolve g) {
  constexpr bool kOne = kFmt == FMT_F16 && kTerms == 3;   // the main format is the refinement's
  extern __shared__ uint8_t smraw[];
  uint8_t* const X = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  float* const Qs = reinterpret_cast<float*>(X + kXBytes);
  float2* const Ps = reinterpret_cast<float2*>(Qs + kQs);
  __shared__ SharedR sh;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  if (tid == 0) {
    tc::mbar_init(&sh.xr, kEpiR);
    for (int t = 0; t < 2; ++t) {
      tc::mbar_init(&sh.pf[t], 1);
      tc::mbar_init(&sh.tr[t], kEpiR);
      tc::mbar_init(&sh.zf[t], 1);
      tc::mbar_init(&sh.zp[t], 1);
      tc::mbar_init(&sh.ze[t], kEpiR);
      tc::mbar_init(&sh.ld[t], 1);
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
  uint32_t nstep = 0, np0 = 0, np1 = 0, nz = 0;   // steps, P tiles and Z blocks so far (per role)

  if (warp < 4) {
  tc::setmaxnreg_dec<kRegsLowR>();
  if (warp == 1) {
    // ------------------------------------------------ MMA issuer
    auto wait = [&](uint64_t* b, uint32_t parity, int more) {
      return (bool)__all_sync(0xffffffffu, tc::mbar_wait_ns(b, parity, more * g.wait_ns));
    };
    const uint32_t x0 = __shfl_sync(0xffffffffu, tc::smem_u32(X), 0);
    bool ok = true;
    while (ok && !sh.err) {
      if (!(ok = wait(&sh.xr, nstep & 1, 8))) break;
      ++nstep;
      tc::tc_fence_after();
      const StepInfo m = sh.mm;
      if (m.term) break;
      const bool three = m.f.terms > 1;
      const uint32_t idp = tc::idesc(m.f.fmt, m.f.fmt, 0, 1, 128, m.n16);
      for (int t = 0; t < m.nrb; ++t) {
        if (tc::elect_one()) {
          product<false>(tmem + kResMaxN * t, x0, 128 * t, 0, 0, m.n16, idp, three);
          tc::mma_commit(&sh.pf[t]);
        }
        __syncwarp();
      }
      if (kTerms == 1 && !three) {   // Z = X T, T in the second plane, over P's accumulators
        for (int t = 0; t < m.nrb && ok; ++t) {
          ok = wait(&sh.tr[t], (t ? np1 : np0) & 1, 1);
          ++(t ? np1 : np0);
        }
        if (!ok) break;
        tc::tc_fence_after();
        for (int t = 0; t < m.nrb; ++t) {
          if (tc::elect_one()) {
            product<false>(tmem + kResMaxN * t, x0, 128 * t, 0, kPlane, m.n16, idp, false);
            tc::mma_commit(&sh.zp[t]);
          }
          __syncwarp();
        }
        continue;
      }
      for (int c = 0; c < m.nch && ok; ++c) {
        const uint32_t idz = tc::idesc(m.f.fmt, m.f.fmt, 0, 1, 128, min(64, m.n16 - 64 * c));
        for (int t = 0; t < m.nrb; ++t, ++nz) {
          const int slot = nz & 1;
          if (c == 0) {
            if (!(ok = wait(&sh.tr[t], (t ? np1 : np0) & 1, 1))) break;
            ++(t ? np1 : np0);
          }
          if (!(ok = wait(&sh.ze[slot], ((nz >> 1) & 1) ^ 1, 1))) break;
          tc::tc_fence_after();
          if (tc::elect_one()) {
            product<true>(tmem + kRing + 64 * slot, x0, 0, tmem + kResMaxN * t, c * kBlk, m.n16, idz, three);
            tc::mma_commit(&sh.zf[slot]);
          }
          __syncwarp();
        }
      }
    }
    if (!ok) sh.err = 1;
  }
  } else {
    tc::setmaxnreg_inc<kRegsEpiR>();
    // ------------------------------------------------ epilogue
    const int etid = tid - 128, ew = warp - 4, q = warp & 3, grp = ew >> 2;
    const uint32_t lane_base = (uint32_t)(32 * q) << 16;
    uint32_t nld = 0, nq0 = 0, nq1 = 0;   // fills; one-term Z products of either row tile
    bool bad = false;
    for (;;) {
      // ---- the next submatrix of at most kResMaxN rows (the last one's finish has used the feed's buffers)
      tc::fence_proxy_async_smem();
      int J = -1;
      for (;;) {
        if (etid == 0) {
          const int k = atomicAdd(g.next, 1);
          sh.fetch = (k < g.count && !sh.err) ? g.order[k] : -1;
        }
        bar_epi();
        J = sh.fetch;
        bar_epi();
        if (J < 0) break;
        if (g.sub_n[J] > kResMaxN) continue;   // k_ns_tc takes it
        if (g.cond && g.prep_status[J] == kSubOk && g.cond[J] > g.cond_max && g.sub_n[J] <= g.ill_max_n) continue;
        if (g.prep_status[J] == kSubOk) break;
        if (etid == 0) {
          g.status[J] = g.prep_status[J];
          g.iters[J] = 0;
          g.rsteps[J] = 0;
          g.tS[J] = 0.0;
          g.tH[J] = 0.0;
        }
      }
      if (J < 0) {
        if (etid == 0) sh.mm.term = 1;
        bar_epi();
        tc::mbar_arrive(&sh.xr);
        break;
      }
      const int n = g.sub_n[J], n16 = (n + 15) & ~15, n64 = (n + 63) & ~63, nrb = (n + 127) / 128, nch = (n16 + 63) / 64;
      // ---- a4: X_0 = (A - mu I) / alpha in the main format, zeros up to n64
      {
        const float* __restrict__ A = g.A + g.a_off[J];
        const float inv = (float)(1.0 / scale_alpha(g.lam, g.lam_g, J, g.mu)), fmu = (float)g.mu;
        const Fmt f{kFmt, kTerms};
        feed(X, A, n, n64, f, reinterpret_cast<uint8_t*>(Qs), sh.ld, nld, g.wait_ns, bad, etid,
             [&](float& x, float& y, int i, int j) {
               x = (i == j && i < n ? x - fmu : x) * inv;
               y = (i == j + 1 && i < n ? y - fmu : y) * inv;
             });
      }
      int phase = 0, refine_left = g.refine_steps, steps = 0, rsteps = 0, status = kSubNotConv;
      float dprev = INFINITY;
      bool ref = kOne;   // X is in the refinement's format
      bool last = false;
      if (etid == 0) sh.mm = StepInfo{0, n16, nrb, nch, Fmt{kFmt, kTerms}};
      tc::fence_proxy_async_smem();
      tc::tc_fence_before();
      bar_epi();
      tc::mbar_arrive(&sh.xr);
      int Jn = -1;
      while (!last) {
        // ---- P -> T, tile by tile
        float part = 0.0f;
        for (int t = 0; t < nrb; ++t) {
          if (!bad) bad = !tc::mbar_wait_ns(&sh.pf[t], (t ? np1 : np0) & 1, g.wait_ns);
          bad = __any_sync(0xffffffffu, bad);
          ++(t ? np1 : np0);
          tc::tc_fence_after();
          const int rbase = 128 * t + 32 * q, row = rbase + lane;
          if (rbase < n64 && !bad) {
            const uint32_t ta = tmem + kResMaxN * t + lane_base;
            const int nsub = (n16 + 31) / 32;
            uint32_t r[32];
            if (grp < nsub) tc::tmem_ld32(ta + 32 * grp, r);
            for (int j = grp; j < nsub; j += 2) {
              const int col0 = 32 * j;
              uint32_t h[16], l[16];
              tc::tmem_wait_ld();
              if (col0 + 16 >= n16) {   // the MMAs left the second half out: it holds anything
#pragma unroll
                for (int u = 16; u < 32; ++u) r[u] = 0;
              }
              // (3I - P)_ij = (I - P)_ij = -P_ij off the diagonal; rows and columns past n are zeros, X's being zeros.
              // On it: P - 1 for the defect, then 3 - P in place of 1 - P
              const bool diag = col0 == rbase;
              if (diag) {
                const float one = row < n ? 1.0f : 0.0f;
#pragma unroll
                for (int u = 0; u < 32; ++u) r[u] = pick(u, lane, __float_as_uint(__uint_as_float(r[u]) - one), r[u]);
              }
              float sq = 0.0f;
              if (!kOne && !ref) scale_split_t<kFmt, (kTerms > 1), true>(r, -1.0f, h, l, sq);
              else scale_split_t<FMT_F16, true, true>(r, -1.0f, h, l, sq);
              if (row < n) part += sq;
              if (diag) {
                uint32_t e = 0;
#pragma unroll
                for (int u = 0; u < 32; ++u) e = pick(u, lane, r[u], e);
                uint32_t th, tl;
                split2(row < n ? 2.0f - __uint_as_float(e) : 0.0f, 0.0f, ref ? FMT_F16 : kFmt, th, tl);
                const uint32_t sel = lane & 1 ? 0x5410u : 0x3254u;   // (low of x, low of t) or (low of t, high of x)
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                  h[u] = pick(u, lane >> 1, __byte_perm(h[u], th, sel), h[u]);
                  l[u] = pick(u, lane >> 1, __byte_perm(l[u], tl, sel), l[u]);
                }
              }
              if (kTerms == 1 && !ref) {
                if (j + 2 < nsub) tc::tmem_ld32(ta + 32 * (j + 2), r);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                  *reinterpret_cast<uint4*>(X + kPlane + unit_at(j >> 1, row, 4 * (j & 1) + u)) =
                      make_uint4(h[4 * u], h[4 * u + 1], h[4 * u + 2], h[4 * u + 3]);
                continue;
              }
              uint32_t o[32];
#pragma unroll
              for (int u = 0; u < 16; ++u) {
                o[u] = h[u];
                o[16 + u] = l[u];
              }
              if (j + 2 < nsub) tc::tmem_ld32(ta + 32 * (j + 2), r);
              tc::tmem_st32(ta + 32 * j, o);
            }
            tc::tmem_wait_st();
          }
          tc::tc_fence_before();
          if (kTerms == 1) tc::fence_proxy_async_smem();
          if (!bad) tc::mbar_arrive(&sh.tr[t]);
        }
        // ---- the defect of X and the decision about the following steps (every thread alike)
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (lane == 0) sh.red[ew] = part;
        if (bar_epi_or(bad)) {
          bad = true;
          break;
        }
        float dsum = 0.0f;
        for (int w = 0; w < 8; ++w) dsum += sh.red[w];
        const float dd = sqrtf(dsum / (float)n);
        steps += 1;
        if (phase == 1) rsteps += 1;   // this step runs in the refinement format
        bool rnxt = ref;
        status = kSubNotConv;
        if (!isfinite(dd)) {
          last = true;
          status = kSubNonFinite;
        } else if (phase == 0) {
          if (dd <= g.tol_ns) {
            if (g.refine_steps == 0) {
              last = true;
              status = dd <= g.tol_accept ? kSubOk : kSubNotConv;
            } else {
              phase = 1;
              refine_left = g.refine_steps;
              rnxt = true;
            }
          }
        } else if (--refine_left <= 0) {
          if (dd <= g.tol_accept) {
            last = true;
            status = kSubOk;
          } else if (dd < dprev) {
            refine_left = 1;           // still converging: one more step (bounded by the step cap below)
          } else {
            last = true;
          }
        }
        const int cap = g.budget ? min(g.max_iter, g.budget[J]) : g.max_iter;
        if (!last && steps >= cap) {
          last = true;
          status = kSubNotConv;
        }
        dprev = dd;
        if (last && etid == 0) {   // what the finish and the next start read, on its way into L2
          const size_t cb = sizeof(double) * (size_t)n * g.nbf[J];
          tc::prefetch_l2(g.Q + g.c_off[J], cb);
          tc::prefetch_l2(g.Sc + g.c_off[J], cb);
          tc::prefetch_l2(g.Hc + g.c_off[J], cb);
          const int kn = *reinterpret_cast<volatile int32_t*>(g.next);   // a guess: another CTA may take it
          if (kn < g.count) {
            Jn = g.order[kn];
            const int nn = g.sub_n[Jn];
            if (nn <= kResMaxN) tc::prefetch_l2(g.A + g.a_off[Jn], sizeof(float) * (size_t)nn * nn);
          }
        }
        // ---- one term: Z -> X', row tile by row tile. Tile t's rows of X are read by tile t's products alone; the lo plane
        // of the refinement's format takes T's place once all of them have completed.
        if (kTerms == 1 && !ref) {
          for (int t = rnxt ? -nrb : 0; t < nrb; ++t) {
            const int w = t < 0 ? t + nrb : t;
            if (!bad) bad = !tc::mbar_wait_ns(&sh.zp[w], (w ? nq1 : nq0) & 1, g.wait_ns);
            bad = __any_sync(0xffffffffu, bad);
            tc::tc_fence_after();
            const int rbase = 128 * w + 32 * q, row = rbase + lane;
            if (t < 0 || rbase >= n64 || bad) continue;
            const uint32_t ta = tmem + kResMaxN * w + lane_base;
#pragma unroll 1
            for (int j = grp; 32 * j < n16; j += 2) {
              uint32_t r[32], h[16], l[16];
              tc::tmem_ld32(ta + 32 * j, r);
              tc::tmem_wait_ld();
              float sq = 0.0f;
              if (!rnxt) scale_split_t<kFmt, false, false>(r, 0.5f, h, l, sq);
              else scale_split_t<FMT_F16, true, false>(r, 0.5f, h, l, sq);
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                uint8_t* at = X + unit_at(j >> 1, row, 4 * (j & 1) + u);
                *reinterpret_cast<uint4*>(at) = make_uint4(h[4 * u], h[4 * u + 1], h[4 * u + 2], h[4 * u + 3]);
                if (rnxt) *reinterpret_cast<uint4*>(at + kPlane) = make_uint4(l[4 * u], l[4 * u + 1], l[4 * u + 2], l[4 * u + 3]);
              }
            }
          }
          ++nq0;
          nq1 += nrb - 1;
          tc::tc_fence_before();
        }
        // ---- else Z -> X', column block by column block (two 32-column chunks, one a group)
        for (int c = 0; c < (kTerms == 1 && !ref ? 0 : nch); ++c) {
          const int col0 = 64 * c + 32 * grp;
          const bool cols = col0 < n16;
          // row tile t's block out of its accumulator, halved and split
          auto take = [&](int t, uint32_t (&h)[16], uint32_t (&l)[16]) {
            const int slot = nz & 1;
            if (!bad) bad = !tc::mbar_wait_ns(&sh.zf[slot], (nz >> 1) & 1, g.wait_ns);
            bad = __any_sync(0xffffffffu, bad);
            ++nz;
            tc::tc_fence_after();
            uint32_t r[32];
            const bool mine = 128 * t + 32 * q < n64 && cols && !bad;
            if (mine) {
              tc::tmem_ld32(tmem + kRing + 64 * slot + lane_base + 32 * grp, r);
              tc::tmem_wait_ld();
            }
            tc::tc_fence_before();
            if (!bad) tc::mbar_arrive(&sh.ze[slot]);
            // rows and columns from n to n16 are zeros of themselves; columns past n16 hold anything and are not read
            float sq = 0.0f;
            if (mine) {
              if (!kOne && !rnxt) scale_split_t<kFmt, (kTerms > 1), false>(r, 0.5f, h, l, sq);
              else scale_split_t<FMT_F16, true, false>(r, 0.5f, h, l, sq);
            }
          };
          auto put = [&](int t, const uint32_t (&h)[16], const uint32_t (&l)[16]) {
            const int rbase = 128 * t + 32 * q, row = rbase + lane;
            if (rbase >= n64 || !cols || bad) return;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              uint8_t* at = X + unit_at(c, row, 4 * grp + u);
              *reinterpret_cast<uint4*>(at) = make_uint4(h[4 * u], h[4 * u + 1], h[4 * u + 2], h[4 * u + 3]);
              if (kTerms > 1 || rnxt)
                *reinterpret_cast<uint4*>(at + kPlane) = make_uint4(l[4 * u], l[4 * u + 1], l[4 * u + 2], l[4 * u + 3]);
            }
          };
          // X's column block may be overwritten once the block's last product has completed
          uint32_t h0[16], l0[16];
          take(0, h0, l0);
          if (nrb == 2) {
            uint32_t h1[16], l1[16];
            take(1, h1, l1);
            put(1, h1, l1);
          }
          put(0, h0, l0);
        }
        if (bar_epi_or(bad)) {
          bad = true;
          break;
        }
        ref = rnxt;
        if (!last) {
          if (etid == 0) sh.mm.f = ref ? Fmt{FMT_F16, 3} : Fmt{kFmt, kTerms};
          tc::fence_proxy_async_smem();
          bar_epi();
          tc::mbar_arrive(&sh.xr);
        }
      }
      if (bad) {   // a wait ran out
        if (etid == 0) {
          sh.err = 1;
          g.status[J] = kSubTimeout;
          g.iters[J] = steps;
          g.rsteps[J] = rsteps;
          g.tS[J] = 0.0;
          g.tH[J] = 0.0;
          atomicExch(g.err, 1);
          sh.mm.term = 1;
        }
        tc::mbar_arrive(&sh.xr);
        break;
      }
      // ---- a7: centre columns of T_J(D) = 1/2 (I - X) T_J(S)^-1 and the FP64 partial traces, eight columns at a time:
      // (32 rows, a quarter of k) per warp, Q staged in FP32, then the FP64 step entry by entry
      const int b = g.nbf[J];
      const double* __restrict__ Q = g.Q + g.c_off[J];
      const double* __restrict__ Sc = g.Sc + g.c_off[J];
      const double* __restrict__ Hc = g.Hc + g.c_off[J];
      double* __restrict__ Dc = g.Dc + g.c_off[J];
      double ps = 0.0, ph = 0.0;
      const bool exact = kExact && exact_xq(n, b);
      const int units = n16 / 16, nitem = ((n + 31) / 32) * kSplit;   // of k: 16 at a time
      for (int cg = 0; cg < b; cg += 8) {
        const int cn = min(8, b - cg);
        {   // all loads in flight together
          double v[kResMaxN * 8 / kEpiR];
#pragma unroll
          for (int u = 0; u < kResMaxN * 8 / kEpiR; ++u) {
            const int e = etid + u * kEpiR;
            v[u] = __ldg(Q + (size_t)min(e >> 3, n - 1) * b + cg + min(e & 7, cn - 1));
          }
#pragma unroll
          for (int u = 0; u < kResMaxN * 8 / kEpiR; ++u) {
            const int e = etid + u * kEpiR, k = e >> 3;
            if (k < n16) Qs[e] = k < n && (e & 7) < cn ? (float)v[u] : 0.0f;
          }
        }
        bar_epi();
        for (int it = ew; it < nitem; it += 8) {
          const int i = 32 * (it / kSplit) + lane, kq = it % kSplit;
          const int k0 = 16 * (units * kq / kSplit), k1 = 16 * (units * (kq + 1) / kSplit);
          uint64_t s[4], e[4];
          if (!kOne && !ref) {
            if (exact) xq_exact<kFmt, (kTerms > 1)>(X, i, k0, k1, Qs, s, e);
            else xq_part<kFmt, (kTerms > 1)>(X, i, k0, k1, Qs, s, e);
          } else {
            if (exact) xq_exact<FMT_F16, true>(X, i, k0, k1, Qs, s, e);
            else xq_part<FMT_F16, true>(X, i, k0, k1, Qs, s, e);
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float2 a = unpair2(s[c]), d = unpair2(e[c]);
            Ps[(kq * 8 + 2 * c) * kResMaxN + i] = make_float2(a.x, d.x);
            Ps[(kq * 8 + 2 * c + 1) * kResMaxN + i] = make_float2(a.y, d.y);
          }
        }
        bar_epi();
        for (int e = etid; e < n * cn; e += kEpiR) {
          const int i = e / cn, c = e - i * cn;
          float s = 0.0f, m = 0.0f;
#pragma unroll
          for (int kq = 0; kq < kSplit; ++kq) {
            const float2 p = Ps[(kq * 8 + c) * kResMaxN + i];
            two_sum(s, m, p.x);
            m += p.y;
          }
          const size_t at = (size_t)i * b + cg + c;
          const double dv = 0.5 * (Q[at] - ((double)s + (double)m));
          Dc[at] = dv;
          ps += dv * Sc[at];
          ph += dv * Hc[at];
        }
        bar_epi();
      }
      double px = 0.0;   // the trace of the final X: (n - Tr X) / 2 eigenvalues lie below mu
      for (int i = etid; i < n; i += kEpiR) {
        const uint32_t at = unit_at(i >> 6, i, (i >> 3) & 7) + 2 * (i & 7);
        float x = from_bits(*reinterpret_cast<const uint16_t*>(X + at), ref ? FMT_F16 : kFmt);
        if (kTerms > 1 || ref) x += from_bits(*reinterpret_cast<const uint16_t*>(X + kPlane + at), ref ? FMT_F16 : kFmt);
        px += x;
      }
      for (int o = 16; o > 0; o >>= 1) {
        ps += __shfl_xor_sync(0xffffffffu, ps, o);
        ph += __shfl_xor_sync(0xffffffffu, ph, o);
        px += __shfl_xor_sync(0xffffffffu, px, o);
      }
      if (lane == 0) {
        sh.dred[0][ew] = ps;
        sh.dred[1][ew] = ph;
        sh.dred[2][ew] = px;
      }
      bar_epi();
      if (etid == 0) {
        double ts = 0.0, th = 0.0, tx = 0.0;
        for (int w = 0; w < 8; ++w) {
          ts += sh.dred[0][w];
          th += sh.dred[1][w];
          tx += sh.dred[2][w];
        }
        if (g.nbelow) g.nbelow[J] = (int32_t)lrint(0.5 * (n - tx));
        g.tS[J] = ts;
        g.tH[J] = th;
        g.iters[J] = steps;
        g.rsteps[J] = rsteps;
        g.status[J] = status == kSubOk && !(isfinite(ts) && isfinite(th)) ? (int32_t)kSubNonFinite : status;
      }
    }
  }

  // every role has left its loop; after a wait that ran out, wait (bounded) for the MMAs still in flight
  __syncthreads();
  if (sh.err && warp == 1 && lane == 0) {
    tc::mma_commit(&sh.idle);
    tc::mbar_wait_ns(&sh.idle, 0, 50000000ull);
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------ the inverse square root
// a2-a3 for submatrices of up to 192 rows whose inverse square root converges in two steps (Eqs. inv1-inv3 with Z_0 = I),
// with the same layout: T_0 = 3I - Y_0 stays in tensor memory as the A operand of every product of the iteration (all of
// them are polynomials of T_J(S) and commute), and shared memory holds the other operand, overwritten column block by
// column block by the product's result:
//   Y_1 = T_0 Y_0 / 2,  T_1 = 3I - T_0 Y_1 / 2 (V_1 = Z_1 Y_1, Z_1 = T_0 / 2),  Z_2 = T_0 T_1 / 4,
//   X = Z_2 Z_2 / c (P product; X in FP32 to memory and over its accumulators as the A operand),  A_J = X T_J(H0).
// T_J(S) and T_J(H0) are read once and A_J and X written once, 0.71 MB at n = 172; nothing else moves. 27,000 submatrices
// of 120-192 rows take 9.8 ms; k_ns_tc, which they used before, took 17.6 ms on them (every product's operands from L2 or
// DRAM). At 6.5 TB/s the traffic alone would take 3.0 ms, the MMAs 2.9 ms: what bounds it is the epilogue, serial with
// the products of one submatrix. Submatrices that need more steps are marked kSubAgain for k_ns_tc.
struct InvInfo { int op, n16, nrb, nch; };   // op 0: T x B in column blocks, 1: B x B in row tiles, 2: the end

struct SharedI {
  uint64_t xr, pf[2], zf[2], ze[2], ld[2], idle;
  uint32_t tmem;
  int err, fetch;
  InvInfo mm;
  float red[8];
};

__global__ void __launch_bounds__(kThreadsR, 1) k_inv_res(InvSolve g) {
  extern __shared__ uint8_t smraw[];
  uint8_t* const X = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  __shared__ SharedI sh;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  if (tid == 0) {
    tc::mbar_init(&sh.xr, kEpiR);
    for (int t = 0; t < 2; ++t) {
      tc::mbar_init(&sh.pf[t], 1);
      tc::mbar_init(&sh.zf[t], 1);
      tc::mbar_init(&sh.ze[t], kEpiR);
      tc::mbar_init(&sh.ld[t], 1);
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
  uint32_t nop = 0, np0 = 0, np1 = 0, nz = 0;   // products, P tiles and column blocks so far (per role)

  if (warp < 4) {
    tc::setmaxnreg_dec<kRegsLowR>();
    if (warp == 1) {
      auto wait = [&](uint64_t* b, uint32_t parity, int more) {
        return (bool)__all_sync(0xffffffffu, tc::mbar_wait_ns(b, parity, more * g.wait_ns));
      };
      const uint32_t x0 = __shfl_sync(0xffffffffu, tc::smem_u32(X), 0);
      bool ok = true;
      while (ok && !sh.err) {
        if (!(ok = wait(&sh.xr, nop & 1, 8))) break;
        ++nop;
        tc::tc_fence_after();
        const InvInfo m = sh.mm;
        if (m.op == 2) break;
        if (m.op == 1) {
          const uint32_t id = tc::idesc(FMT_F16, FMT_F16, 0, 1, 128, m.n16);
          for (int t = 0; t < m.nrb; ++t) {
            if (tc::elect_one()) {
              product<false>(tmem + kResMaxN * t, x0, 128 * t, 0, 0, m.n16, id, true);
              tc::mma_commit(&sh.pf[t]);
            }
            __syncwarp();
          }
          continue;
        }
        for (int c = 0; c < m.nch && ok; ++c) {
          const uint32_t id = tc::idesc(FMT_F16, FMT_F16, 0, 1, 128, min(64, m.n16 - 64 * c));
          for (int t = 0; t < m.nrb; ++t, ++nz) {
            const int slot = nz & 1;
            if (!(ok = wait(&sh.ze[slot], ((nz >> 1) & 1) ^ 1, 1))) break;
            tc::tc_fence_after();
            if (tc::elect_one()) {
              product<true>(tmem + kRing + 64 * slot, x0, 0, tmem + kResMaxN * t, c * kBlk, m.n16, id, true);
              tc::mma_commit(&sh.zf[slot]);
            }
            __syncwarp();
          }
        }
      }
      if (!ok) sh.err = 1;
    }
  } else {
    tc::setmaxnreg_inc<kRegsEpiR>();
    const int etid = tid - 128, ew = warp - 4, q = warp & 3, grp = ew >> 2;
    const uint32_t lane_base = (uint32_t)(32 * q) << 16;
    float* const wf = reinterpret_cast<float*>(X + kXBytes) + 1024 * ew;   // this warp's 32 x 32 staging
    bool bad = false;
    uint32_t nld = 0;
    int kn = -1;   // thread 0: the next submatrix's place, once it has been drawn
    // the operands are ready: product `op` may start
    auto go = [&](int op, int n16, int nrb, int nch) {
      if (etid == 0) sh.mm = InvInfo{op, n16, nrb, nch};
      tc::fence_proxy_async_smem();
      tc::tc_fence_before();
      bar_epi();
      tc::mbar_arrive(&sh.xr);
    };
    for (;;) {
      if (etid == 0) {
        const int k = kn >= 0 ? kn : atomicAdd(g.next, 1);
        sh.fetch = (k < g.count && !sh.err) ? g.order[k] : -1;
        kn = -1;
      }
      bar_epi();
      const int J = sh.fetch;
      bar_epi();
      if (J < 0) {
        go(2, 0, 0, 0);
        break;
      }
      const int n = g.sub_n[J], n16 = (n + 15) & ~15, n64 = (n + 63) & ~63, nrb = (n + 127) / 128, nch = (n16 + 63) / 64;
      const double* __restrict__ S = g.ws + (g.a_off[J] - g.a_base);
      const double* __restrict__ H = S + g.chunk_n2;
      auto total = [&](float p) -> float {   // sum over the epilogue's threads
        for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
        if (lane == 0) sh.red[ew] = p;
        bar_epi();
        float d = 0.0f;
        for (int w = 0; w < 8; ++w) d += sh.red[w];
        bar_epi();
        return d;
      };
      // a 32 x 32 chunk (row = lane) in FP32 to an n x n array, through the warp's staging so that a store
      // instruction writes 32 consecutive entries of a row
      auto out = [&](float* __restrict__ dst, int rbase, int col0, const uint32_t (&r)[32]) __attribute__((always_inline)) {
        // pairs of entries: 2-entry unit p of row i at p ^ (i & 15)
        __syncwarp();
        float2* const wf2 = reinterpret_cast<float2*>(wf);
#pragma unroll
        for (int p = 0; p < 16; ++p)
          wf2[lane * 16 + (p ^ (lane & 15))] = make_float2(__uint_as_float(r[2 * p]), __uint_as_float(r[2 * p + 1]));
        __syncwarp();
        const int rows = min(32, n - rbase), p = lane & 15, col = col0 + 2 * p;
        float* at = dst + (size_t)(rbase + (lane >> 4)) * n + col;
        if ((n & 1) == 0 && (reinterpret_cast<uintptr_t>(dst) & 7) == 0) {   // two rows an instruction, 8 bytes a lane
          if (col < n) {
#pragma unroll 8
            for (int i = lane >> 4; i < rows; i += 2, at += 2 * n) *reinterpret_cast<float2*>(at) = wf2[i * 16 + (p ^ (i & 15))];
          }
        } else {
          for (int i = lane >> 4; i < rows; i += 2, at += 2 * n) {
            const float2 x = wf2[i * 16 + (p ^ (i & 15))];
            if (col < n) at[0] = x.x;
            if (col + 1 < n) at[1] = x.y;
          }
        }
      };
      if (etid == 0) tc::prefetch_l2(H, sizeof(double) * (size_t)n * n);
      double tr = 0.0;   // c = Tr T_J(S) / n
#pragma unroll
      for (int k = 0; k < kResMaxN / 32; ++k) {
        const int i = min(lane + 32 * k, n - 1);
        const double d = __ldg(S + (size_t)i * n + i);
        tr += lane + 32 * k < n ? d : 0.0;
      }
      for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
      const double cc = tr / n;
      const float inv = (float)(1.0 / cc);
      int status = kSubOk, steps = 1;
      bool last0 = false;
      // half 0: the iteration on Y_0 = T_J(S) / c, up to X; half 1: A_J = X T_J(H0). (One copy of the code for both and for
      // every product: what the epilogue runs stays in the instruction cache.)
#pragma unroll 1
      for (int half = 0; half < (g.Aout ? 2 : 1) && status == kSubOk; ++half) {
        const double* __restrict__ M = half ? H : S;
        const float scale = half ? 1.0f : inv;
        float part = 0.0f;   // ||I - Y_0||_F^2
        const Fmt f3{FMT_F16, 3};
        const uint32_t big = feed(X, M, n, n64, f3, X + kXBytes + 32 * 1024, sh.ld, nld, g.wait_ns, bad, etid,
                                  [&](float& x, float& y, int i, int j) {
                                    x *= scale;
                                    y *= scale;
                                    const float e0 = i == j ? 1.0f - x : x, e1 = i == j + 1 ? 1.0f - y : y;
                                    part = fmaf(e0, e0, fmaf(e1, e1, part));
                                  });
        if (big >= kBeyond) {   // T_J(S): left to the FP64 preparation; T_J(H0): a NaN that makes every row of A_J one
          part = INFINITY;
          *reinterpret_cast<uint32_t*>(X) = 0x7FFF7FFFu;
        }
        if (half == 0) {
          const float d0 = sqrtf(total(part) / (float)n);   // its barriers also publish Y_0
          last0 = d0 <= g.tol_inv;
          if (!(cc > 0.0) || !isfinite(cc) || !isfinite(d0)) {   // the FP64 preparation takes it
            status = kSubRefine;
            break;
          }
          // T_0 = 3I - Y_0 into tensor memory (each lane its row); over Y_0 as well when step 0 is the last
#pragma unroll 1
          for (int t = 0; t < nrb; ++t) {
            const int rbase = 128 * t + 32 * q, row = rbase + lane;
            if (rbase >= n64) continue;
#pragma unroll 1
            for (int j = grp; 32 * j < n16; j += 2) {
              uint32_t r[32], o[32], h[16], l[16];
              const float d3 = row < n && 32 * j == rbase ? 3.0f : 0.0f;
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const uint8_t* at = X + unit_at(j >> 1, row, 4 * (j & 1) + u);
                const uint4 a = *reinterpret_cast<const uint4*>(at), b = *reinterpret_cast<const uint4*>(at + kPlane);
                const uint32_t hw[4] = {a.x, a.y, a.z, a.w}, lw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                  const float2 x = __half22float2(*reinterpret_cast<const __half2*>(&hw[w]));
                  const float2 y = __half22float2(*reinterpret_cast<const __half2*>(&lw[w]));
                  const float a0 = -(x.x + y.x), a1 = -(x.y + y.y);
                  const int k = 8 * u + 2 * w;
                  r[k] = pick(k, lane, __float_as_uint(d3 + a0), __float_as_uint(a0));
                  r[k + 1] = pick(k + 1, lane, __float_as_uint(d3 + a1), __float_as_uint(a1));
                }
              }
              float sq = 0.0f;
              scale_split_t<FMT_F16, true, false>(r, 1.0f, h, l, sq);
#pragma unroll
              for (int u = 0; u < 16; ++u) {
                o[u] = h[u];
                o[16 + u] = l[u];
              }
              tc::tmem_st32(tmem + kResMaxN * t + lane_base + 32 * j, o);
              if (last0) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  uint8_t* at = X + unit_at(j >> 1, row, 4 * (j & 1) + u);
                  *reinterpret_cast<uint4*>(at) = make_uint4(h[4 * u], h[4 * u + 1], h[4 * u + 2], h[4 * u + 3]);
                  *reinterpret_cast<uint4*>(at + kPlane) = make_uint4(l[4 * u], l[4 * u + 1], l[4 * u + 2], l[4 * u + 3]);
                }
              }
            }
          }
          tc::tmem_wait_st();
        }
        // products with A in tensor memory, in column blocks: 0: Y_1 = P / 2, 1: T_1 = 3I - P / 2 and its defect, 2: Z_2 =
        // P / 4, each over the operand; 4: A_J = P in FP32
#pragma unroll 1
        for (int s = half ? 4 : last0 ? 3 : 0; s != 3 && s < 5; ++s) {
          const float m = s == 2 ? 0.25f : s == 1 ? -0.5f : 0.5f;
          go(0, n16, nrb, nch);
          float sum = 0.0f;
#pragma unroll 1
          for (int c = 0; c < nch; ++c) {
            const int col0 = 64 * c + 32 * grp;
            const bool cols = col0 < n16;
            auto take = [&](int t, uint32_t (&h)[16], uint32_t (&l)[16]) __attribute__((always_inline)) {
              const int slot = nz & 1;
              if (!bad) bad = !tc::mbar_wait_ns(&sh.zf[slot], (nz >> 1) & 1, g.wait_ns);
              bad = __any_sync(0xffffffffu, bad);
              ++nz;
              tc::tc_fence_after();
              uint32_t r[32];
              const int rbase = 128 * t + 32 * q, row = rbase + lane;
              const bool mine = rbase < n64 && cols && !bad;
              if (mine) {
                tc::tmem_ld32(tmem + kRing + 64 * slot + lane_base + 32 * grp, r);
                tc::tmem_wait_ld();
              }
              tc::tc_fence_before();
              if (!bad) tc::mbar_arrive(&sh.ze[slot]);
              if (!mine) return;
              if (s == 4) {
                out(g.Aout + g.a_off[J], rbase, col0, r);
                return;
              }
              if (col0 + 16 >= n16) {   // the MMAs left the second half out: it holds anything
#pragma unroll
                for (int u = 16; u < 32; ++u) r[u] = 0;
              }
              // T_1: off the diagonal -P / 2; on it first P - 2, whose -1/2-fold is 1 - P / 2, then 2 more
              const bool diag = s == 1 && col0 == rbase;
              if (diag) {
                const float two = row < n ? 2.0f : 0.0f;
#pragma unroll
                for (int u = 0; u < 32; ++u) r[u] = pick(u, lane, __float_as_uint(__uint_as_float(r[u]) - two), r[u]);
              }
              float sq = 0.0f;
              scale_split_t<FMT_F16, true, true>(r, m, h, l, sq);
              if (row < n) sum += sq;
              if (diag) {
                uint32_t e = 0;
#pragma unroll
                for (int u = 0; u < 32; ++u) e = pick(u, lane, r[u], e);
                uint32_t th, tl;
                split2(row < n ? 2.0f - 0.5f * __uint_as_float(e) : 0.0f, 0.0f, FMT_F16, th, tl);
                const uint32_t sel = lane & 1 ? 0x5410u : 0x3254u;
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                  h[u] = pick(u, lane >> 1, __byte_perm(h[u], th, sel), h[u]);
                  l[u] = pick(u, lane >> 1, __byte_perm(l[u], tl, sel), l[u]);
                }
              }
            };
            auto put = [&](int t, const uint32_t (&h)[16], const uint32_t (&l)[16]) __attribute__((always_inline)) {
              const int rbase = 128 * t + 32 * q, row = rbase + lane;
              if (s == 4 || rbase >= n64 || !cols || bad) return;
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                uint8_t* at = X + unit_at(c, row, 4 * grp + u);
                *reinterpret_cast<uint4*>(at) = make_uint4(h[4 * u], h[4 * u + 1], h[4 * u + 2], h[4 * u + 3]);
                *reinterpret_cast<uint4*>(at + kPlane) = make_uint4(l[4 * u], l[4 * u + 1], l[4 * u + 2], l[4 * u + 3]);
              }
            };
            // the operand's column block may be overwritten once the block's last product has completed
            uint32_t h0[16], l0[16];
            take(0, h0, l0);
            if (nrb == 2) {
              uint32_t h1[16], l1[16];
              take(1, h1, l1);
              put(1, h1, l1);
            }
            put(0, h0, l0);
          }
          if (s == 1) {
            const float d1 = sqrtf(total(sum) / (float)n);
            steps = 2;
            if (!isfinite(d1)) status = kSubRefine;
            else if (d1 > g.tol_inv) status = g.max_inv > 2 ? kSubAgain : kSubRefine;
            if (status != kSubOk) break;
          }
        }
        if (half == 1 || status != kSubOk) break;
        if (etid == 0) {
          kn = atomicAdd(g.next, 1);
          if (kn < g.count) {
            const int Jn = g.order[kn];
            tc::prefetch_l2(g.ws + (g.a_off[Jn] - g.a_base), sizeof(double) * (size_t)g.sub_n[Jn] * g.sub_n[Jn]);
          }
        }
        // X = Z Z / c, tile by tile: FP32 to memory, and over the accumulators as the next product's A
        const float m = inv * (last0 ? 0.25f : 1.0f);
        float* __restrict__ Xo = g.Xout + (g.a_off[J] - g.a_base);
        go(1, n16, nrb, nch);
#pragma unroll 1
        for (int t = 0; t < nrb; ++t) {
          if (!bad) bad = !tc::mbar_wait_ns(&sh.pf[t], (t ? np1 : np0) & 1, g.wait_ns);
          bad = __any_sync(0xffffffffu, bad);
          ++(t ? np1 : np0);
          tc::tc_fence_after();
          const int rbase = 128 * t + 32 * q;
          if (rbase < n64 && !bad) {
            const uint32_t ta = tmem + kResMaxN * t + lane_base;
#pragma unroll 1
            for (int j = grp; 32 * j < n16; j += 2) {
              uint32_t r[32], h[16], l[16], o[32];
              tc::tmem_ld32(ta + 32 * j, r);
              tc::tmem_wait_ld();
              float sq = 0.0f;
              scale_split_t<FMT_F16, true, false>(r, m, h, l, sq);
#pragma unroll
              for (int u = 0; u < 16; ++u) {
                o[u] = h[u];
                o[16 + u] = l[u];
              }
              tc::tmem_st32(ta + 32 * j, o);
#pragma unroll
              for (int u = 0; u < 32; ++u) r[u] = __float_as_uint(m * __uint_as_float(r[u]));
              out(Xo, rbase, 32 * j, r);
            }
            tc::tmem_wait_st();
          }
        }
        tc::tc_fence_before();
        bar_epi();   // every P tile has been waited for: Z may be overwritten
      }
      if (bar_epi_or(bad)) {   // a wait ran out
        if (etid == 0) {
          sh.err = 1;
          g.prep_out[J] = kSubTimeout;
          atomicExch(g.err, 1);
        }
        go(2, 0, 0, 0);
        break;
      }
      if (etid == 0) {
        g.prep_out[J] = status;
        if (status == kSubAgain) g.again_list[atomicAdd(g.again, 1)] = J;
        else {
          const double prods = 3.0 * steps - (g.Aout ? 1.0 : 2.0), n3 = (double)n * n * n;
          atomicAdd(&g.flops[0], 2.0 * n3 * prods);
          atomicAdd(&g.flops[1], 6.0 * n3 * prods);
        }
      }
    }
  }

  __syncthreads();
  if (sh.err && warp == 1 && lane == 0) {
    tc::mma_commit(&sh.idle);
    tc::mbar_wait_ns(&sh.idle, 0, 50000000ull);
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

}  // namespace

template <typename K>
static bool split_fits(K* kernel) {
  cudaFuncAttributes at{};
  const bool ok = cudaFuncGetAttributes(&at, reinterpret_cast<const void*>(kernel)) == cudaSuccess;
  if (!ok) cudaGetLastError();
  return ok && at.numRegs == kRegsLaunchR;
}

bool inv_res_ready() { return split_fits(&k_inv_res); }

template <typename K>
static nolsm_status ready(K* kernel, const char* name, uint32_t smem) {
  if (!split_fits(kernel)) {
    set_error("%s was not built with the %d registers per thread that its register split needs", name, kRegsLaunchR);
    return NOLSM_ERR_UNSUPPORTED;
  }
  NOLSM_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  return NOLSM_OK;
}

nolsm_status launch_ns_res(const ResSolve& a, int sms, cudaStream_t st) {
  if (a.count <= 0) return NOLSM_OK;
  ResSolve g = a;
  if (g.wait_ns == 0) g.wait_ns = kWaitNsR;
  NOLSM_CUDA_TRY(cudaMemsetAsync(g.next, 0, sizeof(int32_t), st));
  auto run = [&](auto* kernel) -> nolsm_status {
    NOLSM_TRY(ready(kernel, "k_ns_res", kSmemR));
    kernel<<<std::min(sms, a.count), kThreadsR, kSmemR, st>>>(g);
    return NOLSM_OK;
  };
  auto pick = [&](auto exact) -> nolsm_status {
    constexpr bool kE = decltype(exact)::value;
    if (a.main_fmt.fmt == FMT_BF16) return a.main_fmt.terms > 1 ? run(&k_ns_res<FMT_BF16, 3, kE>) : run(&k_ns_res<FMT_BF16, 1, kE>);
    return a.main_fmt.terms > 1 ? run(&k_ns_res<FMT_F16, 3, kE>) : run(&k_ns_res<FMT_F16, 1, kE>);
  };
  NOLSM_TRY(a.exact_xq ? pick(std::true_type{}) : pick(std::false_type{}));
  NOLSM_LAUNCH_CHECK();
  return NOLSM_OK;
}

nolsm_status launch_inv_res(const InvSolve& a, int sms, cudaStream_t st) {
  if (a.count <= 0) return NOLSM_OK;
  InvSolve g = a;
  if (g.wait_ns == 0) g.wait_ns = kWaitNsR;
  NOLSM_TRY(ready(&k_inv_res, "k_inv_res", kSmemI));
  NOLSM_CUDA_TRY(cudaMemsetAsync(g.next, 0, sizeof(int32_t), st));
  k_inv_res<<<std::min(sms, a.count), kThreadsR, kSmemI, st>>>(g);
  NOLSM_LAUNCH_CHECK();
  return NOLSM_OK;
}

}  // namespace nolsm
