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
//
// The streaming kernel (k_ns_tc), which these submatrices used before and larger ones still use, keeps the operands of
// two submatrices per SM in global memory: 0.6 MB of TMA traffic a product at n = 172, more than the L2 holds over 152
// SMs (14.6 GB of DRAM traffic on 4,096 submatrices). Here the products are bound by the MMAs, 12,100 cycles a step at
// n = 172 in the three-term split, and the epilogue of T tile 0 and of the Z blocks runs beside them.
//
// Roles: warp 1 issues the MMAs (converged, one elected lane), warps 4-11 are the epilogue (two groups of four, even
// and odd 32-column chunks), which also starts and finishes the submatrices. All waits are bounded.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

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
static_assert(kExtra >= 64 * 128, "the second row tile's A reads up to 64 rows past the last block");
static_assert(kSmemR <= 227 * 1024, "shared memory");
constexpr uint32_t kRing = 2 * kResMaxN;          // tensor memory column of the first Z accumulator
constexpr uint64_t kWaitNsR = 2000000000ull;

struct StepInfo { int term, n16, nrb, nch; Fmt f; };   // what the MMA warp needs of a step

struct SharedR {
  uint64_t xr, pf[2], tr[2], zf[2], ze[2], idle;
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

// u == k ? a : b as an instruction that the compiler does not fold into an indexed (local memory) array access: local
// memory shares its bandwidth with the MMAs' operands
__device__ __forceinline__ uint32_t pick(int u, int k, uint32_t a, uint32_t b) {
  uint32_t r;
  asm("{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %1, %2;\n\tselp.b32 %0, %3, %4, p;\n\t}" : "=r"(r) : "r"(u), "r"(k), "r"(a), "r"(b));
  return r;
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

__global__ void __launch_bounds__(kThreadsR, 1) k_ns_res(ResSolve g) {
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
      tc::mbar_init(&sh.ze[t], kEpiR);
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
      return (bool)__all_sync(0xffffffffu, tc::mbar_wait(b, parity, tc::globaltimer() + more * g.wait_ns));
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
    for (;;) {
      // ---- the next submatrix of at most kResMaxN rows
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
        const Fmt f = g.main_fmt;
        // eight rows a warp pass; sixteen lanes along a row, four adjacent columns a lane, in three blocks of 64 columns:
        // 48 loads in flight (no condition holds a load back), then 8-byte stores of hi and lo
        for (int i0 = 8 * ew; i0 < n64; i0 += 64) {
          float v[4][3][4];
          const int jl = 4 * (lane & 15);
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const float* row = A + min(i0 + 2 * r + (lane >> 4), n - 1) * n;
#pragma unroll
            for (int t = 0; t < 3; ++t)
#pragma unroll
              for (int u = 0; u < 4; ++u) v[r][t][u] = __ldg(row + min(64 * t + jl + u, n - 1));
          }
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int i = i0 + 2 * r + (lane >> 4);
#pragma unroll
            for (int t = 0; t < 3; ++t) {
              float w[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const int j = 64 * t + jl + u;
                w[u] = i < n && j < n ? (v[r][t][u] - (i == j ? fmu : 0.0f)) * inv : 0.0f;
              }
              uint2 h, l;
              split2(w[0], w[1], f.fmt, h.x, l.x);
              split2(w[2], w[3], f.fmt, h.y, l.y);
              uint8_t* at = X + unit_at(t, i, (lane & 15) >> 1) + 8 * (lane & 1);
              if (64 * t < n64) {
                *reinterpret_cast<uint2*>(at) = h;
                if (f.terms > 1) *reinterpret_cast<uint2*>(at + kPlane) = l;
              }
            }
          }
        }
      }
      int phase = 0, refine_left = g.refine_steps, steps = 0, rsteps = 0, status = kSubNotConv;
      float dprev = INFINITY;
      Fmt fcur = g.main_fmt;
      bool last = false, bad = false;
      if (etid == 0) sh.mm = StepInfo{0, n16, nrb, nch, fcur};
      tc::fence_proxy_async_smem();
      tc::tc_fence_before();
      bar_epi();
      tc::mbar_arrive(&sh.xr);
      int Jn = -1;
      while (!last) {
        // ---- P -> T, tile by tile
        float part = 0.0f;
        for (int t = 0; t < nrb; ++t) {
          if (!bad) bad = !tc::mbar_wait(&sh.pf[t], (t ? np1 : np0) & 1, tc::globaltimer() + g.wait_ns);
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
              scale_split<true>(r, -1.0f, fcur, h, l, sq);
              if (row < n) part += sq;
              if (diag) {
                uint32_t e = 0;
#pragma unroll
                for (int u = 0; u < 32; ++u) e = pick(u, lane, r[u], e);
                uint32_t th, tl;
                split2(row < n ? 2.0f - __uint_as_float(e) : 0.0f, 0.0f, fcur.fmt, th, tl);
                const uint32_t sel = lane & 1 ? 0x5410u : 0x3254u;   // (low of x, low of t) or (low of t, high of x)
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                  h[u] = pick(u, lane >> 1, __byte_perm(h[u], th, sel), h[u]);
                  l[u] = pick(u, lane >> 1, __byte_perm(l[u], tl, sel), l[u]);
                }
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
        Fmt fnxt = fcur;
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
              fnxt = g.refine_fmt;
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
        // ---- Z -> X', column block by column block (two 32-column chunks, one a group)
        for (int c = 0; c < nch; ++c) {
          const int col0 = 64 * c + 32 * grp;
          const bool cols = col0 < n16;
          // row tile t's block out of its accumulator, halved and split
          auto take = [&](int t, uint32_t (&h)[16], uint32_t (&l)[16]) {
            const int slot = nz & 1;
            if (!bad) bad = !tc::mbar_wait(&sh.zf[slot], (nz >> 1) & 1, tc::globaltimer() + g.wait_ns);
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
            if (mine) scale_split<false>(r, 0.5f, fnxt, h, l, sq);
          };
          auto put = [&](int t, const uint32_t (&h)[16], const uint32_t (&l)[16]) {
            const int rbase = 128 * t + 32 * q, row = rbase + lane;
            if (rbase >= n64 || !cols || bad) return;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              uint8_t* at = X + unit_at(c, row, 4 * grp + u);
              *reinterpret_cast<uint4*>(at) = make_uint4(h[4 * u], h[4 * u + 1], h[4 * u + 2], h[4 * u + 3]);
              if (fnxt.terms > 1)
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
        fcur = fnxt;
        if (!last) {
          if (etid == 0) sh.mm.f = fcur;
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
      const int units = n16 / 16, nitem = ((n + 31) / 32) * kSplit;   // of k: 16 at a time
      for (int cg = 0; cg < b; cg += 8) {
        const int cn = min(8, b - cg);
        for (int e = etid; e < n16 * 8; e += kEpiR) {
          const int k = e >> 3, c = e & 7;
          Qs[e] = (k < n && c < cn) ? (float)Q[(size_t)k * b + cg + c] : 0.0f;
        }
        bar_epi();
        for (int it = ew; it < nitem; it += 8) {
          const int i = 32 * (it / kSplit) + lane, kq = it % kSplit;
          const int k0 = 16 * (units * kq / kSplit), k1 = 16 * (units * (kq + 1) / kSplit);
          uint64_t s[4], e[4];
          if (fcur.fmt == FMT_BF16) {
            if (fcur.terms > 1) xq_part<FMT_BF16, true>(X, i, k0, k1, Qs, s, e);
            else xq_part<FMT_BF16, false>(X, i, k0, k1, Qs, s, e);
          } else {
            if (fcur.terms > 1) xq_part<FMT_F16, true>(X, i, k0, k1, Qs, s, e);
            else xq_part<FMT_F16, false>(X, i, k0, k1, Qs, s, e);
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
        float x = from_bits(*reinterpret_cast<const uint16_t*>(X + at), fcur.fmt);
        if (fcur.terms > 1) x += from_bits(*reinterpret_cast<const uint16_t*>(X + kPlane + at), fcur.fmt);
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
    tc::mbar_wait(&sh.idle, 0, tc::globaltimer() + 50000000ull);
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

}  // namespace

nolsm_status launch_ns_res(const ResSolve& a, int sms, cudaStream_t st) {
  if (a.count <= 0) return NOLSM_OK;
  ResSolve g = a;
  if (g.wait_ns == 0) g.wait_ns = kWaitNsR;
  cudaFuncAttributes at{};
  NOLSM_CUDA_TRY(cudaFuncGetAttributes(&at, reinterpret_cast<const void*>(&k_ns_res)));
  if (at.numRegs != kRegsLaunchR) {
    set_error("k_ns_res was built with %d registers per thread; its register split needs exactly %d", at.numRegs,
              kRegsLaunchR);
    return NOLSM_ERR_UNSUPPORTED;
  }
  NOLSM_CUDA_TRY(cudaFuncSetAttribute(k_ns_res, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemR));
  NOLSM_CUDA_TRY(cudaMemsetAsync(g.next, 0, sizeof(int32_t), st));
  k_ns_res<<<std::min(sms, a.count), kThreadsR, kSmemR, st>>>(g);
  NOLSM_LAUNCH_CHECK();
  return NOLSM_OK;
}

}  // namespace nolsm
