// Operand formats of the tensor-core kernels and the splitting of FP32 values into them.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace nolsm {

enum : int { FMT_F16 = 0, FMT_BF16 = 1, FMT_E4M3 = 2 };

struct Fmt {
  int fmt;    // FMT_F16 / FMT_BF16 / FMT_E4M3
  int terms;  // 1 or 3 (E4M3: 1)
};

__device__ __forceinline__ float from_bits(uint16_t b, int fmt) {
  if (fmt == FMT_BF16) return __bfloat162float(__ushort_as_bfloat16(b));
  return __half2float(__ushort_as_half(b));
}

// Two values rounded to the 2-byte format (packed) and their low parts x - round(x) rounded likewise.
__device__ __forceinline__ void split2(float a, float b, int fmt, uint32_t& hi, uint32_t& lo) {
  if (fmt == FMT_BF16) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const float2 hf = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(a - hf.x, b - hf.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
  } else {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 hf = __half22float2(h);
    const __half2 l = __floats2half2_rn(a - hf.x, b - hf.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
  }
}

// s + c <- s + c + p with s = fl(s + p) and the rounding error of that sum added to c (Knuth's TwoSum).
__device__ __forceinline__ void two_sum(float& s, float& c, float p) {
  const float t = s + p;
  const float z = t - s;
  c += (s - (t - z)) + (p - z);
  s = t;
}

// Packed pairs of FP32 numbers: two operations per instruction.
__device__ __forceinline__ uint64_t pair2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpair2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// s + e <- s + e + a x in pairs, na = -a: the product's rounding error by FMA, the sum's by TwoSum, whatever the order of
// magnitude of the two; e collects them in FP32.
__device__ __forceinline__ void add_product2(uint64_t& s, uint64_t& e, uint64_t a, uint64_t na, uint64_t x) {
  const uint64_t neg = pair2(-1.0f, -1.0f);
  const uint64_t p = mul2(a, x), m = fma2(na, x, p);   // p - a x
  const uint64_t t = add2(s, p), z = fma2(s, neg, t);  // t - s
  const uint64_t d = add2(fma2(fma2(z, neg, t), neg, s), fma2(z, neg, p));
  e = fma2(m, neg, add2(e, d));
  s = t;
}

// How X Q sums its products: in FP32, eight or sixteen at a time between compensated additions, or each with its own
// rounding error where n x b is large (b above 13 at n = 192, above 8 at n = 300, any b from n = 440 on): what the plain
// sums lose there is 3e-8 of D. 512 submatrices of 23 functions a molecule: 24.0 ms without, 25.0 with it.
__host__ __device__ inline bool exact_xq(int n, int b) { return 4 * ((n + 63) & ~63) * ((b + 7) & ~7) + 8 * n * b > 32768; }

// u == k ? a : b as an instruction that the compiler does not fold into an indexed (local memory) array access: local
// memory shares its bandwidth with the MMAs' operands
__device__ __forceinline__ uint32_t pick(int u, int k, uint32_t a, uint32_t b) {
  uint32_t r;
  asm("{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %1, %2;\n\tselp.b32 %0, %3, %4, p;\n\t}" : "=r"(r) : "r"(u), "r"(k), "r"(a), "r"(b));
  return r;
}

// m times 32 accumulators of one row as packed hi (and lo) pairs, and with kSq the sum of the squares added to sq.
template <int kFmt, bool kLo, bool kSq>
__device__ __forceinline__ void scale_split_t(const uint32_t (&r)[32], float m, uint32_t (&h)[16], uint32_t (&l)[16],
                                              float& sq) {
  const uint64_t mm = pair2(m, m), neg = pair2(-1.0f, -1.0f);
  uint64_t s0 = 0, s1 = 0;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const uint64_t v = mul2(pair2(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1])), mm);
    if (kSq) (j & 1 ? s1 : s0) = fma2(v, v, j & 1 ? s1 : s0);
    const float2 f = unpair2(v);
    float2 hf;
    if (kFmt == FMT_BF16) {
      const __nv_bfloat162 b = __floats2bfloat162_rn(f.x, f.y);
      h[j] = *reinterpret_cast<const uint32_t*>(&b);
      hf = make_float2(__uint_as_float(h[j] << 16), __uint_as_float(h[j] & 0xFFFF0000u));
    } else {
      const __half2 b = __floats2half2_rn(f.x, f.y);
      h[j] = *reinterpret_cast<const uint32_t*>(&b);
      hf = __half22float2(b);
    }
    if (kLo) {
      const float2 e = unpair2(fma2(pair2(hf.x, hf.y), neg, v));
      if (kFmt == FMT_BF16) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(e.x, e.y);
        l[j] = *reinterpret_cast<const uint32_t*>(&b);
      } else {
        const __half2 b = __floats2half2_rn(e.x, e.y);
        l[j] = *reinterpret_cast<const uint32_t*>(&b);
      }
    }
  }
  if (kSq) {
    const float2 a = unpair2(s0), b = unpair2(s1);
    sq += (a.x + a.y) + (b.x + b.y);
  }
}
template <bool kSq>
__device__ __forceinline__ void scale_split(const uint32_t (&r)[32], float m, Fmt f, uint32_t (&h)[16], uint32_t (&l)[16],
                                            float& sq) {
  if (f.fmt == FMT_BF16) {
    if (f.terms > 1) scale_split_t<FMT_BF16, true, kSq>(r, m, h, l, sq);
    else scale_split_t<FMT_BF16, false, kSq>(r, m, h, l, sq);
  } else {
    if (f.terms > 1) scale_split_t<FMT_F16, true, kSq>(r, m, h, l, sq);
    else scale_split_t<FMT_F16, false, kSq>(r, m, h, l, sq);
  }
}

}  // namespace nolsm
