// fp64_int.cuh -- correctly rounded FP64 quotient, square root and product on the integer
// and FP32 pipes, and comparisons on the bits.
//
// Why: the SM's FP64 pipe takes 2 lanes a clock, so an FP64 instruction of a warp holds it
// for 16 clocks, while integer and FP32 instructions issue at up to 4 warps a clock
// (measured: add, multiply-add and funnel shift 0.5 clocks per warp and SM, 32 x 32 -> 64
// multiplication 1.0).  A quotient or a root of the compiler is 7-9 FP64 instructions:
// measured 142 and 142 clocks per warp and SM, independent operations, full occupancy.
// The forms below take about 55 integer instructions and one FP32 seed, 17 clocks each,
// and leave the FP64 pipe to the sums and products.
//
// Method: schoolbook long division in two 27..31-bit digits with a 32-bit reciprocal (one
// Newton step on the FP32 seed), and the same for the root with a reciprocal square root;
// then rounding by the sign of the exact remainder at the midpoint between the two
// candidate results, computed modulo 2^64 (the remainder is far below 2^63).  A quotient
// or root of two 53-bit numbers is never such a midpoint, so there are no ties.
// Bounds: the two digits come out 0 to 3 units below the exact quotient (root), where half
// a unit of the result is 16 to 32 of these units; the midpoint test needs less than half.
// The result is therefore the IEEE one, bit for bit, whatever the seed's error within
// 2^-21.9 (tests: seeds moved by +-2 ulp, all 2^23 leading mantissas).
//
// Operands outside 2^-510 <= |x| < 2^512 (subnormal, infinite, NaN, negative under a root)
// take the instruction; a zero numerator gives the signed zero.  That branch is written in
// the asm block so that the surrounding code stays one basic block for the compiler: the
// FP32-bulk unit is compiled with contraction, and what is fused there must not depend on
// how a quotient is formed.
#pragma once
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define RR_HD __host__ __device__ __forceinline__
#else
#define RR_HD inline
#endif

namespace rr {
namespace fpi {

// FP32 seeds.  Any approximation with a relative error of at most 2^-21.9 gives the
// same results (the bounds below use only that).
struct HwSeed {
#if defined(__CUDA_ARCH__)
  static __device__ __forceinline__ float rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
  }
  static __device__ __forceinline__ float rsqrt(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
  }
#endif
};

RR_HD uint32_t mulhi(uint32_t a, uint32_t b) {
#if defined(__CUDA_ARCH__)
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
// the high word of (hi:lo) << n, and the low word of (hi:lo) >> n (0 < n < 32)
RR_HD uint32_t shl_hi(uint32_t hi, uint32_t lo, uint32_t n) {
#if defined(__CUDA_ARCH__)
  return __funnelshift_l(lo, hi, n);
#else
  return (hi << n) | (lo >> (32 - n));
#endif
}
RR_HD uint32_t shr_lo(uint32_t hi, uint32_t lo, uint32_t n) {
#if defined(__CUDA_ARCH__)
  return __funnelshift_r(lo, hi, n);
#else
  return (lo >> n) | (hi << (32 - n));
#endif
}
RR_HD uint32_t hi_word(double x) {
#if defined(__CUDA_ARCH__)
  return (uint32_t)__double2hiint(x);
#else
  uint64_t u;
  std::memcpy(&u, &x, 8);
  return (uint32_t)(u >> 32);
#endif
}
RR_HD uint32_t lo_word(double x) {
#if defined(__CUDA_ARCH__)
  return (uint32_t)__double2loint(x);
#else
  uint64_t u;
  std::memcpy(&u, &x, 8);
  return (uint32_t)u;
#endif
}
RR_HD double make(uint32_t hi, uint32_t lo) {
#if defined(__CUDA_ARCH__)
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t u = ((uint64_t)hi << 32) | lo;
  double x;
  std::memcpy(&x, &u, 8);
  return x;
#endif
}
RR_HD float as_float(uint32_t u) {
#if defined(__CUDA_ARCH__)
  return __uint_as_float(u);
#else
  float f;
  std::memcpy(&f, &u, 4);
  return f;
#endif
}
RR_HD uint32_t float_bits(float f) {
#if defined(__CUDA_ARCH__)
  return __float_as_uint(f);
#else
  uint32_t u;
  std::memcpy(&u, &f, 4);
  return u;
#endif
}

// High words of |x| in [kLo, kLo + kSpan): 2^-510 <= |x| < 2^512.  Quotients of two such
// numbers are normal (exponent difference at most 1021).
constexpr uint32_t kLo = 513u << 20, kSpan = 1022u << 20;

// 1/bm (1 <= bm < 2, the mantissa Bhi:Blo) as a 32-bit fraction, at most 9 units (2^-32)
// too small and never too large: the seed is lowered by 2^-21 (more than its error), so the
// Newton step's correction is positive, and the step's own roundings (4 units) are covered
// by the 5 taken off it.
template <class Seed>
RR_HD uint32_t recip32(uint32_t Bhi, uint32_t Blo) {
  const float f = as_float((shl_hi(Bhi, Blo, 3) & 0x7fffffu) | 0x3f800000u);
  const uint32_t r0 = float_bits(Seed::rcp(f) + (1.0f - 4.76837158203125e-7f)) << 9;
  const uint32_t b32 = shl_hi(Bhi, Blo, 11);
  const uint32_t p = mulhi(r0, b32);
  return mulhi(r0, p * 0xfffffffeu - 5u) + r0;
}

// a / b for 2^-510 <= |a|, |b| < 2^512.
template <class Seed>
RR_HD double div_fast(double a, double b) {
  const uint32_t ahi = hi_word(a), alo = lo_word(a), bhi = hi_word(b), blo = lo_word(b);
  const uint32_t ma = ahi & 0x7fffffffu, mb = bhi & 0x7fffffffu;
  const uint32_t Ahi = (ahi & 0xfffffu) | 0x100000u, Bhi = (bhi & 0xfffffu) | 0x100000u;
  const uint32_t r = recip32<Seed>(Bhi, blo);
  const uint32_t q1 = mulhi(shl_hi(Ahi, alo, 11), r);
  // A 2^31 - q1 B < 10 B: first digit's remainder, then the next 27 bits of the quotient
  const uint64_t rem = (((uint64_t)shr_lo(Ahi, alo, 1) << 32) | (alo << 31)) -
                       ((uint64_t)q1 * blo + ((uint64_t)(q1 * Bhi) << 32));
  const uint32_t q2 = mulhi((uint32_t)(rem >> 25), r);
  const uint64_t Q = (uint64_t)q1 * 0x8000000u + q2;
  const uint32_t Qhi = (uint32_t)(Q >> 32), Qlo = (uint32_t)Q;
  // T = 2m + 1: the midpoint above the truncated result m (54 bits); Q's top bit says
  // whether a/b's mantissa is >= 1
  const uint32_t sh = (Qhi >> 26) + 4u;
  const uint32_t Tlo = shr_lo(Qhi, Qlo, sh) | 1u, Thi = Qhi >> sh;
  // sign of T B - A 2^(57 - sh): negative when the quotient is above the midpoint
  const uint32_t t = mulhi(Tlo, blo) + Thi * blo + Tlo * Bhi - (alo << (26u - sh));
  const uint64_t m = ((((uint64_t)Thi << 32) | Tlo) >> 1) + (t >> 31);
  const uint32_t E = (ma - Ahi) - (mb - Bhi) + (1017u << 20) + (sh << 20);
  const uint32_t hi = ((uint32_t)(m >> 32) + E) | ((ahi ^ bhi) & 0x80000000u);
  return make(hi, (uint32_t)m);
}

// sqrt(x) for 2^-510 <= x < 2^512.
template <class Seed>
RR_HD double sqrt_fast(double x) {
  const uint32_t hi = hi_word(x), lo = lo_word(x);
  const uint32_t par = ~(hi >> 20) & 1u;  // 1: odd power of two
  const float f = as_float(((shl_hi(hi, lo, 3) & 0xffffffu) ^ 0x800000u) + 0x3f800000u);
  const uint32_t y0 = float_bits(Seed::rsqrt(f) + (1.0f - 4.76837158203125e-7f)) << 9;
  const uint64_t M = ((((uint64_t)((hi & 0xfffffu) | 0x100000u)) << 32) | lo) << par;
  const uint32_t m32 = (uint32_t)(M >> 22);
  const uint32_t v = mulhi(mulhi(y0, y0), m32);
  const uint32_t y = mulhi(y0, v * 0xfffffffeu + (0x80000000u - 6u)) + y0;
  const uint32_t s0 = mulhi(m32, y);
  const uint64_t rem = (M << 8) - (uint64_t)s0 * s0;
  const uint32_t s1 = mulhi((uint32_t)(rem >> 4), y);
  const uint64_t Q = (uint64_t)s0 * 0x8000000u + s1;
  const uint64_t T = (Q >> 4) | 1u;
  const uint32_t Tlo = (uint32_t)T, Thi = (uint32_t)(T >> 32);
  // sign of T^2 - M 2^54
  const uint32_t t = mulhi(Tlo, Tlo) + Tlo * (Thi + Thi) - ((uint32_t)M << 22);
  const uint64_t m = (T >> 1) + (t >> 31);
  const uint32_t E = ((hi + (1021u << 20)) >> 1) & 0xfff00000u;
  return make((uint32_t)(m >> 32) + E, (uint32_t)m);
}

// A product takes ~30 integer instructions, 14 clocks per warp and SM, against 18.7 measured
// for the instruction, and runs beside it: two sums and two products per turn, 78 clocks
// with FP64 products, 39 with these (8 to 32 warps per SM).  It has no fallback of its own:
// an FP64 instruction with every lane predicated off still holds the pipe (78 clocks again),
// so callers test a window of their operands once and branch around a whole evaluation.
// a b for normal a, b and a product in the normal range: the 106-bit product of the
// mantissas from four 32 x 32 -> 64 multiplications, rounded to nearest even.  ZEROS: a
// and b may also be zeros.
template <bool ZEROS = false>
RR_HD double mul_fast(double a, double b) {
  const uint32_t ahi = hi_word(a), alo = lo_word(a), bhi = hi_word(b), blo = lo_word(b);
  // A 2^10 and B: the sums below stay within 64 bits
  const uint32_t Ah = ((shl_hi(ahi, alo, 10) & 0x3fffffffu) | 0x40000000u), Al = alo << 10;
  const uint32_t Bh = (bhi & 0xfffffu) | 0x100000u;
  const uint64_t w0 = (uint64_t)Al * blo;
  const uint64_t w1 = (uint64_t)Ah * blo + (uint32_t)(w0 >> 32);
  const uint64_t w2 = (uint64_t)Al * Bh + w1;
  const uint64_t w3 = (uint64_t)Ah * Bh + (uint32_t)(w2 >> 32);
  const uint32_t h = (uint32_t)(w3 >> 32), m = (uint32_t)w3, l = (uint32_t)w2;
  const uint32_t s = 2u - (h >> 19);  // normalising shift: 2 where the product is below 2
  const uint32_t mh = shl_hi(h, m, s), ml = shl_hi(m, l, s);
  const uint32_t r = (l << s) | ((uint32_t)w0 != 0u ? 1u : 0u);
  // round half to even: carry of the bits below + half - 1 + last bit
  const uint32_t up = (uint32_t)(((uint64_t)r + (0x7fffffffu + (ml & 1u))) >> 32);
  const uint32_t ea = ahi & 0x7ff00000u, eb = bhi & 0x7ff00000u;
  const uint32_t E = ea + eb - (1022u << 20) - (s << 20);
  uint64_t z = (((uint64_t)(mh + E) << 32) | ml) + up;
  if (ZEROS && (ea == 0u || eb == 0u)) z = 0u;
  return make((uint32_t)(z >> 32) | ((ahi ^ bhi) & 0x80000000u), (uint32_t)z);
}

// x as a float, rounded to nearest even, for 2^-126 <= |x| < 2^127 or zero.
RR_HD float to_float_fast(double x) {
  const uint32_t hi = hi_word(x), lo = lo_word(x);
  const uint32_t m = shl_hi(hi & 0x7fffffffu, lo, 3) - (896u << 23);
  const uint32_t up = (uint32_t)(((uint64_t)(lo << 3) + (0x7fffffffu + (m & 1u))) >> 32);
  const bool zero = ((hi & 0x7fffffffu) | lo) == 0u;
  return as_float((zero ? 0u : m + up) | (hi & 0x80000000u));
}
// a normal float or zero as a double
RR_HD double to_double_fast(float f) {
  const uint32_t u = float_bits(f), m = u & 0x7fffffffu;
  return make((u & 0x80000000u) | (m ? (m >> 3) + (896u << 20) : 0u), m << 29);
}

// Comparisons on the bits (an FP64 comparison takes the FP64 pipe like a product).
RR_HD uint64_t bits(double x) { return ((uint64_t)hi_word(x) << 32) | lo_word(x); }
constexpr uint64_t kInf = 0x7ff0000000000000ull;
// x > y for y >= 0 (false where x is NaN)
RR_HD bool gt_nonneg(double x, double y) { return bits(x) > bits(y) && bits(x) <= kInf; }
// x > 0
RR_HD bool pos(double x) { return bits(x) - 1u < kInf; }
// a zero, or 2^(lo-1023) <= |x| < 2^(lo+n-1023)
RR_HD bool in_window_or_zero(double x, uint32_t lo, uint32_t n) {
  const uint32_t h = hi_word(x) & 0x7fffffffu;
  return h - (lo << 20) < (n << 20) || (h | lo_word(x)) == 0u;
}
// |x| > |y| (false where either is NaN)
RR_HD bool mag_gt(double x, double y) {
  const uint64_t u = bits(x) & 0x7fffffffffffffffull, v = bits(y) & 0x7fffffffffffffffull;
  return u > v && u <= kInf;
}
// |x| <= y for y >= 0 (false where x is NaN)
RR_HD bool mag_le(double x, double y) { return (bits(x) & 0x7fffffffffffffffull) <= bits(y); }
// 0 <= x < 1, for an x that is not a negative number (false where it is NaN)
RR_HD bool below_one(double x) { return hi_word(x) < 0x3ff00000u; }
// 2^(lo-1023) <= |x| < 2^(lo+n-1023)
RR_HD bool in_window(double x, uint32_t lo, uint32_t n) {
  return (hi_word(x) & 0x7fffffffu) - (lo << 20) < (n << 20);
}

#if defined(__CUDACC__)
// a / b.
__device__ __forceinline__ double div(double a, double b) {
  const uint32_t ahi = hi_word(a), alo = lo_word(a), bhi = hi_word(b);
  const uint32_t ma = ahi & 0x7fffffffu, mb = bhi & 0x7fffffffu;
  const bool za = (ma | alo) == 0u;
  const bool plain = (mb - kLo < kSpan) && ((ma - kLo < kSpan) || za);
  double q = div_fast<HwSeed>(a, b);
  if (za) q = make((ahi ^ bhi) & 0x80000000u, 0u);
  asm("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %1, 0;\n\t@p bra DONE;\n\tdiv.rn.f64 %0, %2, %3;\nDONE:\n\t}"
      : "+d"(q)
      : "r"((int)plain), "d"(a), "d"(b));
  return q;
}

// (float)x and (double)f: a conversion takes the FP64 pipe like a product.  The instruction
// stays for the rest of the range, behind a call (a branch that is not turned into predicates).
static __device__ __noinline__ float to_float_slow(double x) { return (float)x; }
static __device__ __noinline__ double to_double_slow(float f) { return (double)f; }
__device__ __forceinline__ float to_float(double x) {
  return in_window_or_zero(x, 897, 253) ? to_float_fast(x) : to_float_slow(x);
}
__device__ __forceinline__ double to_double(float f) {
  const uint32_t m = float_bits(f) & 0x7fffffffu;
  return m - 0x00800000u < 0x7f000000u || m == 0u ? to_double_fast(f) : to_double_slow(f);
}

// sqrt(x).
__device__ __forceinline__ double sqrt(double x) {
  double s = sqrt_fast<HwSeed>(x);
  asm("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %1, 0;\n\t@p bra DONE;\n\tsqrt.rn.f64 %0, %2;\nDONE:\n\t}"
      : "+d"(s)
      : "r"((int)(hi_word(x) - kLo < kSpan)), "d"(x));
  return s;
}
#endif

}  // namespace fpi
}  // namespace rr
