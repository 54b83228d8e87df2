// gbh_intmath.cuh -- FP64 building blocks computed on the integer pipes.
//
// On GB300 a warp's FP64 instruction holds the FP64 pipe of its SM
// sub-partition for 64 cycles (2 lanes per SM clock), and the kernels of the
// scheme are bound by that pipe with about 12% of the issue slots used.  An
// integer multiply-add with a 64-bit result (IMAD.WIDE), a funnel shift or a
// 64-bit add takes 2 cycles there and runs beside the FP64 pipe without
// slowing it: measured, 4 DFMA alone 258 cycles, with 128 IMAD.WIDE 259.
// So a function that takes three FP64 instructions (192 cycles) is cheaper as
// 30 integer ones, and chains of products, quotients and roots of positive
// numbers are cheaper still when they stay in an unpacked form and are rounded
// once at their end.
//
// Wide: a positive number as a 63-bit mantissa and an exponent,
//     value = (h 2^32 + l) 2^(e - 1023 - 62),  2^62 <= h 2^32 + l < 2^63,
// e in the biased form of a double; a reciprocal, a root or a product of them may
// be up to 64 units below 2^62, which products, sums, roots and the rounding take
// (and wide_rcp_low, where a reciprocal is taken of one).  Products,
// reciprocals and roots are computed to a relative error below 2^-58 (stated at
// each), so a double rounded from a chain of them (wide_pack, to nearest) is
// within 0.55 ulp of the exact value: tighter than the same chain of FP64
// operations, each of which rounds to half an ulp.  Exponents are plain ints
// and do not overflow.  Reciprocal and root start from the FP32 approximations
// (relative error below 2^-22) and take one Newton step in 32-bit fixed point
// and one against the exact residual in 64 bits (the classical iterations for
// 1/x and 1/sqrt(x), see e.g. Muller et al., Handbook of Floating-Point
// Arithmetic, ch. 5).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define GBH_HD __host__ __device__ __forceinline__
#else
#define GBH_HD inline
#endif
#ifndef __CUDA_ARCH__
#include <cmath>
#include <cstring>
#endif

namespace gbh {

struct Wide {
  uint32_t h, l;
  int e;
};

namespace imath {

GBH_HD uint32_t hi32(uint64_t x) { return (uint32_t)(x >> 32); }
GBH_HD uint32_t lo32(uint64_t x) { return (uint32_t)x; }
GBH_HD uint64_t pair(uint32_t h, uint32_t l) { return ((uint64_t)h << 32) | l; }
GBH_HD uint64_t mulu(uint32_t a, uint32_t b) { return (uint64_t)a * b; }
GBH_HD int64_t muls(int32_t a, int32_t b) { return (int64_t)a * b; }

// the low 32 bits of (h:l) >> n, n < 32
GBH_HD uint32_t shr_lo(uint32_t h, uint32_t l, int n) {
#ifdef __CUDA_ARCH__
  return __funnelshift_r(l, h, n);
#else
  return (uint32_t)(pair(h, l) >> (n & 31));
#endif
}
// the high 32 bits of (h:l) << n, n < 32
GBH_HD uint32_t shl_hi(uint32_t h, uint32_t l, int n) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(l, h, n);
#else
  return hi32(pair(h, l) << (n & 31));
#endif
}

GBH_HD uint32_t bits_of(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t u;
  memcpy(&u, &x, 4);
  return u;
#endif
}
GBH_HD float float_of(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float x;
  memcpy(&x, &u, 4);
  return x;
#endif
}
GBH_HD float rcp_seed(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / x;
#endif
}
GBH_HD float rsqrt_seed(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / sqrtf(x);
#endif
}

}  // namespace imath

// The magnitude of the double with high word hi and low word lo (exponent
// field e as it stands: 0 and subnormals read as 2^-1023 (1 + f), infinities
// and NaN as 2^1024 (1 + f); the caller decides what those mean).
GBH_HD Wide wide_unpack(uint32_t hi, uint32_t lo) {
  Wide r;
  r.h = (imath::shl_hi(hi, lo, 10) & 0x3fffffffu) | 0x40000000u;
  r.l = lo << 10;
  r.e = (int)((hi >> 20) & 0x7ffu);
  return r;
}

// The bit pattern of the double nearest to a (exact ties upwards), for a
// normal result.  The mantissa's rounding carry runs into the exponent field.
GBH_HD uint64_t wide_pack(const Wide& a) {
  const uint64_t m = imath::pair(a.h, a.l) + 512;
  return imath::pair((imath::hi32(m) >> 10) + ((uint32_t)(a.e - 1) << 20),
                     imath::shr_lo(imath::hi32(m), imath::lo32(m), 10));
}

// a b: relative error below 2^-59 (the low product is left out; a shift by 1
// or 2 brings the product back to 63 bits).
GBH_HD Wide wide_mul(const Wide& a, const Wide& b) {
  using namespace imath;
  const uint64_t t = mulu(a.h, b.l) + mulu(a.l, b.h);   // < 2^64, as h < 2^31
  const uint64_t p = mulu(a.h, b.h) + hi32(t);          // [2^60, 2^62)
  const uint32_t ph = hi32(p), pl = lo32(p);
  const int top = (int)(ph >> 29);                      // 1: p >= 2^61
  Wide r;
  r.h = shl_hi(ph, pl, 2 - top);
  r.l = pl << (2 - top);
  r.e = a.e + b.e - 1023 + top;
  return r;
}

// a + b: relative error below 2^-61 (the bits shifted out of the smaller one).
GBH_HD Wide wide_add(const Wide& a, const Wide& b) {
  using namespace imath;
  const int d = a.e - b.e;
  const bool sw = d < 0;
  const uint64_t big = sw ? pair(b.h, b.l) : pair(a.h, a.l);
  const uint64_t small = sw ? pair(a.h, a.l) : pair(b.h, b.l);
  const int n = sw ? -d : d;
  const uint64_t sum = big + (small >> (n < 63 ? n : 63));
  const int top = (int)(hi32(sum) >> 31);
  Wide r;
  r.h = hi32(sum) >> top;
  r.l = shr_lo(hi32(sum), lo32(sum), top);
  r.e = (sw ? b.e : a.e) + top;
  return r;
}

// 1 / a: relative error below 2^-58.5.  a is at least 2^62: unpacked, a product
// of unpacked numbers, or a sum whose larger term is one of them.
GBH_HD Wide wide_rcp(const Wide& a) {
  using namespace imath;
  // seed: R0 = 1/f in units of 2^-31, f in [1, 2) the leading 24 bits of a; n0 = -R0
  const uint32_t rb = bits_of(rcp_seed(float_of((a.h >> 7) + 0x3f000000u)));
  const int32_t n0 = (int32_t)(0x3e800000u * 128u - rb * 128u);
  // -h R0 = -(1 - e0) in units of 2^-61; its bits 12.. are e0 in units of 2^-49
  const uint64_t p0 = (uint64_t)muls((int32_t)a.h, n0);
  const int32_t e0 = (int32_t)shr_lo(hi32(p0), lo32(p0), 12);
  // R1 = R0 (1 + e0): relative error below 2^-29.4, R1 <= 2^31
  const int32_t x = (int32_t)hi32((uint64_t)muls(n0, e0));
  const uint32_t r1 = 0u - ((uint32_t)n0 + (uint32_t)(x >> 17));
  // E = a R1 - 1 in units of 2^-61 (|E| < 2^32), c = R1 E in units of 2^-60;
  // the signed reading of r1 = 2^31 is harmless: then 0 <= E < 2^32
  const uint64_t E = mulu(a.h, r1) + pair(0xe0000000u, hi32(mulu(a.l, r1)));
  const uint64_t c = (uint64_t)muls((int32_t)hi32(E), (int32_t)r1) + hi32(mulu(lo32(E), r1));
  // R1 - c in units of 2^-63, less one unit so that the result stays below 2^63
  Wide r;
  r.h = r1 + ~shl_hi(hi32(c), lo32(c), 3);
  r.l = ~(lo32(c) << 3);
  r.e = 2045 - a.e;
  return r;
}

// 1 / a of a number that may lie below 2^62, as a sum whose larger term is a root:
// taken as 2^62 there, which changes the result by as many units of 2^-62 as it
// lies below (three for a root).  wide_rcp itself is off by 2^-21 on such numbers:
// its seed's 1/f exceeds 1.  Three instructions, so not in every reciprocal.
GBH_HD Wide wide_rcp_low(const Wide& a) {
  const bool low = a.h < 0x40000000u;
  return wide_rcp(Wide{low ? 0x40000000u : a.h, low ? 0u : a.l, a.e});
}

// sqrt(a): relative error below 2^-57.
GBH_HD Wide wide_sqrt(const Wide& a) {
  using namespace imath;
  const int odd = ~a.e & 1;                                  // 2^odd m in [1, 4) has an even exponent
  const uint32_t H = shl_hi(a.h, a.l, odd), L = a.l << odd;   // in units of 2^-62
  // seed: R0 = 1/sqrt(f) in units of 2^-31, below 2^31
  // (from f >= 1: a product or root a few units below 2^62 is taken there)
  const uint32_t hs = a.h > 0x40000000u ? a.h : 0x40000000u;
  const uint32_t rb = bits_of(rsqrt_seed(float_of((hs >> 7) + 0x3f000000u + ((uint32_t)odd << 23))));
  const uint32_t r0 = (rb - 0x3e800001u) * 128u;
  // R0^2 in units of 2^-32 (rounded); d0 = H R0^2 - 1 in units of 2^-49
  const uint64_t q = mulu(r0, r0) + (1u << 29);
  const uint64_t p0 = mulu(H, shl_hi(hi32(q), lo32(q), 2));
  const int32_t d0 = (int32_t)shr_lo(hi32(p0), lo32(p0), 13);
  // R1 = R0 (1 - d0/2) in units of 2^-32, three units low so that it is below
  // 1/sqrt(a) (relative error below 2^-28.9)
  const uint64_t x = (uint64_t)muls((int32_t)r0, d0) + (1ull << 48);
  const uint32_t r1 = 2u * r0 - 3u - (uint32_t)((int32_t)hi32(x) >> 17);
  // S1 = a R1 in units of 2^-31 (below sqrt(a)), the residual a - S1^2 in
  // units of 2^-62 (0 .. 2^37) and S1 + (a - S1^2) R1 / 2
  const uint64_t p1 = mulu(H, r1);
  const uint32_t s1 = shl_hi(hi32(p1), lo32(p1), 1);
  const uint64_t R = pair(H, L) - mulu(s1, s1);
  const uint64_t s = pair(s1, 0) + hi32(mulu(lo32(R), r1)) + mulu(hi32(R), r1);
  Wide r;
  r.h = hi32(s) >> 1;
  r.l = shr_lo(hi32(s), lo32(s), 1);
  r.e = (a.e + 1023 - odd) >> 1;
  return r;
}

// sign(p) min(|m + p| / 4, |m|, |p|) where the doubles with bit patterns m and p
// have the same strict sign, else +0: half the MC-limited slope of the
// differences m and p, |m + p| / 4 rounded once to nearest even (as the FP64 sum
// would be).  With a <= b the magnitudes, (a + b) / 4 < a needs b < 3 a, so the
// exponents differ by at most 2 there and the 53-bit mantissas add exactly in 64
// bits.  For a below 2^-1021 the result is a itself.
GBH_HD uint64_t half_slope(uint64_t m, uint64_t p) {
  using namespace imath;
  const uint32_t mh = hi32(m) & 0x7fffffffu, ph = hi32(p) & 0x7fffffffu;
  const bool less = pair(mh, lo32(m)) < pair(ph, lo32(p));
  const uint32_t ah = less ? mh : ph, al = less ? lo32(m) : lo32(p);
  const uint32_t bh = less ? ph : mh, bl = less ? lo32(p) : lo32(m);
  const int ea = (int)(ah >> 20), d = (int)(bh >> 20) - ea;
  const uint32_t fa = (ah & 0xfffffu) | 0x100000u, fb = (bh & 0xfffffu) | 0x100000u;
  const int n = d < 3 ? d : 3;
  const uint64_t S = pair(fa, al) + pair(shl_hi(fb, bl, n), bl << n);   // (a + b) 2^(1075 - ea), from 2^53
  const int top = (int)(hi32(S) >> 22) & 1;                              // S >= 2^54 (below 2^55 where it is taken)
  const uint32_t lsb = shr_lo(hi32(S), lo32(S), 1 + top) & 1u;
  const uint64_t r = S + (uint32_t)top + lsb;
  const uint32_t ch = (hi32(r) >> (1 + top)) + ((uint32_t)(ea - 2 + top) << 20);
  const uint32_t cl = shr_lo(hi32(r), lo32(r), 1 + top);
  const bool central = d < 3 && ea > 1 && pair(ch, cl) < pair(ah, al);
  const bool zero = (int32_t)(hi32(m) ^ hi32(p)) < 0 || (ah | al) == 0;
  const uint32_t h = (central ? ch : ah) | (hi32(p) & 0x80000000u);
  return pair(zero ? 0u : h, zero ? 0u : (central ? cl : al));
}

}  // namespace gbh
