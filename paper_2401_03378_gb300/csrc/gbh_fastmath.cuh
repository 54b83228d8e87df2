// gbh_fastmath.cuh -- FP64 building blocks that keep work off the FP64 pipe.
//
// On GB300 the FP64 pipe retires 2 lanes per SM per clock while the integer
// and FP32 pipes retire 64-128; with everything in FP64 the stage kernel was bound
// by FP64 issue at an eighth of the SM's issue slots.  So:
//  * reciprocal and square root are computed on the integer pipes
//    (gbh_intmath.cuh), within 0.52 and 0.56 ulp.  They took 3 and 5 FP64
//    instructions of 64 issue cycles each; 29 of the 80 a face needs.  3-D step
//    of 256^3: 20.88 -> 16.71 ms, of 128^3: 3.105 -> 2.495 ms, 96-problem 2-D
//    ensemble 8.52 -> 6.88 ms.
//    All take positive (the reciprocal: also negative), normal, finite
//    inputs -- what the scheme feeds them.
//  * comparisons, min / max and sign tests of doubles are done on the bit
//    patterns with 64-bit integer operations (ALU pipe), which give the same
//    decisions as the IEEE comparisons for non-NaN values.
//  * in the stage kernel every FP64 add and multiply is an FMA whose three
//    operands are per-thread registers: a + b = fma(a, 1, b), a - b =
//    fma(-b, 1, a), a * b = fma(a, b, -0), the same results as the plain
//    operations (the product is exact inside the FMA, and x + (-0) = x for
//    every x, zeros included).  Measured on GB300 (gbh_fp64_probe): such an
//    FMA issues at 1.99 lanes per SM clock, while DADD, DMUL and an FMA with
//    a constant-bank, immediate or warp-uniform operand issue at 1.68.  The
//    constants (1, -0, the equation-of-state constants, dt/dx) get there
//    through reg_const: their bit patterns OR-ed with a run-time zero that
//    depends on the thread index, so the compiler can neither fold them into
//    constant operands nor keep them in uniform registers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gbh_internal.h"
#include "gbh_intmath.cuh"

namespace gbh {

__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ double bitsd(long long b) { return __longlong_as_double(b); }

__device__ __forceinline__ double add(double a, double b, const Rk& k) { return fma(a, k.one, b); }
__device__ __forceinline__ double sub(double a, double b, const Rk& k) { return fma(-b, k.one, a); }
__device__ __forceinline__ double mul(double a, double b, const Rk& k) { return fma(a, b, k.nz); }

// A run-time zero that depends on the thread index (p.opaque is 0).
__device__ __forceinline__ long long thread_zero(const Eos& p) { return p.opaque & (long long)threadIdx.x; }

// x in a per-thread register (z = thread_zero(...)).
__device__ __forceinline__ double reg_const(double x, long long z) { return bitsd(dbits(x) | z); }

// The constants of e in per-thread registers.
__device__ __forceinline__ Eos reg_eos(const Eos& p, long long z) {
  Eos e = p;
  e.gamma = reg_const(p.gamma, z);
  e.gm1 = reg_const(p.gm1, z);
  e.g_gm1 = reg_const(p.g_gm1, z);
  e.hgm1 = reg_const(p.hgm1, z);
  e.k.one = reg_const(p.k.one, z);
  e.k.nz = reg_const(p.k.nz, z);
  return e;
}

// Magnitudes and signs of doubles on the integer pipe.  The magnitude key is
// the bit pattern shifted left by one (the sign bit drops out): magnitudes of
// doubles order like these unsigned integers.  Masking the sign bit off with
// an AND would say the same, but the compiler turns that pattern into an FP64
// absolute-value operation (a DADD on the FP64 pipe, the resource this kernel
// is bound by), and it does not do so for the shift.
__device__ __forceinline__ unsigned long long mag_key(double x) { return (unsigned long long)dbits(x) << 1; }
__device__ __forceinline__ unsigned long long sign_bit(double x) {
  return ((unsigned long long)dbits(x) >> 63) << 63;
}

// x / 2 for any finite x on the integer pipe: one off the exponent field when
// |x| >= 2^-1021, else the magnitude bits shifted right (exact except that
// the last bit of a subnormal result is truncated)
__device__ __forceinline__ double half_any(double x) {
  const unsigned long long m2 = mag_key(x);
  return bitsd(m2 >= (4ULL << 52) ? dbits(x) - (1LL << 52) : (long long)(sign_bit(x) | (m2 >> 2)));
}

// x / 4 for any finite x on the integer pipe: two off the exponent field when
// |x| >= 2^-1020, else the magnitude bits shifted right by two (which moves
// the result by less than 2^-1022)
__device__ __forceinline__ double quarter_any(double x) {
  const unsigned long long m2 = mag_key(x);
  return bitsd(m2 >= (6ULL << 52) ? dbits(x) - (2LL << 52) : (long long)(sign_bit(x) | (m2 >> 3)));
}

// The unpacked magnitude of x, and x from a bit pattern held as two words.
__device__ __forceinline__ Wide wide_of(double x) {
  return wide_unpack((uint32_t)((unsigned long long)dbits(x) >> 32), (uint32_t)dbits(x));
}

// 1/x on the integer pipes (gbh_intmath.cuh), within 0.52 ulp: no FP64
// operation (3 before).  NaN for zeros, subnormals, infinities, NaN and |x| >= 2^1022.
__device__ __forceinline__ double rcp_nr(double x) {
  const Wide a = wide_of(x);
  const long long r = (long long)(wide_pack(wide_rcp(a)) | sign_bit(x));
  return bitsd((unsigned)(a.e - 1) < 2044u ? r : 0x7ff8000000000000LL);
}
__device__ __forceinline__ double rcp_nr(double x, const Rk&) { return rcp_nr(x); }

// sqrt(x) on the integer pipes (gbh_intmath.cuh), within 0.56 ulp: no FP64
// operation (5 before).  NaN for zeros, subnormals, negative values, infinities and NaN.
__device__ __forceinline__ double sqrt_nr(double x) {
  const Wide a = wide_of(x);
  const unsigned field = (unsigned)((unsigned long long)dbits(x) >> 52);   // sign and exponent
  return bitsd(field - 1u < 2046u ? (long long)wide_pack(wide_sqrt(a)) : 0x7ff8000000000000LL);
}
__device__ __forceinline__ double sqrt_nr(double x, const Rk&) { return sqrt_nr(x); }

// 1/sqrt(x) as the rounded root's reciprocal, the form the adjoint's 1/c takes.
__device__ __forceinline__ double rsqrt_nr(double x) { return rcp_nr(sqrt_nr(x)); }

// ---- integer-domain comparisons -------------------------------------------

// Key whose signed-integer order is the numeric order of non-NaN doubles
// (negative values have their magnitude bits flipped).
__device__ __forceinline__ long long order_key(double x) {
  const long long b = dbits(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}

__device__ __forceinline__ double min_d(double a, double b) { return order_key(b) < order_key(a) ? b : a; }
__device__ __forceinline__ double max_d(double a, double b) { return order_key(a) < order_key(b) ? b : a; }
__device__ __forceinline__ bool less_d(double a, double b) { return order_key(a) < order_key(b) && ((dbits(a) | dbits(b)) << 1) != 0; }

// x >= 0 (true for +0 and -0), x < 0, x > 0.  (-0 is tested by its exact bit
// pattern: a test of the bits below the sign against zero is turned into an
// FP64 compare by the compiler.)
__device__ __forceinline__ bool ge0(double x) {
  const long long b = dbits(x);
  return b >= 0 || b == (long long)0x8000000000000000ULL;
}
__device__ __forceinline__ bool lt0(double x) { return !ge0(x); }
__device__ __forceinline__ bool gt0(double x) { return dbits(x) > 0; }

__device__ __forceinline__ double sel(bool c, double a, double b) { return c ? a : b; }

}  // namespace gbh
