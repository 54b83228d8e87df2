// gbh_device.cuh -- per-cell and per-face FP64 arithmetic of the stage kernel.
//
// The intra-stage calculations of the paper's hydrodynamics variants
// (Sec. 4.2, Alg. "Intra stage calculations for Spark") are calcLims
// (reconstruction), calcFlux (face fluxes), updSoln (flux-difference update)
// and calcEos (equation of state).  The numerics they leave open are read as:
// ideal-gas EOS with floors, MC-limited piecewise-linear reconstruction of
// primitive variables, and the HLLC flux (Toro's star state, Einfeldt /
// Roe-average wave-speed bounds).
//
// The formulas are arranged to keep work off the FP64 pipe, whose warp
// instruction takes 64 cycles of an SM sub-partition: products, quotients and
// roots of the equation of state and of the HLLC flux run on the integer pipes in
// unpacked form (gbh_intmath.cuh), the HLLC star state is reduced to two quotients,
// every comparison is done on bit patterns (gbh_fastmath.cuh), and what stays FP64
// are sums and differences of numbers of either sign.  Results agree with the plain
// formulas to rounding.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gbh_fastmath.cuh"
#include "gbh_internal.h"

namespace gbh {

// The bit pattern of x by its two words (the compiler does not look through
// the intrinsics, so masked sign bits do not become FP64 operations).
__device__ __forceinline__ uint64_t word_pair(double x) {
  return imath::pair((uint32_t)__double2hiint(x), (uint32_t)__double2loint(x));
}

// Wide -> double, for a result in the normal range.
__device__ __forceinline__ double wide_double(const Wide& a) { return bitsd((long long)wide_pack(a)); }

__device__ __forceinline__ uint32_t hi_word(double x) { return (uint32_t)((unsigned long long)dbits(x) >> 32); }

// The unpacked magnitude of x, with zeros (and subnormals) as numbers so small
// that no product of the scheme brings them back into the range of a double.
__device__ __forceinline__ Wide wide_of0(double x) {
  Wide a = wide_of(x);
  a.e = a.e == 0 ? -8192 : a.e;
  return a;
}

// Wide -> double with the bits of `top` (a sign bit; a NaN's exponent and
// quiet bits) OR-ed in: below the normal range a zero, above it an infinity.
__device__ __forceinline__ double wide_signed(const Wide& a, uint32_t top) {
  const uint64_t m = wide_pack(a);
  const bool in = (unsigned)(a.e - 1) < 2046u;
  const uint32_t out = a.e > 0 ? 0x7ff00000u : 0u;
  return bitsd((long long)imath::pair((in ? imath::hi32(m) : out) | top, in ? imath::lo32(m) : 0u));
}

// The unpacked magnitude of a sum of squares, with an infinity as a number so
// large that no product of the scheme brings it back into the range of a double.
__device__ __forceinline__ Wide wide_of_squares(double x) {
  Wide a = wide_of(x);
  a.e = a.e == 2047 ? 8192 : a.e;
  return a;
}

// 0 or 1: the sign of x (as a number, not a masked word: the compiler turns an
// XOR of masked sign bits into an FP64 negation).
__device__ __forceinline__ uint32_t sign01(double x) { return hi_word(x) >> 31; }

// Infinity or NaN.
__device__ __forceinline__ bool not_finite(double x) { return (hi_word(x) & 0x7ff00000u) == 0x7ff00000u; }

// z + 0 where x is finite and below 2^1017 in magnitude, else NaN: FP32 arithmetic on
// the high word, whose exponent field is all ones from there.  One instruction of
// the otherwise idle FP32 pipe; callers look closer where the sum is not +0.
__device__ __forceinline__ float watch(double x, float z) { return fmaf(__uint_as_float(hi_word(x)), 0.0f, z); }

// A NaN's high word where a face has no flux, else 0.  Not finite: a density or
// pressure, the squared velocity jump (which a velocity that is not makes so) or the
// contact speed's numerator; the unpacked form would take them as numbers.  Zero: the
// contact speed's denominator m = |m_L| + |m_R|, where both sound speeds are lost in
// the velocities they are added to (a sum of two products with a zero has an exponent
// below -5000, any other one above -600).  Without a branch, which would keep the two
// halves of the face from being scheduled together (1.2% of a step).
__device__ __forceinline__ uint32_t no_flux_mask(const double WL[5], const double WR[5], double du2, double num,
                                                 const Wide& m) {
  auto larger = [](uint32_t a, uint32_t b) { return a > b ? a : b; };
  const uint32_t rho = larger(hi_word(WL[0]), hi_word(WR[0])), p = larger(hi_word(WL[4]), hi_word(WR[4]));
  const uint32_t top = larger(larger(rho, p), larger(hi_word(du2), hi_word(num) & 0x7fffffffu));
  return top >= 0x7ff00000u || m.e <= -4096 ? 0x7fffffffu : 0u;
}

// calcEos role: conserved (rho, mx, my, mz, E) -> primitive (rho, u, v, w, p),
// p = (gamma-1) (E - (mx^2 + my^2 + mz^2) / (2 rho)).  Floors rho at small_rho and
// p at small_p (floored_rho, floored_p) and leaves 1/rho in ir.  On the integer pipes but
// for the subtraction: 8 FP64 instructions of 64 cycles became 1 and about 200
// more integer ones.  A conserved variable that is not finite, or beyond 2^1017, makes u,
// v and w NaN, and p NaN or the floor (through the FP32 watch: exact tests took 0.5% of a
// step); prim_beyond gives what the plain formulas do there.
__device__ __forceinline__ void cons_to_prim_flags(const double U[5], double W[5], const Eos& e, Wide& ir,
                                                   bool& floored_rho, bool& floored_p) {
  float z = 0.0f;
#pragma unroll
  for (int v = 0; v < 5; ++v) z = watch(U[v], z);
  const uint32_t bad = __float_as_uint(z);
  double rho = U[0];
  floored_rho = less_d(rho, e.small_rho);
  if (floored_rho) rho = e.small_rho;
  ir = wide_rcp(wide_of(rho));
  const Wide mx = wide_of0(U[1]), my = wide_of0(U[2]), mz = wide_of0(U[3]);
  const double u = wide_signed(wide_mul(mx, ir), sign01(U[1]) << 31 | bad);
  const double v = wide_signed(wide_mul(my, ir), sign01(U[2]) << 31 | bad);
  const double w = wide_signed(wide_mul(mz, ir), sign01(U[3]) << 31 | bad);
  const Wide m2 = wide_mul(wide_add(wide_add(wide_mul(mx, mx), wide_mul(my, my)), wide_mul(mz, mz)), ir);
  const double ein = sub(U[4], wide_signed(Wide{m2.h, m2.l, m2.e - 1}, 0u), e.k);
  double p = wide_signed(wide_mul(e.wgm1, wide_of0(ein)), sign01(ein) << 31 | bad);
  floored_p = less_d(p, e.small_p);
  if (floored_p) p = e.small_p;
  W[0] = rho; W[1] = u; W[2] = v; W[3] = w; W[4] = p;
}

// W of cons_to_prim_flags where a velocity is not finite, by the plain FP64 formulas:
// an infinite momentum is an infinite velocity at the pressure floor, and numbers beyond
// 2^1017 are numbers.  For the CFL speed of given states (dt = 0 beside an infinite
// momentum).
__device__ __forceinline__ void prim_beyond(const double U[5], double W[5], const Wide& ir, const Eos& e) {
  if (!not_finite(W[1]) && !not_finite(W[2]) && !not_finite(W[3])) return;
  const double r = not_finite(W[0]) ? bitsd(0x7ff8000000000000LL) : wide_signed(ir, 0u);
#pragma unroll
  for (int v = 1; v < 4; ++v) W[v] = mul(U[v], r, e.k);
  const double m2 = fma(U[3], W[3], fma(U[2], W[2], mul(U[1], W[1], e.k)));
  const double p = mul(e.gm1, fma(-0.5, m2, U[4]), e.k);
  const bool nan = mag_key(p) > mag_key(bitsd(0x7ff0000000000000LL));
  W[4] = nan ? bitsd(0x7ff8000000000000LL) : less_d(p, e.small_p) ? e.small_p : p;
}

// The same; returns 1 when a floor applied.
__device__ __forceinline__ int cons_to_prim_ir(const double U[5], double W[5], const Eos& e, Wide& ir) {
  bool fr, fp;
  cons_to_prim_flags(U, W, e, ir, fr, fp);
  return fr || fp ? 1 : 0;
}

__device__ __forceinline__ int cons_to_prim(const double U[5], double W[5], const Eos& e) {
  Wide ir;
  return cons_to_prim_ir(U, W, e, ir);
}

// calcLims role: half of the MC-limited slope at q0,
//   sigma/2 = sign(dp) * min(|dm+dp|/4, |dm|, |dp|) if dm, dp have the same strict sign, else 0,
// so that the face values are q0 -/+ sigma/2.  Sign test and minimum on bit
// patterns.
__device__ __forceinline__ double mc_half_slope(double qm, double q0, double qp) {
  const double dm = q0 - qm;
  const double dp = qp - q0;
  const double s4 = 0.25 * (dm + dp);
  const unsigned long long am = mag_key(dm), ap = mag_key(dp), as = mag_key(s4);
  unsigned long long m = am < ap ? am : ap;
  m = as < m ? as : m;
  const bool same = ((dbits(dm) ^ dbits(dp)) >= 0) && am != 0 && ap != 0;
  return bitsd(same ? (long long)((m >> 1) | sign_bit(dp)) : 0LL);
}

// Half the MC-limited slope from the differences dm = q0 - qm, dp = qp - q0:
//   sigma/2 = sign(dp) * min(|dm+dp|, 4|dm|, 4|dp|) / 4
// if dm, dp have the same strict sign, else 0, so the face values are
// q0 -/+ sigma/2.  On the integer pipes (gbh_intmath.cuh), the bits of the FP64
// form: the sum there took 64 cycles of the FP64 pipe, here about 24 more integer
// instructions (256^3 step 12.05 -> 11.72 ms, 96-problem ensemble 5.29 -> 4.98 ms; the
// face values' two sums cost more as integer work than they free: 13.05 ms).
__device__ __forceinline__ double mc_half_slope_d(double dm, double dp, const Rk&) {
  return bitsd((long long)half_slope(word_pair(dm), word_pair(dp)));
}

// max(a, b) of non-negative doubles on the integer pipe (their bit patterns
// order like their values; fmax is an FP64-pipe instruction).  A NaN operand
// is passed over, as fmax passes it over.
__device__ __forceinline__ double max_nonneg(double a, double b) {
  constexpr unsigned long long kInf = 0x7ff0000000000000ULL;
  unsigned long long x = (unsigned long long)dbits(a), y = (unsigned long long)dbits(b);
  x = x > kInf ? 0ULL : x;
  y = y > kInf ? 0ULL : y;
  return bitsd((long long)(x > y ? x : y));
}

// Maximum over the NT threads of a CTA (whole warps, at most 32, or a power of two
// below 32) of non-negative values: xor shuffles within each warp (over the lanes the
// CTA has), then the warps' maxima through s_warp[NT/32] and one more warp of shuffles.  The
// result is valid in thread 0; every thread of the CTA must call it.
template <int NT>
__device__ __forceinline__ double block_max(double v, double* s_warp) {
  static_assert(NT < 32 ? (NT & (NT - 1)) == 0 : NT % 32 == 0 && NT <= 1024);
  constexpr int WL = NT < 32 ? NT : 32;
  constexpr unsigned mask = WL == 32 ? 0xffffffffu : ((1u << WL) - 1u);
#pragma unroll
  for (int o = WL / 2; o > 0; o >>= 1) v = max_nonneg(v, __shfl_xor_sync(mask, v, o));
  if constexpr (NT > 32) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) s_warp[warp] = v;
    __syncthreads();
    if (warp == 0) {
      v = lane < NW ? s_warp[lane] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v = max_nonneg(v, __shfl_xor_sync(0xffffffffu, v, o));
    }
  }
  return v;
}

// The sum of the inverse cell widths that signal_speed_ir takes, in its order.
__device__ __forceinline__ double inv_width_sum(const Eos& e, double idx, double idy, double idz, bool dim3) {
  return dim3 ? add(add(idx, idy, e.k), idz, e.k) : add(idx, idy, e.k);
}

// Signal-speed sum of one cell for the CFL rule,
// sum_d (|u_d| + c) / dx_d = c (1/dx + 1/dy [+ 1/dz]) + |u| / dx + |v| / dy [+ |w| / dz];
// W and ir = 1 / W[0] from cons_to_prim_ir, isum = inv_width_sum(...).
__device__ __forceinline__ double signal_speed_ir(const double W[5], const Wide& ir, const Eos& e, double idx,
                                                  double idy, double idz, double isum, bool dim3) {
  const Wide c = wide_sqrt(wide_mul(wide_mul(e.wgamma, wide_of(W[4])), ir));
  const double c_d = not_finite(W[4]) ? W[4] : wide_double(c);
  double s = fma(fabs(W[1]), idx, mul(c_d, isum, e.k));
  s = fma(fabs(W[2]), idy, s);
  if (dim3) s = fma(fabs(W[3]), idz, s);
  return s;
}

// calcFlux role: HLLC flux through a face whose normal is the first velocity
// component of the rotated states WL (low side) and WR (high side):
// W = (rho, u_n, u_t1, u_t2, p).  F is returned in the same rotated order.
//
// Wave speeds: S_L = min(u_L - c_L, u~ - c~), S_R = max(u_R + c_R, u~ + c~)
// with Roe averages (sqrt(rho) weights); contact speed
// S* = (p_R - p_L + m_L u_L - m_R u_R) / (m_L - m_R), m_K = rho_K (S_K - u_K).
// Side K = L when S* >= 0, else R.  With delta = (S* - u_K) / (S_K - S*),
// Toro's star state satisfies
//   U*_K - U_K = delta [rho_K, rho_K S_K, rho_K v_K, rho_K w_K, h_K + m_K S*]
// (h = E + p), so F = F_K + S_K (U*_K - U_K) becomes, with g = S_K delta and
// t = u_K + g,
//   F0 = rho_K t,  F1 = F0 u_K + p_K + g m_K,  F2 = v_K F0,  F3 = w_K F0,
//   F4 = h_K t + g m_K S*.
// When the whole fan lies on one side (S_L >= 0, or S_R <= 0) g = 0 and
// F = F_K; otherwise t = u_K + g = S* (S_K - u_K) / (S_K - S*).
//
// The Roe averages are evaluated in an algebraically equal form: with
// s = sqrt(rho_L rho_R) the weights are w_L = s / (s + rho_R) and
// w_R = rho_R / (s + rho_R); and, because H_K = c_K^2 / (gamma-1) + |u_K|^2 / 2 and
// w_L + w_R = 1,
//   c~^2 = (gamma-1) (H~ - |u~|^2 / 2) = w_L c_L^2 + w_R c_R^2
//          + (gamma-1)/2 w_L w_R |u_L - u_R|^2
//        = w_L c_L^2 + w_R (c_R^2 + (gamma-1)/2 w_L |u_L - u_R|^2),
// a sum of non-negative terms (no cancellation at high Mach number), so the
// transverse Roe velocities and H~ are not formed.  h_K is formed for the
// chosen side only, and u~ = u_L - w_R (u_L - u_R).
//
// From the densities and pressures to c_L, c_R, w_R and c~ everything is
// positive, so this part is a chain of Wide numbers on the integer pipes
// (gbh_intmath.cuh): 12 products, 3 sums, 2 reciprocals and 4 roots in about
// 350 integer instructions where the FP64 pipe had 16 instructions beside the
// roots' and reciprocals' own (64 issue cycles each, against 1 to 2).  The
// chain carries 57 bits and rounds only its four results.  80 -> 37 FP64
// instructions a face with the remaining roots and reciprocals; of that the
// chain: 256^3 step 16.71 -> 14.07 ms, 96-problem 2-D ensemble 6.88 -> 5.71 ms.
// The quotients S* and t, whose factors are already unpacked, follow the same
// way (m_L - m_R is a sum of two negative numbers), as do m_K, h_K, rho_K t and
// g m_K: 26 FP64 instructions a face are left (256^3 step 14.07 -> 12.33 ms).  The
// sums of squares and the products with v_K and w_K stay on the FP64 pipe: a
// face takes about 960 integer instructions (gbh_op_count_probe), and with these
// seven in integer form too (19 FP64, about 100 more) the integer pipes were the
// longer ones inside the face passes (96-problem ensemble 4.89 -> 4.73 ms, 256^3
// 11.74 -> 11.62 ms).  Results that can leave the range of a double go through
// wide_signed, and no_flux_mask says where there is no flux: 0.7% of a step.
__device__ __forceinline__ void hllc_flux(const double WL[5], const double WR[5], const Eos& e,
                                          double F[5]) {
  const Rk& k = e.k;
  const double rL = WL[0], uL = WL[1], vL = WL[2], wL = WL[3], pL = WL[4];
  const double rR = WR[0], uR = WR[1], vR = WR[2], wR = WR[3], pR = WR[4];

  // the wave speeds' positive part, on the integer pipes
  const Wide RL = wide_of(rL), RR = wide_of(rR);
  const Wide P = wide_mul(RL, RR);
  const Wide g_P = wide_mul(e.wgamma, wide_rcp(P));        // gamma / (rho_L rho_R)
  const Wide cL2 = wide_mul(wide_of(pL), wide_mul(RR, g_P)), cR2 = wide_mul(wide_of(pR), wide_mul(RL, g_P));
  const double cL = wide_double(wide_sqrt(cL2)), cR = wide_double(wide_sqrt(cR2));
  const Wide sP = wide_sqrt(P);
  const Wide D = wide_rcp_low(wide_add(sP, RR));
  const Wide wl = wide_mul(sP, D), wr = wide_mul(RR, D);   // Roe weights

  const double du = sub(uL, uR, k), dv = sub(vL, vR, k), dw = sub(wL, wR, k);
  const double ut = fma(-wide_double(wr), du, uL);         // w_L u_L + w_R u_R
  const double du2_d = fma(dw, dw, fma(dv, dv, mul(du, du, k)));
  const Wide du2 = wide_of(du2_d);
  const Wide ct2 = wide_add(wide_mul(wl, cL2),
                            wide_mul(wr, wide_add(cR2, wide_mul(wide_mul(e.whgm1, wl), du2))));
  const double ct = wide_double(wide_sqrt(ct2));

  const double SL = min_d(sub(uL, cL, k), sub(ut, ct, k));
  const double SR = max_d(add(uR, cR, k), add(ut, ct, k));
  const double dL = sub(SL, uL, k), dR = sub(SR, uR, k);   // <= 0 and >= 0
  const Wide DL = wide_of0(dL), DR = wide_of0(dR);
  const Wide ML = wide_mul(RL, DL), MR = wide_mul(RR, DR); // |m_L|, |m_R|
  const double mL = wide_signed(ML, 0x80000000u), mR = wide_signed(MR, 0u);
  // S* = num / (m_L - m_R) = -num / (|m_L| + |m_R|)
  const double num = fma(-mR, uR, fma(mL, uL, sub(pR, pL, k)));
  const Wide MS = wide_add(ML, MR);
  const uint32_t bad = no_flux_mask(WL, WR, du2_d, num, MS);   // OR-ed into S* and t, from where it reaches every flux
  const Wide WS = wide_mul(wide_of0(num), wide_rcp(MS));
  const uint32_t ssgn = sign01(num) ^ 1u;
  const double Ss = wide_signed(WS, ssgn << 31 | bad);

  const bool left = ge0(Ss);
  const double rK = sel(left, rL, rR), uK = sel(left, uL, uR), vK = sel(left, vL, vR);
  const double wK = sel(left, wL, wR), pK = sel(left, pL, pR);
  const double SK = sel(left, SL, SR);
  const bool fan = left ? lt0(SL) : gt0(SR);

  // t = u_K + g; S_K - S* != 0 inside the fan, and t = u_K (g = 0) outside it
  const double SKs = sub(SK, Ss, k);
  const Wide WT = wide_mul(wide_mul(WS, left ? DL : DR), wide_rcp(wide_of(SKs)));
  const Wide T = fan ? WT : wide_of0(uK);
  const uint32_t tsgn = fan ? ssgn ^ sign01(SKs) ^ (left ? 1u : 0u) : sign01(uK);
  const double t = wide_signed(T, tsgn << 31 | bad);
  const double g = sub(t, uK, k);
  const Wide RK = wide_of(rK);
  // E + p of the chosen side
  const Wide kin = wide_mul(RK, wide_of_squares(fma(wK, wK, fma(vK, vK, mul(uK, uK, k)))));
  const double hK = wide_signed(wide_add(Wide{kin.h, kin.l, kin.e - 1}, wide_mul(e.wg_gm1, wide_of(pK))), 0u);
  const Wide F0 = wide_mul(RK, T);
  const Wide GM = wide_mul(wide_of0(g), left ? ML : MR);   // |g m_K|
  const uint32_t gmsgn = sign01(g) ^ (left ? 1u : 0u);
  F[0] = wide_signed(F0, tsgn << 31 | bad);
  F[1] = add(fma(F[0], uK, pK), wide_signed(GM, gmsgn << 31), k);
  F[2] = mul(vK, F[0], k);
  F[3] = mul(wK, F[0], k);
  F[4] = fma(hK, t, wide_signed(wide_mul(GM, WS), (gmsgn ^ ssgn) << 31));
}

}  // namespace gbh
