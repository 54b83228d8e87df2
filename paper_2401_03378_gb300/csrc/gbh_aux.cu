// gbh_aux.cu -- guard-cell fill, CFL time-step reduction, state check and the
// FP64 throughput probe.
#include <cuda_runtime.h>
#include <stdint.h>

#include "gbh_check.cuh"
#include "gbh_device.cuh"
#include "gbh_internal.h"

namespace gbh {
namespace {

constexpr int kThreads = 256;

// q / d; FAST: by a multiplication with m = 2^32 / d + 1, exact for q < 2^32 / d
// (the launcher checks the range).
struct Divisor {
  unsigned d, m;
};
template <bool FAST>
__device__ __forceinline__ unsigned div_by(unsigned q, const Divisor& v) {
  return FAST ? __umulhi(q, v.m) : q / v.d;
}

// Cell (i, j, k) of a block's padded array.  In 32 bits where the divisions by
// multiplication are exact (FAST): such a block has far fewer than 2^31 padded cells.
template <bool FAST>
__device__ __forceinline__ long long padded_index(const Layout& L, int i, int j, int k) {
  return FAST ? (k * L.nyp + j) * L.nxp + i : ((long long)k * L.nyp + j) * L.nxp + i;
}

// The guard cells of a block, numbered: the z guard planes (all their cells),
// then in every interior plane the 2 g full rows and the 2 g x guards of each
// interior row.
struct FillMap {
  Divisor plane, row, ring, side;   // nyp nxp; nxp; guard cells of an interior plane; 2 g
  unsigned nzg, cells;              // cells of the z guard planes; all guard cells
  int parts;                        // CTAs per block
};

// fill_guardcells (Sec. 4.2).  A CTA takes one of `parts` shares of a block's
// guard cells.  The value of a guard cell is resolved directly, without passes
// that depend on one another:
//  1. for each dimension d in which the cell lies outside the block and the
//     block's face in that direction is an outflow edge, its coordinate is
//     clamped to the nearest interior index (outflow is applied in the order
//     x, then y, then z; clamps in different dimensions commute);
//  2. the remaining outside dimensions give a lattice offset; the cell is the
//     interior cell of the neighbour block at that offset (full table).
// Both steps depend only on which of the 27 (9) regions around the block the
// cell lies in, so the CTA resolves them once per region into shared memory: a
// shift from the guard cell to its source, with a coordinate clamped where the
// region's flags say so.  Every source is an interior cell, so the in-place fill
// has no read/write overlap.  An offset with no neighbour and no outflow face is
// left untouched.  512 blocks of 16^3 + 4 guards (199 MB written, 84 MB read, each
// about 2.4 times, through L2): 136 -> 76 us (83 with 8-byte accesses), bound by the L2 traffic of 32-byte x
// guards; resolving every cell with 64-bit divisions and table reads was the rest.
template <bool FAST, int X>
__global__ void __launch_bounds__(kThreads) fill_kernel(const FillArgs a, const FillMap m) {
  const Layout& L = a.lay;
  const bool d3 = L.ndim == 3;
  const int b = blockIdx.x / m.parts, part = blockIdx.x - b * m.parts;
  __shared__ long long s_shift[27];
  __shared__ int s_flags[27];               // bits 0-2: clamp x, y, z; bit 3: no source
  if (threadIdx.x < (d3 ? 27 : 9)) {
    const int e = threadIdx.x;
    int o[3] = {e % 3 - 1, e / 3 % 3 - 1, d3 ? e / 9 - 1 : 0};
    int flags = 0;
    for (int d = 0; d < L.ndim; ++d)
      if (o[d] != 0 && __ldg(a.face_nbr + 6 * b + 2 * d + (o[d] > 0 ? 1 : 0)) == GBH_BC_OUTFLOW) {
        flags |= 1 << d;
        o[d] = 0;
      }
    int src = b;
    if (o[0] != 0 || o[1] != 0 || o[2] != 0) {
      src = __ldg(a.nbr + (d3 ? 27 * b + (o[2] + 1) * 9 : 9 * b) + (o[1] + 1) * 3 + (o[0] + 1));
      if (src < 0) flags |= 8;
    }
    s_flags[e] = flags;
    s_shift[e] = (long long)src * L.bstride -
                 ((long long)(o[2] * L.nz * L.nyp + o[1] * L.ny) * L.nxp + o[0] * L.nx);
  }
  __syncthreads();
  const long long lim = (long long)L.nblocks * L.bstride - 4 * L.vstride;
  const unsigned full = 2u * L.g * L.nxp;
  for (unsigned t = part * kThreads + threadIdx.x; t < m.cells / X; t += m.parts * kThreads) {
    const unsigned q = X * t;
    int ii, jj, kk;
    if (q < m.nzg) {
      const unsigned p = div_by<FAST>(q, m.plane), r = q - p * m.plane.d;
      jj = (int)div_by<FAST>(r, m.row);
      ii = (int)r - jj * L.nxp;
      kk = (int)p < L.gz ? (int)p : (int)p + L.nz;
    } else {
      const unsigned q2 = q - m.nzg, p = div_by<FAST>(q2, m.ring), r = q2 - p * m.ring.d;
      kk = (int)p + L.gz;
      if (r < full) {
        const int row = (int)div_by<FAST>(r, m.row);
        jj = row < L.g ? row : L.ny + row;
        ii = (int)r - row * L.nxp;
      } else {
        const unsigned r2 = r - full;
        const int row = (int)div_by<FAST>(r2, m.side), t = (int)r2 - row * 2 * L.g;
        jj = L.g + row;
        ii = t < L.g ? t : L.nx + t;
      }
    }
    const int ox = ii < L.g ? 0 : ii >= L.g + L.nx ? 2 : 1, oy = jj < L.g ? 0 : jj >= L.g + L.ny ? 2 : 1;
    const int oz = kk < L.gz ? 0 : kk >= L.gz + L.nz ? 2 : 1;
    const int e = (d3 ? 9 * oz : 0) + 3 * oy + ox;
    const int flags = s_flags[e];
    if (flags & 8) continue;
    const int si = flags & 1 ? (ox ? L.g + L.nx - 1 : L.g) : ii;
    const int sj = flags & 2 ? (oy ? L.g + L.ny - 1 : L.g) : jj;
    const int sk = flags & 4 ? (oz ? L.gz + L.nz - 1 : L.gz) : kk;
    const long long so = GBH_IX(s_shift[e] + padded_index<FAST>(L, si, sj, sk), lim);
    const long long dof = GBH_IX((long long)b * L.bstride + padded_index<FAST>(L, ii, jj, kk), lim);
    if constexpr (X == 2) {
      double2 v[5];
      if (flags & 1) {
#pragma unroll
        for (int n = 0; n < 5; ++n) v[n].x = v[n].y = a.U[so + n * L.vstride];
      } else {
#pragma unroll
        for (int n = 0; n < 5; ++n) v[n] = *reinterpret_cast<const double2*>(a.U + so + n * L.vstride);
      }
#pragma unroll
      for (int n = 0; n < 5; ++n) *reinterpret_cast<double2*>(a.U + dof + n * L.vstride) = v[n];
    } else {
      double v[5];
#pragma unroll
      for (int n = 0; n < 5; ++n) v[n] = a.U[so + n * L.vstride];
#pragma unroll
      for (int n = 0; n < 5; ++n) a.U[dof + n * L.vstride] = v[n];
    }
  }
}

// CFL reduction: max over the interior cells of the signal-speed sum, into
// smax_acc, or with `problem` into the accumulator of the block's problem (one
// atomicMax per CTA and block on the bit pattern, which orders like the
// non-negative value).  A CTA takes one of `parts` shares of a block's cells; with
// parts = 0 the next kThreads cells of the list's blocks one after another (blocks
// of fewer cells; no `problem`).  nx = ny = 2^lg.  512 blocks of 16^3: 92 -> 55 us (the
// 64-bit divisions of a cell index and 17 of 22 FP64 instructions a cell are gone);
// 65536 blocks of 4^2: 39 us, 219 with a CTA to each block.
__global__ void __launch_bounds__(kThreads) dt_reduce_kernel(const DtArgs a, const int* problem, int parts, int lg) {
  const Layout& L = a.lay;
  const unsigned per = (unsigned)(L.nx * L.ny * L.nz);
  const bool d3 = L.ndim == 3;
  const long long zt = thread_zero(a.eos);
  const Eos e = reg_eos(a.eos, zt);   // FP64 constants in per-thread registers (gbh_fastmath.cuh)
  __shared__ double red[kThreads / 32];
  const int nb = a.block_list ? a.nlist : L.nblocks;
  const unsigned total = (unsigned)nb * per;          // with parts = 0 (below 2^32: the state would not fit)
  const int items = parts ? nb * parts : (int)((total + kThreads - 1) / kThreads);
  double smax = 0.0;
  for (int s = blockIdx.x; s < items; s += gridDim.x) {
    int slot, part = 0;
    unsigned cell = threadIdx.x;
    if (parts) {
      slot = s / parts;
      part = s - slot * parts;
    } else {
      const unsigned first = (unsigned)s * kThreads, lo = first / per, t = first - lo * per + threadIdx.x, sub = t / per;
      slot = (int)(lo + sub);
      cell = t - sub * per;
      if (slot >= nb) break;                           // no barrier in this form's loop
    }
    const int b = a.block_list ? __ldg(a.block_list + slot) : slot;
    const double ix = reg_const(__ldg(a.inv_dx + 3 * b), zt), iy = reg_const(__ldg(a.inv_dx + 3 * b + 1), zt);
    const double iz = reg_const(__ldg(a.inv_dx + 3 * b + 2), zt);
    const double isum = inv_width_sum(e, ix, iy, iz, d3);
    const double* src = a.U + GBH_IX((long long)b * L.bstride, (long long)L.nblocks * L.bstride);
    if (problem) smax = 0.0;
    for (unsigned t = part * kThreads + cell; t < per; t += (parts ? parts : 1) * kThreads) {
      const int i = t & (L.nx - 1), j = (t >> lg) & (L.nx - 1), k = t >> (2 * lg);
      const long long o = GBH_IX(((long long)(k + L.gz) * L.nyp + (j + L.g)) * L.nxp + (i + L.g), L.vstride);
      double U[5], W[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) U[v] = __ldg(src + o + v * L.vstride);
      Wide ir;
      cons_to_prim_ir(U, W, e, ir);
      prim_beyond(U, W, ir, e);
      smax = max_nonneg(smax, signal_speed_ir(W, ir, e, ix, iy, iz, isum, d3));
    }
    if (problem) {
      const double m = block_max<kThreads>(smax, red);
      if (threadIdx.x == 0) atomicMax(a.smax_acc + __ldg(problem + b), (unsigned long long)__double_as_longlong(m));
      __syncthreads();
    }
  }
  if (!problem) {
    const double m = block_max<kThreads>(smax, red);
    if (threadIdx.x == 0) atomicMax(a.smax_acc, (unsigned long long)__double_as_longlong(m));
  }
}

// dt = cfl / smax per problem; also records it and clears the accumulator for
// its next use.
__global__ void dt_finalize_kernel(unsigned long long* acc, double cfl, double* dt_out, double* hist, int n) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const double smax = __longlong_as_double((long long)acc[p]);
    const double dt = cfl / smax;
    dt_out[p] = dt;
    if (hist) hist[p] = dt;
    acc[p] = 0ull;
  }
}

__global__ void __launch_bounds__(kThreads) check_kernel(const double* U, const Layout L, const Eos e,
                                                         unsigned long long* count) {
  const long long per = (long long)L.nx * L.ny * L.nz;
  const long long total = per * L.nblocks;
  unsigned long long bad = 0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int b = (int)(t / per);
    long long r = t - (long long)b * per;
    const int i = (int)(r % L.nx);
    r /= L.nx;
    const int j = (int)(r % L.ny);
    const int k = (int)(r / L.ny);
    const long long o = GBH_IX((long long)b * L.bstride + ((long long)(k + L.gz) * L.nyp + (j + L.g)) * L.nxp + (i + L.g),
                               (long long)L.nblocks * L.bstride - 4 * L.vstride);
    double u[5];
    bool finite = true;
    for (int v = 0; v < 5; ++v) {
      u[v] = U[o + v * L.vstride];
      finite = finite && isfinite(u[v]);
    }
    const double p = e.gm1 * (u[4] - 0.5 * (u[1] * u[1] + u[2] * u[2] + u[3] * u[3]) / u[0]);
    if (!finite || !(u[0] > e.small_rho) || !(p > e.small_p)) ++bad;
  }
  if (bad) atomicAdd(count, bad);
}

// Interior cells between the padded and the interior-only layouts of the nb
// blocks that start at `padded` and `interior`: one thread per cell,
// consecutive threads along x, so both sides read and write whole rows of nx
// doubles (coalesced).  The launcher keeps 5 nx ny nz nb below 2^30, so the
// cell index and its decomposition are 32-bit.
__global__ void __launch_bounds__(kThreads) interior_copy_kernel(double* padded, double* interior, const Layout L,
                                                                 int nb, bool to_padded) {
  const unsigned per = (unsigned)(L.nx * L.ny * L.nz), cells = 5u * per, total = cells * (unsigned)nb;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const unsigned bl = t / cells;
    unsigned r = t - bl * cells;
    const unsigned v = r / per;
    r -= v * per;
    const unsigned i = r % (unsigned)L.nx;
    r /= (unsigned)L.nx;
    const unsigned j = r % (unsigned)L.ny, k = r / (unsigned)L.ny;
    const long long o = (long long)bl * L.bstride + (long long)v * L.vstride +
                        ((long long)(k + L.gz) * L.nyp + (j + L.g)) * L.nxp + (i + L.g);
    if (to_padded)
      padded[GBH_IX(o, (long long)nb * L.bstride)] = interior[GBH_IX(t, total)];
    else
      interior[GBH_IX(t, total)] = padded[GBH_IX(o, (long long)nb * L.bstride)];
  }
}

// 8 independent FMA chains per thread; the multiplier and addend keep the
// values bounded (fixed point 1.0).  Only the first `lanes` lanes of each
// warp run the chains (to measure how the FP64 pipe charges partial warps).
// FP64 pipe probe: 8 independent chains per thread, run by the first `lanes`
// lanes of each warp.  FORM 0: x = fma(x, m, c) with m, c compile-time
// constants (constant-bank operands); 1: the same with m, c in per-thread
// registers (their bit patterns OR-ed with a run-time zero that depends on the
// thread index, so the compiler can neither fold them into constants nor keep
// them in warp-uniform registers); 2: x = x + c (DADD); 3: x = x * m (DMUL),
// c and m in per-thread registers; 4: as 1 with m, c warp-uniform (OR-ed with
// the run-time zero alone).
template <int FORM>
__global__ void fp64_probe_kernel(int iters, int lanes, long long zero, double* out) {
  const long long z = FORM == 4 ? zero : (zero & (long long)threadIdx.x);
  const double m = FORM == 0 ? 0.999999999 : __longlong_as_double(__double_as_longlong(0.999999999) | z);
  const double c = FORM == 0 ? 1e-9 : __longlong_as_double(__double_as_longlong(1e-9) | z);
  double x[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) x[k] = 1.0 + 1e-3 * threadIdx.x + 0.1 * k;
  const int n = (int)(threadIdx.x & 31) < lanes ? iters : 0;
  for (int i = 0; i < n; ++i) {
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = FORM == 2 ? x[k] + c : FORM == 3 ? x[k] * m : fma(x[k], m, c);
  }
  double sum = 0.0;
#pragma unroll
  for (int k = 0; k < 8; ++k) sum += x[k];
  out[blockIdx.x * (long long)blockDim.x + threadIdx.x] = sum;
}

// FP64 instruction count of one call of each arithmetic building block of the
// stage kernel, in the form the kernel uses (register constants, register-FMA
// adds and multiplies).  Each thread makes `iters` dependent calls on the 10
// doubles io[10 t .. 10 t + 9]; the next call's inputs take the low bit of
// the XOR of every output of the last one into their last mantissa bits with
// an integer XOR, so no part of a call can be hoisted or folded and the chain
// adds no FP64 work: ncu's FP64 instruction counters of a launch divided by
// threads x iters are the instructions of one call.
template <int FN>
__global__ void op_count_kernel(int iters, const Eos e0, double* io) {
  const long long zt = thread_zero(e0);
  const Eos e = reg_eos(e0, zt);
  const Rk& rk = e.k;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  double x[10];
#pragma unroll
  for (int v = 0; v < 10; ++v) x[v] = io[10 * t + v];
  const double c1 = reg_const(0.3, zt), c2 = reg_const(0.2, zt), c3 = reg_const(0.1, zt);
  long long fb = 0;
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int v = 0; v < 10; ++v) x[v] = bitsd(dbits(x[v]) ^ (fb & 1));
    fb = 0;
    if constexpr (FN == 0) {          // cons -> prim of one cell
      double W[5];
      fb ^= cons_to_prim(x, W, e);
#pragma unroll
      for (int v = 0; v < 5; ++v) fb ^= dbits(W[v]);
    } else if constexpr (FN == 1) {   // one x/y slope work item (three cells) of one variable
      const double d0 = sub(x[1], x[0], rk), d1 = sub(x[2], x[1], rk), d2 = sub(x[3], x[2], rk);
      const double d3 = sub(x[4], x[3], rk);
      const double t0 = mc_half_slope_d(d0, d1, rk), t1 = mc_half_slope_d(d1, d2, rk);
      const double t2 = mc_half_slope_d(d2, d3, rk);
      const double q[6] = {sub(x[1], t0, rk), add(x[1], t0, rk), sub(x[2], t1, rk), add(x[2], t1, rk),
                           sub(x[3], t2, rk), add(x[3], t2, rk)};
#pragma unroll
      for (int v = 0; v < 6; ++v) fb ^= dbits(q[v]);
    } else if constexpr (FN == 2) {   // one HLLC face
      double F[5];
      hllc_flux(x, x + 5, e, F);
#pragma unroll
      for (int v = 0; v < 5; ++v) fb ^= dbits(F[v]);
    } else if constexpr (FN == 3) {   // the 3-D flux-difference update of one variable
      double r = fma(-c1, sub(x[1], x[2], rk), x[0]);
      r = fma(-c2, sub(x[3], x[4], rk), r);
      r = fma(-c3, sub(x[5], x[6], rk), r);
      fb ^= dbits(r);
    } else if constexpr (FN == 4) {   // the second-stage combine of one variable
      fb ^= dbits(half_any(add(x[1], x[0], rk)));
    } else if constexpr (FN == 5) {   // CFL epilogue of one cell: cons -> prim and 3-D signal speed
      double W[5];
      Wide ir;
      cons_to_prim_ir(x, W, e, ir);
      fb ^= dbits(signal_speed_ir(W, ir, e, c1, c2, c3, c1, true));
    } else if constexpr (FN == 6) {   // z march: the next z slope and face states of one variable
      const double dn = sub(x[1], x[0], rk);
      const double tz = mc_half_slope_d(x[2], dn, rk);
      fb ^= dbits(sub(x[0], tz, rk)) ^ dbits(add(x[0], tz, rk)) ^ dbits(dn);
    } else {                           // the two face states of a block-boundary face, one variable
      const double d0 = sub(x[1], x[0], rk), d1 = sub(x[2], x[1], rk), d2 = sub(x[3], x[2], rk);
      fb ^= dbits(add(x[1], mc_half_slope_d(d0, d1, rk), rk)) ^ dbits(sub(x[2], mc_half_slope_d(d1, d2, rk), rk));
    }
  }
#pragma unroll
  for (int v = 0; v < 10; ++v) io[10 * t + v] = bitsd(dbits(x[v]) ^ (fb & 1));
}

// Self-test of the refined reciprocal / square roots: out[6][n] =
// rcp_nr, 1.0/x, rsqrt_nr, 1.0/sqrt(x), sqrt_nr, sqrt(x).
__global__ void fastmath_selftest_kernel(const double* x, double* out, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double v = x[i];
    out[i] = rcp_nr(v);
    out[n + i] = 1.0 / v;
    out[2 * n + i] = rsqrt_nr(v);
    out[3 * n + i] = 1.0 / sqrt(v);
    out[4 * n + i] = sqrt_nr(v);
    out[5 * n + i] = sqrt(v);
  }
}

// Self-test of the integer-pipe helpers the stage kernel relies on:
// out[6][n] = half_any(x), quarter_any(x), mc_half_slope_d(x, y) with the
// constants in per-thread registers, ge0(x) (1 or 0), min_d(x, y), max_d(x, y).
__global__ void bits_selftest_kernel(const double* x, const double* y, double* out, long long n, long long zero) {
  const long long z = zero & (long long)threadIdx.x;
  const Rk k{reg_const(1.0, z), reg_const(-0.0, z)};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double a = x[i], b = y[i];
    out[i] = half_any(a);
    out[n + i] = quarter_any(a);
    out[2 * n + i] = mc_half_slope_d(a, b, k);
    out[3 * n + i] = ge0(a) ? 1.0 : 0.0;
    out[4 * n + i] = min_d(a, b);
    out[5 * n + i] = max_d(a, b);
  }
}

#ifdef GBH_CHECK
// One index past a 4-element buffer: the check counts it and redirects the
// store to element 0 (the access stays inside the buffer).
__global__ void check_selftest_kernel(double* buf) {
  const long long i = 4;
  buf[GBH_IX(i, 4)] = 1.0;
}
#endif

int grid_for(long long work, int threads) {
  long long g = (work + threads - 1) / threads;
  if (g > 152LL * 16) g = 152LL * 16;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

GBH_CHECK_TAKE(check_take_aux)

long long check_selftest() {
#ifdef GBH_CHECK
  double* buf = nullptr;
  if (cudaMalloc(&buf, 4 * sizeof(double)) != cudaSuccess) return -1;
  const long long before = check_take_aux();
  check_selftest_kernel<<<1, 1>>>(buf);
  const cudaError_t e = cudaDeviceSynchronize();
  cudaFree(buf);
  if (e != cudaSuccess || before < 0) return -1;
  return check_take_aux();
#else
  return -1;
#endif
}

cudaError_t launch_fill(const FillArgs& a, cudaStream_t s) {
  const Layout& L = a.lay;
  auto div = [](unsigned d) { return Divisor{d, (unsigned)((1ull << 32) / d + 1)}; };
  const unsigned ring = (unsigned)(2 * L.g * L.nxp + L.ny * 2 * L.g);
  const unsigned long long nzg = 2ull * L.gz * L.nyp * L.nxp, cells = nzg + (unsigned long long)L.nz * ring;
  // multiply-high quotients: exact while the dividend times the divisor stays
  // below 2^32 (all but blocks of very many planes)
  const bool fast = cells * (unsigned long long)(L.nyp * L.nxp) < (1ull << 32);
  // two cells a thread (16-byte accesses) where every run of guard cells starts on
  // an even cell of a 16-byte aligned state: nx is even, so an even g does
  const bool pairs = fast && L.g % 2 == 0 && ((uintptr_t)a.U & 15u) == 0;
  const long long want = (152LL * 16 + L.nblocks - 1) / L.nblocks;
  const long long most = (long long)(cells / (pairs ? 2 : 1) + kThreads - 1) / kThreads;
  const int parts = (int)(want < 1 ? 1 : want < most ? want : most);
  const FillMap m{div((unsigned)(L.nyp * L.nxp)), div((unsigned)L.nxp), div(ring), div(2u * L.g),
                  (unsigned)nzg, (unsigned)cells, parts};
  const unsigned grid = (unsigned)(L.nblocks * parts);
  if (!fast)
    fill_kernel<false, 1><<<grid, kThreads, 0, s>>>(a, m);
  else if (pairs)
    fill_kernel<true, 2><<<grid, kThreads, 0, s>>>(a, m);
  else
    fill_kernel<true, 1><<<grid, kThreads, 0, s>>>(a, m);
  return cudaGetLastError();
}

cudaError_t launch_interior_copy(double* padded, double* interior, const Layout& L, int b0, int nb,
                                 bool to_padded, cudaStream_t s) {
  const long long cells = 5LL * L.nx * L.ny * L.nz;
  const long long per_launch = (1LL << 30) / cells > 0 ? (1LL << 30) / cells : 1;
  for (long long b = b0; b < (long long)b0 + nb; b += per_launch) {
    const int n = (int)((long long)b0 + nb - b < per_launch ? (long long)b0 + nb - b : per_launch);
    interior_copy_kernel<<<grid_for(cells * n, kThreads), kThreads, 0, s>>>(padded + b * L.bstride,
                                                                           interior + b * cells, L, n, to_padded);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_dt_reduce(const DtArgs& a, const int* problem, cudaStream_t s) {
  const Layout& L = a.lay;
  const long long nb = a.block_list ? a.nlist : L.nblocks, per = (long long)L.nx * L.ny * L.nz;
  const int lg = L.nx == 16 ? 4 : L.nx == 8 ? 3 : 2;
  // shares of a block: a power of two (whole rounds of threads), enough CTAs for the
  // chip's dispatch to even out
  const long long most = (per + kThreads - 1) / kThreads;
  int parts = 1;
  while (parts < most && nb * parts < 152LL * 16) parts *= 2;
  // blocks smaller than a CTA one after another, where they have no problems of
  // their own: a CTA with a block of 4^2 to itself has 16 of 256 threads at work
  if (!problem && per < kThreads) parts = 0;
  const long long items = parts ? nb * parts : (nb * per + kThreads - 1) / kThreads, cap = 152LL * 64;
  dt_reduce_kernel<<<(int)(items < cap ? items : cap), kThreads, 0, s>>>(a, problem, parts, lg);
  return cudaGetLastError();
}

cudaError_t launch_dt_finalize(unsigned long long* acc, double cfl, double* dt_out, double* hist,
                               cudaStream_t s, int n) {
  dt_finalize_kernel<<<(n + 255) / 256, n < 256 ? n : 256, 0, s>>>(acc, cfl, dt_out, hist, n);
  return cudaGetLastError();
}

cudaError_t launch_check(const double* U, Layout lay, Eos eos, unsigned long long* count,
                         cudaStream_t s) {
  const long long work = (long long)lay.nblocks * lay.nx * lay.ny * lay.nz;
  check_kernel<<<grid_for(work, kThreads), kThreads, 0, s>>>(U, lay, eos, count);
  return cudaGetLastError();
}

cudaError_t launch_bits_selftest(const double* x, const double* y, double* out, long long n, cudaStream_t s) {
  bits_selftest_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(x, y, out, n, 0);
  return cudaGetLastError();
}

cudaError_t launch_fastmath_selftest(const double* x, double* out, long long n, cudaStream_t s) {
  fastmath_selftest_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(x, out, n);
  return cudaGetLastError();
}

cudaError_t launch_op_count(int fn, int blocks, int threads, int iters, const Eos& e, double* io, cudaStream_t s) {
  switch (fn) {
    case 0: op_count_kernel<0><<<blocks, threads, 0, s>>>(iters, e, io); break;
    case 1: op_count_kernel<1><<<blocks, threads, 0, s>>>(iters, e, io); break;
    case 2: op_count_kernel<2><<<blocks, threads, 0, s>>>(iters, e, io); break;
    case 3: op_count_kernel<3><<<blocks, threads, 0, s>>>(iters, e, io); break;
    case 4: op_count_kernel<4><<<blocks, threads, 0, s>>>(iters, e, io); break;
    case 5: op_count_kernel<5><<<blocks, threads, 0, s>>>(iters, e, io); break;
    case 6: op_count_kernel<6><<<blocks, threads, 0, s>>>(iters, e, io); break;
    case 7: op_count_kernel<7><<<blocks, threads, 0, s>>>(iters, e, io); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_fp64_probe(int blocks, int threads, int iters, int lanes, int form, double* out, cudaStream_t s) {
  switch (form) {
    case 0: fp64_probe_kernel<0><<<blocks, threads, 0, s>>>(iters, lanes, 0, out); break;
    case 1: fp64_probe_kernel<1><<<blocks, threads, 0, s>>>(iters, lanes, 0, out); break;
    case 2: fp64_probe_kernel<2><<<blocks, threads, 0, s>>>(iters, lanes, 0, out); break;
    case 3: fp64_probe_kernel<3><<<blocks, threads, 0, s>>>(iters, lanes, 0, out); break;
    case 4: fp64_probe_kernel<4><<<blocks, threads, 0, s>>>(iters, lanes, 0, out); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace gbh
