"""The per-cell and per-face arithmetic of the kernels (gbh_device.cuh) compiled
for the host, so that its edge cases can be checked on the CPU.

The header is device code without launches: with the few intrinsics it uses
written out below, g++ compiles it as it stands.  The FP32 seeds of the
reciprocal and root are then the host's correctly rounded ones.  The one FP32
rule that matters to the results, that an operation with a NaN result gives the
pattern 0x7fffffff, is applied where the header reads the bits of a float."""
import ctypes as C
import os
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>
static struct { unsigned x = 0; } threadIdx;
static inline long long __double_as_longlong(double x) { long long r; std::memcpy(&r, &x, 8); return r; }
static inline double __longlong_as_double(long long x) { double r; std::memcpy(&r, &x, 8); return r; }
static inline unsigned __float_as_uint(float x) {
  unsigned r;
  std::memcpy(&r, &x, 4);
  return x != x ? 0x7fffffffu : r;
}
static inline float __uint_as_float(unsigned x) { float r; std::memcpy(&r, &x, 4); return r; }
static inline int __double2hiint(double x) { return (int)(__double_as_longlong(x) >> 32); }
static inline int __double2loint(double x) { return (int)__double_as_longlong(x); }
template <class T> static inline T __shfl_xor_sync(unsigned, T v, int) { return v; }
static inline void __syncthreads() {}
#include "gbh_device.cuh"
using namespace gbh;

static Eos eos(const double* q) {          // gamma, small_rho, small_p
  Eos e{};
  e.gamma = q[0]; e.gm1 = q[0] - 1; e.g_gm1 = q[0] / (q[0] - 1); e.hgm1 = 0.5 * (q[0] - 1);
  e.small_rho = q[1]; e.small_p = q[2];
  e.k.one = 1.0; e.k.nz = -0.0;
  e.wgamma = wide_of(e.gamma); e.wgm1 = wide_of(e.gm1); e.whgm1 = wide_of(e.hgm1); e.wg_gm1 = wide_of(e.g_gm1);
  return e;
}
extern "C" {
void hd_hllc(const double* q, long n, const double* WL, const double* WR, double* F) {
  const Eos e = eos(q);
  for (long i = 0; i < 5 * n; i += 5) hllc_flux(WL + i, WR + i, e, F + i);
}
// W and the floor count of a stage; W as the CFL reduction takes it and its speed for
// inverse cell widths d
void hd_prim(const double* q, long n, const double* U, const double* d, double* W, int* hit, double* Wd, double* speed) {
  const Eos e = eos(q);
  for (long i = 0; i < n; ++i) {
    Wide ir;
    hit[i] = cons_to_prim_ir(U + 5 * i, W + 5 * i, e, ir);
    std::memcpy(Wd + 5 * i, W + 5 * i, 5 * sizeof(double));
    prim_beyond(U + 5 * i, Wd + 5 * i, ir, e);
    speed[i] = signal_speed_ir(Wd + 5 * i, ir, e, d[0], d[1], d[2], inv_width_sum(e, d[0], d[1], d[2], true), true);
  }
}
// s / (s + b) with s = sqrt(a): the Roe weight's form, from the unpacked numbers
void hd_weight(long n, const double* a, const double* b, double* r) {
  for (long i = 0; i < n; ++i) {
    const Wide s = wide_sqrt(wide_of(a[i]));
    r[i] = wide_double(wide_mul(s, wide_rcp_low(wide_add(s, wide_of(b[i])))));
  }
}
}
"""


def _cuda_include():
    from paper_2401_03378_gb300.build import nvcc
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")


def build(tmp):
    """The library, compiled into the directory tmp."""
    src, out = os.path.join(tmp, "hostdevice.cpp"), os.path.join(tmp, "libhostdevice.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    inc = [_cuda_include(), os.path.join(os.path.dirname(_cuda_include()), "targets/x86_64-linux/include"),
           os.path.join(os.path.dirname(_cuda_include()), "targets/sbsa-linux/include"),
           os.path.join(ROOT, "paper_2401_03378_gb300/csrc")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-fPIC", "-shared", "-w",
                    *[x for i in inc for x in ("-I", i)], src, "-o", out], check=True)
    return C.CDLL(out)


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


class HostDevice:
    def __init__(self, tmp, gamma=1.4, small_rho=1e-12, small_p=1e-14):
        self.lib = build(str(tmp))
        self.q = np.array([gamma, small_rho, small_p])

    def hllc(self, WL, WR):
        WL, WR = (np.ascontiguousarray(np.atleast_2d(x), dtype=np.float64) for x in (WL, WR))
        F = np.empty_like(WL)
        self.lib.hd_hllc(_p(self.q), C.c_long(len(WL)), _p(WL), _p(WR), _p(F))
        return F

    def prim(self, U, inv_dx=(1.0, 2.0, 3.0), beyond=False):
        """(W, floor count, CFL speed); beyond: W as the CFL reduction takes it."""
        U = np.ascontiguousarray(np.atleast_2d(U), dtype=np.float64)
        d = np.array(inv_dx, dtype=np.float64)
        W, Wd = np.empty_like(U), np.empty_like(U)
        hit, s = np.empty(len(U), dtype=np.int32), np.empty(len(U))
        self.lib.hd_prim(_p(self.q), C.c_long(len(U)), _p(U), _p(d), _p(W), _p(hit), _p(Wd), _p(s))
        return (Wd if beyond else W), hit, s

    def weight(self, a, b):
        a, b = (np.ascontiguousarray(x, dtype=np.float64) for x in (a, b))
        r = np.empty_like(a)
        self.lib.hd_weight(C.c_long(len(a)), _p(a), _p(b), _p(r))
        return r
