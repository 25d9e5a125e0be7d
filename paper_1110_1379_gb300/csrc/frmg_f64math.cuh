// frmg_f64math.cuh -- FP64 reciprocal, reciprocal square root and e^u - 1 in as
// few FP64 instructions as their accuracy allows.
//
// GB300 issues one FP64 warp instruction per 16 cycles and SM, 1/64 of the FP32
// rate, so the FP64 smoother, residual and prolongation take the time of
// their FP64 instructions.  These functions replace the library's division,
// square root and expm1 there; with the regrouped face sums (OpAcc<double>)
// and one reciprocal per update they took a colour of a sweep at 128^3 from 221
// to 144 us (66 FP64 instructions per update, 80 % of the pipe's rate), the
// residual from 225 to 158 us and the prolongation from 143 to 127 us.
#pragma once

#include <cuda_runtime.h>

namespace frmg {

// v is normal and at least 2^20 away from the ends of the exponent's range (an
// integer test of the high word: zeros, infinities and NaN fail it too).
__device__ __forceinline__ bool f64_tame(double v) {
  return ((__double2hiint(v) >> 20) & 0x7ff) - 21u < 2005u;
}

// 1/v: the hardware's approximation (about 20 bits) and one step of the
// third-order iteration r (1 + e + e^2), e = 1 - v r (the geometric series cut
// after e^2; its remainder e^3 is below 2^-57): error below 0.55 ulp.  v tame.
__device__ __forceinline__ double f64_rcp(double v) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(v));
  const double e = fma(-v, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// 1/sqrt(v): the hardware's approximation and one step of Halley's third-order
// iteration, r (1 + e/2 + 3 e^2/8), e = 1 - v r^2 (the binomial series of
// (1 - e)^(-1/2)): error below 1.05 ulp (half an ulp from v r, half from the last
// step).  v > 0 and tame.
__device__ __forceinline__ double f64_rsqrt(double v) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(v));
  const double e = fma(-v * r, r, 1.0);
  return fma(r * e, fma(0.375, e, 0.5), r);
}

// 2^(i/16), i = -8 .. 7, rounded, and the relative rounding error of each.
__device__ const double kExpTab[32] = {
    0x1.6a09e667f3bcdp-1,   0x1.7a11473eb0187p-1,   0x1.8ace5422aa0dbp-1,
    0x1.9c49182a3f090p-1,   0x1.ae89f995ad3adp-1,   0x1.c199bdd85529cp-1,
    0x1.d5818dcfba487p-1,   0x1.ea4afa2a490dap-1,   0x1.0000000000000p+0,
    0x1.0b5586cf9890fp+0,   0x1.172b83c7d517bp+0,   0x1.2387a6e756238p+0,
    0x1.306fe0a31b715p+0,   0x1.3dea64c123422p+0,   0x1.4bfdad5362a27p+0,
    0x1.5ab07dd485429p+0,   -0x1.3b3efbf5e2229p-54, -0x1.b32dcb94da51dp-56,
    0x1.db72fc1f0eab4p-55,  0x1.1affc2b91ce27p-56,  0x1.c1a7792cb3386p-55,
    0x1.36eae30af0cb3p-56,  0x1.4a385a63d07a7p-56,  -0x1.ff7128fd391f1p-55,
    0x0.0p+0,               0x1.79aa65d837b6cp-54,  -0x1.01b15eaa59348p-55,
    0x1.68efde3a8a893p-54,  0x1.34d754db0abb6p-55,  0x1.59f48a72a4c6cp-55,
    0x1.690cebb7aafb0p-56,  0x1.063e1e21c5409p-54};

// e^u = t (1 + p) with t = 2^(k/16) and p = e^r - 1, u = k ln2/16 + r, |r| <=
// ln2/32: the table-driven method of P. T. P. Tang, "Table-driven
// implementation of the Expm1 function in IEEE floating-point arithmetic",
// ACM TOMS 18 (1992) 211, with a 16-entry table and the Taylor series of p to
// degree 7 (remainder below 2^-54 relative to r).  |u| < 700.
__device__ __forceinline__ void f64_exp_parts(double u, double &t, double &p) {
  const double shift = 0x1.8p52;
  const double ks = fma(u, 0x1.71547652b82fep+4, shift);  // 16 / ln2
  const int k = __double2loint(ks);
  const double kd = ks - shift;
  // ln2/16 in two pieces, the first with 20 trailing zero bits: k times it is exact
  double r = fma(-kd, 0x1.62e42fee00000p-5, u);
  r = fma(-kd, 0x1.a39ef35793c76p-37, r);
  const int m = (k + 8) >> 4, i = (k + 8) & 15;
  const double t0 = __ldg(kExpTab + i), dt = __ldg(kExpTab + 16 + i);
  t = __hiloint2double(__double2hiint(t0) + (m << 20), __double2loint(t0));
  const double r2 = r * r;
  const double a = fma(r, 1.0 / 6.0, 0.5), b = fma(r, 1.0 / 120.0, 1.0 / 24.0),
               c = fma(r, 1.0 / 5040.0, 1.0 / 720.0);
  p = fma(fma(fma(c, r2, b), r2, a), r2, r + dt);
}

// e^u - 1 = (t - 1) + t p, the first bracket exact; for |u| < ln2/32 the series
// itself.  Largest errors found (2e7 arguments per range): 0.85 ulp for |u| <
// ln2/32, 2.24 ulp from there to 0.035 (r, r + dt and p, each as large as the
// result, are rounded), 1.24 ulp to 0.1, 1.03 ulp beyond; below 0.3 ulp of e^u for
// |u| < 0.4.  14 FP64 instructions.
__device__ __forceinline__ double f64_expm1(double u) {
  if (!(fabs(u) < 700.0)) return expm1(u);  // overflow, -1, NaN
  double t, p;
  f64_exp_parts(u, t, p);
  return fma(t, p, t - 1.0);
}

// e^u, error below 0.55 ulp.
__device__ __forceinline__ double f64_exp(double u) {
  if (!(fabs(u) < 700.0)) return exp(u);
  double t, p;
  f64_exp_parts(u, t, p);
  return fma(t, p, t);
}

}  // namespace frmg
