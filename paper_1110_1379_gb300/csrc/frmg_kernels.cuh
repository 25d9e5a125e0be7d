// frmg_kernels.cuh -- device code of the f(R) FAS multigrid solver (sm_103a).
//
// Operator (Sec. IV Eq. discrete_fR times c~^2, Sec. V.B.1 Eq. bc_modified_fR_op)
// in u = ln(f_R/fbar_R), as a nonlinear operator A with right-hand side f:
//
//   A_i(u) = (alpha/2) sum_j (e^{u_i} + e^{u_j}) (u_j - u_i) + beta (e^{-u_i/2} - 1)
//   finest level:  A(u) = gamma (rho - 1);  coarse levels: A^H(u^H) = f^H (FAS).
//
// Two evaluation modes share one code path:
//  * plain (BG = false): u is the unknown itself.  Cache x = expm1(u), so
//    B = e^u = 1 + x.
//  * background (BG = true, FP32 inside the mixed-precision loop): the unknown
//    is a correction delta on a fixed FP32 background ub (E = e^{ub}), and the
//    kernels evaluate N(delta) = A(ub + delta) - A(ub) in a form where every
//    term carries a factor of delta:
//      (alpha/2) sum_j [ (E_i x_i + E_j x_j)(ub_j - ub_i) + (B_i + B_j)(d_j - d_i) ]
//      + beta e^{-ub_i/2} (e^{-d_i/2} - 1),    x = expm1(delta), B = E (1 + x).
//    so that FP32 rounding is relative to the correction, not to u.
// Both modes give the same Newton derivative (Eq. bc_modified_fR_dop):
//   dA_i/du_i = (alpha/2) sum_j [ B_i (u_j - u_i) - (B_i + B_j) ] - (beta/2) e^{-u_i/2}.
//
// Refinement patches: a ghost neighbour outside the patch takes
//   u_g = u_b - r u_b + r u_i with r = -1, b_g = exp(u_g)     (Eq. u_i-1jk),
// so its face contributes (B_i + B_g)(u_g - u_i) and, because u_g depends on
// u_i, (B_i - B_g)(u_g - u_i) - 2 (B_i + B_g) to the derivative.
//
// Red-black ordering: colour = (i + j + k) & 1, red (0) first.
// Layout: [n2][n1][n0], x fastest.  Packed boundary faces: -x,+x,-y,+y,-z,+z,
// face normal to axis a indexed by the other axes p < q as c[q]*n[p] + c[p].
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

#include "frmg_dfmath.cuh"
#include "frmg_f64math.cuh"

namespace frmg {

template <typename T>
struct Grid {
  T *u;            // unknown (delta in background mode), buffer 0
  T *u2;           // buffer 1: the tiled smoother reads one buffer and writes the other
  T *x2;           // buffer 1 of the x cache (ping-pongs with u)
  T *x;            // cache: expm1(u)
  const T *f;      // right-hand side storage; f_i = fs * (f[i] - fo); null = 0
                   // (FP32 grids store f_i itself: fs = 1, fo = 0)
  T *uR;           // R u^h saved for the FAS correction (coarse levels)
  const float *ubg;  // background (BG mode), null otherwise
  const float *Ebg;  // exp(background)
  const T *bnd;    // packed Dirichlet faces (null: periodic)
  long long foff[6];
  long long ncell;
  int n0, n1, n2;
  int field;       // index into the active-flag array
  T ah;            // alpha / 2
  T beta;
  T fs, fo;
  T cap;           // Newton step cap
  T relax;         // relaxation factor of the Newton update (1: plain Newton-GS)
  FastDiv fd0, fd1;  // division by n0 and n1 (cell index -> (i, j, k))
};

// (i, j, k) of the linear cell index c < ncell: 32-bit multiply-shift division
// below 2^31 cells, 64-bit division above.
template <typename T>
__device__ __forceinline__ void cell_ijk(const Grid<T> &G, long long c, int &i, int &j, int &k) {
  if (G.ncell < (1ll << 31)) {
    const unsigned cu = (unsigned)c, q = fdiv(cu, G.fd0), q2 = fdiv(q, G.fd1);
    i = (int)(cu - q * (unsigned)G.n0);
    j = (int)(q - q2 * (unsigned)G.n1);
    k = (int)q2;
  } else {
    i = (int)(c % G.n0);
    const long long r = c / G.n0;
    j = (int)(r % G.n1);
    k = (int)(r / G.n1);
  }
}

// ----------------------------------------------------------------------------
// math wrappers (library functions; no re-derived constants)
__device__ __forceinline__ float m_exp(float v) { return expf(v); }
__device__ __forceinline__ double m_exp(double v) { return exp(v); }
// FP32 e^d - 1 used by every FP32 kernel (so all of them see the same cache
// values): the Taylor series to degree 6 for |d| < 1/16 (truncation below
// 1e-12 relative, which keeps small corrections exact to FP32 rounding), and
// the correctly rounded-to-1-ulp exponential minus one otherwise (strongly
// screened cells reach |u| ~ 10, where the SFU approximation's error of a few
// ulp per unit of |u| would set the FP32 residual floor).
// Every FP32 operation of the shared operator code is written out as an
// explicit rounding (fmaf, __fadd_rn, __fmul_rn, ...), so that no kernel's
// compiler contraction can change it: the scalar and the packed (two cells per
// instruction, below) evaluations are then the same bit for bit.
__device__ __forceinline__ float m_expm1_taylor(float d) {
  float p = fmaf(d, 1.0f / 720.0f, 1.0f / 120.0f);
  p = fmaf(d, p, 1.0f / 24.0f);
  p = fmaf(d, p, 1.0f / 6.0f);
  p = fmaf(d, p, 0.5f);
  p = fmaf(d, p, 1.0f);
  return __fmul_rn(d, p);
}
__device__ __forceinline__ float m_expm1(float d) {
  if (fabsf(d) < 0.0625f) return m_expm1_taylor(d);
  return __fsub_rn(expf(d), 1.0f);
}
__device__ __forceinline__ double m_expm1(double v) { return f64_expm1(v); }
__device__ __forceinline__ float m_sqrt(float v) { return sqrtf(v); }
__device__ __forceinline__ double m_sqrt(double v) { return sqrt(v); }
__device__ __forceinline__ float m_rsqrt(float v) { return rsqrtf(v); }
__device__ __forceinline__ double m_rsqrt(double v) { return rsqrt(v); }

__device__ __forceinline__ int wrapmod(int v, int n) {
  int r = v % n;
  return r < 0 ? r + n : r;
}

__device__ __forceinline__ int find_grid(const int *off, int ngrid, int b) {
  int lo = 0, hi = ngrid;  // off[lo] <= b < off[hi]
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (off[mid] <= b)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// Grid view whose u is the current buffer (par selects buffer 0 or 1).
template <typename T>
__device__ __forceinline__ Grid<T> view(const Grid<T> *grids, int g, int par) {
  Grid<T> G = grids[g];
  if (par) {
    G.u = G.u2;
    G.x = G.x2;
  }
  return G;
}

__device__ __forceinline__ bool grid_active(const int *active, int field) {
  return active == nullptr || active[field] != 0;
}

template <typename T>
__device__ __forceinline__ long long idx3(const Grid<T> &G, int i, int j, int k) {
  return ((long long)k * G.n1 + j) * G.n0 + i;
}

// Boundary value of the face f (0..5) at the boundary cell (i,j,k).
template <typename T>
__device__ __forceinline__ T face_value(const Grid<T> &G, int f, int i, int j, int k) {
  long long o;
  if (f < 2)
    o = (long long)k * G.n1 + j;
  else if (f < 4)
    o = (long long)k * G.n0 + i;
  else
    o = (long long)j * G.n0 + i;
  return G.bnd[G.foff[f] + o];
}

// Contribution of one regular face (neighbour values given).
template <typename T, bool BG>
__device__ __forceinline__ void face_vals(T dj, T xj, T ubj, T Ej, T di, T Ei, T xi, T Bi, T ubi,
                                          T &acc, T &dacc) {
  T Bj = BG ? Ej + Ej * xj : T(1) + xj;
  T dd = dj - di;
  T w;
  if (BG) {
    T gd = ubj - ubi;
    acc += (Ei * xi + Ej * xj) * gd + (Bi + Bj) * dd;
    w = gd + dd;
  } else {
    acc += (Bi + Bj) * dd;
    w = dd;
  }
  dacc += Bi * w - (Bi + Bj);
}

template <typename T, bool BG>
__device__ __forceinline__ void face_ghost(T ubf, T di, T Ei, T xi, T Bi, T ubi, T &acc,
                                           T &dacc) {
  T w, Bg;
  if (BG) {
    T ubgh = T(2) * ubf - ubi;   // background ghost
    T Eg = m_exp(ubgh);
    T xg = -xi / (T(1) + xi);    // expm1(-delta_i)
    T gd = ubgh - ubi;
    T dd = T(-2) * di;           // delta_g - delta_i
    Bg = Eg + Eg * xg;
    acc += (Ei * xi + Eg * xg) * gd + (Bi + Bg) * dd;
    w = gd + dd;
  } else {
    T ug = T(2) * ubf - di;
    Bg = m_exp(ug);
    w = ug - di;
    acc += (Bi + Bg) * w;
  }
  dacc += (Bi - Bg) * w - T(2) * (Bi + Bg);
}

// Face-sum accumulator of one cell: own values at construction, one call per
// face (regular neighbour or patch ghost), then the two sums
//   acc  = sum_faces (flux term),   dacc = sum_faces d(flux term)/du_i.
// The generic form adds (B_i + B_j)(u_j - u_i) face by face.  The plain FP32
// form (the bulk of the mixed-precision work) regroups the same sum as
//   acc  = (B_i + 1) S1 + S2,   dacc = B_i S1 - n (B_i + 1) - S3,
//   S1 = sum (u_j - u_i),  S2 = sum x_j (u_j - u_i),  S3 = sum x_j,
// over the n regular faces (B_j = 1 + x_j), four operations per face instead
// of six; every FP32 kernel uses this one accumulator, so all of them evaluate
// the same discrete operator.
template <typename T, bool BG>
struct OpAcc {
  T di, Ei, xi, Bi, ubi;
  T acc = T(0), dacc = T(0);
  __device__ __forceinline__ OpAcc(T d, T E, T x, T B, T ub) : di(d), Ei(E), xi(x), Bi(B), ubi(ub) {}
  __device__ __forceinline__ void reg(T dj, T xj, T ubj, T Ej) {
    face_vals<T, BG>(dj, xj, ubj, Ej, di, Ei, xi, Bi, ubi, acc, dacc);
  }
  __device__ __forceinline__ void ghost(T ubf) {
    face_ghost<T, BG>(ubf, di, Ei, xi, Bi, ubi, acc, dacc);
  }
  __device__ __forceinline__ void done(T &a, T &da) const {
    a = acc;
    da = dacc;
  }
};

template <>
struct OpAcc<float, false> {
  float di, Ei, xi, Bi, ubi;
  float S1 = 0.f, S2 = 0.f, S3 = 0.f, ga = 0.f, gd = 0.f;
  int n = 0;
  __device__ __forceinline__ OpAcc(float d, float E, float x, float B, float ub)
      : di(d), Ei(E), xi(x), Bi(B), ubi(ub) {}
  __device__ __forceinline__ void reg(float dj, float xj, float, float) {
    const float dd = __fsub_rn(dj, di);
    S1 = __fadd_rn(S1, dd);
    S2 = fmaf(xj, dd, S2);
    S3 = __fadd_rn(S3, xj);
    n++;
  }
  __device__ __forceinline__ void ghost(float ubf) {
    face_ghost<float, false>(ubf, di, Ei, xi, Bi, ubi, ga, gd);
  }
  __device__ __forceinline__ void done(float &a, float &da) const {
    const float nf = (float)n;
    const float b1 = __fadd_rn(Bi, 1.0f);
    a = __fadd_rn(fmaf(b1, S1, S2), ga);
    da = __fadd_rn(__fsub_rn(fmaf(Bi, S1, __fmul_rn(-nf, b1)), S3), gd);
  }
};

// The same regrouping in FP64 (24 FP64 operations for the six faces instead of
// 36); a ghost's terms join the sums directly.
template <>
struct OpAcc<double, false> {
  double di, Ei, xi, Bi, ubi;
  double S1 = 0.0, S2 = 0.0, S3 = 0.0;
  int n = 0;
  __device__ __forceinline__ OpAcc(double d, double E, double x, double B, double ub)
      : di(d), Ei(E), xi(x), Bi(B), ubi(ub) {}
  __device__ __forceinline__ void reg(double dj, double xj, double, double) {
    const double dd = dj - di;
    S1 += dd;
    S2 = fma(xj, dd, S2);
    S3 += xj;
    n++;
  }
  __device__ __forceinline__ void ghost(double ubf) {
    double ga = 0.0, gd = 0.0;
    face_ghost<double, false>(ubf, di, Ei, xi, Bi, ubi, ga, gd);
    S2 += ga;
    S3 -= gd;
  }
  __device__ __forceinline__ void done(double &a, double &da) const {
    const double b1 = Bi + 1.0;
    a = fma(b1, S1, S2);
    da = fma(Bi, S1, (double)-n * b1) - S3;
  }
};

// The FP32 correction form regroups its face sum the same way: with
// P = E x (so B = E + P) and g_j = ub_j - ub_i,
//   acc  = sum (P_i + P_j) g_j + (B_i + B_j)(d_j - d_i)
//        = P_i G1 + G2 + B_i S1 + S2,
//   dacc = sum B_i (g_j + d_j - d_i) - (B_i + B_j) = B_i (G1 + S1) - n B_i - S3,
//   G1 = sum g_j, G2 = sum P_j g_j, S1 = sum (d_j - d_i), S2 = sum B_j (d_j - d_i),
//   S3 = sum B_j,
// nine operations per face instead of about twelve, every rounding explicit.
template <>
struct OpAcc<float, true> {
  float di, Ei, xi, Bi, ubi;
  float G1 = 0.f, G2 = 0.f, S1 = 0.f, S2 = 0.f, S3 = 0.f, ga = 0.f, gd = 0.f;
  int n = 0;
  __device__ __forceinline__ OpAcc(float d, float E, float x, float B, float ub)
      : di(d), Ei(E), xi(x), Bi(B), ubi(ub) {}
  __device__ __forceinline__ void reg(float dj, float xj, float ubj, float Ej) {
    const float Pj = __fmul_rn(Ej, xj);
    reg_pb(dj, Pj, ubj, __fadd_rn(Ej, Pj));
  }
  // the neighbour's P = E x and B = E + P formed beforehand
  __device__ __forceinline__ void reg_pb(float dj, float Pj, float ubj, float Bj) {
    const float dd = __fsub_rn(dj, di), g = __fsub_rn(ubj, ubi);
    G1 = __fadd_rn(G1, g);
    G2 = fmaf(Pj, g, G2);
    S1 = __fadd_rn(S1, dd);
    S2 = fmaf(Bj, dd, S2);
    S3 = __fadd_rn(S3, Bj);
    n++;
  }
  __device__ __forceinline__ void ghost(float ubf) {
    face_ghost<float, true>(ubf, di, Ei, xi, Bi, ubi, ga, gd);
  }
  __device__ __forceinline__ void done(float &a, float &da) const {
    const float nf = (float)n;
    const float Pi = __fmul_rn(Ei, xi);
    a = __fadd_rn(__fadd_rn(fmaf(Pi, G1, G2), fmaf(Bi, S1, S2)), ga);
    da = __fadd_rn(__fsub_rn(fmaf(Bi, __fadd_rn(G1, S1), __fmul_rn(-nf, Bi)), S3), gd);
  }
};

// 1 / sqrt(B) and e^{-d/2} - 1 = -x / (B + sqrt B), B = 1 + x, for any B
// (0, infinite and NaN ones too).
__device__ __noinline__ double2 mass_wide(double xi) {
  const double B1 = 1.0 + xi, s = sqrt(B1);
  return make_double2(1.0 / s, -xi / (B1 + s));
}

// Mass term and final assembly:  N = (alpha/2) acc + beta F (e^{-d/2} - 1),
// dN = (alpha/2) dacc - (beta/2) F e^{-d/2},  F = e^{-ub/2}.
// FP32 uses the SFU reciprocal square root and reciprocal (the same expression
// in every FP32 kernel, so all of them see one and the same discrete operator).
__device__ __forceinline__ void finish_op(double xi, double Ei, double acc, double dacc,
                                          double ah, double beta, bool bg, double &N,
                                          double &dN) {
  const double B1 = 1.0 + xi;
  const double bF = bg ? beta * rsqrt(Ei) : beta;
  double2 m;
  if (f64_tame(B1)) {
    m.x = f64_rsqrt(B1);
    m.y = -xi * f64_rcp(fma(B1, m.x, B1));
  } else {
    m = mass_wide(xi);
  }
  N = fma(ah, acc, bF * m.y);
  dN = fma(ah, dacc, -0.5 * bF * m.x);
}

// SFU reciprocal and reciprocal square root (PTX rcp.approx / rsqrt.approx,
// subnormals flushed: every FP32 quantity here is far from the subnormal range).
__device__ __forceinline__ float sfu_rcp(float v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float sfu_rsqrt(float v) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

__device__ __forceinline__ void finish_op(float xi, float Ei, float acc, float dacc, float ah,
                                          float beta, bool bg, float &N, float &dN) {
  const float B1 = __fadd_rn(1.0f, xi);
  const float rs = sfu_rsqrt(B1);  // e^{-d/2}
  const float s = __fmul_rn(B1, rs);  // e^{d/2}
  const float y = __fmul_rn(-xi, sfu_rcp(__fadd_rn(B1, s)));
  const float bF = bg ? __fmul_rn(beta, sfu_rsqrt(Ei)) : beta;  // beta F
  N = fmaf(ah, acc, __fmul_rn(bF, y));
  dN = fmaf(ah, dacc, -__fmul_rn(__fmul_rn(0.5f, bF), rs));
}

__device__ __forceinline__ float newton_step(float r, float dN) {
  return __fmul_rn(-r, sfu_rcp(dN));
}
// relaxed Newton step w (N - f) / -dN of a cell
__device__ __forceinline__ float newton_du(float N, float f, float dN, float w) {
  return __fmul_rn(w, newton_step(__fsub_rn(N, f), dN));
}

// The FP64 Newton step with the library's division and root: where the
// products below leave the range of FP64 (u above about 350, B = 0, non-finite
// values).
__device__ __noinline__ double newton_wide(double xi, double acc, double dacc, double f, double ah,
                                           double beta, double relax) {
  const double B1 = 1.0 + xi, s = sqrt(B1);
  const double N = ah * acc + beta * (-xi / (B1 + s));
  const double dN = ah * dacc - 0.5 * beta / s;
  return relax * (-(N - f) / dN);
}

// The clamped, relaxed Newton step of a cell from its face sums.  FP64, plain
// form: with q = B + sqrt(B) both N - f and dN are multiplied by q, so that one
// reciprocal serves the mass term and the step.
template <typename T, bool BG>
__device__ __forceinline__ T newton_from_sums(T xi, T Ei, T acc, T dacc, T f, T ah, T beta, T cap,
                                              T relax) {
  if constexpr (sizeof(T) == 8 && !BG) {
    const T B1 = T(1) + xi, rs = f64_rsqrt(B1), q = fma(B1, rs, B1);
    const T num = fma(-beta, xi, fma(ah, acc, -f) * q);
    const T den = fma(ah, dacc, T(-0.5) * beta * rs) * q;
    T du;
    // (num below 2^1004, so that relax num is finite; a NaN of num or of rs at
    // B = 0 fails the tests too)
    if (f64_tame(den) && ((__double2hiint(num) >> 20) & 0x7ff) < 2027)
      du = -relax * num * f64_rcp(den);
    else
      du = newton_wide(xi, acc, dacc, f, ah, beta, relax);
    // the comparison by the high words first (an FP64 comparison takes the FP64 pipe)
    if ((__double2hiint(du) & 0x7fffffff) < __double2hiint(cap)) return du;
    return du > cap ? cap : (du < -cap ? -cap : du);
  } else {
    T N, dN;
    finish_op(xi, Ei, acc, dacc, ah, beta, BG, N, dN);
    const T du = newton_du(N, f, dN, relax);
    return du > cap ? cap : (du < -cap ? -cap : du);
  }
}

// ---- packed FP32 pairs (add2, sub2, fma2, mul2, splat2 of frmg_dfmath.cuh)
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// m_expm1 of two values: the Taylor branch packed, the exponential branch per lane
__device__ __forceinline__ float2 m_expm1_2(float2 d) {
  float2 p = fma2(d, splat2(1.0f / 720.0f), splat2(1.0f / 120.0f));
  p = fma2(d, p, splat2(1.0f / 24.0f));
  p = fma2(d, p, splat2(1.0f / 6.0f));
  p = fma2(d, p, splat2(0.5f));
  p = fma2(d, p, splat2(1.0f));
  float2 r = mul2(d, p);
  if (!(fabsf(d.x) < 0.0625f)) r.x = __fsub_rn(expf(d.x), 1.0f);
  if (!(fabsf(d.y) < 0.0625f)) r.y = __fsub_rn(expf(d.y), 1.0f);
  return r;
}

// expm1 of two values of the full variable without a branch (the full u has
// cells on both sides of m_expm1's threshold in most warps, which then run its
// two branches): d = n ln2 + r, |r| <= ln2 / 2, with ln2 in two parts (Cody and
// Waite 1980), expm1(r) by its Taylor series to degree 7 (truncation below
// r^7 / 8! = 1.5e-8), 2^n expm1(r) + (2^n - 1).  n = 0 near zero, so small d
// keep their relative accuracy.  d below -88 counts as -88 (n = -127, 2^-127
// counts as 0: -1), n is at most 127 (infinity from d = 88.73 on), a NaN stays
// one.  Relative error <= 1.6e-7 up to d = 88 (6.3e-7 up to 88.7), m_expm1 9.2e-7
// (expf(d) - 1 just above its threshold).
// Sweep with prolongation at 512^3 0.896 -> 0.851 ms; on a batch of 48 grids of
// 32^3 to 128^3 0.337 -> 0.288, its plain sweeps 0.215 -> 0.201.
__device__ __forceinline__ float max_nan(float a, float b) {  // NaN if one is
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 m_expm1_full2(float2 d) {
  const float magic = 12582912.0f;  // 1.5 2^23: the sum's low bits are n
  d = make_float2(max_nan(d.x, -88.0f), max_nan(d.y, -88.0f));
  float2 t = fma2(d, splat2(1.44269504f), splat2(magic));
  t.x = fminf(t.x, magic + 127.0f);
  t.y = fminf(t.y, magic + 127.0f);
  const float2 n = sub2(t, splat2(magic));
  // ln2 = 0.693359375 (10 bits, n times it is exact) - 2.12194440e-4
  float2 r = fma2(n, splat2(-0.693359375f), d);
  r = fma2(n, splat2(2.12194440e-4f), r);
  float2 p = fma2(r, splat2(1.0f / 5040.0f), splat2(1.0f / 720.0f));
  p = fma2(r, p, splat2(1.0f / 120.0f));
  p = fma2(r, p, splat2(1.0f / 24.0f));
  p = fma2(r, p, splat2(1.0f / 6.0f));
  p = fma2(r, p, splat2(0.5f));
  p = fma2(r, p, splat2(1.0f));
  p = mul2(r, p);
  const float2 s = make_float2(__int_as_float((__float_as_int(t.x) << 23) + (127 << 23)),
                               __int_as_float((__float_as_int(t.y) << 23) + (127 << 23)));
  return fma2(s, p, add2(s, splat2(-1.0f)));
}
// the same of one value, operation for operation
__device__ __forceinline__ float m_expm1_full(float d) {
  const float magic = 12582912.0f;
  d = max_nan(d, -88.0f);
  const float t = fminf(fmaf(d, 1.44269504f, magic), magic + 127.0f);
  const float n = __fsub_rn(t, magic);
  const float r = fmaf(n, 2.12194440e-4f, fmaf(n, -0.693359375f, d));
  float p = fmaf(r, 1.0f / 5040.0f, 1.0f / 720.0f);
  p = fmaf(r, p, 1.0f / 120.0f);
  p = fmaf(r, p, 1.0f / 24.0f);
  p = fmaf(r, p, 1.0f / 6.0f);
  p = fmaf(r, p, 0.5f);
  p = __fmul_rn(r, fmaf(r, p, 1.0f));
  const float s = __int_as_float((__float_as_int(t) << 23) + (127 << 23));
  return fmaf(s, p, __fadd_rn(s, -1.0f));
}

// The plain-form Newton update of two cells at once, operation for operation
// the scalar OpAcc<float, false> (six regular faces), finish_op and newton_du:
// own (u, x), right-hand side f, neighbour u and x in the face order -x, +x,
// -y, +y, -z, +z; returns the two new u.
__device__ __forceinline__ float2 newton2_plain(float2 di, float2 xi, float2 fi, const float2 *nu,
                                                const float2 *nx, float ah, float beta, float cap,
                                                float relax) {
  const float2 Bi = add2(splat2(1.0f), xi);
  float2 S1 = sub2(nu[0], di), S2, S3 = nx[0];
  S2 = mul2(nx[0], S1);  // fmaf(x, dd, 0) rounds as the product
#pragma unroll
  for (int f = 1; f < 6; f++) {
    const float2 dd = sub2(nu[f], di);
    S1 = add2(S1, dd);
    S2 = fma2(nx[f], dd, S2);
    S3 = add2(S3, nx[f]);
  }
  const float2 b1 = add2(Bi, splat2(1.0f));
  const float2 acc = fma2(b1, S1, S2);
  const float2 dacc = sub2(fma2(Bi, S1, mul2(splat2(-6.0f), b1)), S3);
  // finish_op
  const float2 B1 = add2(splat2(1.0f), xi);
  const float2 rs = make_float2(sfu_rsqrt(B1.x), sfu_rsqrt(B1.y));
  const float2 sv = mul2(B1, rs);
  const float2 den = add2(B1, sv);
  const float2 y = mul2(neg2(xi), make_float2(sfu_rcp(den.x), sfu_rcp(den.y)));
  const float2 N = fma2(splat2(ah), acc, mul2(splat2(beta), y));
  const float2 dN = fma2(splat2(ah), dacc, neg2(mul2(splat2(0.5f * beta), rs)));
  // newton_du, clamp, update
  const float2 r = sub2(N, fi);
  const float2 q = make_float2(sfu_rcp(dN.x), sfu_rcp(dN.y));
  float2 du = mul2(splat2(relax), mul2(neg2(r), q));
  du.x = fminf(fmaxf(du.x, -cap), cap);
  du.y = fminf(fmaxf(du.y, -cap), cap);
  return add2(di, du);
}

// Face sums of the operator and its derivative at cell (i,j,k) from global
// memory, with the cell's own u, x and E.
template <typename T, bool BG>
__device__ __forceinline__ void cell_sums(const Grid<T> &G, int i, int j, int k, long long c,
                                          T &di, T &xi, T &Ei, T &acc, T &dacc) {
  di = G.u[c];
  xi = G.x[c];
  Ei = BG ? (T)G.Ebg[c] : T(1);
  const T ubi = BG ? (T)G.ubg[c] : T(0);
  const T Bi = BG ? Ei + Ei * xi : T(1) + xi;
  OpAcc<T, BG> A(di, Ei, xi, Bi, ubi);
  const bool dir = G.bnd != nullptr;
  const long long sx = 1, sy = G.n0, sz = (long long)G.n0 * G.n1;
  auto nb = [&](long long cj) {
    A.reg(G.u[cj], G.x[cj], BG ? (T)G.ubg[cj] : T(0), BG ? (T)G.Ebg[cj] : T(1));
  };
  // -x, +x
  if (i > 0) nb(c - sx);
  else if (!dir) nb(c + (G.n0 - 1) * sx);
  else A.ghost(face_value(G, 0, i, j, k));
  if (i < G.n0 - 1) nb(c + sx);
  else if (!dir) nb(c - (G.n0 - 1) * sx);
  else A.ghost(face_value(G, 1, i, j, k));
  // -y, +y
  if (j > 0) nb(c - sy);
  else if (!dir) nb(c + (G.n1 - 1) * sy);
  else A.ghost(face_value(G, 2, i, j, k));
  if (j < G.n1 - 1) nb(c + sy);
  else if (!dir) nb(c - (G.n1 - 1) * sy);
  else A.ghost(face_value(G, 3, i, j, k));
  // -z, +z
  if (k > 0) nb(c - sz);
  else if (!dir) nb(c + (G.n2 - 1) * sz);
  else A.ghost(face_value(G, 4, i, j, k));
  if (k < G.n2 - 1) nb(c + sz);
  else if (!dir) nb(c - (G.n2 - 1) * sz);
  else A.ghost(face_value(G, 5, i, j, k));
  A.done(acc, dacc);
}

// A_i (or N_i) and its derivative at cell (i,j,k).
template <typename T, bool BG>
__device__ __forceinline__ void cell_eval(const Grid<T> &G, int i, int j, int k, long long c,
                                          T &N, T &dN) {
  T di, xi, Ei, acc, dacc;
  cell_sums<T, BG>(G, i, j, k, c, di, xi, Ei, acc, dacc);
  finish_op(xi, Ei, acc, dacc, G.ah, G.beta, BG, N, dN);
}

template <typename T>
__device__ __forceinline__ T rhs_at(const Grid<T> &G, long long c) {
  return G.f ? G.fs * (G.f[c] - G.fo) : T(0);
}

template <typename T, bool BG>
__device__ __forceinline__ void ngs_update(const Grid<T> &G, int i, int j, int k) {
  long long c = idx3(G, i, j, k);
  T di, xi, Ei, acc, dacc;
  cell_sums<T, BG>(G, i, j, k, c, di, xi, Ei, acc, dacc);
  const T unew = di + newton_from_sums<T, BG>(xi, Ei, acc, dacc, rhs_at(G, c), G.ah, G.beta,
                                              G.cap, G.relax);
  G.u[c] = unew;
  G.x[c] = m_expm1(unew);
}

// ---------------------------------------------------------------------------
// Threads per block of the one-thread-per-cell kernels without a block sum.
// FP64: the FP64 pipes bound them, and small blocks spread a small level over
// all SMs (32^3: 512 warps on 152 SMs).
template <typename T>
__host__ __device__ constexpr int cell_threads() {
  return sizeof(T) == 8 ? 64 : 256;
}

// One colour of a red-black Newton-Gauss-Seidel sweep; one thread per cell of
// that colour.  off[] maps blocks to grids (n0/2 * n1 * n2 threads per grid).
template <typename T, bool BG>
__global__ void k_smooth(const Grid<T> *grids, const int *off, int ngrid, int colour,
                         const int *active, int par) {
  int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<T> G = view(grids, g, par);
  if (!grid_active(active, G.field)) return;
  long long t = (long long)(blockIdx.x - off[g]) * blockDim.x + threadIdx.x;
  if (2 * t >= G.ncell) return;
  int i, j, k;
  cell_ijk(G, 2 * t, i, j, k);  // even cell of the pair
  i += (j + k + colour) & 1;
  ngs_update<T, BG>(G, i, j, k);
}

// Block-level (sum of squares, max |v|) partials, one pair per block.
template <int NT>
__device__ __forceinline__ void block_reduce2(double s, double m, double *out_s, double *out_m) {
  __shared__ double ss[NT / 32], sm[NT / 32];
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_down_sync(0xffffffffu, s, o);
    m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
  }
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    ss[w] = s;
    sm[w] = m;
  }
  __syncthreads();
  if (w == 0) {
    s = (l < NT / 32) ? ss[l] : 0.0;
    m = (l < NT / 32) ? sm[l] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      s += __shfl_down_sync(0xffffffffu, s, o);
      m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
    }
    if (l == 0) {
      *out_s = s;
      *out_m = m;
    }
  }
}

// Block-level (sum of squares, max |v|) from FP32 per-thread values, reduced in
// FP32 (relative error ~1e-6, ample for a stopping criterion) and written as
// FP64 once per block: FP64 arithmetic runs at 1/64 of the FP32 rate here.
template <int NT>
__device__ __forceinline__ void block_reduce2f(float s, float m, double *out_s, double *out_m) {
  __shared__ float ssf[NT / 32], smf[NT / 32];
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_down_sync(0xffffffffu, s, o);
    m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, o));
  }
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    ssf[w] = s;
    smf[w] = m;
  }
  __syncthreads();
  if (w == 0) {
    s = (l < NT / 32) ? ssf[l] : 0.0f;
    m = (l < NT / 32) ? smf[l] : 0.0f;
    for (int o = 16; o > 0; o >>= 1) {
      s += __shfl_down_sync(0xffffffffu, s, o);
      m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, o));
    }
    if (l == 0) {
      *out_s = (double)s;
      *out_m = (double)m;
    }
  }
}

// d = A(u) - f over every cell; optional output array and per-block partial
// norms (partial[2*block], partial[2*block+1]).  One thread per cell.
template <typename T, bool BG, int NT>
__global__ void __launch_bounds__(NT) k_residual(const Grid<T> *grids, const int *off, int ngrid,
                                                 T *const *dout, double *partial,
                                                 const int *active, int par) {
  int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<T> G = view(grids, g, par);
  float s = 0.0f, m = 0.0f;
  long long t = (long long)(blockIdx.x - off[g]) * NT + threadIdx.x;
  if (grid_active(active, G.field) && t < G.ncell) {
    int i, j, k;
    cell_ijk(G, t, i, j, k);
    T N, dN;
    cell_eval<T, BG>(G, i, j, k, t, N, dN);
    T d = N - rhs_at(G, t);
    if (dout && dout[g]) dout[g][t] = d;
    const float df_ = (float)d;
    s = df_ * df_;
    m = fabsf(df_);
  }
  if (partial) block_reduce2f<NT>(s, m, &partial[2 * blockIdx.x], &partial[2 * blockIdx.x + 1]);
}

// Per-grid sums of the block partials: out[2g] = sum of squares, out[2g+1] = max.
// Blocks past ngrid append pairs that are summed already.
__global__ void k_reduce_partials(const double *partial, const int *off, int ngrid, double *out,
                                  const double *done = nullptr) {
  int g = blockIdx.x;
  if (g >= ngrid) {
    if (done && threadIdx.x < 2) out[2 * g + threadIdx.x] = done[2 * (g - ngrid) + threadIdx.x];
    return;
  }
  double s = 0.0, m = 0.0;
  for (int b = off[g] + threadIdx.x; b < off[g + 1]; b += blockDim.x) {
    s += partial[2 * b];
    m = fmax(m, partial[2 * b + 1]);
  }
  block_reduce2<256>(s, m, &out[2 * g], &out[2 * g + 1]);
}

// First stage of the per-grid sums for long partial lists: block (c, g)
// reduces partials [off[g] + c CH, min(off[g] + (c + 1) CH, off[g + 1])) into
// tmp[2 (g nch + c)] (zeros when the range is empty); k_reduce_partials then
// sums each grid's nch entries (offsets g nch).
template <int CH>
__global__ void k_reduce_partials_chunks(const double *partial, const int *off, int nch,
                                         double *tmp) {
  const int g = blockIdx.y, c = blockIdx.x;
  const int b0 = off[g] + c * CH, b1 = min(b0 + CH, off[g + 1]);
  double s = 0.0, m = 0.0;
  for (int b = b0 + threadIdx.x; b < b1; b += blockDim.x) {
    s += partial[2 * b];
    m = fmax(m, partial[2 * b + 1]);
  }
  block_reduce2<256>(s, m, &tmp[2 * (g * nch + c)], &tmp[2 * (g * nch + c) + 1]);
}

// Second stage: out[2g] = sum, out[2g+1] = max of tmp[g nch .. (g+1) nch).
__global__ void k_reduce_chunks(const double *tmp, int nch, int ngrid, double *out) {
  const int g = blockIdx.x;
  if (g >= ngrid) return;
  double s = 0.0, m = 0.0;
  for (int c = threadIdx.x; c < nch; c += blockDim.x) {
    s += tmp[2 * (g * nch + c)];
    m = fmax(m, tmp[2 * (g * nch + c) + 1]);
  }
  block_reduce2<256>(s, m, &out[2 * g], &out[2 * g + 1]);
}

// Fused residual + restriction (Sec. V.B.2): for each coarse cell, the 8 fine
// children give  u^H = uR = mean(u^h),  x^H = expm1(u^H),  f^H <- mean(d^h)
// (the coarse operator is added by k_fas_rhs).  One thread per fine cell, the
// children of a coarse cell in eight neighbouring lanes; a block's 32 coarse
// cells are written by its first warp.  Optionally accumulates per-block
// (sum d^2, max |d|) of the fine residual.  (One thread per coarse cell left
// most SMs idle on small FP64 levels: 45 us at 32^3 against 8 us.)
template <typename T, bool BG>
__global__ void __launch_bounds__(256)
    k_resid_restrict(const Grid<T> *fine, const Grid<T> *coarse, const int *off, int ngrid,
                     const int *active, int fpar, int cpar, double *partial) {
  __shared__ T cu[32], cd[32];
  int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<T> F = view(fine, g, fpar);
  const Grid<T> C = view(coarse, g, cpar);
  const bool on = grid_active(active, F.field);
  const long long c0 = (long long)(blockIdx.x - off[g]) * 32;
  const long long t = c0 + (threadIdx.x >> 3);
  T d = T(0), u = T(0);
  if (on && t < C.ncell) {
    const int q = threadIdx.x & 7;
    int I, J, K;
    cell_ijk(C, t, I, J, K);
    const int i = 2 * I + (q & 1), j = 2 * J + ((q >> 1) & 1), k = 2 * K + (q >> 2);
    const long long c = idx3(F, i, j, k);
    T N, dN;
    cell_eval<T, BG>(F, i, j, k, c, N, dN);
    d = N - rhs_at(F, c);
    u = F.u[c];
  }
  const float df_ = (float)d;
  // even lanes add up u, odd lanes d (one addition per step for the two sums)
  const bool odd = threadIdx.x & 1;
  const T give = odd ? u : d;
  T s = (odd ? d : u) + __shfl_xor_sync(0xffffffffu, give, 1);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 4);
  if ((threadIdx.x & 7) == 0) cu[threadIdx.x >> 3] = s;
  if ((threadIdx.x & 7) == 1) cd[threadIdx.x >> 3] = s;
  __syncthreads();
  if (threadIdx.x < 32 && on && c0 + threadIdx.x < C.ncell) {
    const long long w = c0 + threadIdx.x;
    const T uh = cu[threadIdx.x] * T(0.125);
    C.uR[w] = uh;
    C.u[w] = uh;
    C.x[w] = m_expm1(uh);
    const_cast<T *>(C.f)[w] = cd[threadIdx.x] * T(0.125);
  }
  // fine-grid residual norm partials (the residual after pre-smoothing)
  if (partial)
    block_reduce2f<256>(df_ * df_, fabsf(df_), &partial[2 * blockIdx.x],
                        &partial[2 * blockIdx.x + 1]);
}

// f^H = A^H(R u^h) - R d^h, in place over the R d^h stored in f (fs = 1, fo = 0).
template <typename T, bool BG>
__global__ void k_fas_rhs(const Grid<T> *grids, const int *off, int ngrid, const int *active,
                          int par) {
  int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<T> G = view(grids, g, par);
  if (!grid_active(active, G.field)) return;
  long long t = (long long)(blockIdx.x - off[g]) * blockDim.x + threadIdx.x;
  if (t >= G.ncell) return;
  int i, j, k;
  cell_ijk(G, t, i, j, k);
  T N, dN;
  cell_eval<T, BG>(G, i, j, k, t, N, dN);
  T *f = const_cast<T *>(G.f);
  f[t] = N - f[t];
}

// Truncation-error estimate of Sec. V.B.2 on the coarse grid of a V-cycle
// level, tau = A^H(R u) - R A^h(u), after k_resid_restrict has put R u (and
// its x) into the coarse grid and R d = R(A^h(u) - f^h) into its f: then
// R A^h(u) = f^H + R f^h.  The density terms of the operator cancel between
// the two and are not part of A.  One thread per coarse cell; per-block
// partials (sum tau^2, max |tau|).
template <typename T>
__global__ void __launch_bounds__(256)
    k_tau(const Grid<T> *fine, const Grid<T> *coarse, const int *off, int ngrid, int fpar,
          int cpar, double *partial) {
  int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<T> F = view(fine, g, fpar);
  const Grid<T> C = view(coarse, g, cpar);
  float ss = 0.0f, mx = 0.0f;
  long long t = (long long)(blockIdx.x - off[g]) * blockDim.x + threadIdx.x;
  if (t < C.ncell) {
    int I, J, K;
    cell_ijk(C, t, I, J, K);
    T N, dN;
    cell_eval<T, false>(C, I, J, K, t, N, dN);
    T rf = T(0);
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int i = 2 * I + (q & 1), j = 2 * J + ((q >> 1) & 1), k = 2 * K + (q >> 2);
      rf += rhs_at(F, idx3(F, i, j, k));
    }
    const T tau = N - (C.f[t] + rf * T(0.125));
    const float tf = (float)tau;
    ss = tf * tf;
    mx = fabsf(tf);
  }
  block_reduce2f<256>(ss, mx, &partial[2 * blockIdx.x], &partial[2 * blockIdx.x + 1]);
}

// u^h += P (u^H - R u^h), trilinear 27/9/3/1 over 64 (Sec. V.A.3); x^h refreshed.
// One thread per coarse cell writes its 8 children: the correction
// e = u^H - R u^h of the 3x3x3 coarse neighbourhood is interpolated separably
// (weights 3/4 for the containing cell, 1/4 for the neighbour on the child's
// side, per axis; their products are the paper's 27/9/3/1 over 64).
// Patches: coarse neighbours outside the grid contribute 0.
template <typename T>
__global__ void __launch_bounds__(256) k_prolong(const Grid<T> *fine, const Grid<T> *coarse,
                                                 const int *off, int ngrid, const int *active,
                                                 int fpar, int cpar) {
  int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<T> &Fg = fine[g];
  const Grid<T> &Cg = coarse[g];
  if (!grid_active(active, Fg.field)) return;
  const int c0 = Cg.n0, c1 = Cg.n1, c2 = Cg.n2;
  long long t = (long long)(blockIdx.x - off[g]) * blockDim.x + threadIdx.x;
  if (t >= (long long)c0 * c1 * c2) return;
  const T *__restrict__ uH = cpar ? Cg.u2 : Cg.u;
  const T *__restrict__ uR = Cg.uR;
  T *__restrict__ uf = fpar ? Fg.u2 : Fg.u;
  T *__restrict__ xf = fpar ? Fg.x2 : Fg.x;
  const bool dir = Fg.bnd != nullptr;
  int I, J, K;
  cell_ijk(Cg, t, I, J, K);
  // e over the 3x3x3 neighbourhood, index [dz][dy][dx] with d = -1, 0, 1
  T e[3][3][3];
#pragma unroll
  for (int dz = 0; dz < 3; dz++) {
    int kk = K + dz - 1;
    bool vz = kk >= 0 && kk < c2;
    kk = kk < 0 ? kk + c2 : (kk >= c2 ? kk - c2 : kk);
#pragma unroll
    for (int dy = 0; dy < 3; dy++) {
      int jj = J + dy - 1;
      bool vy = jj >= 0 && jj < c1;
      jj = jj < 0 ? jj + c1 : (jj >= c1 ? jj - c1 : jj);
#pragma unroll
      for (int dx = 0; dx < 3; dx++) {
        int ii = I + dx - 1;
        bool vx = ii >= 0 && ii < c0;
        ii = ii < 0 ? ii + c0 : (ii >= c0 ? ii - c0 : ii);
        long long ci = ((long long)kk * c1 + jj) * c0 + ii;
        bool valid = !dir || (vx && vy && vz);
        e[dz][dy][dx] = valid ? uH[ci] - uR[ci] : T(0);
      }
    }
  }
  const T w3 = T(0.75), w1 = T(0.25);
  // along x: child a = 0 uses (dx = 1, 0), a = 1 uses (dx = 1, 2)
  T ex[2][3][3];
#pragma unroll
  for (int dz = 0; dz < 3; dz++)
#pragma unroll
    for (int dy = 0; dy < 3; dy++) {
      ex[0][dz][dy] = w3 * e[dz][dy][1] + w1 * e[dz][dy][0];
      ex[1][dz][dy] = w3 * e[dz][dy][1] + w1 * e[dz][dy][2];
    }
  T exy[2][2][3];
#pragma unroll
  for (int a = 0; a < 2; a++)
#pragma unroll
    for (int dz = 0; dz < 3; dz++) {
      exy[a][0][dz] = w3 * ex[a][dz][1] + w1 * ex[a][dz][0];
      exy[a][1][dz] = w3 * ex[a][dz][1] + w1 * ex[a][dz][2];
    }
  const int f0 = Fg.n0, f1 = Fg.n1;
#pragma unroll
  for (int cz = 0; cz < 2; cz++)
#pragma unroll
    for (int cy = 0; cy < 2; cy++) {
      const long long fi = ((long long)(2 * K + cz) * f1 + (2 * J + cy)) * f0 + 2 * I;
#pragma unroll
      for (int a = 0; a < 2; a++) {
        const T corr = w3 * exy[a][cy][1] + w1 * exy[a][cy][cz == 0 ? 0 : 2];
        const T un = uf[fi + a] + corr;
        uf[fi + a] = un;
        xf[fi + a] = m_expm1(un);
      }
    }
}

// Tiled FP32 prolongation and correction (same interpolation as k_prolong,
// evaluated in the order z, y, x): a block owns a 64 x 16 fine tile (32 x 8
// coarse cells) and a chunk of kc coarse planes.  The correction
// e = u^H - R u^h of the coarse tile plus a one-cell halo is staged in shared
// memory for planes K-1, K, K+1 (ring of three); for each of the fine planes
// 2K and 2K+1 the z-interpolated coarse plane is formed once in shared memory,
// and each thread corrects its fine x-pairs (y- then x-interpolation,
// weights 3/4 and 1/4 per axis) with 8-byte loads and stores, refreshing
// x = expm1(u).  Patches: coarse cells outside the grid contribute 0.
constexpr int kPlTX = 64, kPlTY = 16;
template <bool DIR, bool BG>
__global__ void __launch_bounds__(256)
    k_prolong_tiled(const Grid<float> *fine, const Grid<float> *coarse, const int *off, int ngrid,
                    int kc, const int *active, int fpar, int cpar) {
  constexpr int CX = kPlTX / 2 + 2, CY = kPlTY / 2 + 2, CP = CX * CY;
  constexpr int NQ = (CP + 255) / 256;
  __shared__ float se[3][CP];
  __shared__ float sz[CP];
  const int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<float> &Fg = fine[g];
  const Grid<float> &Cg = coarse[g];
  if (!grid_active(active, Fg.field)) return;
  const int n0 = Fg.n0, n1 = Fg.n1;
  const int c0 = Cg.n0, c1 = Cg.n1, c2 = Cg.n2;
  const float *__restrict__ uH = cpar ? Cg.u2 : Cg.u;
  const float *__restrict__ uR = Cg.uR;
  float *__restrict__ uf = fpar ? Fg.u2 : Fg.u;
  float *__restrict__ xf = fpar ? Fg.x2 : Fg.x;
  const int ntx = (n0 + kPlTX - 1) / kPlTX, nty = (n1 + kPlTY - 1) / kPlTY;
  int b = blockIdx.x - off[g];
  const int X0 = (b % ntx) * kPlTX;
  b /= ntx;
  const int Y0 = (b % nty) * kPlTY;
  b /= nty;
  const int K0 = b * kc, K1 = min(K0 + kc, c2);
  // coarse staging table: entry q = threadIdx.x + k 256 of the CX x CY tile
  int qoff[NQ];
  bool qok[NQ];
#pragma unroll
  for (int k = 0; k < NQ; k++) {
    const int q = threadIdx.x + k * 256;
    qoff[k] = 0;
    qok[k] = false;
    if (q < CP) {
      int I = X0 / 2 - 1 + q % CX, J = Y0 / 2 - 1 + q / CX;
      if (DIR) {
        qok[k] = I >= 0 && I < c0 && J >= 0 && J < c1;
      } else {
        I = wrapmod(I, c0);
        J = wrapmod(J, c1);
        qok[k] = true;
      }
      qoff[k] = J * c0 + I;
    }
  }
  const long long cplane = (long long)c0 * c1;
  // wrapped index of the next coarse plane to stage
  int kw = DIR ? K0 - 1 : wrapmod(K0 - 1, c2);
  auto stage = [&](int slot, int K) {
    const bool vz = !DIR || (K >= 0 && K < c2);
    const long long zo = (long long)kw * cplane;
#pragma unroll
    for (int k = 0; k < NQ; k++) {
      const int q = threadIdx.x + k * 256;
      if (q >= CP) continue;
      float e = 0.0f;
      if (qok[k] && vz) {
        const long long i = zo + qoff[k];
        e = uH[i] - uR[i];
      }
      se[slot][q] = e;
    }
    kw = DIR ? kw + 1 : (kw + 1 == c2 ? 0 : kw + 1);
  };
  const int lane = threadIdx.x & 31, r0 = threadIdx.x >> 5;  // pair, first row
  const long long fplane = (long long)n0 * n1;
  const float w3 = 0.75f, w1 = 0.25f;
  stage(0, K0 - 1);
  stage(1, K0);
  int sm = 0, sc = 1, sp = 2;  // ring slots of planes K-1, K, K+1
  for (int K = K0; K < K1; K++) {
    stage(sp, K + 1);
    __syncthreads();
#pragma unroll
    for (int cz = 0; cz < 2; cz++) {
      const int so = cz ? sp : sm;
      for (int q = threadIdx.x; q < CP; q += 256) sz[q] = w3 * se[sc][q] + w1 * se[so][q];
      __syncthreads();
      const int k = 2 * K + cz;
      const int fx = X0 + 2 * lane;
#pragma unroll
      for (int rr = 0; rr < 2; rr++) {
        const int row = r0 + 8 * rr;
        const int j = Y0 + row;
        if (j >= n1 || fx >= n0) continue;
        const int jy = row / 2 + 1, jy2 = (row & 1) ? jy + 1 : jy - 1;
        const int ix = lane + 1;
        const float *za = sz + jy * CX, *zb = sz + jy2 * CX;
        const float em = w3 * za[ix - 1] + w1 * zb[ix - 1];
        const float e0 = w3 * za[ix] + w1 * zb[ix];
        const float ep = w3 * za[ix + 1] + w1 * zb[ix + 1];
        const long long fi = (long long)k * fplane + (long long)j * n0 + fx;
        const float2 u = *reinterpret_cast<const float2 *>(uf + fi);
        const float un0 = u.x + (w3 * e0 + w1 * em);
        const float un1 = u.y + (w3 * e0 + w1 * ep);
        *reinterpret_cast<float2 *>(uf + fi) = make_float2(un0, un1);
        // (x as the sweeps of this form compute it)
        *reinterpret_cast<float2 *>(xf + fi) =
            BG || DIR ? make_float2(m_expm1(un0), m_expm1(un1))
                      : m_expm1_full2(make_float2(un0, un1));
      }
      __syncthreads();
    }
    const int t = sm;
    sm = sc;
    sc = sp;
    sp = t;
  }
}

// Block sum of two values (all threads get the result).
template <int NT, typename A>
__device__ __forceinline__ void block_sum2(A a, A b, A &ra, A &rb) {
  __shared__ A sa[NT / 32], sb[NT / 32];
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) {
    sa[w] = a;
    sb[w] = b;
  }
  __syncthreads();
  A ta = A(0), tb = A(0);
  for (int q = 0; q < NT / 32; q++) {
    ta += sa[q];
    tb += sb[q];
  }
  ra = ta;
  rb = tb;
}

// Block sum of one value per thread into *out (shared), written by thread 0.
template <int NT, typename A>
__device__ __forceinline__ void block_sum1(A a, A *out) {
  __shared__ A sa[NT / 32];
  for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sa[w] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    A t = A(0);
    for (int q = 0; q < NT / 32; q++) t += sa[q];
    *out = t;
  }
}

// Coarsest level: one block per grid, Newton-Gauss-Seidel sweeps until
// rms <= max(rel * rms0, abs_floor) (at least one sweep, at most maxit).
// stop_on_stall also stops when a sweep does not lower the rms.
// meanfix (periodic grids): after every sweep, one Newton step on a constant
// shift c of the whole grid.  On a periodic grid the flux terms telescope, so
// sum_i (N_i - f_i) depends on c only through the mass term, whose derivative
// is -(beta/2) sum_i F_i e^{-d_i/2}; the step removes the error of the
// constant mode, which plain relaxation damps by only ~beta/(12 alpha) per
// sweep when the Laplacian dominates (stiff coarsest problems).
template <typename T, bool BG, int NT>
__global__ void __launch_bounds__(NT) k_coarsest(const Grid<T> *grids, int ngrid, double rel,
                                                 double abs_floor, int maxit, int stop_on_stall,
                                                 const int *active, int par, int meanfix) {
  int g = blockIdx.x;
  if (g >= ngrid) return;
  Grid<T> G = view(grids, g, par);
  if (!grid_active(active, G.field)) return;
  // sums in the precision of the grid: FP64 arithmetic runs at 1/64 of the
  // FP32 rate here, and the FP32 levels' stopping test needs no more
  using A = typename std::conditional<sizeof(T) == 4, float, double>::type;
  __shared__ A red_s;
  __shared__ int stop;
  const long long n = G.ncell;
  // a grid of up to 16 KB per array is relaxed in shared memory (u and its
  // x cache copied in and back; the same updates in the same order)
  constexpr int CAPN = 16384 / (int)sizeof(T);
  __shared__ T cs_u[CAPN], cs_x[CAPN];
  T *const gu = G.u;
  T *const gx = G.x;
  const bool local = n <= CAPN;
  if (local) {
    for (long long t = threadIdx.x; t < n; t += NT) {
      cs_u[t] = gu[t];
      cs_x[t] = gx[t];
    }
    __syncthreads();
    G.u = cs_u;
    G.x = cs_x;
  }
  const int hx = G.n0 >> 1;
  const long long nh = (long long)hx * G.n1 * G.n2;
  const bool shift = meanfix && G.bnd == nullptr;
  A thr = A(0), prev = A(0);
  for (int it = -1; it < maxit; it++) {
    if (it >= 0) {
      for (int colour = 0; colour < 2; colour++) {
        for (long long t = threadIdx.x; t < nh; t += NT) {
          int i, j, k;
          cell_ijk(G, 2 * t, i, j, k);
          ngs_update<T, BG>(G, i + ((j + k + colour) & 1), j, k);
        }
        __syncthreads();
      }
      if (shift) {
        A S = A(0), D = A(0);
        for (long long t = threadIdx.x; t < n; t += NT) {
          int i, j, k;
          cell_ijk(G, t, i, j, k);
          T N, dN;
          cell_eval<T, BG>(G, i, j, k, t, N, dN);
          S += (A)(N - rhs_at(G, t));
          const T Ei = BG ? (T)G.Ebg[t] : T(1);
          const T F = BG ? m_rsqrt(Ei) : T(1);
          D += A(0.5) * (A)G.beta * (A)(F * m_rsqrt(T(1) + G.x[t]));
        }
        A St, Dt;
        block_sum2<NT, A>(S, D, St, Dt);
        A c = Dt > A(0) ? St / Dt : A(0);
        const A cap = (A)G.cap;
        c = c > cap ? cap : (c < -cap ? -cap : c);
        __syncthreads();
        for (long long t = threadIdx.x; t < n; t += NT) {
          const T un = G.u[t] + (T)c;
          G.u[t] = un;
          G.x[t] = m_expm1(un);
        }
        __syncthreads();
      }
    }
    A s = A(0);
    for (long long t = threadIdx.x; t < n; t += NT) {
      int i, j, k;
      cell_ijk(G, t, i, j, k);
      T N, dN;
      cell_eval<T, BG>(G, i, j, k, t, N, dN);
      const A d = (A)(N - rhs_at(G, t));
      s += d * d;
    }
    block_sum1<NT, A>(s, &red_s);
    __syncthreads();
    if (threadIdx.x == 0) {
      const A rms = sqrt(red_s / (A)n);
      int st = 0;
      if (it < 0) {
        thr = fmax((A)rel * rms, (A)abs_floor);
        if (rms <= thr) st = 1;
      } else {
        if (rms <= thr) st = 1;
        if (stop_on_stall && rms >= prev) st = 1;
      }
      prev = rms;
      stop = st;
    }
    __syncthreads();
    if (stop) break;
  }
  if (local) {
    __syncthreads();
    for (long long t = threadIdx.x; t < n; t += NT) {
      gu[t] = cs_u[t];
      gx[t] = cs_x[t];
    }
  }
}

// Generic 8-child average (full weighting on cell-centred grids).
template <typename T>
__global__ void k_restrict_avg(const T *fine, int nf0, int nf1, int nf2, T *coarse) {
  int nc0 = nf0 >> 1, nc1 = nf1 >> 1, nc2 = nf2 >> 1;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)nc0 * nc1 * nc2) return;
  int I = (int)(t % nc0);
  long long r = t / nc0;
  int J = (int)(r % nc1);
  int K = (int)(r / nc1);
  T s = T(0);
#pragma unroll
  for (int c = 0; c < 8; c++) {
    int i = 2 * I + (c & 1), j = 2 * J + ((c >> 1) & 1), k = 2 * K + (c >> 2);
    s += fine[((long long)k * nf1 + j) * nf0 + i];
  }
  coarse[t] = s * T(0.125);
}

// Background of the correction form on a level from the next finer one: mean
// of the 8 children and its exponential, for every active grid of the set.
__global__ void __launch_bounds__(256)
    k_bg_restrict(const Grid<float> *fine, const Grid<float> *coarse, const int *off, int ngrid,
                  const int *active) {
  const int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<float> &F = fine[g];
  const Grid<float> &C = coarse[g];
  if (!grid_active(active, F.field)) return;
  const long long t = (long long)(blockIdx.x - off[g]) * 256 + threadIdx.x;
  if (t >= C.ncell) return;
  int I, J, K;
  cell_ijk(C, t, I, J, K);
  float s = 0.0f;
#pragma unroll
  for (int q = 0; q < 8; q++)
    s += F.ubg[idx3(F, 2 * I + (q & 1), 2 * J + ((q >> 1) & 1), 2 * K + (q >> 2))];
  const float ub = s * 0.125f;
  const_cast<float *>(C.ubg)[t] = ub;
  const_cast<float *>(C.Ebg)[t] = expf(ub);
}

// ---------------------------------------------------------------------------
// Tiled FP32 smoother with temporal blocking: S full red-black sweeps per pass.
//
// A block owns a TX x TY tile of one grid and a chunk of zc planes; it marches
// along z with a ring of 2S+2 planes (tile plus a halo of 2S cells in x and y)
// in shared memory.  At the step that loads plane p, stage q (q = 0 .. 2S-1,
// colour q & 1: red first) updates plane p-1-q on the tile grown by 2S-1-q
// cells, so that plane p-2S is final and its tile cells are written out.
// Halo cells are updated redundantly by neighbouring blocks from identical
// inputs; a pass reads the current buffer and writes the other one (blocks
// load their halos from the unmodified input), which makes the result equal to
// S sweeps of k_smooth.  x = expm1(u) is recomputed from u on load and written
// in place for the kernels that follow.
template <int S, int TX, int TY>
struct TileCfg {
  static constexpr int H = 2 * S;                   // halo
  static constexpr int LX = TX + 2 * H, LY = TY + 2 * H, PL = LX * LY, NS = 2 * S + 2;
  static constexpr int PX = LX / 2;                 // x-pairs per row
  static constexpr int RPT = 2;                     // rows per thread (independent updates)
  static constexpr int NT = PX * LY / RPT;          // threads per block
  static constexpr size_t smem(bool bg) { return (size_t)NS * PL * sizeof(float) * (bg ? 5 : 3); }
  static_assert(LY % RPT == 0, "rows must split evenly over threads");
};

// ---------------------------------------------------------------------------
// Tiled FP32 smoother with temporal blocking: S full red-black sweeps per pass.
//
// A block owns a TX x TY tile of one grid and a chunk of zc planes; it marches
// along z with a ring of 2S+2 planes (tile plus a halo of 2S cells in x and y)
// in shared memory.  At the step that loads plane p, stage q (q = 0 .. 2S-1,
// colour q & 1: red first) updates plane p-1-q on the tile grown by 2S-1-q
// cells, so that plane p-2S is final and its tile cells are written out.
// Halo cells are updated redundantly by neighbouring blocks from identical
// inputs; a pass reads the current buffer and writes the other one (blocks
// load their halos from the unmodified input), which makes the result equal to
// S sweeps of k_smooth.  The x = expm1(u) cache ping-pongs with u.
//
// Each thread owns one x-pair in each of RPT rows (LY/RPT rows apart) for the
// whole pass: it loads and stores its pairs with 8-byte accesses (x-pairs
// start at even x, and n0 is even, so a pair never straddles the periodic
// seam), and at every stage it updates, in each of its rows, the one cell of
// its pair that has the stage's colour if that cell lies in the stage's
// region; the RPT updates are independent, which gives the scheduler
// instruction-level parallelism.  The right-hand side is kept in shared memory
// with the plane.  The global loads of plane p+1 are
// issued into registers before the stages of step p and stored to shared
// memory after them.
template <bool BG, bool DIR, int S, int TX, int TY>
__global__ void __launch_bounds__(TileCfg<S, TX, TY>::NT)
    k_smooth_tiled(const Grid<float> *grids, const int *off, int ngrid, int zc, const int *active,
                   int par) {
  using C = TileCfg<S, TX, TY>;
  constexpr int H = C::H, LX = C::LX, LY = C::LY, PL = C::PL, NS = C::NS, PX = C::PX;
  constexpr int RPT = C::RPT;
  extern __shared__ float smem[];
  float *sd = smem;
  float *sx = smem + NS * PL;
  float *sf = smem + 2 * NS * PL;
  float *sub = smem + 3 * NS * PL;
  float *sE = smem + 4 * NS * PL;
  const int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<float> &Gg = grids[g];
  if (!grid_active(active, Gg.field)) return;
  const float *__restrict__ uin = par ? Gg.u2 : Gg.u;
  float *__restrict__ uout = par ? Gg.u : Gg.u2;
  const float *__restrict__ xin = par ? Gg.x2 : Gg.x;
  float *__restrict__ xout = par ? Gg.x : Gg.x2;
  const float *__restrict__ fin = Gg.f;
  const float *__restrict__ ubin = Gg.ubg;
  const float *__restrict__ Ein = Gg.Ebg;
  const float fs = Gg.fs, fo = Gg.fo, ah = Gg.ah, beta = Gg.beta, cap = Gg.cap,
              relax = Gg.relax;
  const int n0 = Gg.n0, n1 = Gg.n1, n2 = Gg.n2;
  constexpr bool dir = DIR;  // patch (Dirichlet faces) or periodic grid
  const int ntx = (n0 + TX - 1) / TX, nty = (n1 + TY - 1) / TY;
  int b = blockIdx.x - off[g];
  const int X0 = (b % ntx) * TX;
  b /= ntx;
  const int Y0 = (b % nty) * TY;
  b /= nty;
  const int Z0 = b * zc;
  const int Z1 = min(Z0 + zc, n2);

  const int ly0 = threadIdx.x / PX;
  const int lx0 = 2 * (threadIdx.x - ly0 * PX);
  const int gx0 = X0 - H + lx0;
  int gxw0;
  if (dir)
    gxw0 = (gx0 < 0 || gx0 >= n0) ? -1 : gx0;
  else
    gxw0 = wrapmod(gx0, n0);
  int ly[RPT], gy[RPT], gyw[RPT], rowo[RPT];
  bool mine[RPT], writer[RPT];
#pragma unroll
  for (int r = 0; r < RPT; r++) {
    ly[r] = ly0 + r * (LY / RPT);
    gy[r] = Y0 - H + ly[r];
    if (dir)
      gyw[r] = (gy[r] < 0 || gy[r] >= n1) ? -1 : gy[r];
    else
      gyw[r] = wrapmod(gy[r], n1);
    mine[r] = gyw[r] >= 0 && gxw0 >= 0;
    rowo[r] = ly[r] * LX + lx0;
    writer[r] = mine[r] && ly[r] >= H && ly[r] < H + TY && lx0 >= H && lx0 < H + TX &&
                gx0 < n0 && gy[r] < n1;
  }

  float2 pd[RPT], px[RPT], pf[RPT], pu[RPT], pE[RPT];
#pragma unroll
  for (int r = 0; r < RPT; r++) {
    pd[r] = make_float2(0.f, 0.f);
    px[r] = pd[r];
    pf[r] = pd[r];
    pu[r] = pd[r];
    pE[r] = make_float2(1.f, 1.f);
  }
  auto fetch = [&](int p) {
    if (dir && (p < 0 || p >= n2)) return;
    const long long zo = (long long)wrapmod(p, n2) * n1;
#pragma unroll
    for (int r = 0; r < RPT; r++) {
      if (!mine[r]) continue;
      const long long gi = (zo + gyw[r]) * n0 + gxw0;
      pd[r] = *reinterpret_cast<const float2 *>(uin + gi);
      px[r] = *reinterpret_cast<const float2 *>(xin + gi);
      if (fin) pf[r] = *reinterpret_cast<const float2 *>(fin + gi);  // scaled at commit
      if (BG) {
        pu[r] = *reinterpret_cast<const float2 *>(ubin + gi);
        pE[r] = *reinterpret_cast<const float2 *>(Ein + gi);
      }
    }
  };
  auto commit = [&](int p) {
    const int base = wrapmod(p, NS) * PL;
#pragma unroll
    for (int r = 0; r < RPT; r++) {
      const int o = base + rowo[r];
      sd[o] = pd[r].x;
      sd[o + 1] = pd[r].y;
      sx[o] = px[r].x;
      sx[o + 1] = px[r].y;
      sf[o] = fin ? fs * (pf[r].x - fo) : 0.0f;
      sf[o + 1] = fin ? fs * (pf[r].y - fo) : 0.0f;
      if (BG) {
        sub[o] = pu[r].x;
        sub[o + 1] = pu[r].y;
        sE[o] = pE[r].x;
        sE[o + 1] = pE[r].y;
      }
    }
  };
  auto stage = [&](int p, int q) {
    const int m = p - 1 - q;
    const int R = 2 * S - 1 - q;
    const int colour = q & 1;
    if (m < Z0 - R || m >= Z1 + R || (dir && (m < 0 || m >= n2))) return;
    const int sl = wrapmod(m, NS), slm = wrapmod(m - 1, NS), slp = wrapmod(m + 1, NS);
#pragma unroll
    for (int r = 0; r < RPT; r++) {
      const int par01 = (X0 - H + gy[r] + m + colour) & 1;
      const int lx = lx0 + par01;
      if (!mine[r] || ly[r] < H - R || ly[r] >= H + TY + R || lx < H - R || lx >= H + TX + R)
        continue;
      const int li = rowo[r] + par01;
      const int o = sl * PL + li;
      const float di = sd[o], xi = sx[o];
      const float Ei = BG ? sE[o] : 1.0f;
      const float ubi = BG ? sub[o] : 0.0f;
      const float Bi = BG ? Ei + Ei * xi : 1.0f + xi;
      OpAcc<float, BG> A(di, Ei, xi, Bi, ubi);
      const int gxw = gxw0 + par01, gyr = gyw[r];
#define FR_NB(OFF) A.reg(sd[OFF], sx[OFF], BG ? sub[OFF] : 0.0f, BG ? sE[OFF] : 1.0f)
      if (dir && gxw == 0)
        A.ghost(face_value(Gg, 0, gxw, gyr, m));
      else
        FR_NB(o - 1);
      if (dir && gxw == n0 - 1)
        A.ghost(face_value(Gg, 1, gxw, gyr, m));
      else
        FR_NB(o + 1);
      if (dir && gyr == 0)
        A.ghost(face_value(Gg, 2, gxw, gyr, m));
      else
        FR_NB(o - LX);
      if (dir && gyr == n1 - 1)
        A.ghost(face_value(Gg, 3, gxw, gyr, m));
      else
        FR_NB(o + LX);
      if (dir && m == 0)
        A.ghost(face_value(Gg, 4, gxw, gyr, m));
      else
        FR_NB(slm * PL + li);
      if (dir && m == n2 - 1)
        A.ghost(face_value(Gg, 5, gxw, gyr, m));
      else
        FR_NB(slp * PL + li);
#undef FR_NB
      float acc, dacc;
      A.done(acc, dacc);
      float N, dN;
      finish_op(xi, Ei, acc, dacc, ah, beta, BG, N, dN);
      float du = newton_du(N, sf[o], dN, relax);
      du = fminf(fmaxf(du, -cap), cap);
      const float dn = di + du;
      sd[o] = dn;
      sx[o] = m_expm1(dn);
    }
  };

  fetch(Z0 - H);
  commit(Z0 - H);
  __syncthreads();
  for (int p = Z0 - H; p < Z1 + H; p++) {
    const bool more = p + 1 < Z1 + H;
    if (more) fetch(p + 1);
#pragma unroll
    for (int q = 0; q < 2 * S; q++) {
      stage(p, q);
      __syncthreads();
    }
    const int w = p - H;
    if (w >= Z0 && w < Z1) {
      const int base = wrapmod(w, NS) * PL;
#pragma unroll
      for (int r = 0; r < RPT; r++) {
        if (!writer[r]) continue;
        const int o = base + rowo[r];
        const long long gi = ((long long)w * n1 + gy[r]) * n0 + gx0;
        *reinterpret_cast<float2 *>(uout + gi) = make_float2(sd[o], sd[o + 1]);
        *reinterpret_cast<float2 *>(xout + gi) = make_float2(sx[o], sx[o + 1]);
      }
    }
    if (more) commit(p + 1);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Tiled FP32 smoother, one full red-black sweep per pass, rows of the tile
// distributed over warps.
//
// Same schedule as k_smooth_tiled with S = 1: a block owns a 64 x TY tile of
// one grid and an even number zc of planes and marches along z.  At the step
// that brings in plane p it updates the red cells of plane p-1 on the tile
// grown by one cell, then the black cells of plane p-2 on the tile, and
// writes plane p-2 out; the halo of two cells is loaded from the input buffer
// and the result goes to the other buffer, so the pass equals one sweep of
// k_smooth.  What differs is the layout and the work mapping:
//  * each plane is stored split by colour.  The six neighbours of a cell have
//    the other colour, so for the colour-c cell of x-pair e they are entries
//    e and e -+ 1 (x), e -+ PX (y) of the other colour's array, and entry e of
//    it in planes m -+ 1 (z); u and x = expm1(u) are interleaved, so each
//    neighbour is one 8-byte shared-memory access, stride-1 across a warp;
//  * a warp updates whole rows of pairs (lane = pair), so the position of the
//    colour-c cell inside the pair is the same for the whole warp, and only
//    the one extra cell per row of the grown red region (at the left or right
//    end of the row) is handled by two warps as a separate column task;
//  * the global loads of a plane go through fixed per-thread tables (row
//    offset, flags) built once, and the next plane's wrapped offset advances
//    by one plane per step.
template <int TY>
struct RBCfg {
  static constexpr int TX = 64, H = 2;
  static constexpr int LX = TX + 2 * H, LY = TY + 2 * H, PX = LX / 2, PP = PX * LY;
  static constexpr int NW = TY / 2, NT = 32 * NW;  // warps, threads
  static constexpr int NLD = (PP + NT - 1) / NT;   // plane-load rounds per thread
  // ring slots of (u, x) [and (ub, E)]; the right-hand side is kept per
  // colour: a red half-plane is read one step after it is loaded, a black one
  // two steps after, so two red and three black half-slots suffice
  static constexpr int NS = 4, NFR = 2, NFB = 3;
  static constexpr int NE = TY + 2;                // edge cells of the red region
  static constexpr size_t smem(bool bg) {
    return (size_t)NS * 2 * PP * sizeof(float2) * (bg ? 2 : 1) +
           (size_t)(NFR + NFB) * PP * sizeof(float);
  }
  // resident blocks per SM that shared memory allows, at most 3 (a fourth
  // block of 256 threads caps the registers at 64 per thread: measured slower)
  static constexpr int minb(bool bg) {
    const int bysm = (int)(228 * 1024 / (smem(bg) + 1024));
    const int byth = 1024 / NT < 3 ? 1024 / NT : 3;
    return bysm < 1 ? 1 : (bysm < byth ? bysm : byth);
  }
  static_assert(TY % 4 == 0 && NW >= 4 && NE <= 64, "tile height");
};

template <bool BG, bool DIR, int TY>
__global__ void __launch_bounds__(RBCfg<TY>::NT, RBCfg<TY>::minb(BG))
    k_smooth_rb(const Grid<float> *grids, const int *off, int ngrid, int zc, const int *active,
                int par) {
  using C = RBCfg<TY>;
  constexpr int TX = C::TX, H = C::H, PX = C::PX, PP = C::PP, NW = C::NW, NT = C::NT;
  constexpr int NLD = C::NLD, NS = C::NS, NFR = C::NFR, NFB = C::NFB;
  extern __shared__ float4 smem_rb[];
  // plain form: (u, x) per cell; correction form: (u, x, ub, E) per cell, so a
  // neighbour is one 16-byte access (half the shared-memory instructions)
  float2 *sux = reinterpret_cast<float2 *>(smem_rb);  // [NS][2][PP] (plain)
  float4 *s4 = smem_rb;                               // [NS][2][PP] (correction form)
  // right-hand side: red half-slots [NFR][PP], then black half-slots [NFB][PP]
  float *sfv = reinterpret_cast<float *>(sux + NS * 2 * PP * (BG ? 2 : 1));
  // cell e of a slot/colour offset: (u, x, ub, E); ub = 0, E = 1 in the plain form
  auto cell = [&](int i) -> float4 {
    if (BG) return s4[i];
    const float2 v = sux[i];
    return make_float4(v.x, v.y, 0.f, 1.f);
  };
  auto put_ux = [&](int i, float u, float x) {
    if (BG)
      *reinterpret_cast<float2 *>(&s4[i]) = make_float2(u, x);
    else
      sux[i] = make_float2(u, x);
  };
  const int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<float> &Gg = grids[g];
  if (!grid_active(active, Gg.field)) return;
  const float *__restrict__ uin = par ? Gg.u2 : Gg.u;
  float *__restrict__ uout = par ? Gg.u : Gg.u2;
  const float *__restrict__ xin = par ? Gg.x2 : Gg.x;
  float *__restrict__ xout = par ? Gg.x : Gg.x2;
  const float *__restrict__ fin = Gg.f;
  const float *__restrict__ ubin = Gg.ubg;
  const float *__restrict__ Ein = Gg.Ebg;
  const float fs = Gg.fs, fo = Gg.fo, ah = Gg.ah, beta = Gg.beta, cap = Gg.cap,
              relax = Gg.relax;
  const int n0 = Gg.n0, n1 = Gg.n1, n2 = Gg.n2;
  const int ntx = (n0 + TX - 1) / TX, nty = (n1 + TY - 1) / TY;
  int b = blockIdx.x - off[g];
  const int X0 = (b % ntx) * TX;
  b /= ntx;
  const int Y0 = (b % nty) * TY;
  b /= nty;
  const int Z0 = b * zc;  // zc is even, so plane p has the parity of its step
  const int Z1 = min(Z0 + zc, n2);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long plane = (long long)n0 * n1;

  // plane-load tables: pair q = threadIdx.x + k NT of the (TX + 4) x (TY + 4) tile
  int roff[NLD];
  unsigned ldf[NLD];  // bit 0: load, bit 1: write out, bit 2: parity of the row
#pragma unroll
  for (int k = 0; k < NLD; k++) {
    const int q = threadIdx.x + k * NT;
    roff[k] = 0;
    ldf[k] = 0;
    if (q < PP) {
      const int ly = q / PX, px = q - (q / PX) * PX;
      const int gx = X0 - H + 2 * px, gy = Y0 - H + ly;
      bool ok;
      int gxw, gyw;
      if (DIR) {
        ok = gx >= 0 && gx < n0 && gy >= 0 && gy < n1;
        gxw = gx;
        gyw = gy;
      } else {
        ok = true;
        gxw = wrapmod(gx, n0);
        gyw = wrapmod(gy, n1);
      }
      const bool wr = ok && ly >= H && ly < H + TY && px >= 1 && px < PX - 1 && gx < n0 &&
                      gy < n1;
      roff[k] = ok ? gyw * n0 + gxw : 0;
      ldf[k] = (ok ? 1u : 0u) | (wr ? 2u : 0u) | ((unsigned)(ly & 1) << 2);
    }
  }
  float2 pd[NLD], pq[NLD], pf[NLD], pu[NLD], pE[NLD];
#pragma unroll
  for (int k = 0; k < NLD; k++) {
    pd[k] = make_float2(0.f, 0.f);
    pq[k] = pd[k];
    pf[k] = pd[k];
    pu[k] = pd[k];
    pE[k] = make_float2(1.f, 1.f);
  }
  auto fetch = [&](long long zoff) {
#pragma unroll
    for (int k = 0; k < NLD; k++) {
      if (!(ldf[k] & 1u)) continue;
      const long long gi = zoff + roff[k];
      pd[k] = *reinterpret_cast<const float2 *>(uin + gi);
      pq[k] = *reinterpret_cast<const float2 *>(xin + gi);
      // raw values: arithmetic on them here would wait for the load
      if (fin) pf[k] = *reinterpret_cast<const float2 *>(fin + gi);
      if (BG) {
        pu[k] = *reinterpret_cast<const float2 *>(ubin + gi);
        pE[k] = *reinterpret_cast<const float2 *>(Ein + gi);
      }
    }
  };
  // plane of parity pb into (u, x) slot offset so and the f half-slot offsets
  // fr (red) and fb (black); the even-x cell of a pair has colour (y + z) & 1
  auto commit = [&](int pb, int so, int fr, int fb) {
#pragma unroll
    for (int k = 0; k < NLD; k++) {
      const int q = threadIdx.x + k * NT;
      if (q >= PP) continue;
      const int c0 = (int)((ldf[k] >> 2) & 1u) ^ pb;
      const int i0 = so + c0 * PP + q, i1 = so + (c0 ^ 1) * PP + q;
      if (BG) {
        s4[i0] = make_float4(pd[k].x, pq[k].x, pu[k].x, pE[k].x);
        s4[i1] = make_float4(pd[k].y, pq[k].y, pu[k].y, pE[k].y);
      } else {
        sux[i0] = make_float2(pd[k].x, pq[k].x);
        sux[i1] = make_float2(pd[k].y, pq[k].y);
      }
      sfv[(c0 ? fb : fr) + q] = fin ? fs * (pf[k].x - fo) : 0.0f;
      sfv[(c0 ? fr : fb) + q] = fin ? fs * (pf[k].y - fo) : 0.0f;
    }
  };
  // Newton update of the colour-Q cell of pair (ly, px) of plane m; s is its x
  // position in the pair; oc, om, op are the (u, x) slot offsets of planes m,
  // m - 1, m + 1 (colour Q's array at oc + Q PP), ofq the f offset.  Split in
  // three: gather (the shared-memory reads), compute (registers and, on patch
  // faces, the boundary values) and store, so that two independent updates
  // can read all their operands before either writes (the compiler cannot
  // tell that a write of one colour never feeds a read of the other).
  struct CellIn {
    float4 own, lft, rgt, nym, nyp, nzm, nzp;
    float f;
    int e, gx, gy;
  };
  auto gather = [&](auto Qc, int ly, int px, int s, int oc, int om, int op, int ofq) {
    constexpr int Q = decltype(Qc)::value;
    CellIn c;
    c.gx = X0 - H + 2 * px + s;
    c.gy = Y0 - H + ly;
    const int e = ly * PX + px;
    c.e = e;
    const int cq = Q * PP, co = (Q ^ 1) * PP;
    const int V = oc + co;
    const int ex = s ? e + 1 : e - 1;
    c.own = cell(oc + cq + e);
    const float4 nin = cell(V + e), nxo = cell(V + ex);
    c.lft = s ? nin : nxo;
    c.rgt = s ? nxo : nin;
    c.nym = cell(V + e - PX);
    c.nyp = cell(V + e + PX);
    c.nzm = cell(om + co + e);
    c.nzp = cell(op + co + e);
    c.f = sfv[ofq + e];
    return c;
  };
  auto inside = [&](const CellIn &c) {
    return !DIR || (c.gx >= 0 && c.gx < n0 && c.gy >= 0 && c.gy < n1);
  };
  // new (u, x) of the cell
  auto compute = [&](const CellIn &c, int m) -> float2 {
    const int gx = c.gx, gy = c.gy;
    const float di = c.own.x, xi = c.own.y;
    const float Ei = BG ? c.own.w : 1.0f;
    const float ubi = BG ? c.own.z : 0.0f;
    const float Bi = BG ? Ei + Ei * xi : 1.0f + xi;
    OpAcc<float, BG> A(di, Ei, xi, Bi, ubi);
    if (DIR && gx == 0)
      A.ghost(face_value(Gg, 0, gx, gy, m));
    else
      A.reg(c.lft.x, c.lft.y, c.lft.z, c.lft.w);
    if (DIR && gx == n0 - 1)
      A.ghost(face_value(Gg, 1, gx, gy, m));
    else
      A.reg(c.rgt.x, c.rgt.y, c.rgt.z, c.rgt.w);
    if (DIR && gy == 0)
      A.ghost(face_value(Gg, 2, gx, gy, m));
    else
      A.reg(c.nym.x, c.nym.y, c.nym.z, c.nym.w);
    if (DIR && gy == n1 - 1)
      A.ghost(face_value(Gg, 3, gx, gy, m));
    else
      A.reg(c.nyp.x, c.nyp.y, c.nyp.z, c.nyp.w);
    if (DIR && m == 0)
      A.ghost(face_value(Gg, 4, gx, gy, m));
    else
      A.reg(c.nzm.x, c.nzm.y, c.nzm.z, c.nzm.w);
    if (DIR && m == n2 - 1)
      A.ghost(face_value(Gg, 5, gx, gy, m));
    else
      A.reg(c.nzp.x, c.nzp.y, c.nzp.z, c.nzp.w);
    float acc, dacc;
    A.done(acc, dacc);
    float N, dN;
    finish_op(xi, Ei, acc, dacc, ah, beta, BG, N, dN);
    float du = newton_du(N, c.f, dN, relax);
    du = fminf(fmaxf(du, -cap), cap);
    const float dn = di + du;
    return make_float2(dn, BG || DIR ? m_expm1(dn) : m_expm1_full(dn));
  };
  auto update = [&](auto Qc, int ly, int px, int s, int m, int oc, int om, int op, int ofq) {
    constexpr int Q = decltype(Qc)::value;
    const CellIn c = gather(Qc, ly, px, s, oc, om, op, ofq);
    if (!inside(c)) return;
    const float2 r = compute(c, m);
    put_ux(oc + Q * PP + c.e, r.x, r.y);
  };
  // two updates of the same colour and plane (rows lya and lyb): both gather
  // before either stores, and their arithmetic interleaves
  auto update2 = [&](auto Qc, int lya, int lyb, int px, int s, int m, int oc, int om, int op,
                     int ofq) {
    constexpr int Q = decltype(Qc)::value;
    const CellIn a = gather(Qc, lya, px, s, oc, om, op, ofq);
    const CellIn b = gather(Qc, lyb, px, s, oc, om, op, ofq);
    if (DIR) {
      if (inside(a)) {
        const float2 r = compute(a, m);
        put_ux(oc + Q * PP + a.e, r.x, r.y);
      }
      if (inside(b)) {
        const float2 r = compute(b, m);
        put_ux(oc + Q * PP + b.e, r.x, r.y);
      }
    } else {
      const float2 ra = compute(a, m), rb = compute(b, m);
      put_ux(oc + Q * PP + a.e, ra.x, ra.y);
      put_ux(oc + Q * PP + b.e, rb.x, rb.y);
    }
  };

  const int P0 = Z0 - H, PE = Z1 + H;
  constexpr int SLOT = 2 * PP;
  // wrapped index of the plane being loaded (periodic grids)
  int pw = DIR ? P0 : wrapmod(P0, n2);
  if (!DIR || (P0 >= 0 && P0 < n2)) fetch((long long)pw * plane);
  // f half-slots: red of plane m at (m & 1) PP, black at (NFR + b) PP with b
  // advancing by one per plane (mod NFB)
  commit(P0 & 1, 0, (P0 & 1) * PP, NFR * PP);
  __syncthreads();
  int cur = 0, bcur = 0;  // ring slot of plane p, black f half-slot of plane p
  for (int p = P0; p < PE; p++) {
    const int pb = p & 1;
    const bool more = p + 1 < PE;
    pw = DIR ? p + 1 : (pw + 1 == n2 ? 0 : pw + 1);
    if (more && (!DIR || (pw >= 0 && pw < n2))) fetch((long long)pw * plane);
    const int o0 = cur * SLOT, o1 = ((cur + 3) & 3) * SLOT, o2 = ((cur + 2) & 3) * SLOT,
              o3 = ((cur + 1) & 3) * SLOT;  // planes p, p-1, p-2, p-3
    const int bnx = bcur == NFB - 1 ? 0 : bcur + 1;  // black f of plane p-2, then p+1
    const int f1 = ((p - 1) & 1) * PP;  // red f of plane p-1 (then of p+1)
    const int f2 = (NFR + bnx) * PP;
    // red cells of plane p-1 on the tile grown by one
    {
      const int m = p - 1;
      if (m >= Z0 - 1 && m < Z1 + 1 && (!DIR || (m >= 0 && m < n2))) {
        const int s = (w + 1 + pb + 1) & 1;  // rows 1 + w + j NW: parity of (ly + m) = s
        update2(std::integral_constant<int, 0>{}, 1 + w, 1 + w + NW, 1 + lane, s, m, o1, o2, o0,
                f1);
        if (w < 2)
          update(std::integral_constant<int, 0>{}, 1 + w + 2 * NW, 1 + lane, s, m, o1, o2, o0,
                 f1);
        if (w == 2 || w == 3) {
          const int idx = (w - 2) * 32 + lane;
          if (idx < C::NE) {
            const int ly = 1 + idx;
            const int se = (ly + m) & 1;
            update(std::integral_constant<int, 0>{}, ly, se ? 0 : PX - 1, se, m, o1, o2, o0, f1);
          }
        }
      }
    }
    __syncthreads();
    // black cells of plane p-2 on the tile
    {
      const int m = p - 2;
      if (m >= Z0 && m < Z1 && (!DIR || (m >= 0 && m < n2))) {
        const int s = (w + m + 1) & 1;  // rows 2 + w + j NW: parity of (ly + m + 1) = s
        update2(std::integral_constant<int, 1>{}, 2 + w, 2 + w + NW, 1 + lane, s, m, o2, o3, o1,
                f2);
      }
    }
    __syncthreads();
    // plane p-2 is final: write the tile out
    {
      const int wz = p - 2;
      if (wz >= Z0 && wz < Z1) {
        const long long woff = (long long)wz * plane;
#pragma unroll
        for (int k = 0; k < NLD; k++) {
          if (!(ldf[k] & 2u)) continue;
          const int q = threadIdx.x + k * NT;
          const int c0 = (int)((ldf[k] >> 2) & 1u) ^ (wz & 1);
          const float4 a = cell(o2 + c0 * PP + q);
          const float4 bb = cell(o2 + (c0 ^ 1) * PP + q);
          *reinterpret_cast<float2 *>(uout + woff + roff[k]) = make_float2(a.x, bb.x);
          *reinterpret_cast<float2 *>(xout + woff + roff[k]) = make_float2(a.y, bb.y);
        }
      }
    }
    if (more) commit(pb ^ 1, o3, f1, f2);
    __syncthreads();
    cur = (cur + 1) & 3;
    bcur = bnx;
  }
}

// ---------------------------------------------------------------------------
// One red-black sweep per launch with register-resident z-columns (plain FP32
// form, and with BG the correction form; the same sweep, cell for cell and bit
// for bit, as k_smooth_rb).
//
// A block owns a 64 x TY tile and a chunk of zc planes and marches along z over
// the planes Z0-2 .. Z1+1.  Every x-pair of the tile plus a halo of two cells
// (34 x (TY + 4) pairs) has one owner thread for the whole march, which keeps
// the pair's red and black cell ((u, x = expm1(u)), in the correction form
// (delta, x, background ub, E = e^ub)) and right-hand sides for the last four
// planes in registers: the z neighbours of an update are the owner's
// own registers, and only the xy exchange goes through shared memory.  At the
// step that loads plane p:
//   1. the pair's u, x and f of plane p (loaded a step earlier; x from the x
//      cache that the writer of u left beside it) are split into its red and
//      black cell, and the black cell, still old, is published to the black
//      half-plane of p;
//   2. the red cells of plane p-1 on the tile grown by one cell are updated:
//      x and y neighbours are black cells of plane p-1 (the other cell of the
//      pair from registers, the rest from the black half-plane published a
//      step earlier), z neighbours are the owner's old black cells of planes
//      p-2 and p; the new values are published to the red half-plane of p-1;
//   3. the black cells of plane p-2 on the tile are updated from the new red
//      cells (red half-plane of p-2, published a step earlier, and the owner's
//      red cells of planes p-3 and p-1), and plane p-2 (u and its x cache) is
//      written out.
// Half-planes are double-buffered by step parity, so a step reads only what
// the previous step wrote and one barrier per step suffices.
// With PRL the sweep is the first one after the coarse-grid correction: every
// arriving cell first gets u += P(u^H - R u^h) from the coarser grid (the
// trilinear 27/9/3/1 prolongation of k_prolong_tiled, z then y then x, same
// arithmetic) and its x is computed from the corrected u, so the separate
// prolongation pass is saved.  The coarse
// correction of the tile, blended in z for the next plane, is staged in
// shared memory during the step before (double-buffered as the half-planes).  The ring of
// register planes is indexed by the step modulo 4, which the loop unrolls into
// compile-time indices; which cell of a pair is red is a per-slot bit flipped
// every plane, applied with selects, so an update is straight-line code and
// the updates of a thread's slots interleave.
// In the correction form a cell is kept and published as its neighbours use it,
// (u, P = E x, ub, B = E + P), and the x and E that only its own update needs
// wait in the thread's own shared memory: bound by issue (60 % of slots), the
// two operations per face saved are 3 % of a sweep (512^3 1.081 -> 1.054 ms).
// 64 x 16 tiles of 512 threads (one block per SM, a sixth fewer halo updates)
// took as long, and planes arriving by 8-byte asynchronous copies 1.67 ms.
// Thread layout (256 threads, 8 warps): warp w owns the interior pairs
// px = 1 + lane of rows 2 + w + 8 j (j < TY / 8), and thread t < NHALO also
// one halo pair: the four halo rows for t < 128, the two halo columns above.
template <int TY, bool BG = false>
struct RCCfg {
  static constexpr int TX = 64, H = 2, PX = TX / 2 + 2, LY = TY + 2 * H, PP = PX * LY;
  static constexpr int NT = 256, NW = NT / 32;
  static constexpr int NI = TY / NW;                  // interior rows per thread
  static constexpr int NSL = NI + 1;                  // pair slots per thread
  static constexpr int NHR = 4 * (TX / 2);            // halo-row pairs
  static constexpr int NHALO = NHR + 2 * LY;          // all halo pairs
#ifndef FR_RC_MINB16
#define FR_RC_MINB16 2
#endif
  // resident blocks per SM (64 x 16 tiles: 2, 124 registers; 3 would cap the
  // registers at 80 and spill)
  // (correction form: four values per cell, 64 x 8 tiles at 2 blocks per SM)
  static constexpr int MINB = BG ? 2 : (TY <= 8 ? 3 : FR_RC_MINB16);
  using Cell = typename std::conditional<BG, float4, float2>::type;
  // coarse tile of the prolongation (fine tile plus halo, +-1 coarse cell)
  static constexpr int CXE = TX / 2 + 4, CYE = TY / 2 + 4, CE = CXE * CYE;
  static constexpr size_t smem(bool prl = false) {
    return (size_t)4 * PP * sizeof(Cell) + (prl ? (size_t)2 * CE * sizeof(float) : 0) +
           (BG ? NT * (4 * sizeof(float2) + 2 * sizeof(float)) : 0);
  }
  static_assert(TY % NW == 0 && NHALO <= NT, "tile height");
  static_assert(!BG || NI == 1, "the correction form keeps the x of one pair per thread");
};

template <bool BG, bool DIR, int TY, bool PRL = false>
__global__ void __launch_bounds__(RCCfg<TY, BG>::NT, RCCfg<TY, BG>::MINB)
    k_smooth_rc(const Grid<float> *grids, const int *off, int ngrid, int zc, const int *active,
                int par, const Grid<float> *coarse = nullptr, int cpar = 0) {
  using C = RCCfg<TY, BG>;
  using Cell = typename C::Cell;
  constexpr int TX = C::TX, PX = C::PX, PP = C::PP, NI = C::NI, NSL = C::NSL;
  constexpr int NHR = C::NHR, NHALO = C::NHALO, LY = C::LY;
  extern __shared__ float4 smem_rc4[];
  // black half-planes [2][PP] (old values), red half-planes [2][PP] (new values)
  Cell *const sbk = reinterpret_cast<Cell *>(smem_rc4);
  Cell *const srd = sbk + 2 * PP;
  float *const sez = reinterpret_cast<float *>(srd + 2 * PP);  // [2][CE] (PRL)
  constexpr int CXE = C::CXE, CE = C::CE;
  // correction form: (x, E) of the thread's black cells [4][NT], x of its
  // updated red cells [2][NT]
  [[maybe_unused]] float2 *const sxe = reinterpret_cast<float2 *>(srd + 2 * PP) + threadIdx.x;
  [[maybe_unused]] float *const sxr =
      reinterpret_cast<float *>(reinterpret_cast<float2 *>(srd + 2 * PP) + 4 * C::NT) + threadIdx.x;
  const int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<float> &Gg = grids[g];
  if (!grid_active(active, Gg.field)) return;
  const float *__restrict__ uin = par ? Gg.u2 : Gg.u;
  const float *__restrict__ xin = par ? Gg.x2 : Gg.x;  // x = expm1(u) of uin
  float *__restrict__ uout = par ? Gg.u : Gg.u2;
  float *__restrict__ xout = par ? Gg.x : Gg.x2;
  const float *__restrict__ fin = Gg.f;
  const float *__restrict__ ubin = Gg.ubg;
  const float *__restrict__ Ein = Gg.Ebg;
  const float ah = Gg.ah, beta = Gg.beta, cap = Gg.cap,
              relax = Gg.relax;
  const int n0 = Gg.n0, n1 = Gg.n1, n2 = Gg.n2;
  const int ntx = (n0 + TX - 1) / TX, nty = (n1 + TY - 1) / TY;
  int b = blockIdx.x - off[g];
  const int X0 = (b % ntx) * TX;
  b /= ntx;
  const int Y0 = (b % nty) * TY;
  b /= nty;
  const int Z0 = b * zc;
  const int Z1 = min(Z0 + zc, n2);
  const int P0 = Z0 - 2, nstep = Z1 - Z0 + 4;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long plane = (long long)n0 * n1;

  // slots: NI interior pairs, then (threads < NHALO) one halo pair.
  // fl: bit 0 load, bit 1 write out, bit 2 / 3 red update of the even / odd
  // cell; ro: 1 if the red cell of plane P0 is the odd one
  int q[NSL], roff[NSL], gyv[NSL], gxe[NSL];
  unsigned fl[NSL], ro[NSL];
#pragma unroll
  for (int s = 0; s < NSL; s++) {
    int px = -1, ly = -1;
    const bool interior = s < NI;
    if (interior) {
      px = 1 + lane;
      ly = 2 + w + C::NW * s;
    } else if ((int)threadIdx.x < NHALO) {
      const int t = threadIdx.x;
      if (t < NHR) {
        const int r = t >> 5;
        px = 1 + lane;
        ly = r < 2 ? r : TY + r;  // rows 0, 1, TY + 2, TY + 3
      } else {
        const int k = t - NHR;
        px = k < LY ? 0 : PX - 1;
        ly = k < LY ? k : k - LY;
      }
    }
    q[s] = 0;
    roff[s] = 0;
    gyv[s] = 0;
    gxe[s] = 0;
    fl[s] = 0;
    ro[s] = 0;
    if (px < 0) continue;
    const int gx = X0 - 2 + 2 * px, gy = Y0 - 2 + ly;
    q[s] = ly * PX + px;
    gyv[s] = gy;
    gxe[s] = gx;
    ro[s] = (unsigned)((gy + P0) & 1);  // gx even: colour of the even cell = (y + z) & 1
    bool ok;
    int gxw, gyw;
    if (DIR) {
      ok = gx >= 0 && gx < n0 && gy >= 0 && gy < n1;
      gxw = gx;
      gyw = gy;
    } else {
      ok = true;
      gxw = wrapmod(gx, n0);
      gyw = wrapmod(gy, n1);
    }
    if (!ok) continue;
    roff[s] = gyw * n0 + gxw;
    unsigned f = 1u;
    // red update on the tile grown by one cell: x in [X0-1, X0+TX], y in [Y0-1, Y0+TY]
    const bool yin = gy >= Y0 - 1 && gy <= Y0 + TY;
    if (yin && gx >= X0 - 1 && gx <= X0 + TX) f |= 4u;
    if (yin && gx + 1 >= X0 - 1 && gx + 1 <= X0 + TX) f |= 8u;
    if (interior && gx < n0 && gy < n1) f |= 2u;
    fl[s] = f;
  }

  // register ring: plane P0 + k in slot k & 3; red and black cell, f
  Cell R[NSL][4], B[NSL][4];
  float FR[NSL][4], FB[NSL][4];
  // prefetched plane (u, f and, in the correction form, ub and E of the even
  // and odd cell)
  // (without the prolongation, x of the arriving u is read from the x cache
  // its writer left beside it; with it, u changes on arrival and x is computed)
  float2 pu[NSL], px[NSL], pf[NSL], pb[NSL], pe[NSL];
#pragma unroll
  for (int s = 0; s < NSL; s++) {
    pu[s] = make_float2(0.f, 0.f);
    px[s] = pu[s];
    pf[s] = pu[s];
    pb[s] = pu[s];
    pe[s] = make_float2(1.f, 1.f);
#pragma unroll
    for (int r = 0; r < 4; r++) {
      R[s][r] = Cell{};
      B[s][r] = Cell{};
      FR[s][r] = 0.f;
      FB[s][r] = 0.f;
    }
  }
  int pw = DIR ? P0 : wrapmod(P0, n2);  // wrapped index of the next plane to load
  auto fetch = [&]() {
    if (!DIR || (pw >= 0 && pw < n2)) {
      const long long zo = (long long)pw * plane;
#pragma unroll
      for (int s = 0; s < NSL; s++) {
        if (!(fl[s] & 1u)) continue;
        pu[s] = *reinterpret_cast<const float2 *>(uin + zo + roff[s]);
        if (!PRL) px[s] = *reinterpret_cast<const float2 *>(xin + zo + roff[s]);
        if (fin) pf[s] = *reinterpret_cast<const float2 *>(fin + zo + roff[s]);
        if (BG) {
          pb[s] = *reinterpret_cast<const float2 *>(ubin + zo + roff[s]);
          pe[s] = *reinterpret_cast<const float2 *>(Ein + zo + roff[s]);
        }
      }
    }
    pw = DIR ? pw + 1 : (pw + 1 == n2 ? 0 : pw + 1);
  };
  fetch();

  // prolongation (PRL): coarse correction e = u^H - R u^h of the coarse cells
  // (X0/2 - 2 + ci, Y0/2 - 2 + cj), blended in z for fine plane p, into sez[b].
  // The coarse values of the next plane are loaded into registers early in a
  // step (ez_load) and blended and stored at its end (ez_store), so that the
  // loads' latency overlaps the step's updates.
  const float w3 = 0.75f, w1 = 0.25f;
  constexpr int NEZ = PRL ? (CE + C::NT - 1) / C::NT : 1;
  float ezH[NEZ][2], ezR[NEZ][2];
  int coff[NEZ];  // offset in a coarse plane of this thread's tile entries (-1: none / zero)
  const float *__restrict__ cuH = nullptr;
  const float *__restrict__ cuR = nullptr;
  int c2 = 1;
  long long cplane = 0;
  if constexpr (PRL) {
    const Grid<float> &Cg = coarse[g];
    cuH = cpar ? Cg.u2 : Cg.u;
    cuR = Cg.uR;
    const int c0 = Cg.n0, c1 = Cg.n1;
    c2 = Cg.n2;
    cplane = (long long)c0 * c1;
#pragma unroll
    for (int r = 0; r < NEZ; r++) {
      const int q = threadIdx.x + r * C::NT;
      coff[r] = -1;
      if (q >= CE) continue;
      const int cj = q / CXE, ci = q - cj * CXE;
      int I = X0 / 2 - 2 + ci, J = Y0 / 2 - 2 + cj;
      if (DIR) {
        if (!(I >= 0 && I < c0 && J >= 0 && J < c1)) continue;
      } else {
        I = wrapmod(I, c0);
        J = wrapmod(J, c1);
      }
      coff[r] = J * c0 + I;
    }
  }
  auto ez_load = [&](int p) {
    if constexpr (PRL) {
      const int pz = DIR ? p : wrapmod(p, n2);
      const int K = pz >> 1, K2 = (pz & 1) ? K + 1 : K - 1;  // nearer, farther coarse plane
      const bool vK = !DIR || (pz >= 0 && pz < n2);
      // K is in [0, c2) for a wrapped pz; K2 wraps by one plane at most
      int K2w = K2;
      bool vK2 = vK;
      if (DIR)
        vK2 = vK && K2 >= 0 && K2 < c2;
      else
        K2w = K2 < 0 ? c2 - 1 : (K2 == c2 ? 0 : K2);
      const long long oa = (long long)K * cplane, ob = (long long)K2w * cplane;
#pragma unroll
      for (int r = 0; r < NEZ; r++) {
        ezH[r][0] = ezR[r][0] = ezH[r][1] = ezR[r][1] = 0.0f;
        if (coff[r] < 0) continue;
        if (vK) {
          ezH[r][0] = cuH[oa + coff[r]];
          ezR[r][0] = cuR[oa + coff[r]];
        }
        if (vK2) {
          ezH[r][1] = cuH[ob + coff[r]];
          ezR[r][1] = cuR[ob + coff[r]];
        }
      }
    }
  };
  auto ez_store = [&](int bsel) {
    if constexpr (PRL) {
#pragma unroll
      for (int r = 0; r < NEZ; r++) {
        const int q = threadIdx.x + r * C::NT;
        if (q >= CE) continue;
        const float ea = ezH[r][0] - ezR[r][0], eb = ezH[r][1] - ezR[r][1];
        sez[bsel * CE + q] = w3 * ea + w1 * eb;
      }
    }
  };
  if constexpr (PRL) {
    ez_load(P0);
    ez_store(0);
    __syncthreads();
  }

  // x of a new u: without the branch in the plain form (on patches its
  // registers would spill)
  auto ex = [](float u) { return BG || DIR ? m_expm1(u) : m_expm1_full(u); };
  // (ub, E) of a cell: (0, 1) in the plain form
  auto bgv = [](const Cell &c) -> float2 {
    if constexpr (BG)
      return make_float2(c.z, c.w);
    else
      return make_float2(0.0f, 1.0f);
  };
  // Newton update of one cell: own cell and f, neighbours -x, +x, -y, +y, -z,
  // +z; the same face order and arithmetic as k_smooth_rb
  auto newton = [&](Cell own, float fi, Cell lf, Cell rt, Cell ym, Cell yp, Cell zm, Cell zp,
                    int gx, int gy, int m) -> float {
    const float di = own.x, xi = own.y;
    const float Ei = bgv(own).y, ubi = bgv(own).x;
    const float Bi = BG ? Ei + Ei * xi : 1.0f + xi;
    OpAcc<float, BG> A(di, Ei, xi, Bi, ubi);
    auto nb = [&](const Cell &c) {
      if constexpr (BG)
        A.reg_pb(c.x, c.y, c.z, c.w);
      else
        A.reg(c.x, c.y, 0.0f, 1.0f);
    };
    if (DIR && gx == 0)
      A.ghost(face_value(Gg, 0, gx, gy, m));
    else
      nb(lf);
    if (DIR && gx == n0 - 1)
      A.ghost(face_value(Gg, 1, gx, gy, m));
    else
      nb(rt);
    if (DIR && gy == 0)
      A.ghost(face_value(Gg, 2, gx, gy, m));
    else
      nb(ym);
    if (DIR && gy == n1 - 1)
      A.ghost(face_value(Gg, 3, gx, gy, m));
    else
      nb(yp);
    if (DIR && m == 0)
      A.ghost(face_value(Gg, 4, gx, gy, m));
    else
      nb(zm);
    if (DIR && m == n2 - 1)
      A.ghost(face_value(Gg, 5, gx, gy, m));
    else
      nb(zp);
    float acc, dacc, N, dN;
    A.done(acc, dacc);
    finish_op(xi, Ei, acc, dacc, ah, beta, BG, N, dN);
    float du = newton_du(N, fi, dN, relax);
    du = fminf(fmaxf(du, -cap), cap);
    return di + du;
  };
  auto sel = [](bool c, Cell a, Cell b) { return c ? a : b; };
  // the plain form's two interior slots are updated as packed pairs
  constexpr bool PACK = !DIR && !BG && NI == 2;
  auto with_u2 = [](const Cell &c, float u, float x) -> Cell {
    Cell r = c;
    r.x = u;
    r.y = x;
    return r;
  };
  // cell of value u (x recomputed) with the background of cell c
  auto with_u = [&](const Cell &c, float u) -> Cell {
    Cell r = c;
    r.x = u;
    r.y = ex(u);
    return r;
  };

  auto step = [&](auto Kc, int k) {
    constexpr int K = decltype(Kc)::value;  // ring slot of plane p
    constexpr int K1 = (K + 3) & 3, K2 = (K + 2) & 3, K3 = (K + 1) & 3;
    constexpr unsigned PK = K & 1, PK1 = K1 & 1, PK2 = K2 & 1;  // plane parities (rel. P0)
    const int p = P0 + k;
    // 1. plane p from the prefetch registers; publish its black cells
    {
      const bool inz = !DIR || (p >= 0 && p < n2);
#pragma unroll
      for (int s = 0; s < NSL; s++) {
        if (!(fl[s] & 1u)) continue;
        if constexpr (PRL) {
          // u += P(e): coarse column ci = px + 1, row cj = ly / 2 + 1 of the
          // tile; the farther row is cj + 1 for odd y, cj - 1 for even y
          const int ly = q[s] / PX, px = q[s] - ly * PX;
          const int ci = px + 1, cj = (ly >> 1) + 1, cj2 = (ly & 1) ? cj + 1 : cj - 1;
          const float *za = sez + PK * CE + cj * CXE, *zb = sez + PK * CE + cj2 * CXE;
          const float em = w3 * za[ci - 1] + w1 * zb[ci - 1];
          const float e0 = w3 * za[ci] + w1 * zb[ci];
          const float ep = w3 * za[ci + 1] + w1 * zb[ci + 1];
          pu[s].x = pu[s].x + (w3 * e0 + w1 * em);
          pu[s].y = pu[s].y + (w3 * e0 + w1 * ep);
        }
        const bool odd = (ro[s] ^ PK) != 0;  // red cell is the odd one
        const float ur = odd ? pu[s].y : pu[s].x, ub = odd ? pu[s].x : pu[s].y;
        // the red cell's x is needed only if this pair's red cell is updated
        const bool needr = s < NI || (fl[s] & (odd ? 8u : 4u));
        if constexpr (PRL) {
          if (needr) {
            px[s] = DIR ? m_expm1_2(pu[s]) : m_expm1_full2(pu[s]);
          } else {
            px[s].x = px[s].y = ex(ub);
          }
        }
        const float xr = odd ? px[s].y : px[s].x, xb = odd ? px[s].x : px[s].y;
        if constexpr (BG) {
          R[s][K] = make_float4(ur, needr ? xr : 0.0f,
                                odd ? pb[s].y : pb[s].x, odd ? pe[s].y : pe[s].x);
          const float Eb = odd ? pe[s].x : pe[s].y, Pb = __fmul_rn(Eb, xb);
          B[s][K] = make_float4(ub, Pb, odd ? pb[s].x : pb[s].y, __fadd_rn(Eb, Pb));
          if (s < NI) sxe[K * C::NT] = make_float2(xb, Eb);
        } else {
          R[s][K] = make_float2(ur, needr ? xr : 0.0f);
          B[s][K] = make_float2(ub, xb);
        }
        if (fin) {
          const float fr = odd ? pf[s].y : pf[s].x, fb = odd ? pf[s].x : pf[s].y;
          FR[s][K] = fr;  // FP32 grids: fs = 1, fo = 0, fs (f - fo) = f exactly
          FB[s][K] = fb;
        } else {
          FR[s][K] = 0.0f;
          FB[s][K] = 0.0f;
        }
        if (inz) sbk[PK * PP + q[s]] = B[s][K];
      }
    }
    if (k + 1 < nstep) {
      fetch();
      ez_load(p + 1);
    }
    // 2. red cells of plane m = p - 1 on the grown tile
    {
      const int m = p - 1;
      if (m >= Z0 - 1 && m <= Z1 && (!DIR || (m >= 0 && m < n2))) {
        if constexpr (PACK) {
          // the two interior slots (same row parity) in packed pairs
          const bool odd = (ro[0] ^ PK1) != 0;
          float2 nu[6], nxv[6];
          float2 di, xi, fi;
#pragma unroll
          for (int s = 0; s < 2; s++) {
            const Cell *bk = sbk + PK1 * PP + q[s];
            const Cell nx = bk[odd ? 1 : -1];
            const Cell in = B[s][K1];
            const Cell c6[6] = {odd ? in : nx, odd ? nx : in, bk[-PX], bk[PX], B[s][K2], B[s][K]};
#pragma unroll
            for (int f = 0; f < 6; f++) {
              (s ? nu[f].y : nu[f].x) = c6[f].x;
              (s ? nxv[f].y : nxv[f].x) = c6[f].y;
            }
            (s ? di.y : di.x) = R[s][K1].x;
            (s ? xi.y : xi.x) = R[s][K1].y;
            (s ? fi.y : fi.x) = FR[s][K1];
          }
          const float2 un = newton2_plain(di, xi, fi, nu, nxv, ah, beta, cap, relax);
          const float2 xn = m_expm1_full2(un);
          R[0][K1] = with_u2(R[0][K1], un.x, xn.x);
          R[1][K1] = with_u2(R[1][K1], un.y, xn.y);
          srd[PK1 * PP + q[0]] = R[0][K1];
          srd[PK1 * PP + q[1]] = R[1][K1];
        }
#pragma unroll
        for (int s = PACK ? 2 : 0; s < NSL; s++) {
          const bool odd = (ro[s] ^ PK1) != 0;
          if (!((s < NI && !DIR) || (fl[s] & (odd ? 8u : 4u)))) continue;
          const Cell *bk = sbk + PK1 * PP + q[s];
          const Cell ym = bk[-PX], yp = bk[PX];
          const Cell nx = bk[odd ? 1 : -1];
          const float un = newton(R[s][K1], FR[s][K1], sel(odd, B[s][K1], nx),
                                  sel(odd, nx, B[s][K1]), ym, yp, B[s][K2], B[s][K],
                                  gxe[s] + (odd ? 1 : 0), gyv[s], m);
          if constexpr (BG) {
            const float xn = ex(un), Er = R[s][K1].w, Pr = __fmul_rn(Er, xn);
            R[s][K1] = make_float4(un, Pr, R[s][K1].z, __fadd_rn(Er, Pr));
            if (s < NI) sxr[PK1 * C::NT] = xn;
          } else {
            R[s][K1] = with_u(R[s][K1], un);
          }
          srd[PK1 * PP + q[s]] = R[s][K1];
        }
      }
    }
    // 3. black cells of plane m = p - 2 on the tile, then plane m is final
    {
      const int m = p - 2;
      if (m >= Z0 && m < Z1 && (!DIR || (m >= 0 && m < n2))) {
        [[maybe_unused]] float2 unp, xnp;
        if constexpr (PACK) {
          const bool odd = (ro[0] ^ PK2) == 0;  // black cell is the odd one
          float2 nu[6], nxv[6];
          float2 di, xi, fi;
#pragma unroll
          for (int s = 0; s < 2; s++) {
            const Cell *rd = srd + PK2 * PP + q[s];
            const Cell nx = rd[odd ? 1 : -1];
            const Cell in = R[s][K2];
            const Cell c6[6] = {odd ? in : nx, odd ? nx : in, rd[-PX], rd[PX], R[s][K3], R[s][K1]};
#pragma unroll
            for (int f = 0; f < 6; f++) {
              (s ? nu[f].y : nu[f].x) = c6[f].x;
              (s ? nxv[f].y : nxv[f].x) = c6[f].y;
            }
            (s ? di.y : di.x) = B[s][K2].x;
            (s ? xi.y : xi.x) = B[s][K2].y;
            (s ? fi.y : fi.x) = FB[s][K2];
          }
          unp = newton2_plain(di, xi, fi, nu, nxv, ah, beta, cap, relax);
          xnp = m_expm1_full2(unp);
        }
#pragma unroll
        for (int s = 0; s < NI; s++) {
          if (DIR && !(fl[s] & 1u)) continue;
          const bool odd = (ro[s] ^ PK2) == 0;  // black cell is the odd one
          if constexpr (PACK) {
            B[s][K2] = with_u2(B[s][K2], s ? unp.y : unp.x, s ? xnp.y : xnp.x);
          } else {
            const Cell *rd = srd + PK2 * PP + q[s];
            const Cell ym = rd[-PX], yp = rd[PX];
            const Cell nx = rd[odd ? 1 : -1];
            Cell own = B[s][K2];
            if constexpr (BG) {
              const float2 xe = sxe[K2 * C::NT];
              own.y = xe.x;
              own.w = xe.y;
            }
            const float un = newton(own, FB[s][K2], sel(odd, R[s][K2], nx), sel(odd, nx, R[s][K2]), ym,
                        yp, R[s][K3], R[s][K1], gxe[s] + (odd ? 1 : 0), gyv[s], m);
            B[s][K2] = with_u(B[s][K2], un);
          }
          if (fl[s] & 2u) {
            Cell rr = R[s][K2];
            if constexpr (BG) rr.y = sxr[PK2 * C::NT];
            const Cell e = sel(odd, rr, B[s][K2]), o = sel(odd, B[s][K2], rr);
            const long long oo = (long long)m * plane + roff[s];
            *reinterpret_cast<float2 *>(uout + oo) = make_float2(e.x, o.x);
            *reinterpret_cast<float2 *>(xout + oo) = make_float2(e.y, o.y);
          }
        }
      }
    }
    if (k + 1 < nstep) ez_store((int)(PK ^ 1u));
    __syncthreads();
  };
  for (int k = 0; k < nstep; k += 4) {
    step(std::integral_constant<int, 0>{}, k);
    if (k + 1 < nstep) step(std::integral_constant<int, 1>{}, k + 1);
    if (k + 2 < nstep) step(std::integral_constant<int, 2>{}, k + 2);
    if (k + 3 < nstep) step(std::integral_constant<int, 3>{}, k + 3);
  }
}

// Tiled FAS right-hand side of a coarse level, f <- A(u) - f (the same
// operator evaluation, face order and arithmetic as k_fas_rhs): a block owns a
// 64 x 16 tile and a chunk of zc planes and marches along z with a ring of
// three planes of (u, x) [and (ub, E)] in shared memory (tile plus a halo of
// one cell); at the step that has loaded plane p it evaluates plane p-1, each
// thread four cells (two rows, x = lane and lane + 32), with f read and written
// in place.  The next plane is prefetched into registers during the evaluation.
constexpr int kFrTX = 64, kFrTY = 16;
// dynamic shared memory of k_fas_rhs_tiled: three planes of the tile plus halo,
// (u, x, ub, E) per cell in the correction form, (u, x) in the plain one
constexpr size_t fas_rhs_tiled_smem(bool bg) {
  return (size_t)3 * (kFrTX + 2) * (kFrTY + 2) * (bg ? sizeof(float4) : sizeof(float2));
}
template <bool BG, bool DIR>
__global__ void __launch_bounds__(256)
    k_fas_rhs_tiled(const Grid<float> *grids, const int *off, int ngrid, int zc,
                    const int *active, int par) {
  constexpr int LX = kFrTX + 2, LY = kFrTY + 2, PC = LX * LY, NT = 256;
  constexpr int NLD = (PC + NT - 1) / NT;
  extern __shared__ float4 sfr[];
  float2 *s2 = reinterpret_cast<float2 *>(sfr);
  auto cellv = [&](int i) -> float4 {
    if (BG) return sfr[i];
    const float2 v = s2[i];
    return make_float4(v.x, v.y, 0.f, 1.f);
  };
  const int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<float> &Gg = grids[g];
  if (!grid_active(active, Gg.field)) return;
  const float *__restrict__ uin = par ? Gg.u2 : Gg.u;
  const float *__restrict__ xin = par ? Gg.x2 : Gg.x;
  const float *__restrict__ ubin = Gg.ubg;
  const float *__restrict__ Ein = Gg.Ebg;
  float *__restrict__ f = const_cast<float *>(Gg.f);
  const float ah = Gg.ah, beta = Gg.beta;
  const int n0 = Gg.n0, n1 = Gg.n1, n2 = Gg.n2;
  const int ntx = (n0 + kFrTX - 1) / kFrTX, nty = (n1 + kFrTY - 1) / kFrTY;
  int b = blockIdx.x - off[g];
  const int X0 = (b % ntx) * kFrTX;
  b /= ntx;
  const int Y0 = (b % nty) * kFrTY;
  b /= nty;
  const int Z0 = b * zc, Z1 = min(Z0 + zc, n2);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long plane = (long long)n0 * n1;
  // plane-load table: cell q = threadIdx.x + k NT of the (TX + 2) x (TY + 2) tile
  int roff[NLD];
  bool lok[NLD];
#pragma unroll
  for (int k = 0; k < NLD; k++) {
    const int q = threadIdx.x + k * NT;
    roff[k] = 0;
    lok[k] = false;
    if (q < PC) {
      const int gx = X0 - 1 + q % LX, gy = Y0 - 1 + q / LX;
      if (DIR) {
        lok[k] = gx >= 0 && gx < n0 && gy >= 0 && gy < n1;
        roff[k] = lok[k] ? gy * n0 + gx : 0;
      } else {
        lok[k] = true;
        roff[k] = wrapmod(gy, n1) * n0 + wrapmod(gx, n0);
      }
    }
  }
  float4 pv[NLD];
  // plane at offset zoff (vz false: outside a patch, never read)
  auto fetch = [&](long long zoff, bool vz) {
#pragma unroll
    for (int k = 0; k < NLD; k++) {
      pv[k] = make_float4(0.f, 0.f, 0.f, 1.f);
      if (!vz || !lok[k]) continue;
      const long long gi = zoff + roff[k];
      pv[k].x = uin[gi];
      pv[k].y = xin[gi];
      if (BG) {
        pv[k].z = ubin[gi];
        pv[k].w = Ein[gi];
      }
    }
  };
  auto commit = [&](int so) {
#pragma unroll
    for (int k = 0; k < NLD; k++) {
      const int q = threadIdx.x + k * NT;
      if (q >= PC) continue;
      if (BG)
        sfr[so + q] = pv[k];
      else
        s2[so + q] = make_float2(pv[k].x, pv[k].y);
    }
  };
  // f <- A(u) - f at tile cell (lx, ly) of plane m; om, oc, op: slots of m-1, m, m+1
  auto eval = [&](int lx, int ly, int m, int om, int oc, int op) {
    const int gx = X0 - 1 + lx, gy = Y0 - 1 + ly;
    if (gx >= n0 || gy >= n1) return;
    const int i = ly * LX + lx;
    const float4 own = cellv(oc + i);
    const float di = own.x, xi = own.y;
    const float Ei = BG ? own.w : 1.0f;
    const float ubi = BG ? own.z : 0.0f;
    const float Bi = BG ? Ei + Ei * xi : 1.0f + xi;
    OpAcc<float, BG> A(di, Ei, xi, Bi, ubi);
    auto nb = [&](int j) {
      const float4 v = cellv(j);
      A.reg(v.x, v.y, v.z, v.w);
    };
    if (DIR && gx == 0) A.ghost(face_value(Gg, 0, gx, gy, m)); else nb(oc + i - 1);
    if (DIR && gx == n0 - 1) A.ghost(face_value(Gg, 1, gx, gy, m)); else nb(oc + i + 1);
    if (DIR && gy == 0) A.ghost(face_value(Gg, 2, gx, gy, m)); else nb(oc + i - LX);
    if (DIR && gy == n1 - 1) A.ghost(face_value(Gg, 3, gx, gy, m)); else nb(oc + i + LX);
    if (DIR && m == 0) A.ghost(face_value(Gg, 4, gx, gy, m)); else nb(om + i);
    if (DIR && m == n2 - 1) A.ghost(face_value(Gg, 5, gx, gy, m)); else nb(op + i);
    float acc, dacc, N, dN;
    A.done(acc, dacc);
    finish_op(xi, Ei, acc, dacc, ah, beta, BG, N, dN);
    const long long c = (long long)m * plane + (long long)gy * n0 + gx;
    f[c] = N - f[c];
  };
  const int P0 = Z0 - 1, PE = Z1 + 1;
  auto inr = [&](int pz) { return !DIR || (pz >= 0 && pz < n2); };
  int pw = DIR ? P0 : wrapmod(P0, n2);
  fetch((long long)pw * plane, inr(P0));
  commit(0);
  __syncthreads();
  int cur = 0;  // ring slot of plane p
  for (int p = P0; p < PE; p++) {
    const bool more = p + 1 < PE;
    pw = DIR ? p + 1 : (pw + 1 == n2 ? 0 : pw + 1);
    if (more) fetch((long long)pw * plane, inr(p + 1));
    const int o0 = cur * PC, o1 = (cur == 0 ? 2 : cur - 1) * PC,
              o2 = (cur == 2 ? 0 : cur + 1) * PC;  // planes p, p-1, p-2
    const int m = p - 1;
    if (m >= Z0 && m < Z1) {
#pragma unroll
      for (int r = 0; r < 2; r++)
#pragma unroll
        for (int h = 0; h < 2; h++) eval(1 + lane + 32 * h, 1 + w + 8 * r, m, o2, o1, o0);
    }
    __syncthreads();
    if (more) commit(o2);
    __syncthreads();
    cur = cur == 2 ? 0 : cur + 1;
  }
}

// ---------------------------------------------------------------------------
// Asynchronous global-to-shared copy of 8 bytes (PTX cp.async; both
// addresses 8-byte aligned); commit_group / wait_group track completion.
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Tiled FP32 residual + restriction (same result as k_resid_restrict).
// A block owns a 64 x 16 fine tile and an even chunk of zc fine planes and
// marches along z; a thread owns the 2 x 2 fine cells of one coarse column.
// The planes arrive by asynchronous copies in a ring of four in shared memory,
// two ahead of the one in use; each thread copies its own cells and the cells
// beyond the tile that only it needs, and keeps its cells of planes m - 1, m,
// m + 1 in registers, so that shared memory is read for the arriving plane and
// the rows above and below only (x neighbours come by shuffles) and one barrier
// per plane suffices.  Without a patch's ghost faces the two cells of an x-pair
// are evaluated as one packed pair.  After every second plane a thread writes
// its coarse cell (u^H = uR = mean u^h, x^H = expm1(u^H), f^H <- mean d^h); the
// fine residual norm is accumulated on the way.
//
// 512^3: 0.379 ms plain, 0.715 ms in the correction form (3 and 5 arrays read,
// 0.28 and 0.44 ms of memory time); with every neighbour of a cell read from
// shared memory, which left one or two blocks per SM, 0.477 and 0.824 ms.
// Bound by instruction issue (packed FP32, shuffles) at 24 warps per SM in the
// plain form, 16 in the correction form.
template <bool BG>
struct RRCfg {
  static constexpr int TX = 64, TY = 16, NT = 256, NW = NT / 32;
  static_assert(TY == 2 * NW && TX == 64, "two rows per warp, one pair per lane");
  static constexpr int NA = BG ? 4 : 2;  // arrays: u, x [, ub, E]
  static constexpr int NS = 4;           // planes in the ring: m, m + 1 and two on their way
  // rows -1 .. 16 of an array, then the columns left and right of the tile; f
  // without either
  static constexpr int EC = (TY + 2) * TX, AN = EC + 2 * TY, PL = NA * AN + TY * TX;
  static constexpr int MINB = BG ? 2 : 3;
  static constexpr size_t smem = (size_t)NS * PL * sizeof(float);
};

template <bool BG, bool DIR>
__global__ void __launch_bounds__(RRCfg<BG>::NT, RRCfg<BG>::MINB)
    k_resid_restrict_tiled(const Grid<float> *fine, const Grid<float> *coarse, const int *off,
                           int ngrid, int zc, const int *active, int fpar, int cpar,
                           double *partial) {
  using C = RRCfg<BG>;
  constexpr int TX = C::TX, TY = C::TY, NT = C::NT, NA = C::NA;
  constexpr bool CV = BG && !DIR;  // (x, E) are published and kept as (P, B)
  extern __shared__ float smem[];
  const int g = find_grid(off, ngrid, blockIdx.x);
  const Grid<float> &Fg = fine[g];
  const Grid<float> &Cg = coarse[g];
  float ss = 0.0f, mx = 0.0f;
  if (grid_active(active, Fg.field)) {
    const float *__restrict__ in[4] = {fpar ? Fg.u2 : Fg.u, fpar ? Fg.x2 : Fg.x, Fg.ubg, Fg.Ebg};
    const float *__restrict__ fin = Fg.f;
    const float ah = Fg.ah, beta = Fg.beta;
    const int n0 = Fg.n0, n1 = Fg.n1, n2 = Fg.n2;
    const int c0 = Cg.n0, c1 = Cg.n1;
    float *__restrict__ cu = cpar ? Cg.u2 : Cg.u;
    float *__restrict__ cR = Cg.uR;
    float *__restrict__ cx = cpar ? Cg.x2 : Cg.x;
    float *__restrict__ cf = const_cast<float *>(Cg.f);
    const int ntx = (n0 + TX - 1) / TX, nty = (n1 + TY - 1) / TY;
    int b = blockIdx.x - off[g];
    const int X0 = (b % ntx) * TX;
    b /= ntx;
    const int Y0 = (b % nty) * TY;
    b /= nty;
    const int Z0 = b * zc;
    const int Z1 = min(Z0 + zc, n2);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int gx = X0 + 2 * lane, gy = Y0 + 2 * w;
    const bool valid = gx < n0 && gy < n1;
    const long long fplane = (long long)n0 * n1;
    // What a lane copies of a plane (offsets, -1: none): 16 bytes of row 2 w
    // (lanes 0 - 15) or 2 w + 1, and of the row beyond the tile (first and last
    // warp).  The first and last lane also copy the cells left and right of the
    // tile.  (Rows are whole quads: a level that has a coarser one has n0 a
    // multiple of 4, see count_levels.)
    auto at = [&](int x, int y) -> int {
      if (DIR) return x >= 0 && x < n0 && y >= 0 && y < n1 ? y * n0 + x : -1;
      return wrapmod(y, n1) * n0 + wrapmod(x, n0);
    };
    const int lx = 4 * (lane & 15), ly = lane >> 4;
    const int o0 = at(X0 + lx, gy + ly);
    const int oh = w == 0 && !ly ? at(X0 + lx, gy - 1)
                                 : (w == C::NW - 1 && !ly ? at(X0 + lx, gy + 2) : -1);
    const int ex = lane == 0 ? X0 - 1 : X0 + TX;
    const bool edge = lane == 0 || lane == 31;
    const int oe = edge ? at(ex, gy) : -1;  // (and the row above: n1 is even)
    // their places in an array's tile, and the own pair of row 2 w
    const int qc = (2 * w + 1 + ly) * TX + lx;
    const int qh = (w == 0 ? 0 : TY + 1) * TX + lx;
    const int qe = C::EC + (lane == 0 ? 0 : TY) + 2 * w;
    const int q0 = (2 * w + 1) * TX + 2 * lane;
    auto inz = [&](int p) { return !DIR || (p >= 0 && p < n2); };
    auto wrapz = [&](int p) { return DIR ? p : (p < 0 ? p + n2 : (p >= n2 ? p - n2 : p)); };

    float2 r[4][NA][2];  // plane (m - 1, m, m + 1 live), array, row
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
      for (int a = 0; a < NA; a++)
        r[k][a][0] = r[k][a][1] = make_float2(a == 3 ? 1.f : 0.f, a == 3 ? 1.f : 0.f);
    auto ld2 = [](const float *p) { return *reinterpret_cast<const float2 *>(p); };
    // copies of plane p into its slot, one commit group
    auto fetch = [&](int p) {
      if (p <= Z1 && inz(p)) {
        const bool own = p >= Z0 && p < Z1;
        const long long zo = (long long)wrapz(p) * fplane;
        float *h = smem + ((p - Z0 + 1) & 3) * C::PL;
#pragma unroll
        for (int a = 0; a < NA; a++) {
          const float *v = in[a] + zo;
          float *ha = h + a * C::AN;
          if (o0 >= 0) cp_async16(ha + qc, v + o0);
          if (own && oh >= 0) cp_async16(ha + qh, v + oh);
          if (own && oe >= 0) {
            cp_async4(ha + qe, v + oe);
            cp_async4(ha + qe + 1, v + oe + n0);
          }
        }
        if (fin && own && o0 >= 0)
          cp_async16(h + NA * C::AN + qc - TX, fin + zo + o0);
      }
      cp_async_commit();
    };
    // (x, E) -> (P, B), P = E x, B = E + P
    auto conv = [](float2 &x, float2 &E) {
      x = mul2(E, x);
      E = add2(E, x);
    };
    float2 su = make_float2(0.f, 0.f), sd = su, s2 = su;

    auto step = [&](auto Kc, int p) {
      constexpr int K = decltype(Kc)::value;  // ring slot of plane p
      constexpr int K1 = (K + 3) & 3, K2 = (K + 2) & 3;
      // 1. plane p + 2 on its way (into the slot of plane p - 2, last read in
      // the step before the last barrier), plane p from its slot
      fetch(p + 2);
      cp_async_wait<2>();
      __syncwarp();  // a warp's rows are copied by all of its lanes
      const float *sp = smem + K * C::PL;
#pragma unroll
      for (int a = 0; a < NA; a++) {
        r[K][a][0] = ld2(sp + a * C::AN + q0);
        r[K][a][1] = ld2(sp + a * C::AN + q0 + TX);
      }
      // 2. residual of plane m = p - 1
      const int m = p - 1;
      if (m >= Z0) {
        const float *sm = smem + K1 * C::PL;
        float2 O[NA][2];
#pragma unroll
        for (int a = 0; a < NA; a++) {
          O[a][0] = r[K1][a][0];
          O[a][1] = r[K1][a][1];
        }
        if (CV) {
          conv(O[1][0], O[NA - 1][0]);
          conv(O[1][1], O[NA - 1][1]);
        }
#pragma unroll
        for (int k = 0; k < 2; k++) {
          // left and right neighbours of the pair, and the row below (k = 0)
          // or above (k = 1) the own two
          float2 L[NA], R[NA], V[NA];
          float lo[NA], hi[NA];
#pragma unroll
          for (int a = 0; a < NA; a++) {
            lo[a] = __shfl_up_sync(0xffffffffu, O[a][k].y, 1);
            hi[a] = __shfl_down_sync(0xffffffffu, O[a][k].x, 1);
          }
          if (edge) {
            float e[NA];
#pragma unroll
            for (int a = 0; a < NA; a++) e[a] = sm[a * C::AN + qe + k];
            if (CV) {
              e[1] = __fmul_rn(e[NA - 1], e[1]);
              e[NA - 1] = __fadd_rn(e[NA - 1], e[1]);
            }
#pragma unroll
            for (int a = 0; a < NA; a++) (lane == 0 ? lo[a] : hi[a]) = e[a];
          }
#pragma unroll
          for (int a = 0; a < NA; a++) {
            L[a] = make_float2(lo[a], O[a][k].x);
            R[a] = make_float2(O[a][k].y, hi[a]);
            V[a] = ld2(sm + a * C::AN + q0 + (k ? 2 * TX : -TX));
          }
          if (CV) conv(V[1], V[NA - 1]);
          const float2 di = r[K1][0][k], xi = r[K1][1][k];
          const float2 f =
              fin ? ld2(sm + NA * C::AN + q0 + (k - 1) * TX) : make_float2(0.f, 0.f);
          float2 d;
          if constexpr (!DIR) {
            float2 Zm[NA], Zp[NA];
#pragma unroll
            for (int a = 0; a < NA; a++) {
              Zm[a] = r[K2][a][k];
              Zp[a] = r[K][a][k];
            }
            if (CV) conv(Zp[1], Zp[NA - 1]);
            float2 S1, S2;
            [[maybe_unused]] float2 G1, G2;  // of the correction form
            auto face = [&](const float2 (&v)[NA], bool first) {
              const float2 dd = sub2(v[0], di);
              S1 = first ? dd : add2(S1, dd);
              S2 = first ? mul2(v[NA - 1], dd) : fma2(v[NA - 1], dd, S2);
              if constexpr (BG) {
                const float2 gg = sub2(v[2], r[K1][NA - 2][k]);
                G1 = first ? gg : add2(G1, gg);
                G2 = first ? mul2(v[1], gg) : fma2(v[1], gg, G2);
              }
            };
            auto other = [&]() {
              float2 t[NA];
#pragma unroll
              for (int a = 0; a < NA; a++) t[a] = O[a][1 - k];
              face(t, false);
            };
            face(L, true);
            face(R, false);
            if (k == 0) face(V, false);
            other();
            if (k == 1) face(V, false);
            face(Zm, false);
            face(Zp, false);
            float2 acc;
            if constexpr (BG) {
              const float2 Ei = r[K1][NA - 1][k];
              acc = add2(fma2(O[1][k], G1, G2), fma2(fma2(Ei, xi, Ei), S1, S2));
            } else {
              acc = fma2(add2(add2(splat2(1.0f), xi), splat2(1.0f)), S1, S2);
            }
            // N of finish_op, in pairs
            const float2 B1 = add2(splat2(1.0f), xi);
            const float2 rs = make_float2(sfu_rsqrt(B1.x), sfu_rsqrt(B1.y));
            const float2 den = add2(B1, mul2(B1, rs));
            const float2 y = mul2(neg2(xi), make_float2(sfu_rcp(den.x), sfu_rcp(den.y)));
            float2 bF = splat2(beta);
            if constexpr (BG) {
              const float2 Ei = r[K1][NA - 1][k];
              bF = mul2(bF, make_float2(sfu_rsqrt(Ei.x), sfu_rsqrt(Ei.y)));
            }
            d = sub2(fma2(splat2(ah), acc, mul2(bF, y)), f);
          } else {
            // cell by cell, with the ghost faces of a patch
#pragma unroll
            for (int ax = 0; ax < 2; ax++) {
              auto lane_of = [&](const float2 &v) { return ax ? v.y : v.x; };
              const int gxq = gx + ax, gyq = gy + k;
              const float dc = lane_of(di), xc = lane_of(xi);
              const float Ei = BG ? lane_of(r[K1][NA - 1][k]) : 1.0f;
              const float ubi = BG ? lane_of(r[K1][NA - 2][k]) : 0.0f;
              const float Bi = BG ? Ei + Ei * xc : 1.0f + xc;
              OpAcc<float, BG> A(dc, Ei, xc, Bi, ubi);
              auto nb = [&](auto get) {
                A.reg(lane_of(get(0)), lane_of(get(1)), BG ? lane_of(get(NA - 2)) : 0.0f,
                      BG ? lane_of(get(NA - 1)) : 1.0f);
              };
              if (gxq == 0) A.ghost(face_value(Fg, 0, gxq, gyq, m));
              else nb([&](int a) { return L[a]; });
              if (gxq == n0 - 1) A.ghost(face_value(Fg, 1, gxq, gyq, m));
              else nb([&](int a) { return R[a]; });
              if (gyq == 0) A.ghost(face_value(Fg, 2, gxq, gyq, m));
              else nb([&](int a) { return k ? O[a][0] : V[a]; });
              if (gyq == n1 - 1) A.ghost(face_value(Fg, 3, gxq, gyq, m));
              else nb([&](int a) { return k ? V[a] : O[a][1]; });
              if (m == 0) A.ghost(face_value(Fg, 4, gxq, gyq, m));
              else nb([&](int a) { return r[K2][a][k]; });
              if (m == n2 - 1) A.ghost(face_value(Fg, 5, gxq, gyq, m));
              else nb([&](int a) { return r[K][a][k]; });
              float acc, dacc, N, dN;
              A.done(acc, dacc);
              finish_op(xc, Ei, acc, dacc, ah, beta, BG, N, dN);
              (ax ? d.y : d.x) = N - lane_of(f);
            }
          }
          if (valid) {
            sd = add2(sd, d);
            su = add2(su, di);
            s2 = fma2(d, d, s2);
            mx = fmaxf(mx, fmaxf(fabsf(d.x), fabsf(d.y)));
          }
        }
        if (((m - Z0) & 1) && valid) {
          const long long cidx = ((long long)(m >> 1) * c1 + (gy >> 1)) * c0 + (gx >> 1);
          const float uh = (su.x + su.y) * 0.125f;
          cR[cidx] = uh;
          cu[cidx] = uh;
          cx[cidx] = m_expm1(uh);
          cf[cidx] = (sd.x + sd.y) * 0.125f;
          su = sd = make_float2(0.f, 0.f);
        }
      }
      if (CV) {  // plane p - 1 becomes the plane below
        conv(r[K1][1][0], r[K1][NA - 1][0]);
        conv(r[K1][1][1], r[K1][NA - 1][1]);
      }
      __syncthreads();
    };
    // planes Z0 - 1 .. Z1; the number of planes is even (zc and n2 are)
    fetch(Z0 - 1);
    fetch(Z0);
    for (int p = Z0 - 1; p <= Z1; p += 4) {
      step(std::integral_constant<int, 0>{}, p);
      step(std::integral_constant<int, 1>{}, p + 1);
      if (p + 2 <= Z1) {
        step(std::integral_constant<int, 2>{}, p + 2);
        step(std::integral_constant<int, 3>{}, p + 3);
      }
    }
    ss = s2.x + s2.y;
    cp_async_wait<0>();
  }
  if (partial) block_reduce2f<NT>(ss, mx, &partial[2 * blockIdx.x], &partial[2 * blockIdx.x + 1]);
}

}  // namespace frmg
