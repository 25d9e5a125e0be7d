// frmg_tail.cuh -- the small levels of a V-cycle in one kernel.
//
// A V-cycle (Sec. V.B.2) spends about eleven dependent steps on every level
// (colours of the sweeps, residual, restriction, FAS right-hand side,
// prolongation).  On a level of at most a few ten thousand cells one launch
// per step costs 5 to 9 microseconds of launch, descriptor and L2 latency and
// leaves most of the GPU idle.  k_tail runs all levels of one grid from such a
// level down to the coarsest and back up in one thread-block cluster: the
// level's planes are dealt out to the cluster's blocks, every array lives in
// the blocks' shared memory for the whole pass, and a step ends at a hardware
// cluster barrier.  Each block also holds copies of u and x of the planes
// above and below its own; whoever writes a cell of a first or last plane
// writes the neighbour's copy too (distributed shared memory), so that the
// operator reads its own block's memory only, at fixed offsets, all loads in
// flight together.  Levels of at most tail_local() cells live in the first
// block alone (block barriers only), a coarsest grid of at most kTailWarp
// cells in its first warp.
//
// The updates are those of k_smooth, k_resid_restrict, k_fas_rhs, k_prolong
// and k_coarsest, cell by cell in the same operation order (the coarsest
// solve's stopping sums are added in another order).
#pragma once

#include <cooperative_groups.h>

#include "frmg_kernels.cuh"

namespace frmg {

namespace cg = cooperative_groups;

constexpr int kTailLev = 8;       // levels of a tail
constexpr int kTailWarp = 128;    // cells of a coarsest grid relaxed by one warp
constexpr int kTailCluster = 16;  // most blocks per cluster

// Threads per block.  FP32: 1024 threads would halve the registers and spill
// (85 against 73 us on the 32^3 tail); FP64 levels have at most 16^3 cells here.
template <typename T>
__host__ __device__ constexpr int tail_threads() {
  return sizeof(T) == 4 ? 512 : 256;
}

// Cells of a level kept in one block.  An FP64 step of n cells takes the FP64
// pipe about 65 cycles per cell on one SM, more than a cluster barrier (600 to
// 900 cycles) already at 8^3 cells; an FP32 step of 8^3 cells takes 1000.
template <typename T>
__host__ __device__ constexpr int tail_local() {
  return sizeof(T) == 4 ? 1024 : 64;
}

// Planes per block of a level (all of them in the first block if it is local).
template <typename T>
inline __host__ __device__ int tail_planes(int n0, int n1, int n2, int cs) {
  if ((long long)n0 * n1 * n2 <= tail_local<T>()) return n2;
  return (n2 + cs - 1) / cs;
}

struct TailOpts {
  int pre, post;
  int fas;    // 1: f of the top level holds R d: form the FAS right-hand side first
  int keepx;  // 1: write x of the top level too (the finest level)
  double crs_rel, crs_abs;
  int crs_maxit, crs_stall, crs_meanfix;
};

// One level: the part that is the same for every block (set up by the host),
// then what depends on the block.  Entry q of a plane of array a is at
// a + plane + kl * plane + q for the own plane kl (u, x, background; kl = -1
// and np are the copies) and at a + kl * plane + q for f, d and R u.  e: the
// correction of the coarser level on the coarse planes that the own planes
// interpolate.
template <typename T>
struct TailLevel {
  int n0, n1, n2, hx, plane, zc, local;
  unsigned u, x, ub, E, f, d, r, e;  // the arrays in shared memory (cells)
  unsigned mh, m0, m1, mz;           // division by hx, n0, n1, zc: (t m) >> 32
  T ah, fs, fo;
  T *gu[2], *gx[2];                  // the grid's arrays (Grid)
  const T *gf;
  const float *gub, *gE;
  const T *bnd;
  long long foff[6];
  int z0, np;                        // own planes [z0, z0 + np)
  int below, above;                  // blocks that own the planes under and over them
  int belowo;                        // own plane 0's copy in the block below (offset in an array)
};

// A grid's tail, as the host lays it out.
template <typename T>
struct TailDesc {
  int nl, field;
  T beta, cap, relax;
  TailLevel<T> lev[kTailLev];
};

// Sets up the block-independent part of level q of a tail laid out from `base`
// cells of shared memory on (bg: with the background arrays); returns its end.
template <typename T>
inline unsigned tail_layout(TailLevel<T> &L, const Grid<T> &G, int cs, bool bg, bool top,
                            unsigned base) {
  auto magic = [](int d) {
    return d <= 1 ? 0u : (unsigned)(((1ull << 32) + (unsigned)d - 1) / (unsigned)d);
  };
  L.n0 = G.n0;
  L.n1 = G.n1;
  L.n2 = G.n2;
  L.hx = G.n0 >> 1;
  L.plane = G.n0 * G.n1;
  L.zc = tail_planes<T>(G.n0, G.n1, G.n2, cs);
  L.local = G.ncell <= tail_local<T>();
  L.mh = magic(L.hx);
  L.m0 = magic(L.n0);
  L.m1 = magic(L.n1);
  L.mz = magic(L.zc);
  L.ah = G.ah;
  L.fs = G.fs;
  L.fo = G.fo;
  L.gu[0] = G.u;
  L.gu[1] = G.u2;
  L.gx[0] = G.x;
  L.gx[1] = G.x2;
  L.gf = G.f;
  L.gub = G.ubg;
  L.gE = G.Ebg;
  L.bnd = G.bnd;
  for (int f = 0; f < 6; f++) L.foff[f] = G.foff[f];
  const unsigned a = (unsigned)((L.zc + 2) * L.plane), b = (unsigned)(L.zc * L.plane);
  L.u = base;
  L.x = L.u + a;
  L.ub = L.x + a;
  L.E = L.ub + (bg ? a : 0);
  L.f = L.E + (bg ? a : 0);
  L.d = L.f + b;
  L.r = L.d + b;
  L.e = L.r + (top ? 0 : b);
  return (L.e + (unsigned)((L.zc / 2 + 3) * (L.plane / 4)) + 3) & ~3u;  // 16-byte aligned
}

// What the steps of one block share.
template <typename T>
struct TailBlock {
  static constexpr int NT = tail_threads<T>();
  using A = typename std::conditional<sizeof(T) == 4, float, double>::type;
  TailDesc<T> D;
  int cs, me;                  // blocks of the cluster, this one
  A red[2 * (NT / 32)];        // a block sum's warp sums
  A slots[2 * kTailCluster];   // a cluster sum's block sums
  float nslot[2 * kTailCluster];  // blocks' residual norms (first block)
};

template <typename T>
__device__ __forceinline__ T *tail_smem() {
  extern __shared__ __align__(16) unsigned char tail_smem_raw[];
  return reinterpret_cast<T *>(tail_smem_raw);
}

// Who works on a step: the cluster (2) or its first block (1).
__device__ __forceinline__ void tail_sync(int mode) {
  if (mode == 2) cg::this_cluster().sync();
  else __syncthreads();
}

template <typename T>
__device__ __forceinline__ T *tail_remote(T *p, int rank) {
  return cg::this_cluster().map_shared_rank(p, rank);
}

// t / d with m = ceil(2^32 / d): exact for t d < 2^32 (a tail's levels have
// far fewer cells); d = 1 has m = 0.
__device__ __forceinline__ int tail_div(int t, unsigned m) {
  return m ? (int)__umulhi((unsigned)t, m) : t;
}

template <typename T>
__device__ __forceinline__ T tail_face(const TailLevel<T> &L, int f, int i, int j, int k) {
  const long long o = f < 2 ? (long long)k * L.n1 + j
                            : (f < 4 ? (long long)k * L.n0 + i : (long long)j * L.n0 + i);
  return __ldg(L.bnd + L.foff[f] + o);
}

template <typename T>
__device__ __forceinline__ void tail_ijk(const TailLevel<T> &L, int t, int &i, int &j, int &kl) {
  const int q = tail_div(t, L.m0);
  kl = tail_div(q, L.m1);
  j = q - kl * L.n1;
  i = t - q * L.n0;
}

// Writes values to an own plane and to the neighbours' copies of the first and
// last plane.
template <typename T, bool DIR>
struct TailPut {
  T *sm, *below, *above;  // this block's shared memory and the neighbours'
  int plane, last, belowo;
  __device__ __forceinline__ explicit TailPut(const TailLevel<T> &L)
      : sm(tail_smem<T>()), plane(L.plane), last(L.np - 1), belowo(L.belowo) {
    below = DIR && L.z0 == 0 ? nullptr : tail_remote(sm, L.below);
    above = DIR && L.z0 + L.np == L.n2 ? nullptr : tail_remote(sm, L.above);
  }
  // entry q of plane kl of the arrays at a and b
  __device__ __forceinline__ void operator()(unsigned a, T va, unsigned b, T vb, int kl,
                                             int q) const {
    sm[a + (kl + 1) * plane + q] = va;
    sm[b + (kl + 1) * plane + q] = vb;
    if (kl == 0 && (!DIR || below)) {
      below[a + belowo + q] = va;
      below[b + belowo + q] = vb;
    }
    if (kl == last && (!DIR || above)) {
      above[a + q] = va;
      above[b + q] = vb;
    }
  }
};

// Face sums at cell (i, j) of own plane kl: cell_sums on the level's
// shared-memory arrays.  All loads come first.
template <typename T, bool BG, bool DIR>
__device__ __forceinline__ void tail_sums(const TailLevel<T> &L, int i, int j, int kl, T &ui,
                                          T &xi, T &Ei, T &acc, T &dacc) {
  const T *sm = tail_smem<T>();
  const int n0 = L.n0, pl = L.plane, o = (kl + 1) * pl + j * n0 + i;
  const bool b0 = i == 0, b1 = i == n0 - 1, b2 = j == 0, b3 = j == L.n1 - 1;
  const int wx = n0 - 1, wy = pl - n0;
  const int nb[6] = {o + (b0 ? wx : -1), o + (b1 ? -wx : 1), o + (b2 ? wy : -n0),
                     o + (b3 ? -wy : n0), o - pl, o + pl};
  T du[6], dx[6], db[6], dE[6];
#pragma unroll
  for (int q = 0; q < 6; q++) {
    du[q] = sm[L.u + nb[q]];
    dx[q] = sm[L.x + nb[q]];
    db[q] = BG ? sm[L.ub + nb[q]] : T(0);
    dE[q] = BG ? sm[L.E + nb[q]] : T(1);
  }
  ui = sm[L.u + o];
  xi = sm[L.x + o];
  Ei = BG ? sm[L.E + o] : T(1);
  const T ubi = BG ? sm[L.ub + o] : T(0);
  const T Bi = BG ? Ei + Ei * xi : T(1) + xi;
  OpAcc<T, BG> A(ui, Ei, xi, Bi, ubi);
  if (DIR) {
    const int k = L.z0 + kl;
    const bool g[6] = {b0, b1, b2, b3, k == 0, k == L.n2 - 1};
#pragma unroll
    for (int q = 0; q < 6; q++) {
      if (g[q]) A.ghost(tail_face(L, q, i, j, k));
      else A.reg(du[q], dx[q], db[q], dE[q]);
    }
  } else {
#pragma unroll
    for (int q = 0; q < 6; q++) A.reg(du[q], dx[q], db[q], dE[q]);
  }
  A.done(acc, dacc);
}

// A_i (or N_i) and its derivative at that cell.
template <typename T, bool BG, bool DIR>
__device__ __forceinline__ void tail_eval(const TailLevel<T> &L, T beta, int i, int j, int kl,
                                          T &ui, T &xi, T &N, T &dN) {
  T Ei, acc, dacc;
  tail_sums<T, BG, DIR>(L, i, j, kl, ui, xi, Ei, acc, dacc);
  finish_op(xi, Ei, acc, dacc, L.ah, beta, BG, N, dN);
}

// Sums of a and b over the threads of a step, the same on every thread;
// another tail_sync has to come before the next call.
template <typename T>
__device__ __forceinline__ void tail_sum2(TailBlock<T> &B, int mode, typename TailBlock<T>::A &a,
                                          typename TailBlock<T>::A &b) {
  using A = typename TailBlock<T>::A;
  constexpr int NW = TailBlock<T>::NT / 32;
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    B.red[2 * w] = a;
    B.red[2 * w + 1] = b;
  }
  __syncthreads();
  a = l < NW ? B.red[2 * l] : A(0);
  b = l < NW ? B.red[2 * l + 1] : A(0);
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (mode == 1) return;
  if ((int)threadIdx.x < B.cs) {
    A *r = tail_remote(B.slots, threadIdx.x);
    r[2 * B.me] = a;
    r[2 * B.me + 1] = b;
  }
  tail_sync(2);
  a = A(0);
  b = A(0);
  for (int q = 0; q < B.cs; q++) {
    a += B.slots[2 * q];
    b += B.slots[2 * q + 1];
  }
}

// The steps below are functions of their own, not inlined, so that every use
// runs the same instructions (inlined everywhere they would not fit the
// instruction cache).

// Red-black sweeps of level l (k_smooth).  The position of a thread's x-pair is
// found once where every thread has at most one.
template <typename T, bool BG, bool DIR>
__device__ __noinline__ void tail_smooth(const TailBlock<T> &B, int l, int sweeps, int mode) {
  const TailLevel<T> &L = B.D.lev[l];
  const T *sm = tail_smem<T>();
  constexpr int nt = TailBlock<T>::NT;
  const int n = L.np * L.n1 * L.hx;
  const TailPut<T, DIR> put(L);
  const T beta = B.D.beta, cap = B.D.cap, relax = B.D.relax;
  int j, kl, i0, c0;
  auto pair = [&](int t) {
    const int q = tail_div(t, L.mh);
    kl = tail_div(q, L.m1);
    j = q - kl * L.n1;
    i0 = 2 * (t - q * L.hx);
    c0 = (j + L.z0 + kl) & 1;
  };
  auto update = [&](int c) {
    const int i = i0 + ((c0 + c) & 1), q = j * L.n0 + i;
    T ui, xi, Ei, acc, dacc;
    const T f = sm[L.f + kl * L.plane + q];
    tail_sums<T, BG, DIR>(L, i, j, kl, ui, xi, Ei, acc, dacc);
    const T un = ui + newton_from_sums<T, BG>(xi, Ei, acc, dacc, f, L.ah, beta, cap, relax);
    put(L.u, un, L.x, m_expm1(un), kl, q);
  };
  const bool one = n <= nt;
  if (one) pair(min((int)threadIdx.x, n - 1));
  for (int s = 0; s < 2 * sweeps; s++) {
    if (one) {
      if ((int)threadIdx.x < n) update(s & 1);
    } else {
      for (int t = threadIdx.x; t < n; t += nt) {
        pair(t);
        update(s & 1);
      }
    }
    tail_sync(mode);
  }
}

// d = A(u) - f (fas = false) or f = A(u) - f in place (fas = true, k_fas_rhs);
// norm: this block's sum d^2 and max |d| go to the first block's nslot.
template <typename T, bool BG, bool DIR>
__device__ __noinline__ void tail_resid(TailBlock<T> &B, int l, bool fas, bool norm, int mode) {
  const TailLevel<T> &L = B.D.lev[l];
  T *sm = tail_smem<T>();
  constexpr int NT = TailBlock<T>::NT;
  const int n = L.np * L.plane;
  const unsigned out = fas ? L.f : L.d;
  float s = 0.0f, m = 0.0f;
  for (int t = threadIdx.x; t < n; t += NT) {
    int i, j, kl;
    tail_ijk(L, t, i, j, kl);
    T ui, xi, N, dN;
    const T f = sm[L.f + t];
    tail_eval<T, BG, DIR>(L, B.D.beta, i, j, kl, ui, xi, N, dN);
    const T d = N - f;
    sm[out + t] = d;
    const float df_ = (float)d;
    s = fmaf(df_, df_, s);
    m = fmaxf(m, fabsf(df_));
  }
  if (norm) {
    float *rf = reinterpret_cast<float *>(B.red);
    for (int q = 16; q > 0; q >>= 1) {
      s += __shfl_down_sync(0xffffffffu, s, q);
      m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, q));
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
      rf[2 * w] = s;
      rf[2 * w + 1] = m;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      s = 0.0f;
      m = 0.0f;
      for (int q = 0; q < NT / 32; q++) {
        s += rf[2 * q];
        m = fmaxf(m, rf[2 * q + 1]);
      }
      float *r = tail_remote(B.nslot, 0);
      r[2 * B.me] = s;
      r[2 * B.me + 1] = m;
    }
  }
  tail_sync(mode);
}

// u and d of level l averaged onto the own planes of level l + 1 (the second
// half of k_resid_restrict).
template <typename T, bool DIR>
__device__ __noinline__ void tail_restrict(const TailBlock<T> &B, int l, int mode) {
  const TailLevel<T> &F = B.D.lev[l], &C = B.D.lev[l + 1];
  T *sm = tail_smem<T>();
  const int n = C.np * C.plane;
  const TailPut<T, DIR> put(C);
  for (int t = threadIdx.x; t < n; t += TailBlock<T>::NT) {
    int I, J, Kl;
    tail_ijk(C, t, I, J, Kl);
    T su = T(0), sd = T(0);
#pragma unroll
    for (int cz = 0; cz < 2; cz++) {
      const int k = 2 * (C.z0 + Kl) + cz, r = tail_div(k, F.mz);
      const T *p = tail_remote(sm, r) + (k - r * F.zc) * F.plane + 2 * J * F.n0 + 2 * I;
#pragma unroll
      for (int cy = 0; cy < 2; cy++)
#pragma unroll
        for (int cx = 0; cx < 2; cx++) {
          const int q = cy * F.n0 + cx;
          sd += p[F.d + q];
          su += p[F.u + F.plane + q];
        }
    }
    const T uh = su * T(0.125);
    const int q = J * C.n0 + I;
    put(C.u, uh, C.x, m_expm1(uh), Kl, q);
    sm[C.f + t] = sd * T(0.125);
    sm[C.r + t] = uh;
  }
  tail_sync(mode);
}

// u of the own planes of level l += P (u^H - R u^h) of level l + 1 (k_prolong).
// The correction on the coarse planes that the own planes need is gathered
// from their owners first.
template <typename T, bool DIR>
__device__ __noinline__ void tail_prolong(const TailBlock<T> &B, int l, int mode) {
  const TailLevel<T> &F = B.D.lev[l], &C = B.D.lev[l + 1];
  T *sm = tail_smem<T>();
  const T w3 = T(0.75), w1 = T(0.25);
  const int n = F.np * F.n1 * F.hx;
  const int K0 = (F.z0 >> 1) - 1;  // first coarse plane gathered
  if (n > 0) {
    const int ne = (((F.z0 + F.np - 1) >> 1) + 2 - K0) * C.plane;
    for (int t = threadIdx.x; t < ne; t += TailBlock<T>::NT) {
      const int s = tail_div(tail_div(t, C.m0), C.m1), q = t - s * C.plane;
      int K = K0 + s;
      const bool out = K < 0 || K >= C.n2;
      K = K < 0 ? K + C.n2 : (K >= C.n2 ? K - C.n2 : K);
      const int r = tail_div(K, C.mz);
      const T *p = tail_remote(sm, r) + (K - r * C.zc) * C.plane + q;
      const T v = p[C.u + C.plane] - p[C.r];
      sm[F.e + t] = DIR && out ? T(0) : v;  // coarse cells outside the grid contribute 0
    }
  }
  __syncthreads();
  const TailPut<T, DIR> put(F);
  for (int t = threadIdx.x; t < n; t += TailBlock<T>::NT) {
    const int q = tail_div(t, F.mh), kl = tail_div(q, F.m1);
    const int j = q - kl * F.n1, I = t - q * F.hx, k = F.z0 + kl;
    // coarse neighbours: the containing cell and the one on the child's side
    const int im = I > 0 ? I - 1 : C.n0 - 1, ip = I < C.n0 - 1 ? I + 1 : 0;
    T exy[2][2];  // [child][z]
#pragma unroll
    for (int z = 0; z < 2; z++) {
      const T *p = sm + F.e + ((k >> 1) + (z ? ((k & 1) ? 1 : -1) : 0) - K0) * C.plane;
      T ex[2][2];
#pragma unroll
      for (int y = 0; y < 2; y++) {
        int J = (j >> 1) + (y ? ((j & 1) ? 1 : -1) : 0);
        const bool vy = J >= 0 && J < C.n1;
        J = J < 0 ? J + C.n1 : (J >= C.n1 ? J - C.n1 : J);
        const T *pe = p + J * C.n0;
        T e0 = pe[im], e1 = pe[I], e2 = pe[ip];
        if (DIR) {
          if (!vy) e0 = e1 = e2 = T(0);
          if (I == 0) e0 = T(0);
          if (I == C.n0 - 1) e2 = T(0);
        }
        ex[0][y] = w3 * e1 + w1 * e0;
        ex[1][y] = w3 * e1 + w1 * e2;
      }
      exy[0][z] = w3 * ex[0][0] + w1 * ex[0][1];
      exy[1][z] = w3 * ex[1][0] + w1 * ex[1][1];
    }
    const int w = j * F.n0 + 2 * I;
#pragma unroll
    for (int a = 0; a < 2; a++) {
      const T un = sm[F.u + (kl + 1) * F.plane + w + a] + (w3 * exy[a][0] + w1 * exy[a][1]);
      put(F.u, un, F.x, m_expm1(un), kl, w + a);
    }
  }
  tail_sync(mode);
}

// Newton-Gauss-Seidel sweeps on level l to the coarsest level's stopping rule
// (k_coarsest).
template <typename T, bool BG, bool DIR>
__device__ __noinline__ void tail_coarsest(TailBlock<T> &B, int l, const TailOpts &o, int mode) {
  using A = typename TailBlock<T>::A;
  const TailLevel<T> &L = B.D.lev[l];
  const T *sm = tail_smem<T>();
  constexpr int nt = TailBlock<T>::NT;
  const int n = L.np * L.plane;
  const A cells = (A)(L.n2 * L.plane);
  const bool shift = !DIR && o.crs_meanfix;
  const TailPut<T, DIR> put(L);
  A thr = A(0), prev = A(0);
  for (int it = -1; it < o.crs_maxit; it++) {
    if (it >= 0) tail_smooth<T, BG, DIR>(B, l, 1, mode);
    // what = 0: sums for the Newton step on a constant shift (periodic grids),
    // what = 1: the residual's square sum
    for (int what = it >= 0 && shift ? 0 : 1; what < 2; what++) {
      A s = A(0), D = A(0);
      for (int t = threadIdx.x; t < n; t += nt) {
        int i, j, kl;
        tail_ijk(L, t, i, j, kl);
        T ui, xi, N, dN;
        const T f = sm[L.f + t];
        tail_eval<T, BG, DIR>(L, B.D.beta, i, j, kl, ui, xi, N, dN);
        const A d = (A)(N - f);
        if (what) {
          s += d * d;
        } else {
          s += d;
          const T F = BG ? m_rsqrt(sm[L.E + L.plane + t]) : T(1);
          D += A(0.5) * (A)B.D.beta * (A)(F * m_rsqrt(T(1) + xi));
        }
      }
      tail_sum2(B, mode, s, D);
      if (what) {
        const A rms = sqrt(s / cells);
        bool stop;
        if (it < 0) {
          thr = fmax((A)o.crs_rel * rms, (A)o.crs_abs);
          stop = rms <= thr;
        } else {
          stop = rms <= thr || (o.crs_stall && rms >= prev);
        }
        prev = rms;
        tail_sync(mode);  // the sums have been read
        if (stop) return;
      } else {
        const A cap = (A)B.D.cap;
        A c = D > A(0) ? s / D : A(0);
        c = c > cap ? cap : (c < -cap ? -cap : c);
        tail_sync(mode);  // every cell and the sums have been read
        for (int t = threadIdx.x; t < n; t += nt) {
          const int kl = tail_div(tail_div(t, L.m0), L.m1), q = t - kl * L.plane;
          const T un = sm[L.u + L.plane + t] + (T)c;
          put(L.u, un, L.x, m_expm1(un), kl, q);
        }
        tail_sync(mode);
      }
    }
  }
}

// tail_coarsest by one warp on a level of at most 64 P cells in one block: a
// lane keeps the positions, right-hand sides and backgrounds of its P x-pairs
// in registers for the whole solve.
template <typename T, bool BG, bool DIR, int P>
__device__ __noinline__ void tail_coarsest_warp(TailBlock<T> &B, int l, const TailOpts &o) {
  using A = typename TailBlock<T>::A;
  const TailLevel<T> &L = B.D.lev[l];
  T *U = tail_smem<T>() + L.u, *X = tail_smem<T>() + L.x;
  const T *sb = tail_smem<T>() + L.ub, *sE = tail_smem<T>() + L.E, *sf = tail_smem<T>() + L.f;
  const int n0 = L.n0, pl = L.plane, n = L.n1 * L.n2 * L.hx;
  const T beta = B.D.beta, cap = B.D.cap, relax = B.D.relax, ah = L.ah;
  const A cells = (A)(2 * n);
  // cell v of pair p: v = 0 red, 1 black
  int at[P][2], nb[P][2][6], ci[P][2], cj[P], ck[P];
  T f[P][2], ub[P][2], E[P][2], gb[P][2][6];
  bool mine[P];
#pragma unroll
  for (int p = 0; p < P; p++) {
    const int t = threadIdx.x + 32 * p;
    mine[p] = t < n;
    const int q = tail_div(mine[p] ? t : 0, L.mh), k = tail_div(q, L.m1), j = q - k * L.n1;
    cj[p] = j;
    ck[p] = k;
#pragma unroll
    for (int v = 0; v < 2; v++) {
      const int i = 2 * ((mine[p] ? t : 0) - q * L.hx) + ((j + k + v) & 1);
      const int c = (k + 1) * pl + j * n0 + i;
      ci[p][v] = i;
      at[p][v] = c;
      nb[p][v][0] = i > 0 ? c - 1 : c + n0 - 1;
      nb[p][v][1] = i < n0 - 1 ? c + 1 : c - (n0 - 1);
      nb[p][v][2] = j > 0 ? c - n0 : c + pl - n0;
      nb[p][v][3] = j < L.n1 - 1 ? c + n0 : c - (pl - n0);
      nb[p][v][4] = k > 0 ? c - pl : c + (L.n2 - 1) * pl;
      nb[p][v][5] = k < L.n2 - 1 ? c + pl : c - (L.n2 - 1) * pl;
      f[p][v] = sf[c - pl];
      ub[p][v] = BG ? sb[c] : T(0);
      E[p][v] = BG ? sE[c] : T(1);
      if (DIR) {
        const bool g[6] = {i == 0, i == n0 - 1, j == 0, j == L.n1 - 1, k == 0, k == L.n2 - 1};
#pragma unroll
        for (int w = 0; w < 6; w++) gb[p][v][w] = g[w] ? tail_face(L, w, i, j, k) : T(0);
      }
    }
  }
  // face sums of a cell, its u and x
  auto sums = [&](int p, int v, T &ui, T &xi, T &a, T &da) {
    T du[6], dx[6], db[6], dE[6];
#pragma unroll
    for (int q = 0; q < 6; q++) {
      const int c = nb[p][v][q];
      du[q] = U[c];
      dx[q] = X[c];
      db[q] = BG ? sb[c] : T(0);
      dE[q] = BG ? sE[c] : T(1);
    }
    ui = U[at[p][v]];
    xi = X[at[p][v]];
    const T Ei = E[p][v], Bi = BG ? Ei + Ei * xi : T(1) + xi;
    OpAcc<T, BG> acc(ui, Ei, xi, Bi, ub[p][v]);
    const int i = ci[p][v], j = cj[p], k = ck[p];
    const bool g[6] = {i == 0, i == n0 - 1, j == 0, j == L.n1 - 1, k == 0, k == L.n2 - 1};
#pragma unroll
    for (int q = 0; q < 6; q++) {
      if (DIR && g[q]) acc.ghost(gb[p][v][q]);
      else acc.reg(du[q], dx[q], db[q], dE[q]);
    }
    acc.done(a, da);
  };
  auto sum = [&](A a) {
    for (int q = 16; q > 0; q >>= 1) a += __shfl_xor_sync(0xffffffffu, a, q);
    return a;
  };
  const bool shift = !DIR && o.crs_meanfix;
  A thr = A(0), prev = A(0);
  for (int it = -1; it < o.crs_maxit; it++) {
    if (it >= 0) {
#pragma unroll
      for (int v = 0; v < 2; v++) {
#pragma unroll
        for (int p = 0; p < P; p++) {
          if (!mine[p]) continue;
          T ui, xi, a, da;
          sums(p, v, ui, xi, a, da);
          const T un = ui + newton_from_sums<T, BG>(xi, E[p][v], a, da, f[p][v], ah, beta, cap,
                                                    relax);
          U[at[p][v]] = un;
          X[at[p][v]] = m_expm1(un);
        }
        __syncwarp();
      }
    }
    for (int what = it >= 0 && shift ? 0 : 1; what < 2; what++) {
      A s = A(0), D = A(0);
#pragma unroll
      for (int p = 0; p < P; p++)
#pragma unroll
        for (int v = 0; v < 2; v++) {
          if (!mine[p]) continue;
          T ui, xi, a, da, N, dN;
          sums(p, v, ui, xi, a, da);
          finish_op(xi, E[p][v], a, da, ah, beta, BG, N, dN);
          const A d = (A)(N - f[p][v]);
          if (what) {
            s += d * d;
          } else {
            s += d;
            const T F = BG ? m_rsqrt(E[p][v]) : T(1);
            D += A(0.5) * (A)beta * (A)(F * m_rsqrt(T(1) + xi));
          }
        }
      s = sum(s);
      if (what) {
        const A rms = sqrt(s / cells);
        bool stop;
        if (it < 0) {
          thr = fmax((A)o.crs_rel * rms, (A)o.crs_abs);
          stop = rms <= thr;
        } else {
          stop = rms <= thr || (o.crs_stall && rms >= prev);
        }
        prev = rms;
        if (stop) return;
      } else {
        D = sum(D);
        const A cp = (A)cap;
        A c = D > A(0) ? s / D : A(0);
        c = c > cp ? cp : (c < -cp ? -cp : c);
        __syncwarp();  // every cell has been read
#pragma unroll
        for (int p = 0; p < P; p++)
#pragma unroll
          for (int v = 0; v < 2; v++) {
            if (!mine[p]) continue;
            const T un = U[at[p][v]] + (T)c;
            U[at[p][v]] = un;
            X[at[p][v]] = m_expm1(un);
          }
        __syncwarp();
      }
    }
  }
}

// One V-cycle from level `skip` of every tail of the set down and up; one
// cluster per grid.
// The top level is read from u buffer pin and written to buffer pout.  norms
// (if not null, and the grid has a coarser level): entries 2g, 2g + 1 receive
// sum d^2 and max |d| of the top level after its pre-smoothing.
//
// Bound: latency of the dependent steps (at 2 GHz, plain form, 32^3 on 16
// blocks: 4600 cycles a colour at 32^3, 1850 at 16^3, 950 at 8^3; 15,000 for
// the coarsest solve at 4^3); barriers take 58 % of a warp's time.  The 32^3 tail
// takes 53 to 56 us (plain) and 67 us (correction form) with V(2,2), 40 to 43 and
// 52 to 60 us with V(1,1); its 35 launches took 240 us.  16 blocks per cluster are
// the fastest for up to 8 grids (8 blocks: 64 and 85 us); with more grids
// clusters of 8 let more of them run at once (28 patches of 32 to 64 cells:
// 120 against 133 us).
template <typename T, bool BG, bool DIR>
__global__ void __launch_bounds__(tail_threads<T>(), 1)
    k_tail(const TailDesc<T> *desc, int skip, int pin, int pout, TailOpts o, const int *active,
           double *norms) {
  constexpr int NT = tail_threads<T>();
  T *sm = tail_smem<T>();
  __shared__ TailBlock<T> B;
  const int cs = (int)cg::this_cluster().num_blocks(), me = (int)cg::this_cluster().block_rank();
  const int g = blockIdx.x / cs;
  const int tid = threadIdx.x;
  {
    const int *src = reinterpret_cast<const int *>(desc + g);
    int *dst = reinterpret_cast<int *>(&B.D);
    for (int t = tid; t < (int)(sizeof(TailDesc<T>) / sizeof(int)); t += NT) dst[t] = src[t];
  }
  __syncthreads();
  if (!grid_active(active, B.D.field)) return;  // the whole cluster
  const int nl = B.D.nl - skip;
  if (skip > 0) {
    // levels skip .. of the tail
    constexpr int NW = (int)(sizeof(TailLevel<T>) / sizeof(int));
    int *dst = reinterpret_cast<int *>(&B.D.lev[0]);
    for (int l = 0; l < nl; l++) {
      for (int t = tid; t < NW; t += NT) dst[l * NW + t] = dst[(l + skip) * NW + t];
      __syncthreads();
    }
  }
  if (tid < nl) {
    TailLevel<T> &L = B.D.lev[tid];
    L.z0 = min(me * L.zc, L.n2);
    L.np = min(L.zc, L.n2 - L.z0);
    // the own first plane is the upper copy of the block below, the own last
    // plane the lower copy of the block above
    const int lo = L.z0 > 0 ? L.z0 - 1 : L.n2 - 1;
    const int hi = L.z0 + L.np < L.n2 ? L.z0 + L.np : 0;
    L.below = tail_div(lo, L.mz);
    L.above = tail_div(hi, L.mz);
    L.belowo = (lo - L.below * L.zc + 2) * L.plane;
  }
  if (tid == 0) {
    B.cs = cs;
    B.me = me;
  }
  __syncthreads();
  const TailLevel<T> &L0 = B.D.lev[0];
  const long long c0 = (long long)L0.z0 * L0.plane;
  const int ntop = L0.np * L0.plane;
  if (ntop > 0) {
    // the top level's own planes and, from global memory too, the copied ones,
    // 16 bytes at a time (a plane holds a multiple of four cells) unless an
    // FP64 array of the caller's starts at an odd multiple of 8 bytes
    constexpr int W = 16 / (int)sizeof(T);
    const T *gu = L0.gu[pin], *gx = L0.gx[pin], *gf = L0.gf;
    const int pl = L0.plane, z0 = L0.z0, n2 = L0.n2, n = ntop + 2 * pl;
    const T fs = L0.fs, fo = L0.fo;
    auto cell = [&](int t) {
      const int kl = tail_div(tail_div(t, L0.m0), L0.m1) - 1;
      int k = z0 + kl;
      k = k < 0 ? k + n2 : (k >= n2 ? k - n2 : k);
      return k * pl + t - (kl + 1) * pl;
    };
    if (sizeof(T) == 4 ||
        ((reinterpret_cast<size_t>(gu) | reinterpret_cast<size_t>(gf)) & 15) == 0) {
      for (int t = W * tid; t < n; t += W * NT) {
        const int c = cell(t);
        const int4 vu = *reinterpret_cast<const int4 *>(gu + c);
        const int4 vx = *reinterpret_cast<const int4 *>(gx + c);
        int4 vb, vE;
        if (BG) {
          vb = *reinterpret_cast<const int4 *>(L0.gub + c);
          vE = *reinterpret_cast<const int4 *>(L0.gE + c);
        }
        *reinterpret_cast<int4 *>(sm + L0.u + t) = vu;
        *reinterpret_cast<int4 *>(sm + L0.x + t) = vx;
        if (BG) {
          *reinterpret_cast<int4 *>(sm + L0.ub + t) = vb;
          *reinterpret_cast<int4 *>(sm + L0.E + t) = vE;
        }
      }
      for (int t = W * tid; t < ntop; t += W * NT) {
        T v[W];
        *reinterpret_cast<int4 *>(v) = gf ? *reinterpret_cast<const int4 *>(gf + c0 + t)
                                          : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int q = 0; q < W; q++) v[q] = gf ? fs * (v[q] - fo) : T(0);
        *reinterpret_cast<int4 *>(sm + L0.f + t) = *reinterpret_cast<int4 *>(v);
      }
    } else {
      for (int t = tid; t < n; t += NT) {
        const int c = cell(t);
        sm[L0.u + t] = gu[c];
        sm[L0.x + t] = gx[c];
      }
      for (int t = tid; t < ntop; t += NT) sm[L0.f + t] = gf ? fs * (gf[c0 + t] - fo) : T(0);
    }
  }
  int lf = 0;  // first level kept in one block
  while (lf < nl && !B.D.lev[lf].local) lf++;
  tail_sync(2);
  if (BG) {
    // background of the coarser levels: mean of the 8 children, exponential
    for (int l = 1; l < nl; l++) {
      const TailLevel<T> &F = B.D.lev[l - 1], &C = B.D.lev[l];
      const TailPut<T, DIR> put(C);
      for (int t = tid; t < C.np * C.plane; t += NT) {
        int I, J, Kl;
        tail_ijk(C, t, I, J, Kl);
        T s = T(0);
#pragma unroll
        for (int cz = 0; cz < 2; cz++) {
          const int k = 2 * (C.z0 + Kl) + cz, r = tail_div(k, F.mz);
          const T *p = tail_remote(sm, r) + F.ub + (k - r * F.zc + 1) * F.plane + 2 * J * F.n0 +
                       2 * I;
          s += p[0];
          s += p[1];
          s += p[F.n0];
          s += p[F.n0 + 1];
        }
        const T ub = s * T(0.125);
        put(C.ub, ub, C.E, m_exp(ub), Kl, J * C.n0 + I);
      }
      if (l < lf) tail_sync(2);
      else __syncthreads();
    }
  }
  if (o.fas && (lf > 0 || me == 0)) tail_resid<T, BG, DIR>(B, 0, true, false, lf > 0 ? 2 : 1);
  // down: the levels dealt out to the cluster
  for (int l = 0; l < lf; l++) {
    if (l == nl - 1) {
      tail_coarsest<T, BG, DIR>(B, l, o, 2);
      break;
    }
    tail_smooth<T, BG, DIR>(B, l, o.pre, 2);
    tail_resid<T, BG, DIR>(B, l, false, norms && l == 0, 2);
    if (l + 1 < lf) {
      tail_restrict<T, DIR>(B, l, 2);
      tail_resid<T, BG, DIR>(B, l + 1, true, false, 2);
    }
  }
  // the levels of the first block, down and up
  if (lf < nl) {
    if (me == 0) {
      if (lf > 0) {
        tail_restrict<T, DIR>(B, lf - 1, 1);
        tail_resid<T, BG, DIR>(B, lf, true, false, 1);
      }
      for (int l = lf; l < nl - 1; l++) {
        tail_smooth<T, BG, DIR>(B, l, o.pre, 1);
        tail_resid<T, BG, DIR>(B, l, false, norms && l == 0, 1);
        tail_restrict<T, DIR>(B, l, 1);
        tail_resid<T, BG, DIR>(B, l + 1, true, false, 1);
      }
      const int nc = B.D.lev[nl - 1].n2 * B.D.lev[nl - 1].plane;
      if (nc > kTailWarp)
        tail_coarsest<T, BG, DIR>(B, nl - 1, o, 1);
      else if (tid < 32 && nc > 64)
        tail_coarsest_warp<T, BG, DIR, 2>(B, nl - 1, o);
      else if (tid < 32)
        tail_coarsest_warp<T, BG, DIR, 1>(B, nl - 1, o);
      __syncthreads();
      for (int l = nl - 2; l >= lf; l--) {
        tail_prolong<T, DIR>(B, l, 1);
        tail_smooth<T, BG, DIR>(B, l, o.post, 1);
      }
    }
    tail_sync(2);
  }
  // up: the cluster's levels
  for (int l = min(lf, nl - 1) - 1; l >= 0; l--) {
    tail_prolong<T, DIR>(B, l, 2);
    tail_smooth<T, BG, DIR>(B, l, o.post, 2);
  }
  {
    T *gu = L0.gu[pout], *gx = L0.gx[pout];
    for (int t = tid; t < ntop; t += NT) {
      gu[c0 + t] = sm[L0.u + L0.plane + t];
      if (o.keepx) gx[c0 + t] = sm[L0.x + L0.plane + t];
    }
  }
  if (norms && nl > 1 && me == 0 && tid == 0) {
    double s = 0.0, m = 0.0;
    for (int q = 0; q < (lf > 0 ? cs : 1); q++) {
      s += (double)B.nslot[2 * q];
      m = fmax(m, (double)B.nslot[2 * q + 1]);
    }
    norms[2 * g] = s;
    norms[2 * g + 1] = m;
  }
}

}  // namespace frmg
