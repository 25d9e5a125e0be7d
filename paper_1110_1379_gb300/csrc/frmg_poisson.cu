// frmg_poisson.cu -- the modified Poisson equation for the potential Phi.
//
// Sec. III.B gives the equation in code units and Eq. (discrete_poisson) its
// 7-point discretisation,
//   (1/h^2)[sum of the six neighbours - 6 phi_i] = s_i,
//   s_i = 2 Om a (rho_i - 1) - (1/6) Om a^4 [(n a^2 xi)^(1/(n+1)) e^{-u~_i/(n+1)}
//                                            - 3 (a^-3 + 4 OL/Om)],
// which for n = 1, in the f(R) solver's variable u = u~ - ubar (ubar: the
// homogeneous solution, where the bracket vanishes), reads
//   s_i = 2 gamma (rho_i - 1) - (beta/2) (e^{-u_i/2} - 1),
//   gamma = Om a,  beta = Om a^4 (a^-3 + 4 OL/Om).
// On a refinement patch a missing neighbour is the ghost 2 phi_b - phi_i
// (Eq. phi_b with mask ratio -1), which is Eq. (bc_modified_poisson).  The
// operator is linear, so the multigrid is the correction scheme of Sec. V.A.2:
// on coarser levels L^H e^H = R(s - L phi)^h with e = 0 on patch boundaries
// (Eq. bc_modified_poisson_coarse: only the left-hand side is modified), and
// e^h += P e^H with the trilinear 27/9/3/1 weights of Sec. V.A.3 (coarse cells
// outside a patch contribute 0).
//
// Precision follows the f(R) solve: phi, the source, the fine defect and its
// norm are double-float pairs (hi + lo, ~48-bit significands) on the FP32
// pipes, and the correction equation L e = -d is solved by FP32 V-cycles;
// phi += e.  On a periodic grid the equation has a solution only for a source
// of zero mean, so the source's mean is removed (and reported) and phi is
// returned with zero mean.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "frmg.h"
#include "frmg_dfmath.cuh"
#include "frmg_internal.h"
#include "frmg_perdevice.h"

using namespace frmg;

namespace {

struct PError {
  int status;
  std::string msg;
};

#define PCK(call)                                                                       \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess)                                                              \
      throw PError{FR_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)};       \
  } while (0)

#define PLAUNCH(ctx)                                                                    \
  do {                                                                                  \
    frmg_launch_counter(ctx)++;                                                         \
    cudaError_t e_ = cudaGetLastError();                                                \
    if (e_ != cudaSuccess)                                                              \
      throw PError{FR_ECUDA, std::string("kernel launch: ") + cudaGetErrorString(e_)};  \
  } while (0)

constexpr int kNT = 256;

long long nblk(long long n) { return (n + kNT - 1) / kNT; }

// ------------------------------------------------------------------ device
struct PLevel {
  float *e;        // correction (current buffer)
  float *e_alt;    // second buffer of the tiled smoother (null: not tiled)
  float *f;        // right-hand side of the correction equation
  int n0, n1, n2;
  long long ncell;
  FastDiv fd0, fd1;
  float h2;        // h^2
  float relax;     // relaxation factor of the smoother (1: Gauss-Seidel)
  int patch;       // 1: Dirichlet (ghost = -e on the boundary), 0: periodic
};

__device__ __forceinline__ void decomp(const PLevel &L, unsigned t, int &i, int &j, int &k) {
  const unsigned q = fdiv(t, L.fd0), q2 = fdiv(q, L.fd1);
  i = (int)(t - q * (unsigned)L.n0);
  j = (int)(q - q2 * (unsigned)L.n1);
  k = (int)q2;
}

// sum of the six neighbours of (i,j,k) and the number of missing ones (patch)
__device__ __forceinline__ float nbsum(const PLevel &L, const float *e, int i, int j, int k,
                                       long long c, int &nmiss) {
  const long long sy = L.n0, sz = (long long)L.n0 * L.n1;
  float s = 0.0f;
  nmiss = 0;
  if (L.patch) {
    if (i > 0) s += e[c - 1]; else nmiss++;
    if (i < L.n0 - 1) s += e[c + 1]; else nmiss++;
    if (j > 0) s += e[c - sy]; else nmiss++;
    if (j < L.n1 - 1) s += e[c + sy]; else nmiss++;
    if (k > 0) s += e[c - sz]; else nmiss++;
    if (k < L.n2 - 1) s += e[c + sz]; else nmiss++;
  } else {
    s += e[i > 0 ? c - 1 : c + (L.n0 - 1)];
    s += e[i < L.n0 - 1 ? c + 1 : c - (L.n0 - 1)];
    s += e[j > 0 ? c - sy : c + (L.n1 - 1) * sy];
    s += e[j < L.n1 - 1 ? c + sy : c - (L.n1 - 1) * sy];
    s += e[k > 0 ? c - sz : c + (L.n2 - 1) * sz];
    s += e[k < L.n2 - 1 ? c + sz : c - (L.n2 - 1) * sz];
  }
  return s;
}

// Gauss-Seidel value of a cell, (sum of its neighbours in the grid - h^2 f) /
// (6 + missing neighbours), with the diagonal's reciprocal as a constant (at
// most three neighbours are missing: every dimension is at least 2); every
// smoother uses this one expression.
__device__ __forceinline__ float gs_value(float sum, float h2f, int nm) {
  const float inv = nm == 0   ? 1.0f / 6.0f
                    : nm == 1 ? 1.0f / 7.0f
                    : nm == 2 ? 1.0f / 8.0f
                              : 1.0f / 9.0f;
  return (sum - h2f) * inv;
}

// Red-black Gauss-Seidel on L e = f (one colour per launch): with the ghosts
// -e_i on patch faces, e_i = (sum of the neighbours in the grid - h^2 f_i) / (6 + missing),
// over-relaxed as e_i += w (that value - e_i) when relax = w != 1.
__global__ void __launch_bounds__(kNT) k_lsmooth(PLevel L, int colour) {
  const long long half = L.ncell / 2;
  const long long t = (long long)blockIdx.x * kNT + threadIdx.x;
  if (t >= half) return;
  // cell 2t or 2t+1 along x, whichever has the colour (n0 even)
  int i, j, k;
  decomp(L, (unsigned)(2 * t), i, j, k);
  i += (i + j + k + colour) & 1;
  const long long c = ((long long)k * L.n1 + j) * L.n0 + i;
  int nm;
  const float s = nbsum(L, L.e, i, j, k, c, nm);
  const float gs = gs_value(s, L.h2 * L.f[c], nm);
  L.e[c] = fmaf(L.relax, gs - L.e[c], L.e[c]);
}

// Tiled red-black Gauss-Seidel on L e = f, one full sweep per pass (the
// schedule of the f(R) solver's tiled smoother): a block owns a 64 x 16 tile
// and a chunk of zc planes and marches along z with a ring of four planes of e
// and f in shared memory (the tile plus a halo of two cells).  At the step for
// plane p it updates the red cells of plane p-1 on the tile grown by one cell,
// then the black cells of plane p-2 on the tile, and writes plane p-2 to the
// other buffer (the halos are read from the unmodified input, so the pass
// equals one sweep of k_lsmooth).  Each plane is stored colour-split: per
// x-pair q = (ly, px) of the tile, array c holds the pair's cell of colour c
// (the even-x cell has colour (ly + z) & 1), so the six neighbours of a cell
// are the opposite colour's entries q, q -+ 1, q -+ PX of its own and the
// adjacent planes, and a warp's accesses (lane = x-pair) are contiguous.
// Warps update whole rows of the tile; the next plane is prefetched into
// registers during the updates.
template <bool PATCH>
__global__ void __launch_bounds__(256, 4) k_lsmooth_tiled(PLevel L, int zc) {
  constexpr int TX = 64, TY = 16, H = 2, LX = TX + 2 * H, LY = TY + 2 * H, PX = LX / 2;
  constexpr int PP = PX * LY, NW = TY / 2, NT = 32 * NW, NLD = (PP + NT - 1) / NT, NS = 4;
  constexpr int NE = TY + 2, PL = 2 * PP;
  __shared__ __align__(16) float se[NS * PL];  // [slot][colour][pair]
  __shared__ __align__(16) float sf[NS * PL];
  const int n0 = L.n0, n1 = L.n1, n2 = L.n2;
  const int ntx = (n0 + TX - 1) / TX, nty = (n1 + TY - 1) / TY;
  int b = blockIdx.x;
  const int X0 = (b % ntx) * TX;
  b /= ntx;
  const int Y0 = (b % nty) * TY;
  b /= nty;
  const int Z0 = b * zc, Z1 = min(Z0 + zc, n2);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long plane = (long long)n0 * n1;
  const float *__restrict__ ein = L.e;
  float *__restrict__ eout = L.e_alt;
  const float *__restrict__ fin = L.f;
  const float h2 = L.h2, relax = L.relax;
  auto wrapm = [](int v, int n) {
    int r = v % n;
    return r < 0 ? r + n : r;
  };
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
      bool ok = true;
      int gxw = gx, gyw = gy;
      if (PATCH) {
        ok = gx >= 0 && gx < n0 && gy >= 0 && gy < n1;
      } else {
        gxw = wrapm(gx, n0);
        gyw = wrapm(gy, n1);
      }
      const bool wr = ok && ly >= H && ly < H + TY && px >= 1 && px < PX - 1 && gx < n0 &&
                      gy < n1;
      roff[k] = ok ? gyw * n0 + gxw : 0;
      ldf[k] = (ok ? 1u : 0u) | (wr ? 2u : 0u) | ((unsigned)(ly & 1) << 2);
    }
  }
  float2 pe[NLD], pf[NLD];
#pragma unroll
  for (int k = 0; k < NLD; k++) {
    pe[k] = make_float2(0.f, 0.f);
    pf[k] = pe[k];
  }
  auto fetch = [&](long long zoff) {
#pragma unroll
    for (int k = 0; k < NLD; k++) {
      if (!(ldf[k] & 1u)) continue;
      pe[k] = *reinterpret_cast<const float2 *>(ein + zoff + roff[k]);
      pf[k] = *reinterpret_cast<const float2 *>(fin + zoff + roff[k]);
    }
  };
  // plane of parity pb into slot offset so
  auto commit = [&](int pb, int so) {
#pragma unroll
    for (int k = 0; k < NLD; k++) {
      const int q = threadIdx.x + k * NT;
      if (q >= PP) continue;
      const int c0 = (int)((ldf[k] >> 2) & 1u) ^ pb;
      se[so + c0 * PP + q] = pe[k].x;
      se[so + (c0 ^ 1) * PP + q] = pe[k].y;
      sf[so + c0 * PP + q] = pf[k].x;
      sf[so + (c0 ^ 1) * PP + q] = pf[k].y;
    }
  };
  // Gauss-Seidel update of the colour-Q cell of pair (ly, px) of plane m; s is
  // its x position in the pair; oc, om, op the slot offsets of planes m, m-1, m+1
  auto update = [&](int Q, int ly, int px, int s, int m, int oc, int om, int op) {
    const int gx = X0 - H + 2 * px + s, gy = Y0 - H + ly;
    if (PATCH && (gx < 0 || gx >= n0 || gy < 0 || gy >= n1)) return;
    const int e = ly * PX + px;
    const int cq = oc + Q * PP + e, V = oc + (Q ^ 1) * PP + e;
    const int o = (Q ^ 1) * PP + e;
    float sum = 0.0f;
    int nm = 0;
    if (!PATCH || gx > 0) sum += se[s ? V : V - 1]; else nm++;
    if (!PATCH || gx < n0 - 1) sum += se[s ? V + 1 : V]; else nm++;
    if (!PATCH || gy > 0) sum += se[V - PX]; else nm++;
    if (!PATCH || gy < n1 - 1) sum += se[V + PX]; else nm++;
    if (!PATCH || m > 0) sum += se[om + o]; else nm++;
    if (!PATCH || m < n2 - 1) sum += se[op + o]; else nm++;
    const float gs = gs_value(sum, h2 * sf[cq], nm);
    se[cq] = fmaf(relax, gs - se[cq], se[cq]);
  };
  const int P0 = Z0 - H, PE = Z1 + H;
  auto inr = [&](int pz) { return !PATCH || (pz >= 0 && pz < n2); };
  int pw = PATCH ? P0 : wrapm(P0, n2);
  if (inr(P0)) fetch((long long)pw * plane);
  commit(P0 & 1, 0);
  __syncthreads();
  int cur = 0;
  for (int p = P0; p < PE; p++) {
    const bool more = p + 1 < PE;
    pw = PATCH ? p + 1 : (pw + 1 == n2 ? 0 : pw + 1);
    if (more && inr(p + 1)) fetch((long long)pw * plane);
    const int o0 = cur * PL, o1 = ((cur + 3) & 3) * PL, o2 = ((cur + 2) & 3) * PL,
              o3 = ((cur + 1) & 3) * PL;  // planes p, p-1, p-2, p-3
    {
      const int m = p - 1;  // red cells, tile grown by one
      if (m >= Z0 - 1 && m < Z1 + 1 && inr(m)) {
        const int s = (w + p) & 1;  // rows 1 + w + j NW: (ly + m) & 1
#pragma unroll
        for (int j = 0; j < 3; j++) {
          if (j == 2 && w >= 2) break;
          update(0, 1 + w + j * NW, 1 + lane, s, m, o1, o2, o0);
        }
        if (w == 2 || w == 3) {
          const int idx = (w - 2) * 32 + lane;
          if (idx < NE) {
            const int ly = 1 + idx, se_ = (ly + m) & 1;
            update(0, ly, se_ ? 0 : PX - 1, se_, m, o1, o2, o0);
          }
        }
      }
    }
    __syncthreads();
    {
      const int m = p - 2;  // black cells, tile
      if (m >= Z0 && m < Z1 && inr(m)) {
        const int s = (w + m + 1) & 1;  // rows 2 + w + j NW: (ly + m + 1) & 1
#pragma unroll
        for (int j = 0; j < 2; j++) update(1, 2 + w + j * NW, 1 + lane, s, m, o2, o3, o1);
      }
    }
    __syncthreads();
    {
      const int wz = p - 2;
      if (wz >= Z0 && wz < Z1) {
        const long long woff = (long long)wz * plane;
#pragma unroll
        for (int k = 0; k < NLD; k++)
          if (ldf[k] & 2u) {
            const int q = threadIdx.x + k * NT;
            const int c0 = (int)((ldf[k] >> 2) & 1u) ^ (wz & 1);
            *reinterpret_cast<float2 *>(eout + woff + roff[k]) =
                make_float2(se[o2 + c0 * PP + q], se[o2 + (c0 ^ 1) * PP + q]);
          }
      }
    }
    if (more) commit((p + 1) & 1, o3);
    __syncthreads();
    cur = (cur + 1) & 3;
  }
}

// Residual d = f - L e of the 8 children of each coarse cell, averaged into
// the coarse right-hand side; coarse e = 0.  Optional per-block (sum d^2, max |d|).
__global__ void __launch_bounds__(kNT) k_lresid_restrict(PLevel F, PLevel C, double *partial) {
  const long long t = (long long)blockIdx.x * kNT + threadIdx.x;
  float ss = 0.0f, mx = 0.0f;
  if (t < C.ncell) {
    int I, J, K;
    decomp(C, (unsigned)t, I, J, K);
    float sd = 0.0f;
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int i = 2 * I + (q & 1), j = 2 * J + ((q >> 1) & 1), k = 2 * K + (q >> 2);
      const long long c = ((long long)k * F.n1 + j) * F.n0 + i;
      int nm;
      const float s = nbsum(F, F.e, i, j, k, c, nm);
      const float d = F.f[c] - (s - (6.0f + (float)nm) * F.e[c]) / F.h2;
      sd += d;
      ss = fmaf(d, d, ss);
      mx = fmaxf(mx, fabsf(d));
    }
    C.f[t] = 0.125f * sd;
    C.e[t] = 0.0f;
  }
  if (partial) {
    for (int o = 16; o > 0; o >>= 1) {
      ss += __shfl_down_sync(0xffffffffu, ss, o);
      mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
    }
    __shared__ float a[kNT / 32], b[kNT / 32];
    if ((threadIdx.x & 31) == 0) {
      a[threadIdx.x >> 5] = ss;
      b[threadIdx.x >> 5] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double s2 = 0.0;
      float m2 = 0.0f;
      for (int w = 0; w < kNT / 32; w++) {
        s2 += (double)a[w];
        m2 = fmaxf(m2, b[w]);
      }
      partial[2 * blockIdx.x] = s2;
      partial[2 * blockIdx.x + 1] = (double)m2;
    }
  }
}

// Asynchronous global-to-shared copies of 4, 8 and 16 bytes (PTX cp.async).
template <int N>
__device__ __forceinline__ void cp_async(void *smem, const void *gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  if constexpr (N == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(sa), "l"(gmem), "n"(N)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Tiled residual + restriction (the residuals of k_lresid_restrict): a block
// owns a 64 x 16 fine tile (32 x 8 coarse cells, one per thread) and a chunk
// of kc coarse planes, and marches over its fine planes.  They arrive by
// asynchronous copies in a ring of four, two ahead of the one in use (16 bytes
// a lane where rows are whole quads, else pairs); a thread keeps its 2 x 2 cells
// of three planes in registers, takes x neighbours by shuffles and the rows
// above and below from shared memory, and evaluates x-pairs as packed FP32
// pairs.  On a patch the cells outside are zeros, and counted.  Bound by HBM and
// the copies' latency; eight cells one by one from shared memory, f by scalar
// loads and a division each took 0.363 ms at 512^3, this 0.196 (the memory time
// of e, f and the coarse arrays is 0.18).  Optional per-block norm partials
// (sum d^2, max |d|).
constexpr int kLrTX = 64, kLrTY = 16;
template <bool PATCH>
__global__ void __launch_bounds__(256, 4) k_lresid_restrict_tiled(PLevel F, PLevel C, int kc,
                                                                  double *partial) {
  constexpr int TX = kLrTX, TY = kLrTY, NT = 256, NW = NT / 32;
  static_assert(TY == 2 * NW && TX == 64, "two rows per warp, one pair per lane");
  // a slot: rows -1 .. 16 of e, the columns left and right of the tile, rows 0 .. 15 of f
  constexpr int EC = (TY + 2) * TX, AN = EC + 2 * TY, PL = AN + TY * TX;
  __shared__ __align__(16) float smem[4 * PL];
  const int n0 = F.n0, n1 = F.n1, n2 = F.n2;
  const int ntx = (n0 + TX - 1) / TX, nty = (n1 + TY - 1) / TY;
  int b = blockIdx.x;
  const int X0 = (b % ntx) * TX;
  b /= ntx;
  const int Y0 = (b % nty) * TY;
  b /= nty;
  const int Z0 = 2 * b * kc, Z1 = min(Z0 + 2 * kc, n2);
  const long long plane = (long long)n0 * n1;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int gx = X0 + 2 * lane, gy = Y0 + 2 * w;
  const bool valid = gx < n0 && gy < n1;
  auto wrapm = [](int v, int n) {
    int r = v % n;
    return r < 0 ? r + n : r;
  };
  // What a lane copies of a plane (offsets, -1: none): 16 bytes of row 2 w
  // (lanes 0 - 15) or 2 w + 1, and of the row beyond the tile (first and last
  // warp), or pairs of both rows; the first and last lane also the cells left
  // and right of the tile.
  auto at = [&](int x, int y) -> int {
    if (PATCH) return x >= 0 && x < n0 && y >= 0 && y < n1 ? y * n0 + x : -1;
    return wrapm(y, n1) * n0 + wrapm(x, n0);
  };
  const bool quad = !(n0 & 3);
  const int lx = quad ? 4 * (lane & 15) : 2 * lane, ly = quad ? lane >> 4 : 0;
  const int o0 = at(X0 + lx, gy + ly);
  const int oh = w == 0 && !(quad && ly) ? at(X0 + lx, gy - 1)
                 : (w == NW - 1 && !(quad && ly) ? at(X0 + lx, gy + 2) : -1);
  const int ex = lane == 0 ? X0 - 1 : X0 + TX;
  const bool edge = lane == 0 || lane == 31;
  const int oe = edge ? at(ex, gy) : -1;  // (and the row above: n1 is even)
  const int qc = (2 * w + 1 + ly) * TX + lx;
  const int qh = (w == 0 ? 0 : TY + 1) * TX + lx;
  const int qe = EC + (lane == 0 ? 0 : TY) + 2 * w;
  const int q0 = (2 * w + 1) * TX + 2 * lane;
  auto inz = [&](int p) { return !PATCH || (p >= 0 && p < n2); };
  if (PATCH) {  // what lies outside the grid is never copied to
    for (int q = threadIdx.x; q < 4 * PL; q += NT) smem[q] = 0.0f;
    __syncthreads();
  }
  auto fetch = [&](int p) {
    if (p <= Z1 && inz(p)) {
      const bool own = p >= Z0 && p < Z1;
      const long long zo = (long long)(PATCH ? p : (p < 0 ? p + n2 : (p >= n2 ? p - n2 : p))) * plane;
      float *h = smem + ((p - Z0 + 1) & 3) * PL;
      const float *v = F.e + zo, *fv = F.f + zo;
      if (quad) {
        if (o0 >= 0) {
          cp_async<16>(h + qc, v + o0);
          if (own) cp_async<16>(h + AN + qc - TX, fv + o0);
        }
        if (own && oh >= 0) cp_async<16>(h + qh, v + oh);
      } else {
        if (o0 >= 0) {
          cp_async<8>(h + qc, v + o0);
          cp_async<8>(h + qc + TX, v + o0 + n0);
          if (own) {
            cp_async<8>(h + AN + qc - TX, fv + o0);
            cp_async<8>(h + AN + qc, fv + o0 + n0);
          }
        }
        if (own && oh >= 0) cp_async<8>(h + qh, v + oh);
      }
      if (own && oe >= 0) {
        cp_async<4>(h + qe, v + oe);
        cp_async<4>(h + qe + 1, v + oe + n0);
      }
    }
    cp_async_commit();
  };
  auto ld2 = [](const float *p) { return *reinterpret_cast<const float2 *>(p); };
  const float h2 = F.h2, rh2 = 1.0f / h2;
  float2 sd = make_float2(0.f, 0.f), s2 = sd;
  float mx = 0.0f;
  float2 r[4][2];  // the own rows of planes m - 1, m, m + 1 (by plane modulo 4)
  r[3][0] = r[3][1] = r[2][0] = r[2][1] = sd;

  auto step = [&](auto Kc, int p) {
    constexpr int K = decltype(Kc)::value, K1 = (K + 3) & 3, K2 = (K + 2) & 3;
    fetch(p + 2);  // into the slot of plane p - 2, last read before the last barrier
    cp_async_wait<2>();
    __syncwarp();  // a warp's rows are copied by all of its lanes
#pragma unroll
    for (int k = 0; k < 2; k++)
      r[K][k] = inz(p) ? ld2(smem + K * PL + q0 + k * TX) : make_float2(0.f, 0.f);
    const int m = p - 1;
    if (m >= Z0) {
      const float *sm = smem + K1 * PL;
#pragma unroll
      for (int k = 0; k < 2; k++) {
        const float2 own = r[K1][k];
        float lo = __shfl_up_sync(0xffffffffu, own.y, 1);
        float hi = __shfl_down_sync(0xffffffffu, own.x, 1);
        if (edge) (lane == 0 ? lo : hi) = sm[qe + k];
        const float2 V = ld2(sm + q0 + (k ? 2 * TX : -TX));
        float2 R = make_float2(own.y, hi);
        float2 cnt = make_float2(6.0f, 6.0f);
        if (PATCH) {
          // lanes at the end of a ragged row: the pair beyond it holds zeros
          const float my = (float)((gy + k == 0) + (gy + k == n1 - 1) + (m == 0) + (m == n2 - 1));
          cnt.x += my + (float)(gx == 0);
          cnt.y += my + (float)(gx + 2 == n0);
        }
        float2 t = add2(make_float2(lo, own.x), R);
        t = add2(t, k ? r[K1][0] : V);
        t = add2(t, k ? V : r[K1][1]);
        t = add2(t, r[K2][k]);
        t = add2(t, r[K][k]);
        // one rounding, as in k_lresid_restrict: with 6 e rounded first, a large
        // constant part of e (free on a periodic grid) left a residual of its own
        t = fma2(make_float2(-cnt.x, -cnt.y), own, t);
        // t / h^2: the product with the rounded reciprocal and one correction
        // by its exact remainder (Markstein 1990)
        float2 q = mul2(t, splat2(rh2));
        q = fma2(fma2(q, splat2(-h2), t), splat2(rh2), q);
        const float2 d = sub2(ld2(sm + AN + q0 + (k - 1) * TX), q);
        if (valid) {
          sd = add2(sd, d);
          s2 = fma2(d, d, s2);
          mx = fmaxf(mx, fmaxf(fabsf(d.x), fabsf(d.y)));
        }
      }
      if (((m - Z0) & 1) && valid) {
        const long long t = ((long long)(m >> 1) * C.n1 + (gy >> 1)) * C.n0 + (gx >> 1);
        C.f[t] = 0.125f * (sd.x + sd.y);
        C.e[t] = 0.0f;
        sd = make_float2(0.f, 0.f);
      }
    }
    __syncthreads();
  };
  fetch(Z0 - 1);
  fetch(Z0);
  for (int p = Z0 - 1; p <= Z1; p += 4) {  // an even number of planes
    step(std::integral_constant<int, 0>{}, p);
    step(std::integral_constant<int, 1>{}, p + 1);
    if (p + 2 <= Z1) {
      step(std::integral_constant<int, 2>{}, p + 2);
      step(std::integral_constant<int, 3>{}, p + 3);
    }
  }
  cp_async_wait<0>();
  float ss = s2.x + s2.y;
  if (partial) {
    for (int o = 16; o > 0; o >>= 1) {
      ss += __shfl_down_sync(0xffffffffu, ss, o);
      mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
    }
    __shared__ float a[NT / 32], bm[NT / 32];
    if ((threadIdx.x & 31) == 0) {
      a[threadIdx.x >> 5] = ss;
      bm[threadIdx.x >> 5] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double s2 = 0.0;
      float m2 = 0.0f;
      for (int w = 0; w < NT / 32; w++) {
        s2 += (double)a[w];
        m2 = fmaxf(m2, bm[w]);
      }
      partial[2 * blockIdx.x] = s2;
      partial[2 * blockIdx.x + 1] = (double)m2;
    }
  }
}

// e^h += P e^H: trilinear, per axis 3/4 on the containing coarse cell and 1/4
// on the neighbour on the child's side (products: 27/9/3/1 over 64).
__global__ void __launch_bounds__(kNT) k_lprolong(PLevel F, PLevel C) {
  const long long t = (long long)blockIdx.x * kNT + threadIdx.x;
  if (t >= F.ncell) return;
  int i, j, k;
  decomp(F, (unsigned)t, i, j, k);
  const int I = i >> 1, J = j >> 1, K = k >> 1;
  const int di = (i & 1) ? 1 : -1, dj = (j & 1) ? 1 : -1, dk = (k & 1) ? 1 : -1;
  float acc = 0.0f;
#pragma unroll
  for (int q = 0; q < 8; q++) {
    int ii = I + ((q & 1) ? di : 0), jj = J + (((q >> 1) & 1) ? dj : 0),
        kk = K + ((q >> 2) ? dk : 0);
    const float w = ((q & 1) ? 0.25f : 0.75f) * (((q >> 1) & 1) ? 0.25f : 0.75f) *
                    ((q >> 2) ? 0.25f : 0.75f);
    bool in = true;
    if (C.patch) {
      in = ii >= 0 && ii < C.n0 && jj >= 0 && jj < C.n1 && kk >= 0 && kk < C.n2;
    } else {
      ii = ii < 0 ? ii + C.n0 : (ii >= C.n0 ? ii - C.n0 : ii);
      jj = jj < 0 ? jj + C.n1 : (jj >= C.n1 ? jj - C.n1 : jj);
      kk = kk < 0 ? kk + C.n2 : (kk >= C.n2 ? kk - C.n2 : kk);
    }
    if (in) acc = fmaf(w, C.e[((long long)kk * C.n1 + jj) * C.n0 + ii], acc);
  }
  F.e[t] += acc;
}

// Tiled e^h += P e^H (the interpolation of k_lprolong, evaluated in the order
// z, y, x): a block owns a 64 x 16 fine tile (32 x 8 coarse cells) and a chunk
// of kc coarse planes; the coarse tile plus a one-cell halo is staged in
// shared memory for planes K-1, K, K+1 (ring of three), the z-interpolated
// plane is formed once per fine plane, and each thread corrects fine x-pairs
// with 8-byte loads and stores.  Patches: coarse cells outside the grid
// contribute 0.
constexpr int kLpTX = 64, kLpTY = 16;
template <bool PATCH>
__global__ void __launch_bounds__(256) k_lprolong_tiled(PLevel F, PLevel C, int kc) {
  constexpr int CX = kLpTX / 2 + 2, CY = kLpTY / 2 + 2, CP = CX * CY;
  constexpr int NQ = (CP + 255) / 256;
  __shared__ float se[3][CP];
  __shared__ float sz[CP];
  const int n0 = F.n0, n1 = F.n1;
  const int c0 = C.n0, c1 = C.n1, c2 = C.n2;
  const float *__restrict__ eH = C.e;
  float *__restrict__ ef = F.e;
  const int ntx = (n0 + kLpTX - 1) / kLpTX, nty = (n1 + kLpTY - 1) / kLpTY;
  int b = blockIdx.x;
  const int X0 = (b % ntx) * kLpTX;
  b /= ntx;
  const int Y0 = (b % nty) * kLpTY;
  b /= nty;
  const int K0 = b * kc, K1 = min(K0 + kc, c2);
  auto wrapm = [](int v, int n) {
    int r = v % n;
    return r < 0 ? r + n : r;
  };
  int qoff[NQ];
  bool qok[NQ];
#pragma unroll
  for (int k = 0; k < NQ; k++) {
    const int q = threadIdx.x + k * 256;
    qoff[k] = 0;
    qok[k] = false;
    if (q < CP) {
      int I = X0 / 2 - 1 + q % CX, J = Y0 / 2 - 1 + q / CX;
      if (PATCH) {
        qok[k] = I >= 0 && I < c0 && J >= 0 && J < c1;
      } else {
        I = wrapm(I, c0);
        J = wrapm(J, c1);
        qok[k] = true;
      }
      qoff[k] = J * c0 + I;
    }
  }
  const long long cplane = (long long)c0 * c1;
  int kw = PATCH ? K0 - 1 : wrapm(K0 - 1, c2);  // wrapped index of the next plane staged
  auto stage = [&](int slot, int K) {
    const bool vz = !PATCH || (K >= 0 && K < c2);
    const long long zo = (long long)kw * cplane;
#pragma unroll
    for (int k = 0; k < NQ; k++) {
      const int q = threadIdx.x + k * 256;
      if (q >= CP) continue;
      se[slot][q] = (qok[k] && vz) ? eH[zo + qoff[k]] : 0.0f;
    }
    kw = PATCH ? kw + 1 : (kw + 1 == c2 ? 0 : kw + 1);
  };
  const int lane = threadIdx.x & 31, r0 = threadIdx.x >> 5;
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
        const float2 v = *reinterpret_cast<const float2 *>(ef + fi);
        *reinterpret_cast<float2 *>(ef + fi) =
            make_float2(v.x + (w3 * e0 + w1 * em), v.y + (w3 * e0 + w1 * ep));
      }
      __syncthreads();
    }
    const int t = sm;
    sm = sc;
    sc = sp;
    sp = t;
  }
}

// Coarsest level: one block, red-black sweeps until the rms residual falls by
// 1e-3 of its value before the first sweep (at most maxit sweeps) or stops falling.
__global__ void __launch_bounds__(kNT) k_lcoarsest(PLevel L, int maxit) {
  __shared__ float red[kNT / 32];
  __shared__ float r0s, rprev;
  auto rms = [&]() -> float {
    float ss = 0.0f;
    for (long long c = threadIdx.x; c < L.ncell; c += kNT) {
      int i, j, k;
      decomp(L, (unsigned)c, i, j, k);
      int nm;
      const float s = nbsum(L, L.e, i, j, k, c, nm);
      const float d = L.f[c] - (s - (6.0f + (float)nm) * L.e[c]) / L.h2;
      ss = fmaf(d, d, ss);
    }
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_down_sync(0xffffffffu, ss, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.0f;
    for (int w = 0; w < kNT / 32; w++) tot += red[w];
    __syncthreads();
    return sqrtf(tot / (float)L.ncell);
  };
  const float r0 = rms();
  if (threadIdx.x == 0) {
    r0s = r0;
    rprev = r0;
  }
  __syncthreads();
  for (int it = 0; it < maxit; it++) {
    for (int colour = 0; colour < 2; colour++) {
      for (long long t = threadIdx.x; t < L.ncell / 2; t += kNT) {
        int i, j, k;
        decomp(L, (unsigned)(2 * t), i, j, k);
        i += (i + j + k + colour) & 1;
        const long long c = ((long long)k * L.n1 + j) * L.n0 + i;
        int nm;
        const float s = nbsum(L, L.e, i, j, k, c, nm);
        L.e[c] = gs_value(s, L.h2 * L.f[c], nm);
      }
      __syncthreads();
    }
    const float r = rms();
    const bool stop = r <= 1e-3f * r0s || !(r < rprev);
    __syncthreads();
    if (threadIdx.x == 0) rprev = r;
    __syncthreads();
    if (stop) break;
  }
}

// ---- the small levels of a V-cycle in one cluster
//
// As the f(R) solver's tail (frmg_tail.cuh): the levels from one of at most
// kLtCells cells down to the coarsest and back up run in one launch, each
// level's planes dealt out to the blocks of one thread-block cluster, e and f in
// shared memory, with copies of the e planes above and below a block's own
// that their owner keeps up to date; levels of at most kLtLocal cells live in the
// first block.  A launch per step costs 3 to 4 us of host and launch time on
// these levels, ten steps per level (V(2,2)).  Same updates as k_lsmooth, k_lresid_restrict,
// k_lprolong and k_lcoarsest (whose sums are added in another order).
namespace cg = cooperative_groups;

constexpr int kLtNT = 512, kLtLev = 8, kLtCluster = 16;
constexpr long long kLtCells = 110592;  // 48^3: what fits 16 blocks' shared memory
constexpr int kLtLocal = 4096;          // 16^3: a step of one block is shorter than a barrier

struct LtLevel {
  int n0, n1, n2, hx, plane, zc, local;
  unsigned e, f, d, g;       // arrays in shared memory: e (with the copies), f, residual,
                             // the coarser level's correction that the own planes take
  unsigned mh, m0, m1, mz;   // division by hx, n0, n1, zc: (t m) >> 32
  float h2;
  float *ge, *gf;            // the level's arrays in global memory
  int z0, np, below, above, belowo;
};
struct LtDesc {
  int nl, patch, pre, post;
  float relax;
  LtLevel lev[kLtLev];
};

// Lays out nl levels on clusters of cs blocks; returns the bytes per block.
size_t lt_layout(LtDesc &D, const PLevel *lev, int nl, int cs) {
  auto magic = [](int d) {
    return d <= 1 ? 0u : (unsigned)(((1ull << 32) + (unsigned)d - 1) / (unsigned)d);
  };
  unsigned end = 0;
  D.nl = nl;
  for (int l = 0; l < nl; l++) {
    LtLevel &L = D.lev[l];
    const PLevel &G = lev[l];
    L.n0 = G.n0;
    L.n1 = G.n1;
    L.n2 = G.n2;
    L.hx = G.n0 / 2;
    L.plane = G.n0 * G.n1;
    L.local = G.ncell <= kLtLocal;
    L.zc = L.local ? G.n2 : (G.n2 + cs - 1) / cs;
    L.mh = magic(L.hx);
    L.m0 = magic(L.n0);
    L.m1 = magic(L.n1);
    L.mz = magic(L.zc);
    L.h2 = G.h2;
    L.ge = G.e;
    L.gf = G.f;
    L.e = end;
    L.f = L.e + (unsigned)((L.zc + 2) * L.plane);
    L.d = L.f + (unsigned)(L.zc * L.plane);
    L.g = L.d + (unsigned)(L.zc * L.plane);
    end = L.g + (unsigned)((L.zc / 2 + 3) * (L.plane / 4 + 1));
  }
  return (size_t)end * sizeof(float);
}

struct LtBlock {
  LtDesc D;
  int cs, me;
  float red[kLtNT / 32], slots[kLtCluster];
};

__device__ __forceinline__ float *lt_smem() {
  extern __shared__ __align__(16) float lt_smem_raw[];
  return lt_smem_raw;
}
__device__ __forceinline__ void lt_sync(bool all) {
  if (all) cg::this_cluster().sync();
  else __syncthreads();
}
__device__ __forceinline__ float *lt_remote(float *p, int r) {
  return cg::this_cluster().map_shared_rank(p, r);
}
__device__ __forceinline__ int lt_div(int t, unsigned m) {
  return m ? (int)__umulhi((unsigned)t, m) : t;
}

// Writes e of the own planes, and the neighbours' copies of the outer ones.
template <bool PATCH>
struct LtPut {
  float *sm, *below, *above;
  int plane, last, belowo;
  unsigned e;
  __device__ __forceinline__ explicit LtPut(const LtLevel &L)
      : sm(lt_smem()), plane(L.plane), last(L.np - 1), belowo(L.belowo), e(L.e) {
    below = PATCH && L.z0 == 0 ? nullptr : lt_remote(sm, L.below);
    above = PATCH && L.z0 + L.np == L.n2 ? nullptr : lt_remote(sm, L.above);
  }
  __device__ __forceinline__ void operator()(float v, int kl, int q) const {
    sm[e + (kl + 1) * plane + q] = v;
    if (kl == 0 && (!PATCH || below)) below[e + belowo + q] = v;
    if (kl == last && (!PATCH || above)) above[e + q] = v;
  }
};

// Sum of the six neighbours (in the grid) of cell (i, j) of own plane kl.
template <bool PATCH>
__device__ __forceinline__ float lt_nbsum(const LtLevel &L, int i, int j, int kl, float &own,
                                          int &nm) {
  const float *sm = lt_smem();
  const int n0 = L.n0, pl = L.plane, o = (int)L.e + (kl + 1) * pl + j * n0 + i;
  const bool b[6] = {i == 0, i == n0 - 1, j == 0, j == L.n1 - 1, L.z0 + kl == 0,
                     L.z0 + kl == L.n2 - 1};
  const int wx = n0 - 1, wy = pl - n0;
  const float v[6] = {sm[b[0] ? o + wx : o - 1],  sm[b[1] ? o - wx : o + 1],
                      sm[b[2] ? o + wy : o - n0], sm[b[3] ? o - wy : o + n0],
                      sm[o - pl],                 sm[o + pl]};
  own = sm[o];
  float s = 0.0f;
  nm = 0;
#pragma unroll
  for (int q = 0; q < 6; q++) {
    if (PATCH && b[q]) nm++;
    else s += v[q];
  }
  return s;
}

template <bool PATCH>
__device__ __noinline__ void lt_smooth(const LtBlock &B, int l, int sweeps, float relax,
                                       bool all) {
  const LtLevel &L = B.D.lev[l];
  const float *sm = lt_smem();
  const LtPut<PATCH> put(L);
  const int n = L.np * L.n1 * L.hx;
  for (int s = 0; s < 2 * sweeps; s++) {
    for (int t = threadIdx.x; t < n; t += kLtNT) {
      const int q = lt_div(t, L.mh), kl = lt_div(q, L.m1), j = q - kl * L.n1;
      const int i = 2 * (t - q * L.hx) + ((j + L.z0 + kl + s) & 1);
      float own;
      int nm;
      const float sum = lt_nbsum<PATCH>(L, i, j, kl, own, nm);
      const float gs = gs_value(sum, L.h2 * sm[L.f + kl * L.plane + j * L.n0 + i], nm);
      put(fmaf(relax, gs - own, own), kl, j * L.n0 + i);
    }
    lt_sync(all);
  }
}

// d = f - L e on the own planes; returns this thread's sum of d^2.
template <bool PATCH>
__device__ __noinline__ float lt_resid(const LtBlock &B, int l) {
  const LtLevel &L = B.D.lev[l];
  float *sm = lt_smem();
  const int n = L.np * L.plane;
  float ss = 0.0f;
  for (int t = threadIdx.x; t < n; t += kLtNT) {
    const int q = lt_div(t, L.m0), kl = lt_div(q, L.m1), j = q - kl * L.n1, i = t - q * L.n0;
    float own;
    int nm;
    const float sum = lt_nbsum<PATCH>(L, i, j, kl, own, nm);
    const float d = sm[L.f + t] - (sum - (6.0f + (float)nm) * own) / L.h2;
    sm[L.d + t] = d;
    ss = fmaf(d, d, ss);
  }
  return ss;
}

// f of level l + 1 = mean of the children's d, e = 0 (own planes and copies)
__device__ __noinline__ void lt_restrict(const LtBlock &B, int l, bool all) {
  const LtLevel &F = B.D.lev[l], &C = B.D.lev[l + 1];
  float *sm = lt_smem();
  const int n = C.np * C.plane;
  if (n > 0)
    for (int t = threadIdx.x; t < n + 2 * C.plane; t += kLtNT) sm[C.e + t] = 0.0f;
  for (int t = threadIdx.x; t < n; t += kLtNT) {
    const int q = lt_div(t, C.m0), Kl = lt_div(q, C.m1), J = q - Kl * C.n1, I = t - q * C.n0;
    float sd = 0.0f;
#pragma unroll
    for (int z = 0; z < 2; z++) {
      const int k = 2 * (C.z0 + Kl) + z, r = lt_div(k, F.mz);
      const float *p = lt_remote(sm, r) + F.d + (k - r * F.zc) * F.plane + 2 * J * F.n0 + 2 * I;
      sd += p[0];
      sd += p[1];
      sd += p[F.n0];
      sd += p[F.n0 + 1];
    }
    sm[C.f + t] = 0.125f * sd;
  }
  lt_sync(all);
}

template <bool PATCH>
__device__ __noinline__ void lt_prolong(const LtBlock &B, int l, bool all) {
  const LtLevel &F = B.D.lev[l], &C = B.D.lev[l + 1];
  float *sm = lt_smem();
  const int n = F.np * F.plane, K0 = (F.z0 >> 1) - 1;
  if (n > 0) {
    const int ne = (((F.z0 + F.np - 1) >> 1) + 2 - K0) * C.plane;
    for (int t = threadIdx.x; t < ne; t += kLtNT) {
      const int s = lt_div(lt_div(t, C.m0), C.m1), q = t - s * C.plane;
      int K = K0 + s;
      const bool out = K < 0 || K >= C.n2;
      K = K < 0 ? K + C.n2 : (K >= C.n2 ? K - C.n2 : K);
      const int r = lt_div(K, C.mz);
      const float v = lt_remote(sm, r)[C.e + (K - r * C.zc + 1) * C.plane + q];
      sm[F.g + t] = PATCH && out ? 0.0f : v;
    }
  }
  __syncthreads();
  const LtPut<PATCH> put(F);
  for (int t = threadIdx.x; t < n; t += kLtNT) {
    const int q = lt_div(t, F.m0), kl = lt_div(q, F.m1), j = q - kl * F.n1, i = t - q * F.n0;
    const int k = F.z0 + kl, I = i >> 1, J = j >> 1, K = k >> 1;
    const int di = (i & 1) ? 1 : -1, dj = (j & 1) ? 1 : -1, dk = (k & 1) ? 1 : -1;
    float acc = 0.0f;
#pragma unroll
    for (int c = 0; c < 8; c++) {
      int ii = I + ((c & 1) ? di : 0), jj = J + (((c >> 1) & 1) ? dj : 0);
      const int kk = K + ((c >> 2) ? dk : 0);
      const float w = ((c & 1) ? 0.25f : 0.75f) * (((c >> 1) & 1) ? 0.25f : 0.75f) *
                      ((c >> 2) ? 0.25f : 0.75f);
      const bool in = !PATCH || (ii >= 0 && ii < C.n0 && jj >= 0 && jj < C.n1);
      ii = ii < 0 ? ii + C.n0 : (ii >= C.n0 ? ii - C.n0 : ii);
      jj = jj < 0 ? jj + C.n1 : (jj >= C.n1 ? jj - C.n1 : jj);
      const float v = sm[F.g + (kk - K0) * C.plane + jj * C.n0 + ii];
      if (in) acc = fmaf(w, v, acc);
    }
    put(sm[F.e + F.plane + t] + acc, kl, t - kl * F.plane);
  }
  lt_sync(all);
}

// Gauss-Seidel sweeps to k_lcoarsest's stopping rule.
template <bool PATCH>
__device__ __noinline__ void lt_coarsest(LtBlock &B, int l, int maxit, bool all) {
  const float cells = (float)(B.D.lev[l].n2 * B.D.lev[l].plane);
  float r0 = 0.0f, prev = 0.0f;
  for (int it = -1; it < maxit; it++) {
    if (it >= 0) lt_smooth<PATCH>(B, l, 1, 1.0f, all);
    float ss = lt_resid<PATCH>(B, l);
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const int lane = threadIdx.x & 31;
    if (lane == 0) B.red[threadIdx.x >> 5] = ss;
    __syncthreads();
    ss = lane < kLtNT / 32 ? B.red[lane] : 0.0f;
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (all) {
      if ((int)threadIdx.x < B.cs) lt_remote(B.slots, threadIdx.x)[B.me] = ss;
      lt_sync(true);
      ss = 0.0f;
      for (int q = 0; q < B.cs; q++) ss += B.slots[q];
    }
    const float r = sqrtf(ss / cells);
    lt_sync(all);  // the sums have been read
    if (it < 0) r0 = r;
    else if (r <= 1e-3f * r0 || !(r < prev)) return;
    prev = r;
  }
}

template <bool PATCH>
__global__ void __launch_bounds__(kLtNT, 1) k_ltail(const LtDesc *desc) {
  __shared__ LtBlock B;
  float *sm = lt_smem();
  const int tid = threadIdx.x;
  const int cs = (int)cg::this_cluster().num_blocks(), me = (int)cg::this_cluster().block_rank();
  {
    const int *src = reinterpret_cast<const int *>(desc);
    int *dst = reinterpret_cast<int *>(&B.D);
    for (int t = tid; t < (int)(sizeof(LtDesc) / sizeof(int)); t += kLtNT) dst[t] = src[t];
  }
  __syncthreads();
  const int nl = B.D.nl, pre = B.D.pre, post = B.D.post;
  const float relax = B.D.relax;
  if (tid < nl) {
    LtLevel &L = B.D.lev[tid];
    L.z0 = min(me * L.zc, L.n2);
    L.np = min(L.zc, L.n2 - L.z0);
    const int lo = L.z0 > 0 ? L.z0 - 1 : L.n2 - 1;
    const int hi = L.z0 + L.np < L.n2 ? L.z0 + L.np : 0;
    L.below = lt_div(lo, L.mz);
    L.above = lt_div(hi, L.mz);
    L.belowo = (lo - L.below * L.zc + 2) * L.plane;
  }
  if (tid == 0) {
    B.cs = cs;
    B.me = me;
  }
  __syncthreads();
  const LtLevel &T = B.D.lev[0];
  const long long c0 = (long long)T.z0 * T.plane;
  const int ntop = T.np * T.plane;
  // the top level: f from global memory, e = 0
  for (int t = tid; t < ntop; t += kLtNT) sm[T.f + t] = T.gf[c0 + t];
  if (ntop > 0)
    for (int t = tid; t < ntop + 2 * T.plane; t += kLtNT) sm[T.e + t] = 0.0f;
  int lf = 0;  // first level kept in one block
  while (lf < nl && !B.D.lev[lf].local) lf++;
  lt_sync(true);
  for (int l = 0; l < lf; l++) {
    if (l == nl - 1) {
      lt_coarsest<PATCH>(B, l, 500, true);
      break;
    }
    lt_smooth<PATCH>(B, l, pre, relax, true);
    lt_resid<PATCH>(B, l);
    lt_sync(true);
    if (l + 1 < lf) lt_restrict(B, l, true);
  }
  if (lf < nl) {
    if (me == 0) {
      if (lf > 0) lt_restrict(B, lf - 1, false);
      for (int l = lf; l < nl - 1; l++) {
        lt_smooth<PATCH>(B, l, pre, relax, false);
        lt_resid<PATCH>(B, l);
        __syncthreads();
        lt_restrict(B, l, false);
      }
      lt_coarsest<PATCH>(B, nl - 1, 500, false);
      for (int l = nl - 2; l >= lf; l--) {
        lt_prolong<PATCH>(B, l, false);
        lt_smooth<PATCH>(B, l, post, relax, false);
      }
    }
    lt_sync(true);
  }
  for (int l = min(lf, nl - 1) - 1; l >= 0; l--) {
    lt_prolong<PATCH>(B, l, true);
    lt_smooth<PATCH>(B, l, post, relax, true);
  }
  for (int t = tid; t < ntop; t += kLtNT) T.ge[c0 + t] = sm[T.e + T.plane + t];
}

// Blocks per cluster the current device takes (16 where it can); also sets the
// kernel's attributes there.
constexpr size_t kLtSmem = 220 * 1024;
template <bool PATCH>
int lt_cluster() {
  static PerDevice<int> best;
  int dev = 0;
  PCK(cudaGetDevice(&dev));
  return best.get(dev, []() {
    auto *k = k_ltail<PATCH>;
    PCK(cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    PCK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLtSmem));
    for (int cs = kLtCluster; cs > 0; cs /= 2) {
      cudaLaunchConfig_t c = {};
      c.gridDim = dim3(cs);
      c.blockDim = dim3(kLtNT);
      c.dynamicSmemBytes = kLtSmem;
      cudaLaunchAttribute a[1];
      a[0].id = cudaLaunchAttributeClusterDimension;
      a[0].val.clusterDim.x = cs;
      a[0].val.clusterDim.y = a[0].val.clusterDim.z = 1;
      c.attrs = a;
      c.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k, &c) == cudaSuccess && n > 0) return cs;
      cudaGetLastError();
    }
    return 1;
  });
}

// ---- double-float fine level

struct PFine {
  float2 *phi;         // phi (hi, lo)
  float2 *s;           // source (hi, lo)
  const double *phib;  // patch faces (FP64) or null
  long long foff[6];
  int n0, n1, n2;
  long long ncell;
  FastDiv fdh, fd1;    // division by n0 / 2 and n1
  float ih2h, ih2l;    // 1/h^2 as a double-float pair
};

// Sum of v over NV values of a block's shared array, one per lane of its first
// warp, in FP64; on lane 0.
template <int NV>
__device__ __forceinline__ double warp_sum64(const double *v) {
  const int lane = threadIdx.x & 31;
  double s = lane < NV ? v[lane] : 0.0;
  for (int o = NV / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// Block (sum, max) of a double-float per-thread value (of four cells): partial[2
// b] = sum (as FP64), partial[2 b + 1] = max |value| (the max is taken on the
// high parts).  Eight threads' values are added as pairs, the 32 sums of such
// groups in FP64 (five FP64 warp instructions per 1024 cells).
__device__ __forceinline__ void block_df_partial(df v, float amax, double *partial) {
  __shared__ double ws[kNT / 8];
  __shared__ float wm[kNT / 32];
  static_assert(kNT / 8 == 32, "one group per lane");
  for (int o = 4; o > 0; o >>= 1) {
    const df w = {__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)};
    v = df_add(v, w);
  }
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  const int lane = threadIdx.x & 31;
  if ((lane & 7) == 0) ws[threadIdx.x >> 3] = join_bits(v.h, v.l);
  if (lane == 0) wm[threadIdx.x >> 5] = amax;
  __syncthreads();
  if (threadIdx.x < 32) {
    const double s = warp_sum64<32>(ws);
    amax = lane < kNT / 32 ? wm[lane] : 0.0f;
    for (int o = 4; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if (lane == 0) {
      partial[2 * blockIdx.x] = s;
      partial[2 * blockIdx.x + 1] = (double)amax;
    }
  }
}

// The double-float passes over the fine grid work on x-pairs (every n0 is
// even), the pair arithmetic on packed FP32 pairs; the sums take kPP pairs per
// thread, 256 apart, so that their block reduction (about 150 instructions) is
// shared by 2 kPP cells.  At 512^3: source 3.20 -> 2.04 ms, sum of phi 0.80 ->
// 0.20 ms, defect 1.47 -> 1.18 ms (one cell per thread before).
constexpr int kPP = 2;

__device__ __forceinline__ df2 ld_df2(const float2 *p, long long pair) {
  const float4 v = reinterpret_cast<const float4 *>(p)[pair];
  return {make_float2(v.x, v.z), make_float2(v.y, v.w)};
}
__device__ __forceinline__ void st_df2(float2 *p, long long pair, const df2 &v) {
  reinterpret_cast<float4 *>(p)[pair] = make_float4(v.h.x, v.l.x, v.h.y, v.l.y);
}
// cells c0 and c1 of an FP64 array of the caller's (aligned to 8 bytes only)
__device__ __forceinline__ df2 split2(const double *p, long long c0, long long c1) {
  const df a = split_bits(p[c0]), b = split_bits(p[c1]);
  return {make_float2(a.h, b.h), make_float2(a.l, b.l)};
}

// s = 2 gamma (rho - 1) - (beta/2)(e^{-u/2} - 1) and phi = phi0, both as
// pairs; per-block partial sums of s (for its mean).
__global__ void __launch_bounds__(kNT)
    k_psource(PFine P, const double *rho, const double *u, const double *phi0, float g2h,
              float g2l, float bh, float bl, float ln2h, float ln2l, double *partial) {
  df2 v = {splat2(0.f), splat2(0.f)};
  float am = 0.0f;
#pragma unroll
  for (int q = 0; q < kPP; q++) {
    const long long t = ((long long)blockIdx.x * kPP + q) * kNT + threadIdx.x;
    const long long c0 = 2 * t;
    if (c0 >= P.ncell) break;
    // (the last pair of an odd number of cells holds one cell twice)
    const bool two = c0 + 1 < P.ncell;
    const long long c1 = two ? c0 + 1 : c0;
    const df2 r = split2(rho, c0, c1), uu = split2(u, c0, c1);
    const df2 e = df_exp2(df2{mul2(uu.h, splat2(-0.5f)), mul2(uu.l, splat2(-0.5f))}, ln2h,
                          ln2l);  // exact halving
    df2 s = df_sub2(df_mul2(df_add_f2(r, -1.0f), df2{splat2(g2h), splat2(g2l)}),
                    df_mul2(df_add_f2(e, -1.0f), df2{splat2(bh), splat2(bl)}));
    const df2 p0 = phi0 ? split2(phi0, c0, c1) : df2{splat2(0.f), splat2(0.f)};
    if (two) {
      st_df2(P.s, t, s);
      st_df2(P.phi, t, p0);
    } else {
      P.s[c0] = make_float2(s.h.x, s.l.x);
      P.phi[c0] = make_float2(p0.h.x, p0.l.x);
      s.h.y = s.l.y = 0.0f;
    }
    v = df_add2(v, s);
    am = fmaxf(am, fmaxf(fabsf(s.h.x), fabsf(s.h.y)));
  }
  block_df_partial(df_add(df{v.h.x, v.l.x}, df{v.h.y, v.l.y}), am, partial);
}

// Fine defect d = L(phi) - (s - smean) in double-float; the FP32 correction
// problem gets f = -d and e = 0.  Per-block partials of (d^2, max |d|).  One
// x-pair per thread.  The neighbours are added pair by pair, each sum
// normalised: with the low parts left to one FP32 sum the defect's rounding
// error was 1.35 times as large (rms 4.8 against 3.5 units of 2^-48 |phi| / h^2).
__global__ void __launch_bounds__(kNT)
    k_pdefect(PFine P, float smh, float sml, float *f32, float *e32, double *partial) {
  const long long t = (long long)blockIdx.x * kNT + threadIdx.x;
  float ss = 0.0f, mx = 0.0f;
  if (t < (P.ncell >> 1)) {
    const unsigned tu = (unsigned)t, q = fdiv(tu, P.fdh), q2 = fdiv(q, P.fd1);
    const int i = 2 * (int)(tu - q * (unsigned)(P.n0 >> 1)),
              j = (int)(q - q2 * (unsigned)P.n1), k = (int)q2;
    const long long c = 2 * t, sy = P.n0, sz = (long long)P.n0 * P.n1;
    const df2 pi = ld_df2(P.phi, t);
    const bool pat = P.phib != nullptr;
    float2 nb = splat2(6.0f);  // neighbours inside
    // ghost 2 phi_b - phi_i: phi_b enters here, -phi_i with the diagonal
    auto ghost = [&](int f, long long o) {
      const df b = split_bits(P.phib[P.foff[f] + o]);
      return make_float2(2.0f * b.h, 2.0f * b.l);
    };
    // -x of the pair's left cell, +x of its right cell
    float2 xl, xr;
    if (i > 0 || !pat) {
      xl = P.phi[i > 0 ? c - 1 : c + P.n0 - 1];
    } else {
      xl = ghost(0, (long long)k * P.n1 + j);
      nb.x -= 1.0f;
    }
    if (i + 2 < P.n0 || !pat) {
      xr = P.phi[i + 2 < P.n0 ? c + 2 : c + 2 - P.n0];
    } else {
      xr = ghost(1, (long long)k * P.n1 + j);
      nb.y -= 1.0f;
    }
    // cell 0: xl + cell 1; cell 1: cell 0 + xr
    df2 acc = df_add2(df2{make_float2(xl.x, pi.h.x), make_float2(xl.y, pi.l.x)},
                      df2{make_float2(pi.h.y, xr.x), make_float2(pi.l.y, xr.y)});
    auto add = [&](const df2 &v) { acc = df_add2(acc, v); };
    auto pair_face = [&](bool inside, long long in, long long wrap, int f, long long o) {
      if (inside || !pat) {
        add(ld_df2(P.phi, (inside ? in : wrap) >> 1));
      } else {
        const float2 g0 = ghost(f, o), g1 = ghost(f, o + 1);
        add(df2{make_float2(g0.x, g1.x), make_float2(g0.y, g1.y)});
        nb = sub2(nb, splat2(1.0f));
      }
    };
    const long long oy = (long long)k * P.n0 + i, oz = (long long)j * P.n0 + i;
    pair_face(j > 0, c - sy, c + (P.n1 - 1) * sy, 2, oy);
    pair_face(j < P.n1 - 1, c + sy, c - (P.n1 - 1) * sy, 3, oy);
    pair_face(k > 0, c - sz, c + (P.n2 - 1) * sz, 4, oz);
    pair_face(k < P.n2 - 1, c + sz, c - (P.n2 - 1) * sz, 5, oz);
    // diagonal: -(6 + missing) phi_i = -(12 - nb) phi_i
    const float2 dg = sub2(nb, splat2(12.0f));
    const df2 m = two_prod2(pi.h, dg);
    add(fast_two_sum2(m.h, fma2(pi.l, dg, m.l)));
    df2 d = df_mul2(acc, df2{splat2(P.ih2h), splat2(P.ih2l)});
    d = df_sub2(d, df_sub2(ld_df2(P.s, t), df2{splat2(smh), splat2(sml)}));
    const float2 dv = add2(d.h, d.l);
    reinterpret_cast<float2 *>(f32)[t] = make_float2(-dv.x, -dv.y);
    reinterpret_cast<float2 *>(e32)[t] = make_float2(0.0f, 0.0f);
    ss = fmaf(dv.y, dv.y, dv.x * dv.x);
    mx = fmaxf(fabsf(dv.x), fabsf(dv.y));
  }
  // sixteen threads' squares are added in FP32, the block's 16 sums in FP64
  for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  __shared__ double a[kNT / 16];
  __shared__ float b[kNT / 32];
  const int lane = threadIdx.x & 31;
  if ((lane & 15) == 0) a[threadIdx.x >> 4] = (double)ss;
  if (lane == 0) b[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x < 32) {
    const double s2 = warp_sum64<kNT / 16>(a);
    mx = lane < kNT / 32 ? b[lane] : 0.0f;
    for (int o = 4; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) {
      partial[2 * blockIdx.x] = s2;
      partial[2 * blockIdx.x + 1] = (double)mx;
    }
  }
}

// phi += e (pair arithmetic)
__global__ void __launch_bounds__(kNT) k_pupdate(PFine P, const float *e) {
  const long long t = (long long)blockIdx.x * kNT + threadIdx.x;
  if (t >= P.ncell) return;
  const float2 p = P.phi[t];
  df s = two_sum(p.x, e[t]);
  s.l += p.y;
  s = fast_two_sum(s.h, s.l);
  P.phi[t] = make_float2(s.h, s.l);
}

// per-block sums of phi (for its mean)
__global__ void __launch_bounds__(kNT) k_pphisum(PFine P, double *partial) {
  const long long np = P.ncell >> 1;
  df2 v = {splat2(0.f), splat2(0.f)};
#pragma unroll
  for (int q = 0; q < kPP; q++) {
    const long long t = ((long long)blockIdx.x * kPP + q) * kNT + threadIdx.x;
    if (t < np) v = df_add2(v, ld_df2(P.phi, t));
  }
  block_df_partial(df_add(df{v.h.x, v.l.x}, df{v.h.y, v.l.y}), 0.0f, partial);
}

// phi64 = phi - mean
__global__ void __launch_bounds__(kNT) k_pfinal(PFine P, float mh, float ml, double *out) {
  const long long t = (long long)blockIdx.x * kNT + threadIdx.x;
  if (t >= P.ncell) return;
  const float2 v = P.phi[t];
  const df p = df_sub(df{v.x, v.y}, df{mh, ml});
  out[t] = join_bits(p.h, p.l);
}

// ------------------------------------------------------------------ host
void split_host(double v, float &h, float &l) {
  h = (float)v;
  l = (float)(v - (double)h);
}

bool on_device(const void *p) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

struct Arena {
  frmg_ctx *c;
  std::vector<void *> ptrs;
  explicit Arena(frmg_ctx *c_) : c(c_) {}
  template <typename T>
  T *get(size_t n) {
    void *p = nullptr;
    try {
      p = frmg_alloc(c, n * sizeof(T));
    } catch (...) {
      throw PError{FR_ENOMEM, "device allocation failed"};
    }
    ptrs.push_back(p);
    return (T *)p;
  }
  ~Arena() {
    for (void *p : ptrs) frmg_release(c, p);
  }
};

// Sum and max of n (sum, max) pairs of per-block partials: block b reduces
// pairs [b kRedCH, (b + 1) kRedCH) in a fixed order (FP64) into pair b of out.
constexpr int kRedCH = 4096;
__global__ void __launch_bounds__(kNT) k_psum_pairs(const double *in, long long n, double *out) {
  __shared__ double ss[kNT / 32], sm[kNT / 32];
  const long long b0 = (long long)blockIdx.x * kRedCH;
  const long long b1 = b0 + kRedCH < n ? b0 + kRedCH : n;
  double s = 0.0, m = 0.0;
  for (long long i = b0 + threadIdx.x; i < b1; i += kNT) {
    s += in[2 * i];
    m = fmax(m, in[2 * i + 1]);
  }
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_down_sync(0xffffffffu, s, o);
    m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
  }
  if ((threadIdx.x & 31) == 0) {
    ss[threadIdx.x >> 5] = s;
    sm[threadIdx.x >> 5] = m;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0, mm = 0.0;
    for (int w = 0; w < kNT / 32; w++) {
      t += ss[w];
      mm = fmax(mm, sm[w]);
    }
    out[2 * blockIdx.x] = t;
    out[2 * blockIdx.x + 1] = mm;
  }
}

// Device-side sum (and max) of nb partial pairs in one or two reduction
// launches; only the final pair crosses to the host.  tmp holds at least
// 2 (ceil(nb / kRedCH) + 1) doubles; nb <= kRedCH^2.
struct PartialSum {
  frmg_ctx *ctx;
  double *tmp;
  double *pinned;
  cudaStream_t st;
  void operator()(const double *dpart, long long nb, double &sum, double &mx) const {
    const long long n2 = (nb + kRedCH - 1) / kRedCH;
    k_psum_pairs<<<(unsigned)n2, kNT, 0, st>>>(dpart, nb, tmp);
    PLAUNCH(ctx);
    const double *res = tmp;
    if (n2 > 1) {
      k_psum_pairs<<<1, kNT, 0, st>>>(tmp, n2, tmp + 2 * n2);
      PLAUNCH(ctx);
      res = tmp + 2 * n2;
    }
    PCK(cudaMemcpyAsync(pinned, res, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
    PCK(cudaStreamSynchronize(st));
    sum = pinned[0];
    mx = pinned[1];
  }
};

int level_count(const int n[3]) {
  int L = 1, m[3] = {n[0], n[1], n[2]};
  while (true) {
    bool ok = true;
    for (int d = 0; d < 3; d++) ok = ok && (m[d] % 2 == 0) && (m[d] / 2 >= 4);
    if (!ok) break;
    for (int d = 0; d < 3; d++) m[d] /= 2;
    L++;
  }
  return L;
}

struct PoissonSolver {
  frmg_ctx *ctx;
  cudaStream_t st;
  std::vector<PLevel> lev;
  int pre = 2, post = 2;

  std::vector<int> zc, nblk_t;  // tiled smoother: z-chunk and blocks per level (0: not tiled)
  std::vector<int> kc_p, nblk_p;  // tiled prolongation onto a level: coarse planes per block
                                  // and blocks (0: one thread per fine cell)
  std::vector<int> kc_r, nblk_r;  // tiled residual + restriction from a level (same layout)
  int tail = 1 << 30;     // first level of the one-cluster tail (none)
  LtDesc *tail_d = nullptr;
  int tail_cs = 1;
  size_t tail_smem = 0;

  // The tail begins at the first level below the finest whose levels fit it.
  void set_tail(Arena &A) {
    const int nl = (int)lev.size();
    const bool patch = lev[0].patch != 0;
    // a coarsest grid of odd sides keeps the launched levels (x-pairs)
    if (lev.back().n0 % 2 || lev.back().n1 % 2 || lev.back().n2 % 2) return;
    const int cs = patch ? lt_cluster<true>() : lt_cluster<false>();
    LtDesc D, best;
    memset(&D, 0, sizeof(D));
    D.patch = patch;
    D.pre = pre;
    D.post = post;
    D.relax = lev[0].relax;
    int at = nl;
    for (int l = nl - 1; l >= 1 && nl - l <= kLtLev && lev[l].ncell <= kLtCells; l--) {
      const int c = lev[l].ncell <= kLtLocal ? 1 : cs;
      const size_t b = lt_layout(D, &lev[l], nl - l, c);
      if (b > kLtSmem) break;
      at = l;
      best = D;
      tail_cs = c;
      tail_smem = b;
    }
    if (at == nl) return;
    tail = at;
    tail_d = A.get<LtDesc>(1);
    PCK(cudaMemcpyAsync(tail_d, &best, sizeof(best), cudaMemcpyHostToDevice, st));
    PCK(cudaStreamSynchronize(st));  // best has been read
  }
  template <bool PATCH>
  void run_tail() {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)tail_cs);
    c.blockDim = dim3(kLtNT);
    c.dynamicSmemBytes = tail_smem;
    c.stream = st;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeClusterDimension;
    a[0].val.clusterDim.x = tail_cs;
    a[0].val.clusterDim.y = a[0].val.clusterDim.z = 1;
    c.attrs = a;
    c.numAttrs = 1;
    PCK(cudaLaunchKernelEx(&c, k_ltail<PATCH>, (const LtDesc *)tail_d));
    PLAUNCH(ctx);
  }

  void smooth(int l, int n) {
    for (int it = 0; it < n; it++) {
      PLevel &L = lev[l];
      if (nblk_t[l] > 0) {
        if (L.patch)
          k_lsmooth_tiled<true><<<nblk_t[l], 256, 0, st>>>(L, zc[l]);
        else
          k_lsmooth_tiled<false><<<nblk_t[l], 256, 0, st>>>(L, zc[l]);
        PLAUNCH(ctx);
        std::swap(L.e, L.e_alt);
        continue;
      }
      for (int c = 0; c < 2; c++) {
        k_lsmooth<<<nblk(L.ncell / 2), kNT, 0, st>>>(L, c);
        PLAUNCH(ctx);
      }
    }
  }
  void vcycle(int l, double *partial0) {
    if (l == tail) {
      if (lev[l].patch) run_tail<true>();
      else run_tail<false>();
      return;
    }
    if (l == (int)lev.size() - 1) {
      k_lcoarsest<<<1, kNT, 0, st>>>(lev[l], 500);
      PLAUNCH(ctx);
      return;
    }
    smooth(l, pre);
    double *part = l == 0 ? partial0 : nullptr;
    if (nblk_r[l] > 0) {
      if (lev[l].patch)
        k_lresid_restrict_tiled<true><<<nblk_r[l], 256, 0, st>>>(lev[l], lev[l + 1], kc_r[l], part);
      else
        k_lresid_restrict_tiled<false><<<nblk_r[l], 256, 0, st>>>(lev[l], lev[l + 1], kc_r[l],
                                                                  part);
    } else {
      k_lresid_restrict<<<nblk(lev[l + 1].ncell), kNT, 0, st>>>(lev[l], lev[l + 1], part);
    }
    PLAUNCH(ctx);
    vcycle(l + 1, nullptr);
    if (nblk_p[l] > 0) {
      if (lev[l].patch)
        k_lprolong_tiled<true><<<nblk_p[l], 256, 0, st>>>(lev[l], lev[l + 1], kc_p[l]);
      else
        k_lprolong_tiled<false><<<nblk_p[l], 256, 0, st>>>(lev[l], lev[l + 1], kc_p[l]);
    } else {
      k_lprolong<<<nblk(lev[l].ncell), kNT, 0, st>>>(lev[l], lev[l + 1]);
    }
    PLAUNCH(ctx);
    smooth(l, post);
  }
};

}  // namespace

extern "C" int fr_poisson_solve(frmg_ctx *ctx, const double *density, const double *u,
                                const int dims[3], double box_mpc_h, double a, double omega_m,
                                double fr0_abs, const double *phib, double h, double tol,
                                double *phi_inout, const fr_opts *opts, fr_stats *stats,
                                double *src_mean, void *stream) {
  try {
    const auto t0 = std::chrono::steady_clock::now();
    if (!ctx || !density || !u || !dims || !phi_inout)
      throw PError{FR_EINVAL, "NULL argument"};
    PCK(cudaSetDevice(frmg_device(ctx)));
    for (int d = 0; d < 3; d++)
      if (dims[d] < 2 || (dims[d] & 1)) throw PError{FR_EINVAL, "dims must be even and >= 2"};
    const long long nc = (long long)dims[0] * dims[1] * dims[2];
    if (nc >= (1ll << 31)) throw PError{FR_EINVAL, "grid too large (at most 2^31 - 1 cells)"};
    if (!(tol >= 0)) throw PError{FR_EINVAL, "tol must be >= 0"};
    fr_opts o;
    fr_opts_default(&o);
    if (opts) o = *opts;
    if (o.pre < 0 || o.post < 0 || o.pre + o.post < 1 || o.max_vcycles < 1 || o.max_outer < 1)
      throw PError{FR_EINVAL, "invalid options"};
    if (!(o.relax > 0 && o.relax < 2)) throw PError{FR_EINVAL, "relax must be in (0, 2)"};
    if (h <= 0) h = 1.0 / dims[0];
    double k6[6];
    int stc = fr_constants(box_mpc_h, dims[0], a, omega_m, fr0_abs, k6);
    if (stc != FR_OK) return stc;
    const double beta = k6[1], gamma = k6[2];
    cudaStream_t st = (cudaStream_t)stream;
    Arena A(ctx);
    // inputs on the device
    auto dev_in = [&](const double *p, long long n) -> const double * {
      if (!p) return nullptr;
      if (on_device(p)) return p;
      double *d = A.get<double>(n);
      PCK(cudaMemcpyAsync(d, p, n * sizeof(double), cudaMemcpyHostToDevice, st));
      return d;
    };
    long long nface = 2ll * dims[1] * dims[2] + 2ll * dims[0] * dims[2] + 2ll * dims[0] * dims[1];
    const double *drho = dev_in(density, nc);
    const double *du = dev_in(u, nc);
    const double *dphib = dev_in(phib, nface);
    const bool phi_dev = on_device(phi_inout);
    const double *dphi0 = dev_in(phi_inout, nc);
    double *dphi_out = phi_dev ? phi_inout : A.get<double>(nc);

    PFine P;
    memset(&P, 0, sizeof(P));
    P.n0 = dims[0];
    P.n1 = dims[1];
    P.n2 = dims[2];
    P.ncell = nc;
    P.fdh = make_fastdiv((unsigned)(P.n0 / 2));
    P.fd1 = make_fastdiv((unsigned)P.n1);
    P.phi = A.get<float2>(nc);
    P.s = A.get<float2>(nc);
    P.phib = dphib;
    {
      long long off = 0;
      const long long fs[6] = {(long long)dims[1] * dims[2], (long long)dims[1] * dims[2],
                               (long long)dims[0] * dims[2], (long long)dims[0] * dims[2],
                               (long long)dims[0] * dims[1], (long long)dims[0] * dims[1]};
      for (int f = 0; f < 6; f++) {
        P.foff[f] = off;
        off += fs[f];
      }
    }
    split_host(1.0 / (h * h), P.ih2h, P.ih2l);
    // multigrid levels of the correction equation
    PoissonSolver S{ctx, st, {}, o.pre, o.post, {}, {}, {}, {}, {}, {}};
    {
      const int nl = level_count(dims);
      int m[3] = {dims[0], dims[1], dims[2]};
      double hl = h;
      for (int l = 0; l < nl; l++) {
        PLevel L;
        L.n0 = m[0];
        L.n1 = m[1];
        L.n2 = m[2];
        L.ncell = (long long)m[0] * m[1] * m[2];
        L.fd0 = make_fastdiv((unsigned)m[0]);
        L.fd1 = make_fastdiv((unsigned)m[1]);
        L.h2 = (float)(hl * hl);
        L.relax = (float)o.relax;
        L.patch = phib != nullptr;
        L.e = A.get<float>(L.ncell);
        L.f = A.get<float>(L.ncell);
        L.e_alt = nullptr;
        PCK(cudaMemsetAsync(L.e, 0, L.ncell * sizeof(float), st));
        // tiled smoother on levels large enough to fill the GPU with 64 x 16
        // tiles; z-chunks minimise (waves of 4 resident blocks per SM) x
        // (planes per block, chunk + 4)
        int zcl = 0, nbt = 0;
        if (m[0] >= 32 && m[1] >= 16 && m[2] >= 8) {
          int sms = 0, dev = 0;
          PCK(cudaGetDevice(&dev));
          PCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
          const long long slots = 4ll * std::max(sms, 1);
          const long long tiles = (long long)((m[0] + 63) / 64) * ((m[1] + 15) / 16);
          double best = 1e300;
          for (int c = 1; c <= m[2]; c++) {
            const int z = (m[2] + c - 1) / c;
            const long long blocks = tiles * ((m[2] + z - 1) / z);
            const double cost = std::ceil((double)blocks / slots) * (z + 4);
            if (cost < best - 1e-9) {
              best = cost;
              zcl = z;
            }
          }
          const long long blocks = tiles * ((m[2] + zcl - 1) / zcl);
          if (blocks >= sms) {
            nbt = (int)blocks;
            L.e_alt = A.get<float>(L.ncell);
          } else {
            zcl = 0;
          }
        }
        S.zc.push_back(zcl);
        S.nblk_t.push_back(nbt);
        // tiled prolongation onto this level (from the next coarser one) and
        // residual + restriction from it, where the 64 x 16 tiles times chunks
        // of coarse planes fill the GPU: the chunk minimises (waves of resident
        // blocks, 8 and 4 per SM) x (chunk + the planes read beyond it)
        int kcp = 0, nbp = 0, kcr = 0, nbr = 0;
        if (l + 1 < nl && nbt > 0) {
          int sms = 0, dev = 0;
          PCK(cudaGetDevice(&dev));
          PCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
          const long long tiles = (long long)((m[0] + 63) / 64) * ((m[1] + 15) / 16);
          const int c2 = m[2] / 2;
          auto pick = [&](int per_sm, int beyond, int &kc, int &nb) {
            const long long slots = (long long)per_sm * std::max(sms, 1);
            double best = 1e300;
            for (int c = 1; c <= c2; c++) {
              const int z = (c2 + c - 1) / c;
              const long long blocks = tiles * ((c2 + z - 1) / z);
              const double cost = std::ceil((double)blocks / slots) * (z + beyond);
              if (cost < best - 1e-9) {
                best = cost;
                kc = z;
              }
            }
            nb = (int)(tiles * ((c2 + kc - 1) / kc));
          };
          pick(8, 1, kcp, nbp);
          pick(4, 2, kcr, nbr);
        }
        S.kc_p.push_back(kcp);
        S.nblk_p.push_back(nbp);
        S.kc_r.push_back(kcr);
        S.nblk_r.push_back(nbr);
        S.lev.push_back(L);
        for (int d = 0; d < 3; d++) m[d] /= 2;
        hl *= 2.0;
      }
    }
    S.set_tail(A);
    // blocks of the double-float passes: one x-pair per thread, kPP pairs per
    // thread in the sums, one cell per thread
    const long long np = nc / 2, nbp = nblk(np), nbs = nblk((np + kPP - 1) / kPP), nb = nblk(nc);
    double *partial = A.get<double>(2 * nbp);
    double *pin = frmg_pinned(ctx, 2);
    if (!pin) throw PError{FR_ENOMEM, "pinned host allocation failed"};
    if (nb > (long long)kRedCH * kRedCH) throw PError{FR_EINVAL, "grid too large"};
    const PartialSum psum{ctx, A.get<double>(2 * ((nb + kRedCH - 1) / kRedCH + 1)), pin, st};
    float ln2h, ln2l, g2h, g2l, bh, bl;
    split_host(std::log(2.0), ln2h, ln2l);
    split_host(2.0 * gamma, g2h, g2l);
    split_host(0.5 * beta, bh, bl);
    k_psource<<<nbs, kNT, 0, st>>>(P, drho, du, dphi0, g2h, g2l, bh, bl, ln2h, ln2l, partial);
    PLAUNCH(ctx);
    double ssum, smax;
    psum(partial, nbs, ssum, smax);
    const double smean = phib ? 0.0 : ssum / (double)nc;
    if (src_mean) *src_mean = smean;
    float smh, sml;
    split_host(smean, smh, sml);

    fr_stats sv;
    memset(&sv, 0, sizeof(sv));
    sv.tau_rms = std::nan("");  // not evaluated by the linear solve
    auto push = [&](double v) {
      if (sv.nhist < FR_HIST) sv.hist[sv.nhist++] = v;
    };
    double prev = HUGE_VAL;
    int status = FR_ENOCONV;
    // fine-level norm partials of the residual + restriction (one per block)
    const long long nbc = S.lev.size() > 1
                              ? (S.nblk_r[0] > 0 ? (long long)S.nblk_r[0] : nblk(S.lev[1].ncell))
                              : 0;
    double *partial0 = A.get<double>(2 * std::max<long long>(nbc, 1));
    for (int outer = 0; outer < o.max_outer; outer++) {
      k_pdefect<<<nbp, kNT, 0, st>>>(P, smh, sml, S.lev[0].f, S.lev[0].e, partial);
      PLAUNCH(ctx);
      double s2, dmax;
      psum(partial, nbp, s2, dmax);
      const double r = std::sqrt(s2 / (double)nc);
      if (outer == 0) sv.res0_rms = r;
      sv.res_rms = r;
      sv.res_max = dmax;
      sv.outer = outer + 1;
      push(-r);
      if (!(r == r)) throw PError{FR_EDIVERGED, "non-finite residual"};
      if (r <= tol) {
        status = FR_OK;
        break;
      }
      if (outer > 0 && r > prev) throw PError{FR_EDIVERGED, "defect grew"};
      prev = r;
      if (sv.vcycles >= o.max_vcycles) break;
      // FP32 correction solve: stop near the FP32 floor (1e-5 of its start)
      // or when the cycle contraction stalls
      double rp = HUGE_VAL;
      for (int k = 0; k < o.max_vcycles; k++) {
        if (S.lev.size() == 1) {
          k_lcoarsest<<<1, kNT, 0, st>>>(S.lev[0], 500);
          PLAUNCH(ctx);
          sv.vcycles++;
          break;
        }
        S.vcycle(0, partial0);
        sv.vcycles++;
        double a2, am;
        psum(partial0, nbc, a2, am);
        const double rr = std::sqrt(a2 / (double)nc);  // residual after pre-smoothing
        push(rr);
        const double pred = rp < HUGE_VAL ? rr * std::sqrt(rr / rp) : rr;
        if (!(rr < 0.75 * rp) || rr <= 1e-5 * r || pred <= 0.5 * tol ||
            sv.vcycles >= o.max_vcycles)
          break;
        rp = rr;
      }
      k_pupdate<<<nb, kNT, 0, st>>>(P, S.lev[0].e);
      PLAUNCH(ctx);
    }
    // gauge (periodic): phi of zero mean
    double pmean = 0.0;
    if (!phib) {
      k_pphisum<<<nbs, kNT, 0, st>>>(P, partial);
      PLAUNCH(ctx);
      double phisum, pm;
      psum(partial, nbs, phisum, pm);
      pmean = phisum / (double)nc;
    }
    float mh, ml;
    split_host(pmean, mh, ml);
    k_pfinal<<<nb, kNT, 0, st>>>(P, mh, ml, dphi_out);
    PLAUNCH(ctx);
    if (!phi_dev)
      PCK(cudaMemcpyAsync(phi_inout, dphi_out, nc * sizeof(double), cudaMemcpyDeviceToHost, st));
    PCK(cudaStreamSynchronize(st));
    sv.seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    if (stats) *stats = sv;
    if (status != FR_OK) frmg_set_error("no convergence within the V-cycle or outer limits");
    return status;
  } catch (PError &e) {
    frmg_set_error(e.msg);
    if (stream) cudaStreamSynchronize((cudaStream_t)stream);
    return e.status;
  }
}

extern "C" int fr_poisson_source(frmg_ctx *ctx, const double *density, const double *u,
                                 const int dims[3], double box_mpc_h, double a,
                                 double omega_m, double fr0_abs, double *s_out, void *stream) {
  try {
    if (!ctx || !density || !u || !dims || !s_out) throw PError{FR_EINVAL, "NULL argument"};
    PCK(cudaSetDevice(frmg_device(ctx)));
    for (int d = 0; d < 3; d++)
      if (dims[d] < 1) throw PError{FR_EINVAL, "bad dims"};
    const long long nc = (long long)dims[0] * dims[1] * dims[2];
    double k6[6];
    int stc = fr_constants(box_mpc_h, dims[0], a, omega_m, fr0_abs, k6);
    if (stc != FR_OK) return stc;
    cudaStream_t st = (cudaStream_t)stream;
    Arena A(ctx);
    auto dev_in = [&](const double *p) -> const double * {
      if (on_device(p)) return p;
      double *d = A.get<double>(nc);
      PCK(cudaMemcpyAsync(d, p, nc * sizeof(double), cudaMemcpyHostToDevice, st));
      return d;
    };
    const double *drho = dev_in(density), *du = dev_in(u);
    const bool out_dev = on_device(s_out);
    double *ds = out_dev ? s_out : A.get<double>(nc);
    PFine P;
    memset(&P, 0, sizeof(P));
    P.ncell = nc;
    P.phi = A.get<float2>(nc);
    P.s = A.get<float2>(nc);
    const long long nb = nblk(nc), nbs = nblk(((nc + 1) / 2 + kPP - 1) / kPP);
    double *partial = A.get<double>(2 * nbs);
    float ln2h, ln2l, g2h, g2l, bh, bl;
    split_host(std::log(2.0), ln2h, ln2l);
    split_host(2.0 * k6[2], g2h, g2l);
    split_host(0.5 * k6[1], bh, bl);
    k_psource<<<nbs, kNT, 0, st>>>(P, drho, du, nullptr, g2h, g2l, bh, bl, ln2h, ln2l, partial);
    PLAUNCH(ctx);
    PFine Q = P;  // k_pfinal converts its phi array: point it at the source
    Q.phi = P.s;
    k_pfinal<<<nb, kNT, 0, st>>>(Q, 0.f, 0.f, ds);
    PLAUNCH(ctx);
    if (!out_dev) PCK(cudaMemcpyAsync(s_out, ds, nc * sizeof(double), cudaMemcpyDeviceToHost, st));
    PCK(cudaStreamSynchronize(st));
    return FR_OK;
  } catch (PError &e) {
    frmg_set_error(e.msg);
    return e.status;
  }
}
