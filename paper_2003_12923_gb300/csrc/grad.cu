// Analytic gradient of E2 with respect to the Fock matrix and the (ov|ov) integrals.
//
// With A x = -b (A self-adjoint in the determinant inner product <,>) and E2 = <b,x> + E2_S:
//   dE2 = 2 <x, db> + <x, dA x> + dE2_S .
// The adjoint vector of the first-order equation is x itself (A is symmetric); an adjoint
// solve can be run and compared with x.  Contributions (TOP basis, then rotated back):
//   <x, dA x>, one-body part: densities of x contracted over every index but one (the
//       N_o^2 N_v^3 / N_o^3 N_v^2 float64 GEMMs below), plus the N^4 coupling terms, the pair
//       energy of the L blocks and omega;
//   2 <x, db>: the (ov|ov)-dependence of the L-triple right-hand side and the F_vo-dependence
//       of the doubles right-hand side (through the closed-shell Fock block f0);
//   dE2_S: the S-space sum -b_I^2 / D_I differentiated in b_I (integrals) and D_I (diagonal F).
// Conventions: dF is the derivative of E2 evaluated on (F + F^T)/2 (so dF is symmetric) and
// dOVOV[i][a][j][b] the derivative of E2 evaluated on the (ia)<->(jb) symmetrised block.
#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.h"

namespace esmp2 {
namespace {

constexpr double WT = 0.5, WS = 1.0, WX = 0.5, WY = 0.5, WZ = 2.0;
static_assert(WT == WX && WT == WY, "T, X and Y share one density product");

struct GCtx {
  int No, Nv, N;
  int64_t B;
  const double *x, *lam, *ovov, *F;
  double omega;
  __device__ __forceinline__ double X(int blk, int i, int j, int a, int b) const {
    return x[blk * B + (((int64_t)i * No + j) * Nv + a) * Nv + b];
  }
  __device__ __forceinline__ int64_t ov(int i, int a, int j, int b) const {
    return (((int64_t)i * Nv + a) * No + j) * Nv + b;
  }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ double block_sum(double v) {
  __shared__ double sh[32];
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
    t = warp_sum(t);
  }
  __syncthreads();
  return t;  // valid in thread 0
}

// (ov|ov) gradient from the L-triple right-hand side (elementwise part)
__global__ void kg_ovov_L(GCtx c, double *G) {
  const int No = c.No, Nv = c.Nv;
  const double l0 = c.lam[0];
  const int64_t n = (int64_t)No * Nv * No * Nv;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t f = e;
    const int g = (int)(f % Nv); f /= Nv;
    const int q = (int)(f % No); f /= No;
    const int be = (int)(f % Nv);
    const int p = (int)(f / Nv);
    G[e] += l0 * (4.0 * WX * c.X(BX, p, q, be, g) + 4.0 * WY * c.X(BY, p, q, be, g) + 2.0 * WZ * c.X(BZ, p, q, be, g));
  }
}

// per (J, B): partner-weighted sums of x entering the (ov|ov) entries with a TOP index and f0
__global__ void kg_small(GCtx c, double *Gov, double *Gf) {
  const int No = c.No, Nv = c.Nv, N = c.N;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < No * Nv; e += gridDim.x * blockDim.x) {
    const int J = e / Nv, Bv = e % Nv;
    double RX = 0, RY = 0, RZ1 = 0, RZ2 = 0, RT = 0, RS1 = 0, RS2 = 0;
    for (int k = 0; k < No; ++k) {
      const double l = c.lam[k];
      RX += l * c.X(BX, J, k, Bv, k);
      RY += l * c.X(BY, J, k, Bv, k);
      RZ1 += l * c.X(BZ, J, k, Bv, k);
      RZ2 += l * c.X(BZ, k, J, k, Bv);
      RT += l * c.X(BT, k, J, k, Bv);
      RS1 += l * c.X(BS, k, J, k, Bv);
      RS2 += l * c.X(BS, J, k, Bv, k);
    }
    atomicAdd(&Gov[c.ov(0, 0, J, Bv)], 8.0 * WX * RX + 8.0 * WY * RY);
    atomicAdd(&Gov[c.ov(J, 0, 0, Bv)], -8.0 * WX * RX);
    atomicAdd(&Gov[c.ov(J, Bv, 0, 0)], 2.0 * WZ * (RZ1 + RZ2));
    atomicAdd(&Gov[c.ov(0, Bv, J, 0)], -2.0 * WZ * RZ2);
    atomicAdd(&Gf[(int64_t)J * N + No + Bv], 8.0 * WT * RT + 2.0 * WS * (RS1 + RS2));  // 2<x, d b / d f0_BJ>
  }
}

// F1 (F_ov(0,0)), <x,x>, <x_L,x_L>: grid-stride, block partials via atomics into acc[0..2]
__global__ void kg_scalars(GCtx c, double *acc) {
  const int No = c.No, Nv = c.Nv;
  double f1 = 0, nn = 0, nl = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < c.B; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t f = e;
    const int b = (int)(f % Nv); f /= Nv;
    const int a = (int)(f % Nv); f /= Nv;
    const int j = (int)(f % No);
    const int i = (int)(f / No);
    const double t = c.X(BT, i, j, a, b), s = c.X(BS, i, j, a, b), xx = c.X(BX, i, j, a, b),
                 y = c.X(BY, i, j, a, b), z = c.X(BZ, i, j, a, b);
    f1 += WT * t * (xx + y) + WS * s * (z + c.X(BZ, j, i, b, a)) + WX * xx * t + WY * y * t + WZ * z * s;
    nl += WX * xx * xx + WY * y * y + WZ * z * z;
    nn += WT * t * t + WS * s * s;
  }
  nn += nl;
  const double r0 = block_sum(f1), r1 = block_sum(nn), r2 = block_sum(nl);
  if (threadIdx.x == 0) { atomicAdd(&acc[0], r0); atomicAdd(&acc[1], r1); atomicAdd(&acc[2], r2); }
}

// F2: d/dF_ov(0,c), one block per c
__global__ void kg_F2(GCtx c, double *Gf) {
  const int No = c.No, Nv = c.Nv, cc = blockIdx.x;
  double s = 0;
  for (int64_t r = threadIdx.x; r < (int64_t)No * No * Nv; r += blockDim.x) {
    const int b = (int)(r % Nv), ij = (int)(r / Nv), i = ij / No, j = ij % No;
    s += -2.0 * WT * c.X(BT, i, j, 0, b) * c.X(BX, i, j, cc, b)
         - WS * c.X(BS, i, j, b, 0) * c.X(BZ, i, j, b, cc)
         - WS * c.X(BS, i, j, 0, b) * c.X(BZ, j, i, b, cc)
         - 2.0 * WX * c.X(BX, i, j, cc, b) * c.X(BT, i, j, 0, b)
         - WZ * c.X(BZ, i, j, b, cc) * c.X(BS, i, j, b, 0);
  }
  s = block_sum(s);
  if (threadIdx.x == 0) Gf[No + cc] += s;
}

// F3: d/dF_ov(k,0), blocks (k, one of gridDim.y ranges of the sum over (j, a, b))
__global__ void kg_F3(GCtx c, double *Gf) {
  const int No = c.No, Nv = c.Nv, k = blockIdx.x;
  double s = 0;
  for (int64_t r = blockIdx.y * (int64_t)blockDim.x + threadIdx.x; r < (int64_t)No * Nv * Nv; r += (int64_t)gridDim.y * blockDim.x) {
    const int b = (int)(r % Nv), a = (int)((r / Nv) % Nv), j = (int)(r / ((int64_t)Nv * Nv));
    s += -2.0 * WT * c.X(BT, 0, j, a, b) * c.X(BX, k, j, a, b)
         - WS * c.X(BS, j, 0, a, b) * c.X(BZ, j, k, a, b)
         - WS * c.X(BS, 0, j, a, b) * c.X(BZ, j, k, b, a)
         - 2.0 * WX * c.X(BX, k, j, a, b) * c.X(BT, 0, j, a, b)
         - WZ * c.X(BZ, j, k, a, b) * c.X(BS, j, 0, a, b);
  }
  s = block_sum(s);
  if (threadIdx.x == 0) atomicAdd(&Gf[(int64_t)k * c.N + No], s);
}

// F4: d/dF_ov(k,c), one block per (k,c)
__global__ void kg_F4(GCtx c, double *Gf) {
  const int No = c.No, Nv = c.Nv, k = blockIdx.x / Nv, cc = blockIdx.x % Nv;
  double s = 0;
  for (int r = threadIdx.x; r < No * Nv; r += blockDim.x) {
    const int j = r / Nv, b = r % Nv;
    s += 4.0 * WT * c.X(BT, 0, j, 0, b) * (c.X(BX, k, j, cc, b) + c.X(BZ, k, j, cc, b))
         + WS * (c.X(BS, j, 0, b, 0) + c.X(BS, 0, j, 0, b)) * (c.X(BY, j, k, b, cc) + c.X(BZ, j, k, b, cc))
         + 4.0 * WX * c.X(BX, k, j, cc, b) * c.X(BT, 0, j, 0, b)
         + 4.0 * WY * c.X(BY, j, k, b, cc) * c.X(BS, 0, j, 0, b)
         + WZ * c.X(BZ, j, k, b, cc) * c.X(BS, j, 0, b, 0)
         + WZ * c.X(BZ, k, j, cc, b) * c.X(BT, 0, j, 0, b);
  }
  s = block_sum(s);
  if (threadIdx.x == 0) Gf[(int64_t)k * c.N + No + cc] += s;
}

// F5..F8: the t / t' row and column terms of the mixed-spin L blocks; one block per index
__global__ void kg_F5to8(GCtx c, double *Gf) {
  const int No = c.No, Nv = c.Nv, N = c.N;
  int id = blockIdx.x;
  int fam;
  if (id < Nv) fam = 5;
  else if ((id -= Nv) < No) fam = 6;
  else if ((id -= No) < Nv) fam = 7;
  else { id -= Nv; fam = 8; }
  double s = 0;
  for (int r = threadIdx.x; r < No * Nv; r += blockDim.x) {
    const int j = r / Nv, b = r % Nv;
    if (fam == 5) s += 4.0 * WY * c.X(BY, 0, j, 0, b) * c.X(BZ, 0, j, id, b);
    else if (fam == 6) s -= 4.0 * WY * c.X(BY, 0, j, 0, b) * c.X(BZ, id, j, 0, b);
    else if (fam == 7) s += WZ * c.X(BZ, 0, j, id, b) * c.X(BY, 0, j, 0, b);
    else s -= WZ * c.X(BZ, id, j, 0, b) * c.X(BY, 0, j, 0, b);
  }
  s = block_sum(s);
  if (threadIdx.x == 0) {
    if (fam == 5) Gf[(int64_t)No * N + No + id] += s;      // F_vv(0,d)
    else if (fam == 6) Gf[(int64_t)id * N] += s;           // F_oo(l,0)
    else if (fam == 7) Gf[(int64_t)(No + id) * N + No] += s;  // F_vv(a,0)
    else Gf[id] += s;                                      // F_oo(0,i)
  }
}

// scalars into Gf: F_ov(0,0), pair energy of L, omega
__global__ void kg_finish_scalars(GCtx c, const double *acc, double *Gf) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int No = c.No, N = c.N;
  Gf[No] += acc[0];
  Gf[(int64_t)No * N + No] += acc[2];
  Gf[0] -= acc[2];
  for (int u = 0; u < No; ++u) {
    const double w = 2.0 * c.lam[u] * c.lam[u] * acc[1];
    Gf[(int64_t)(No + u) * N + No + u] -= w;
    Gf[(int64_t)u * N + u] += w;
  }
}

// ---- S space: E2_S = sum_I 2 (-b_I^2 / D_I); scatter dE2_S/db_I into (ov|ov), dE2_S/dD_I into diag F
struct SG {
  GCtx c;
  double *Gov, *Gdiag;  // Gdiag[N + 1]: diagonal F gradient and (last) the omega sum
  __device__ void triple(const int *ho, const int *hs, const int *po, const int *ps, double *sdiag) const {
    const int PERM[3][3] = {{0, 1, 2}, {2, 1, 0}, {0, 2, 1}};
    const int PSG[3] = {1, -1, -1};
    const int No = c.No, N = c.N;
    double bI = 0.0;
    for (int t = 0; t < 3; ++t)
      for (int r = 0; r < 3; ++r) {
        const int h3 = PERM[t][2], p3 = PERM[r][2];
        if (hs[h3] != ps[p3] || ho[h3] != po[p3]) continue;
        const int H0 = PERM[t][0], H1 = PERM[t][1], P0 = PERM[r][0], P1 = PERM[r][1];
        double a = 0.0;
        if (ps[P0] == hs[H0] && ps[P1] == hs[H1]) a += c.ovov[c.ov(ho[H0], po[P0], ho[H1], po[P1])];
        if (ps[P0] == hs[H1] && ps[P1] == hs[H0]) a -= c.ovov[c.ov(ho[H1], po[P0], ho[H0], po[P1])];
        bI += PSG[t] * PSG[r] * c.lam[ho[h3]] * a;
      }
    double D = -c.omega;
    for (int k = 0; k < 3; ++k)
      D += c.F[(int64_t)(No + po[k]) * N + No + po[k]] - c.F[(int64_t)ho[k] * N + ho[k]];
    const double gb = -4.0 * bI / D, gd = 2.0 * bI * bI / (D * D);
    for (int t = 0; t < 3; ++t)
      for (int r = 0; r < 3; ++r) {
        const int h3 = PERM[t][2], p3 = PERM[r][2];
        if (hs[h3] != ps[p3] || ho[h3] != po[p3]) continue;
        const int H0 = PERM[t][0], H1 = PERM[t][1], P0 = PERM[r][0], P1 = PERM[r][1];
        const double f = gb * PSG[t] * PSG[r] * c.lam[ho[h3]];
        if (ps[P0] == hs[H0] && ps[P1] == hs[H1]) atomicAdd(&Gov[c.ov(ho[H0], po[P0], ho[H1], po[P1])], f);
        if (ps[P0] == hs[H1] && ps[P1] == hs[H0]) atomicAdd(&Gov[c.ov(ho[H1], po[P0], ho[H0], po[P1])], -f);
      }
    for (int k = 0; k < 3; ++k) {
      atomicAdd(&sdiag[No + po[k]], gd);
      atomicAdd(&sdiag[ho[k]], -gd);
    }
    atomicAdd(&sdiag[N], gd);
  }
};

__device__ void flush_diag(const SG &g, double *sdiag) {
  __syncthreads();
  for (int k = threadIdx.x; k <= g.c.N; k += blockDim.x)
    if (sdiag[k] != 0.0) atomicAdd(&g.Gdiag[k], sdiag[k]);
}

// S-space derivative, the triples with exactly one transition pair (the energy's k_e2s_ab and
// k_e2s_cm enumerate the same ones): b_I is lambda_u times one antisymmetrised integral, so a
// thread that owns the integral sums over the pair u itself, adds its own two (ov|ov) elements
// without atomics (no other thread writes them) and keeps the diagonal sums in registers and
// private shared-memory slots.  One triple at a time with nine scattered float64 atomics each took
// 17.5 ms at No=12 Nv=120, this form 1.0 ms.  (A float32 reciprocal with two Newton steps in place of the
// division was slower: 0.96 ms against 0.76 ms for the two kernels, the conversions share the pipe.)
constexpr int kST = 128;   // threads of the S-space gradient kernels

// shared memory: lu2[No], du[No], sdiag[N + 1], private per-u sums [No][kST]
size_t sgrad_smem(int No, int Nv) { return sizeof(double) * (size_t)(2 * No + No + Nv + 1 + No * kST); }
struct SSh {
  double *lu2, *du, *sdiag, *su;
};
__device__ __forceinline__ SSh s_shared(const SG &g, double *sm) {
  const int No = g.c.No, N = g.c.N;
  SSh s{sm, sm + No, sm + 2 * No, sm + 2 * No + N + 1};
  for (int u = threadIdx.x; u < No; u += blockDim.x) {
    s.lu2[u] = g.c.lam[u] * g.c.lam[u];
    s.du[u] = g.c.F[(int64_t)(No + u) * N + No + u] - g.c.F[(int64_t)u * N + u];
  }
  for (int k = threadIdx.x; k <= N; k += blockDim.x) s.sdiag[k] = 0.0;
  for (int k = threadIdx.x; k < No * kST; k += blockDim.x) s.su[k] = 0.0;
  __syncthreads();
  return s;
}
// per-u sums of the CTA into sdiag (u' particle, u hole), then everything to the gradient
__device__ __forceinline__ void s_flush(const SG &g, const SSh &s) {
  __syncthreads();
  const int No = g.c.No, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int u = warp; u < No; u += kST / 32) {
    double v = 0.0;
    for (int t = lane; t < kST; t += 32) v += s.su[u * kST + t];
    v = warp_sum(v);
    if (lane == 0 && v != 0.0) {
      atomicAdd(&s.sdiag[No + u], v);
      atomicAdd(&s.sdiag[u], -v);
      atomicAdd(&s.sdiag[g.c.N], v);
    }
  }
  flush_diag(g, s.sdiag);
}

// sectors A and B: block = (pair j < k, one of nchunk strided ranges of c), threads over b < c
__global__ void __launch_bounds__(kST) kg_s_ab(SG g, int nchunk) {
  extern __shared__ double sm[];
  const int No = g.c.No, Nv = g.c.Nv, N = g.c.N;
  const SSh s = s_shared(g, sm);
  const int chunk = blockIdx.x % nchunk;
  int kk = blockIdx.x / nchunk, j = 0;
  while (kk >= No - 1 - j) { kk -= No - 1 - j; ++j; }
  const int k = j + 1 + kk;
  const double base = -g.c.F[(int64_t)j * N + j] - g.c.F[(int64_t)k * N + k] - g.c.omega;
  double *su = s.su + threadIdx.x;
  double jk = 0.0;
  for (int b0 = 0; b0 < Nv; b0 += kST) {
    const int b = b0 + threadIdx.x;
    const double eb = b < Nv ? base + g.c.F[(int64_t)(No + b) * N + No + b] : 0.0;
    double gb = 0.0;
    for (int cc = 1 + chunk; cc < Nv; cc += nchunk) {
      if (cc <= b0 || cc == j || cc == k) continue;   // uniform over the CTA
      double gd = 0.0;
      if (b < cc && b != j && b != k) {
        const int64_t i1 = g.c.ov(k, cc, j, b), i2 = g.c.ov(j, cc, k, b);
        const double dg = g.c.ovov[i1] - g.c.ovov[i2], e = eb + g.c.F[(int64_t)(No + cc) * N + No + cc];
        double q1 = 0.0;
        for (int u = 1; u < No; ++u) {
          const double m = (u != j && u != k && u != b && u != cc) ? 2.0 : 1.0;   // sectors A and B, or B alone
          const double r = 1.0 / (s.du[u] + e), q = m * s.lu2[u] * r, d = 2.0 * dg * dg * q * r;
          q1 += q;
          su[u * kST] += d;
          gd += d;
        }
        g.Gov[i1] -= 4.0 * dg * q1;
        g.Gov[i2] += 4.0 * dg * q1;
      }
      gb += gd;
      gd = warp_sum(gd);
      if ((threadIdx.x & 31) == 0 && gd != 0.0) atomicAdd(&s.sdiag[No + cc], gd);
    }
    if (b < Nv && gb != 0.0) atomicAdd(&s.sdiag[No + b], gb);
    jk += gb;
  }
  jk = warp_sum(jk);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&s.sdiag[j], -jk);
    atomicAdd(&s.sdiag[k], -jk);
  }
  s_flush(g, s);
}

// sector C: block = (i, k, one of nchunk strided ranges of a), threads over c
__global__ void __launch_bounds__(kST) kg_s_cm(SG g, int nchunk) {
  extern __shared__ double sm[];
  const int No = g.c.No, Nv = g.c.Nv, N = g.c.N;
  const SSh s = s_shared(g, sm);
  const int chunk = blockIdx.x % nchunk, ik = blockIdx.x / nchunk, i = ik / No, k = ik % No;
  const double base = -g.c.F[(int64_t)i * N + i] - g.c.F[(int64_t)k * N + k] - g.c.omega;
  double *su = s.su + threadIdx.x;
  double sik = 0.0;
  for (int c0 = 0; c0 < Nv; c0 += kST) {
    const int cc = c0 + threadIdx.x;
    const bool on = cc < Nv && cc != k;
    const double ec = cc < Nv ? base + g.c.F[(int64_t)(No + cc) * N + No + cc] : 0.0;
    double gc = 0.0;
    for (int a = chunk; a < Nv; a += nchunk) {
      if (a == i) continue;
      double gd = 0.0;
      if (on) {
        const int64_t i1 = g.c.ov(i, a, k, cc);
        const double gv = g.c.ovov[i1], e = ec + g.c.F[(int64_t)(No + a) * N + No + a];
        double q1 = 0.0;
        for (int u = 1; u < No; ++u) {
          if (u == k || u == cc) continue;
          const double r = 1.0 / (s.du[u] + e), q = s.lu2[u] * r, d = 2.0 * gv * gv * q * r;
          q1 += q;
          su[u * kST] += d;
          gd += d;
        }
        g.Gov[i1] -= 4.0 * gv * q1;
      }
      gc += gd;
      gd = warp_sum(gd);
      if ((threadIdx.x & 31) == 0 && gd != 0.0) atomicAdd(&s.sdiag[No + a], gd);
    }
    if (on) atomicAdd(&s.sdiag[No + cc], gc);
    sik += gc;
  }
  sik = warp_sum(sik);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&s.sdiag[i], -sik);
    atomicAdd(&s.sdiag[k], -sik);
  }
  s_flush(g, s);
}

// the triples that hold a second transition pair (few), one at a time (the energy's k_e2s_gen
// enumerates the same ones): block = (u, x, y) for the three sectors' index pairs
__global__ void __launch_bounds__(kST) kg_s_gen(SG g) {
  extern __shared__ double sdiag[];
  for (int k = threadIdx.x; k <= g.c.N; k += blockDim.x) sdiag[k] = 0.0;
  __syncthreads();
  const int No = g.c.No, Nv = g.c.Nv;
  const int64_t blk = blockIdx.x;
  const int u = (int)(blk / ((int64_t)No * No)), x = (int)((blk / No) % No), y = (int)(blk % No);
  if (u >= 1) {
    const int j = x, k = y;
    if (j < k) {
      for (int e = threadIdx.x; e < 2 * Nv; e += blockDim.x) {
        const int xx = e < Nv ? j : k, yy = e % Nv;
        if (yy == xx || ((yy == j || yy == k) && xx != j)) continue;  // the pair (j, k) once
        const int b = min(xx, yy), cc = max(xx, yy);
        if (j != u && k != u && b != u && cc != u) {   // sector A
          const bool pj = (b == j || cc == j), pk = (b == k || cc == k);
          if (!((pj && j < u) || (pk && k < u)) && !((pj && j == 0) || (pk && k == 0))) {
            const int ho[3] = {u, j, k}, hs[3] = {0, 0, 0}, po[3] = {u, b, cc}, ps[3] = {0, 0, 0};
            g.triple(ho, hs, po, ps, sdiag);
          }
        }
        if (!((j == 0 || k == 0) && (b == 0 || cc == 0))) {   // sector B
          const int ho[3] = {u, j, k}, hs[3] = {0, 1, 1}, po[3] = {u, b, cc}, ps[3] = {0, 1, 1};
          g.triple(ho, hs, po, ps, sdiag);
        }
      }
    }
    const int i = x;
    if (k != u && k >= u && k != 0) {   // sector C: the down particle c == k
      for (int a = threadIdx.x; a < Nv; a += blockDim.x) {
        if (a == i) continue;
        const int ho[3] = {i, u, k}, hs[3] = {0, 1, 1}, po[3] = {a, u, k}, ps[3] = {0, 1, 1};
        g.triple(ho, hs, po, ps, sdiag);
      }
    }
  }
  flush_diag(g, sdiag);
}

__global__ void kg_s_finish(GCtx c, const double *Gdiag, double *Gf) {
  const int No = c.No, N = c.N;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < N; p += gridDim.x * blockDim.x) {
    double v = Gdiag[p];
    // omega = sum_u 2 lam_u^2 (F_u'u' - F_uu); D_I contains -omega
    if (p < No) v += 2.0 * c.lam[p] * c.lam[p] * Gdiag[N];
    else if (p < 2 * No) v -= 2.0 * c.lam[p - No] * c.lam[p - No] * Gdiag[N];
    Gf[(int64_t)p * N + p] += v;
  }
}

// symmetrise: out = (G + G^T) / 2 for an n x n matrix
__global__ void kg_sym(const double *G, double *out, int n) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
    const int p = e / n, q = e % n;
    out[e] = 0.5 * (G[e] + G[(int64_t)q * n + p]);
  }
}

// (ov|ov) symmetrisation over (ia) <-> (jb)
__global__ void kg_sym_ov(const double *G, double *out, int No, int Nv) {
  const int64_t M = (int64_t)No * Nv, n = M * M;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / M, q = e % M;
    out[e] = 0.5 * (G[e] + G[q * M + r]);
  }
}

__global__ void kg_transpose(const double *A, double *At, int n) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x)
    At[(e % n) * n + e / n] = A[e];
}

}  // namespace

// One-body densities of x (the N^5 part of <x, dA x>), accumulated into Gf (N x N).  T, X and Y are
// antisymmetric in both index pairs and S_ij^ab = S_ji^ba, so their sums over rows and over columns are
// the same, and the slices i < j of the first three count twice: a product over the listed slices of the
// three blocks (equal weights) takes 1.5 units of work in place of six, S one in place of two, Z two.
// The float64 pipe bounds them: No=12 Nv=120, all float64 GEMMs of the gradient 6.3 -> 3.8 ms.
static esmp2_status densities(esmp2_handle *h, const double *x, double *Gf) {
  const int No = h->d.No, Nv = h->d.Nv, N = h->d.N, NN = No * No, half = No * (No - 1) / 2;
  const int64_t B = h->d.B, NvNv = (int64_t)Nv * Nv;
  if (esmp2_status s = ensure_slist(h)) return s;
  double *Gv = Gf + (int64_t)No * N + No;
  // virtual: sum over (s, a) of X_s[a][p] X_s[a][q], and (by columns) over (s, b) of X_s[p][b] X_s[q][b]
  auto virt = [&](const double *X, const int *list, int ns, double w, bool cols) {
    Gemm64 g{};
    g.M = Nv; g.N = Nv; g.K = ns * Nv; g.batch = 1; g.alpha = w; g.beta = 1.0; g.sym = 1;
    g.Kin = Nv;
    g.klist = list;
    g.A = X; g.sAm = cols ? Nv : 1; g.sAk = cols ? 1 : Nv; g.sAk1 = NvNv;
    g.B = X; g.sBn = cols ? Nv : 1; g.sBk = cols ? 1 : Nv; g.sBk1 = NvNv;
    g.C = Gv; g.sCm = N; g.sCn = 1;
    gemm64(g, h->stream);
    h->launches += 1;
  };
  // occupied: minus the sum over (j, ab) of X[l][j][ab] X[i][j][ab], and over (i', ab) of X[i'][l][ab] X[i'][i][ab]
  auto occ = [&](const double *X, double w, bool second) {
    Gemm64 g{};
    g.M = No; g.N = No; g.K = (int)(No * NvNv); g.batch = 1; g.alpha = -w; g.beta = 1.0; g.sym = 1;
    if (second) {
      g.Kin = (int)NvNv;
      g.sAk1 = g.sBk1 = (int64_t)No * NvNv;
    }
    g.A = X; g.sAm = second ? NvNv : (int64_t)No * NvNv; g.sAk = 1;
    g.B = X; g.sBn = g.sAm; g.sBk = 1;
    g.C = Gf; g.sCm = N; g.sCn = 1;
    gemm64(g, h->stream);
    h->launches += 1;
  };
  if (!h->x_sym) {   // a vector set by the caller: every sum as it stands
    const double w[5] = {WT, WS, WX, WY, WZ};
    for (int blk = 0; blk < 5; ++blk)
      for (bool second : {false, true}) {
        virt(x + blk * B, nullptr, NN, w[blk], second);
        occ(x + blk * B, w[blk], second);
      }
    return ESMP2_OK;
  }
  if (half) virt(x, h->slist, 3 * half, 4.0 * WT, false);
  virt(x + BS * B, nullptr, NN, 2.0 * WS, false);
  virt(x + BZ * B, nullptr, NN, WZ, false);
  virt(x + BZ * B, nullptr, NN, WZ, true);
  for (int blk : {BT, BX, BY}) occ(x + blk * B, 2.0 * WT, false);
  occ(x + BS * B, 2.0 * WS, false);
  occ(x + BZ * B, WZ, false);
  occ(x + BZ * B, WZ, true);
  return ESMP2_OK;
}

esmp2_status gradient(esmp2_handle *h, double *dF_host, double *dOVOV_host, int adjoint, double *adj_diff) {
  if (!h->solved) { h->err = "esmp2_grad needs a previous esmp2_solve"; return ESMP2_ERR_STATE; }
  const int No = h->d.No, Nv = h->d.Nv, N = h->d.N;
  const int64_t nov = (int64_t)No * Nv * No * Nv, n = h->d.n;
  cudaStream_t st = h->stream;
  if (esmp2_status s0 = x_to_basis(h, 0)) return s0;
  if (adj_diff) *adj_diff = 0.0;
  if (adjoint) {  // A is symmetric: the adjoint solve A^T lambda = -b must return x itself
    double *xs = nullptr;
    cudaError_t ce = cudaMalloc(&xs, sizeof(double) * n);
    if (ce != cudaSuccess) return check_cuda(h, ce, "adjoint");
    cudaMemcpyAsync(xs, h->s64.x, sizeof(double) * n, cudaMemcpyDeviceToDevice, st);
    cudaMemsetAsync(h->s64.x, 0, sizeof(double) * n, st);
    h->x_zero = true;
    h->r_true = false;
    const bool xsym = h->x_sym;
    esmp2_solve_info info{};
    esmp2_status s = solve64(h, 1e-12, 5000, &info);
    if (s != ESMP2_OK && s != ESMP2_ERR_NOT_CONVERGED) { cudaFree(xs); return s; }
    // relative difference |lambda - x| / |x| (plain Euclidean on the stored blocks)
    std::vector<double> a(n), b(n);
    cudaMemcpy(a.data(), h->s64.x, sizeof(double) * n, cudaMemcpyDeviceToHost);
    cudaMemcpy(b.data(), xs, sizeof(double) * n, cudaMemcpyDeviceToHost);
    double dd = 0, xx = 0;
    for (int64_t k = 0; k < n; ++k) { dd += (a[k] - b[k]) * (a[k] - b[k]); xx += b[k] * b[k]; }
    if (adj_diff) *adj_diff = xx > 0 ? std::sqrt(dd / xx) : 0.0;
    cudaMemcpyAsync(h->s64.x, xs, sizeof(double) * n, cudaMemcpyDeviceToDevice, st);
    h->x_zero = false;
    h->x_sym = xsym;
    h->r_true = false;
    cudaStreamSynchronize(st);
    cudaFree(xs);
  }
  double *Gf = nullptr, *Gov = nullptr, *acc = nullptr, *T1 = nullptr, *T2 = nullptr, *Gd = nullptr;
  cudaError_t ce = cudaSuccess;
  auto A = [&](double **p, size_t cnt) { if (ce == cudaSuccess) ce = dmalloc(reinterpret_cast<void **>(p), sizeof(double) * cnt, st); };
  A(&Gf, (size_t)N * N); A(&Gov, (size_t)nov); A(&acc, 4); A(&T1, (size_t)std::max<int64_t>((int64_t)N * N, nov));
  A(&T2, (size_t)std::max<int64_t>((int64_t)N * N, nov)); A(&Gd, (size_t)N + 1);
  double *Ut_d = nullptr, *Wvt_d = nullptr;
  A(&Ut_d, (size_t)No * No); A(&Wvt_d, (size_t)Nv * Nv);
  auto release = [&]() {
    for (double *p : {Gf, Gov, acc, T1, T2, Gd, Ut_d, Wvt_d}) dfree(p, st);
  };
  if (ce != cudaSuccess) {
    release();
    return check_cuda(h, ce, "gradient workspace");
  }
  cudaMemsetAsync(Gf, 0, sizeof(double) * N * N, st);
  cudaMemsetAsync(Gov, 0, sizeof(double) * nov, st);
  cudaMemsetAsync(acc, 0, sizeof(double) * 4, st);
  cudaMemsetAsync(Gd, 0, sizeof(double) * (N + 1), st);
  GCtx c;
  c.No = No; c.Nv = Nv; c.N = N; c.B = h->d.B; c.x = h->s64.x; c.lam = h->lam; c.ovov = h->ovov; c.F = h->F;
  c.omega = h->omega_op;
  if (esmp2_status sd = densities(h, h->s64.x, Gf)) { release(); return sd; }
  kg_ovov_L<<<1216, 256, 0, st>>>(c, Gov);
  kg_small<<<(unsigned)cdiv((int64_t)No * Nv, 128), 128, 0, st>>>(c, Gov, Gf);
  kg_scalars<<<1216, 256, 0, st>>>(c, acc);
  kg_F2<<<Nv, 256, 0, st>>>(c, Gf);
  kg_F3<<<dim3((unsigned)No, (unsigned)std::max<int64_t>(1, std::min<int64_t>(cdiv(1216, No), (int64_t)No * Nv * Nv / 2048))), 256, 0, st>>>(c, Gf);
  kg_F4<<<No * Nv, 128, 0, st>>>(c, Gf);
  kg_F5to8<<<2 * (No + Nv), 128, 0, st>>>(c, Gf);
  kg_finish_scalars<<<1, 32, 0, st>>>(c, acc, Gf);
  SG sg;
  sg.c = c; sg.Gov = Gov; sg.Gdiag = Gd;
  if (No > 1) {   // sums over the small pairs u >= 1
    const int npair = No * (No - 1) / 2, chAB = (int)std::max<int64_t>(1, std::min<int64_t>(Nv / 8, cdiv(1216, npair))),
              chC = (int)std::max<int64_t>(1, std::min<int64_t>(Nv / 8, cdiv(1216, No * No)));
    const size_t shm = sgrad_smem(No, Nv);
    const int lim = (int)sgrad_smem(64, 4096);   // the largest sizes of the library: one limit for every call
    cudaError_t ea = smem_limit_once(reinterpret_cast<const void *>(kg_s_ab), lim);
    if (ea == cudaSuccess) ea = smem_limit_once(reinterpret_cast<const void *>(kg_s_cm), lim);
    if (ea != cudaSuccess) {
      release();
      return check_cuda(h, ea, "gradient shared-memory limit");
    }
    kg_s_ab<<<npair * chAB, kST, shm, st>>>(sg, chAB);
    kg_s_cm<<<No * No * chC, kST, shm, st>>>(sg, chC);
    kg_s_gen<<<No * No * No, kST, sizeof(double) * (N + 1), st>>>(sg);
  }
  kg_s_finish<<<(unsigned)cdiv(N, 128), 128, 0, st>>>(c, Gd, Gf);
  h->launches += 13;
  // dF = W sym(Gf) W^T
  kg_sym<<<256, 256, 0, st>>>(Gf, T1, N);
  Gemm64 g{};
  g.alpha = 1.0; g.beta = 0.0; g.batch = 1; g.M = N; g.N = N; g.K = N;
  g.A = h->W; g.sAm = N; g.sAk = 1; g.B = T1; g.sBk = N; g.sBn = 1; g.C = T2; g.sCm = N; g.sCn = 1;
  gemm64(g, st);
  g.A = T2; g.sAm = N; g.sAk = 1; g.B = h->W; g.sBk = 1; g.sBn = N; g.C = T1; g.sCm = N; g.sCn = 1;
  gemm64(g, st);
  if (dF_host) cudaMemcpyAsync(dF_host, T1, sizeof(double) * N * N, cudaMemcpyDeviceToHost, st);
  // dOVOV: symmetrise, then rotate every index back (in[i'] -> sum_i' U[i][i'] in[i'])
  kg_sym_ov<<<1216, 256, 0, st>>>(Gov, T1, No, Nv);
  kg_transpose<<<64, 256, 0, st>>>(h->U, Ut_d, No);
  kg_transpose<<<256, 256, 0, st>>>(h->Wv, Wvt_d, Nv);
  const int dims[4] = {No, Nv, No, Nv};
  const double *R[4] = {Ut_d, Wvt_d, Ut_d, Wvt_d};
  const int K[4] = {No, Nv, No, Nv};
  double *src = T1, *dst = T2;
  for (int m = 0; m < 4; ++m) {
    mode_product(src, dst, dims, m, R[m], K[m], K[m], st);
    double *t = src; src = dst; dst = t;
  }
  h->launches += 10;
  if (dOVOV_host) cudaMemcpyAsync(dOVOV_host, src, sizeof(double) * nov, cudaMemcpyDeviceToHost, st);
  ce = cudaStreamSynchronize(st);
  release();
  if (ce == cudaSuccess) ce = cudaGetLastError();
  return check_cuda(h, ce, "gradient");
}

}  // namespace esmp2
