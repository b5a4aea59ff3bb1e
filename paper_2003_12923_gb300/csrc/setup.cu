// One-time setup on the device: TOP basis (Sec. II.A, Eqs. 2-4), orbital transforms,
// the closed-shell Fock block f0_vo and the right-hand side b = Q H Psi0 on D+L.
//
// Conventions (shared by construction with every consumer of the TOP basis):
//  * 2 ||C||^2 = 1;
//  * SVD by one-sided (Hestenes) Jacobi on the rows of C, singular values sorted in
//    descending order, column k of V signed so its largest-magnitude component is
//    positive, u_k = C v_k / lambda_k;
//  * AVOs = columns No.. of the product of the Householder reflectors that
//    triangularise V (H = I - 2 w w^T / w^T w, w = x - alpha e_0, alpha = -sign(x_0)|x|).
#include <algorithm>
#include <cmath>

#include "internal.h"
#include "jacobi.h"

namespace esmp2 {
namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 2 |C|^2 = 1 (each spin-adapted CSF of Eq. psi0 has norm^2 2).
__global__ void k_normalise(const double *Cin, double *C, int n) {
  __shared__ double part[32];
  double s = 0.0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) s += Cin[k] * Cin[k];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.0;
    v = warp_sum(v);
    if (threadIdx.x == 0) part[0] = v;
  }
  __syncthreads();
  const double scale = 1.0 / sqrt(2.0 * part[0]);
  for (int k = threadIdx.x; k < n; k += blockDim.x) C[k] = Cin[k] * scale;
}

// One-sided Jacobi SVD of C (No x Nv, No <= 64): rotate the rows of B = J^T C with an
// orthogonal J until they are mutually orthogonal; then C = J diag(|B_k|) (B_k/|B_k|).
// One warp per row pair, pairs of a round disjoint (round-robin ordering).  On entry Jt holds the
// eigenvectors of C C^T as rows and B = Jt C: the rows are orthogonal up to the rounding of C C^T, so
// the sweeps (float64 on one SM: 15 pairs of 400 elements take its pipe 10 us a round) only clean up.
// Outputs: U (No x No), lam (No), V into columns 0..No-1 of Wv (Nv x Nv).
__global__ void __launch_bounds__(1024) k_jacobi_svd(const double *C, double *B, const double *Jt, double *J, double *U,
                                                     double *lam, double *Wv, int No, int Nv) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  __shared__ int rotated;
  __shared__ int perm[64];
  __shared__ double nrm[64];
  for (int k = threadIdx.x; k < No * No; k += blockDim.x) J[k] = Jt[(k % No) * No + k / No];
  __syncthreads();
  const int n = (No & 1) ? No + 1 : No;  // padded with a dummy row when No is odd
  for (int sweep = 0; sweep < 60; ++sweep) {
    if (threadIdx.x == 0) rotated = 0;
    __syncthreads();
    for (int r = 0; r < n - 1; ++r) {
      for (int pi = warp; pi < n / 2; pi += nw) {
        int p, q;
        if (pi == 0) { p = 0; q = 1 + (r % (n - 1)); }
        else { p = 1 + ((pi + r) % (n - 1)); q = 1 + ((n - 1 - pi + r) % (n - 1)); }
        if (p > q) { const int t = p; p = q; q = t; }
        if (q >= No) continue;
        double al = 0.0, be = 0.0, ga = 0.0;
        for (int a = lane; a < Nv; a += 32) {
          const double x = B[p * Nv + a], y = B[q * Nv + a];
          al += x * x; be += y * y; ga += x * y;
        }
        warp_sum3(al, be, ga);
        if (al <= 1e-300 || be <= 1e-300 || ga * ga <= 1e-30 * al * be) continue;
        double c, s;
        jacobi_rotation(al, be, ga, c, s);
        for (int a = lane; a < Nv; a += 32) {
          const double x = B[p * Nv + a], y = B[q * Nv + a];
          B[p * Nv + a] = c * x - s * y;
          B[q * Nv + a] = s * x + c * y;
        }
        for (int i = lane; i < No; i += 32) {
          const double x = J[i * No + p], y = J[i * No + q];
          J[i * No + p] = c * x - s * y;
          J[i * No + q] = s * x + c * y;
        }
        if (lane == 0) rotated = 1;
      }
      __syncthreads();
    }
    const int any = rotated;
    __syncthreads();
    if (!any) break;
  }
  // row norms and descending order
  for (int k = warp; k < No; k += nw) {
    double s = 0.0;
    for (int a = lane; a < Nv; a += 32) s += B[k * Nv + a] * B[k * Nv + a];
    s = warp_sum(s);
    if (lane == 0) nrm[k] = sqrt(s);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < No; ++k) perm[k] = k;
    for (int k = 0; k < No; ++k) {
      int best = k;
      for (int l = k + 1; l < No; ++l)
        if (nrm[perm[l]] > nrm[perm[best]]) best = l;
      const int t = perm[k]; perm[k] = perm[best]; perm[best] = t;
    }
  }
  __syncthreads();
  const double lmax = nrm[perm[0]];
  // V columns, sign convention, u_k = C v_k / lambda_k: a warp per column with a singular value
  // that is not negligible; then warp 0 completes the others (the last ones) in order
  auto finish = [&](int kk, bool live, double l) {   // column kk of Wv holds v_k up to its sign
    double best = -1.0;
    int bi = 0x7fffffff;
    for (int a = lane; a < Nv; a += 32) {   // argmax |v| (first occurrence)
      const double v = fabs(Wv[a * Nv + kk]);
      if (v > best) { best = v; bi = a; }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, off);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if (bi >= Nv) bi = 0;   // NaN input
    const double sg = Wv[bi * Nv + kk] < 0 ? -1.0 : 1.0;
    __syncwarp();
    for (int a = lane; a < Nv; a += 32) Wv[a * Nv + kk] *= sg;
    __syncwarp();
    for (int i = 0; i < No; ++i) {
      double u = sg * J[i * No + perm[kk]];
      if (live) {
        u = 0.0;
        for (int a = lane; a < Nv; a += 32) u += C[i * Nv + a] * Wv[a * Nv + kk];
        u = warp_sum(u) / l;
      }
      if (lane == 0) U[i * No + kk] = u;
    }
    if (lane == 0) lam[kk] = live ? l : 0.0;
  };
  auto is_live = [&](double l) { return l > 1e-12 * lmax && l > 1e-300; };
  for (int kk = warp; kk < No; kk += nw) {
    const int o = perm[kk];
    const double l = nrm[o];
    if (!is_live(l)) continue;
    for (int a = lane; a < Nv; a += 32) Wv[a * Nv + kk] = B[o * Nv + a] / l;
    __syncwarp();
    finish(kk, true, l);
  }
  __syncthreads();
  if (warp == 0) {
    for (int kk = 0; kk < No; ++kk) {
      if (is_live(nrm[perm[kk]])) continue;
      for (int m = 0; m < Nv; ++m) {   // Gram-Schmidt completion with the first unit vector that survives
        double nn = 0.0;
        for (int a = lane; a < Nv; a += 32) {
          double v = (a == m) ? 1.0 : 0.0;
          for (int prev = 0; prev < kk; ++prev) v -= Wv[m * Nv + prev] * Wv[a * Nv + prev];
          Wv[a * Nv + kk] = v;
          nn += v * v;
        }
        nn = warp_sum(nn);
        if (nn > 0.25) {
          const double inv = 1.0 / sqrt(nn);
          for (int a = lane; a < Nv; a += 32) Wv[a * Nv + kk] *= inv;
          break;
        }
      }
      __syncwarp();
      finish(kk, false, 0.0);
      __syncwarp();
    }
  }
}

// Eigenvectors (rows of Vt) of a symmetric matrix A (m x m <= 64 x 64, row pitch ldA, positive
// semi-definite, or any when shifted: A + (1 + largest absolute row sum) I has the same
// eigenvectors): one-sided Jacobi on the rows of B = Vt A held in shared memory, a warp per pair.
// A round is bound by its dependency chain (three reductions, one rotation).
__global__ void __launch_bounds__(1024) k_eig_small(const double *A, int64_t ldA, int m, int shifted, double *Vt) {
  extern __shared__ double sm_eig[];
  double *B = sm_eig, *J = sm_eig + m * m;
  __shared__ double red[32];
  __shared__ int rotated;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  double shift = 0.0;
  if (shifted) {
    double mx = 0.0;
    for (int p = warp; p < m; p += nw) {
      double r = 0.0;
      for (int q = lane; q < m; q += 32) r += fabs(A[p * ldA + q]);
      mx = fmax(mx, warp_sum(r));
    }
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    for (int w = 0; w < nw; ++w) shift = fmax(shift, red[w]);
    shift += 1.0;
  }
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
    const int p = e / m, q = e % m;
    J[e] = p == q ? 1.0 : 0.0;
    B[e] = A[p * ldA + q] + (p == q ? shift : 0.0);
  }
  __syncthreads();
  const int n = m + (m & 1);
  for (int sweep = 0; sweep < 60; ++sweep) {
    if (threadIdx.x == 0) rotated = 0;
    __syncthreads();
    for (int r = 0; r < n - 1; ++r) {
      for (int pi = warp; pi < n / 2; pi += nw) {
        int p, q;
        if (pi == 0) { p = 0; q = 1 + (r % (n - 1)); }
        else { p = 1 + ((pi + r) % (n - 1)); q = 1 + ((n - 1 - pi + r) % (n - 1)); }
        if (p > q) { const int t = p; p = q; q = t; }
        if (q >= m) continue;
        double *bp = B + p * m, *bq = B + q * m, *jp = J + p * m, *jq = J + q * m;
        double al = 0.0, be = 0.0, ga = 0.0;
        for (int k = lane; k < m; k += 32) {
          const double x = bp[k], y = bq[k];
          al += x * x; be += y * y; ga += x * y;
        }
        warp_sum3(al, be, ga);
        if (al <= 1e-300 || be <= 1e-300 || ga * ga <= 1e-30 * al * be) continue;
        double c, s;
        jacobi_rotation(al, be, ga, c, s);
        for (int k = lane; k < m; k += 32) {
          const double x = bp[k], y = bq[k], u = jp[k], v = jq[k];
          bp[k] = c * x - s * y;
          bq[k] = s * x + c * y;
          jp[k] = c * u - s * v;
          jq[k] = s * u + c * v;
        }
        if (lane == 0) rotated = 1;
      }
      __syncthreads();
    }
    const int any = rotated;
    __syncthreads();
    if (!any) break;
  }
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) Vt[e] = J[e];
}

// An orthonormal basis of the complement of orbital 0 of the orthogonal W (n x n, its columns the
// rotated orbitals in the input basis), in the coordinates of the columns 1 .. n-1: the rows
// j != k of H W without column 0, H the Householder reflector that takes column 0 to the input
// orbital k of its largest component.  It is as close to the input orbitals as the complement
// allows, where the Fock matrix is usually close to diagonal, so Jacobi starts from it.
__global__ void k_complement(const double *W, int n, double *J0) {
  __shared__ int k_sh;
  if (threadIdx.x < 32) {
    double best = -1.0;
    int bi = 0x7fffffff;
    for (int a = threadIdx.x; a < n; a += 32) {
      const double v = fabs(W[(int64_t)a * n]);
      if (v > best) { best = v; bi = a; }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, off);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if (threadIdx.x == 0) k_sh = bi < n ? bi : 0;   // (0: NaN input)
  }
  __syncthreads();
  const int k = k_sh, m = n - 1;
  const double vk = W[(int64_t)k * n], f = (vk >= 0.0 ? -1.0 : 1.0) / (1.0 + fabs(vk));
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)m * m; e += (int64_t)gridDim.x * blockDim.x) {
    const int jr = (int)(e / m), b = (int)(e % m) + 1, j = jr < k ? jr : jr + 1;
    J0[e] = W[(int64_t)j * n + b] + f * W[(int64_t)j * n] * W[(int64_t)k * n + b];
  }
}

// Householder reflectors triangularising V (columns 0..No-1 of Wv).  A: Nv x No work copy,
// R: Nv x No reflector vectors (column k holds w_k on rows k..Nv-1), ww: No norms^2.
__global__ void __launch_bounds__(1024) k_householder(const double *Wv, double *A, double *R, double *ww,
                                                      int No, int Nv) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  __shared__ double sh_ww;
  for (int e = threadIdx.x; e < Nv * No; e += blockDim.x) {
    A[e] = Wv[(e / No) * Nv + (e % No)];
    R[e] = 0.0;
  }
  __syncthreads();
  for (int k = 0; k < No; ++k) {
    if (warp == 0) {
      double s = 0.0;
      for (int r = k + lane; r < Nv; r += 32) s += A[r * No + k] * A[r * No + k];
      s = warp_sum(s);
      const double x0 = A[k * No + k];
      const double alpha = -(x0 >= 0 ? 1.0 : -1.0) * sqrt(s);
      double w2 = 0.0;
      for (int r = k + lane; r < Nv; r += 32) {
        const double w = A[r * No + k] - (r == k ? alpha : 0.0);
        R[r * No + k] = w;
        w2 += w * w;
      }
      w2 = warp_sum(w2);
      if (lane == 0) { sh_ww = w2; ww[k] = w2; }
    }
    __syncthreads();
    const double w2 = sh_ww;
    if (w2 > 0.0) {
      for (int col = k + warp; col < No; col += nw) {
        double d = 0.0;
        for (int r = k + lane; r < Nv; r += 32) d += R[r * No + k] * A[r * No + col];
        d = warp_sum(d) * (2.0 / w2);
        for (int r = k + lane; r < Nv; r += 32) A[r * No + col] -= d * R[r * No + k];
      }
    }
    __syncthreads();
  }
}

// AVO column j = H_0 H_1 ... H_{No-1} e_{No+j}, written to Wv[:, No+j].  One warp per column;
// E is Nv-1-No rows of scratch, row j contiguous.
__global__ void k_avo(const double *R, const double *ww, double *E, double *Wv, int No, int Nv) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const int navo = Nv - No;
  if (warp >= navo) return;
  double *e = E + (int64_t)warp * Nv;
  for (int r = lane; r < Nv; r += 32) e[r] = (r == No + warp) ? 1.0 : 0.0;
  __syncwarp();
  for (int k = No - 1; k >= 0; --k) {
    const double w2 = ww[k];
    if (w2 <= 0.0) continue;
    double d = 0.0;
    for (int r = k + lane; r < Nv; r += 32) d += R[r * No + k] * e[r];
    d = warp_sum(d) * (2.0 / w2);
    for (int r = k + lane; r < Nv; r += 32) e[r] -= d * R[r * No + k];
    __syncwarp();
  }
  for (int r = lane; r < Nv; r += 32) Wv[(int64_t)r * Nv + No + warp] = e[r];
}

__global__ void k_assemble_W(const double *U, const double *Wv, double *W, int No, int Nv) {
  const int N = No + Nv;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)N * N;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int p = (int)(e / N), q = (int)(e % N);
    double v = 0.0;
    if (p < No && q < No) v = U[p * No + q];
    else if (p >= No && q >= No) v = Wv[(int64_t)(p - No) * Nv + (q - No)];
    W[e] = v;
  }
}

// omega = sum_u 2 lam_u^2 (F_u'u' - F_uu);  E0 = E_Phi[F] + omega = 2 sum_i F_ii + omega.
__global__ void k_scalars(const double *F, const double *lam, double *scal, int No, int Nv) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int N = No + Nv;
  double om = 0.0, eph = 0.0;
  for (int u = 0; u < No; ++u) {
    om += 2.0 * lam[u] * lam[u] * (F[(int64_t)(No + u) * N + No + u] - F[(int64_t)u * N + u]);
    eph += 2.0 * F[(int64_t)u * N + u];
  }
  scal[0] = om;
  scal[1] = eph + om;
}

// f0_aj: the Fock matrix of the closed-shell determinant Phi, F - G[gamma - gamma_Phi],
// with gamma - gamma_Phi = -2 lam_u^2 on occupied u and +2 lam_u^2 on TOP virtual u'.
__global__ void k_f0vo(const double *F, const double *lam, const double *ooov, const double *ovvt,
                       double *f0, int No, int Nv) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= Nv * No) return;
  const int a = e / No, j = e % No, N = No + Nv;
  double v = F[(int64_t)j * N + No + a];
  for (int u = 0; u < No; ++u) {
    const double w = 2.0 * lam[u] * lam[u];
    const double aj_uu = ooov[(((int64_t)u * No + u) * No + j) * Nv + a];
    const double au_uj = ooov[(((int64_t)u * No + j) * No + u) * Nv + a];
    const double aj_pp = ovvt[(((int64_t)j * Nv + a) * Nv + u) * No + u];
    const double ap_pj = ovvt[(((int64_t)j * Nv + u) * Nv + a) * No + u];
    v += w * (aj_uu - 0.5 * au_uj) - w * (aj_pp - 0.5 * ap_pj);
  }
  f0[e] = v;
}

// b = Q H Psi0 on the stored blocks (Slater-Condon rules with Psi0 = sum_u lam_u (u -> u')):
//  doubles: P(ij)P(ab)[s_ia f0_bj] + P(ij) sum_c <ab||cj> s_ic - P(ab) sum_k <kb||ij> s_ka
//  triples: P(k/ij)P(c/ab)[<ab||ij> s_kc]  (disconnected product of the double and the single)
//  Q[i][u][b][a] = (ia|bu'): the OVVT integrals with the last two index pairs moved so
//  that one of the two OVVT terms of every T/S element runs along b; the other (a and b
//  exchanged) is staged through shared memory.  One CTA per (pair i <= j, 32-row strip of a, T and S
//  or X, Y and Z), b in tiles of 32: both slices (i, j) and (j, i) of every block come from the same
//  two integrals, so each is read once (T, S: twice) for up to six results.  One CTA per block
//  and slice took 11.3 ms at No=30 Nv=400, this form 7.7 ms (9 GB; row segments of 256 bytes in ten
//  streams keep it well below the copy rate).
__global__ void __launch_bounds__(256) k_rhs(const double *lam, const double *f0, const double *ovov,
                                             const double *ooov, const double *Q, double *out, int No, int Nv) {
  __shared__ double tji[32][33], tij[32][33];
  const int64_t sNv = Nv, NvNv = (int64_t)Nv * Nv, B = (int64_t)No * No * NvNv;
  int i = 0, j = blockIdx.y;
  while (j >= No - i) { j -= No - i; ++i; }
  j += i;
  const int a0 = blockIdx.x * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const bool eq = i == j;
#define OVOV(i, a, j, b) ovov[(((int64_t)(i) * sNv + (a)) * No + (j)) * sNv + (b)]
#define OOOV(i, j, k, a) ooov[(((int64_t)(i) * No + (j)) * No + (k)) * sNv + (a)]
#define F0(a, j) f0[(int64_t)(a) * No + (j)]
  double *oij = out + ((int64_t)i * No + j) * NvNv, *oji = out + ((int64_t)j * No + i) * NvNv;
  const double li = lam[i], lj = lam[j], l0 = lam[0];
  if (blockIdx.z == 0) {   // T, S
    const double *Qji = Q + ((int64_t)j * No + i) * NvNv;  // Qji[a][b] = OVVT(j, b, a, i)
    const double *Qij = Q + ((int64_t)i * No + j) * NvNv;  // Qij[a][b] = OVVT(i, b, a, j)
    for (int b0 = 0; b0 < Nv; b0 += 32) {
      const int b = b0 + tx;
      double p[4], q[4];
      __syncthreads();
#pragma unroll
      for (int rr = 0; rr < 4; ++rr) {   // tji[bb][aa] = OVVT(j, a, b, i), tij[bb][aa] = OVVT(i, a, b, j)
        const int r = ty + 8 * rr, a = a0 + r, bb = b0 + r, aa = a0 + tx;
        const bool in = bb < Nv && aa < Nv, on = a < Nv && b < Nv;
        tji[r][tx] = in ? Qji[(int64_t)bb * Nv + aa] : 0.0;
        tij[r][tx] = in ? Qij[(int64_t)bb * Nv + aa] : 0.0;
        p[rr] = on ? Qji[(int64_t)a * Nv + b] : 0.0;
        q[rr] = on ? Qij[(int64_t)a * Nv + b] : 0.0;
      }
      __syncthreads();
#pragma unroll
      for (int rr = 0; rr < 4; ++rr) {
        const int ar = ty + 8 * rr, a = a0 + ar;
        if (a >= Nv || b >= Nv) continue;
        const int64_t ab = (int64_t)a * Nv + b;
        double t = 0.0, s1 = 0.0, s2 = 0.0;   // T_ij, S_ij, S_ji
        if (!eq && a != b) {
          if (a == i) t += li * F0(b, j);
          if (a == j) t -= lj * F0(b, i);
          if (b == i) t -= li * F0(a, j);
          if (b == j) t += lj * F0(a, i);
          t += li * (p[rr] - tji[tx][ar]) - lj * (q[rr] - tij[tx][ar]);
          if (a < No) t -= lam[a] * (OOOV(a, i, j, b) - OOOV(a, j, i, b));
          if (b < No) t += lam[b] * (OOOV(b, i, j, a) - OOOV(b, j, i, a));
        }
        if (a == i) s1 += li * F0(b, j);
        if (b == j) s1 += lj * F0(a, i);
        s1 += li * p[rr] + lj * tij[tx][ar];
        if (a < No) s1 -= lam[a] * OOOV(a, i, j, b);
        if (b < No) s1 -= lam[b] * OOOV(b, j, i, a);
        oij[ab] = t;
        oij[B + ab] = s1;
        if (!eq) {
          if (a == j) s2 += lj * F0(b, i);
          if (b == i) s2 += li * F0(a, j);
          s2 += lj * q[rr] + li * tji[tx][ar];
          if (a < No) s2 -= lam[a] * OOOV(a, j, i, b);
          if (b < No) s2 -= lam[b] * OOOV(b, i, j, a);
          oji[ab] = -t;
          oji[B + ab] = s2;
        }
      }
    }
  } else {   // X, Y: t j k -> t' b c (here j,k,b,c = i,j,a,b);  Z: i t k -> a t' c (here k,c = j,b)
    for (int b = tx; b < Nv; b += 32) {
      double p[4], q[4];
#pragma unroll
      for (int rr = 0; rr < 4; ++rr) {
        const int a = a0 + ty + 8 * rr;
        p[rr] = a < Nv ? OVOV(i, a, j, b) : 0.0;
        q[rr] = a < Nv ? OVOV(j, a, i, b) : 0.0;
      }
#pragma unroll
      for (int rr = 0; rr < 4; ++rr) {
        const int a = a0 + ty + 8 * rr;
        if (a >= Nv) continue;
        const int64_t ab = (int64_t)a * Nv + b;
        double x = 0.0, y = 0.0, z1 = 0.0, z2 = 0.0;   // X_ij, Y_ij, Z_ij, Z_ji
        if (!eq && a != b) {   // lam_t <bc||jk> + P(jk)P(bc)[lam_k d_ck q(j,b)]
          // X: q(j,b) = <t'b||tj> = (t't|bj) - (t'j|bt);  Y: q(j,b) = (t't|bj) (opposite spins)
          x = y = l0 * (p[rr] - q[rr]);
          auto add = [&](double l, int jj, int bb) {
            const double d = OVOV(0, 0, jj, bb);
            x += l * (d - OVOV(jj, 0, 0, bb));
            y += l * d;
          };
          if (b == j) add(lj, i, a);
          if (b == i) add(-li, j, a);
          if (a == j) add(-lj, i, b);
          if (a == i) add(li, j, b);
          if (i == 0 || a == 0 || b == 0) x = 0.0;
        }
        if (j != 0 && b != 0 && !(i == 0 && a == 0)) {
          z1 = l0 * p[rr];
          if (b == j) z1 += lj * OVOV(i, a, 0, 0);
          if (a == i) z1 += li * (OVOV(j, b, 0, 0) - OVOV(0, b, j, 0));
        }
        oij[BX * B + ab] = x;
        oij[BY * B + ab] = y;
        oij[BZ * B + ab] = z1;
        if (!eq) {
          if (i != 0 && b != 0) {
            z2 = l0 * q[rr];
            if (b == i) z2 += li * OVOV(j, a, 0, 0);
            if (a == j) z2 += lj * (OVOV(i, b, 0, 0) - OVOV(0, b, i, 0));
          }
          oji[BX * B + ab] = -x;
          oji[BY * B + ab] = -y;
          oji[BZ * B + ab] = z2;
        }
      }
    }
  }
#undef OVOV
#undef OOOV
#undef F0
}

}  // namespace

static esmp2_status eig_small(esmp2_handle *h, const double *A, int64_t ldA, int m, int shifted, double *Vt) {
  const int lim = (int)(sizeof(double) * 2 * 64 * 64);
  if (cudaError_t e = smem_limit_once(reinterpret_cast<const void *>(k_eig_small), lim)) return check_cuda(h, e, "k_eig_small shared-memory limit");
  k_eig_small<<<1, 1024, sizeof(double) * 2 * (size_t)m * m, h->stream>>>(A, ldA, m, shifted, Vt);
  h->launches += 1;
  return ESMP2_OK;
}

// rows of J0 ((n-1) x (n-1)): start of the Jacobi rotations in the complement of orbital 0 of W (n x n)
void complement_basis(esmp2_handle *h, const double *W, int n, double *J0) {
  k_complement<<<(unsigned)std::min<int64_t>(cdiv((int64_t)(n - 1) * (n - 1), 256), 304), 256, 0, h->stream>>>(W, n, J0);
  h->launches += 1;
}

// eigenvectors (rows of Vt) of F_oo without t (from the identity: the columns of U that belong to
// tiny singular values are orthogonal only to rounding over that value, W_v's always to rounding)
esmp2_status eigvecs_occ(esmp2_handle *h, double *Vt) {
  return eig_small(h, h->F + h->d.N + 1, h->d.N, h->d.No - 1, 1, Vt);
}

esmp2_status check_cuda(esmp2_handle *h, cudaError_t e, const char *what) {
  if (e == cudaSuccess) return ESMP2_OK;
  h->err = std::string(what) + ": " + cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? ESMP2_ERR_OOM : ESMP2_ERR_CUDA;
}

esmp2_status setup_top_basis(esmp2_handle *h) {
  const int No = h->d.No, Nv = h->d.Nv, N = h->d.N;
  cudaStream_t st = h->stream;
  // one pooled workspace: B, A, R (No x Nv each), the Gram matrix, its eigenvectors and J (No x No
  // each), the reflector norms, AVO scratch, and W^T F's intermediate
  const size_t nC = (size_t)No * Nv, nO = (size_t)No * No, nE = (size_t)(Nv - No + 1) * Nv, nF = (size_t)N * N;
  double *ws = nullptr;
  cudaError_t ce = dmalloc(reinterpret_cast<void **>(&ws), sizeof(double) * (3 * nC + 3 * nO + No + nE + nF), st);
  if (ce != cudaSuccess) return check_cuda(h, ce, "setup alloc");
  double *work = ws, *A = work + nC, *R = A + nC, *Gm = R + nC, *Jt = Gm + nO, *Jm = Jt + nO, *ww = Jm + nO, *E = ww + No, *T1 = E + nE;

  k_normalise<<<1, 1024, 0, st>>>(h->C, h->C, No * Nv);
  Gemm64 g{};
  g.alpha = 1.0; g.beta = 0.0; g.batch = 1;
  g.M = No; g.N = No; g.K = Nv; g.sym = 1;   // C C^T
  g.A = h->C; g.sAm = Nv; g.sAk = 1;
  g.B = h->C; g.sBk = 1; g.sBn = Nv;
  g.C = Gm; g.sCm = No; g.sCn = 1;
  gemm64(g, st);
  esmp2_status se = eig_small(h, Gm, No, No, 0, Jt);
  if (se) { dfree(ws, st); return se; }
  g.N = Nv; g.K = No; g.sym = 0;             // B = Jt C
  g.A = Jt; g.sAm = No; g.sAk = 1;
  g.B = h->C; g.sBk = Nv; g.sBn = 1;
  g.C = work; g.sCm = Nv; g.sCn = 1;
  gemm64(g, st);
  h->launches += 2;
  k_jacobi_svd<<<1, 1024, 0, st>>>(h->C, work, Jt, Jm, h->U, h->lam, h->Wv, No, Nv);
  k_householder<<<1, 1024, 0, st>>>(h->Wv, A, R, ww, No, Nv);
  const int navo = Nv - No;
  if (navo > 0) k_avo<<<(unsigned)cdiv((int64_t)navo * 32, 256), 256, 0, st>>>(R, ww, E, h->Wv, No, Nv);
  k_assemble_W<<<256, 256, 0, st>>>(h->U, h->Wv, h->W, No, Nv);
  h->launches += 4 + (navo > 0);
  // F_TOP = W^T F W
  g.M = N; g.N = N; g.K = N;
  g.A = h->F; g.sAm = N; g.sAk = 1;   // h->F holds the input F here
  g.B = h->W; g.sBk = N; g.sBn = 1;
  g.C = T1; g.sCm = N; g.sCn = 1;
  gemm64(g, st);
  g.A = h->W; g.sAm = 1; g.sAk = N;
  g.B = T1; g.sBk = N; g.sBn = 1;
  g.C = h->F; g.sCm = N; g.sCn = 1;
  gemm64(g, st);
  k_scalars<<<1, 32, 0, st>>>(h->F, h->lam, h->scal, No, Nv);
  h->launches += 3;
  ce = cudaGetLastError();
  dfree(ws, st);
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(h->hred, h->scal, sizeof(double) * 2, cudaMemcpyDeviceToHost, st);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
  h->omega = h->hred[0];
  h->E0 = h->hred[1];
  if (ce == cudaSuccess) ce = cudaGetLastError();
  return check_cuda(h, ce, "TOP basis");
}

// Integral transforms + f0 + right-hand side.  ovov_src / ovvv_src are the device inputs
// (read only: the first pass of each transform reads them directly); ovov_in, ooov_in
// and ovvv_in are the handle's work buffers (ooov_in holds a copy of the input, ovvv_in
// No Nv Nv No elements), all consumed.
namespace {
// out[o0][o1][o2][o3] = in[...] with input axis ax[k] running along output axis k.  A CTA iteration
// takes kPermute elements of one (o0, o1), with 32-bit index arithmetic per element: 1.15 GB in and out
// 0.98 -> 0.88 ms; what remains are the strided reads.
constexpr int kPermute = 2048;
__global__ void __launch_bounds__(256) k_permute4(const double *in, double *out, int d0, int d1, int d2, int d3, int a0, int a1,
                                                  int a2, int a3) {
  const int d[4] = {d0, d1, d2, d3};
  int64_t st[4];
  st[3] = 1; st[2] = d3; st[1] = (int64_t)d2 * d3; st[0] = (int64_t)d1 * d2 * d3;
  const int D0 = d[a0], D1 = d[a1], D2 = d[a2], D3 = d[a3], n23 = D2 * D3, nch = (n23 + kPermute - 1) / kPermute;
  const int64_t s2 = st[a2], s3 = st[a3], items = (int64_t)D0 * D1 * nch;
  for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const int64_t oo = it / nch;
    const int ch = (int)(it - oo * nch), o0 = (int)(oo / D1), o1 = (int)(oo - (int64_t)o0 * D1);
    const double *src = in + o0 * st[a0] + o1 * st[a1];
    double *dst = out + oo * n23;
    const int end = min(n23, (ch + 1) * kPermute);
#pragma unroll 4
    for (int e = ch * kPermute + threadIdx.x; e < end; e += 256) {
      const int o2 = e / D3, o3 = e - o2 * D3;
      dst[e] = src[o2 * s2 + o3 * s3];
    }
  }
}

void permute4(esmp2_handle *h, const double *in, double *out, const int d[4], int a0, int a1, int a2, int a3) {
  k_permute4<<<1216, 256, 0, h->stream>>>(in, out, d[0], d[1], d[2], d[3], a0, a1, a2, a3);
  h->launches += 1;
}

}  // namespace

// The N^5 integral transforms of step a1, on the tensor cores from exact digit products (float64
// accuracy): rotations by the occupied U and the contraction of the last OVVV index with the TOP
// virtuals (Nv -> No columns) by the narrow-factor kernel (No <= 32, else float64 GEMMs),
// rotations by W_v (Nv x Nv) as X W_v after moving the rotated index last.
esmp2_status setup_rhs_from(esmp2_handle *h, const double *ovov_src, double *ovov_in, double *ooov_in,
                            const double *ovvv_src, double *ovvv_in, double *scratch) {
  const int No = h->d.No, Nv = h->d.Nv;
  cudaStream_t st = h->stream;
  const bool tc = (int64_t)9 * Nv * 1024 < (1LL << 24);   // exact ten-level digit sums (one term)
  esmp2_status s = ESMP2_OK;
  const double *q_ovvt = nullptr;  // (ia|bu') as [i][u][b][a], for the right-hand side
  {
    const int dims[4] = {No, Nv, No, Nv};
    if (tc) {
      if ((s = mode_product_small(h, ovov_src, scratch, 1, No, (int64_t)Nv * No * Nv, h->U))) return s;  // i
      if ((s = mode_product_small(h, scratch, ovov_in, (int64_t)No * Nv, No, Nv, h->U))) return s;       // j
      if ((s = xwv_split(h, ovov_in, (int64_t)No * Nv * No, scratch))) return s;   // b
      permute4(h, scratch, ovov_in, dims, 0, 2, 3, 1);                              // [i][j][b][a]
      if ((s = xwv_split(h, ovov_in, (int64_t)No * No * Nv, scratch))) return s;   // a
      const int d2[4] = {No, No, Nv, Nv};
      permute4(h, scratch, h->ovov, d2, 0, 3, 1, 2);                                // [i][a][j][b]
    } else {
      if (ovov_src != ovov_in)
        cudaMemcpyAsync(ovov_in, ovov_src, sizeof(double) * h->d.B, cudaMemcpyDeviceToDevice, st);
      double *src = ovov_in, *dst = scratch;
      const double *R[4] = {h->U, h->Wv, h->U, h->Wv};
      const int K[4] = {No, Nv, No, Nv};
      for (int m = 0; m < 4; ++m) {
        mode_product(src, dst, dims, m, R[m], K[m], K[m], st);
        double *t = src; src = dst; dst = t;
      }
      cudaMemcpyAsync(h->ovov, src, sizeof(double) * h->d.B, cudaMemcpyDeviceToDevice, st);
    }
  }
  debug_phase(h, "  ovov transform");
  {
    const int dims[4] = {No, No, No, Nv};
    double *src = ooov_in, *dst = scratch;
    const double *R[4] = {h->U, h->U, h->U, h->Wv};
    const int K[4] = {No, No, No, Nv};
    for (int m = 0; m < 4; ++m) {
      if (m < 3) {
        int64_t P = 1, Q = 1;
        for (int k = 0; k < m; ++k) P *= dims[k];
        for (int k = m + 1; k < 4; ++k) Q *= dims[k];
        if ((s = mode_product_small(h, src, dst, P, No, Q, h->U))) return s;
      } else {
        mode_product(src, dst, dims, m, R[m], K[m], K[m], st);
      }
      double *t = src; src = dst; dst = t;
    }
    cudaMemcpyAsync(h->ooov, src, sizeof(double) * (size_t)No * No * No * Nv, cudaMemcpyDeviceToDevice, st);
  }
  {
    debug_phase(h, "  ooov transform");
    if (h->ovvv_ready) cudaStreamWaitEvent(st, h->ovvv_ready, 0);   // host OVVV copied on a side stream
    int dims[4] = {No, Nv, Nv, Nv};
    if (No <= 32 && tc) {  // c -> u' (first No columns of Wv)
      if ((s = rows_times_narrow(h, ovvv_src, scratch, (int64_t)No * Nv * Nv, No, h->Wv))) return s;
    } else {
      mode_product(ovvv_src, scratch, dims, 3, h->Wv, No, Nv, st);
    }
    dims[3] = No;
    debug_phase(h, "  ovvv last index -> u'");
    if (tc) {
      if ((s = mode_product_small(h, scratch, ovvv_in, 1, No, (int64_t)Nv * Nv * No, h->U))) return s;  // [i][a][b][u]
      permute4(h, ovvv_in, scratch, dims, 0, 3, 1, 2);                             // [i][u][a][b]
      if ((s = xwv_split(h, scratch, (int64_t)No * No * Nv, ovvv_in))) return s;  // b
      const int d2[4] = {No, No, Nv, Nv};
      permute4(h, ovvv_in, scratch, d2, 0, 1, 3, 2);                               // [i][u][b][a]
      if ((s = xwv_split(h, scratch, (int64_t)No * No * Nv, ovvv_in))) return s;  // a
      permute4(h, ovvv_in, h->ovvt, d2, 0, 3, 2, 1);                               // [i][a][b][u]
      q_ovvt = ovvv_in;                                                             // [i][u][b][a]
    } else {
      double *src = scratch, *dst = ovvv_in;
      const double *R[3] = {h->U, h->Wv, h->Wv};
      const int K[3] = {No, Nv, Nv};
      for (int m = 0; m < 3; ++m) {
        mode_product(src, dst, dims, m, R[m], K[m], K[m], st);
        double *t = src; src = dst; dst = t;
      }
      cudaMemcpyAsync(h->ovvt, src, sizeof(double) * (size_t)No * Nv * Nv * No, cudaMemcpyDeviceToDevice, st);
      const int d4[4] = {No, Nv, Nv, No};
      permute4(h, h->ovvt, scratch, d4, 0, 3, 2, 1);                               // [i][u][b][a]
      q_ovvt = scratch;
    }
  }
  debug_phase(h, "  ovvt rotations");
  k_f0vo<<<(unsigned)cdiv((int64_t)No * Nv, 256), 256, 0, st>>>(h->F, h->lam, h->ooov, h->ovvt, h->f0vo, No, Nv);
  k_rhs<<<dim3((unsigned)cdiv(Nv, 32), (unsigned)(No * (No + 1) / 2), 2), 256, 0, st>>>(h->lam, h->f0vo, h->ovov, h->ooov, q_ovvt,
                                                                               h->b, No, Nv);
  h->launches += 2;
  return check_cuda(h, cudaGetLastError(), "rhs");
}

}  // namespace esmp2
