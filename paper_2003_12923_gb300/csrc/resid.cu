// One pass over the amplitudes that are independent under the singlet symmetries (antisymmetric T,
// X, Y; S_ij^ab = S_ji^ba), full-storage float64 vectors, No <= 32, in two forms:
//   * the true residual r = -b - A x of the mixed-precision refinement, in the basis whose occupied
//     orbitals other than t diagonalise F_oo (arrow form of the occupied-index terms);
//   * SIG: y = A x in the TOP basis after the index contractions (sigma.cu index_terms64), the last
//     stage of the float64 sigma, with the partials of <x, y>.
//
// The general float64 sigma (sigma.cu) combines the virtual-index products, adds the couplings to y
// element by element on every stored image (four of T, X, Y, two of S) and leaves r to a further
// pass; float64 runs at two operations per clock and SM, so the coupling pass alone was bound by
// its arithmetic on the images.  Here an amplitude is computed once: T, X, Y on i < j and tile pairs
// ta <= tb (r written to both tiles), S on i <= j (r written to both slices), Z element by element;
// y never goes to memory and the norm is taken on the way.  The slices (j, i) of T, X, Y (the
// negatives) are neither read nor written.  Per residual at No=30 Nv=400 (without the virtual-index
// products): combine 2.5 + arrow sums and intermediates 4.7 + couplings 18.7 + residual 4.4 ms before,
// 13 ms now; the intermediate residuals no longer need their float32 coupling pass.
#include <algorithm>

#include "internal.h"

namespace esmp2 {
namespace {

constexpr int kT = 32, kThreads = 256, kGrid = 1216;

struct RC {
  int No, Nv, N;
  int64_t NvNv, B;
  const double *F;          // Fock matrix of the working basis, N x N
  double omega;
  const double *x, *b;
  const double *P;          // x F: T, X, Y (i < j) and S slices
  const double *Pz;         // Z: F Z (block vector) or nullptr
  const double *yz;         // Z F (Pz != nullptr) or Z F + F Z (Z slices)
  double *r;
  const double *VX, *WZ, *OC1, *OX, *OZ, *G, *H, *CYZ;
  const double *rho, *kap;  // reduced-cost basis: row sums [5 No^2][Nv], column sums of the Z slices
  double *red;
  int64_t base;
  __device__ __forceinline__ double o(int k, int l) const { return __ldg(F + (int64_t)k * N + l); }
  __device__ __forceinline__ double v(int a, int c) const { return __ldg(F + (int64_t)(No + a) * N + No + c); }
  __device__ __forceinline__ double ov(int k, int a) const { return __ldg(F + (int64_t)k * N + No + a); }
  __device__ __forceinline__ int64_t sl(int blk, int i, int j) const { return blk * B + ((int64_t)i * No + j) * NvNv; }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ void cta_partial(double v, double *slot) {
  __shared__ double sh[kThreads / 32];
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) s += sh[w];
    *slot = s;
  }
}
// items [first, last) of the blocked assignment of `items` work items to this CTA
__device__ __forceinline__ void cta_items(int64_t items, int64_t &first, int64_t &last) {
  const int64_t per = (items + gridDim.x - 1) / gridDim.x;
  first = (int64_t)blockIdx.x * per;
  last = min(items, first + per);
}

// T, X, Y: item = (slice i < j, tile pair ta <= tb).  AV (reduced-cost basis): the virtual-index
// terms x F - (x F)^T element-wise from the arrow form of F_vv.
// SIG: the occupied-index terms are in P; y also goes to the slice (j, i), and the slices i = j (zero)
// are items too.
typedef double Tile[kT][kT + 1];
template <int BLK, bool AV, bool SIG>
__device__ __forceinline__ void kr_anti(const RC &c, Tile &Pb /* the transposed product tile, then -r of the tile */) {
  const int nt = (c.Nv + kT - 1) / kT, npairs = nt * (nt + 1) / 2, No = c.No, Nv = c.Nv;
  const int nh = No * (SIG ? No + 1 : No - 1) / 2;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  int64_t first, last;
  cta_items((int64_t)nh * npairs, first, last);
  double nrm = 0.0;
  for (int64_t it = first; it < last; ++it) {
    int k = (int)(it / npairs), tp = (int)(it % npairs), ta = 0, i = 0;
    while (tp >= nt - ta) { tp -= nt - ta; ++ta; }
    const int tb = ta + tp;
    while (k >= (SIG ? No : No - 1) - i) { k -= (SIG ? No : No - 1) - i; ++i; }
    const int j = i + (SIG ? 0 : 1) + k;
    const int64_t so = c.sl(BLK, i, j);
    if (SIG && i == j) {   // uniform
      for (int q = ty; q < kT; q += 8) {
        const int a = ta * kT + q, b = tb * kT + tx, a2 = tb * kT + q, b2 = ta * kT + tx;
        if (a < Nv && b < Nv) c.r[so + (int64_t)a * Nv + b] = 0.0;
        if (a2 < Nv && b2 < Nv) c.r[so + (int64_t)a2 * Nv + b2] = 0.0;
      }
      continue;
    }
    const double *x = c.x + so, *P = c.P + so, *bv = c.b + so;
    double *r = c.r + so, *rj = c.r + c.sl(BLK, j, i);
    const int b = tb * kT + tx;
    double pa[4], xe[4], bb[4];
    if constexpr (!AV) __syncthreads();   // Pb of the previous item has been read
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {
      const int q = ty + 8 * rr, a = ta * kT + q;
      const int64_t e = (int64_t)a * Nv + b;
      const bool in = a < Nv && b < Nv;
      xe[rr] = in ? x[e] : 0.0;
      bb[rr] = !SIG && in ? bv[e] : 0.0;
      if constexpr (!AV) {
        const int a2 = tb * kT + q, b2 = ta * kT + tx;
        pa[rr] = in ? P[e] : 0.0;
        Pb[q][tx] = (a2 < Nv && b2 < Nv) ? P[(int64_t)a2 * Nv + b2] : 0.0;
      }
    }
    const bool i0 = i == 0;
    const double cxe = -c.omega + (BLK == BT ? 0.0 : c.v(0, 0) - c.o(0, 0)) - (SIG ? 0.0 : c.o(i, i) + c.o(j, j));
    const double s1 = i0 ? 1.0 : c.o(0, i), s2 = i0 ? 0.0 : c.o(0, j), f00 = c.ov(0, 0), fi0 = c.ov(i, 0), fj0 = c.ov(j, 0);
    const double *t1p = i0 ? c.OC1 + ((int64_t)BLK * No + j) * c.NvNv : c.x + c.sl(BLK, 0, j);
    const double *t2p = c.x + c.sl(BLK, 0, i0 ? j : i);   // x_i0 = -x_0i (not used for i = 0)
    const double *A1 = nullptr, *A2 = nullptr, *A3 = nullptr, *r1 = nullptr, *r2 = nullptr, *r3 = nullptr;
    if (BLK == BT) {
      A1 = c.x + c.sl(BX, i, j);
      A2 = c.x + c.sl(BY, i, j);
      r1 = c.VX + ((int64_t)i * No + j) * Nv;
      if (i0) { r2 = c.OX + (int64_t)j * c.NvNv; r3 = c.G + (int64_t)j * Nv; }
    } else if (BLK == BX) {
      A1 = c.x + c.sl(BT, i, j);
      A2 = c.x + c.sl(BT, 0, j);
      A3 = c.x + c.sl(BT, 0, i);   // i = 0: not an amplitude row (X needs i >= 1)
    } else {
      A1 = c.x + c.sl(BT, i, j);
      A2 = c.x + c.sl(BS, 0, i);
      A3 = c.x + c.sl(BS, 0, j);
      if (i0) r1 = c.CYZ + (int64_t)j * Nv;
    }
    const bool bin = b < Nv;
    const double fob0 = bin ? c.ov(0, b) : 0.0, fobi = bin ? c.ov(i, b) : 0.0, fobj = bin ? c.ov(j, b) : 0.0;
    double fv0b = 0.0, fvbb = 0.0, xb0 = 0.0;
    if constexpr (AV) {
      fv0b = bin ? c.v(0, b) : 0.0;
      fvbb = bin ? c.v(b, b) : 0.0;
      xb0 = bin ? x[(int64_t)b * Nv] : 0.0;
    }
    // row 0 of the partner slices at b (used by every row of the tile)
    double h1 = 0.0, h2 = 0.0, h3 = 0.0;
    if (bin && BLK == BX) { h1 = A1[b]; h2 = A2[b]; h3 = A3[b]; }
    if (bin && BLK == BY) { h2 = A2[b]; h3 = A3[b]; }
    if constexpr (!AV) __syncthreads();
    double rv[4];
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {
      const int q = ty + 8 * rr, a = ta * kT + q;
      rv[rr] = 0.0;
      const bool ok = a < Nv && bin && (ta < tb || q < tx) && !(BLK == BX && (i0 || a == 0));   // a < b; X: b >= 1 follows
      if (ok) {
        const int64_t ab = (int64_t)a * Nv + b;
        double u = cxe * xe[rr];
        if constexpr (!SIG) {
          u -= s1 * t1p[ab];
          if (!i0) u += s2 * t2p[ab];
        }
        if constexpr (AV) {   // X_ba = -X_ab
          u += fvbb * xe[rr];
          if (a == 0) u -= c.rho[(int64_t)(BLK * No * No + i * No + j) * Nv + b];
          else u += c.v(a, a) * xe[rr] + x[(int64_t)a * Nv] * fv0b - xb0 * c.v(0, a);
        } else {
          u += pa[rr] - Pb[tx][q];
        }
        if (BLK == BT) {
          u += f00 * (A1[ab] + A2[ab]);
          if (a == 0) u -= r1[b];   // a < b, so b >= 1
          if (i0) {
            u -= r2[ab];
            if (a == 0) u += r3[b];
          }
        } else if (BLK == BX) {
          const double foa0 = c.ov(0, a), foai = c.ov(i, a), foaj = c.ov(j, a);
          u += f00 * A1[ab] - foa0 * h1 + fob0 * A1[a] - fi0 * A2[ab] + fj0 * A3[ab] + foai * h2 - foaj * h3 -
               fobi * A2[a] + fobj * A3[a];
        } else {
          u += f00 * A1[ab] + fobj * A2[a] - fobi * A3[a] - c.ov(j, a) * h2 + c.ov(i, a) * h3;
          if (i0 && a == 0) u += r1[b];
        }
        rv[rr] = SIG ? u : -bb[rr] - u;
        nrm += (SIG ? xe[rr] : rv[rr]) * rv[rr];
      }
      if (a < Nv && bin && (ta < tb || q <= tx)) {
        r[(int64_t)a * Nv + b] = rv[rr];
        if (SIG) rj[(int64_t)a * Nv + b] = -rv[rr];
      }
    }
    __syncthreads();
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) Pb[ty + 8 * rr][tx] = -rv[rr];
    __syncthreads();
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {   // element (tb*32 + q, ta*32 + tx) = -r(ta*32 + tx, tb*32 + q)
      const int q = ty + 8 * rr, a = tb * kT + q, b2 = ta * kT + tx;
      if (a < Nv && b2 < Nv && (ta < tb || q > tx)) {
        r[(int64_t)a * Nv + b2] = Pb[tx][q];
        if (SIG) rj[(int64_t)a * Nv + b2] = -Pb[tx][q];
      }
    }
    if constexpr (AV) __syncthreads();
  }
  cta_partial(2.0 * nrm, c.red + c.base + blockIdx.x);   // four images of weight 1/2
}

// S: item = (slice pair i <= j, tile (ta, tb)); r_ji = r_ij^T
template <bool AV, bool SIG>
__device__ __forceinline__ void kr_s(const RC &c, Tile &Pb, Tile &Zt, Tile &Ot) {
  const int nt = (c.Nv + kT - 1) / kT, No = c.No, Nv = c.Nv, npair = No * (No + 1) / 2;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  int64_t first, last;
  cta_items((int64_t)npair * nt * nt, first, last);
  double nrm = 0.0;
  for (int64_t it = first; it < last; ++it) {
    int pi = (int)(it / (nt * nt)), i = 0;
    const int tt = (int)(it % (nt * nt)), ta = tt / nt, tb = tt % nt;
    while (pi >= No - i) { pi -= No - i; ++i; }
    const int j = i + pi;
    if (i == j && ta > tb) continue;   // the mirror of an item already covered (uniform)
    const int64_t sij = c.sl(BS, i, j), sji = c.sl(BS, j, i);
    const double *Zij = c.x + c.sl(BZ, i, j), *Zji = c.x + c.sl(BZ, j, i), *OZj = c.OZ + (int64_t)j * c.NvNv;
    const bool i0 = i == 0, j0 = j == 0;
    __syncthreads();
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {
      const int q = ty + 8 * rr, a2 = tb * kT + q, b2 = ta * kT + tx;
      const bool in = a2 < Nv && b2 < Nv;
      const int64_t e2 = (int64_t)a2 * Nv + b2;
      if constexpr (!AV) Pb[q][tx] = in ? c.P[sji + e2] : 0.0;
      Zt[q][tx] = in ? Zji[e2] : 0.0;
      if (i0) Ot[q][tx] = in ? OZj[e2] : 0.0;
    }
    __syncthreads();
    const double cxe = -c.omega - (SIG ? 0.0 : c.o(i, i) + c.o(j, j)), f00 = c.ov(0, 0);
    const double s1 = i0 ? 1.0 : c.o(0, i), s2 = j0 ? 1.0 : c.o(0, j);
    const double *t1p = i0 ? c.OC1 + ((int64_t)BS * No + j) * c.NvNv : c.x + c.sl(BS, 0, j);
    const double *t2p = c.x + c.sl(BS, i, 0);   // j = 0 (then i = 0): OC1_0 transposed
    const double *WZji = c.WZ + ((int64_t)j * No + i) * Nv, *WZij = c.WZ + ((int64_t)i * No + j) * Nv;
    const bool diag = i == j && ta == tb;
    const int b = tb * kT + tx;
    double fv0b = 0.0, fvbb = 0.0;
    if (AV && b < Nv) { fv0b = c.v(0, b); fvbb = c.v(b, b); }
    double rv[4];
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {
      const int q = ty + 8 * rr, a = ta * kT + q;
      rv[rr] = 0.0;
      if (a < Nv && b < Nv && (!diag || q <= tx)) {
        const int64_t ab = (int64_t)a * Nv + b;
        const double xe = c.x[sij + ab];
        double u = cxe * xe + f00 * (Zij[ab] + Zt[tx][q]);
        if constexpr (!SIG) {
          u -= s1 * t1p[ab];
          if (j0) u -= c.OC1[(int64_t)BS * No * c.NvNv + (int64_t)b * Nv + a];   // sum_m F_mt S_0m^ab = sum_m F_mt S_m0^ba
          else u -= s2 * t2p[ab];
        }
        if constexpr (AV) {   // S_ji^ba = S_ij^ab
          const double *xs = c.x + sij;
          u += b == 0 ? c.rho[(int64_t)(BS * No * No + i * No + j) * Nv + a] : fvbb * xe + xs[(int64_t)a * Nv] * fv0b;
          u += a == 0 ? c.rho[(int64_t)(BS * No * No + j * No + i) * Nv + b] : c.v(a, a) * xe + xs[b] * c.v(0, a);
        } else {
          u += c.P[sij + ab] + Pb[tx][q];
        }
        if (a == 0) u -= WZji[b];
        if (b == 0) u -= WZij[a];
        if (j0) {
          u -= c.OZ[(int64_t)i * c.NvNv + ab];
          if (b == 0) u += c.H[(int64_t)i * Nv + a];
        }
        if (i0) {
          u -= Ot[tx][q];
          if (a == 0) u += c.H[(int64_t)j * Nv + b];
        }
        rv[rr] = SIG ? u : -c.b[sij + ab] - u;
        nrm += (diag && q == tx ? 1.0 : 2.0) * (SIG ? xe : rv[rr]) * rv[rr];
        c.r[sij + ab] = rv[rr];
      }
    }
    __syncthreads();
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) Zt[ty + 8 * rr][tx] = rv[rr];
    __syncthreads();
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {   // r_ji[tb*32 + q][ta*32 + tx] = r_ij[ta*32 + tx][tb*32 + q]
      const int q = ty + 8 * rr, a = tb * kT + q, b2 = ta * kT + tx;
      if (a < Nv && b2 < Nv && (!diag || q > tx)) c.r[sji + (int64_t)a * Nv + b2] = Zt[tx][q];
    }
  }
  cta_partial(nrm, c.red + c.base + blockIdx.x);
}

// Z: a warp per row (slice, a), what depends on the row alone taken once
template <bool AV, bool SIG>
__device__ __forceinline__ void kr_z(const RC &c) {
  const int No = c.No, Nv = c.Nv, lane = threadIdx.x & 31;
  const int64_t rows = (int64_t)No * No * Nv;
  double nrm = 0.0;
  for (int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; row < rows;
       row += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int s = (int)(row / Nv), a = (int)(row - (int64_t)s * Nv), i = s / No, j = s - i * No;
    const int64_t so = (int64_t)BZ * c.B + (int64_t)s * c.NvNv + (int64_t)a * Nv;
    double *r = c.r + so;
    const bool i0 = i == 0;
    if (j == 0 || (i0 && a == 0)) {   // not amplitudes
      for (int b = lane; b < Nv; b += 32) r[b] = 0.0;
      continue;
    }
    const double *x = c.x + so, *bv = c.b + so, *yz = c.yz + (int64_t)s * c.NvNv + (int64_t)a * Nv;
    const double *fz = c.Pz ? c.Pz + so : nullptr;
    const double *Sij = c.x + c.sl(BS, i, j) + (int64_t)a * Nv, *Si0 = c.x + c.sl(BS, i, 0) + (int64_t)a * Nv;
    const double *T0j = c.x + c.sl(BT, 0, j), *Y0j = c.x + c.sl(BY, 0, j);   // row 0
    const double *t1 = (i0 ? c.OC1 + ((int64_t)BZ * No + j) * c.NvNv : c.x + c.sl(BZ, 0, j)) + (int64_t)a * Nv;
    const double *t2 = c.x + c.sl(BZ, i, 0) + (int64_t)a * Nv;
    const double *F0 = c.F + No, *Fj = c.F + (int64_t)j * c.N + No;
    const double cxe = -c.omega + (c.v(0, 0) - c.o(0, 0)) - (SIG ? 0.0 : c.o(i, i) + c.o(j, j)), s1 = i0 ? 1.0 : c.o(0, i), s2 = c.o(0, j);
    const double f00 = c.ov(0, 0), fj0 = c.ov(j, 0), foai = c.ov(i, a), sija0 = Sij[0], si0a0 = Si0[0];
    const double fy = (i0 ? c.v(a, 0) : 0.0) - (a == 0 ? c.o(0, i) : 0.0);
    double xa0 = 0.0, fva = 0.0, fvaa = 0.0;
    const double *x0 = nullptr, *Fv0 = c.F + (int64_t)No * c.N + No;
    if constexpr (AV) {
      xa0 = x[0];
      fva = c.v(0, a);
      fvaa = c.v(a, a);
      x0 = c.x + (int64_t)BZ * c.B + (int64_t)s * c.NvNv;
    }
    for (int b = lane; b < Nv; b += 32) {
      double rb = 0.0;
      if (b != 0) {
        const double xe = x[b];
        double u = cxe * xe + f00 * Sij[b] - __ldg(F0 + b) * sija0 - fj0 * Si0[b] + __ldg(Fj + b) * si0a0 + foai * T0j[b];
        if constexpr (!SIG) u -= s1 * t1[b] + s2 * t2[b];
        if (i0 || a == 0) u += fy * Y0j[b];
        if constexpr (AV) {
          u += c.v(b, b) * xe + xa0 * __ldg(Fv0 + b);
          u += a == 0 ? c.kap[(int64_t)s * Nv + b] : fvaa * xe + fva * x0[b];
        } else {
          u += yz[b];
          if (fz) u += fz[b];
        }
        rb = SIG ? u : -bv[b] - u;
        nrm += (SIG ? xe : rb) * rb;
      }
      r[b] = rb;
    }
  }
  cta_partial(2.0 * nrm, c.red + c.base + blockIdx.x);
}

// All blocks in one launch (grid.y: T, X, Y, Z, S): the small sizes are bound by their launches.  SIG
// without the S part: S of an arbitrary input is left to the element-wise pass of sigma.cu.
template <bool AV, bool SIG>
__global__ void __launch_bounds__(kThreads) k_sym_pass(const __grid_constant__ RC cin) {
  __shared__ Tile t[3];
  RC c = cin;
  c.base = (int64_t)blockIdx.y * kGrid;
  switch (blockIdx.y) {
    case 0: kr_anti<BT, AV, SIG>(c, t[0]); break;
    case 1: kr_anti<BX, AV, SIG>(c, t[0]); break;
    case 2: kr_anti<BY, AV, SIG>(c, t[0]); break;
    case 3: kr_z<AV, SIG>(c); break;
    default: kr_s<AV, SIG>(c, t[0], t[1], t[2]); break;
  }
}

// ---- arrow sums over an occupied index, weights as launch parameters (constant operands)
struct ArrowW64 {
  double fl[32];  // F_l,t for 1 <= l < No, else 0
  double fk[32];  // F_l,t' for l < No, else 0
};
// T, X, Y from the slices i < j: OC1[m] = sum_{l>=1} F_lt x_lm (x_lm = -x_ml for l > m), X also OX[m] =
// sum_l F_l,t' X_lm
template <int BLK>
__device__ __forceinline__ void kr_arrow_anti(int No, int m, int64_t NvNv, int64_t B, int64_t e, const double *__restrict__ x,
                                              double *oc1, double *ox, const ArrowW64 &w) {
  constexpr bool WX = BLK == BX;
  const double *xb = x + BLK * B + e;
  double c = 0.0, r = 0.0, cx = 0.0, rx = 0.0;
#pragma unroll 8
  for (int l = 0; l < m; ++l) {
    const double v = xb[(int64_t)(l * No + m) * NvNv];
    c += w.fl[l] * v;
    if (WX) cx += w.fk[l] * v;
  }
#pragma unroll 8
  for (int l = m + 1; l < No; ++l) {
    const double v = xb[(int64_t)(m * No + l) * NvNv];
    r += w.fl[l] * v;
    if (WX) rx += w.fk[l] * v;
  }
  oc1[((int64_t)BLK * No + m) * NvNv + e] = c - r;
  if (WX) ox[(int64_t)m * NvNv + e] = cx - rx;
}
// S, Z: OC1[m] = sum_{l>=1} F_lt x_lm; Z also OZ[m] = sum_l F_l,t' Z_ml
template <int BLK>
__device__ __forceinline__ void kr_arrow_full(int No, int m, int64_t NvNv, int64_t B, int64_t e, const double *__restrict__ x,
                                              double *oc1, double *oz, const ArrowW64 &w) {
  const double *xb = x + BLK * B + e;
  double c = 0.0, z = 0.0;
#pragma unroll 8
  for (int l = 0; l < No; ++l) {
    c += w.fl[l] * xb[(int64_t)(l * No + m) * NvNv];
    if (BLK == BZ) z += w.fk[l] * xb[(int64_t)(m * No + l) * NvNv];
  }
  oc1[((int64_t)BLK * No + m) * NvNv + e] = c;
  if (BLK == BZ) oz[(int64_t)m * NvNv + e] = z;
}

// One thread per sum: the CTAs of one range of elements (a, b) and all m run side by side, so the second
// read of an amplitude (as x_lm and as -x_ml) hits L2.  Bound by float64 (two to four operations per
// amplitude).  A thread that kept every sum of an element in registers had No times fewer threads:
// No=20 Nv=200 0.57 ms, No=30 Nv=400 3.1 ms; this form 1.8 ms at the latter, 1.7 ms of float64 work.
__global__ void __launch_bounds__(128) k_arrow_sums(int No, int64_t NvNv, int64_t B, const double *__restrict__ x, double *oc1,
                                                    double *ox, double *oz, const __grid_constant__ ArrowW64 w) {
  const int m = blockIdx.x % No;
  const int64_t e = (int64_t)(blockIdx.x / No) * 128 + threadIdx.x;
  if (e >= NvNv) return;
  switch (blockIdx.y) {   // X first: it does the most
    case 0: kr_arrow_anti<BX>(No, m, NvNv, B, e, x, oc1, ox, w); break;
    case 1: kr_arrow_full<BZ>(No, m, NvNv, B, e, x, oc1, oz, w); break;
    case 2: kr_arrow_full<BS>(No, m, NvNv, B, e, x, oc1, oz, w); break;
    case 3: kr_arrow_anti<BT>(No, m, NvNv, B, e, x, oc1, ox, w); break;
    default: kr_arrow_anti<BY>(No, m, NvNv, B, e, x, oc1, ox, w); break;
  }
}

// Hylleraas sums <b, x> and <x, A x> = <x, -b - r> per block on the same independent slices (T, X, Y:
// i < j, counted twice): 10 partials per CTA.  grid.y = block.
__global__ void __launch_bounds__(256) kr_hyll(int No, int64_t NvNv, int64_t B, const double *b, const double *x, const double *r,
                                               double *red) {
  const int blk = blockIdx.y;
  const bool anti = blk == BT || blk == BX || blk == BY;
  const int ns = anti ? No * (No - 1) / 2 : No * No;
  double s0 = 0.0, s1 = 0.0;
  for (int s = blockIdx.x; s < ns; s += gridDim.x) {
    int sl = s;
    if (anti) {
      int k = s, i = 0;
      while (k >= No - 1 - i) { k -= No - 1 - i; ++i; }
      sl = i * No + i + 1 + k;
    }
    const int64_t off = blk * B + (int64_t)sl * NvNv;
    for (int64_t e = threadIdx.x; e < NvNv; e += 256) {
      const double bi = b[off + e], xi = x[off + e];
      s0 = fma(bi, xi, s0);
      s1 = fma(xi, -bi - r[off + e], s1);
    }
  }
  const double f = anti ? 2.0 : 1.0;
  __shared__ double sh[2][8];
  s0 = warp_sum(s0);
  s1 = warp_sum(s1);
  if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = s0; sh[1][threadIdx.x >> 5] = s1; }
  __syncthreads();
  if (threadIdx.x < 2) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += sh[threadIdx.x][w];
    red[(int64_t)(2 * blk + threadIdx.x) * gridDim.x + blockIdx.x] = f * t;
  }
}

}  // namespace

namespace {
void fill(esmp2_handle *h, RC &c, const double *F, const double *x) {
  c.No = h->d.No; c.Nv = h->d.Nv; c.N = h->d.N;
  c.NvNv = (int64_t)h->d.Nv * h->d.Nv;
  c.B = h->d.B;
  c.F = F;
  c.omega = h->omega_op;
  c.x = x;
  c.VX = h->cp.VX; c.WZ = h->cp.WZ; c.OC1 = h->cp.OC1; c.OX = h->cp.OX; c.OZ = h->cp.OZ;
  c.G = h->cp.G; c.H = h->cp.H; c.CYZ = h->cp.CYZ;
  c.red = h->red;
}
}  // namespace

int residual_parts() { return 5 * kGrid; }

// r = -b - A x (the independent slices), partials of <r, r>_w in h->red (residual_parts()); x with the
// singlet symmetries bit for bit.  levels: digit levels of the virtual-index products, 0 float64
// GEMMs; h->arrowv: the reduced-cost basis (element-wise virtual-index terms).
esmp2_status residual_sym(esmp2_handle *h, const double *x, const double *b, double *r, int levels) {
  const int No = h->d.No, Nv = h->d.Nv, N = h->d.N, NN = No * No;
  const int64_t NvNv = (int64_t)Nv * Nv, B = h->d.B;
  cudaStream_t st = h->stream;
  const bool av = h->arrowv;
  const double *F = av ? h->Farr : h->Fsemi;
  double *q = h->s64.q;
  esmp2_status s = ensure_slist(h);
  if (!s && !av) s = ensure_p64(h, levels ? 5 : 4);   // the element-wise form has no products to hold
  if (s) return s;
  RC c{};
  c.P = av ? x : h->P64;   // (av: not read)
  if (av) {
    virt_arrow_sums(h, x);
    c.rho = h->rho64;
    c.kap = h->kap64 + (int64_t)BZ * NN * Nv;
    c.yz = x;   // not read
  } else if (levels) {
    if ((s = virt_split(h, x, q, h->P64, 2, levels, false))) return s;
    c.yz = q + BZ * B;
    c.Pz = h->P64;
  } else {   // T, X, Y, S one-sided, Z both terms
    virt64_list(h, F + (int64_t)No * N + No, N, x, q, h->P64, h->slist, h->nslist - NN, h->nslist);
    c.yz = q + BZ * B;
  }
  ArrowW64 w;
  for (int l = 0; l < 32; ++l) { w.fl[l] = h->arrow_w64[l]; w.fk[l] = h->arrow_w64[32 + l]; }
  const unsigned ga = (unsigned)(No * cdiv(NvNv, 128));
  k_arrow_sums<<<dim3(ga, 5), 128, 0, st>>>(No, NvNv, B, x, h->cp.OC1, h->cp.OX, h->cp.OZ, w);
  launch_intermediates64(h, F, 2, x);
  fill(h, c, F, x);
  c.b = b;
  c.r = r;
  {
    const double bytes = 8.0 * (double)(h->nslist) * NvNv * (av ? 3.0 : 4.0);
    KScope ks(st, ESMP2_KT_COUPLING, bytes, bytes);
    if (av) k_sym_pass<true, false><<<dim3(kGrid, 5), kThreads, 0, st>>>(c);
    else k_sym_pass<false, false><<<dim3(kGrid, 5), kThreads, 0, st>>>(c);
  }
  h->launches += 2;
  return check_cuda(h, cudaGetLastError(), "residual");
}

// The last stage of the float64 sigma in the TOP basis (No <= 32): y from the products P64 with the
// occupied sums folded in (T, X, Y; with s_sym also S) and the Z part already in y; the partials of
// <x, y> over these blocks go to h->red (T, X, Y, Z and, with s_sym, S: residual_parts() in all).
esmp2_status sigma_sym_tail(esmp2_handle *h, const double *x, double *y, bool s_sym, cudaEvent_t after_inter) {
  RC c{};
  launch_intermediates64(h, h->F, 0, x);
  if (after_inter) cudaEventRecord(after_inter, h->stream);
  fill(h, c, h->F, x);
  c.P = h->P64;
  c.yz = y + BZ * h->d.B;
  c.r = y;
  const double bytes = 24.0 * (double)h->d.n * (s_sym ? 1.0 : 0.8);
  KScope ks(h->stream, ESMP2_KT_COUPLING, bytes, bytes);
  k_sym_pass<false, true><<<dim3(kGrid, s_sym ? 5 : 4), kThreads, 0, h->stream>>>(c);
  h->launches += 1;
  return check_cuda(h, cudaGetLastError(), "sigma64");
}

// per-block Hylleraas partials (2 x 5 quantities of hyll_parts() CTAs) from the residual of residual_sym
int hyll_parts() { return 304; }
void hylleraas_sym(esmp2_handle *h, const double *b, const double *x, const double *r) {
  kr_hyll<<<dim3((unsigned)hyll_parts(), 5), 256, 0, h->stream>>>(h->d.No, (int64_t)h->d.Nv * h->d.Nv, h->d.B, b, x, r, h->red);
  h->launches += 1;
}

}  // namespace esmp2
