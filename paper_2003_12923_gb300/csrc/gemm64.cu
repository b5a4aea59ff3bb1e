// Float64 strided batched GEMM and 4-index mode products.
//
// GB300 executes float64 at two multiply-adds per clock and SM (half of one per scheduler), so
// every float64 contraction here is bound by the number of multiply-adds issued, not by loads:
// a 32 x 32 x 16 tile step takes the pipe 8192 clocks against 8 KB of operands.  What matters
// is therefore (1) no multiply-adds on padding, (2) every scheduler of every SM busy:
//   * CTA tile 32 x 32, four warps of 16 x 16; a warp trims its own tile to the matrix in steps of
//     4 rows and 8 columns and the last K chunk to its length (M = No = 20 issues 20 rows, not 64);
//     the warps trade places with the block index so that the trimmed ones do not all sit on the
//     same scheduler;
//   * too few tiles for the chip and a long K: K is cut into slices of at least 64 with their own
//     CTAs, the partial results are summed in a fixed order by a second kernel.
// Measured against 64 x 64 x 16 tiles padded in M, N and K and no K slices: the GEMMs of a gradient of
// No=12 Nv=120 1948 -> 3.8 ms (densities on half of the tiles by symmetry, each sum once); a float64 sigma
// of No=6 Nv=30 0.90 -> 0.094 ms (21 launches of one under-filled wave each, now k_virt64 and the passes of
// sigma.cu and resid.cu), of No=13 Nv=113 10.7 -> 3.65 ms.
#include <algorithm>

#include "internal.h"

namespace esmp2 {
namespace {

constexpr int TS = 32, BK = 16, NT = 128;
constexpr int kSplitTarget = 152 * 6;          // CTAs that keep every scheduler of 152 SMs busy
constexpr int64_t kSplitBytes = 64 << 20;      // limit of the partial results

// one K chunk of a warp's 16 x 16 tile: rows r0 + 4 i (i < mi), columns c0 + 8 j (j < nj) per lane
__device__ __forceinline__ void chunk(const double (*As)[TS + 1], const double (*Bs)[TS + 1], int kn, int r0, int c0,
                                      int mi, int nj, double (&acc)[4][2]) {
  if (mi == 4 && nj == 2) {
#pragma unroll 4
    for (int k = 0; k < kn; ++k) {
      double a[4], b[2];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[k][r0 + 4 * i];
#pragma unroll
      for (int j = 0; j < 2; ++j) b[j] = Bs[k][c0 + 8 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
  } else if (mi > 0 && nj > 0) {
    for (int k = 0; k < kn; ++k) {
      const double b0 = Bs[k][c0], b1 = Bs[k][c0 + 8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (i < mi) {   // uniform over the warp
          const double a = As[k][r0 + 4 * i];
          acc[i][0] = fma(a, b0, acc[i][0]);
          if (nj == 2) acc[i][1] = fma(a, b1, acc[i][1]);
        }
      }
    }
  }
}

__global__ void __launch_bounds__(NT) gemm64_kernel(Gemm64 g, int mtiles, int ntiles, int kper, double *part) {
  __shared__ double As[BK][TS + 1];
  __shared__ double Bs[BK][TS + 1];
  const int tid = threadIdx.x, lane = tid & 31, role = ((tid >> 5) + (int)blockIdx.x) & 3;
  const int ks = (int)(blockIdx.x / ((int64_t)mtiles * ntiles));
  const int tile = (int)(blockIdx.x % ((int64_t)mtiles * ntiles));
  const int m0 = (tile % mtiles) * TS, n0 = (tile / mtiles) * TS;
  if (g.sym && m0 > n0) return;   // the mirror of tile (n0, m0)
  const int wm = (role >> 1) * 16, wn = (role & 1) * 16, ly = lane >> 3, lx = lane & 7;
  const int64_t bz = blockIdx.y;
  const double *A = g.A + bz * g.sAb;
  const double *B = g.B + bz * g.sBb;
  const bool a_kfast = g.sAk == 1;
  const bool b_nfast = g.sBn == 1 || g.sBk != 1;
  const int kbeg = ks * kper, kend = min(g.K, kbeg + kper);
  // rows in steps of 4 and columns in steps of 8 that this warp has inside the matrix
  const int mi = max(0, min(4, (g.M - m0 - wm + 3) >> 2)), nj = max(0, min(2, (g.N - n0 - wn + 7) >> 3));
  double acc[4][2] = {};
  double ra[4], rb[4];
  auto kslice = [&](int gk) { return !g.klist ? gk / g.Kin : gk < kend ? __ldg(g.klist + gk / g.Kin) : 0; };
  auto load = [&](int k0) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int idx = tid + NT * r;
      int m, k;
      if (a_kfast) { k = idx % BK; m = idx / BK; } else { m = idx % TS; k = idx / TS; }
      int gk = k0 + k;
      int64_t ko = (int64_t)gk * g.sAk;
      if (g.Kin > 0) ko = (int64_t)kslice(gk) * g.sAk1 + (int64_t)(gk % g.Kin) * g.sAk;
      ra[r] = (m0 + m < g.M && gk < kend) ? A[(int64_t)(m0 + m) * g.sAm + ko] : 0.0;
      int n;
      if (b_nfast) { n = idx % TS; k = idx / TS; } else { k = idx % BK; n = idx / BK; }
      gk = k0 + k;
      ko = (int64_t)gk * g.sBk;
      if (g.Kin > 0) ko = (int64_t)kslice(gk) * g.sBk1 + (int64_t)(gk % g.Kin) * g.sBk;
      rb[r] = (n0 + n < g.N && gk < kend) ? B[ko + (int64_t)(n0 + n) * g.sBn] : 0.0;
    }
  };
  if (kbeg < kend) load(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int idx = tid + NT * r;
      if (a_kfast) As[idx % BK][idx / BK] = ra[r]; else As[idx / TS][idx % TS] = ra[r];
      if (b_nfast) Bs[idx / TS][idx % TS] = rb[r]; else Bs[idx % BK][idx / BK] = rb[r];
    }
    __syncthreads();
    if (k0 + BK < kend) load(k0 + BK);   // in flight while the pipe works on this chunk
    chunk(As, Bs, min(BK, kend - k0), wm + ly, wn + lx, mi, nj, acc);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int gm = m0 + wm + ly + 4 * i;
    if (gm >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int gn = n0 + wn + lx + 8 * j;
      if (gn >= g.N) continue;
      if (part) {
        part[(((int64_t)ks * gridDim.y + bz) * g.M + gm) * g.N + gn] = acc[i][j];
      } else {
        double *c = g.C + bz * g.sCb + (int64_t)gm * g.sCm + (int64_t)gn * g.sCn;
        *c = (g.beta == 0.0) ? g.alpha * acc[i][j] : fma(g.alpha, acc[i][j], g.beta * *c);
        if (g.sym && m0 < n0) {
          c = g.C + bz * g.sCb + (int64_t)gn * g.sCm + (int64_t)gm * g.sCn;
          *c = (g.beta == 0.0) ? g.alpha * acc[i][j] : fma(g.alpha, acc[i][j], g.beta * *c);
        }
      }
    }
  }
}

// C = alpha sum_k part[k] + beta C, in a fixed order: 32 elements per CTA, eight threads each (a small C
// comes with many slices, and one thread per element was a chain of up to 900 loads)
__global__ void __launch_bounds__(256) gemm64_sum(Gemm64 g, int nsplit, const double *part) {
  __shared__ double sh[8][33];
  const int64_t per = (int64_t)g.batch * g.M * g.N;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int64_t e0 = (int64_t)blockIdx.x * 32; e0 < per; e0 += (int64_t)gridDim.x * 32) {
    const int64_t e = e0 + tx, f = e / g.N;
    const int n = (int)(e - f * g.N), m = (int)(f % g.M);
    const int64_t src = g.sym && m / TS > n / TS ? e + (int64_t)(n - m) * g.N + (m - n) : e;   // element (n, m)
    double s = 0.0;
    if (e < per) {
#pragma unroll 4
      for (int k = ty; k < nsplit; k += 8) s += part[k * per + src];
    }
    sh[ty][tx] = s;
    __syncthreads();
    if (ty == 0 && e < per) {
      for (int w = 1; w < 8; ++w) s += sh[w][tx];
      double *c = g.C + (f / g.M) * g.sCb + (int64_t)m * g.sCm + (int64_t)n * g.sCn;
      *c = (g.beta == 0.0) ? g.alpha * s : fma(g.alpha, s, g.beta * *c);
    }
    __syncthreads();
  }
}

// Virtual-index terms of the float64 sigma, every listed slice in one launch: the first n_one
// entries of the list take P_s = x_s F, the others y_s = x_s F + F x_s (both terms in one
// accumulator).  One CTA per 32 x 32 tile of a slice, trimmed like the GEMM's.  A launch per row
// of slices and term kept the small sizes to a few SMs at a time.
__global__ void __launch_bounds__(NT) k_virt64(const double *Fv, int ldF, const double *x, double *y, double *P, int Nv,
                                               const int *list, int n_one, int nt) {
  __shared__ double As[BK][TS + 1];
  __shared__ double Bs[BK][TS + 1];
  const int tid = threadIdx.x, lane = tid & 31, role = ((tid >> 5) + (int)blockIdx.x) & 3;
  const int li = (int)(blockIdx.x / (unsigned)(nt * nt)), tt = (int)(blockIdx.x % (unsigned)(nt * nt));
  const int m0 = (tt / nt) * TS, n0 = (tt % nt) * TS;
  const int wm = (role >> 1) * 16, wn = (role & 1) * 16, ly = lane >> 3, lx = lane & 7;
  const int64_t off = (int64_t)list[li] * Nv * Nv;
  const double *xs = x + off;
  double *out = (li < n_one ? P : y) + off;
  const int mi = max(0, min(4, (Nv - m0 - wm + 3) >> 2)), nj = max(0, min(2, (Nv - n0 - wn + 7) >> 3));
  const int nc = (Nv + BK - 1) / BK, total = li < n_one ? nc : 2 * nc;
  double acc[4][2] = {};
  double ra[4], rb[4];
  auto load = [&](int q) {   // chunk q: term 1 (x rows, F) then term 2 (F rows, x)
    const bool t1 = q < nc;
    const int k0 = (t1 ? q : q - nc) * BK;
    const double *A = t1 ? xs : Fv, *B = t1 ? Fv : xs;
    const int64_t lda = t1 ? Nv : ldF, ldb = t1 ? ldF : Nv;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int idx = tid + NT * r, k = idx % BK, m = idx / BK, n = idx % TS, kb = idx / TS;
      ra[r] = (m0 + m < Nv && k0 + k < Nv) ? A[(m0 + m) * lda + k0 + k] : 0.0;
      rb[r] = (n0 + n < Nv && k0 + kb < Nv) ? B[(k0 + kb) * ldb + n0 + n] : 0.0;
    }
  };
  load(0);
  for (int q = 0; q < total; ++q) {
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int idx = tid + NT * r;
      As[idx % BK][idx / BK] = ra[r];
      Bs[idx / TS][idx % TS] = rb[r];
    }
    __syncthreads();
    if (q + 1 < total) load(q + 1);
    chunk(As, Bs, min(BK, Nv - (q < nc ? q : q - nc) * BK), wm + ly, wn + lx, mi, nj, acc);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int a = m0 + wm + ly + 4 * i;
    if (a >= Nv) continue;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int b = n0 + wn + lx + 8 * j;
      if (b < Nv) out[(int64_t)a * Nv + b] = acc[i][j];
    }
  }
}

}  // namespace

void virt64_list(esmp2_handle *h, const double *Fv, int ldF, const double *x, double *y, double *P, const int *list,
                 int n_one, int n_list) {
  const int Nv = h->d.Nv, nt = (int)cdiv(Nv, TS);
  const double nv3 = (double)Nv * Nv * Nv, flops = 2.0 * nv3 * n_one + 4.0 * nv3 * (n_list - n_one);
  KScope ks(h->stream, ESMP2_KT_GEMM64, flops, flops);
  k_virt64<<<(unsigned)((int64_t)n_list * nt * nt), NT, 0, h->stream>>>(Fv, ldF, x, y, P, Nv, list, n_one, nt);
  h->launches += 1;
}

void gemm64(const Gemm64 &g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return;
  const int mtiles = (int)cdiv(g.M, TS), ntiles = (int)cdiv(g.N, TS);
  const int64_t tiles = (int64_t)mtiles * ntiles;
  const int64_t active = g.sym ? (int64_t)mtiles * (mtiles + 1) / 2 : tiles;   // tiles that compute
  const double flops = 2.0 * g.M * (double)g.N * g.K * g.batch;
  KScope ks(st, ESMP2_KT_GEMM64, flops, flops);
  // K slices: when the tiles alone leave more than half of the schedulers idle and every slice
  // keeps at least 64 steps (so that its result's write and read stay small beside its work)
  int nsplit = 1;
  double *part = nullptr;
  if (active * g.batch * 2 <= kSplitTarget && g.K >= 128) {
    const int64_t per = (int64_t)g.batch * g.M * g.N * (int64_t)sizeof(double);
    nsplit = (int)std::max<int64_t>(1, std::min<int64_t>({cdiv(kSplitTarget, active * g.batch), g.K / 64, kSplitBytes / per}));
    if (nsplit > 1 && dmalloc(reinterpret_cast<void **>(&part), (size_t)(nsplit * per), st) != cudaSuccess) {
      cudaGetLastError();
      part = nullptr;
      nsplit = 1;
    }
  }
  const int kper = (int)(cdiv(cdiv(std::max(g.K, 1), nsplit), BK) * BK);
  if (part) {   // batch <= kSplitTarget here: one launch
    nsplit = (int)cdiv(g.K, kper);
    gemm64_kernel<<<dim3((unsigned)(tiles * nsplit), (unsigned)g.batch), NT, 0, st>>>(g, mtiles, ntiles, kper, part);
    gemm64_sum<<<(unsigned)std::min<int64_t>(cdiv((int64_t)g.batch * g.M * g.N, 32), 1216), 256, 0, st>>>(g, nsplit, part);
    dfree(part, st);
    return;
  }
  for (int b0 = 0; b0 < g.batch; b0 += 65535) {
    Gemm64 gg = g;
    gg.batch = std::min(65535, g.batch - b0);
    gg.A = g.A + (int64_t)b0 * g.sAb;
    gg.B = g.B + (int64_t)b0 * g.sBb;
    gg.C = g.C + (int64_t)b0 * g.sCb;
    gemm64_kernel<<<dim3((unsigned)tiles, (unsigned)gg.batch), NT, 0, st>>>(gg, mtiles, ntiles, kper, nullptr);
  }
}

void mode_product(const double *in, double *out, const int dims[4], int mode, const double *R,
                  int Kout, int64_t ldR, cudaStream_t st) {
  int64_t P = 1, Q = 1;
  for (int k = 0; k < mode; ++k) P *= dims[k];
  for (int k = mode + 1; k < 4; ++k) Q *= dims[k];
  const int Kin = dims[mode];
  Gemm64 g{};
  g.alpha = 1.0; g.beta = 0.0;
  if (Q == 1) {  // out[p][k'] = sum_k in[p][k] R[k][k']
    g.M = (int)P; g.N = Kout; g.K = Kin; g.batch = 1;
    g.A = in; g.sAm = Kin; g.sAk = 1; g.sAb = 0;
    g.B = R; g.sBk = ldR; g.sBn = 1; g.sBb = 0;
    g.C = out; g.sCm = Kout; g.sCn = 1; g.sCb = 0;
  } else {       // out_p[k'][q] = sum_k R[k][k'] in_p[k][q]
    g.M = Kout; g.N = (int)Q; g.K = Kin; g.batch = (int)P;
    g.A = R; g.sAm = 1; g.sAk = ldR; g.sAb = 0;
    g.B = in; g.sBk = Q; g.sBn = 1; g.sBb = (int64_t)Kin * Q;
    g.C = out; g.sCm = Q; g.sCn = 1; g.sCb = (int64_t)Kout * Q;
  }
  gemm64(g, st);
}

}  // namespace esmp2
