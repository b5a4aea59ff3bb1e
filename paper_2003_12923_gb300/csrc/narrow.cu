// Products with a narrow right factor (at most 32 columns) in float64 accuracy on the tensor cores:
// the rotations of an occupied index (K = No <= 32) and the contraction of the last OVVV index with
// the TOP virtuals (K = Nv, No columns), steps a1 of the transforms and the basis changes of the solves.
//
// Both have only No multiply-adds per element, too few to hide double-float arithmetic on the float32
// pipes (13 operations per multiply-add bound them) and far too many for the float64 pipe.  Here the
// operand is split into eight exact bf16 digit planes of seven bits (digits.cu) on its way through shared
// memory, tcgen05 forms the level sums (levels 2 .. 9, exact in fp32; 2^-55 of the row's largest element
// times the right factor's), and the levels are joined as integers
// and rounded once: one read and one write of HBM, no digit planes in memory.
// No=30 Nv=400: the rotations of a solve 44 -> 16.2 ms against double-float arithmetic, the OVVV
// contraction 27.4 -> 10.6 ms, 2.4 of them for its row exponents (10.3 ms with six-bit digits and one
// scale per Nv x Nv slice, which lost a row's last bits by as much as it was smaller than its slice: an
// element 2^-30 of it kept 11 bits); No=16 Nv=160 rotations 3.7 -> 1.4 ms.
//
// A tile is 128 result rows; persistent CTAs of 28 warps:
//   warps 0, 1   MMA issuer; TMA of the right factor's digit chunks (OVVV form)
//   warps 4..11  epilogue (two warps per TMEM lane quarter)
//   warps 12..27 conversion: float64 from global memory into the eight planes of a 64-byte-swizzled
//                K-major tile, 16-byte shared-memory stores, the next tile's loads in flight
// Digit p of the operand meets the digits 1 .. 9 - p of the right factor, stacked along N (their
// levels are neighbouring accumulators): eight MMAs per K step instead of 36.  Two sets of
// accumulators (2 x 8 levels x 32 columns fill TMEM): the epilogue of a tile runs beside the next one.
//
// A row with a NaN or infinity has the exponent field 0x7FF as its scale (kBadExp) and gets NaN results, so
// does a column of the right factor with one.  Found once per row, not per element: with NaN digits and a
// look at every result (as in digits.cu) the rotations of No=30 Nv=400 took 16.9 ms.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.h"
#include "digit_split.h"
#include "tc_ptx.h"

namespace esmp2 {
namespace nr {

using namespace ptx;

constexpr int P = 8;                    // digit planes of both operands
constexpr int BM = 128, BK = 32;
// Longest sum over K of one launch: every level sum stays below 2^24 (8 pairs x 2^12 x 480) and the joined
// integer below 2^63 (480 / 4 x 2^56).  The OVVV product of a larger Nv runs in K ranges of equal length,
// added in float64.
constexpr int K_MAX = 480;
constexpr int W = 7;                    // bits per digit
constexpr int A_PLANE = BM * 64, A_STAGE = P * A_PLANE;   // 64 KB
// result columns of a tile, 32 or 16 (No <= 16)
template <int BN> constexpr int b_plane() { return BN * 64; }
template <int BN> constexpr int smem_bytes() { return 1024 + 2 * A_STAGE + 2 * P * b_plane<BN>(); }
constexpr int NTHREADS = 896;

struct Args {
  const double *in;
  double *out;
  int64_t rows, tiles;
  int K, N, nk;      // K: length of the sum of this launch
  int64_t Q;         // occupied form: row c = p Q + q reads in[(p K + k) Q + q], writes out[(p N + n) Q + q]
  const double *R;   // occupied form: right factor, K x N row-major
  const int *es;     // OVVV form: binary exponent of every row, ...
  const int *eR;     // ... that of the right factor, a mask of its columns with a NaN or infinity,
  int ld, k0, add;   // ... row pitch, first K element, and whether out is added to
  int vec;           // OVVV form: 16-byte loads
  int *err;
};

// byte offset of 16-byte group c of row r in a K-major tile of 64-byte rows, 64-byte swizzle
__device__ __forceinline__ uint32_t sw64(int r, int c) { return (uint32_t)(r * 64 + ((c ^ ((r >> 1) & 3)) << 4)); }

// digits of eight consecutive K elements of one row, 16 bytes per plane, to dst + (p - 1) pitch
__device__ __forceinline__ void put_digits(uint8_t *dst, int64_t pitch, const double (&v)[8], int e) {
  long long U[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) U[k] = digit_word<P, W>(v[k], e);
  uint32_t sg[4], rg[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    sg[k] = sign_pair(v[2 * k], v[2 * k + 1]);
    rg[k] = range_pair(v[2 * k], v[2 * k + 1]);
  }
#pragma unroll
  for (int p = 1; p <= P; ++p)
    *reinterpret_cast<uint4 *>(dst + (p - 1) * pitch) =
        make_uint4(digit_pair<P, W>(U[0], U[1], sg[0], rg[0], p), digit_pair<P, W>(U[2], U[3], sg[1], rg[1], p),
                   digit_pair<P, W>(U[4], U[5], sg[2], rg[2], p), digit_pair<P, W>(U[6], U[7], sg[3], rg[3], p));
}
__device__ __forceinline__ void store_digits(uint8_t *tile, int plane_bytes, int row, int c, const double (&v)[8], int e) {
  put_digits(tile + sw64(row, c), plane_bytes, v, e);
}
__device__ __forceinline__ int hi_abs(double v) { return __double2hiint(v) & 0x7FFFFFFF; }   // high word of |v|
__device__ __forceinline__ int hi_finite(double v) { return non_finite(v) ? 0 : hi_abs(v); }
// binary exponent of a row whose largest hi_abs is hi (as k_slice_exp; kBadExp: it is not finite)
constexpr int kBadExp = 2047 - 1021;
__device__ __forceinline__ int exp_of(int hi) { return hi >> 20 ? (hi >> 20) - 1021 : 0; }

// OVVV form: binary exponent of every row (length n, pitch n), a warp per row.  The scale of the whole Nv x Nv slice would cost a small row the bits it is smaller by.
// (No=30 Nv=400: the pass over 15.4 GB takes 2.4 ms, one CTA per slice took 2.0.)
__global__ void __launch_bounds__(256) k_row_exp(const double *x, int64_t rows, int n, int *es) {
  const int lane = threadIdx.x & 31;
  const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (r >= rows) return;
  const double *src = x + r * n;
  int m = 0;
#pragma unroll 8
  for (int c = lane; c < n; c += 32) m = max(m, hi_abs(src[c]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) es[r] = exp_of(m);
}

// OVVV form: digit planes of the right factor, out[p][n][k] (row pitch Kp) from column n < N of M (K x ldM),
// rows N .. bn and the pad columns zero; eR: its exponent and the mask of its non-finite columns; one CTA
__global__ void __launch_bounds__(1024) k_factor_digits(const double *M, int ldM, int K, int N, int Kp, int bn,
                                                        __nv_bfloat16 *out, int *eR) {
  __shared__ int mx;
  __shared__ unsigned bad;
  if (threadIdx.x == 0) { mx = 0; bad = 0; }
  __syncthreads();
  int m = 0;
  for (int u = threadIdx.x; u < K * N; u += 1024) {
    const double v = M[(int64_t)(u / N) * ldM + u % N];
    m = max(m, hi_finite(v));
    if (non_finite(v)) atomicOr(&bad, 1u << (u % N));
  }
  atomicMax(&mx, m);
  __syncthreads();
  const int e = exp_of(mx);
  if (threadIdx.x == 0) { eR[0] = e; eR[1] = (int)bad; }
  for (int u = threadIdx.x; u < bn * (Kp >> 3); u += 1024) {
    const int n = u % bn, c = (u / bn) * 8;
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = (n < N && c + k < K) ? M[(int64_t)(c + k) * ldM + n] : 0.0;
    put_digits(reinterpret_cast<uint8_t *>(out + (int64_t)n * Kp + c), (int64_t)bn * Kp * 2, v, e);
  }
}

// ROW: OVVV form; BN: result columns.  A conversion thread takes
// eight K elements of a row; the occupied form with BN = 16 has K <= 16 and half as many of these per
// tile, so its two halves of the conversion warps take turns.
template <bool ROW, int BN>
__global__ void __launch_bounds__(NTHREADS, 1) k_narrow(const __grid_constant__ CUtensorMap tB, const __grid_constant__ Args g) {
  constexpr int B_PLANE = b_plane<BN>(), B_STAGE = P * B_PLANE, ACC = 256;   // TMEM columns per accumulator set
  constexpr bool HALF = !ROW && BN == 16;
  constexpr bool SMALL = !ROW;   // occupied form (K <= 32): every level sum is below 2^20
  constexpr int CW = HALF ? 8 : 16;   // conversion warps per chunk
  extern __shared__ uint8_t smem_raw[];
  uint8_t *sA = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *sB = sA + 2 * A_STAGE;
  __shared__ uint64_t a_full[2], a_empty[2], b_full[2], acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_base;
  __shared__ int fail, rmax, rexp[8][BM];
  __shared__ unsigned rbad;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) { mbar_init(&a_full[s], CW); mbar_init(&a_empty[s], 1); mbar_init(&b_full[s], 1); mbar_init(&acc_full[s], 1); mbar_init(&acc_empty[s], 8); }
    fail = 0;
    rmax = 0;
    rbad = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int k = threadIdx.x; k < 8 * BM; k += NTHREADS) (&rexp[0][0])[k] = 0;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  int eR = 0;
  if constexpr (ROW) {
    eR = __ldg(g.eR);
  } else {   // the right factor's digits, row n = column n of R, once per CTA
    __syncthreads();
    int m = 0;
    for (int e = threadIdx.x; e < g.K * g.N; e += NTHREADS) {
      m = max(m, hi_finite(g.R[e]));
      if (non_finite(g.R[e])) atomicOr(&rbad, 1u << (e % g.N));
    }
    atomicMax(&rmax, m);
    __syncthreads();
    eR = exp_of(rmax);
    for (int u = threadIdx.x; u < BN * 4; u += NTHREADS) {   // (every K group: unused ones are zero)
      const int n = u >> 2, c = u & 3;
      double v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = (n < g.N && c * 8 + k < g.K) ? g.R[(c * 8 + k) * g.N + n] : 0.0;
      store_digits(sB, B_PLANE, n, c, v, eR);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = tmem_base;

  if (warp == 0) {
    if (lane == 0) {  // ------------------------------------------------ MMA issuer
      int st = 0, ab = 0;
      uint32_t ph = 0, aph = 1;
      bool ok = true;
      const uint64_t dA = sdesc64(smem_u32(sA)), dB = sdesc64(smem_u32(sB));
      for (int64_t t = blockIdx.x; t < g.tiles && ok; t += gridDim.x) {
        if (!mbar_wait(&acc_empty[ab], aph)) { ok = false; break; }
        tc_after();
        const uint32_t acc = tmem + (uint32_t)(ab * ACC);
        for (int kc = 0; kc < g.nk; ++kc) {
          if (!mbar_wait(&a_full[st], ph) || (ROW && !mbar_wait(&b_full[st], ph))) { ok = false; break; }
          const int ks = g.K - kc * BK > 16 ? 2 : 1;
          const uint64_t B = dB + (ROW ? (uint64_t)(st * (B_STAGE / 16)) : 0ull);
          for (int k = 0; k < ks; ++k) {
#pragma unroll
            for (int i = 1; i <= P; ++i) {   // operand digit P + 1 - i, right-factor digits 1 .. i
              const uint64_t A = dA + (uint64_t)(st * (A_STAGE / 16) + (P - i) * (A_PLANE / 16) + 2 * k);
              const uint32_t d0 = acc + (uint32_t)((P - i) * BN);
              if (kc == 0 && k == 0) {       // the lowest level of the group is met for the first time
                umma_bf16(d0, A, B, idesc_bf16(BM, BN), 0u);
                if (i > 1) umma_bf16(d0 + BN, A, B + B_PLANE / 16, idesc_bf16(BM, (i - 1) * BN), 1u);
              } else {
                umma_bf16(d0, A, B + 2 * k, idesc_bf16(BM, i * BN), 1u);
              }
            }
          }
          umma_commit(&a_empty[st]);
          st ^= 1;
          ph ^= (uint32_t)(st == 0);
        }
        if (!ok) break;
        umma_commit(&acc_full[ab]);
        ab ^= 1;
        aph ^= (uint32_t)(ab == 0);
      }
      if (!ok) atomicExch(&fail, 1);
    }
  } else if (warp == 1) {
    if (ROW && lane == 0) {  // ------------------------------------------ right-factor chunks
      int st = 0;
      uint32_t ph = 1;
      int64_t it = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < g.tiles && ok; t += gridDim.x)
        for (int kc = 0; kc < g.nk; ++kc, ++it) {
          if (!mbar_wait(&a_empty[st], ph)) { ok = false; break; }
          mbar_expect_tx(&b_full[st], (uint32_t)B_STAGE);
#pragma unroll
          for (int p = 0; p < P; ++p) tma_3d(sB + st * B_STAGE + p * B_PLANE, &tB, &b_full[st], g.k0 + kc * BK, 0, p);
          st ^= 1;
          ph ^= (uint32_t)(st == 0);
        }
      if (!ok) atomicExch(&fail, 1);
      for (int64_t j = it > 2 ? it - 2 : 0; j < it; ++j) mbar_wait(&b_full[j & 1], (uint32_t)((j >> 1) & 1), 100000000ull);
    }
  } else if (warp >= 12) {  // ------------------------------------------- conversion
    const int cw = warp - 12, grp = HALF ? cw >> 3 : 0;
    // occupied form: 8 rows by 4 K groups per warp (HALF: 16 by 2), consecutive lanes on consecutive
    // rows; OVVV form: 8 rows, the 4 K groups of a row on neighbouring lanes
    const int row = HALF ? (cw & 7) * 16 + (lane & 15) : ROW ? cw * 8 + (lane >> 2) : cw * 8 + (lane & 7);
    const int kg = HALF ? lane >> 4 : ROW ? lane & 3 : lane >> 3;
    double v[8];
    auto load = [&](int64_t t, int kc) {
      const int64_t r = t * BM + row;
      if constexpr (!ROW) {
        const int64_t p = r < g.rows ? r / g.Q : 0;
        const double *src = g.in + (p * g.K + kg * 8) * g.Q + (r - p * g.Q);
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = (r < g.rows && kg * 8 + k < g.K) ? src[(int64_t)k * g.Q] : 0.0;
      } else {
        const int k0 = kc * BK + kg * 8;
        const double *src = g.in + r * g.ld + g.k0 + k0;
        if (g.vec) {
#pragma unroll
          for (int k = 0; k < 8; k += 2) {
            const double2 w = (r < g.rows && k0 + k < g.K) ? *reinterpret_cast<const double2 *>(src + k) : make_double2(0.0, 0.0);
            v[k] = w.x;
            v[k + 1] = w.y;
          }
        } else {
#pragma unroll
          for (int k = 0; k < 8; ++k) v[k] = (r < g.rows && k0 + k < g.K) ? src[k] : 0.0;
        }
      }
    };
    // HALF: group 0 fills stage 0 with this CTA's even tiles, group 1 stage 1 with its odd ones
    const int64_t t0 = blockIdx.x + (HALF ? (int64_t)grp * gridDim.x : 0), dt = (HALF ? 2 : 1) * (int64_t)gridDim.x;
    int st = grp, slot = grp;
    uint32_t ph = 1;
    bool ok = true;
    if (t0 < g.tiles) load(t0, 0);
    for (int64_t t = t0; t < g.tiles && ok; t += dt) {
      for (int kc = 0; kc < g.nk; ++kc) {
        double w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k] = v[k];
        if (kc + 1 < g.nk) load(t, kc + 1);   // in flight while this chunk is converted
        else if (t + dt < g.tiles) load(t + dt, 0);
        int e;
        if constexpr (!ROW) {   // the row's own scale: the largest of its K elements
          int m = 0;
#pragma unroll
          for (int k = 0; k < 8; ++k) m = max(m, hi_abs(w[k]));
          if constexpr (!HALF) m = max(m, __shfl_xor_sync(0xffffffffu, m, 8));
          m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
          e = exp_of(m);
          // eight slots: this one was last read eight tiles back, and the conversion of the tile two
          // before this one waited for MMAs that came after the epilogue six tiles back
          if (kg == 0) rexp[slot][row] = m;
        } else {
          const int64_t r = t * BM + row;
          e = r < g.rows ? __ldg(g.es + r) : 0;
        }
        // every warp waits for itself: a wait that runs out ends the conversion for good
        ok = __all_sync(0xffffffffu, mbar_wait(&a_empty[st], ph));
        if (!ok) break;
        store_digits(sA + st * A_STAGE, A_PLANE, row, kg, w, e);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&a_full[st]);
        if constexpr (HALF) {
          ph ^= 1;
        } else {
          st ^= 1;
          ph ^= (uint32_t)(st == 0);
        }
      }
      slot = (slot + (HALF ? 2 : 1)) & 7;
    }
    if (!ok) atomicExch(&fail, 1);
  } else if (warp >= 4) {  // -------------------------------------------- epilogue
    const int quarter = warp & 3, chalf = (warp - 4) >> 2;
    uint32_t lt = 0;
    for (int64_t t = blockIdx.x; t < g.tiles; t += gridDim.x, ++lt) {
      const int ab = (int)(lt & 1);
      if (!mbar_wait(&acc_full[ab], (lt >> 1) & 1)) { if (lane == 0) atomicExch(&fail, 1); break; }
      __syncwarp();
      tc_after();
      const int row = quarter * 32 + lane;
      const int64_t r = t * BM + row;
      const int er = ROW ? (r < g.rows ? __ldg(g.es + r) : 0) : exp_of(rexp[lt & 7][row]), e = er + eR - 56;
      const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(ab * ACC + chalf * (BN / 2));
      double *dst = nullptr;
      int64_t pitch = 1;
      if (r < g.rows) {
        if constexpr (ROW) {
          dst = g.out + r * g.N;
        } else {
          const int64_t p = r / g.Q;
          dst = g.out + p * g.N * g.Q + (r - p * g.Q);
          pitch = g.Q;
        }
      }
#pragma unroll
      for (int c4 = 0; c4 < BN / 8; ++c4) {
        uint32_t q[P][4];
#pragma unroll
        for (int l = 0; l < P; ++l) tmem_ld4(taddr + (uint32_t)(l * BN + c4 * 4), q[l]);
        tmem_wait();
        if (c4 == BN / 8 - 1) {
          tc_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[ab]);   // the MMAs of the tile after the next may start
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float f[P];
#pragma unroll
          for (int l = 0; l < P; ++l) {
            keep(q[l][c]);
            f[l] = __uint_as_float(q[l][c]);
          }
          // in units of the level before the last one, to stay within 64 bits
          const long long V = join_levels<P - 1, SMALL, W, P>(f) + round128(__float2int_rn(f[P - 1]));
          const int n = chalf * (BN / 2) + c4 * 4 + c;
          if (dst && n < g.N) {
            const double v = scale_i64(V, e);
            dst[n * pitch] = ROW && g.add ? dst[n * pitch] + v : v;
          }
        }
      }
      const unsigned bad = er == kBadExp ? ~0u : ROW ? (unsigned)__ldg(g.eR + 1) : rbad;
      if (bad && dst) {
        for (int n = chalf * (BN / 2); n < min(g.N, (chalf + 1) * (BN / 2)); ++n)
          if ((bad >> n) & 1) dst[n * pitch] = __longlong_as_double(0x7FF8000000000000ll);
      }
      __syncwarp();
    }
  }
  tc_before();
  __syncthreads();
  if (warp == 0) {
    tc_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
  if (threadIdx.x == 0 && fail) atomicOr(g.err, 1);
}

template <bool ROW, int BN>
esmp2_status launch(esmp2_handle *h, const CUtensorMap &mB, nr::Args &g) {
  if (g.rows <= 0) return ESMP2_OK;
  constexpr int smem = smem_bytes<BN>();
  if (cudaError_t e = smem_limit_once(reinterpret_cast<const void *>(k_narrow<ROW, BN>), smem))
    return check_cuda(h, e, "k_narrow shared-memory limit");
  g.tiles = cdiv(g.rows, BM);
  g.nk = (g.K + BK - 1) / BK;
  g.err = h->dflag;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  k_narrow<ROW, BN><<<(unsigned)std::min<int64_t>(g.tiles, sms), NTHREADS, smem, h->stream>>>(mB, g);
  h->launches += 1;
  return check_cuda(h, cudaGetLastError(), "k_narrow");
}

}  // namespace nr

// out[p][n][q] = sum_k R[k][n] in[p][k][q] (R: K x K, row pitch K): on the tensor cores for K <= 32, else
// a float64 GEMM.  in and out must not overlap.
esmp2_status mode_product_small(esmp2_handle *h, const double *in, double *out, int64_t P, int K, int64_t Q, const double *R) {
  if (K <= nr::BK) {
    if (esmp2_status s = ensure_dflag(h)) return s;
    nr::Args g{};
    g.in = in; g.out = out;
    g.rows = P * Q;
    g.K = K; g.N = K; g.Q = Q;
    g.R = R;
    return K <= 16 ? nr::launch<false, 16>(h, CUtensorMap{}, g) : nr::launch<false, 32>(h, CUtensorMap{}, g);
  }
  Gemm64 g{};
  g.alpha = 1.0; g.beta = 0.0;
  g.M = K; g.N = (int)Q; g.K = K; g.batch = (int)P;
  g.A = R; g.sAm = 1; g.sAk = K; g.sAb = 0;
  g.B = in; g.sBk = Q; g.sBn = 1; g.sBb = (int64_t)K * Q;
  g.C = out; g.sCm = Q; g.sCn = 1; g.sCb = (int64_t)K * Q;
  gemm64(g, h->stream);
  h->launches += 1;
  return ESMP2_OK;
}

// out[m][n] = sum_k in[m][k] M[k][n], n < N <= 32, for M rows of length Nv: the first N columns of the
// Nv x Nv matrix Mat.  in is read twice, for the power-of-two scale of each row and for the product.
esmp2_status rows_times_narrow(esmp2_handle *h, const double *in, double *out, int64_t M, int N, const double *Mat) {
  const int Nv = h->d.Nv, Nvp = (Nv + 7) & ~7, bn = N <= 16 ? 16 : 32;
  if (esmp2_status s = ensure_dflag(h)) return s;
  // the factor's digit planes, its exponent, the rows' exponents
  const size_t dig_bytes = sizeof(__nv_bfloat16) * (size_t)nr::P * bn * Nvp;   // a multiple of 256
  uint8_t *ws = nullptr;
  cudaError_t e = dmalloc(reinterpret_cast<void **>(&ws), dig_bytes + sizeof(int) * (size_t)(M + 4), h->stream);
  if (e != cudaSuccess) return check_cuda(h, e, "row exponents");
  int *eR = reinterpret_cast<int *>(ws + dig_bytes), *es = eR + 4;
  nr::k_factor_digits<<<1, 1024, 0, h->stream>>>(Mat, Nv, Nv, N, Nvp, bn, reinterpret_cast<__nv_bfloat16 *>(ws), eR);
  nr::k_row_exp<<<(unsigned)cdiv(M, 8), 256, 0, h->stream>>>(in, M, Nv, es);
  h->launches += 2;
  CUtensorMap mB;
  const uint64_t dims[3] = {(uint64_t)Nvp, (uint64_t)bn, (uint64_t)nr::P};
  const uint64_t str[2] = {(uint64_t)Nvp * 2, (uint64_t)Nvp * bn * 2};
  const uint32_t box[3] = {nr::BK, (uint32_t)bn, 1};
  if (!tma_map_bf16(&mB, ws, 3, dims, str, box, 64)) {
    dfree(ws, h->stream);
    h->err = "tensor map encoding failed";
    return ESMP2_ERR_CUDA;
  }
  nr::Args g{};
  g.in = in; g.out = out;
  g.rows = M;
  g.N = N; g.Q = 1;
  g.es = es;
  g.eR = eR;
  g.ld = Nv;
  g.vec = (Nv % 2) == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0;
  const int parts = (Nv + nr::K_MAX - 1) / nr::K_MAX;
  const int kper = ((Nv + parts - 1) / parts + nr::BK - 1) / nr::BK * nr::BK;   // <= K_MAX, a multiple of BK
  static_assert(nr::K_MAX % nr::BK == 0, "a K range ends on a chunk");
  esmp2_status s = ESMP2_OK;
  for (int k0 = 0; k0 < Nv && !s; k0 += kper) {
    g.k0 = k0;
    g.K = std::min(kper, Nv - k0);
    g.add = k0 > 0;
    s = bn == 16 ? nr::launch<true, 16>(h, mB, g) : nr::launch<true, 32>(h, mB, g);
  }
  dfree(ws, h->stream);
  return s;
}

}  // namespace esmp2
