// Float64-accurate products with F_vv (and the orbital rotations) from exact bf16 digit products
// on the 5th-generation tensor cores: the N_o^2 N_v^3 terms of Table 1 to float64 accuracy, with
// GB300's float64 pipe (two multiply-adds per clock and SM) out of the inner loop.
//
// Digits (Ozaki-type splitting): with 2^e the smallest power of two above 2 max |x_s|, z = x / 2^e
// lies in (-1/2, 1/2); Z = round(z 64^P) is an integer of magnitude <= 2^(6P-1) and the balanced
// base-64 digits of |Z|, Z = +-sum_{p=1..P} d_p 64^(P-p), d_p in [-32, 31] (d_1 in [0, 32]), give z
// to within 64^-P / 2.  Every digit is exact in bf16, every product of two an integer of magnitude
// <= 2^10.  Level L = p + q collects the digit pairs of one weight in one fp32 accumulator: a sum
// over K = Nv of at most L - 1 pairs stays below 2^24 whenever Nv (L - 1) 2^10 < 2^24, so the
// tensor cores add exactly.  The levels 2 .. Lmax are joined as integers and rounded to float64
// once.
//
// The rows of all slices are stacked: one GEMM with M = rows, N = K = Nv per operand
// (transposed copies of the slices that need F x as well, (x^T F)^T = F x).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "digit_split.h"
#include "internal.h"
#include "tc_ptx.h"

namespace esmp2 {
namespace dg {

using namespace ptx;

constexpr int BM = 128;                  // rows of a tile (TMEM lanes)
constexpr int BK = 64;                   // K elements of a chunk (128 bytes of bf16, the swizzle span)
constexpr int A_BYTES = BM * 128;        // one x digit plane of a chunk
constexpr int SMEM_MAX = 232448 - 2048;  // dynamic shared memory of a CTA (room for the barriers)
constexpr int NTHREADS = 320;            // producer warp, MMA warp, 8 epilogue warps
constexpr int kMaxLevels = 10;

// A tile keeps the accumulators of ALL its levels in TMEM at once (NLEV x BN <= 512 columns) and
// walks K once: a K chunk brings every digit plane of 128 rows of x and of BN columns of F a
// single time, and digit p of x meets the digits 1 .. Lmax - p of F, stacked along N, in one to
// three MMAs (their levels p + 1 .. Lmax are neighbouring accumulators).  Against one pass over K
// per digit pair and a float64 read-modify-write of the tile per level this moves 2.2 times fewer
// operand bytes through L2, reads no output, and takes the float64 conversion per element and
// level (the float64 pipe, not the tensor cores, had been the limit: 2 x 7 of its operations per
// element at eight levels) out of the kernel.  The eight contractions of a No=30 Nv=400 step: 147 ms
// before, 47 ms now (tensor pipe 18 -> 62 %); 58 ms with K chunks of 32 (64-byte rows: the copy
// engine's row rate), 118 ms when the two issuing threads divided a 64-bit counter by the ring
// length at every step.  A float64 sigma (FP64_TC) at No=20 Nv=200: 5.3 -> 0.9 ms of contraction.
template <int NLEV> struct Geo;          // BN: columns of a tile, a multiple of 16
template <> struct Geo<9> { static constexpr int BN = 48; };
template <> struct Geo<8> { static constexpr int BN = 64; };
template <> struct Geo<7> { static constexpr int BN = 64; };
template <> struct Geo<6> { static constexpr int BN = 80; };
template <> struct Geo<5> { static constexpr int BN = 96; };
template <> struct Geo<4> { static constexpr int BN = 96; };

// two buffers of F digit planes, the rest of shared memory a ring of x digit planes (6 or 7)
template <int NLEV> constexpr int fbuf_bytes() { return NLEV * Geo<NLEV>::BN * 128; }
template <int NLEV> constexpr int slots() { return (SMEM_MAX - 1024 - 2 * fbuf_bytes<NLEV>()) / A_BYTES; }

struct Args {
  int64_t R;          // stacked rows, r = job * Nv + a
  int64_t tiles;      // m_tiles * n_tiles
  int Nv, n_tiles, nk;
  const int *jobs;    // slice * 2 + transposed, or nullptr: job k is slice k, not transposed
  const int *es;      // binary exponent of the digits of each slice
  int eF;             // that of the right operand
  int per_block;      // slices per amplitude block (No^2)
  int vec2;           // rows of y and P start on 16-byte boundaries
  int one[5];         // per block: 1 = the plain job's product goes to P, 0 = to y
  double *y, *P;      // [slice][Nv][Nv]; a transposed job stores its product transposed into P
  int *err;
};

template <int NLEV, bool SMALL>   // SMALL: every level sum is below 2^22
__global__ void __launch_bounds__(NTHREADS, 1)
    k_levels(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tF,
             const __grid_constant__ Args g) {
  constexpr int BN = Geo<NLEV>::BN, PF = BN * 128 /* bytes of one F plane of a chunk */, FBUF = NLEV * PF;
  constexpr int SLOTS = slots<NLEV>();
  constexpr int PPM = 256 / BN;          // F planes one MMA spans (N <= 256)
  extern __shared__ uint8_t smem_raw[];
  uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *fbuf = ring + SLOTS * A_BYTES;   // two buffers of NLEV F planes
  __shared__ uint64_t full[SLOTS], empty[SLOTS], fempty[2], acc_full, acc_empty;
  __shared__ uint32_t tmem_base;
  __shared__ int fail;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < SLOTS; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int s = 0; s < 2; ++s) mbar_init(&fempty[s], 1);
    mbar_init(&acc_full, 1);
    mbar_init(&acc_empty, 8);
    fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = tmem_base;

  if (warp == 0) {
    if (lane == 0) {  // ------------------------------------------------ TMA producer
      // ring positions as running 32-bit counters: one thread issues every copy (and another one
      // every MMA), so the instructions between two issues are on the kernel's critical path
      int st = 0, fb = 0;
      uint32_t ph = 1, fph = 1, laps = 0;   // parities of the next wait on an empty slot / F buffer
      bool ok = true;
      for (int64_t t = blockIdx.x; t < g.tiles && ok; t += gridDim.x) {
        const int a0 = (int)(t / g.n_tiles) * BM, b0 = (int)(t % g.n_tiles) * BN;
        for (int kc = 0; kc < g.nk && ok; ++kc) {
          if (!mbar_wait(&fempty[fb], fph)) { ok = false; break; }
          uint8_t *F = fbuf + fb * FBUF;
          // step i = 1 .. NLEV brings x digit NLEV + 1 - i and F digit i: the MMAs of step i need
          // the F digits 1 .. i, all of which have then arrived
#pragma unroll
          for (int i = 1; i <= NLEV; ++i) {
            if (!mbar_wait(&empty[st], ph)) { ok = false; break; }
            mbar_expect_tx(&full[st], (uint32_t)(A_BYTES + PF));
            tma_3d(ring + st * A_BYTES, &tA, &full[st], kc * BK, a0, NLEV - i);
            tma_3d(F + (i - 1) * PF, &tF, &full[st], kc * BK, b0, i - 1);
            if (++st == SLOTS) { st = 0; ph ^= 1; laps = 1; }
          }
          fb ^= 1;
          fph ^= (uint32_t)(fb == 0);
        }
      }
      if (!ok) atomicExch(&fail, 1);
      // wait (bounded) until no copy of this CTA is still in flight: slots before st belong to the
      // current lap (parity ph ^ 1 of their full barrier), the others to the one before
      for (int j = 0; j < SLOTS; ++j)
        if (j < st) mbar_wait(&full[j], ph ^ 1, 100000000ull);
        else if (laps) mbar_wait(&full[j], ph, 100000000ull);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ------------------------------------------------ MMA issuer
      int st = 0, fb = 0;
      uint32_t ph = 0, aph = 1;
      bool ok = true;
      // descriptors: the constant part and the start address in units of 16 bytes
      const uint64_t dring = sdesc128(smem_u32(ring)), dfb = sdesc128(smem_u32(fbuf));
      for (int64_t t = blockIdx.x; t < g.tiles && ok; t += gridDim.x) {
        if (!mbar_wait(&acc_empty, aph)) { ok = false; break; }
        aph ^= 1;
        tc_after();
        for (int kc = 0; kc < g.nk && ok; ++kc) {
          const int ks = min(BK / 16, (g.Nv - kc * BK + 15) / 16);   // K steps of 16 in this chunk
          const uint64_t F = dfb + (uint64_t)(fb * (FBUF / 16));
#pragma unroll
          for (int i = 1; i <= NLEV; ++i) {
            if (!mbar_wait(&full[st], ph)) { ok = false; break; }
            const uint64_t A = dring + (uint64_t)(st * (A_BYTES / 16));
            const uint32_t d0 = tmem + (uint32_t)((NLEV - i) * BN);
            // F digits 1 .. i go to the accumulators of the levels p + 1 .. Lmax (p = NLEV + 1 - i);
            // the first of them is met here for the first time
            if (kc == 0) {
              umma_bf16(d0, A, F, idesc_bf16(BM, BN), 0u);
#pragma unroll
              for (int q = 1; q < i; q += PPM)
                umma_bf16(d0 + (uint32_t)(q * BN), A, F + (uint64_t)(q * PF / 16), idesc_bf16(BM, (i - q < PPM ? i - q : PPM) * BN), 1u);
            } else {
#pragma unroll
              for (int q = 0; q < i; q += PPM)
                umma_bf16(d0 + (uint32_t)(q * BN), A, F + (uint64_t)(q * PF / 16), idesc_bf16(BM, (i - q < PPM ? i - q : PPM) * BN), 1u);
            }
            for (int k = 1; k < ks; ++k) {
#pragma unroll
              for (int q = 0; q < i; q += PPM)
                umma_bf16(d0 + (uint32_t)(q * BN), A + 2 * k, F + (uint64_t)(q * PF / 16 + 2 * k), idesc_bf16(BM, (i - q < PPM ? i - q : PPM) * BN), 1u);
            }
            umma_commit(&empty[st]);
            if (++st == SLOTS) { st = 0; ph ^= 1; }
          }
          if (ok) umma_commit(&fempty[fb]);
          fb ^= 1;
        }
        if (!ok) break;
        umma_commit(&acc_full);
      }
      if (!ok) atomicExch(&fail, 1);
    }
  } else {  // ---------------------------------------------------------- epilogue
    // warp w reads TMEM lanes 32 (w % 4) .. +31; the two warps of a quarter split the columns
    constexpr int HC = BN / 2;
    const int quarter = warp & 3, chalf = (warp - 2) >> 2;
    uint32_t lt = 0;
    for (int64_t t = blockIdx.x; t < g.tiles; t += gridDim.x, ++lt) {
      if (!mbar_wait(&acc_full, lt & 1)) { if (lane == 0) atomicExch(&fail, 1); break; }
      tc_after();
      const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(chalf * HC);
      // levels 2 .. joined in int64 (bounded by Nv 2^10 64^(levels - 1) < 2^63 for eight levels and
      // the supported Nv; the ninth is rounded in at the weight of the eighth, 64^-9)
      long long V[HC];
#pragma unroll
      for (int c8 = 0; c8 < HC / 8; ++c8) {
        uint32_t r[NLEV][8];
#pragma unroll
        for (int l = 0; l < NLEV; ++l) tmem_ld8(taddr + (uint32_t)(l * BN + c8 * 8), r[l]);
        tmem_wait();
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          constexpr int NI = NLEV < 8 ? NLEV : 8;
          float f[NI];
#pragma unroll
          for (int l = 0; l < NLEV; ++l) keep(r[l][c]);
#pragma unroll
          for (int l = 0; l < NI; ++l) f[l] = __uint_as_float(r[l][c]);
          long long v = join_levels<NI, SMALL>(f);
          if constexpr (NLEV > 8) v += round64(__float2int_rn(__uint_as_float(r[8][c])));
          V[c8 * 8 + c] = no_value(f[0]) ? kNoValue : v;
        }
      }
      tc_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty);   // the next tile's MMAs run during the stores
      const int64_t r = (t / g.n_tiles) * BM + quarter * 32 + lane;
      if (r < g.R) {
        const int b0 = (int)(t % g.n_tiles) * BN + chalf * HC;
        const int job = (int)(r / g.Nv), a = (int)(r - (int64_t)job * g.Nv);
        const int jc = g.jobs ? g.jobs[job] : 2 * job, s = jc >> 1;
        const int e = g.es[s] + g.eF - 6 * (NLEV < 8 ? NLEV + 1 : 9);
        const int64_t off = (int64_t)s * g.Nv * g.Nv;
        if (jc & 1) {   // F x_s from the transposed copy: consecutive lanes are consecutive columns
          double *dst = g.P + off + a;
#pragma unroll
          for (int c = 0; c < HC; ++c)
            if (b0 + c < g.Nv) dst[(int64_t)(b0 + c) * g.Nv] = scale_or_nan(V[c], e);
        } else {
          double *dst = (g.one[s / g.per_block] ? g.P : g.y) + off + (int64_t)a * g.Nv + b0;
          if (g.vec2) {
#pragma unroll
            for (int c = 0; c < HC; c += 2)
              if (b0 + c < g.Nv)
                *reinterpret_cast<double2 *>(dst + c) = make_double2(scale_or_nan(V[c], e), scale_or_nan(V[c + 1], e));
          } else {
#pragma unroll
            for (int c = 0; c < HC; ++c)
              if (b0 + c < g.Nv) dst[c] = scale_or_nan(V[c], e);
          }
        }
      }
      __syncwarp();
    }
  }
  tc_before();
  __syncthreads();
  if (warp == 1) {
    tc_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
  if (threadIdx.x == 0 && fail) atomicOr(g.err, 1);
}

// ---------------------------------------------------------------------------- digit splits
// Exponent of one Nv x Nv matrix, element (r, c) at r ld + c cs (one CTA); infinities and NaN do not take part.
__global__ void k_mat_exp(const double *x, int n, int64_t ld, int64_t cs, int *es) {
  __shared__ double red[32];
  double m = 0.0;
  for (int64_t e = threadIdx.x; e < (int64_t)n * n; e += blockDim.x) {
    const double v = x[(e / n) * ld + (e % n) * cs];
    if (!non_finite(v)) m = fmax(m, fabs(v));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) {
      int e = 0;
      if (m > 0.0) frexp(m, &e);   // m = f 2^e with f in [0.5, 1): 2 max |x| < 2^(e+1)
      *es = m > 0.0 ? e + 1 : 0;
    }
  }
}
// its P digit planes, out[p][r][c] with row pitch Nvp, pad columns zero; NaN digits for an infinity or NaN
__global__ void k_mat_digits(const double *x, int n, int Nvp, int64_t ld, int64_t cs, const int *es, int P,
                             __nv_bfloat16 *out) {
  const int64_t plane = (int64_t)n * Nvp;
  const double scale = ldexp(1.0, 6 * P - *es);
  for (int r = blockIdx.x; r < n; r += gridDim.x) {
    for (int c = threadIdx.x; c < Nvp; c += blockDim.x) {
      const double v = c < n ? x[r * ld + c * cs] : 0.0;
      __nv_bfloat16 *dst = out + (int64_t)r * Nvp + c;
      if (non_finite(v)) {
        for (int p = 0; p < P; ++p) dst[p * plane] = __ushort_as_bfloat16(0x7FFF);
        continue;
      }
      long long Z = __double2ll_rn(v * scale);
      for (int p = P - 1; p > 0; --p) {   // least significant digit first
        const long long d = ((Z + 32) & 63) - 32;
        Z = (Z - d) >> 6;                 // exact: Z - d is a multiple of 64
        dst[p * plane] = __int2bfloat16_rn((int)d);
      }
      dst[0] = __int2bfloat16_rn((int)Z);  // leading digit, |Z| <= 32
    }
  }
}

// Exponent of each slice (one CTA per slice): the largest exponent field decides, so the maximum
// runs on the high words as integers (a float64 comparison per element would be bound by the
// float64 pipe); infinities and NaN do not take part.
__global__ void __launch_bounds__(256) k_slice_exp(const double *x, int n /* Nv^2 */, int *es, const int *list) {
  __shared__ int red[8];
  const int s = list ? list[blockIdx.x] : (int)blockIdx.x;
  const int2 *X = reinterpret_cast<const int2 *>(x + (int64_t)s * n);
  int m = 0;
#pragma unroll 8
  for (int e = threadIdx.x; e < n; e += 256) {
    const int h = X[e].y & 0x7FFFFFFF;
    m = max(m, h < 0x7FF00000 ? h : 0);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) m = max(m, red[w]);
    es[s] = m >> 20 ? (m >> 20) - 1021 : 0;   // max |x| < 2^(field - 1022), and one more bit
  }
}

// Digit planes of the stacked rows, out[p][job Nv + a][c] (row pitch Nvp, pad columns zero): plain
// jobs row by row, a warp per row and two columns per lane (one 128-byte line per plane and warp).
template <int P>
__global__ void __launch_bounds__(256) k_digits(const double *x, int Nv, int Nvp, const int *es, const int *jobs,
                                                int njobs, int64_t plane, __nv_bfloat16 *out, int vec) {
  const int lane = threadIdx.x & 31;
  const int64_t rows = (int64_t)njobs * Nv;
  for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; r < rows;
       r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int job = (int)(r / Nv), a = (int)(r - (int64_t)job * Nv);
    const int jc = jobs ? jobs[job] : 2 * job;
    if (jc & 1) continue;   // k_digits_t
    const int s = jc >> 1, e = es[s];
    const double *src = x + ((int64_t)s * Nv + a) * Nv;
    __nv_bfloat16 *dst = out + r * Nvp;
    for (int c = 2 * lane; c < Nvp; c += 64) {
      double2 v = make_double2(0.0, 0.0);
      if (vec) {
        if (c < Nv) v = *reinterpret_cast<const double2 *>(src + c);
      } else {
        if (c < Nv) v.x = src[c];
        if (c + 1 < Nv) v.y = src[c + 1];
      }
      const long long U0 = digit_word<P>(v.x, e), U1 = digit_word<P>(v.y, e);
      const uint32_t sg = sign_pair_nan(v.x, v.y), rg = range_pair(v.x, v.y);
#pragma unroll
      for (int p = 1; p <= P; ++p)
        *reinterpret_cast<uint32_t *>(dst + (p - 1) * plane + c) = digit_pair<P>(U0, U1, sg, rg, p);
    }
  }
}
// the transposed jobs (the last ones of the list, from job first on): rows are the columns of the
// slice, 32 of them by 64 through shared memory
template <int P>
__global__ void __launch_bounds__(256) k_digits_t(const double *x, int Nv, int Nvp, const int *es, const int *jobs,
                                                  int first, int njobs, int64_t plane, __nv_bfloat16 *out) {
  __shared__ double t[64][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nr = (Nv + 31) / 32, nc = (Nvp + 63) / 64;
  const int64_t items = (int64_t)(njobs - first) * nr * nc;
  for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const int job = first + (int)(it / (nr * nc)), tt = (int)(it % (nr * nc)), a0 = (tt / nc) * 32, c0 = (tt % nc) * 64;
    const int s = jobs[job] >> 1, e = es[s];
    const double *src = x + (int64_t)s * Nv * Nv;
    __syncthreads();
    for (int q = w; q < 64; q += 8)
      t[q][lane] = (c0 + q < Nv && a0 + lane < Nv) ? src[(int64_t)(c0 + q) * Nv + a0 + lane] : 0.0;
    __syncthreads();
    const int c = 2 * lane;
    if (c0 + c >= Nvp) continue;
    for (int q = w; q < 32 && a0 + q < Nv; q += 8) {
      const long long U0 = digit_word<P>(t[c][q], e), U1 = digit_word<P>(t[c + 1][q], e);
      const uint32_t sg = sign_pair_nan(t[c][q], t[c + 1][q]), rg = range_pair(t[c][q], t[c + 1][q]);
      __nv_bfloat16 *dst = out + ((int64_t)job * Nv + a0 + q) * Nvp + c0 + c;
#pragma unroll
      for (int p = 1; p <= P; ++p)
        *reinterpret_cast<uint32_t *>(dst + (p - 1) * plane) = digit_pair<P>(U0, U1, sg, rg, p);
    }
  }
}

// Job lists (slice * 2 + transposed): T, X, Y slices with i < j (every slice when sym = 0), S, Z, then
// the transposed copies of the slices that take both terms (sym = 0 all, 1 S and Z, 2 Z).  slices:
// the plain slices alone.
__global__ void k_job_list(int No, int sym, int *jobs, int *slices) {
  const int NN = No * No, half = No * (No - 1) / 2, h1 = sym ? half : NN;
  const int plain = 3 * h1 + 2 * NN, extra = sym == 0 ? 5 * NN : sym == 1 ? 2 * NN : NN;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < plain + extra; e += gridDim.x * blockDim.x) {
    int s;
    if (e >= plain) {
      const int f = e - plain;
      s = sym == 0 ? f : sym == 1 ? (f < NN ? NN + f : 3 * NN + f) : 4 * NN + f;
      jobs[e] = 2 * s + 1;
      continue;
    }
    if (e < 3 * h1) {
      const int blk = e / h1 == 0 ? 0 : (e / h1 == 1 ? 2 : 3);
      int k = e % h1;
      if (sym) {
        int i = 0;
        while (k >= No - 1 - i) { k -= No - 1 - i; ++i; }
        k = i * No + i + 1 + k;
      }
      s = blk * NN + k;
    } else {
      const int f = e - 3 * h1;
      s = (f < NN ? 1 : 4) * NN + f % NN;
    }
    jobs[e] = 2 * s;
    if (slices) slices[e] = s;
  }
}

// y += P on the slices that took both terms
__global__ void __launch_bounds__(256) k_add64(const double *P, double *y, int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) y[e] += P[e];
}

}  // namespace dg

namespace {

// 3-D tensor map {Nvp, rows, planes} of bf16, box 64 x box_rows x 1, 128-byte swizzle
bool digit_map(CUtensorMap *m, const void *base, int Nvp, int64_t rows, int64_t plane_elems, int planes, int box_rows) {
  const uint64_t dims[3] = {(uint64_t)Nvp, (uint64_t)rows, (uint64_t)planes};
  const uint64_t str[2] = {(uint64_t)Nvp * 2, (uint64_t)plane_elems * 2};
  const uint32_t box[3] = {dg::BK, (uint32_t)box_rows, 1};
  return tma_map_bf16(m, base, 3, dims, str, box, 128);
}

template <int NLEV>
const char *launch_levels(cudaStream_t st, const void *xd, int64_t xplane, const void *Fd, int Fplanes, dg::Args g) {
  constexpr int BN = dg::Geo<NLEV>::BN;
  constexpr int smem = dg::slots<NLEV>() * dg::A_BYTES + 2 * dg::fbuf_bytes<NLEV>() + 1024;
  static_assert(smem <= dg::SMEM_MAX && dg::slots<NLEV>() >= 4, "shared memory of the digit-level kernel");
  const int Nv = g.Nv, Nvp = (Nv + 7) & ~7;
  CUtensorMap mA, mF;
  if (!digit_map(&mA, xd, Nvp, g.R, xplane, NLEV, dg::BM) || !digit_map(&mF, Fd, Nvp, Nv, (int64_t)Nv * Nvp, Fplanes, BN))
    return "tensor map encoding failed";
  const bool small = (int64_t)Nv * NLEV * 1024 < (1 << 22);
  const void *fn = small ? reinterpret_cast<const void *>(dg::k_levels<NLEV, true>) : reinterpret_cast<const void *>(dg::k_levels<NLEV, false>);
  if (smem_limit_once(fn, smem) != cudaSuccess)
    return "cannot raise the shared-memory limit of the digit-level kernel";
  g.n_tiles = (Nv + BN - 1) / BN;
  g.nk = (Nv + dg::BK - 1) / dg::BK;
  g.tiles = cdiv(g.R, dg::BM) * g.n_tiles;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const unsigned grid = (unsigned)std::min<int64_t>(g.tiles, sms);
  if (small) dg::k_levels<NLEV, true><<<grid, dg::NTHREADS, smem, st>>>(mA, mF, g);
  else dg::k_levels<NLEV, false><<<grid, dg::NTHREADS, smem, st>>>(mA, mF, g);
  return nullptr;
}

// digit planes of the jobs' rows, then every level of every tile; levels 5 .. 10
template <int NLEV>
const char *run_levels(esmp2_handle *h, const double *x, const int *jobs, int nplain, int njobs, const void *Fd, dg::Args g,
                       double alg, double exec) {
  const int Nv = g.Nv, Nvp = (Nv + 7) & ~7;
  const int64_t plane = (int64_t)njobs * Nv * Nvp;
  __nv_bfloat16 *xd = static_cast<__nv_bfloat16 *>(h->xdig);
  const int vec = (Nv % 2) == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0;
  dg::k_digits<NLEV><<<1216, 256, 0, h->stream>>>(x, Nv, Nvp, g.es, jobs, nplain, plane, xd, vec);
  if (njobs > nplain) {
    dg::k_digits_t<NLEV><<<1216, 256, 0, h->stream>>>(x, Nv, Nvp, g.es, jobs, nplain, njobs, plane, xd);
    h->launches += 1;
  }
  KScope ks(h->stream, ESMP2_KT_DIGITS, alg, exec);
  h->launches += 2;
  return launch_levels<NLEV>(h->stream, xd, plane, Fd, kDigitPlanes, g);
}

esmp2_status run_digits(esmp2_handle *h, const double *x, const int *jobs, int nplain, int njobs, const void *Fd, dg::Args g,
                        int levels, double alg, double per_pair) {
  const int Nvp = (g.Nv + 7) & ~7;
  levels = std::max(levels, 5);   // fewer levels than five would gain nothing
  const size_t plane = sizeof(__nv_bfloat16) * (size_t)g.Nv * Nvp;   // one digit plane of a slice
  const size_t one = plane * (levels - 1), need = one * njobs;
  if (need > h->xdig_bytes && !h->xdig_final) {   // stream-ordered: the old planes are released after their last use
    // The transforms of the set-up take what they need.  The first call on a whole block vector takes nine
    // planes of the job list of sym = 1 (of the longest, sym = 0, where that is small: a second pass would
    // cost No=1 Nv=40 a third of its 60 us), and that stays: a caller may have captured what works on it.
    // Calls that need more, or all of them where there was less room, work in passes.
    const int NN = h->d.No * h->d.No;
    h->xdig_final = jobs || njobs > NN;
    const size_t least = plane * kDigitPlanes, full = least * h->njobs[0];
    size_t room = !h->xdig_final ? need : full <= (size_t)256 << 20 ? full : least * h->njobs[1];
    dfree(h->xdig, h->stream);
    h->xdig = nullptr;
    h->xdig_bytes = 0;
    cudaError_t e = dmalloc(&h->xdig, room, h->stream);
    while (e != cudaSuccess && room > least) {
      cudaGetLastError();
      e = dmalloc(&h->xdig, room = std::max(least, room / 2), h->stream);
    }
    if (e != cudaSuccess) {
      h->xdig = nullptr;
      h->xdig_final = false;
      return check_cuda(h, e, "digit planes");
    }
    h->xdig_bytes = room;
  }
  const int per = (int)std::min<size_t>(njobs, h->xdig_bytes / one);   // jobs of one pass
  g.vec2 = (g.Nv % 2) == 0 && (reinterpret_cast<uintptr_t>(g.y) | reinterpret_cast<uintptr_t>(g.P)) % 16 == 0;
  const char *m = nullptr;
  double *const y0 = g.y;
  const int *const es0 = g.es;
  for (int j0 = 0; j0 < njobs && !m; j0 += per) {
    const int nj = std::min(per, njobs - j0), np = std::max(0, std::min(nj, nplain - j0));
    const double part = (double)nj / njobs, a = part * alg, e = part * 0.5 * levels * (levels - 1) * per_pair;
    const int *jl = jobs ? jobs + j0 : nullptr;
    g.R = (int64_t)nj * g.Nv;
    g.jobs = jl;
    const int64_t off = jobs ? 0 : (int64_t)j0 * g.Nv * g.Nv;   // without a list, job k of the pass is slice k
    const double *xp = x + off;
    g.y = y0 + off;
    g.es = es0 + (jobs ? 0 : j0);
    switch (levels) {
      case 5: m = run_levels<4>(h, xp, jl, np, nj, Fd, g, a, e); break;
      case 6: m = run_levels<5>(h, xp, jl, np, nj, Fd, g, a, e); break;
      case 7: m = run_levels<6>(h, xp, jl, np, nj, Fd, g, a, e); break;
      case 8: m = run_levels<7>(h, xp, jl, np, nj, Fd, g, a, e); break;
      case 9: m = run_levels<8>(h, xp, jl, np, nj, Fd, g, a, e); break;
      default: m = run_levels<9>(h, xp, jl, np, nj, Fd, g, a, e); break;
    }
  }
  if (m) { h->err = m; return ESMP2_ERR_CUDA; }
  return check_cuda(h, cudaGetLastError(), "digit levels");
}

}  // namespace

int split_levels_for(double tol) {
  // keep 2^{-6 (Lmax - 1)} at or below 1e-4 tol (refinement and energy stay float64-exact)
  const double need = std::log2(1e4 / std::max(tol, 1e-300)) / 6.0;
  return std::max(2, std::min(dg::kMaxLevels, (int)std::ceil(need) + 1));
}

bool split_supported(const esmp2_handle *h, int levels) {
  if (levels < 2 || levels > dg::kMaxLevels) return false;
  return 2LL * h->d.Nv * (levels - 1) * 1024 < (1LL << 24);
}

// device error flag of the bounded waits
esmp2_status ensure_dflag(esmp2_handle *h) {
  if (h->dflag) return ESMP2_OK;
  cudaError_t e = dmalloc(reinterpret_cast<void **>(&h->dflag), sizeof(int), h->stream);
  if (e != cudaSuccess) { h->dflag = nullptr; return check_cuda(h, e, "device flag"); }
  return check_cuda(h, cudaMemsetAsync(h->dflag, 0, sizeof(int), h->stream), "device flag");
}

// plain slices of the symmetric forms (T, X, Y with i < j, all of S and Z)
esmp2_status ensure_slist(esmp2_handle *h) {
  if (h->slist) return ESMP2_OK;
  const int No = h->d.No, NN = No * No, half = No * (No - 1) / 2, nl = 3 * half + 2 * NN;
  // slist, then the job lists of sym = 0, 1, 2
  const int nj[3] = {10 * NN, nl + 2 * NN, nl + NN};
  cudaError_t e = dmalloc(reinterpret_cast<void **>(&h->slist), sizeof(int) * (size_t)(nl + nj[0] + nj[1] + nj[2]), h->stream);
  if (e != cudaSuccess) { h->slist = nullptr; return check_cuda(h, e, "slice list"); }
  h->nslist = nl;
  int *p = h->slist + nl;
  for (int sym = 0; sym < 3; ++sym) {
    h->jobs[sym] = p;
    h->njobs[sym] = nj[sym];
    dg::k_job_list<<<(unsigned)cdiv(nj[sym], 256), 256, 0, h->stream>>>(No, sym, p, sym == 1 ? h->slist : nullptr);
    p += nj[sym];
  }
  h->launches += 3;
  return check_cuda(h, cudaGetLastError(), "slice list");
}

esmp2_status ensure_split(esmp2_handle *h) {
  if (h->Fdig) return ESMP2_OK;
  if (esmp2_status s0 = ensure_slist(h)) return s0;
  const int No = h->d.No, Nv = h->d.Nv, N = h->d.N, Nvp = (Nv + 7) & ~7;
  const int S = 5 * No * No;
  cudaError_t e = dmalloc(&h->Fdig, sizeof(__nv_bfloat16) * (size_t)kDigitPlanes * Nv * Nvp, h->stream);
  if (e == cudaSuccess) e = dmalloc(reinterpret_cast<void **>(&h->es), sizeof(int) * (size_t)(S + 4), h->stream);
  if (e != cudaSuccess) {
    dfree(h->Fdig, h->stream); dfree(h->es, h->stream);
    h->Fdig = nullptr; h->es = nullptr;
    return check_cuda(h, e, "split workspace");
  }
  if (esmp2_status s0 = ensure_dflag(h)) return s0;
  // digits of F_vv (the same block in the TOP and the semicanonical-occupied basis); the
  // leading digits do not depend on how many are kept
  const double *Fv = h->F + (int64_t)No * N + No;
  dg::k_mat_exp<<<1, 1024, 0, h->stream>>>(Fv, Nv, N, 1, h->es + S);
  dg::k_mat_digits<<<256, 256, 0, h->stream>>>(Fv, Nv, Nvp, N, 1, h->es + S, kDigitPlanes, static_cast<__nv_bfloat16 *>(h->Fdig));
  h->launches += 2;
  e = cudaMemcpyAsync(&h->eF, h->es + S, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  return check_cuda(h, e, "split setup");
}

// sym = 1: T, X, Y slices (exactly antisymmetric) take only x F on i < j into p64 and the
// caller forms y_ij = P_ij - P_ij^T; S and Z slices take x F + F x into y (F x by way of p64).
// sym = 2: as sym = 1, and the S slices (S_ij^ab = S_ji^ba exactly) also take only x F into
// p64: F x_ij = (x_ji F)^T, so the caller forms y_ij = P_ij + P_ji^T.
// sym = 0: every slice takes both terms into y (any input).
// p64: a full block vector (5 blocks).  join = false: F x stays in p64 (the caller adds it).
esmp2_status virt_split(esmp2_handle *h, const double *x, double *y, double *p64, int sym, int levels, bool join) {
  if (!split_supported(h, levels)) { h->err = "digit-split contraction not exact for this Nv"; return ESMP2_ERR_UNSUPPORTED; }
  esmp2_status s = ensure_split(h);
  if (s) return s;
  const int No = h->d.No, Nv = h->d.Nv, NN = No * No;
  const int nplain = sym ? h->nslist : 5 * NN, njobs = h->njobs[sym];
  dg::k_slice_exp<<<nplain, 256, 0, h->stream>>>(x, Nv * Nv, h->es, sym ? h->slist : nullptr);
  h->launches += 1;
  dg::Args g{};
  g.Nv = Nv;
  g.es = h->es;
  g.eF = h->eF;
  g.per_block = NN;
  for (int b = 0; b < 5; ++b) g.one[b] = sym && (b == BT || b == BX || b == BY || (sym == 2 && b == BS));
  g.y = y;
  g.P = p64;
  g.err = h->dflag;
  // the method's work is one contraction of the block vector, however many digit pairs
  // emulate it; the tensor cores execute every pair on the stored slices
  const double per_pair = 2.0 * njobs * (double)Nv * Nv * Nv;
  if ((s = run_digits(h, x, h->jobs[sym], nplain, njobs, h->Fdig, g, levels, sym ? alg_virtual_flops(No, Nv) : per_pair, per_pair)))
    return s;
  if (!join) return check_cuda(h, cudaGetLastError(), "virt_split");
  const int64_t B = h->d.B;
  if (sym == 0) dg::k_add64<<<2432, 256, 0, h->stream>>>(p64, y, 5 * B);
  else {
    if (sym == 1) { dg::k_add64<<<2432, 256, 0, h->stream>>>(p64 + BS * B, y + BS * B, B); h->launches += 1; }
    dg::k_add64<<<2432, 256, 0, h->stream>>>(p64 + BZ * B, y + BZ * B, B);
  }
  h->launches += 1;
  return check_cuda(h, cudaGetLastError(), "virt_split");
}

// the digit planes of M^T (Nv x Nv), built on first use
static esmp2_status ensure_matrix_digits(esmp2_handle *h, const double *M, void **dig, int *eM, int eslot) {
  const int No = h->d.No, Nv = h->d.Nv, Nvp = (Nv + 7) & ~7;
  if (!*dig) {
    cudaError_t e = dmalloc(dig, sizeof(__nv_bfloat16) * (size_t)kDigitPlanes * Nv * Nvp, h->stream);
    if (e != cudaSuccess) return check_cuda(h, e, "rotation digits");
    int *ed = h->es + 5 * No * No + eslot;
    dg::k_mat_exp<<<1, 1024, 0, h->stream>>>(M, Nv, 1, Nv, ed);
    dg::k_mat_digits<<<256, 256, 0, h->stream>>>(M, Nv, Nvp, 1, Nv, ed, kDigitPlanes, static_cast<__nv_bfloat16 *>(*dig));
    e = cudaMemcpyAsync(eM, ed, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    h->launches += 2;
    if (e != cudaSuccess) return check_cuda(h, e, "rotation digits");
  }
  return ESMP2_OK;
}

// Y = X M (rows x Nv times an Nv x Nv matrix M, rows a multiple of Nv) in float64 accuracy from
// exact digit products on the tensor cores (ten levels): the right-factor form of the orbital
// rotations (M = W_v for the integral transforms, the virtual rotation of the reduced-cost
// basis).  X is read as rows/Nv slices of Nv x Nv.  The digit planes of M^T (row b' holds column
// b' of M, the K-major right operand) are built on first use into *dig with the power-of-two
// scale in es[eslot] (device) and *eM (host).
esmp2_status xwm_split(esmp2_handle *h, const double *X, int64_t rows, double *Y, const double *M, void **dig,
                       int *eM, int eslot) {
  esmp2_status s = ensure_split(h);
  if (s) return s;
  const int No = h->d.No, Nv = h->d.Nv;
  const int S = (int)(rows / Nv), levels = dg::kMaxLevels;
  if (rows % Nv != 0 || S > 5 * No * No || (int64_t)(levels - 1) * Nv * 1024 >= (1LL << 24)) {
    h->err = "xwm_split: unsupported shape";
    return ESMP2_ERR_UNSUPPORTED;
  }
  if ((s = ensure_matrix_digits(h, M, dig, eM, eslot))) return s;
  dg::k_slice_exp<<<S, 256, 0, h->stream>>>(X, Nv * Nv, h->es, nullptr);
  h->launches += 1;
  dg::Args g{};
  g.Nv = Nv;
  g.es = h->es;
  g.eF = *eM;
  g.per_block = S;
  g.y = Y;
  g.err = h->dflag;
  const double fl = 2.0 * (double)rows * Nv * Nv;   // one float64-accurate rotation
  return run_digits(h, X, nullptr, S, S, *dig, g, levels, fl, fl);
}

esmp2_status xwv_split(esmp2_handle *h, const double *X, int64_t rows, double *Y) {
  return xwm_split(h, X, rows, Y, h->Wv, &h->Rdig, &h->eR, 1);
}

}  // namespace esmp2
