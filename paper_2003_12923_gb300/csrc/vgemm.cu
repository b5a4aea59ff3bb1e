// Virtual-index contraction of the inner sigma as one dense GEMM on the 5th-generation tensor
// cores (the N_o^2 N_v^3 terms of Table 1, Eq. qfq_replacement): bf16 operands (kind::f16) or
// float32 operands read as tf32 (kind::tf32), fp32 accumulation in TMEM.
//
// Every slice s of the packed inner vector is an Nv x Nv matrix X_s with rows a and columns
// c; the terms of a slice are X_s F and F X_s (F = F_vv, symmetric).  Stacking the rows of
// all slices gives one matrix A with rows r = (s, a), and
//     P = A F,   P[r][b] = sum_c A[r][c] F[c][b]
// is a plain GEMM with M = (#slices) Nv, N = K = Nv: no per-slice tile padding.  The second
// term of each slice is the transpose of a first term: F X_s = -(X_s F)^T for the
// antisymmetric T, X, Y slices, F S_ij = (S_ji F)^T for the spin-flip-symmetric S slices,
// and for Z the operand also holds the transposed slices Z_s^T, whose rows of P are stored
// transposed here, (Z_s^T F)^T = F Z_s.  The coupling pass forms y from P.
//
// Structure (persistent, 576 threads):
//   each CTA owns one column tile b0 .. b0 + Nt - 1 of the result (columns split over nN
//   tiles) and keeps that tile's panel W[b][c] (all K) resident in shared memory;
//   warp 0      TMA producer: 2-D tiled bulk copies of 128-row x 64-byte A chunks (32 bf16 or
//               16 float32 columns; 64-byte swizzle) into a ring of 5 to 8 slots (what the
//               panel leaves)
//   warp 1      one thread issues tcgen05.mma (M = 128, N = Nt, K = 16 bf16 or 8 tf32, 32 bytes
//               of each operand row per instruction), commits to mbarriers
//   warps 2..17 epilogue: tcgen05.ld 32x32b from one of two TMEM accumulators (2 x Nt
//               columns), fp32 stores of P rows (16-byte vectors) or of transposed rows (one
//               128-byte segment per column and warp).  Four warps share a TMEM lane quarter, each
//               with two eight-column loads in flight: with two warps per quarter, one load at a
//               time, 64-bit row divisions and the masks taken element by element the epilogue, not the
//               operands or the MMAs, set the pace (No=10 Nv=400: plain rotation 68 us, scaled one
//               245 us a launch; now 67 and 73 us)
// Every mbarrier wait is bounded (globaltimer); a wait that runs out raises the error flag,
// the CTA waits (bounded) for its own copies in flight and frees its TMEM.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.h"
#include "tc_ptx.h"

namespace esmp2 {
namespace vg {

using namespace ptx;

constexpr int BM = 128;                 // accumulator rows (TMEM lanes)
constexpr int CHUNK_B = 64;             // bytes of one operand row per K chunk (the swizzle span)
constexpr int MAX_STAGES = 8;
constexpr int A_STAGE = BM * CHUNK_B;   // 8 KB
// K elements per chunk and per MMA: bf16 32 and 16, tf32 16 and 8 (both 32 bytes per MMA).  Chunks of
// 128-byte rows leave room for five ring slots only with three column tiles instead of two at
// Nv = 400 and were slower (51 launches of the No=30 Nv=400 step: 41 against 35 ms).
template <bool TF32> struct Kind {
  static constexpr int BK = TF32 ? 16 : 32;
  static constexpr int KMMA = TF32 ? 8 : 16;
};
constexpr int EPI_WARPS = 16, NTHREADS = 64 + 32 * EPI_WARPS;
// dynamic shared memory per CTA: the 232448-byte opt-in limit less room for the kernel's
// static shared memory (barriers, TMEM address, flags, the epilogue's 10 KB staging tile and 1 KB table)
constexpr int SMEM_MAX = 232448 - 2048 - 11264;
// Instruction descriptor: D fp32 (bits 4-5 = 1); A and B format (bits 7-9, 10-12) bf16 = 1 of
// kind::f16 or tf32 = 2 of kind::tf32; both K-major; N >> 3 at bit 17, M >> 4 at bit 24.
template <bool TF32>
__device__ __forceinline__ uint32_t idesc(int M, int N) {
  const uint32_t fmt = TF32 ? 2u : 1u;
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
template <bool TF32>
__device__ __forceinline__ void umma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if constexpr (TF32)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(
            d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
  else
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
            d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

struct Args {
  int64_t rows;         // rows of A and of the result, r = (slice, a)
  int64_t rows_normal;  // rows [0, rows_normal) go to P[r][b]; later rows to PT (transposed)
  int Nv;               // rows per slice (transposed part) and columns of the result
  int nk;               // K chunks (nk * BK >= Nv)
  int nN;               // column tiles; CTA c works on tile c % nN
  int Nt;               // columns of a column tile (multiple of 16, <= 256)
  int stages;           // ring slots (<= MAX_STAGES)
  int64_t m_tiles;      // ceil(rows / BM)
  float *P;             // [rows_normal][ldp]
  float *PT;            // [(rows - rows_normal) / Nv][Nv][ldp]: PT[s][b][c] = result row (s, c), column b
  int ldp;              // row pitch of P and PT (elements, a multiple of 4)
  int *err;             // device error flag
  // transposed rows stored as bf16 into PT16 instead of PT, optionally scaled element-wise
  // by the inverse diagonal of the reduced-cost basis (the preconditioner's middle factor):
  // element (slice s, a, b) of the stored slice times valid ? 1 / ((lam[a] + lam[b]) - occ[s]) : 0
  __nv_bfloat16 *PT16;
  const float *lam;     // [Nv] or nullptr (no scaling)
  const float *occ;     // [slices]
  const int *code;      // [slices]: block | 8 (i == 0) | 16 (j == 0)
};

template <bool TF32>
__global__ void __launch_bounds__(NTHREADS, 1)
    k_vgemm(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tF, Args g) {
  constexpr int BK = Kind<TF32>::BK, KMMA = Kind<TF32>::KMMA;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int STAGES = g.stages;
  uint8_t *ring = smem;                                  // STAGES x A_STAGE
  uint8_t *panel = smem + STAGES * A_STAGE;              // nk chunks of Nt rows x 64 bytes
  __shared__ uint64_t full[MAX_STAGES], empty[MAX_STAGES], acc_full[2], acc_empty[2], pbar;
  __shared__ uint32_t tmem_base;
  __shared__ int fail;
  // bf16 transposed output: per epilogue warp one 8-column x 32-row chunk, turned so that each
  // lane stores 8 consecutive rows of one column as a 16-byte vector
  __shared__ __align__(16) __nv_bfloat16 stg[EPI_WARPS][8][40];
  __shared__ __align__(16) float slam[256];   // lam of the CTA's column tile
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nt = blockIdx.x % g.nN, group = gridDim.x / g.nN, gi = blockIdx.x / g.nN;
  const int b0 = nt * g.Nt, nvalid = min(g.Nt, g.Nv - b0), nmma = (nvalid + 15) & ~15;
  const uint32_t chunk_bytes = (uint32_t)g.Nt * CHUNK_B;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&acc_full[s], 1); mbar_init(&acc_empty[s], EPI_WARPS); }
    mbar_init(&pbar, 1);
    fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (g.lam)
    for (int k = threadIdx.x; k < nvalid; k += NTHREADS) slam[k] = g.lam[b0 + k];
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
      bool ok = true;
      // the column tile's F panel, once
      mbar_expect_tx(&pbar, chunk_bytes * (uint32_t)g.nk);
      for (int kc = 0; kc < g.nk; ++kc) tma_2d(panel + kc * chunk_bytes, &tF, &pbar, kc * BK, b0);
      // ring positions as running counters: this thread and the MMA issuer are serial chains, and a
      // 64-bit division per chunk by the (runtime) ring length was the longest link in both
      int st = 0;
      uint32_t ph = 1, laps = 0;   // parity of the next wait on an empty slot
      for (int64_t m = gi; m < g.m_tiles && ok; m += group) {
        for (int kc = 0; kc < g.nk; ++kc) {
          if (!mbar_wait(&empty[st], ph)) { ok = false; break; }
          mbar_expect_tx(&full[st], (uint32_t)A_STAGE);
          tma_2d(ring + st * A_STAGE, &tA, &full[st], kc * BK, (int)(m * BM));
          if (++st == STAGES) { st = 0; ph ^= 1; laps = 1; }
        }
      }
      if (!ok) atomicExch(&fail, 1);
      // wait (bounded) until no copy of this CTA is still in flight: slots before st belong to the
      // current lap (parity ph ^ 1 of their full barrier), the others to the one before
      mbar_wait(&pbar, 0, 100000000ull);
      for (int j = 0; j < STAGES; ++j)
        if (j < st) mbar_wait(&full[j], ph ^ 1, 100000000ull);
        else if (laps) mbar_wait(&full[j], ph, 100000000ull);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ------------------------------------------------ MMA issuer
      bool ok = mbar_wait(&pbar, 0);
      tc_after();
      const uint32_t id = idesc<TF32>(BM, nmma);
      const uint64_t pan = sdesc64(smem_u32(panel)), rg = sdesc64(smem_u32(ring));
      int st = 0, lt = 0;
      uint32_t ph = 0;
      for (int64_t m = gi; m < g.m_tiles && ok; m += group, ++lt) {
        const int ab = lt & 1;
        const uint32_t ar = (uint32_t)(lt >> 1);
        if (!mbar_wait(&acc_empty[ab], (ar & 1) ^ 1)) { ok = false; break; }
        tc_after();
        const uint32_t d = tmem + (uint32_t)(ab * 256);
        for (int kc = 0; kc < g.nk; ++kc) {
          if (!mbar_wait(&full[st], ph)) { ok = false; break; }
          const uint64_t a = rg + (uint64_t)(st * (A_STAGE / 16)), b = pan + (uint64_t)(kc * (chunk_bytes / 16));
          umma<TF32>(d, a, b, id, kc > 0 ? 1u : 0u);
          if (g.Nv - kc * BK > KMMA) umma<TF32>(d, a + 2, b + 2, id, 1u);   // skip the K step past Nv
          umma_commit(&empty[st]);
          if (++st == STAGES) { st = 0; ph ^= 1; }
        }
        if (!ok) break;
        umma_commit(&acc_full[ab]);
      }
      if (!ok) atomicExch(&fail, 1);
    }
  } else {  // ---------------------------------------------------------- epilogue
    const int quarter = warp & 3, part = (warp - 2) >> 2, ew = warp - 2;
    const int units = (nvalid + 7) >> 3;   // eight-column units, dealt to the four warps of a quarter in turn
    int lt = 0;
    for (int64_t m = gi; m < g.m_tiles; m += group, ++lt) {
      const int ab = lt & 1;
      const uint32_t ar = (uint32_t)(lt >> 1);
      if (!mbar_wait(&acc_full[ab], ar & 1)) { if (lane == 0) atomicExch(&fail, 1); break; }
      __syncwarp();
      tc_after();
      const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(ab * 256);
      // rows fit 32 bits (checked by the host)
      const uint32_t r = (uint32_t)(m * BM) + (uint32_t)(quarter * 32 + lane), rn = (uint32_t)g.rows_normal;
      const bool in = r < (uint32_t)g.rows, normal = r < rn;
      float *dst = nullptr;     // column b (< Nv) of this row
      __nv_bfloat16 *dst16 = nullptr;
      int64_t tpitch = 1;
      uint32_t rc = 0;          // transposed rows: row within the slice
      float2 rsum = make_float2(0.f, 0.f);   // lam of the row, occupied part of the slice
      bool dead = false, no0 = false, nodiag = false;   // scaled output: masks of the row
      if (in && normal) {
        dst = g.P + (int64_t)r * g.ldp;
      } else if (in) {
        const uint32_t q = r - rn, s = q / (uint32_t)g.Nv;
        rc = q - s * (uint32_t)g.Nv;
        if (g.PT16) dst16 = g.PT16 + (int64_t)s * g.Nv * g.ldp + rc;
        else dst = g.PT + (int64_t)s * g.Nv * g.ldp + rc;   // column b at dst + b * ldp
        tpitch = g.ldp;
        if (g.lam) {   // stored element (a = column, b = rc): the masks of the block vector
          const int code = g.code[s], blk = code & 7;
          const bool i0 = (code & 8) != 0, j0 = (code & 16) != 0;
          dead = (blk == 2 && (i0 || j0 || rc == 0)) || (blk == 4 && (j0 || rc == 0));
          no0 = blk == 2 || (blk == 4 && i0);
          nodiag = blk == 0 || blk == 2 || blk == 3;
          rsum = make_float2(g.lam[rc], g.occ[s]);
        }
      }
      // the warp's 32 rows form one run of a transposed slice (same slice, consecutive rows
      // starting on a multiple of 8): the staged 16-byte stores apply
      const uint32_t rc0 = __shfl_sync(0xffffffffu, rc, 0);
      const bool run = g.PT16 && __all_sync(0xffffffffu, in && !normal && rc == rc0 + lane) && (rc0 & 7) == 0;
      for (int u0 = part; u0 < units; u0 += 8) {
        uint32_t w[2][8];
        const bool second = u0 + 4 < units;   // uniform
        tmem_ld8(taddr + (uint32_t)(u0 * 8), w[0]);
        if (second) tmem_ld8(taddr + (uint32_t)(u0 * 8 + 32), w[1]);
        tmem_wait();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (h == 1 && !second) break;
          const int c = (u0 + 4 * h) * 8, bc = b0 + c, mcol = min(8, nvalid - c);
          float v[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            keep(w[h][q]);
            v[q] = __uint_as_float(w[h][q]);
          }
          if (g.PT16) {
            if (g.lam) {   // the approximate reciprocal serves the preconditioner: the denominator of
                           // (a, b) and of its image (b, a) is the same float, so M stays symmetric
              const float4 la = *reinterpret_cast<const float4 *>(&slam[c]), lb = *reinterpret_cast<const float4 *>(&slam[c + 4]);
              const float lc[8] = {la.x, la.y, la.z, la.w, lb.x, lb.y, lb.z, lb.w};
#pragma unroll
              for (int q = 0; q < 8; ++q) v[q] = dead ? 0.f : v[q] * rcp_approx((lc[q] + rsum.x) - rsum.y);
              if (no0 && bc == 0) v[0] = 0.f;
              if (nodiag && rc - (uint32_t)bc < 8u) {
#pragma unroll
                for (int q = 0; q < 8; ++q)
                  if ((uint32_t)(bc + q) == rc) v[q] = 0.f;
              }
            }
            if (run) {   // all 32 lanes here (every row of the warp is in range)
              __nv_bfloat16(*st)[40] = stg[ew];
              __syncwarp();
#pragma unroll
              for (int q = 0; q < 8; ++q) st[q][lane] = __float2bfloat16_rn(v[q]);
              __syncwarp();
              const int j = lane >> 2, hh = (lane & 3) * 8;   // column bc + j, rows hh .. hh + 7 of the run
              if (j < mcol)
                *reinterpret_cast<uint4 *>(dst16 - lane + (int64_t)(bc + j) * tpitch + hh) = *reinterpret_cast<const uint4 *>(&st[j][hh]);
            } else if (dst16) {
#pragma unroll
              for (int q = 0; q < 8; ++q)
                if (q < mcol) dst16[(int64_t)(bc + q) * tpitch] = __float2bfloat16_rn(v[q]);
            }
          } else if (dst) {
            if (normal && mcol == 8) {
              float4 *d4 = reinterpret_cast<float4 *>(dst + bc);
              d4[0] = make_float4(v[0], v[1], v[2], v[3]);
              d4[1] = make_float4(v[4], v[5], v[6], v[7]);
            } else {
#pragma unroll
              for (int q = 0; q < 8; ++q)
                if (q < mcol) dst[(int64_t)(bc + q) * tpitch] = v[q];
            }
          }
        }
      }
      tc_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[ab]);
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

}  // namespace vg

// Column tiling of the GEMM: the fewest column tiles (each at most 256 columns, a multiple of
// 16) whose resident panel and an operand ring of at least 5 slots fit the shared memory of
// one CTA; the ring takes what is left, up to MAX_STAGES slots.  bk: K elements per chunk.
static bool vgemm_tiling(int ncols, int Kc, int bk, int *nN, int *Nt, int *nk, int *stages, int *smem) {
  const int k = (Kc + bk - 1) / bk;
  for (int n = 1; n <= 64; ++n) {
    const int t = (((ncols + n - 1) / n) + 15) & ~15;
    const int fixed = 1024 + k * t * vg::CHUNK_B;
    if (t > 256 || fixed + 5 * vg::A_STAGE > vg::SMEM_MAX) continue;
    const int st = std::min(vg::MAX_STAGES, (vg::SMEM_MAX - fixed) / vg::A_STAGE);
    // at least 120 KB, so one CTA per SM: each CTA holds all 512 TMEM columns
    *nN = n; *Nt = t; *nk = k; *stages = st; *smem = std::max(fixed + st * vg::A_STAGE, 120 * 1024);
    return true;
  }
  return false;
}

// P = A W on the tensor cores.  A: rows x Nvp (row pitch Nvp elements), W: Nv x Nvp (row b of
// W is column b of the right factor), both bf16, or both float32 read as tf32 (tf32 = true).
esmp2_status vgemm(esmp2_handle *h, const void *A, int64_t rows, int64_t rows_normal, const void *W, float *P,
                   float *PT, int ldp, double alg_flops, bool tf32, const VgemmOut *out) {
  const int Nv = h->d.Nv, Nvp = (Nv + 7) & ~7;
  const int bk = tf32 ? vg::Kind<true>::BK : vg::Kind<false>::BK, esz = tf32 ? 4 : 2;
  int nN = 0, Nt = 0, nk = 0, stages = 0, smem = 0;
  if (!vgemm_tiling(Nv, Nv, bk, &nN, &Nt, &nk, &stages, &smem) || (ldp & 3) || rows <= 0) {
    h->err = "vgemm: unsupported shape";
    return ESMP2_ERR_UNSUPPORTED;
  }
  if (rows >= (int64_t)1 << 31) {
    h->err = "vgemm: too many rows";
    return ESMP2_ERR_UNSUPPORTED;
  }
  if (rows_normal < rows && (rows - rows_normal) % Nv != 0) {
    h->err = "vgemm: transposed rows must be whole slices";
    return ESMP2_ERR_UNSUPPORTED;
  }
  CUtensorMap mA, mW;
  if (!tma_map_2d(&mA, A, tf32, (uint64_t)Nvp, (uint64_t)rows, (uint64_t)Nvp * esz, (uint32_t)bk, vg::BM, 64) ||
      !tma_map_2d(&mW, W, tf32, (uint64_t)Nvp, (uint64_t)Nv, (uint64_t)Nvp * esz, (uint32_t)bk, (uint32_t)Nt, 64)) {
    h->err = "vgemm: tensor map encoding failed";
    return ESMP2_ERR_CUDA;
  }
  const void *fn = tf32 ? reinterpret_cast<const void *>(vg::k_vgemm<true>)
                        : reinterpret_cast<const void *>(vg::k_vgemm<false>);
  if (cudaError_t e = smem_limit_once(fn, vg::SMEM_MAX)) return check_cuda(h, e, "vgemm shared-memory limit");
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  vg::Args g{};
  g.rows = rows;
  g.rows_normal = rows_normal;
  g.Nv = Nv;
  g.nk = nk;
  g.nN = nN;
  g.Nt = Nt;
  g.stages = stages;
  g.m_tiles = (rows + vg::BM - 1) / vg::BM;
  g.P = P;
  g.PT = PT;
  g.ldp = ldp;
  g.err = h->dflag;
  if (out) {
    g.PT16 = static_cast<__nv_bfloat16 *>(out->PT16);
    g.lam = out->lam;
    g.occ = out->occ;
    g.code = out->code;
  }
  const int family = out ? out->family : ESMP2_KT_CONTRACTION;
  const int64_t per_group = std::max<int64_t>(1, std::min<int64_t>(g.m_tiles, sms / nN));
  const int grid = (int)(per_group * nN);
  const double exec = 2.0 * (double)g.m_tiles * vg::BM * (double)Nv * (double)nN * Nt;
  {
    KScope ks(h->stream, family, alg_flops, exec);
    if (tf32) vg::k_vgemm<true><<<grid, vg::NTHREADS, smem, h->stream>>>(mA, mW, g);
    else vg::k_vgemm<false><<<grid, vg::NTHREADS, smem, h->stream>>>(mA, mW, g);
  }
  h->launches += 1;
  return check_cuda(h, cudaGetLastError(), "vgemm");
}

}  // namespace esmp2
