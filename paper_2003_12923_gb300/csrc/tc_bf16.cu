// Virtual-index contractions of the sigma build on the 5th-generation tensor cores.
//
// For every slice s = (block, i, j) of the block vector (an Nv x Nv matrix X_s) the two
// virtual-index terms of the one-body operator are
//     Y_s = X_s F + F X_s            (F = F_vv, symmetric)
// i.e. the N_o^2 N_v^3 part of Table 1.  One CTA tile is (s, 128 rows a, <= 256 columns b);
// both terms accumulate into the same fp32 TMEM accumulator:
//     term 2: A = X_s[a-tile][c]   (K-major)   B = F[b-tile][c]      (K-major)
//     term 1: A = F[a-tile][c]     (K-major)   B = X_s[c][b-tile]    (MN-major)
// so each output element is written once.  Operands are bf16 (rounded copies of x and F),
// accumulation fp32.
//
// Structure (persistent, one CTA per SM, 320 threads):
//   warp 0      TMA producer: 3-D tiled bulk copies, 128-byte swizzle, 4-slot ring
//   warp 1      tcgen05.mma issuer (one elected thread), commits to mbarriers
//   warps 2..9  epilogue: tcgen05.ld 32x32b from the accumulator (two warps per lane
//               quarter, each half of the columns), fp32 or float64 stores
// Two TMEM accumulators (2 x 256 columns) let the epilogue of tile k overlap the main
// loop of tile k+1.  Every mbarrier wait is bounded by a globaltimer limit; a wait that
// runs out sets an error flag, skips the remaining work and the CTA still waits (bounded)
// for its own copies in flight and frees its TMEM before returning.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>
#include <mutex>
#include <map>
#include <cstdlib>

#include "internal.h"
#include "tc_ptx.h"

namespace esmp2 {
namespace tc {

using namespace ptx;

constexpr int BM = 128;           // accumulator rows (TMEM lanes)
constexpr int BN_MAX = 256;       // accumulator columns per tile
constexpr int BK = 64;            // K elements per stage (128 bytes of bf16)
constexpr int STAGES = 4;          // ring slots; a slot holds the operands of one term
constexpr int A_BYTES = BM * BK * 2;          // 16 KB
constexpr int B_BYTES = BN_MAX * BK * 2;      // 32 KB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024;
constexpr int NTHREADS = 320;     // producer warp, MMA warp, 8 epilogue warps

// Shared-memory matrix descriptor (tcgen05): start >> 4, LBO >> 4 at bit 16, SBO >> 4 at
// bit 32, descriptor version 1 at bit 46, layout type at bit 61 (2 = 128-byte swizzle).
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46) | (2ull << 61);
}
// Instruction descriptor, kind::f16: D fp32 (bit 4), A bf16 (bits 7-9 = 1), B bf16
// (bits 10-12 = 1), A K-major, B major at bit 16, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)b_mn_major << 16) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}

struct Args {
  int Nv;            // virtual orbitals (rows and columns of every slice)
  int nslices;       // slices of this launch
  const int *slices; // global slice index of each launched slice (nullptr: 0 .. nslices-1)
  int per_block;     // slices per amplitude block (No^2); block of slice s = s / per_block
  int tm[5];         // per block: 1 = x F only, 2 = x F + F x, 3 = F x only
  int a_tiles;       // ceil(Nv / 128)
  int b_tiles;       // column tiles per slice
  int bn;            // columns of a full column tile (multiple of 16, <= 256)
  int nk;            // K chunks: ceil(Nv / 64)
  int64_t tiles;     // nslices * a_tiles * b_tiles
  float *y32;        // [S][Nv][Nv]
  double *y64;       // not null: the same values are stored here, as float64, instead of y32
  int vec64;         // rows of y64 start on 16-byte boundaries
  int mirror;        // slices of T, X, Y (i < j listed) also write -y into slice (j, i)
  int No;
  int *err;          // error flag (device)
  uint64_t wait_ns;  // limit of every mbarrier wait (0: kWaitNs)
  int no_copies;     // failure-detection self-test only: the producer issues no copies, so the
                     // first wait on a full slot runs out with nothing in flight
};

__device__ __forceinline__ int slice_of(const Args &g, int64_t li) {
  return g.slices ? g.slices[li] : (int)li;
}
__device__ __forceinline__ int terms_of(const Args &g, int s) { return g.tm[s / g.per_block]; }

__global__ void __launch_bounds__(NTHREADS, 1)
    k_virt(const __grid_constant__ CUtensorMap tXa, const __grid_constant__ CUtensorMap tXb,
           const __grid_constant__ CUtensorMap tFa, const __grid_constant__ CUtensorMap tFb, Args g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t full[STAGES], empty[STAGES], acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_base;
  __shared__ int fail;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&acc_full[s], 1); mbar_init(&acc_empty[s], 8); }
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
  // launched programmatically behind its operand conversion: the set-up above overlaps it, and the
  // operands are complete from here on (returns at once for an ordinary launch)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const uint32_t tmem = tmem_base;
  const uint64_t lim = g.wait_ns ? g.wait_ns : kWaitNs;
  const int per_slice = g.a_tiles * g.b_tiles;

  if (warp == 0) {
    if (lane == 0) {  // ------------------------------------------------ TMA producer
      int64_t it = 0;
      bool ok = true;
      const uint32_t bytesXF = (uint32_t)(A_BYTES + g.bn * BK * 2);
      const int nb1 = (g.bn + 63) / 64;   // 64-column boxes of the MN-major X tile
      const uint32_t bytesFX = (uint32_t)(A_BYTES + nb1 * 64 * BK * 2);
      if (g.no_copies) ok = false;
      for (int64_t t = blockIdx.x; t < g.tiles && ok; t += gridDim.x) {
        const int s = slice_of(g, t / per_slice), rem = (int)(t % per_slice);
        const int terms = terms_of(g, s);
        const int a0 = (rem / g.b_tiles) * BM, b0 = (rem % g.b_tiles) * g.bn;
        for (int kc = 0; kc < g.nk && ok; ++kc) {
          const int c0 = kc * BK;
          for (int term = 1; term <= 2; ++term, ++it) {   // 1: x F, 2: F x
            if ((term == 1 && terms == 3) || (term == 2 && terms == 1)) { --it; continue; }
            const int st = (int)(it % STAGES);
            const uint32_t rnd = (uint32_t)(it / STAGES);
            if (!mbar_wait(&empty[st], (rnd & 1) ^ 1, lim)) { ok = false; break; }
            uint8_t *A = smem + st * STAGE_BYTES, *B = A + A_BYTES;
            if (term == 1) {   // A = X_s rows (128 x 64), B = F rows b (bn x 64), both K-major
              mbar_expect_tx(&full[st], bytesXF);
              tma_3d(A, &tXa, &full[st], c0, a0, s);
              tma_3d(B, &tFb, &full[st], c0, b0, 0);
            } else {           // A = F rows a (128 x 64), B = X_s[c][b] (4 boxes of 64 x 64, MN-major)
              mbar_expect_tx(&full[st], bytesFX);
              tma_3d(A, &tFa, &full[st], c0, a0, 0);
#pragma unroll
              for (int q = 0; q < nb1; ++q) tma_3d(B + q * (BK * 128), &tXb, &full[st], b0 + 64 * q, c0, s);
            }
          }
        }
      }
      if (!ok && !g.no_copies) atomicExch(&fail, 1);
      // wait (bounded) until no copy of this CTA is still in flight
      for (int64_t j = it > STAGES ? it - STAGES : 0; j < it; ++j)
        mbar_wait(&full[j % STAGES], (uint32_t)((j / STAGES) & 1), 100000000ull);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ------------------------------------------------ MMA issuer
      int64_t it = 0;
      int lt = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < g.tiles && ok; t += gridDim.x, ++lt) {
        const int s = slice_of(g, t / per_slice), rem = (int)(t % per_slice);
        const int terms = terms_of(g, s);
        const int b0 = (rem % g.b_tiles) * g.bn;
        const int nvalid = min(g.bn, g.Nv - b0);
        const int nmma = (nvalid + 15) & ~15;
        const uint32_t id2 = idesc_bf16(BM, nmma, 0), id1 = idesc_bf16(BM, nmma, 1);
        const int ab = lt & 1;
        const uint32_t ar = (uint32_t)(lt >> 1);
        if (!mbar_wait(&acc_empty[ab], (ar & 1) ^ 1, lim)) { ok = false; break; }
        tc_after();
        const uint32_t d = tmem + (uint32_t)(ab * BN_MAX);
        bool first = true;
        for (int kc = 0; kc < g.nk && ok; ++kc) {
          const int ksteps = min(BK / 16, (g.Nv - kc * BK + 15) / 16);
          for (int term = 1; term <= 2; ++term, ++it) {
            if ((term == 1 && terms == 3) || (term == 2 && terms == 1)) { --it; continue; }
            const int st = (int)(it % STAGES);
            const uint32_t rnd = (uint32_t)(it / STAGES);
            if (!mbar_wait(&full[st], rnd & 1, lim)) { ok = false; break; }
            tc_after();
            const uint32_t A = smem_u32(smem + st * STAGE_BYTES), B = A + A_BYTES;
            for (int k = 0; k < ksteps; ++k) {
              if (term == 1)   // X_s[a][c] F[c][b]
                umma_bf16(d, sdesc(A + 32 * k, 16, 1024), sdesc(B + 32 * k, 16, 1024), id2, first ? 0u : 1u);
              else             // F[a][c] X_s[c][b]
                umma_bf16(d, sdesc(A + 32 * k, 16, 1024), sdesc(B + 2048 * k, BK * 128, 1024), id1, first ? 0u : 1u);
              first = false;
            }
            umma_commit(&empty[st]);
          }
        }
        if (!ok) break;
        umma_commit(&acc_full[ab]);
      }
      if (!ok) atomicExch(&fail, 1);
    }
  } else {  // ---------------------------------------------------------- epilogue
    // warp w reads TMEM lanes 32 (w % 4) .. +31 (the tcgen05.ld lane rule); the two warps of
    // a lane quarter split the tile's columns
    const int quarter = warp & 3, chalf = (warp - 2) >> 2;
    int lt = 0;
    for (int64_t t = blockIdx.x; t < g.tiles; t += gridDim.x, ++lt) {
      const int s = slice_of(g, t / per_slice), rem = (int)(t % per_slice);
      const int a0 = (rem / g.b_tiles) * BM, b0 = (rem % g.b_tiles) * g.bn;
      const int nvalid = min(g.bn, g.Nv - b0);
      const int ab = lt & 1;
      const uint32_t ar = (uint32_t)(lt >> 1);
      if (!mbar_wait(&acc_full[ab], ar & 1, lim)) {
        if (lane == 0) atomicExch(&fail, 1);
        break;
      }
      tc_after();
      const int row = quarter * 32 + lane;
      const int a = a0 + row;
      const int64_t off = ((int64_t)s * g.Nv + a) * g.Nv + b0;
      const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(ab * BN_MAX);
      const int hc = ((nvalid + 31) / 32) * 16;   // columns per half, a multiple of 16
      const int c_begin = chalf * hc, c_end = min(nvalid, c_begin + hc);
      float *dst = g.y32 + off;
      float *dmr = nullptr;   // mirror slice (j, i) of an antisymmetric block
      if (g.mirror) {
        const int blk = s / g.per_block, ij = s % g.per_block;
        if (blk == 0 || blk == 2 || blk == 3) {
          const int sm = blk * g.per_block + (ij % g.No) * g.No + ij / g.No;
          dmr = g.y32 + ((int64_t)sm * g.Nv + a) * g.Nv + b0;
        }
      }
      for (int c = c_begin; c < c_end; c += 16) {
        float v[16];
        tmem_ld16(taddr + (uint32_t)c, v);
        if (a < g.Nv) {
          const int m = min(16, nvalid - c);
          if (g.y64) {
            double *q64 = g.y64 + off + c;
            if (m == 16 && g.vec64) {
#pragma unroll
              for (int q = 0; q < 8; ++q) reinterpret_cast<double2 *>(q64)[q] = make_double2(v[2 * q], v[2 * q + 1]);
            } else {
              for (int q = 0; q < m; ++q) q64[q] = (double)v[q];
            }
          } else if (m == 16 && (g.Nv & 3) == 0) {
            float4 *d4 = reinterpret_cast<float4 *>(dst + c);
#pragma unroll
            for (int q = 0; q < 4; ++q) d4[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            if (dmr) {
              float4 *m4 = reinterpret_cast<float4 *>(dmr + c);
#pragma unroll
              for (int q = 0; q < 4; ++q)
                m4[q] = make_float4(-v[4 * q], -v[4 * q + 1], -v[4 * q + 2], -v[4 * q + 3]);
            }
          } else {
            for (int q = 0; q < m; ++q) dst[c + q] = v[q];
            if (dmr)
              for (int q = 0; q < m; ++q) dmr[c + q] = -v[q];
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

// Both operands of the allocation-free contraction in one launch: bf16 rows (pitch Nvp, pad columns
// zero) of F, then of x; a thread converts eight columns.  Lets the contraction behind it start its
// set-up at once.  The call is a chain of latencies at small sizes: S=16 Nv=64 took 38.5 us with six
// dependent operations (flag memset, two conversions, contraction, float32 -> float64 pass, flag copy)
// and takes 22.3 us with these two launches and a flag that the host reads itself.
__global__ void __launch_bounds__(128) k_noalloc_operands(const double *F, const double *x, int Nv, int Nvp, int64_t rows,
                                                          __nv_bfloat16 *Fb, __nv_bfloat16 *xb) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int c8 = Nvp >> 3;
  const int64_t n = rows * c8;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = e / c8;
    const int c = (int)(e - r * c8) * 8;
    const bool isF = r < Nv;
    if (!isF) r -= Nv;
    const double *src = (isF ? F : x) + r * Nv;
    __align__(16) __nv_bfloat16 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = __float2bfloat16_rn(c + q < Nv ? (float)src[c + q] : 0.f);
    *reinterpret_cast<uint4 *>((isF ? Fb : xb) + r * Nvp + c) = *reinterpret_cast<uint4 *>(v);
  }
}

// bf16 copies: dst[s][r][c] (row pitch Nvp) = src[s][r][c] (row pitch Nv); pad columns zero.
template <typename T>
__global__ void k_to_bf16(const T *src, __nv_bfloat16 *dst, int64_t rows, int Nv, int Nvp) {
  const int64_t n = rows * Nvp;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / Nvp;
    const int c = (int)(e % Nvp);
    dst[e] = __float2bfloat16_rn(c < Nv ? (float)src[r * Nv + c] : 0.f);
  }
}

__global__ void k_fvv_bf16(const double *F, int No, int Nv, int Nvp, __nv_bfloat16 *dst) {
  const int N = No + Nv;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < Nv * Nvp; e += gridDim.x * blockDim.x) {
    const int r = e / Nvp, c = e % Nvp;
    dst[e] = __float2bfloat16_rn(c < Nv ? (float)F[(int64_t)(No + r) * N + No + c] : 0.f);
  }
}

}  // namespace tc

// ------------------------------------------------------------------------ host side
namespace {
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

bool get_encode() {
  if (g_encode) return true;
  cudaDriverEntryPointQueryResult q;
  void *fn = nullptr;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !fn)
    return false;
  g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  return true;
}

}  // namespace

bool tma_map_bf16(CUtensorMap *m, const void *base, int rank, const uint64_t *dims, const uint64_t *strides_bytes,
                  const uint32_t *box, int swizzle_bytes) {
  if (!get_encode()) return false;
  const uint32_t estr[3] = {1, 1, 1};
  return g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(base),
                  reinterpret_cast<const cuuint64_t *>(dims), reinterpret_cast<const cuuint64_t *>(strides_bytes),
                  reinterpret_cast<const cuuint32_t *>(box), estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  swizzle_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tma_map_2d(CUtensorMap *m, const void *base, bool f32, uint64_t inner, uint64_t outer, uint64_t row_bytes,
                uint32_t box_inner, uint32_t box_outer, int swizzle_bytes) {
  if (!get_encode()) return false;
  const uint64_t dims[2] = {inner, outer};
  const uint64_t strides[1] = {row_bytes};
  const uint32_t box[2] = {box_inner, box_outer};
  const uint32_t estr[2] = {1, 1};
  const CUtensorMapSwizzle sw = swizzle_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                : swizzle_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                : swizzle_bytes == 32 ? CU_TENSOR_MAP_SWIZZLE_32B
                                                      : CU_TENSOR_MAP_SWIZZLE_NONE;
  CUresult r = g_encode(m, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                        const_cast<void *>(base), reinterpret_cast<const cuuint64_t *>(dims),
                        reinterpret_cast<const cuuint64_t *>(strides), reinterpret_cast<const cuuint32_t *>(box), estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

namespace {
// Fills the tile geometry of `g` and launches k_virt.  xd: bf16 x [S][Nv][Nvp]; Fd: bf16 F [Nv][Nvp];
// Nvp = Nv rounded up to 8 (16-byte row pitch).
// overlap: the launch before it on the stream is k_noalloc_operands, whose tail it may overlap.
const char *launch_virt(cudaStream_t st, const void *xd, int S, const void *Fd, tc::Args &g, double alg_flops,
                        double exec_flops, bool overlap = false) {
  const int Nv = g.Nv, Nvp = (Nv + 7) & ~7;
  if (!get_encode()) return "cuTensorMapEncodeTiled unavailable";
  if (g.nslices <= 0) return nullptr;
  CUtensorMap mXa, mXb, mFa, mFb;
  const uint64_t dX[3] = {(uint64_t)Nvp, (uint64_t)Nv, (uint64_t)S};
  const uint64_t sX[2] = {(uint64_t)Nvp * 2, (uint64_t)Nvp * Nv * 2};
  const uint64_t dF[3] = {(uint64_t)Nvp, (uint64_t)Nv, 1};
  g.a_tiles = (Nv + tc::BM - 1) / tc::BM;
  if (g.bn <= 0 || g.bn > tc::BN_MAX || (g.bn & 15)) {   // default column tile: fewest tiles of <= 256
    g.b_tiles = (Nv + tc::BN_MAX - 1) / tc::BN_MAX;
    g.bn = ((Nv + g.b_tiles - 1) / g.b_tiles + 15) & ~15;
  } else {
    g.b_tiles = (Nv + g.bn - 1) / g.bn;
  }
  g.nk = (Nv + tc::BK - 1) / tc::BK;
  g.tiles = (int64_t)g.nslices * g.a_tiles * g.b_tiles;
  const uint32_t boxXa[3] = {64, 128, 1}, boxXb[3] = {64, 64, 1}, boxFa[3] = {64, 128, 1};
  const uint32_t boxFb[3] = {64, (uint32_t)g.bn, 1};
  if (!tma_map_bf16(&mXa, xd, 3, dX, sX, boxXa, 128) || !tma_map_bf16(&mXb, xd, 3, dX, sX, boxXb, 128) ||
      !tma_map_bf16(&mFa, Fd, 3, dF, sX, boxFa, 128) || !tma_map_bf16(&mFb, Fd, 3, dF, sX, boxFb, 128))
    return "tensor map encoding failed";
  if (smem_limit_once(reinterpret_cast<const void *>(tc::k_virt), tc::SMEM_BYTES) != cudaSuccess)
    return "cannot raise the shared-memory limit of the tensor-core kernel";
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = (int)std::min<int64_t>(g.tiles, sms);
  KScope ks(st, ESMP2_KT_CONTRACTION, alg_flops, exec_flops);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(tc::NTHREADS);
  cfg.dynamicSmemBytes = tc::SMEM_BYTES;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, tc::k_virt, mXa, mXb, mFa, mFb, g) == cudaSuccess ? nullptr : "k_virt launch failed";
}

tc::Args plain_args(int Nv, int S, float *y, int *err) {
  tc::Args g{};
  g.Nv = Nv;
  g.nslices = S;
  g.slices = nullptr;
  g.per_block = S;
  for (int b = 0; b < 5; ++b) g.tm[b] = 2;
  g.y32 = y;
  g.err = err;
  return g;
}
}  // namespace

// Inner-solve form: only T, X, Y slices with i < j and every S, Z slice are contracted; the
// slice (j, i) of T, X, Y receives -y_ij (the blocks are antisymmetric under i <-> j).
// bn: column tile width (0 = the default, fewest tiles of at most 256 columns).
static esmp2_status virt_bf16_sym_bn(esmp2_handle *h, const void *xb, const void *Fb, float *y, int *err, int bn) {
  if (esmp2_status s0 = ensure_slist(h)) return s0;
  const int No = h->d.No, S = 5 * No * No, half = No * (No - 1) / 2;
  const double nv = h->d.Nv, nv3 = nv * nv * nv;
  tc::Args g = plain_args(h->d.Nv, S, y, err);
  g.bn = bn;
  g.nslices = h->nslist;
  g.slices = h->slist;
  g.per_block = No * No;
  g.No = No;
  g.mirror = 1;
  // both terms of a slice share one pass (two one-term passes were measured slower: No=30
  // Nv=400 inner contraction 4.2 ms against 2.0 ms)
  const double exec1 = 4.0 * nv3 * 3 * half + 4.0 * nv3 * 2 * No * No;
  if (const char *m = launch_virt(h->stream, xb, S, Fb, g, alg_virtual_flops(No, h->d.Nv), exec1)) {
    h->err = m;
    return ESMP2_ERR_CUDA;
  }
  h->launches += 1;
  return check_cuda(h, cudaGetLastError(), "virt_bf16_sym");
}

// Tile table keyed by (No, Nv): on the first inner contraction of a shape in this process,
// the candidate column tile widths are timed on the handle's own operands (CUDA events,
// one warm-up and one timed launch each) and the fastest is kept for every later call.
// Candidates: the default, half of it, and 256 when Nv > 256.
namespace {
std::mutex g_tile_mu;
std::map<std::pair<int, int>, int> g_tile_table;
}  // namespace

int tuned_column_tile(esmp2_handle *h, const void *xb, const void *Fb, float *y, int *err) {
  const std::pair<int, int> key(h->d.No, h->d.Nv);
  {
    std::lock_guard<std::mutex> lk(g_tile_mu);
    auto it = g_tile_table.find(key);
    if (it != g_tile_table.end()) return it->second;
  }
  const int Nv = h->d.Nv;
  const int nt = (Nv + tc::BN_MAX - 1) / tc::BN_MAX;
  const int def = ((Nv + nt - 1) / nt + 15) & ~15;
  std::vector<int> cand = {def};
  const int halfw = ((def / 2) + 15) & ~15;
  if (halfw >= 32 && halfw != def) cand.push_back(halfw);
  if (Nv > tc::BN_MAX && def != tc::BN_MAX) cand.push_back(tc::BN_MAX);
  int best = def;
  float best_ms = 1e30f;
  cudaEvent_t e0, e1;
  if (cand.size() > 1 && cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess) {
    for (int bn : cand) {
      if (virt_bf16_sym_bn(h, xb, Fb, y, err, bn)) continue;
      cudaEventRecord(e0, h->stream);
      if (virt_bf16_sym_bn(h, xb, Fb, y, err, bn)) continue;
      cudaEventRecord(e1, h->stream);
      float ms = 0.f;
      if (cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess && ms < best_ms) {
        best_ms = ms;
        best = bn;
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
  }
  std::lock_guard<std::mutex> lk(g_tile_mu);
  g_tile_table[key] = best;
  return best;
}

esmp2_status virt_bf16_sym(esmp2_handle *h, const void *xb, const void *Fb, float *y, int *err) {
  return virt_bf16_sym_bn(h, xb, Fb, y, err, tuned_column_tile(h, xb, Fb, y, err));
}

// y[s][a][b] = sum_c xb[s][a][c] F[c][b] + sum_c F[a][c] xb[s][c][b]  for S slices (fp32 out).
// xb: bf16 [S][Nv][Nvp], Fb: bf16 [Nv][Nvp], Nvp = Nv rounded up to 8 (16-byte row pitch).
esmp2_status virt_bf16(esmp2_handle *h, const void *xb, const void *Fb, int S, float *y, int *err) {
  tc::Args g = plain_args(h->d.Nv, S, y, err);
  const double nv = h->d.Nv, exec = 4.0 * nv * nv * nv * S;
  const double alg = S == 5 * h->d.No * h->d.No ? alg_virtual_flops(h->d.No, h->d.Nv) : exec;
  if (const char *m = launch_virt(h->stream, xb, S, Fb, g, alg, exec)) { h->err = m; return ESMP2_ERR_CUDA; }
  h->launches += 1;
  return check_cuda(h, cudaGetLastError(), "virt_bf16");
}

void to_bf16_f64(esmp2_handle *h, const double *src, void *dst, int64_t rows) {
  const int Nv = h->d.Nv, Nvp = (Nv + 7) & ~7;
  tc::k_to_bf16<double><<<1216, 256, 0, h->stream>>>(src, static_cast<__nv_bfloat16 *>(dst), rows, Nv, Nvp);
  h->launches += 1;
}
void to_bf16_f32(esmp2_handle *h, const float *src, void *dst, int64_t rows) {
  const int Nv = h->d.Nv, Nvp = (Nv + 7) & ~7;
  tc::k_to_bf16<float><<<1216, 256, 0, h->stream>>>(src, static_cast<__nv_bfloat16 *>(dst), rows, Nv, Nvp);
  h->launches += 1;
}
void fvv_bf16(esmp2_handle *h, const double *F, void *dst) {
  const int Nv = h->d.Nv, Nvp = (Nv + 7) & ~7;
  tc::k_fvv_bf16<<<256, 256, 0, h->stream>>>(F, h->d.No, Nv, Nvp, static_cast<__nv_bfloat16 *>(dst));
  h->launches += 1;
}

}  // namespace esmp2

// ---------------------------------------------------------------------------------------
// Allocation-free variant of the bf16 virtual-index contraction.
//
// Some callers cannot allocate device memory at the point where they need this
// contraction: code that runs while another framework owns the whole device heap through
// its own caching allocator (a cudaMalloc there fails or fragments that allocator's
// budget), and latency-critical loops where a cudaMalloc/cudaFree pair would synchronise
// the device.  For them the scratch (bf16 copies of x and F) lives in one file-scope device array
// of ESMP2_NOALLOC_MAX_BYTES.  The size limit of a request also counts a float32 product, which the
// epilogue no longer writes: the limit is part of the call's contract.
// Every GPU that loads this library holds that array until the process exits.
namespace esmp2 {
namespace {

__device__ __align__(256) unsigned char g_noalloc_scratch[ESMP2_NOALLOC_MAX_BYTES];

constexpr int kMaxDevices = 64;
unsigned char *g_noalloc_ptr[kMaxDevices] = {nullptr};

// Error flag of the allocation-free contraction, one cache line per device.  Managed: the host clears
// and reads it without a launch or a copy, and the kernel touches it only when a wait has run out.
// The host may touch it while kernels of other streams run (cudaDevAttrConcurrentManagedAccess, which
// every GB300 has).
__managed__ int g_noalloc_flag[kMaxDevices][32];

inline size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace
}  // namespace esmp2

extern "C" esmp2_status esmp2_virtual_contraction_noalloc(const double *x, const double *Fvv, double *y, int S,
                                                         int Nv, void *stream) {
  using namespace esmp2;
  if (!x || !Fvv || !y || S < 1 || Nv < 1) return ESMP2_ERR_INVALID_ARG;
  const int Nvp = (Nv + 7) & ~7;
  const size_t off_F = 256;
  const size_t off_x = off_F + align256(sizeof(__nv_bfloat16) * (size_t)Nv * Nvp);
  const size_t off_y = off_x + align256(sizeof(__nv_bfloat16) * (size_t)S * Nv * Nvp);
  const size_t total = off_y + align256(sizeof(float) * (size_t)S * Nv * Nv);
  if (total > (size_t)ESMP2_NOALLOC_MAX_BYTES) return ESMP2_ERR_UNSUPPORTED;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ESMP2_ERR_CUDA;
  if (!g_noalloc_ptr[dev]) {  // one-time set-up on this device
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return ESMP2_ERR_CUDA;
    g_noalloc_ptr[dev] = static_cast<unsigned char *>(p);
  }
  if (!get_encode()) return ESMP2_ERR_CUDA;
  unsigned char *base = g_noalloc_ptr[dev];
  auto *Fb = reinterpret_cast<__nv_bfloat16 *>(base + off_F);
  auto *xb = reinterpret_cast<__nv_bfloat16 *>(base + off_x);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  volatile int *flag = g_noalloc_flag[dev];
  *flag = 0;
  const int64_t rows = (int64_t)(S + 1) * Nv;
  tc::k_noalloc_operands<<<(unsigned)std::min<int64_t>((rows * (Nvp / 8) + 127) / 128, 2432), 128, 0, st>>>(
      Fvv, x, Nv, Nvp, rows, Fb, xb);
  tc::Args g = plain_args(Nv, S, nullptr, g_noalloc_flag[dev]);
  g.y64 = y;
  g.vec64 = (Nv & 1) == 0 && (reinterpret_cast<uintptr_t>(y) & 15) == 0;
  const double exec = 4.0 * (double)Nv * Nv * Nv * S;
  if (launch_virt(st, xb, S, Fb, g, exec, exec, true)) return ESMP2_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return ESMP2_ERR_CUDA;
  if (cudaGetLastError() != cudaSuccess) return ESMP2_ERR_CUDA;
  return *flag ? ESMP2_ERR_TIMEOUT : ESMP2_OK;
}

// ---------------------------------------------------------------------------------------
// Failure-detection self-test of the bounded waits (the paper has no counterpart).
// One CTA of the tensor-core kernel runs on a 16 x 16 slice held in the allocation-free
// scratch array with its producer told to issue no copies: the MMA warp's first wait on a
// full slot and the epilogue's first wait on the accumulator run out after wait_ms with
// nothing in flight (no copy, no MMA, no TMEM load was issued), the CTA frees its TMEM and
// raises the error flag, and the host reads the flag like any other call.
extern "C" esmp2_status esmp2_selftest_bounded_wait(int wait_ms, void *stream) {
  using namespace esmp2;
  if (wait_ms < 1 || wait_ms > 2000) return ESMP2_ERR_INVALID_ARG;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ESMP2_ERR_CUDA;
  if (!g_noalloc_ptr[dev]) {
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return ESMP2_ERR_CUDA;
    g_noalloc_ptr[dev] = static_cast<unsigned char *>(p);
  }
  if (!get_encode()) return ESMP2_ERR_CUDA;
  const int Nv = 16;
  unsigned char *base = g_noalloc_ptr[dev];
  int *err = reinterpret_cast<int *>(base);
  void *op = base + 256;                                // operand maps need a valid address only
  float *y32 = reinterpret_cast<float *>(base + 4096);  // never written: no tile completes
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(base, 0, 8192, st) != cudaSuccess) return ESMP2_ERR_CUDA;
  tc::Args g = plain_args(Nv, 1, y32, err);
  g.wait_ns = (uint64_t)wait_ms * 1000000ull;
  g.no_copies = 1;
  if (launch_virt(st, op, 1, op, g, 0.0, 0.0)) return ESMP2_ERR_CUDA;
  int flag = 0;
  if (cudaMemcpyAsync(&flag, err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return ESMP2_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return ESMP2_ERR_CUDA;
  if (cudaGetLastError() != cudaSuccess) return ESMP2_ERR_CUDA;
  return flag ? ESMP2_ERR_TIMEOUT : ESMP2_OK;
}
