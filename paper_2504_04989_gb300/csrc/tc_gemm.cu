// tc_gemm.cu -- batched real GEMM on the 5th-generation tensor cores:
//   C_b (M x N, FP32) = A_b (M x K) * B_b^T,   B_b stored N x K,
// A and B K-major (K contiguous), TF32 (FP32 storage) or BF16 operands, FP32
// accumulation in tensor memory.
//
// One CTA computes a 128 x BN tile, BN = 128, or 256 when
// N > 128 (a product with N in (128, 256], as the Krylov products' 2b real
// columns, then reads each row panel of A once).  Operand tiles of 128 (A) and BN (B) rows x 128
// bytes of K are staged by TMA (128-byte swizzle) through a ring of shared
// buffers guarded by mbarriers; one thread issues tcgen05.mma (4 per stage,
// 32 bytes of K each) into a BN-column TMEM accumulator and commits each
// stage back to the producer; eight further warps read the accumulator with
// tcgen05.ld and store it through shared memory, 128 bytes of a row per eight
// lanes (C = alpha A B^T + beta C, the old values loaded before any store).  A
// CTA walks over several tiles with two accumulators, so the next tile's loads
// and products run under the storing of this one (2048 x 120 x 360 on 65 slices,
// added to C with split copies: 357 -> 258 us; TF32, 2048 x 120 x 2048: 470 -> 440).  Every wait is bounded: on a
// timeout the kernel records an error flag instead of hanging.  The split-TF32 epilogue can also write
// hi / lo copies of C for a following product.
//
// A third mode keeps FP32 accuracy on the TF32 units ("split TF32"): each
// operand is split as x = hi + lo with hi = x rounded to TF32 and lo = x - hi
// (exact in FP32), and the tile product is hi*hi + hi*lo + lo*hi accumulated
// in the same TMEM tile (about 22 significant bits per product; lo*lo, below
// FP32 rounding, is dropped).  Four operand tiles per stage: three stages of 128
// bytes of K at 128 columns, four of 64 bytes at 256 columns.
//
// Complex products use it without moving the big operand: an interleaved
// complex matrix X (rows x cols) is the real matrix [Re Im Re Im ...] of
// rows x 2cols, so X * Y = real(X) * E(Y)^T with a small expanded real form
// E(Y) of the thin factor (see expand_* below).  X^H Y with both factors tall
// takes their de-interleaved columns instead (split_deinterleave): one real
// product of the rows Re x_c, Im x_c against those of Y, combined 2 x 2.
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_common.cuh"

namespace tsvd {

constexpr int TC_BM = 128;
constexpr int TC_DRAIN = 256;  // threads that read the accumulator (8 warps, 4 KB of staging each), then one TMA and one MMA warp
constexpr int TC_THREADS = TC_DRAIN + 64;
// MODE 0: TF32, 1: BF16, 2: split TF32; BN: 128 or 256 columns per tile
template <int MODE, int BN>
constexpr int tc_row() { return MODE == 2 && BN == 256 ? 64 : 128; }  // bytes of K per stage
template <int MODE, int BN>
constexpr int tc_a_bytes() { return TC_BM * tc_row<MODE, BN>(); }
template <int MODE, int BN>
constexpr int tc_b_bytes() { return BN * tc_row<MODE, BN>(); }
template <int MODE, int BN>
constexpr int tc_stage_bytes() {  // A, B[, A lo, B lo]
  return (MODE == 2 ? 2 : 1) * (tc_a_bytes<MODE, BN>() + tc_b_bytes<MODE, BN>());
}
template <int MODE, int BN>
constexpr int tc_stages() { return MODE == 2 && BN == 128 ? 3 : 4; }
template <int MODE, int BN>
constexpr int tc_smem() { return tc_stages<MODE, BN>() * tc_stage_bytes<MODE, BN>() + 1024 + 256 + TC_DRAIN / 32 * 4096; }

// hi = x rounded to the nearest TF32 (lo = x - hi is exact in FP32)
__device__ __forceinline__ float tf32_hi(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// instruction descriptor: D FP32, A/B TF32 (kind::tf32) or BF16 (kind::f16),
// both K-major, M = 128, N = BN
template <bool BF16, int BN>
__device__ __forceinline__ uint32_t instr_desc() {
  static_assert(BN % 16 == 0 && BN >= 16 && BN <= 256, "M = 128 takes N in [16, 256], a multiple of 16");
  const uint32_t fmt = BF16 ? 1u : 2u;
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(TC_BM >> 4) << 24);
}

template <int MODE, int BN>
__global__ void __launch_bounds__(TC_THREADS, 1) k_tc_gemm(const __grid_constant__ CUtensorMap tmA,
                                                           const __grid_constant__ CUtensorMap tmB,
                                                           const __grid_constant__ CUtensorMap tmA2,
                                                           const __grid_constant__ CUtensorMap tmB2,
                                                           float* __restrict__ C, long ldc, long sC, int M, int N, int nk,
                                                           int batch, int* __restrict__ err, float alpha, float beta,
                                                           TcSplitOut o2) {
  constexpr bool BF16 = MODE == 1, SPLIT = MODE == 2;
  constexpr int STAGES = tc_stages<MODE, BN>(), SB = tc_stage_bytes<MODE, BN>();
  static_assert(tc_smem<MODE, BN>() <= 227 * 1024, "the stages must fit the opt-in shared memory of a CTA");
  constexpr int AB = tc_a_bytes<MODE, BN>(), BB = tc_b_bytes<MODE, BN>(), ROW = tc_row<MODE, BN>();
  auto desc = [](uint32_t addr) { return ROW == 64 ? smem_desc_sw64(addr) : smem_desc_sw128(addr); };
  extern __shared__ unsigned char tc_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)tc_raw + 1023) & ~(uintptr_t)1023);
  // o: A, B, A lo, B lo (every offset a multiple of 1024 bytes)
  auto operand = [&](int s, int o) {
    return smem_u32(base + s * SB + (o & 1) * AB + (o >> 1) * (AB + BB));
  };
  uint64_t* bars = (uint64_t*)(base + STAGES * SB);  // full[S], empty[S], tfull[2], tempty[2]
  uint32_t* tslot = (uint32_t*)(bars + 2 * STAGES + 4);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tn = (N + BN - 1) / BN, tm = (M + TC_BM - 1) / TC_BM;
  const int tiles = tn * tm * batch;  // at least one element each: within an int
  struct Tile {
    int n0, m0, bz;
  };
  auto tile = [&](int t) {  // columns fastest: neighbouring CTAs share rows of A
    const int r = t / tn;
    return Tile{(t % tn) * BN, (r % tm) * TC_BM, r / tm};
  };
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES);
  const uint32_t tfull = smem_u32(bars + 2 * STAGES), tempty = tfull + 16;
  constexpr int KE = ROW / (BF16 ? 2 : 4);  // elements of K per stage

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(tfull + 8 * s, 1);
      mbar_init(tempty + 8 * s, TC_DRAIN);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(2 * BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tslot;

  // stages are counted through all tiles of the CTA and two accumulators alternate, so loads and
  // products of the next tile run under the writing of this one
  if (tid == TC_DRAIN) {  // TMA producer
    Ring<STAGES> r;
    long filled = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
      const Tile w = tile(t);
      for (int kb = 0; kb < nk; ++kb, ++filled, r.next()) {
        const int s = r.s;
        if (!mbar_wait(empty0 + 8 * s, r.ph ^ 1)) {
          ok = false;
          break;
        }
        const uint32_t bar = full0 + 8 * s;
        mbar_expect_tx(bar, SB);
        tma_load_3d(operand(s, 0), &tmA, kb * KE, w.m0, w.bz, bar);
        tma_load_3d(operand(s, 1), &tmB, kb * KE, w.n0, w.bz, bar);
        if (SPLIT) {
          tma_load_3d(operand(s, 2), &tmA2, kb * KE, w.m0, w.bz, bar);
          tma_load_3d(operand(s, 3), &tmB2, kb * KE, w.n0, w.bz, bar);
        }
      }
    }
    ring_drain(r, filled, full0);
  } else if (tid == TC_DRAIN + 32) {  // MMA issuer
    const uint32_t idesc = instr_desc<BF16, BN>();
    Ring<STAGES> r;
    Ring<2> ra;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x, ra.next()) {
      const int a = ra.s;
      if (!mbar_wait(tempty + 8 * a, ra.ph ^ 1)) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
      const uint32_t d = tmem + (uint32_t)(a * BN);
      for (int kb = 0; kb < nk; ++kb, r.next()) {
        const int s = r.s;
        if (!mbar_wait(full0 + 8 * s, r.ph)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint64_t ad = desc(operand(s, 0)), bd = desc(operand(s, 1));
#pragma unroll
        for (int kk = 0; kk < ROW / 32; ++kk) {  // 32 bytes of K per instruction: advance the start address by 2 x 16 B
          mma_issue<BF16>(d, ad + 2 * kk, bd + 2 * kk, idesc, (kb | kk) != 0);
          if (SPLIT) {
            const uint64_t ad2 = desc(operand(s, 2)), bd2 = desc(operand(s, 3));
            mma_issue<BF16>(d, ad + 2 * kk, bd2 + 2 * kk, idesc, 1);
            mma_issue<BF16>(d, ad2 + 2 * kk, bd + 2 * kk, idesc, 1);
          }
        }
        mma_commit(empty0 + 8 * s);
      }
      if (ok) mma_commit(tfull + 8 * a);
    }
  } else if (warp < TC_DRAIN / 32) {
    const int row0 = (warp & 3) * 32, col0 = (warp >> 2) * (BN / 2);
    float4* stg = (float4*)(base + STAGES * SB + 256) + warp * 256;  // 32 rows x 32 floats, swizzled
    const int q8 = lane & 7;
    Ring<2> ra;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, ra.next()) {
      const Tile w = tile(t);
      const int a = ra.s;
      if (!__all_sync(0xffffffffu, mbar_wait(tfull + 8 * a, ra.ph))) {
        if (lane == 0) atomicExch(err, 1);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
      // 32 columns at a time through shared memory, so that eight lanes write 128 bytes of a row
#pragma unroll 1
      for (int c0 = 0; c0 < BN / 2; c0 += 32) {
        const uint32_t ta = tmem + ((uint32_t)row0 << 16) + (uint32_t)(a * BN + col0 + c0);
        uint32_t r[32];
#pragma unroll
        for (int h = 0; h < 32; h += 16)
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
              "%14, %15}, [%16];"
              : "=r"(r[h]), "=r"(r[h + 1]), "=r"(r[h + 2]), "=r"(r[h + 3]), "=r"(r[h + 4]), "=r"(r[h + 5]),
                "=r"(r[h + 6]), "=r"(r[h + 7]), "=r"(r[h + 8]), "=r"(r[h + 9]), "=r"(r[h + 10]), "=r"(r[h + 11]),
                "=r"(r[h + 12]), "=r"(r[h + 13]), "=r"(r[h + 14]), "=r"(r[h + 15])
              : "r"(ta + (uint32_t)h));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (c0 + 32 == BN / 2) {  // the accumulator has been read
          asm volatile("tcgen05.fence::before_thread_sync;");
          mbar_arrive(tempty + 8 * a);
        }
        if (w.n0 + col0 + c0 >= N) continue;
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 8; ++q)
          stg[lane * 8 + (q ^ q8)] =
              make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]), __uint_as_float(r[4 * q + 2]),
                          __uint_as_float(r[4 * q + 3]));
        __syncwarp();
        const int col = w.n0 + col0 + c0 + 4 * q8, left = N - col;
        float* Cb = C + (long)w.bz * sC + col;
        float4 v[8], old[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int rr = 4 * i + (lane >> 3), row = w.m0 + row0 + rr;
          v[i] = stg[rr * 8 + (q8 ^ (rr & 7))];
          if (beta == 0.0f || row >= M || left <= 0) continue;  // the old values all loaded first
          const float* src = Cb + (long)row * ldc;
          if (left >= 4 && ((uintptr_t)src & 15) == 0) {
            old[i] = *(const float4*)src;
          } else {
            old[i].x = src[0];
            old[i].y = left > 1 ? src[1] : 0.f;
            old[i].z = left > 2 ? src[2] : 0.f;
            old[i].w = left > 3 ? src[3] : 0.f;
          }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int rr = 4 * i + (lane >> 3), row = w.m0 + row0 + rr;
          if (row >= M || left <= 0) continue;
          // C = alpha A B^T + beta C
          float4 x = make_float4(alpha * v[i].x, alpha * v[i].y, alpha * v[i].z, alpha * v[i].w);
          if (beta != 0.0f)
            x = make_float4(fmaf(beta, old[i].x, x.x), fmaf(beta, old[i].y, x.y), fmaf(beta, old[i].z, x.z),
                            fmaf(beta, old[i].w, x.w));
          auto put = [&](float* dst, float4 y) {
            if (left >= 4 && ((uintptr_t)dst & 15) == 0) {
              *(float4*)dst = y;
            } else {
              dst[0] = y.x;
              if (left > 1) dst[1] = y.y;
              if (left > 2) dst[2] = y.z;
              if (left > 3) dst[3] = y.w;
            }
          };
          put(Cb + (long)row * ldc, x);
          if (o2.Rhi) {  // split copy in C's layout
            const float4 hi = make_float4(tf32_hi(x.x), tf32_hi(x.y), tf32_hi(x.z), tf32_hi(x.w));
            const long off = (long)w.bz * o2.sr + (long)row * o2.ldr + col;
            put(o2.Rhi + off, hi);
            put(o2.Rlo + off, make_float4(x.x - hi.x, x.y - hi.y, x.z - hi.z, x.w - hi.w));
          }
        }
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN));
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// rows x K (elements) per batch, row stride ld, batch stride sb (elements); boxes of
// box_rows rows x row bytes of K
static int make_map(CUtensorMap* tm, const void* ptr, int rows, int K, long ld, long sb, int batch, bool bf16,
                    int box_rows = TC_BM, int row = 128) {
  auto enc = get_encode();
  if (!enc) return TSVD_ERR_CUDA;
  const size_t es = bf16 ? 2 : 4;
  cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)(ld * es), (cuuint64_t)(sb * es)};
  cuuint32_t box[3] = {(cuuint32_t)(row / es), (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(tm, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, (void*)ptr, dims,
                   strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   row == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? TSVD_OK : TSVD_ERR_UNSUPPORTED;
}

bool tc_gemm_supported(const void* A, long lda, long sA, const void* B, long ldb, long sB, int batch, bool bf16) {
  const long es = bf16 ? 2 : 4;
  auto al = [](long bytes) { return bytes % 16 == 0; };
  if (((uintptr_t)A & 15) || ((uintptr_t)B & 15)) return false;
  if (!al(lda * es) || !al(ldb * es)) return false;
  if (batch > 1 && (!al(sA * es) || !al(sB * es))) return false;
  return batch <= 65535;
}

template <int MODE, int BN>
static int tc_launch(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& ta2, const CUtensorMap& tb2,
                     float* C, long ldc, long sC, int M, int N, int nk, int batch, int* err, cudaStream_t s,
                     float alpha = 1.0f, float beta = 0.0f, const TcSplitOut& o2 = TcSplitOut()) {
  const long tiles = (long)cdiv(N, BN) * cdiv(M, TC_BM) * batch;
  if (cudaFuncSetAttribute(k_tc_gemm<MODE, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem<MODE, BN>()) !=
      cudaSuccess) {
    cudaGetLastError();
    return TSVD_ERR_CUDA;
  }
  k_tc_gemm<MODE, BN><<<(unsigned)std::min<long>(tiles, SMS), TC_THREADS, tc_smem<MODE, BN>(), s>>>(
      ta, tb, ta2, tb2, C, ldc, sC, M, N, nk, batch, err, alpha, beta, o2);
  TSVD_LAUNCHED();
  return TSVD_OK;
}
// tile width: 256 columns when N > 128 (one tile row covers the whole of N <= 256)
static int tc_bn(int N) { return N > 128 ? 256 : 128; }

int tc_gemm(const void* A, long lda, long sA, int M, const void* B, long ldb, long sB, int N, int K, float* C, long ldc,
            long sC, int batch, bool bf16, int* err, cudaStream_t s) {
  if (M <= 0 || N <= 0 || batch <= 0) return TSVD_OK;
  if (!tc_gemm_supported(A, lda, sA, B, ldb, sB, batch, bf16)) return TSVD_ERR_UNSUPPORTED;
  CUtensorMap ta, tb;
  const int bn = tc_bn(N);
  TSVD_TRY(make_map(&ta, A, M, K, lda, sA, batch, bf16));
  TSVD_TRY(make_map(&tb, B, N, K, ldb, sB, batch, bf16, bn));
  const int kelem = bf16 ? 64 : 32;
  const int nk = (K + kelem - 1) / kelem;
  if (bf16)
    return bn == 256 ? tc_launch<1, 256>(ta, tb, ta, tb, C, ldc, sC, M, N, nk, batch, err, s)
                     : tc_launch<1, 128>(ta, tb, ta, tb, C, ldc, sC, M, N, nk, batch, err, s);
  return bn == 256 ? tc_launch<0, 256>(ta, tb, ta, tb, C, ldc, sC, M, N, nk, batch, err, s)
                   : tc_launch<0, 128>(ta, tb, ta, tb, C, ldc, sC, M, N, nk, batch, err, s);
}

int tc_gemm_split(const float* Ahi, const float* Alo, long lda, long sA, int M, const float* Bhi, const float* Blo,
                  long ldb, long sB, int N, int K, float* C, long ldc, long sC, int batch, int* err, cudaStream_t s,
                  float alpha, float beta, const TcSplitOut* out2) {
  if (M <= 0 || N <= 0 || batch <= 0) return TSVD_OK;
  if (!tc_gemm_supported(Ahi, lda, sA, Bhi, ldb, sB, batch, false) ||
      !tc_gemm_supported(Alo, lda, sA, Blo, ldb, sB, batch, false))
    return TSVD_ERR_UNSUPPORTED;
  // columns per tile: shared memory feeds the products (every instruction reads its 128 rows of A and
  // BN of B, 160 KB per 32 terms at 128 columns with the filling, 240 KB at 256, against 128 bytes per
  // clock), so a term of K costs a tile of 256 about 1.5 times one of 128.  The 48 products of a T-SVD
  // of 2048 x 2048 x 128 took 12.2 ms with 128 columns throughout, 11.1 so (one tile per CTA).
  const long rows = (long)cdiv(M, TC_BM) * batch;
  const bool wide = 3 * cdiv(rows * cdiv(N, 256), SMS) <= 2 * cdiv(rows * cdiv(N, 128), SMS);
  const int bn = wide ? 256 : 128, row = wide ? 64 : 128;
  CUtensorMap ta, tb, ta2, tb2;
  TSVD_TRY(make_map(&ta, Ahi, M, K, lda, sA, batch, false, TC_BM, row));
  TSVD_TRY(make_map(&tb, Bhi, N, K, ldb, sB, batch, false, bn, row));
  TSVD_TRY(make_map(&ta2, Alo, M, K, lda, sA, batch, false, TC_BM, row));
  TSVD_TRY(make_map(&tb2, Blo, N, K, ldb, sB, batch, false, bn, row));
  const TcSplitOut o2 = out2 ? *out2 : TcSplitOut();
  return wide ? tc_launch<2, 256>(ta, tb, ta2, tb2, C, ldc, sC, M, N, (K + 15) / 16, batch, err, s, alpha, beta, o2)
              : tc_launch<2, 128>(ta, tb, ta2, tb2, C, ldc, sC, M, N, (K + 31) / 32, batch, err, s, alpha, beta, o2);
}

// ---------------------------------------------------------------------------
// Expanded real forms of a thin complex factor Y (K x N per batch, interleaved,
// leading dim ldy), as E (2N x 2K per batch, leading dim lde), so that for an
// interleaved complex X (rows x K) seen as a real rows x 2K matrix,
// real(X) * E^T is the interleaved complex product:
//   mode 0 (X Y):       E[2n][2k] = Yr, E[2n][2k+1] = -Yi, E[2n+1][2k] = Yi, E[2n+1][2k+1] = Yr
//   mode 1 (conj(X) Y): E[2n][2k] = Yr, E[2n][2k+1] =  Yi, E[2n+1][2k] = Yi, E[2n+1][2k+1] = -Yr
// ---------------------------------------------------------------------------
template <typename O>
__device__ __forceinline__ O cvt_out(float v);
template <>
__device__ __forceinline__ float cvt_out<float>(float v) {
  return v;
}
template <>
__device__ __forceinline__ __nv_bfloat16 cvt_out<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}

// 32 x 32 tiles of Y (k rows x n columns) through shared memory: reads
// coalesced along n (Y's rows), writes coalesced along k (E's rows).
template <typename O>
__global__ void __launch_bounds__(256) k_expand(const float2* __restrict__ Y, long ldy, long sy, int K, int N,
                                                O* __restrict__ E, long lde, long se, int mode) {
  __shared__ float2 t[32][33];
  const int b = blockIdx.z, k0 = blockIdx.y * 32, n0 = blockIdx.x * 32;
  const float2* Yb = Y + (long)b * sy;
  for (int kk = threadIdx.y; kk < 32; kk += blockDim.y) {
    const int k = k0 + kk, n = n0 + threadIdx.x;
    t[kk][threadIdx.x] = (k < K && n < N) ? Yb[(long)k * ldy + n] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  O* Eb = E + (long)b * se;
  for (int nn = threadIdx.y; nn < 32; nn += blockDim.y) {
    const int n = n0 + nn, k = k0 + threadIdx.x;
    if (n >= N || k >= K) continue;
    const float2 y = t[threadIdx.x][nn];
    O* e0 = Eb + (long)(2 * n) * lde + 2 * k;
    O* e1 = e0 + lde;
    if (mode == 0) {
      e0[0] = cvt_out<O>(y.x);
      e0[1] = cvt_out<O>(-y.y);
      e1[0] = cvt_out<O>(y.y);
      e1[1] = cvt_out<O>(y.x);
    } else {
      e0[0] = cvt_out<O>(y.x);
      e0[1] = cvt_out<O>(y.y);
      e1[0] = cvt_out<O>(y.y);
      e1[1] = cvt_out<O>(-y.x);
    }
  }
}

int expand_thin(const float2* Y, long ldy, long sy, int K, int N, void* E, long lde, long se, int batch, int mode,
                bool bf16, cudaStream_t s) {
  if ((long)batch * K * N <= 0) return TSVD_OK;
  if (batch > 65535 || cdiv(K, 32) > 65535) return TSVD_ERR_UNSUPPORTED;
  dim3 grid(cdiv(N, 32), cdiv(K, 32), batch), block(32, 8);
  if (bf16)
    k_expand<__nv_bfloat16><<<grid, block, 0, s>>>(Y, ldy, sy, K, N, (__nv_bfloat16*)E, lde, se, mode);
  else
    k_expand<float><<<grid, block, 0, s>>>(Y, ldy, sy, K, N, (float*)E, lde, se, mode);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

// rows x cols FP32 (leading dim ldx) to BF16 (round to nearest even) or FP32
// with leading dim ldy; the padding columns are zeroed
template <typename O>
__global__ void k_copy_rows(const float* __restrict__ x, long ldx, O* __restrict__ y, long ldy, int cols, long rows) {
  const long total = rows * ldy;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    const long r = i / ldy;
    const long c = i % ldy;
    y[i] = cvt_out<O>(c < cols ? x[r * ldx + c] : 0.0f);
  }
}

int copy_rows(const float* x, long ldx, void* y, long ldy, int cols, long rows, bool bf16, cudaStream_t s) {
  const long total = rows * ldy;
  if (total <= 0) return TSVD_OK;
  const unsigned grid = std::min<long>(cdiv(total, 256), 8192);
  if (bf16) k_copy_rows<__nv_bfloat16><<<grid, 256, 0, s>>>(x, ldx, (__nv_bfloat16*)y, ldy, cols, rows);
  else k_copy_rows<float><<<grid, 256, 0, s>>>(x, ldx, (float*)y, ldy, cols, rows);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

// ---------------------------------------------------------------------------
// Split operands for the split-TF32 mode: hi = x rounded to the nearest TF32
// (cvt.rna.tf32.f32), lo = x - hi (exact in FP32).
// ---------------------------------------------------------------------------

// Columns [0, fill) of hi / lo rows (leading dim ldy) from rows x cols FP32 (leading dim ldx, zeros from
// cols on): 2^lg lanes per row, W floats per lane.  Bound: its bytes (the eight passes of a T-SVD of 2048 x 2048 x
// 128, 4 GB: 1.01 ms with an element and two 64-bit divisions per thread, 0.65 so).
template <int W>
__global__ void __launch_bounds__(256) k_split_rows(const float* __restrict__ x, long ldx, float* __restrict__ hi,
                                                    float* __restrict__ lo, long ldy, int cols, int fill, long rows,
                                                    int lg) {
  const int lane = threadIdx.x & 31, sub = lane & ((1 << lg) - 1);
  const long warps = (long)gridDim.x * 8 << (5 - lg);
  for (long r = ((long)blockIdx.x * 8 + (threadIdx.x >> 5) << (5 - lg)) + (lane >> lg); r < rows; r += warps) {
    const float* src = x + r * ldx;
    float *h = hi + r * ldy, *l = lo + r * ldy;
#pragma unroll 4
    for (int c = sub * W; c < fill; c += W << lg) {
      if constexpr (W == 4) {
        const float4 v = c < cols ? *(const float4*)(src + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 y = make_float4(tf32_hi(v.x), tf32_hi(v.y), tf32_hi(v.z), tf32_hi(v.w));
        *(float4*)(h + c) = y;
        *(float4*)(l + c) = make_float4(v.x - y.x, v.y - y.y, v.z - y.z, v.w - y.w);
      } else {
        const float v = c < cols ? src[c] : 0.f, y = tf32_hi(v);
        h[c] = y;
        l[c] = v - y;
      }
    }
  }
}

static int split_fill(const float* x, long ldx, float* hi, float* lo, long ldy, int cols, int fill, long rows,
                      cudaStream_t s) {
  if (rows <= 0 || fill <= 0) return TSVD_OK;
  const bool vec = (((uintptr_t)x | (uintptr_t)hi | (uintptr_t)lo) & 15) == 0 && ldx % 4 == 0 && ldy % 4 == 0 &&
                   cols % 4 == 0 && fill % 4 == 0;
  int lg = 0;
  while (lg < 5 && (vec ? 4 : 1) << lg < fill) ++lg;
  const unsigned grid = (unsigned)std::min<long>(cdiv(rows, 8L << (5 - lg)), SMS * 16);
  if (vec) k_split_rows<4><<<grid, 256, 0, s>>>(x, ldx, hi, lo, ldy, cols, fill, rows, lg);
  else k_split_rows<1><<<grid, 256, 0, s>>>(x, ldx, hi, lo, ldy, cols, fill, rows, lg);
  TSVD_LAUNCHED();
  return TSVD_OK;
}
// rows x cols FP32 (leading dim ldx) to hi / lo rows of leading dim ldy (padding zeroed)
int split_rows(const float* x, long ldx, float* hi, float* lo, long ldy, int cols, long rows, cudaStream_t s) {
  return split_fill(x, ldx, hi, lo, ldy, cols, (int)ldy, rows, s);
}
// columns [0, cols) of FP32 rows (leading dim ldx) -> hi (nearest TF32) / lo rows of leading dim ldy;
// the other columns of the destination rows are left as they are
int split_block(const float* x, long ldx, float* hi, float* lo, long ldy, int cols, long rows, cudaStream_t s) {
  return split_fill(x, ldx, hi, lo, ldy, cols, cols, rows, s);
}

// per slice: complex X (rows x cols, interleaved, leading dim cols) transposed
// to XT (cols x rows complex = real rows of 2 rows floats, leading dim ldt),
// split into hi / lo; 32 x 32 complex tiles through shared memory
__global__ void k_split_transpose(const float2* __restrict__ X, int rows, int cols, long ldx, long sx,
                                  float* __restrict__ hi, float* __restrict__ lo, long ldt, long st) {
  __shared__ float2 t[32][33];
  const int b = blockIdx.z;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  const float2* Xb = X + (long)b * sx;
  for (int rr = threadIdx.y; rr < 32; rr += blockDim.y) {
    const int r = r0 + rr, c = c0 + threadIdx.x;
    t[rr][threadIdx.x] = (r < rows && c < cols) ? Xb[(long)r * ldx + c] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  float* hb = hi + (long)b * st;
  float* lb = lo + (long)b * st;
  for (int cc = threadIdx.y; cc < 32; cc += blockDim.y) {
    const int c = c0 + cc, r = r0 + threadIdx.x;
    if (c < cols && r < rows) {
      const float2 v = t[threadIdx.x][cc];
      const float hx = tf32_hi(v.x), hy = tf32_hi(v.y);
      hb[(long)c * ldt + 2 * r] = hx;
      hb[(long)c * ldt + 2 * r + 1] = hy;
      lb[(long)c * ldt + 2 * r] = v.x - hx;
      lb[(long)c * ldt + 2 * r + 1] = v.y - hy;
    }
  }
}

int split_transpose(const float2* X, int rows, int cols, int batch, float* hi, float* lo, long ldt, cudaStream_t s) {
  if (rows <= 0 || cols <= 0 || batch <= 0) return TSVD_OK;
  if (batch > 65535) return TSVD_ERR_UNSUPPORTED;
  // zero the padding columns of every row once (2 rows .. ldt)
  if (ldt > 2L * rows) {
    if (cudaMemset2DAsync(hi + 2L * rows, ldt * sizeof(float), 0, (ldt - 2L * rows) * sizeof(float),
                          (size_t)batch * cols, s) != cudaSuccess ||
        cudaMemset2DAsync(lo + 2L * rows, ldt * sizeof(float), 0, (ldt - 2L * rows) * sizeof(float),
                          (size_t)batch * cols, s) != cudaSuccess)
      return TSVD_ERR_CUDA;
  }
  dim3 grid(cdiv(cols, 32), cdiv(rows, 32), batch), block(32, 8);
  k_split_transpose<<<grid, block, 0, s>>>(X, rows, cols, cols, (long)rows * cols, hi, lo, ldt, (long)cols * ldt);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

// per slice: the columns of a complex X (rows x cols, leading dim ldx) as real rows of
// length `rows`: row 2c the real parts of column c, row 2c+1 the imaginary parts, split
// into hi / lo (leading dim ldt, batch stride st); 32 x 32 complex tiles through shared memory
__global__ void k_split_deinterleave(const float2* __restrict__ X, int rows, int cols, long ldx, long sx,
                                     float* __restrict__ hi, float* __restrict__ lo, long ldt, long st) {
  __shared__ float2 t[32][33];
  const int b = blockIdx.z;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  const float2* Xb = X + (long)b * sx;
  for (int rr = threadIdx.y; rr < 32; rr += blockDim.y) {
    const int r = r0 + rr, c = c0 + threadIdx.x;
    t[rr][threadIdx.x] = (r < rows && c < cols) ? Xb[(long)r * ldx + c] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  float* hb = hi + (long)b * st;
  float* lb = lo + (long)b * st;
  for (int cc = threadIdx.y; cc < 32; cc += blockDim.y) {
    const int c = c0 + cc, r = r0 + threadIdx.x;
    if (c < cols && r < rows) {
      const float2 v = t[threadIdx.x][cc];
      const float hx = tf32_hi(v.x), hy = tf32_hi(v.y);
      hb[(long)(2 * c) * ldt + r] = hx;
      hb[(long)(2 * c + 1) * ldt + r] = hy;
      lb[(long)(2 * c) * ldt + r] = v.x - hx;
      lb[(long)(2 * c + 1) * ldt + r] = v.y - hy;
    }
  }
}

int split_deinterleave(const float2* X, int rows, int cols, long ldx, long sx, int batch, float* hi, float* lo,
                       long ldt, long st, cudaStream_t s) {
  if (rows <= 0 || cols <= 0 || batch <= 0) return TSVD_OK;
  if (batch > 65535) return TSVD_ERR_UNSUPPORTED;
  dim3 grid(cdiv(cols, 32), cdiv(rows, 32), batch), block(32, 8);
  k_split_deinterleave<<<grid, block, 0, s>>>(X, rows, cols, ldx, sx, hi, lo, ldt, st);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

// expanded real form (as expand_thin, FP32) split into hi / lo; same tiling
__global__ void __launch_bounds__(256) k_expand_split(const float2* __restrict__ Y, long ldy, long sy, int K, int N,
                                                      float* __restrict__ Eh, float* __restrict__ El, long lde,
                                                      long se, int mode) {
  __shared__ float2 t[32][33];
  const int b = blockIdx.z, k0 = blockIdx.y * 32, n0 = blockIdx.x * 32;
  const float2* Yb = Y + (long)b * sy;
  for (int kk = threadIdx.y; kk < 32; kk += blockDim.y) {
    const int k = k0 + kk, n = n0 + threadIdx.x;
    t[kk][threadIdx.x] = (k < K && n < N) ? Yb[(long)k * ldy + n] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  for (int nn = threadIdx.y; nn < 32; nn += blockDim.y) {
    const int n = n0 + nn, k = k0 + threadIdx.x;
    if (n >= N || k >= K) continue;
    const float2 y = t[threadIdx.x][nn];
    const float v[4] = {y.x, mode == 0 ? -y.y : y.y, y.y, mode == 0 ? y.x : -y.x};
    const long o0 = (long)b * se + (long)(2 * n) * lde + 2 * k;
    const long off[4] = {o0, o0 + 1, o0 + lde, o0 + lde + 1};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float h = tf32_hi(v[q]);
      Eh[off[q]] = h;
      El[off[q]] = v[q] - h;
    }
  }
}

int expand_thin_split(const float2* Y, long ldy, long sy, int K, int N, float* Eh, float* El, long lde, long se,
                      int batch, int mode, cudaStream_t s) {
  if ((long)batch * K * N <= 0) return TSVD_OK;
  if (batch > 65535 || cdiv(K, 32) > 65535) return TSVD_ERR_UNSUPPORTED;
  dim3 grid(cdiv(N, 32), cdiv(K, 32), batch), block(32, 8);
  k_expand_split<<<grid, block, 0, s>>>(Y, ldy, sy, K, N, Eh, El, lde, se, mode);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

}  // namespace tsvd
