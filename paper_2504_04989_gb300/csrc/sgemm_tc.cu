// sgemm_tc.cu -- FP32 complex GEMM on the BF16 tensor cores, exact operands.
//
// Each operand is the sum of three BF16 numbers, x = b0 + b1 + b2, each the nearest to what is left:
// 8 + 8 + 8 bits, so the split is exact.  The six products b_i b_j with i + j <= 2 are accumulated on
// tcgen05 (those left out lie below 2^-26 of the product, under half its FP32 rounding), at the price of
// three of the TF32 rate.  The tensor cores truncate when they add to an accumulator (measured: a sum
// kept in TMEM shrinks by about 2e-8 per instruction, 1.4e-5 after 1024 complex terms), so an accumulator
// holds 32 terms of K of b0 b0 only, two instructions on products of 16 bits that rarely lose any,
// and is then read and added to sums in registers, rounded to nearest, in runs of eight
// readings; the five small products, 2^-9 of those and less, have accumulators of their own that are read once a run.
// Two pairs of accumulators alternate so that the reading runs under the next products, and a CTA walks over several
// tiles so that the next tile's loads and products run under the writing of this one.  Against exact dot products the
// result is closer than FP32 multiply-adds' at every K (the figures stand at sgemm_tc_better).
//
// Near the ends of FP32's range the parts or their products leave it: an entry below 2^-100 (its b2), a sum below
// 2^-98 per term with products below 2^-100 in it, results that are not finite.  The pass over the operands notes how
// small the entries of each row get, and the elements concerned are left to k_redo.
//
// A complex product is the real product of the interleaved rows of op(A) with the
// expanded real form of op(B) (rows 2n and 2n + 1 per column n, as in tc_gemm.cu),
// both written as three planes by one pass over the operands.
//
// Bound: shared memory, 136 KB read and filled per 128 x 128 x 32 block (1063 clocks at 128
// bytes per clock; the products alone take 768).
#include <cuda_bf16.h>

#include <cmath>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_common.cuh"
#include "tc_redo.cuh"

namespace tsvd {

constexpr int SG_D = 3;                  // BF16 parts
constexpr int SG_BM = 128, SG_BN = 128;  // complex rows x real columns
constexpr int SG_KB = 64;                // K per stage: rows of 128 bytes, 128-byte swizzle
constexpr int SG_STAGES = 2;
constexpr int SG_KA = 32;                // K per reading of the accumulators
constexpr int SG_TILE = SG_BM * SG_KB * 2;        // one part of either operand
constexpr int SG_STAGE_BYTES = 2 * SG_D * SG_TILE;  // A, B
constexpr int SG_RUN = 8;                // readings summed before they join the total
constexpr int SG_DRAIN = 256;            // threads reading the accumulators, then one TMA and one MMA warp
constexpr int SG_THREADS = SG_DRAIN + 64;
constexpr int SG_OUT = SG_BN / 2;        // columns per reading thread
constexpr int SG_SMEM = SG_STAGES * SG_STAGE_BYTES + 1024 + 256 + SG_DRAIN / 32 * 4096;  // 4 KB per reading warp
static_assert(SG_SMEM <= 227 * 1024, "the stages must fit a CTA's shared memory");

// one operand as its pass sees it: rows (columns of op(B)) of K elements
struct SplitOp {
  const float2* S;
  long ld, ss;
  int rows;
  bool trans;  // stored K x rows, else rows x K
  bool conj;   // enters conjugated
  uint8_t* low;  // [batch][rows][lowk]: per 32 of K, bits 0 to 3: an entry below 2^-25, 2^-50, 2^-75, 2^-100
  uint32_t* D;   // planes of the parts, [batch][3][rows, or 2 rows for op(B)][ldk]
  __host__ __device__ unsigned blocks(int K) const { return (unsigned)((rows + 31) / 32) * ((K + 31) / 32); }
};
__host__ __device__ __forceinline__ int sg_lowk(int K) { return ((K + 31) / 32 + 7) / 8 * 8; }  // read 8 bytes at a time

// the three parts' bits
__device__ __forceinline__ void bf16_parts(float x, uint32_t (&b)[SG_D]) {
#pragma unroll
  for (int s = 0; s < SG_D; ++s) {
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    b[s] = __bfloat16_as_ushort(h);
    x -= __bfloat162float(h);
  }
}

// Both operands to planes of parts: blocks, tiles and rows as in k_dig_pack.  Also clears the marks.
__global__ void __launch_bounds__(256) k_split_pack(const SplitOp A, const SplitOp B, int K, long ldk,
                                                    const Marks<float2> marks) {
  __shared__ float2 t[32][33];
  const bool first = blockIdx.x < A.blocks(K);
  const SplitOp& o = first ? A : B;
  const int blk = first ? blockIdx.x : blockIdx.x - A.blocks(K), b = blockIdx.z;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int kblocks = (K + 31) / 32, kb = blk % kblocks, k0 = kb * 32, r0 = blk / kblocks * 32, rows = o.rows;
  marks.clear(((long)b * gridDim.x + blockIdx.x) * 256 + threadIdx.x, (long)gridDim.z * gridDim.x * 256);
  const float2* S = o.S + (long)b * o.ss;
  if (o.trans) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = k0 + ty + 8 * i, r = r0 + tx;
      t[ty + 8 * i][tx] = (k < K && r < rows) ? S[(long)k * o.ld + r] : make_float2(0.f, 0.f);
    }
    __syncthreads();
  }
  const int k = k0 + tx;
  const long plane = (long)rows * (first ? 1 : 2) * (ldk / 2);  // 32-bit words of a plane
  const uint32_t sign = (o.conj == first) ? 0x8000u : 0u;  // of the imaginary part in the first row
  const int lowk = sg_lowk(K);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + 8 * i;  // the same for the whole warp
    if (r >= rows) break;
    float2 v = make_float2(0.f, 0.f);
    if (k < K) v = o.trans ? t[tx][ty + 8 * i] : S[(long)r * o.ld + k];
    const float x = v.x != 0.f ? fabsf(v.x) : 1.f, y = v.y != 0.f ? fabsf(v.y) : 1.f;
    const unsigned least = __reduce_min_sync(0xffffffffu, __float_as_uint(fminf(x, y))) >> 23;  // its exponent
    if (tx < (kb == kblocks - 1 ? lowk - kb : 1))  // the last block fills up the row
      o.low[((long)b * rows + r) * lowk + kb + tx] =
          tx ? 0 : (least < 102) + 2 * (least < 77) + 4 * (least < 52) + 8 * (least < 27);
    if (k >= K) continue;
    uint32_t re[SG_D], im[SG_D];
    bf16_parts(v.x, re);
    bf16_parts(v.y, im);
    uint32_t* dst = o.D + (long)b * SG_D * plane + (long)(first ? r : 2 * r) * (ldk / 2) + k;
#pragma unroll
    for (int s = 0; s < SG_D; ++s) {
      dst[s * plane] = re[s] | ((im[s] ^ sign) << 16);
      if (!first) dst[s * plane + ldk / 2] = (im[s] ^ (sign ^ 0x8000u)) | (re[s] << 16);
    }
  }
}

__global__ void __launch_bounds__(SG_THREADS, 1) k_sgemm_tc(const __grid_constant__ CUtensorMap tmA,
                                                            const __grid_constant__ CUtensorMap tmB,
                                                            const uint8_t* __restrict__ lowA,
                                                            const uint8_t* __restrict__ lowB,
                                                            const __grid_constant__ Marks<float2> marks,
                                                            float2* __restrict__ C, long ldc, long sC, int M, int N,
                                                            int K, int batch, float alpha, int beta, TcOpts st) {
  extern __shared__ unsigned char sg_raw[];
  const int nk = (2 * K + SG_KB - 1) / SG_KB, na = (2 * K + SG_KA - 1) / SG_KA;  // stages and readings of a tile
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tn = (2 * N + SG_BN - 1) / SG_BN, tm = (M + SG_BM - 1) / SG_BM;
  const int tiles = tn * tm * batch;  // at least one element each: within an int
  struct Tile {
    int n0, m0, bz;
  };
  auto tile = [&](int t) {  // columns fastest: neighbouring CTAs share rows of A
    const int r = t / tn;
    return Tile{(t % tn) * SG_BN, (r % tm) * SG_BM, r / tm};
  };
  unsigned char* base = (unsigned char*)(((uintptr_t)sg_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(base + SG_STAGES * SG_STAGE_BYTES);  // full[S], empty[S], tfull[2], tempty[2]
  uint32_t* tslot = (uint32_t*)(bars + 2 * SG_STAGES + 4);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + SG_STAGES);
  const uint32_t tfull = smem_u32(bars + 2 * SG_STAGES), tempty = tfull + 16;
  if (tid == 0) {
    for (int s = 0; s < SG_STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(tfull + 8 * s, 1);
      mbar_init(tempty + 8 * s, SG_DRAIN);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tslot;
  auto wait = [&](uint32_t bar, uint32_t parity) { return !st.expire && mbar_wait(bar, parity); };

  // stages and accumulators are counted through all tiles of the CTA, so loads and products of the
  // next tile run under the writing of this one
  if (tid == SG_DRAIN) {  // TMA producer
    Ring<SG_STAGES> r;
    long filled = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
      const Tile w = tile(t);
      for (int kb = 0; kb < nk; ++kb, ++filled, r.next()) {
        const int s = r.s;
        if (!wait(empty0 + 8 * s, r.ph ^ 1)) {
          ok = false;
          break;
        }
        const uint32_t dst = smem_u32(base + s * SG_STAGE_BYTES), bar = full0 + 8 * s;
        mbar_expect_tx(bar, SG_STAGE_BYTES);
        tma_load_3d(dst, &tmA, kb * SG_KB, w.m0, w.bz * SG_D, bar);
        tma_load_3d(dst + SG_D * SG_TILE, &tmB, kb * SG_KB, w.n0, w.bz * SG_D, bar);
      }
    }
    ring_drain(r, filled, full0);
  } else if (tid == SG_DRAIN + 32) {  // MMA issuer
    const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(SG_BM >> 4) << 24);  // FP32 += BF16 BF16^T
    const uint32_t idesc1 = idesc0 | ((uint32_t)(SG_BN >> 3) << 17), idesc2 = idesc0 | ((uint32_t)(2 * SG_BN >> 3) << 17);
    Ring<SG_STAGES> r;
    Ring<2> ra;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
      for (int kb = 0; ok && kb < nk; ++kb, r.next()) {
        const int s = r.s;
        if (!wait(full0 + 8 * s, r.ph)) {
          ok = false;
          break;
        }
        const uint32_t sm = smem_u32(base + s * SG_STAGE_BYTES);
        uint64_t pa[SG_D], pb[SG_D];
#pragma unroll
        for (int i = 0; i < SG_D; ++i) {
          pa[i] = smem_desc_sw128(sm + i * SG_TILE);
          pb[i] = smem_desc_sw128(sm + (SG_D + i) * SG_TILE);
        }
        const int parts = min(SG_KB / SG_KA, na - kb * (SG_KB / SG_KA));
        for (int p = 0; p < parts; ++p, ra.next()) {
          const int a = ra.s;
          if (!wait(tempty + 8 * a, ra.ph ^ 1)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t d = tmem + (uint32_t)(a * 2 * SG_BN);
          const int j = kb * (SG_KB / SG_KA) + p;
          const bool fresh = (j & (SG_RUN - 1)) < 2;  // the run's first use of this pair
#pragma unroll
          for (int kk = 0; kk < SG_KA / 16; ++kk) {
            const int at = 2 * (p * (SG_KA / 16) + kk);  // 32 bytes of K
            if (kk == 0) {
              mma_issue<true>(d, pa[0] + at, pb[0] + at, idesc1, 0);
              mma_issue<true>(d + SG_BN, pa[0] + at, pb[1] + at, idesc1, fresh ? 0 : 1);
            } else {
              mma_issue<true>(d, pa[0] + at, pb[0] + at, idesc2, 1);  // b0 b0 | b0 b1
            }
            mma_issue<true>(d + SG_BN, pa[0] + at, pb[2] + at, idesc1, 1);
            mma_issue<true>(d + SG_BN, pa[1] + at, pb[0] + at, idesc1, 1);
            mma_issue<true>(d + SG_BN, pa[1] + at, pb[1] + at, idesc1, 1);
            mma_issue<true>(d + SG_BN, pa[2] + at, pb[0] + at, idesc1, 1);
          }
          mma_commit(tfull + 8 * a);
        }
        if (ok) mma_commit(empty0 + 8 * s);
      }
    }
  } else if (warp < SG_DRAIN / 32) {
    const int row0 = (warp & 3) * 32, col0 = (warp >> 2) * SG_OUT;
    const uint32_t tw = tmem + ((uint32_t)row0 << 16) + (uint32_t)col0;
    float4* stg = (float4*)(base + SG_STAGES * SG_STAGE_BYTES + 256) + warp * 256;  // 32 rows x 32 floats
    Ring<2> ra;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
      const Tile w = tile(t);
      // notes of small entries in this lane's row and column: the first 256 of K ahead of the sums
      const int lr = min(w.m0 + row0 + lane, M - 1), lc = min((w.n0 + col0) / 2 + lane, N - 1), lowk = sg_lowk(K);
      const uint2* pr = (const uint2*)(lowA + ((long)w.bz * M + lr) * lowk);
      const uint2* pc = (const uint2*)(lowB + ((long)w.bz * N + lc) * lowk);
      const uint2 rl = pr[0], cl = pc[0];
      float run[SG_OUT], tot[SG_OUT];
#pragma unroll
      for (int q = 0; q < SG_OUT; ++q) run[q] = tot[q] = 0.f;
      for (int kb = 0; kb < na && ok; ++kb, ra.next()) {
        const int a = ra.s;
        ok = wait(tfull + 8 * a, ra.ph);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        // the sums of b0 b0; those of the small products at the run's last use of the pair
        const int halves = kb + 2 >= min(na, (kb & ~(SG_RUN - 1)) + SG_RUN) ? 2 : 1;
        for (int h = 0; h < halves; ++h) {
#pragma unroll
          for (int q0 = 0; q0 < SG_OUT; q0 += 16) {
            uint32_t r[16];
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                "%14, %15}, [%16];"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                  "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                : "r"(tw + (uint32_t)((2 * a + h) * SG_BN + q0)));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int u = 0; u < 16; ++u) run[q0 + u] += __uint_as_float(r[u]);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        mbar_arrive(tempty + 8 * a);
        if ((kb & (SG_RUN - 1)) == SG_RUN - 1 || kb == na - 1) {
#pragma unroll
          for (int q = 0; q < SG_OUT; ++q) {
            tot[q] += run[q];
            run[q] = 0.f;
          }
        }
      }
      if (!ok && lane == 0 && st.err) atomicExch(st.err, 1);
      // results that are not finite, or entries near the lower end of the range: the warp looks which of its elements
      // (rare)
      float zero = 0.f;
#pragma unroll
      for (int q = 0; q < SG_OUT; ++q) zero = fmaf(tot[q], 0.f, zero);
      uint32_t rlow = rl.x | rl.y, clow = cl.x | cl.y;
#pragma unroll 4
      for (int q = 1; q < lowk / 8; ++q) {
        const uint2 x = pr[q], y = pc[q];
        rlow |= x.x | x.y;
        clow |= y.x | y.y;
      }
      auto level = [](uint32_t x) {  // entries of at least 2^(-25 (level + 1)); 4: smaller ones
        x |= x >> 16;
        return __popc((x | x >> 8) & 15u);
      };
      const int rlev = level(rlow), clev = level(clow);
      const int rtop = __reduce_max_sync(0xffffffffu, rlev), ctop = __reduce_max_sync(0xffffffffu, clev);
      // products below 2^-100 among them, or parts below 2^-124
      const bool spoiled = ok && (__any_sync(0xffffffffu, zero != zero) || rtop + ctop > 2);
      const float least = 0x1p-98f * (2.f * (float)K);
      // 32 columns at a time through shared memory, so that eight lanes write 128 bytes of a row
#pragma unroll
      for (int c0 = 0; c0 < SG_OUT; c0 += 32) {
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 8; ++q)
          stg[lane * 8 + (q ^ (lane & 7))] =
              make_float4(tot[c0 + 4 * q], tot[c0 + 4 * q + 1], tot[c0 + 4 * q + 2], tot[c0 + 4 * q + 3]);
        __syncwarp();
        const int cb = (w.n0 + col0 + c0) >> 1, col = cb + 2 * (lane & 7);
        if (cb >= N) continue;
#pragma unroll 2
        for (int i = 0; i < 8; ++i) {
          const int r = 4 * i + (lane >> 3), row = w.m0 + row0 + r;
          if (w.m0 + row0 + 4 * i >= M) break;  // the same for the whole warp
          const float4 x = stg[r * 8 + ((lane & 7) ^ (r & 7))];
          float2* dst = C + (long)w.bz * sC + (long)row * ldc + col;
          float2 v[2] = {make_float2(alpha * x.x, alpha * x.y), make_float2(alpha * x.z, alpha * x.w)};
          bool out[2] = {row < M && col < N, row < M && col + 1 < N};
          if (spoiled) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int rl4 = __shfl_sync(0xffffffffu, rlev, r);
              const int cl4 = __shfl_sync(0xffffffffu, clev, c0 / 2 + 2 * (lane & 7) + u);
              const float big = fmaxf(fabsf(v[u].x), fabsf(v[u].y));
              const bool mark = out[u] && (!(fabsf(v[u].x) <= FLT_MAX && fabsf(v[u].y) <= FLT_MAX) ||
                                           max(rl4, cl4) > 3 || (rl4 + cl4 > 2 && big < least));
              marks.put(M, N, w.bz, w.m0 + row0 + 4 * i, cb + u, mark, row, col + u, lane);
              out[u] = out[u] && !mark;
            }
          }
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if (!ok) v[u] = make_float2(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000));
            if (beta && out[u]) v[u] = cadd(v[u], dst[u]);
          }
          if (out[0] && out[1] && ((uintptr_t)dst & 15) == 0) {
            *(float4*)dst = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
          } else {
            if (out[0]) dst[0] = v[0];
            if (out[1]) dst[1] = v[1];
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
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static int split_map(CUtensorMap* tm, const void* ptr, int rows, int K2, long ldk, int planes) {
  auto enc = get_encode();
  if (!enc) return TSVD_ERR_CUDA;
  cuuint64_t dims[3] = {(cuuint64_t)K2, (cuuint64_t)rows, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)(ldk * 2), (cuuint64_t)(ldk * 2 * rows)};
  cuuint32_t box[3] = {(cuuint32_t)SG_KB, 128, (cuuint32_t)SG_D};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)ptr, dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? TSVD_OK : TSVD_ERR_UNSUPPORTED;
}

static long sg_ldk(int K) { return (2L * K + 7) / 8 * 8; }
static size_t sg_slice_bytes(int M, int N, int K) {
  return SG_D * 2 * (size_t)sg_ldk(K) * (M + 2 * (size_t)N) + (size_t)sg_lowk(K) * ((size_t)M + N) +
         Marks<float2>::bytes(M, N, 1);
}
size_t sgemm_tc_bytes(int M, int N, int K, int batch) {
  return std::min<size_t>(sg_slice_bytes(M, N, K) * batch, (size_t)3 << 30) + sg_slice_bytes(M, N, K) + 2048;
}

// Estimated times in microseconds of the two forms: a SIMT tile takes 0.104 (64 x 64) or 0.25 us (128 x
// 64) per term of K and SM, K split as cgemm splits it.  Measured, product with its operand pass: 1024 x
// 1024 x 1024 on 33 slices 5.08 -> 1.61 ms (the product alone 1.28: 220 TFLOP/s); 2048 x 100 x 2048 on 17 takes 706 us
// (366), 512 x 60 x 512 on 33 85 us (37).  Error, 2-norm, in 2^-24, normal
// data, K = 32, 60, 128, 512, 2048: 0.8, 0.9, 1.1, 1.4, 1.7, the SIMT kernels 1.7, 2.3, 3.4, 6.8, 13.6; positive data
// 0.8, 0.9, 1.1, 1.0, 1.2, SIMT 1.4, 2.0, 2.9, 5.9, 11.7 (two TF32 parts and three products, as this was: 2.1 .. 2.6
// and 1.7 .. 1.9, from K = 56 on below SIMT only).
bool sgemm_tc_better(const GemmArgs& g, size_t bytes) {
  if (g.K < 1 || g.M < 1 || g.N < 1 || g.K > (1 << 24)) return false;
  const size_t slice = sg_slice_bytes(g.M, g.N, g.K) + 2048;
  if (bytes < slice) return false;
  const double wtiles = (double)cdiv(g.M, 128) * cdiv(g.N, 64) * g.batch;
  const bool wide = g.K >= 1024 || wtiles >= 2 * SMS;
  const double stiles = wide ? wtiles : (double)cdiv(g.M, 64) * cdiv(g.N, 64) * g.batch;
  double ks = std::min(16.0, std::max(1.0, std::floor(wide ? (4 * SMS + stiles - 1) / stiles : 2 * SMS / stiles)));
  ks = std::min(ks, std::max(1.0, g.K / 64.0));
  const double simt = 4.0 + (ks > 1.0 ? 3.0 : 0.0) + std::ceil(stiles * ks / SMS) * (g.K / ks) * (wide ? 0.25 : 0.104);
  const double tiles = (double)cdiv(g.M, SG_BM) * cdiv(2L * g.N, SG_BN) * g.batch;
  const double tile_us = 3.0 + cdiv(2L * g.K, SG_KB) * 0.55;
  const double pack_us = ((double)slice * 1.4 * g.batch) / 4.0e6;
  const double calls = std::ceil((double)g.batch * slice / (double)bytes);
  return simt > 10.0 * calls + pack_us + std::ceil(tiles / SMS) * tile_us;
}

int sgemm_tc(const GemmArgs& g, void* ws, size_t bytes, cudaStream_t s, TcOpts st) {
  const long ldk = sg_ldk(g.K);
  const int N2 = 2 * g.N;
  const uintptr_t p0 = ((uintptr_t)ws + 255) & ~(uintptr_t)255;
  const size_t off = p0 - (uintptr_t)ws + 1280;  // alignments
  const int nb = bytes < off ? 0 : (int)std::min<size_t>(g.batch, (bytes - off) / sg_slice_bytes(g.M, g.N, g.K));
  if (nb < 1) return TSVD_ERR_WORKSPACE;
  if (g.C == g.A || g.C == g.B) return TSVD_ERR_INVALID_ARG;  // k_redo reads the operands once more
  auto up = [](uintptr_t p) { return (p + 255) & ~(uintptr_t)255; };
  uint32_t* DA = (uint32_t*)p0;
  uint32_t* DB = (uint32_t*)up(p0 + (size_t)nb * SG_D * g.M * ldk * 2);
  uint8_t* lowA = (uint8_t*)up((uintptr_t)DB + (size_t)nb * SG_D * N2 * ldk * 2);
  uint8_t* lowB = lowA + (size_t)nb * g.M * sg_lowk(g.K);
  const Marks<float2> marks = Marks<float2>::at(up((uintptr_t)(lowB + (size_t)nb * g.N * sg_lowk(g.K))), g.M, g.N, nb);
  if (cudaFuncSetAttribute(k_sgemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM) != cudaSuccess) {
    cudaGetLastError();
    return TSVD_ERR_CUDA;
  }
  for (int b0 = 0; b0 < g.batch; b0 += nb) {
    const int n = std::min(nb, g.batch - b0);
    const float2* A = (const float2*)g.A + (long)b0 * g.sA;
    const float2* B = (const float2*)g.B + (long)b0 * g.sB;
    const SplitOp oa{A, g.lda, g.sA, g.M, g.opA == 'H', g.opA == 'H', lowA, DA};
    const SplitOp ob{B, g.ldb, g.sB, g.N, g.opB == 'N', g.opB == 'H', lowB, DB};
    k_split_pack<<<dim3(oa.blocks(g.K) + ob.blocks(g.K), 1, n), 256, 0, s>>>(oa, ob, g.K, ldk, marks);
    TSVD_LAUNCHED();
    CUtensorMap ma, mb;
    TSVD_TRY(split_map(&ma, DA, g.M, 2 * g.K, ldk, n * SG_D));
    TSVD_TRY(split_map(&mb, DB, N2, 2 * g.K, ldk, n * SG_D));
    const long tiles = (long)cdiv(N2, SG_BN) * cdiv(g.M, SG_BM) * n;
    float2* Cb = (float2*)g.C + (long)b0 * g.sC;
    k_sgemm_tc<<<(unsigned)std::min<long>(tiles, SMS), SG_THREADS, SG_SMEM, s>>>(
        ma, mb, lowA, lowB, marks, Cb, g.ldc, g.sC, g.M, g.N, g.K, n, (float)g.alpha, g.beta != 0.0, st);
    TSVD_LAUNCHED();
    TSVD_TRY(redo_marked<float2>(marks, {A, B, g.lda, g.sA, g.ldb, g.sB, g.K, g.opA == 'H', g.opB == 'H'}, Cb,
                                 g.ldc, g.sC, g.M, g.N, n, g.alpha, g.beta != 0.0, false, s));
  }
  return TSVD_OK;
}

}  // namespace tsvd
