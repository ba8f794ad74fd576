// sgemm_tc.cu -- FP32 complex GEMM on the TF32 tensor cores with FP32 accuracy.
//
// Each operand is split x = hi + lo, hi the nearest TF32 and lo the nearest TF32 of
// the rest (2^-23 relative), and hi hi + hi lo + lo hi is accumulated on tcgen05.  The
// tensor cores truncate when they add to an accumulator (measured: a sum kept in TMEM
// shrinks by about 2e-8 per instruction, 1.4e-5 after 1024 complex terms), so an
// accumulator holds 32 terms of K only -- hi hi and the two small products apart, as B's hi
// and lo rows lie one after another and one instruction multiplies A hi with both -- and
// is then read and added to sums in registers, rounded to nearest, in runs of eight
// readings; two pairs of accumulators alternate so that the reading runs under the next
// products, and a CTA walks over several tiles so that the next tile's loads and products
// run under the writing of this one.  Against exact dot products of normal data the result
// is closer than FP32 multiply-adds' (the figures stand at sgemm_tc_better).
//
// A complex product is the real product of the interleaved rows of op(A) with the
// expanded real form of op(B) (rows 2n and 2n + 1 per column n, as in tc_gemm.cu),
// both written as hi / lo rows by one pass over each operand.
//
// Bound: shared memory, 144 KB read and filled per 128 x 128 x 32 block (1125 clocks at 128
// bytes per clock; the products alone take 768).  K = 100 (2048 x 2048 on 65 slices, most of it
// writing): 2.13 -> 1.70 ms by walking over tiles; K = 1024: 1.82 -> 1.81 ms by reading A hi
// once for both, 1.92 with 16 reading warps instead of 8.
#include <cmath>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_common.cuh"
#include "tc_redo.cuh"

namespace tsvd {

constexpr int SG_BM = 128, SG_BN = 128;  // complex rows x real columns
constexpr int SG_KB = 32;                // K per stage: rows of 128 bytes, 128-byte swizzle
constexpr int SG_STAGES = 3;
constexpr int SG_TILE = SG_BM * SG_KB * 4;
constexpr int SG_STAGE_BYTES = 4 * SG_TILE;  // A hi, A lo, B hi, B lo
constexpr int SG_RUN = 8;                // readings summed before they join the total
constexpr int SG_DRAIN = 256;            // threads reading the accumulators, then one TMA and one MMA warp
constexpr int SG_THREADS = SG_DRAIN + 64;
constexpr int SG_OUT = SG_BN / 2;        // columns per reading thread
constexpr int SG_SMEM = SG_STAGES * SG_STAGE_BYTES + 1024 + 256 + SG_DRAIN / 32 * 4096;  // 4 KB per reading warp
static_assert(SG_SMEM <= 227 * 1024, "the stages must fit a CTA's shared memory");

__device__ __forceinline__ float rna_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// one operand as k_split_pack sees it: rows (columns of op(B)) of K elements
struct SplitOp {
  const float2* S;
  long ld, ss;
  int rows;
  bool trans;  // stored K x rows, else rows x K
  bool conj;   // enters conjugated
  float *Hi, *Lo;
  __host__ __device__ unsigned blocks(int K) const { return (unsigned)((rows + 31) / 32) * ((K + 31) / 32); }
};

// Both operands to hi / lo rows of 2K floats (row length ldk): blocks and rows as in k_dig_pack.  Also clears
// the marks.
__global__ void __launch_bounds__(256) k_split_pack(const SplitOp A, const SplitOp B, int K, long ldk,
                                                    const Marks<float2> marks) {
  __shared__ float2 t[32][33];
  const bool first = blockIdx.x < A.blocks(K);
  const SplitOp& o = first ? A : B;
  const int blk = first ? blockIdx.x : blockIdx.x - A.blocks(K), b = blockIdx.z;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int kblocks = (K + 31) / 32, k0 = blk % kblocks * 32, r0 = blk / kblocks * 32, rows = o.rows;
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
  if (k >= K) return;
  const long so = (long)b * rows * (first ? 1 : 2) * ldk;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + 8 * i;
    if (r >= rows) continue;
    float2 v = o.trans ? t[tx][ty + 8 * i] : S[(long)r * o.ld + k];
    if (o.conj) v.y = -v.y;
    const float hx = rna_tf32(v.x), hy = rna_tf32(v.y), lx = rna_tf32(v.x - hx), ly = rna_tf32(v.y - hy);
    const long at = so + (long)(first ? r : 2 * r) * ldk + 2 * k;
    if (first) {
      *(float2*)(o.Hi + at) = make_float2(hx, hy);
      *(float2*)(o.Lo + at) = make_float2(lx, ly);
    } else {
      *(float2*)(o.Hi + at) = make_float2(hx, -hy);
      *(float2*)(o.Lo + at) = make_float2(lx, -ly);
      *(float2*)(o.Hi + at + ldk) = make_float2(hy, hx);
      *(float2*)(o.Lo + at + ldk) = make_float2(ly, lx);
    }
  }
}

__global__ void __launch_bounds__(SG_THREADS, 1) k_sgemm_tc(const __grid_constant__ CUtensorMap tmAh,
                                                            const __grid_constant__ CUtensorMap tmAl,
                                                            const __grid_constant__ CUtensorMap tmBh,
                                                            const __grid_constant__ CUtensorMap tmBl,
                                                            const __grid_constant__ Marks<float2> marks,
                                                            float2* __restrict__ C, long ldc, long sC, int M, int N,
                                                            int nk, int batch, float alpha, int beta) {
  extern __shared__ unsigned char sg_raw[];
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
        if (!mbar_wait(empty0 + 8 * s, r.ph ^ 1)) {
          ok = false;
          break;
        }
        const uint32_t dst = smem_u32(base + s * SG_STAGE_BYTES), bar = full0 + 8 * s;
        mbar_expect_tx(bar, SG_STAGE_BYTES);
        tma_load_3d(dst, &tmAh, kb * SG_KB, w.m0, w.bz, bar);
        tma_load_3d(dst + 2 * SG_TILE, &tmBh, kb * SG_KB, w.n0, w.bz, bar);
        tma_load_3d(dst + SG_TILE, &tmAl, kb * SG_KB, w.m0, w.bz, bar);
        tma_load_3d(dst + 3 * SG_TILE, &tmBl, kb * SG_KB, w.n0, w.bz, bar);
      }
    }
    ring_drain(r, filled, full0);
  } else if (tid == SG_DRAIN + 32) {  // MMA issuer
    const uint32_t idesc0 = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(SG_BM >> 4) << 24);  // FP32 += TF32 TF32^T
    const uint32_t idesc1 = idesc0 | ((uint32_t)(SG_BN >> 3) << 17), idesc2 = idesc0 | ((uint32_t)(2 * SG_BN >> 3) << 17);
    const long last = (long)((tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1) * nk;
    Ring<SG_STAGES> r;
    Ring<2> ra;
    for (long g = 0; g < last; ++g, r.next(), ra.next()) {
      const int s = r.s, a = ra.s;
      if (!mbar_wait(tempty + 8 * a, ra.ph ^ 1)) break;
      if (!mbar_wait(full0 + 8 * s, r.ph)) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
      const uint32_t sm = smem_u32(base + s * SG_STAGE_BYTES);
      const uint64_t ah = smem_desc_sw128(sm), al = smem_desc_sw128(sm + SG_TILE);
      const uint64_t bb = smem_desc_sw128(sm + 2 * SG_TILE);  // B hi, B lo: 256 rows
      const uint32_t d = tmem + (uint32_t)(a * 2 * SG_BN);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) mma_issue<false>(d, ah + 2 * kk, bb + 2 * kk, idesc2, kk > 0);  // 32 bytes of K
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) mma_issue<false>(d + SG_BN, al + 2 * kk, bb + 2 * kk, idesc1, 1);
      mma_commit(empty0 + 8 * s);
      mma_commit(tfull + 8 * a);
    }
  } else if (warp < SG_DRAIN / 32) {
    const int row0 = (warp & 3) * 32, col0 = (warp >> 2) * SG_OUT;
    const uint32_t tw = tmem + ((uint32_t)row0 << 16) + (uint32_t)col0;
    float4* stg = (float4*)(base + SG_STAGES * SG_STAGE_BYTES + 256) + warp * 256;  // 32 rows x 32 floats
    Ring<2> ra;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
      const Tile w = tile(t);
      float run[SG_OUT], tot[SG_OUT];
#pragma unroll
      for (int q = 0; q < SG_OUT; ++q) run[q] = tot[q] = 0.f;
      for (int kb = 0; kb < nk && ok; ++kb, ra.next()) {
        const int a = ra.s;
        ok = mbar_wait(tfull + 8 * a, ra.ph);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
        for (int q0 = 0; q0 < SG_OUT; q0 += 8) {
          uint32_t r[2][8];  // hi hi, the small products
#pragma unroll
          for (int h = 0; h < 2; ++h)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(r[h][0]), "=r"(r[h][1]), "=r"(r[h][2]), "=r"(r[h][3]), "=r"(r[h][4]), "=r"(r[h][5]),
                           "=r"(r[h][6]), "=r"(r[h][7])
                         : "r"(tw + (uint32_t)((2 * a + h) * SG_BN + q0)));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int u = 0; u < 8; ++u) run[q0 + u] += __uint_as_float(r[0][u]) + __uint_as_float(r[1][u]);
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        mbar_arrive(tempty + 8 * a);
        if ((kb & (SG_RUN - 1)) == SG_RUN - 1 || kb == nk - 1) {
#pragma unroll
          for (int q = 0; q < SG_OUT; ++q) {
            tot[q] += run[q];
            run[q] = 0.f;
          }
        }
      }
      // operands that are not finite, or whose hi part overflowed: the warp looks which of its elements (rare)
      float zero = 0.f;
#pragma unroll
      for (int q = 0; q < SG_OUT; ++q) zero = fmaf(tot[q], 0.f, zero);
      const bool spoiled = __any_sync(0xffffffffu, ok && zero != zero);
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
              const bool mark = out[u] && !(fabsf(v[u].x) <= FLT_MAX && fabsf(v[u].y) <= FLT_MAX);
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
static int split_map(CUtensorMap* tm, const float* ptr, int rows, int K2, long ldk, int batch) {
  auto enc = get_encode();
  if (!enc) return TSVD_ERR_CUDA;
  cuuint64_t dims[3] = {(cuuint64_t)K2, (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)(ldk * 4), (cuuint64_t)(ldk * 4 * rows)};
  cuuint32_t box[3] = {(cuuint32_t)SG_KB, 128, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, (void*)ptr, dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? TSVD_OK : TSVD_ERR_UNSUPPORTED;
}

static long sg_ldk(int K) { return (2L * K + 3) / 4 * 4; }
static size_t sg_slice_bytes(int M, int N, int K) {
  return 8 * (size_t)sg_ldk(K) * (M + 2 * (size_t)N) + Marks<float2>::bytes(M, N, 1);
}
size_t sgemm_tc_bytes(int M, int N, int K, int batch) {
  return std::min<size_t>(sg_slice_bytes(M, N, K) * batch, (size_t)3 << 30) + sg_slice_bytes(M, N, K) + 2048;
}

// Estimated times in microseconds of the two forms: a SIMT tile takes 0.104 (64 x 64) or 0.25 us (128 x
// 64) per term of K and SM, K split as cgemm splits it.  Measured, product with its operand passes: 1024 x
// 1024 x 1024 on 33 slices 5.08 -> 1.56 ms (the product alone 1.23: 230 TFLOP/s), 2048 x 100 x 2048 on
// 17 1230 -> 561 us, 512 x 60 x 512 on 33 109 -> 70.  Error, 2-norm, normal data, K = 97, 512, 1024,
// 2048, 4096: 1.4, 1.4, 1.4, 1.6, 1.8e-7, the SIMT kernels 1.8, 4.0, 2.6, 4.2, 4.5e-7.
bool sgemm_tc_better(const GemmArgs& g, size_t bytes) {
  if (g.K < 1 || g.M < 1 || g.N < 1 || g.K > (1 << 24)) return false;
  const size_t slice = sg_slice_bytes(g.M, g.N, g.K) + 2048;
  if (bytes < slice) return false;
  const double wtiles = (double)cdiv(g.M, 128) * cdiv(g.N, 64) * g.batch;
  const bool wide = g.K >= 1024 || wtiles >= 2 * 152;
  const double stiles = wide ? wtiles : (double)cdiv(g.M, 64) * cdiv(g.N, 64) * g.batch;
  double ks = std::min(16.0, std::max(1.0, std::floor(wide ? (4 * 152 + stiles - 1) / stiles : 2 * 152 / stiles)));
  ks = std::min(ks, std::max(1.0, g.K / 64.0));
  const double simt = 4.0 + (ks > 1.0 ? 3.0 : 0.0) + std::ceil(stiles * ks / 152) * (g.K / ks) * (wide ? 0.25 : 0.104);
  const double tiles = (double)cdiv(g.M, SG_BM) * cdiv(2L * g.N, SG_BN) * g.batch;
  const double tile_us = 3.0 + cdiv(2L * g.K, SG_KB) * 0.55;
  const double pack_us = ((double)slice * 1.4 * g.batch) / 4.0e6;
  const double calls = std::ceil((double)g.batch * slice / (double)bytes);
  return simt > 10.0 * calls + pack_us + std::ceil(tiles / 152.0) * tile_us;
}

int sgemm_tc(const GemmArgs& g, void* ws, size_t bytes, cudaStream_t s) {
  const long ldk = sg_ldk(g.K);
  const int N2 = 2 * g.N;
  const uintptr_t p0 = ((uintptr_t)ws + 255) & ~(uintptr_t)255;
  const size_t off = p0 - (uintptr_t)ws + 1280;  // alignments
  const int nb = bytes < off ? 0 : (int)std::min<size_t>(g.batch, (bytes - off) / sg_slice_bytes(g.M, g.N, g.K));
  if (nb < 1) return TSVD_ERR_WORKSPACE;
  if (g.C == g.A || g.C == g.B) return TSVD_ERR_INVALID_ARG;  // k_redo reads the operands once more
  auto up = [](uintptr_t p) { return (p + 255) & ~(uintptr_t)255; };
  const size_t an = (size_t)nb * g.M * ldk * 4, bn = (size_t)nb * N2 * ldk * 4;
  float* Ah = (float*)p0;
  float* Al = (float*)up(p0 + an);
  float* Bh = (float*)up((uintptr_t)Al + an);
  float* Bl = (float*)up((uintptr_t)Bh + bn);
  const Marks<float2> marks = Marks<float2>::at(up((uintptr_t)Bl + bn), g.M, g.N, nb);
  if (cudaFuncSetAttribute(k_sgemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM) != cudaSuccess) {
    cudaGetLastError();
    return TSVD_ERR_CUDA;
  }
  for (int b0 = 0; b0 < g.batch; b0 += nb) {
    const int n = std::min(nb, g.batch - b0);
    const float2* A = (const float2*)g.A + (long)b0 * g.sA;
    const float2* B = (const float2*)g.B + (long)b0 * g.sB;
    const SplitOp oa{A, g.lda, g.sA, g.M, g.opA == 'H', g.opA == 'H', Ah, Al};
    const SplitOp ob{B, g.ldb, g.sB, g.N, g.opB == 'N', g.opB == 'H', Bh, Bl};
    k_split_pack<<<dim3(oa.blocks(g.K) + ob.blocks(g.K), 1, n), 256, 0, s>>>(oa, ob, g.K, ldk, marks);
    TSVD_LAUNCHED();
    CUtensorMap mah, mal, mbh, mbl;
    TSVD_TRY(split_map(&mah, Ah, g.M, 2 * g.K, ldk, n));
    TSVD_TRY(split_map(&mal, Al, g.M, 2 * g.K, ldk, n));
    TSVD_TRY(split_map(&mbh, Bh, N2, 2 * g.K, ldk, n));
    TSVD_TRY(split_map(&mbl, Bl, N2, 2 * g.K, ldk, n));
    const long tiles = (long)cdiv(N2, SG_BN) * cdiv(g.M, SG_BM) * n;
    float2* Cb = (float2*)g.C + (long)b0 * g.sC;
    k_sgemm_tc<<<(unsigned)std::min<long>(tiles, 152), SG_THREADS, SG_SMEM, s>>>(
        mah, mal, mbh, mbl, marks, Cb, g.ldc, g.sC, g.M, g.N, cdiv(2L * g.K, SG_KB), n, (float)g.alpha,
        g.beta != 0.0);
    TSVD_LAUNCHED();
    TSVD_TRY(redo_marked<float2>(marks, {A, B, g.lda, g.sA, g.ldb, g.sB, g.K, g.opA == 'H', g.opB == 'H'}, Cb,
                                 g.ldc, g.sC, g.M, g.N, n, g.alpha, g.beta != 0.0, false, s));
  }
  return TSVD_OK;
}

}  // namespace tsvd
