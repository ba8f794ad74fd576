// dgemm_tc.cu -- FP64 complex GEMM as exact digit products on the BF16 tensor cores.
//
// GB300 has two FP64 multiply-adds per SM and clock, 1/2000 of its BF16 rate, so an
// FP64 product of any size is bound by that pipe.  Here each row of op(A) and each
// column of op(B) is scaled by a power of two to integers of at most 2^55 (the rounding
// of that step, 2^-56 of the row's scale, is the only one before the result)
// and written in seven balanced base-256 digits, X = sum_s d_s 256^(6-s), -128 <=
// d_s <= 128, each exact in BF16.  The digit pairs (s, t) with s + t <= 7 (34 of
// 49; the rest lie below 2^-62 of the leading product) are multiplied on tcgen05.
// Pairs with equal s + t have equal weight and share one accumulator, so a tile
// has eight FP32 accumulators of 64 columns, all 512 columns of TMEM; the digits of
// B lie one after another in shared memory, so one instruction multiplies a digit
// of A with several digits of B into neighbouring accumulators.  Every product is
// an integer below 2^14: after 192 terms of K the accumulators (sums below 2^24 for
// the five leading levels whatever the data) are read, converted and added up in two
// 64-bit integers per element, and the result is rounded once to FP64.  Error, 2-norm,
// against exact dot products of normal data: 5e-17 to 7e-17 for K = 97 .. 2048 (FP64
// multiply-adds: 3.1e-16 to 3.6e-16), of data graded over twelve decades 1.5e-16 to
// 2.7e-16 (2.3e-16 to 4.0e-16).
//
// A complex product is the real product of the interleaved rows of op(A) with the
// expanded real form of op(B) (rows 2n and 2n + 1 per column n, as in tc_gemm.cu).
//
// Bound: the tensor cores, 34 BF16 products per multiply-add (56 TFLOP/s of FP64
// work at the measured BF16 rate, against 1.1 on the FP64 units), and for thin
// products the two passes over the operands (largest exponents, digits).  1024 x 1024
// x 1024 on 5 slices: 36.7 -> 1.26 ms, 512 x 60 x 512 on 33: 4.09 -> 0.28 ms, of which
// the product itself about 0.09.
#include <cuda_bf16.h>

#include <cmath>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_common.cuh"
#include "tc_redo.cuh"

namespace tsvd {

constexpr int DG_D = 7;        // digits
constexpr int DG_L = 8;        // levels s + t = 0 .. 7
constexpr int DG_BM = 128;     // complex rows per tile
constexpr int DG_BN = 64;      // real columns per tile (32 complex)
constexpr int DG_KB = 32;      // K per stage: rows of 64 bytes, 64-byte swizzle
constexpr int DG_STAGES = 2;
constexpr int DG_CHUNK = 6;    // stages between two readings of the accumulators (192 terms)
constexpr int DG_A_BYTES = DG_D * DG_BM * DG_KB * 2, DG_B_BYTES = DG_D * DG_BN * DG_KB * 2;
constexpr int DG_STAGE_BYTES = DG_A_BYTES + DG_B_BYTES;
constexpr int DG_SMEM = DG_STAGES * DG_STAGE_BYTES + 1024 + 256;
// threads that read the accumulators (16 warps: 5.7 ms for the products of a 512 x 512 x 64 T-SVD, 6.3 with 8,
// whose sums took all registers), then one TMA and one MMA warp
constexpr int DG_DRAIN = 512;
constexpr int DG_THREADS = DG_DRAIN + 64;
constexpr int DG_OUT = DG_BN / 4;  // real columns per draining thread
static_assert(DG_SMEM <= 227 * 1024, "two stages must fit a CTA's shared memory");
static_assert(DG_L * DG_BN == 512, "the accumulators take the whole of TMEM");
static_assert(5 * (1 << 14) * DG_CHUNK * DG_KB < (1 << 24), "sums of the five leading levels stay exact");

// ---------------------------------------------------------------------------
// operands
// ---------------------------------------------------------------------------
__device__ __forceinline__ int expo(double2 v) {
  const int a = (__double2hiint(v.x) >> 20) & 0x7ff, b = (__double2hiint(v.y) >> 20) & 0x7ff;
  return max(max(a, b), 1);  // subnormals scale as 2^-1022
}

// one operand as its passes see it: rows (columns of op(B)) of K elements
struct DigOp {
  const double2* S;
  long ld, ss;
  int rows;
  bool trans;  // stored K x rows, else rows x K
  bool conj;   // enters conjugated
  int* E;      // largest biased exponent of each row (zeroed before where trans), [batch][rows]
  uint32_t* D; // digit planes, [batch][7][rows, or 2 rows for op(B)][ldk]
  __host__ __device__ unsigned expo_blocks(int K) const {
    return trans ? (unsigned)((rows + 31) / 32) * ((K + 63) / 64) : (unsigned)((rows + 7) / 8);
  }
  __host__ __device__ unsigned pack_blocks(int K) const { return (unsigned)((rows + 31) / 32) * ((K + 31) / 32); }
};

// The largest exponents of both operands' rows: of rows as stored by a warp each, of stored columns by 32 columns x 64 of K
// per block.  Also clears the marks.
__global__ void __launch_bounds__(256) k_dig_expo(const DigOp A, const DigOp B, int K, const Marks<double2> marks) {
  __shared__ int red[8][32];
  const bool first = blockIdx.x < A.expo_blocks(K);
  const DigOp& o = first ? A : B;
  const int blk = first ? blockIdx.x : blockIdx.x - A.expo_blocks(K), b = blockIdx.z;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  marks.clear(((long)b * gridDim.x + blockIdx.x) * 256 + threadIdx.x, (long)gridDim.z * gridDim.x * 256);
  const double2* S = o.S + (long)b * o.ss;
  int e = 1;
  if (!o.trans) {
    const int r = blk * 8 + ty;
    if (r >= o.rows) return;
    const double2* p = S + (long)r * o.ld;
#pragma unroll 4
    for (int k = tx; k < K; k += 32) e = max(e, expo(p[k]));
    e = __reduce_max_sync(0xffffffffu, e);
    if (tx == 0) o.E[(long)b * o.rows + r] = e;
    return;
  }
  const int kb = (K + 63) / 64, r = blk / kb * 32 + tx, k0 = blk % kb * 64;
  if (r < o.rows) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = k0 + ty + 8 * i;
      if (k < K) e = max(e, expo(S[(long)k * o.ld + r]));
    }
  }
  red[ty][tx] = e;
  __syncthreads();
  if (ty == 0 && r < o.rows) {
#pragma unroll
    for (int i = 1; i < 8; ++i) e = max(e, red[i][tx]);
    atomicMax(o.E + (long)b * o.rows + r, e);
  }
}

// x as an integer in units of 2^(E - 1077), |X| <= 2^55 (round half away from zero), its bytes
// biased by 128: digit s is byte 6 - s minus 128 (the leading one with its carry: at most 128)
__device__ __forceinline__ unsigned long long biased_digits(double x, int E) {
  const unsigned long long u = __double_as_longlong(x);
  const int ex = (int)(u >> 52) & 0x7ff;
  unsigned long long m = u & 0xfffffffffffffull;
  m |= ex ? (1ull << 52) : 0;
  const int sh = E - max(ex, 1) - 2;  // >= -2
  if (sh < 0) m <<= -sh;
  else if (sh > 54) m = 0;
  else if (sh > 0) m = (m + (1ull << (sh - 1))) >> sh;
  return 0x80808080808080ull + ((long long)u < 0 ? 0ull - m : m);
}
// the BF16 bits of byte - 128
__device__ __forceinline__ uint32_t digit_bf16(unsigned long long y, int s) {
  const uint32_t byte = (uint32_t)(y >> (8 * (6 - s))) & (s == 0 ? 0x1ffu : 0xffu);
  return __float_as_uint(__uint_as_float(0x4B000000u | byte) - (8388608.0f + 128.0f)) >> 16;
}

// Both operands to digit planes, 32 rows x 32 of K per block (all along blockIdx.x: rows / 32 passes the 65535 of
// the other dimensions); stored columns are read through a 32 x 32 tile.  op(A): rows (ar, ai); op(B):
// two rows 2r and 2r + 1 per column r, (yr, -yi) and (yi, yr).
__global__ void __launch_bounds__(256) k_dig_pack(const DigOp A, const DigOp B, int K, long ldk) {
  __shared__ double2 t[32][33];
  const bool first = blockIdx.x < A.pack_blocks(K);
  const DigOp& o = first ? A : B;
  const int blk = first ? blockIdx.x : blockIdx.x - A.pack_blocks(K), b = blockIdx.z;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int kblocks = (K + 31) / 32, k0 = blk % kblocks * 32, r0 = blk / kblocks * 32, rows = o.rows;
  const double2* S = o.S + (long)b * o.ss;
  if (o.trans) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = k0 + ty + 8 * i, r = r0 + tx;
      t[ty + 8 * i][tx] = (k < K && r < rows) ? S[(long)k * o.ld + r] : make_double2(0.0, 0.0);
    }
    __syncthreads();
  }
  const int k = k0 + tx;
  if (k >= K) return;
  const long plane = (long)rows * (first ? 1 : 2) * (ldk / 2);  // 32-bit words of a digit plane
  const uint32_t sign = (o.conj == first) ? 0x8000u : 0u;  // of the imaginary part in the first row
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + 8 * i;
    if (r >= rows) continue;
    const double2 v = o.trans ? t[tx][ty + 8 * i] : S[(long)r * o.ld + k];
    const int e = o.E[(long)b * rows + r];
    const unsigned long long x = biased_digits(v.x, e), y = biased_digits(v.y, e);
    uint32_t* dst = o.D + (long)b * DG_D * plane + (long)(first ? r : 2 * r) * (ldk / 2) + k;
#pragma unroll
    for (int s = 0; s < DG_D; ++s) {
      const uint32_t re = digit_bf16(x, s), im = digit_bf16(y, s);
      dst[s * plane] = re | ((im ^ sign) << 16);
      if (!first) dst[s * plane + ldk / 2] = (im ^ (sign ^ 0x8000u)) | (re << 16);
    }
  }
}

// ---------------------------------------------------------------------------
// the product
// ---------------------------------------------------------------------------
// (hi 2^32 + lo) 2^e rounded to nearest, in integer arithmetic (FP64 conversions run on the FP64 pipe)
__device__ __forceinline__ double fixed_to_double(long long hi, long long lo, int e) {
  __int128 v = ((__int128)hi << 32) + lo;
  if (v == 0) return 0.0;
  const bool neg = v < 0;
  unsigned __int128 a = neg ? (unsigned __int128)(-v) : (unsigned __int128)v;
  const unsigned long long ah = (unsigned long long)(a >> 64);
  const int lz = ah ? __clzll(ah) : 64 + __clzll((unsigned long long)a);
  a <<= lz;
  const unsigned long long top = (unsigned long long)(a >> 64);
  const unsigned rem = (unsigned)((top & 0x7ff) << 1) | ((unsigned long long)a != 0 ? 1u : 0u);
  unsigned long long m = top >> 11;
  m += (rem > 0x800u || (rem == 0x800u && (m & 1))) ? 1 : 0;
  const int be = 127 - lz + e + 1023;  // biased exponent of the leading bit
  if (be >= 1 && be < 2046) {
    const unsigned long long bits = ((unsigned long long)be << 52) + (m - (1ull << 52));
    return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0)));
  }
  return scalbn(neg ? -(double)m : (double)m, be - 1023 - 52);
}

__global__ void __launch_bounds__(DG_THREADS, 1) k_dgemm_tc(const __grid_constant__ CUtensorMap tmA,
                                                            const __grid_constant__ CUtensorMap tmB,
                                                            const int* __restrict__ EA, const int* __restrict__ EB,
                                                            const __grid_constant__ Marks<double2> marks,
                                                            double2* __restrict__ C, long ldc, long sC, int M, int N,
                                                            int nk, int batch, double alpha, int beta, int upper) {
  extern __shared__ unsigned char dg_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tn = (2 * N + DG_BN - 1) / DG_BN, tm = (M + DG_BM - 1) / DG_BM;
  const int tiles = tn * tm * batch;  // at least one element each: within an int
  struct Tile {
    int n0, m0, bz;
    bool skip;
  };
  auto tile = [&](int t) {  // columns fastest: neighbouring CTAs share rows of A
    const int r = t / tn;
    Tile w{(t % tn) * DG_BN, (r % tm) * DG_BM, r / tm, false};
    w.skip = upper && w.n0 / 2 + DG_BN / 2 <= w.m0;  // Hermitian product: mirrored afterwards
    return w;
  };
  if (upper && (int)gridDim.x == tiles && tile(blockIdx.x).skip) return;
  unsigned char* base = (unsigned char*)(((uintptr_t)dg_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(base + DG_STAGES * DG_STAGE_BYTES);  // full[S], empty[S], tfull, tempty
  uint32_t* tslot = (uint32_t*)(bars + 2 * DG_STAGES + 2);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + DG_STAGES);
  const uint32_t tfull = smem_u32(bars + 2 * DG_STAGES), tempty = tfull + 8;
  if (tid == 0) {
    for (int s = 0; s < DG_STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, DG_DRAIN);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tslot;
  const int chunks = (nk + DG_CHUNK - 1) / DG_CHUNK;

  // stages and readings are counted through all tiles of the CTA, so loads and products of the next
  // tile run under the rounding and writing of this one
  if (tid == DG_DRAIN) {  // TMA producer
    Ring<DG_STAGES> r;
    long filled = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
      const Tile w = tile(t);
      if (w.skip) continue;
      for (int kb = 0; kb < nk; ++kb, ++filled, r.next()) {
        const int s = r.s;
        if (!mbar_wait(empty0 + 8 * s, r.ph ^ 1)) {
          ok = false;
          break;
        }
        const uint32_t dst = smem_u32(base + s * DG_STAGE_BYTES);
        mbar_expect_tx(full0 + 8 * s, DG_STAGE_BYTES);
        tma_load_3d(dst, &tmA, kb * DG_KB, w.m0, w.bz * DG_D, full0 + 8 * s);
        tma_load_3d(dst + DG_A_BYTES, &tmB, kb * DG_KB, w.n0, w.bz * DG_D, full0 + 8 * s);
      }
    }
    ring_drain(r, filled, full0);
  } else if (tid == DG_DRAIN + 32) {  // MMA issuer
    const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(DG_BM >> 4) << 24);  // FP32 += BF16 BF16^T
    Ring<DG_STAGES> r;
    Ring<1> ra;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
      if (tile(t).skip) continue;
      for (int c = 0; ok && c < chunks; ++c, ra.next()) {
        if (!mbar_wait(tempty, ra.ph ^ 1)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        const int k1 = min(nk, (c + 1) * DG_CHUNK);
        for (int kb = c * DG_CHUNK; kb < k1; ++kb, r.next()) {
          const int s = r.s;
          if (!mbar_wait(full0 + 8 * s, r.ph)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t sa = smem_u32(base + s * DG_STAGE_BYTES), sb = sa + DG_A_BYTES;
#pragma unroll
          for (int kk = 0; kk < DG_KB / 16; ++kk) {
            const bool first = kb == c * DG_CHUNK && kk == 0;
            // digit i of A with the digits j of B, as many as 256 columns per instruction; level i + j
            auto mul = [&](int i, int j, int nj, bool acc) {
              mma_issue<true>(tmem + (uint32_t)((i + j) * DG_BN),
                              smem_desc_sw64(sa + i * (DG_BM * DG_KB * 2)) + 2 * kk,
                              smem_desc_sw64(sb + j * (DG_BN * DG_KB * 2)) + 2 * kk,
                              idesc0 | ((uint32_t)(nj * DG_BN >> 3) << 17), acc ? 1u : 0u);
            };
            mul(0, 0, 4, !first);
            mul(0, 4, 3, !first);
            mul(1, 0, 4, true);
            mul(1, 4, 2, true);
            mul(1, 6, 1, !first);  // level 7 begins here
            mul(2, 0, 4, true);
            mul(2, 4, 2, true);
            mul(3, 0, 4, true);
            mul(3, 4, 1, true);
            mul(4, 0, 4, true);
            mul(5, 0, 3, true);
            mul(6, 0, 2, true);
          }
          mma_commit(empty0 + 8 * s);
        }
        if (ok) mma_commit(tfull);
      }
    }
  } else if (warp < DG_DRAIN / 32) {
    const int col0 = (warp >> 2) * DG_OUT;
    const uint32_t tw = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)col0;
    Ring<1> ra;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
      if (tile(t).skip) continue;
      long long hi[DG_OUT], lo[DG_OUT];
#pragma unroll
      for (int q = 0; q < DG_OUT; ++q) hi[q] = lo[q] = 0;
      for (int c = 0; ok && c < chunks; ++c, ra.next()) {
        ok = mbar_wait(tfull, ra.ph);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
        for (int q0 = 0; q0 < DG_OUT; q0 += 4) {
          uint32_t r[DG_L][4];
#pragma unroll
          for (int l = 0; l < DG_L; ++l)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(r[l][0]), "=r"(r[l][1]), "=r"(r[l][2]), "=r"(r[l][3])
                         : "r"(tw + (uint32_t)(l * DG_BN + q0)));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            int v[DG_L];
#pragma unroll
            for (int l = 0; l < DG_L; ++l) v[l] = __float2int_rn(__uint_as_float(r[l][u]));
            long long h = hi[q0 + u], lw = lo[q0 + u];
            h += (long long)v[0] * (1 << 24);
            h += (long long)v[1] * (1 << 16);
            h += (long long)v[2] * (1 << 8);
            h += (long long)v[3];
            lw += (long long)v[4] * (1 << 24);
            lw += (long long)v[5] * (1 << 16);
            lw += (long long)v[6] * (1 << 8);
            lw += (long long)v[7];
            hi[q0 + u] = h;
            lo[q0 + u] = lw;
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        mbar_arrive(tempty);
      }
      const Tile w = tile(t);
      const int row0 = w.m0 + (warp & 3) * 32, row = row0 + lane;
      if (row0 >= M) continue;
      const int ea = row < M ? EA[(long)w.bz * M + row] : 0;
      double2* crow = C + (long)w.bz * sC + (long)row * ldc;
#pragma unroll
      for (int q = 0; q < DG_OUT; q += 2) {
        const int col = (w.n0 + col0 + q) >> 1;
        if (col >= N) continue;  // the same for the whole warp
        const int eb = EB[(long)w.bz * N + col];
        // a row or column holding an infinity or NaN: its digits say nothing, left to k_redo
        const bool mark = ok && row < M && (ea >= 0x7ff || eb >= 0x7ff);
        marks.put(M, N, w.bz, row0, col, mark, row, col, lane);
        if (mark || row >= M) continue;
        const int e = ea + eb + 40 - 2 * 1077;  // the levels carry 256^5 = 2^40
        double2 v = make_double2(fixed_to_double(hi[q], lo[q], e), fixed_to_double(hi[q + 1], lo[q + 1], e));
        if (!ok) v = make_double2(__longlong_as_double(0x7ff8000000000000ll), __longlong_as_double(0x7ff8000000000000ll));
        if (alpha != 1.0) v = cscale(v, alpha);
        if (beta) v = cadd(v, crow[col]);
        crow[col] = v;
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
static int digit_map(CUtensorMap* tm, const void* ptr, int rows, int K2, long ldk, int planes, int box_rows) {
  auto enc = get_encode();
  if (!enc) return TSVD_ERR_CUDA;
  cuuint64_t dims[3] = {(cuuint64_t)K2, (cuuint64_t)rows, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)(ldk * 2), (cuuint64_t)(ldk * 2 * rows)};
  cuuint32_t box[3] = {(cuuint32_t)DG_KB, (cuuint32_t)box_rows, (cuuint32_t)DG_D};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)ptr, dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? TSVD_OK : TSVD_ERR_UNSUPPORTED;
}

static long dg_ldk(int K) { return (2L * K + 7) / 8 * 8; }
static size_t dg_slice_bytes(int M, int N, int K) {
  return (size_t)DG_D * dg_ldk(K) * 2 * (M + 2 * (size_t)N) + 4 * ((size_t)M + N) + Marks<double2>::bytes(M, N, 1);
}
size_t dgemm_tc_bytes(int M, int N, int K, int batch) {
  return std::min<size_t>(dg_slice_bytes(M, N, K) * batch, (size_t)3 << 30) + dg_slice_bytes(M, N, K) + 2048;
}

// Estimated times in microseconds of the two forms; the digit form from about 2e7 multiply-adds on
// (128 x 64 x 128 on 5 slices: 265 us on the FP64 units, 78 us here; 64 x 15 x 64 on 9 slices: 19 us
// there, about 25 us of launches here).
bool dgemm_tc_better(const GemmArgs& g, size_t bytes) {
  if (g.K < 1 || g.M < 1 || g.N < 1 || g.K > (1 << 20)) return false;
  const size_t slice = dg_slice_bytes(g.M, g.N, g.K) + 2048;
  if (bytes < slice) return false;
  const double simt = 4.0 * g.M * g.N * (double)g.K * g.batch / 5.0e5;
  const double tiles = (double)cdiv(g.M, DG_BM) * cdiv(2L * g.N, DG_BN) * g.batch;
  const double tile_us = 2.0 + (cdiv(2L * g.K, DG_KB) * 1.5 + cdiv(2L * g.K, DG_KB * DG_CHUNK) * 1.5);
  const double pack_us = ((double)slice * 1.3 * g.batch) / 3.0e6;
  const double calls = std::ceil((double)g.batch * slice / (double)bytes);
  return simt > 25.0 * calls + pack_us + std::ceil(tiles / 152.0) * tile_us;
}

int dgemm_tc(const GemmArgs& g, void* ws, size_t bytes, cudaStream_t s, bool upper) {
  const long ldk = dg_ldk(g.K);
  const int N2 = 2 * g.N;
  // slices per pass: the digits of both operands in the scratch
  uintptr_t p0 = ((uintptr_t)ws + 255) & ~(uintptr_t)255;
  const size_t off = p0 - (uintptr_t)ws + 1024;  // alignments
  const int nb = bytes < off ? 0 : (int)std::min<size_t>(g.batch, (bytes - off) / dg_slice_bytes(g.M, g.N, g.K));
  if (nb < 1) return TSVD_ERR_WORKSPACE;
  if (g.C == g.A || g.C == g.B) return TSVD_ERR_INVALID_ARG;  // k_redo reads the operands once more
  auto up = [](uintptr_t p) { return (p + 255) & ~(uintptr_t)255; };
  uint32_t* DA = (uint32_t*)p0;
  uint32_t* DB = (uint32_t*)up(p0 + (size_t)nb * DG_D * g.M * ldk * 2);
  int* EA = (int*)up((uintptr_t)DB + (size_t)nb * DG_D * N2 * ldk * 2);
  int* EB = EA + (size_t)nb * g.M;
  const Marks<double2> marks = Marks<double2>::at(up((uintptr_t)(EB + (size_t)nb * g.N)), g.M, g.N, nb);
  if (cudaFuncSetAttribute(k_dgemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, DG_SMEM) != cudaSuccess) {
    cudaGetLastError();
    return TSVD_ERR_CUDA;
  }
  for (int b0 = 0; b0 < g.batch; b0 += nb) {
    const int n = std::min(nb, g.batch - b0);
    const bool ta = g.opA == 'H', tb = g.opB == 'N';
    const double2* A = (const double2*)g.A + (long)b0 * g.sA;
    const double2* B = (const double2*)g.B + (long)b0 * g.sB;
    const DigOp oa{A, g.lda, g.sA, g.M, ta, ta, EA, DA}, ob{B, g.ldb, g.sB, g.N, tb, !tb, EB, DB};
    if ((ta || tb) && cudaMemsetAsync(EA, 0, sizeof(int) * (size_t)nb * (g.M + g.N), s) != cudaSuccess)
      return TSVD_ERR_CUDA;
    k_dig_expo<<<dim3(oa.expo_blocks(g.K) + ob.expo_blocks(g.K), 1, n), 256, 0, s>>>(oa, ob, g.K, marks);
    TSVD_LAUNCHED();
    k_dig_pack<<<dim3(oa.pack_blocks(g.K) + ob.pack_blocks(g.K), 1, n), 256, 0, s>>>(oa, ob, g.K, ldk);
    TSVD_LAUNCHED();
    CUtensorMap ma, mb;
    TSVD_TRY(digit_map(&ma, DA, g.M, 2 * g.K, ldk, n * DG_D, DG_BM));
    TSVD_TRY(digit_map(&mb, DB, N2, 2 * g.K, ldk, n * DG_D, DG_BN));
    const long tiles = (long)cdiv(N2, DG_BN) * cdiv(g.M, DG_BM) * n;  // one per CTA where some are skipped
    const unsigned grid = (unsigned)(upper ? tiles : std::min<long>(tiles, 152));
    double2* Cb = (double2*)g.C + (long)b0 * g.sC;
    k_dgemm_tc<<<grid, DG_THREADS, DG_SMEM, s>>>(ma, mb, EA, EB, marks, Cb, g.ldc, g.sC, g.M, g.N,
                                                 cdiv(2L * g.K, DG_KB), n, g.alpha, g.beta != 0.0, upper ? 1 : 0);
    TSVD_LAUNCHED();
    TSVD_TRY(redo_marked<double2>(marks, {A, B, g.lda, g.sA, g.ldb, g.sB, g.K, ta, !tb}, Cb, g.ldc, g.sC, g.M, g.N, n,
                                  g.alpha, g.beta != 0.0, upper, s));
  }
  return TSVD_OK;
}

}  // namespace tsvd
