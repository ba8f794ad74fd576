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

// largest biased exponent of every row of a stored rows x cols matrix (one warp per row)
__global__ void __launch_bounds__(256) k_dig_expo_rows(const double2* __restrict__ S, long ld, long ss, int rows,
                                                       int cols, int* __restrict__ E) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, b = blockIdx.y;
  if (r >= rows) return;
  const double2* p = S + (long)b * ss + (long)r * ld;
  int e = 1;
#pragma unroll 4
  for (int c = lane; c < cols; c += 32) e = max(e, expo(p[c]));
  e = __reduce_max_sync(0xffffffffu, e);
  if (lane == 0) E[(long)b * rows + r] = e;
}

// the same of every column (E zeroed before; rows in pieces of 64 along blockIdx.y)
__global__ void __launch_bounds__(256) k_dig_expo_cols(const double2* __restrict__ S, long ld, long ss, int rows,
                                                       int cols, int* __restrict__ E) {
  __shared__ int red[8][32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, b = blockIdx.z;
  const int c = blockIdx.x * 32 + tx, r0 = blockIdx.y * 64;
  int e = 1;
  if (c < cols) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = r0 + ty + 8 * i;
      if (r < rows) e = max(e, expo(S[(long)b * ss + (long)r * ld + c]));
    }
  }
  red[ty][tx] = e;
  __syncthreads();
  if (ty == 0 && c < cols) {
#pragma unroll
    for (int i = 1; i < 8; ++i) e = max(e, red[i][tx]);
    atomicMax(E + (long)b * cols + c, e);
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

// One stored complex matrix to digit planes D[(b * 7 + s)][row][2K] (row length ldk elements).
//   TRANS: stored K x rows (read through 32 x 32 tiles), else rows x K;
//   EXPAND: op(B), two rows 2r and 2r + 1 per column r: (yr, -yi) and (yi, yr); else op(A): (ar, ai);
//   conj: the stored matrix enters conjugated.
// Blocks of 32 rows x 32 of K, all along blockIdx.x: rows / 32 passes the 65535 of the other two.
template <bool TRANS, bool EXPAND>
__global__ void __launch_bounds__(256) k_dig_pack(const double2* __restrict__ S, long ld, long ss, int rows, int K,
                                                  bool conj, const int* __restrict__ E, uint32_t* __restrict__ D,
                                                  long ldk) {
  __shared__ double2 t[TRANS ? 32 : 1][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, b = blockIdx.z;
  const int kblocks = (K + 31) / 32, k0 = blockIdx.x % kblocks * 32, r0 = blockIdx.x / kblocks * 32;
  S += (long)b * ss;
  if (TRANS) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = k0 + ty + 8 * i, r = r0 + tx;
      t[ty + 8 * i][tx] = (k < K && r < rows) ? S[(long)k * ld + r] : make_double2(0.0, 0.0);
    }
    __syncthreads();
  }
  const int k = k0 + tx;
  if (k >= K) return;
  const long plane = (long)rows * (EXPAND ? 2 : 1) * (ldk / 2);  // 32-bit words of a digit plane
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + 8 * i;
    if (r >= rows) continue;
    const double2 v = TRANS ? t[tx][ty + 8 * i] : S[(long)r * ld + k];
    const int e = E[(long)b * rows + r];
    const unsigned long long x = biased_digits(v.x, e), y = biased_digits(v.y, e);
    uint32_t* dst = D + (long)b * DG_D * plane + (long)(EXPAND ? 2 * r : r) * (ldk / 2) + k;
    const uint32_t sign = (conj != EXPAND) ? 0x8000u : 0u;  // of the imaginary part in the first row
#pragma unroll
    for (int s = 0; s < DG_D; ++s) {
      const uint32_t re = digit_bf16(x, s), im = digit_bf16(y, s);
      dst[s * plane] = re | ((im ^ sign) << 16);
      if (EXPAND) dst[s * plane + ldk / 2] = (im ^ (sign ^ 0x8000u)) | (re << 16);
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
                                                            const __grid_constant__ DotSrc<double2> src,
                                                            const int* __restrict__ EA, const int* __restrict__ EB,
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
      const int row = w.m0 + (warp & 3) * 32 + lane;
      if (row < M) {
        const int ea = EA[(long)w.bz * M + row];
        double2* crow = C + (long)w.bz * sC + (long)row * ldc;
#pragma unroll
        for (int q = 0; q < DG_OUT; q += 2) {
          const int col = (w.n0 + col0 + q) >> 1;
          if (col < N) {
            const int eb = EB[(long)w.bz * N + col];
            double2 v;
            if (ok && ea < 0x7ff && eb < 0x7ff) {
              const int e = ea + eb + 40 - 2 * 1077;  // the levels carry 256^5 = 2^40
              v = make_double2(fixed_to_double(hi[q], lo[q], e), fixed_to_double(hi[q + 1], lo[q + 1], e));
            } else if (ok && src.A) {  // a row or column holding an infinity or NaN
              v = direct_dot(src, w.bz, row, col);
            } else {  // (or its operand overwritten in place, or a pipeline that gave up)
              v = make_double2(__longlong_as_double(0x7ff8000000000000ll), __longlong_as_double(0x7ff8000000000000ll));
            }
            if (alpha != 1.0) v = cscale(v, alpha);
            if (beta) v = cadd(v, crow[col]);
            crow[col] = v;
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
  return (size_t)DG_D * dg_ldk(K) * 2 * (M + 2 * (size_t)N) + 4 * ((size_t)M + N);
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
  const size_t avail = bytes - (p0 - (uintptr_t)ws) - 1024;
  const int nb = (int)std::min<size_t>(g.batch, avail / dg_slice_bytes(g.M, g.N, g.K));
  if (nb < 1) return TSVD_ERR_WORKSPACE;
  auto up = [](uintptr_t p) { return (p + 255) & ~(uintptr_t)255; };
  uint32_t* DA = (uint32_t*)p0;
  uint32_t* DB = (uint32_t*)up(p0 + (size_t)nb * DG_D * g.M * ldk * 2);
  int* EA = (int*)up((uintptr_t)DB + (size_t)nb * DG_D * N2 * ldk * 2);
  int* EB = EA + (size_t)nb * g.M;
  if (cudaFuncSetAttribute(k_dgemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, DG_SMEM) != cudaSuccess) {
    cudaGetLastError();
    return TSVD_ERR_CUDA;
  }
  for (int b0 = 0; b0 < g.batch; b0 += nb) {
    const int n = std::min(nb, g.batch - b0);
    const bool ta = g.opA == 'H', tb = g.opB == 'N';
    const double2* A = (const double2*)g.A + (long)b0 * g.sA;
    const double2* B = (const double2*)g.B + (long)b0 * g.sB;
    if ((ta || tb) && cudaMemsetAsync(EA, 0, sizeof(int) * (size_t)nb * (g.M + g.N), s) != cudaSuccess)
      return TSVD_ERR_CUDA;
    if (ta) k_dig_expo_cols<<<dim3(cdiv(g.M, 32), cdiv(g.K, 64), n), 256, 0, s>>>(A, g.lda, g.sA, g.K, g.M, EA);
    else k_dig_expo_rows<<<dim3(cdiv(g.M, 8), n), 256, 0, s>>>(A, g.lda, g.sA, g.M, g.K, EA);
    TSVD_LAUNCHED();
    if (tb) k_dig_expo_cols<<<dim3(cdiv(g.N, 32), cdiv(g.K, 64), n), 256, 0, s>>>(B, g.ldb, g.sB, g.K, g.N, EB);
    else k_dig_expo_rows<<<dim3(cdiv(g.N, 8), n), 256, 0, s>>>(B, g.ldb, g.sB, g.N, g.K, EB);
    TSVD_LAUNCHED();
    const dim3 ga(cdiv(g.K, 32) * cdiv(g.M, 32), 1, n), gb(cdiv(g.K, 32) * cdiv(g.N, 32), 1, n);
    if (ta) k_dig_pack<true, false><<<ga, 256, 0, s>>>(A, g.lda, g.sA, g.M, g.K, true, EA, DA, ldk);
    else k_dig_pack<false, false><<<ga, 256, 0, s>>>(A, g.lda, g.sA, g.M, g.K, false, EA, DA, ldk);
    TSVD_LAUNCHED();
    if (tb) k_dig_pack<true, true><<<gb, 256, 0, s>>>(B, g.ldb, g.sB, g.N, g.K, false, EB, DB, ldk);
    else k_dig_pack<false, true><<<gb, 256, 0, s>>>(B, g.ldb, g.sB, g.N, g.K, true, EB, DB, ldk);
    TSVD_LAUNCHED();
    CUtensorMap ma, mb;
    TSVD_TRY(digit_map(&ma, DA, g.M, 2 * g.K, ldk, n * DG_D, DG_BM));
    TSVD_TRY(digit_map(&mb, DB, N2, 2 * g.K, ldk, n * DG_D, DG_BN));
    const long tiles = (long)cdiv(N2, DG_BN) * cdiv(g.M, DG_BM) * n;  // one per CTA where some are skipped
    const unsigned grid = (unsigned)(upper ? tiles : std::min<long>(tiles, 152));
    const DotSrc<double2> src{g.C == g.A || g.C == g.B ? nullptr : A, B, g.lda, g.sA, g.ldb, g.sB, g.K, ta, !tb};
    k_dgemm_tc<<<grid, DG_THREADS, DG_SMEM, s>>>(ma, mb, src, EA, EB, (double2*)g.C + (long)b0 * g.sC, g.ldc, g.sC, g.M,
                                                 g.N, cdiv(2L * g.K, DG_KB), n, g.alpha, g.beta != 0.0, upper ? 1 : 0);
    TSVD_LAUNCHED();
  }
  return TSVD_OK;
}

}  // namespace tsvd
