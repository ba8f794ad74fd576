// dgemm_tc.cu -- FP64 complex GEMM as exact digit products on the BF16 tensor cores, a form of the
// error-free splitting of a matrix product into integer slices (Ozaki, Ogita, Oishi and Rump 2012).
//
// GB300 has two FP64 multiply-adds per SM and clock, 1/2000 of its BF16 rate, so an
// FP64 product of any size is bound by that pipe.  Here each row of op(A) and each
// column of op(B) is scaled by a power of two to integers below 2^62 and written in
// eight balanced base-256 digits, X = sum_s d_s 256^(7-s), -128 <= d_s <= 128 (the leading
// one at most 64), each exact in BF16.  An entry within 2^-9 of its row's largest is held
// exactly, one 2^-k below it with 62 - k bits.  The digit pairs (s, t) with s + t <= 7 (36 of
// 64; the rest lie below 2^-60 of the scales) are multiplied on tcgen05.
// Pairs with equal s + t have equal weight and share one accumulator, so a tile
// has eight FP32 accumulators of 64 columns, all 512 columns of TMEM; the digits of
// B lie one after another in shared memory, so one instruction multiplies a digit
// of A with several digits of B into neighbouring accumulators.  Every product is
// an integer of at most 2^14: after 192 terms of K the accumulators (sums below 2^24 for
// the six leading levels whatever the data) are read, converted and added up in two
// 64-bit integers per element, and the result is rounded once to FP64.
//
// Uneven scales.  FP64 multiply-adds keep 53 bits of every product; digits keep what is large in its
// row or column, and lose a small entry of A that meets a large one of B.  So (1) an exact power of two per k
// makes the columns of op(A) (or the rows of op(B), whichever a sample shows to be the more even within) equally
// large and gives their scales to the other operand, whose columns then take their own: features times their weights, W
// times R^-1, C^H times U_c and U S times V^H become even; (2) every element shows that its terms are not
// small next to its scales, or is left to k_redo, which adds them up in FP64:
//   |C_ij| is at least 2^-7 of (scale of row i) (scale of column j), or
//   the entry of row i that meets the largest one of column j is within 2^-5 of its scale, or the other way round, or
//   the entries within 2^-5 and within 2^-8 of their scales that meet one another add up to 2^-7: bits of the two
//   levels, counted word by word until they do.  This shows it for the products of orthonormal columns, which cancel
//   to zeros, where the columns are concentrated and have their largest entries in different rows (of a
//   2048 x 2048 x 128 T-SVD's Q^H Q and Q^H W the two tests above leave 7 to 25 % of the elements, this one 1 %).
// Each says that sum |a||b| is at least 2^-7 of the scales, against an error of at most about 2^-59 of them per
// term: 2.4 times the worst case of FP64 multiply-adds, 2 K u sum |a||b|, where those are only just met.  Errors as
// measured stand at dgemm_tc_better.
//
// A complex product is the real product of the interleaved rows of op(A) with the
// expanded real form of op(B) (rows 2n and 2n + 1 per column n, as in tc_gemm.cu).
//
// Bound: the tensor cores, 36 BF16 products per multiply-add (53 TFLOP/s of FP64
// work at the measured BF16 rate, against 1.1 on the FP64 units), and for thin
// products the three passes over the operands (sampled scales, largest exponents, digits).
#include <cuda_bf16.h>

#include <cmath>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_common.cuh"
#include "tc_redo.cuh"

namespace tsvd {

constexpr int DG_D = 8;        // digits
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
static_assert(5 * (1 << 14) * DG_CHUNK * DG_KB < (1 << 24), "sums of the six leading levels stay exact");
constexpr int DG_OFF = 8192;     // added to exponents, so that 0 says: a row without an entry
constexpr int DG_INF = 1 << 20;  // a row with an infinity or NaN

// ---------------------------------------------------------------------------
// operands
// ---------------------------------------------------------------------------
// largest biased exponent of the two parts, subnormals as 2^-1022; 0: zero, 0x7ff: not finite
__device__ __forceinline__ int expo(double2 v) {
  const unsigned long long x = __double_as_longlong(v.x) << 1, y = __double_as_longlong(v.y) << 1;
  const int e = max((int)(x >> 53), (int)(y >> 53));
  return (x | y) == 0 ? 0 : max(e, 1);
}

// one operand as its passes see it: rows (columns of op(B)) of K elements
struct DigOp {
  const double2* S;
  long ld, ss;
  int rows;
  bool trans;  // stored K x rows, else rows x K
  bool conj;   // enters conjugated
  int sign;    // its entries of k take sign * shift[k] to their exponents
  // [batch][rows] 2^32 (bound of the row's exponents + DG_OFF, 0, DG_INF) + the k of the largest entry
  unsigned long long* top;
  uint2* near;              // [batch][rows][K / 32] which entries are within 2^-5 and within 2^-8 of that bound
  uint32_t* D;              // digit planes, [batch][8][rows, or 2 rows for op(B)][ldk]
  __host__ __device__ unsigned expo_blocks(int K) const {
    return trans ? (unsigned)((rows + 31) / 32) * ((K + 63) / 64) : (unsigned)((rows + 7) / 8);
  }
  __host__ __device__ unsigned pack_blocks(int K) const { return (unsigned)((rows + 31) / 32) * ((K + 31) / 32); }
};

// Of 32 entries of op(A)(:, k) and of op(B)(k, :), spread over it, the mean exponent (0 where all are zero) and how
// far the largest lies above it, zeros counted as 64 below: 32 k per block, 8 of its threads on each.  Also zeroes what
// the next pass takes maxima into.
__global__ void __launch_bounds__(256) k_dig_sample(const DigOp A, const DigOp B, int K, float4* __restrict__ stat) {
  __shared__ int red[2][3][8][32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, b = blockIdx.z, k = blockIdx.x * 32 + tx;
  int e[2][4];
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const DigOp& o = w ? B : A;
    const double2* S = o.S + (long)b * o.ss;
    const int n = min(o.rows, 32);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      // pairs of neighbours where there are enough: a sector of stored columns holds both
      const int q = ty + 8 * u, r = o.rows < 64 ? (int)((long)q * o.rows / n) : (int)((long)(q >> 1) * o.rows / 16) + (q & 1);
      e[w][u] = (q < n && k < K) ? expo(o.trans ? S[(long)k * o.ld + r] : S[(long)r * o.ld + k]) : 0;
    }
  }
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const DigOp& o = w ? B : A;
    for (int r = blockIdx.x * 256 + threadIdx.x; r < o.rows; r += gridDim.x * 256) o.top[(long)b * o.rows + r] = 0;
    int sum = 0, cnt = 0, big = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int x = e[w][u] < 0x7ff ? e[w][u] : 0;
      sum += x;
      cnt += x > 0;
      big = max(big, x);
    }
    red[w][0][ty][tx] = sum;
    red[w][1][ty][tx] = cnt;
    red[w][2][ty][tx] = big;
  }
  __syncthreads();
  if (ty >= 2 || k >= K) return;
  int sum = 0, cnt = 0, big = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    sum += red[ty][0][q][tx];
    cnt += red[ty][1][q][tx];
    big = max(big, red[ty][2][q][tx]);
  }
  const int n = min(ty ? B.rows : A.rows, 32);
  const float mean = (float)sum / (float)max(cnt, 1);
  float* out = (float*)(stat + (long)b * K + k) + ty;
  out[0] = mean;
  out[2] = cnt ? ((float)big - mean) + 64.f * (float)(n - cnt) / (float)n : 64.f;
}

// The power of two that op(A)(:, k) takes over from op(B)(k, :): what brings the mean exponent of the more even
// operand's column or row to that of 32 k spread over K, if it is off by more than 1.25 (a sample of evenly scaled
// data stays below, and an entry more or less does not change it); where that is all zero, what brings the other's
// there.  A sample that misleads costs time, not accuracy.
struct DigShift {
  const float4* stat;
  float ra, rb;
  bool byA;
  __device__ DigShift(const float4* t, int b, int K) : stat(t + (long)b * K) {  // by whole warps
    const int lane = threadIdx.x & 31;
    const float4 v = stat[(long)lane * K / 32];
    const int na = __popc(__ballot_sync(0xffffffffu, v.x > 0.f)), nb = __popc(__ballot_sync(0xffffffffu, v.y > 0.f));
    float s[3] = {v.x, v.y, v.z - v.w};
#pragma unroll
    for (int q = 0; q < 3; ++q)
      for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
    ra = s[0] / (float)max(na, 1);
    rb = s[1] / (float)max(nb, 1);
    byA = s[2] <= 16.f;  // of 32: B only where it is plainly the more even
  }
  __device__ int operator()(int k) const {
    const float4 v = stat[k];
    const bool a = v.x > 0.f && (byA || v.y <= 0.f);
    const float t = a ? ra - v.x : v.y > 0.f ? v.y - rb : 0.f;
    return fabsf(t) <= 1.25f ? 0 : (int)rintf(t);
  }
};

// The largest shifted exponents of both operands' rows: of rows as stored by a warp each, of stored columns by 32
// columns x 64 of K per block.  Also clears the marks.
__global__ void __launch_bounds__(256) k_dig_expo(const DigOp A, const DigOp B, int K, const float4* __restrict__ stat,
                                                  const Marks<double2> marks) {
  __shared__ unsigned long long red[8][32];
  const bool first = blockIdx.x < A.expo_blocks(K);
  const DigOp& o = first ? A : B;
  const int blk = first ? blockIdx.x : blockIdx.x - A.expo_blocks(K), b = blockIdx.z;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  marks.clear(((long)b * gridDim.x + blockIdx.x) * 256 + threadIdx.x, (long)gridDim.z * gridDim.x * 256);
  const double2* S = o.S + (long)b * o.ss;
  const DigShift shift(stat, b, K);
  int e = 0, ke = 0;
  auto take = [&](double2 v, int k) {
    const int x = expo(v), l = x == 0 ? 0 : x == 0x7ff ? DG_INF : x + o.sign * shift(k) + DG_OFF;
    if (l > e) {
      e = l;
      ke = k;
    }
  };
  if (!o.trans) {
    const int r = blk * 8 + ty;
    if (r >= o.rows) return;
    const double2* p = S + (long)r * o.ld;
#pragma unroll 4
    for (int k = tx; k < K; k += 32) take(p[k], k);
    const int m = __reduce_max_sync(0xffffffffu, e);
    const int km = __reduce_max_sync(0xffffffffu, e == m ? ke : 0);
    if (tx == 0) o.top[(long)b * o.rows + r] = ((unsigned long long)m << 32) + km;
    return;
  }
  const int kb = (K + 63) / 64, r = blk / kb * 32 + tx, k0 = blk % kb * 64;
  if (r < o.rows) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = k0 + ty + 8 * i;
      if (k < K) take(S[(long)k * o.ld + r], k);
    }
  }
  red[ty][tx] = ((unsigned long long)e << 32) + ke;
  __syncthreads();
  if (ty == 0 && r < o.rows) {
    unsigned long long m = red[0][tx];
#pragma unroll
    for (int i = 1; i < 8; ++i) m = max(m, red[i][tx]);
    if (m >> 32) atomicMax(o.top + (long)b * o.rows + r, m);
  }
}

// x 2^shift as an integer in units of 2^(E - 1084), below 2^62 (round half away from zero); E without DG_OFF and
// less the shift
__device__ __forceinline__ long long digit_int(double x, int E) {
  const unsigned long long u = __double_as_longlong(x);
  const int ex = (int)(u >> 52) & 0x7ff;
  unsigned long long m = u & 0xfffffffffffffull;
  m |= ex ? (1ull << 52) : 0;
  const int sh = E - max(ex, 1) - 9;  // >= -9 for every entry but 0
  if (sh < 0) m <<= min(-sh, 9);
  else if (sh > 54) m = 0;
  else if (sh > 0) m = (m + (1ull << (sh - 1))) >> sh;
  return (long long)u < 0 ? -(long long)m : (long long)m;
}
// the BF16 bits of digit s, from y = X + 0x8080808080808080 (digit s is byte 7 - s minus 128)
__device__ __forceinline__ uint32_t digit_bf16(unsigned long long y, int s) {
  const uint32_t byte = (uint32_t)(y >> (8 * (7 - s))) & 0xffu;
  return __float_as_uint(__uint_as_float(0x4B000000u | byte) - (8388608.0f + 128.0f)) >> 16;
}

// Both operands to digit planes, 32 rows x 32 of K per block (all along blockIdx.x: rows / 32 passes the 65535 of
// the other dimensions); stored columns are read through a 32 x 32 tile.  op(A): rows (ar, ai); op(B):
// two rows 2r and 2r + 1 per column r, (yr, -yi) and (yi, yr).  Notes which entries are near their row's scale.
__global__ void __launch_bounds__(256) k_dig_pack(const DigOp A, const DigOp B, int K, long ldk,
                                                  const float4* __restrict__ stat) {
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
  const bool in = k < K;
  const DigShift shift(stat, b, K);
  const int sk = in ? o.sign * shift(k) : 0;
  const long plane = (long)rows * (first ? 1 : 2) * (ldk / 2);  // 32-bit words of a digit plane
  const uint32_t sign = (o.conj == first) ? 0x8000u : 0u;  // of the imaginary part in the first row
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + 8 * i;  // the same for the whole warp
    if (r >= rows) break;
    const long br = (long)b * rows + r;
    const int e = (int)(o.top[br] >> 32) - DG_OFF - sk;
    double2 v = make_double2(0.0, 0.0);
    if (in) v = o.trans ? t[tx][ty + 8 * i] : S[(long)r * o.ld + k];
    const long long X = digit_int(v.x, e), Y = digit_int(v.y, e);
    const long long big = max(llabs(X), llabs(Y));
    const uint2 near =
        make_uint2(__ballot_sync(0xffffffffu, big >= 1ll << 57), __ballot_sync(0xffffffffu, big >= 1ll << 54));
    if (tx == 0) o.near[br * kblocks + blk % kblocks] = near;
    if (!in) continue;
    const unsigned long long x = 0x8080808080808080ull + X, y = 0x8080808080808080ull + Y;
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
                                                            const unsigned long long* __restrict__ topA,
                                                            const unsigned long long* __restrict__ topB,
                                                            const uint2* __restrict__ nearA,
                                                            const uint2* __restrict__ nearB,
                                                            const __grid_constant__ Marks<double2> marks,
                                                            double2* __restrict__ C, long ldc, long sC, int M, int N,
                                                            int K, int batch, double alpha, int beta, int upper,
                                                            TcOpts st) {
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
  auto wait = [&](uint32_t bar, uint32_t parity) { return !st.expire && mbar_wait(bar, parity); };
  const int nk = (2 * K + DG_KB - 1) / DG_KB, chunks = (nk + DG_CHUNK - 1) / DG_CHUNK;

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
        if (!wait(empty0 + 8 * s, r.ph ^ 1)) {
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
        if (!wait(tempty, ra.ph ^ 1)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        const int k1 = min(nk, (c + 1) * DG_CHUNK);
        for (int kb = c * DG_CHUNK; kb < k1; ++kb, r.next()) {
          const int s = r.s;
          if (!wait(full0 + 8 * s, r.ph)) {
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
            mul(0, 4, 4, !first);
            mul(1, 0, 4, true);
            mul(1, 4, 3, true);
            mul(2, 0, 4, true);
            mul(2, 4, 2, true);
            mul(3, 0, 4, true);
            mul(3, 4, 1, true);
            mul(4, 0, 4, true);
            mul(5, 0, 3, true);
            mul(6, 0, 2, true);
            mul(7, 0, 1, true);
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
        ok = wait(tfull, ra.ph);
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
      if (!ok && lane == 0 && st.err) atomicExch(st.err, 1);
      const Tile w = tile(t);
      const int row0 = w.m0 + (warp & 3) * 32, row = row0 + lane;
      if (row0 >= M) continue;
      const long ra = (long)w.bz * M + min(row, M - 1);
      const unsigned long long ta = topA[ra];
      const int ea = (int)(ta >> 32);
      double2* crow = C + (long)w.bz * sC + (long)row * ldc;
#pragma unroll
      for (int q = 0; q < DG_OUT; q += 2) {
        const int col = (w.n0 + col0 + q) >> 1;
        if (col >= N) continue;  // the same for the whole warp
        const long rb = (long)w.bz * N + col;
        const unsigned long long tb = topB[rb];
        const int eb = (int)(tb >> 32);
        // left to k_redo: an operand that is not finite, or terms that may be small next to the scales
        auto large = [](long long h, long long l) { return llabs(h + (l >> 32)) >= 1ll << 29; };  // 2^-7 of the scales
        bool mark = ok && row < M && min(ea, eb) > 0 && !large(hi[q], lo[q]) && !large(hi[q + 1], lo[q + 1]);
        if (mark) {
          const int ka = (int)(uint32_t)ta, kb = (int)(uint32_t)tb, kw = (K + 31) / 32;
          const uint2 *na = nearA + ra * kw, *nb = nearB + rb * kw;
          mark = !((na[kb / 32].x >> (kb & 31) | nb[ka / 32].x >> (ka & 31)) & 1u);
          if (mark) {
            // each pair is worth the product of its levels, 2^-5 = 2^-8 (1 + 7): in units of 2^-16
            int sum = 0;
#pragma unroll 4
            for (int w = 0; w < kw && sum < 512; ++w) {
              const uint2 x = na[w], y = nb[w];
              sum += __popc(x.y & y.y) + 7 * (__popc(x.x & y.y) + __popc(x.y & y.x)) + 49 * __popc(x.x & y.x);
            }
            mark = sum < 512;
          }
        }
        mark |= ok && row < M && max(ea, eb) >= DG_INF;
        marks.put(M, N, w.bz, row0, col, mark, row, col, lane);
        if (mark || row >= M) continue;
        const int e = ea + eb - 2 * DG_OFF + 56 - 2 * 1084;  // the levels carry 256^7 = 2^56
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
  return (size_t)DG_D * dg_ldk(K) * 2 * (M + 2 * (size_t)N) + 8 * (1 + (size_t)((K + 31) / 32)) * ((size_t)M + N) +
         16 * (size_t)K + Marks<double2>::bytes(M, N, 1);
}
size_t dgemm_tc_bytes(int M, int N, int K, int batch) {
  return std::min<size_t>(dg_slice_bytes(M, N, K) * batch, (size_t)3 << 30) + dg_slice_bytes(M, N, K) + 2048;
}

// Estimated times in microseconds of the two forms; the digit form from about 2e7 multiply-adds on
// (128 x 64 x 128 on 5 slices, just below: 74 us on the FP64 units, 78 us here; 64 x 15 x 64 on 9 slices:
// 19 us there, about 25 us of launches here).  With its passes 1024 x 1024 x 1024 on 5 slices takes
// 1240 us (the product alone 1066), 512 x 60 x 512 on 33 slices 312 (160).
// Error, 2-norm, and the largest of an element in u sum |a||b|, FP64 multiply-adds (GemmCfg<double2>) in brackets:
// normal data, K = 16: 4.7e-17, 1.5 (1.4e-16, 4.4), 97: 4.7e-17, 0.5 (3.3e-16, 4.5), 2048: 4.7e-17, 0.1 (4.0e-16,
// 0.6); every entry over twelve decades of its own 1.5e-16, 7.8 (2.6e-16, 12); columns of A over eight decades
// 5.0e-17, 1.0 (3.6e-16, 8.3); columns of A and rows of B against each other over 3, 6, 12, 17 decades 4.8e-17, 0.4
// (2.8e-16, 1.8) each.
bool dgemm_tc_better(const GemmArgs& g, size_t bytes) {
  if (g.K < 1 || g.M < 1 || g.N < 1 || g.K > (1 << 20)) return false;
  const size_t slice = dg_slice_bytes(g.M, g.N, g.K) + 2048;
  if (bytes < slice) return false;
  const double simt = 4.0 * g.M * g.N * (double)g.K * g.batch / 5.0e5;
  const double tiles = (double)cdiv(g.M, DG_BM) * cdiv(2L * g.N, DG_BN) * g.batch;
  const double tile_us = 2.0 + (cdiv(2L * g.K, DG_KB) * 1.5 + cdiv(2L * g.K, DG_KB * DG_CHUNK) * 1.5);
  const double pack_us = ((double)slice * 1.3 * g.batch) / 3.0e6;
  const double calls = std::ceil((double)g.batch * slice / (double)bytes);
  return simt > 25.0 * calls + pack_us + std::ceil(tiles / SMS) * tile_us;
}

int dgemm_tc(const GemmArgs& g, void* ws, size_t bytes, cudaStream_t s, bool upper, TcOpts st) {
  const long ldk = dg_ldk(g.K);
  const int N2 = 2 * g.N;
  // slices per pass: the digits of both operands in the scratch
  uintptr_t p0 = ((uintptr_t)ws + 255) & ~(uintptr_t)255;
  const size_t off = p0 - (uintptr_t)ws + 1536;  // alignments
  const int nb = bytes < off ? 0 : (int)std::min<size_t>(g.batch, (bytes - off) / dg_slice_bytes(g.M, g.N, g.K));
  if (nb < 1) return TSVD_ERR_WORKSPACE;
  if (g.C == g.A || g.C == g.B) return TSVD_ERR_INVALID_ARG;  // k_redo reads the operands once more
  auto up = [](uintptr_t p) { return (p + 255) & ~(uintptr_t)255; };
  uint32_t* DA = (uint32_t*)p0;
  uint32_t* DB = (uint32_t*)up(p0 + (size_t)nb * DG_D * g.M * ldk * 2);
  float4* stat = (float4*)up((uintptr_t)DB + (size_t)nb * DG_D * N2 * ldk * 2);
  unsigned long long* topA = (unsigned long long*)(stat + (size_t)nb * g.K);
  unsigned long long* topB = topA + (size_t)nb * g.M;
  const size_t kw = cdiv(g.K, 32);
  uint2* nearA = (uint2*)(topB + (size_t)nb * g.N);
  uint2* nearB = nearA + (size_t)nb * g.M * kw;
  const Marks<double2> marks = Marks<double2>::at(up((uintptr_t)(nearB + (size_t)nb * g.N * kw)), g.M, g.N, nb);
  if (cudaFuncSetAttribute(k_dgemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, DG_SMEM) != cudaSuccess) {
    cudaGetLastError();
    return TSVD_ERR_CUDA;
  }
  for (int b0 = 0; b0 < g.batch; b0 += nb) {
    const int n = std::min(nb, g.batch - b0);
    const bool ta = g.opA == 'H', tb = g.opB == 'N';
    const double2* A = (const double2*)g.A + (long)b0 * g.sA;
    const double2* B = (const double2*)g.B + (long)b0 * g.sB;
    const DigOp oa{A, g.lda, g.sA, g.M, ta, ta, 1, topA, nearA, DA};
    const DigOp ob{B, g.ldb, g.sB, g.N, tb, !tb, -1, topB, nearB, DB};
    k_dig_sample<<<dim3(cdiv(g.K, 32), 1, n), 256, 0, s>>>(oa, ob, g.K, stat);
    TSVD_LAUNCHED();
    k_dig_expo<<<dim3(oa.expo_blocks(g.K) + ob.expo_blocks(g.K), 1, n), 256, 0, s>>>(oa, ob, g.K, stat, marks);
    TSVD_LAUNCHED();
    k_dig_pack<<<dim3(oa.pack_blocks(g.K) + ob.pack_blocks(g.K), 1, n), 256, 0, s>>>(oa, ob, g.K, ldk, stat);
    TSVD_LAUNCHED();
    CUtensorMap ma, mb;
    TSVD_TRY(digit_map(&ma, DA, g.M, 2 * g.K, ldk, n * DG_D, DG_BM));
    TSVD_TRY(digit_map(&mb, DB, N2, 2 * g.K, ldk, n * DG_D, DG_BN));
    const long tiles = (long)cdiv(N2, DG_BN) * cdiv(g.M, DG_BM) * n;  // one per CTA where some are skipped
    const unsigned grid = (unsigned)(upper ? tiles : std::min<long>(tiles, SMS));
    double2* Cb = (double2*)g.C + (long)b0 * g.sC;
    k_dgemm_tc<<<grid, DG_THREADS, DG_SMEM, s>>>(ma, mb, topA, topB, nearA, nearB, marks, Cb, g.ldc, g.sC, g.M, g.N,
                                                 g.K, n, g.alpha, g.beta != 0.0, upper ? 1 : 0, st);
    TSVD_LAUNCHED();
    TSVD_TRY(redo_marked<double2>(marks, {A, B, g.lda, g.sA, g.ldb, g.sB, g.K, ta, !tb}, Cb, g.ldc, g.sC, g.M, g.N, n,
                                  g.alpha, g.beta != 0.0, upper, s));
  }
  return TSVD_OK;
}

}  // namespace tsvd
