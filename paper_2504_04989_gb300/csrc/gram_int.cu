// gram_int.cu -- the Hermitian Gram G = C C^H of the small SVD of Alg. 2
// (T-SVD(C) through the eigenpairs of C C^H) on the FP32 path, summed exactly
// in integer arithmetic.
//
// C^H (n2 x m per slice) holds FP32 data.  Each column i is written as
// 2^(e_i - B) times a vector of integers of at most B+1 bits (one power of two
// per column, e_i the exponent of the column's largest component), which moves
// every entry by at most 2^(e_i - B - 1): a perturbation of C of the size of its
// own FP32 rounding.  The Gram of the scaled integers is then exact in 64-bit
// integer multiply-adds, and G_ij = 2^(e_i + e_j - 2B) sum_l conj(q_li) q_lj is
// rounded once, to FP64.  An FP32 Gram would put rounding errors of the order
// eps32 ||C||^2 on the small eigenvalues sigma_i^2 the method keeps; this form
// keeps the error at the level of a perturbation of C itself, as the FP64 Gram
// does, while running on the integer pipe instead of GB300's narrow FP64 unit.
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_common.cuh"

namespace tsvd {

// mantissa bits B: 2 products per component and n2 terms must stay below 2^63
static int gram_bits(int n2) {
  int lg = 0;
  while ((1L << lg) < n2) ++lg;
  return std::min(23, (61 - lg) / 2);
}

// columns of one slice in tiles of 32, 8 row groups per column: exponent of the
// column's largest |component| (max over the groups in shared memory), then
// the scaled integers (round to nearest even)
__global__ void __launch_bounds__(256) k_gram_quantize(const float2* __restrict__ CH, long ldc, long sC, int n2,
                                                       int m, int B, int2* __restrict__ Q, int* __restrict__ colexp) {
  __shared__ float smx[8][32];
  const int cx = threadIdx.x & 31, ry = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + cx;
  const int k = blockIdx.y;
  const bool ok = i < m;
  const float2* src = CH + (long)k * sC + i;
  float mx = 0.0f;
  if (ok)
#pragma unroll 8
    for (int l = ry; l < n2; l += 8) {
      const float2 x = src[(long)l * ldc];
      mx = fmaxf(mx, fmaxf(fabsf(x.x), fabsf(x.y)));
    }
  smx[ry][cx] = mx;
  __syncthreads();
  float cm = 0.0f;
#pragma unroll
  for (int r = 0; r < 8; ++r) cm = fmaxf(cm, smx[r][cx]);
  if (!ok) return;
  int e = 0;
  if (cm > 0.0f) frexpf(cm, &e);  // cm < 2^e
  if (ry == 0) colexp[(long)k * m + i] = e;
  if (!Q) return;  // the exponents only (the digit form quantizes as it writes its digits)
  int2* dst = Q + (long)k * n2 * m + i;
  for (int l = ry; l < n2; l += 8) {
    const float2 x = src[(long)l * ldc];
    dst[(long)l * m] = make_int2((int)rintf(ldexpf(x.x, B - e)), (int)rintf(ldexpf(x.y, B - e)));
  }
}

// ---------------------------------------------------------------------------
// The same exact Gram on the BF16 tensor cores.  Every integer q (|q| <= 2^B,
// B <= 23) is written in three balanced base-256 digits, q = sum_s d_s 256^(2-s),
// -128 <= d_s <= 128: exact in BF16.  Row 2i of digit plane s holds digit s of the
// real parts of column i of C^H along l, row 2i + 1 that of the imaginary parts.
// A tile of 128 x 64 rows multiplies all nine digit pairs (s, t); those of equal
// s + t have equal weight and share one FP32 accumulator, five accumulators of 64
// columns in TMEM, and as the three digits of the second operand lie one after
// another in shared memory, one instruction multiplies a digit of the first with all
// three into neighbouring accumulators.  A digit product is at most 2^14 and at most
// three share an accumulator, so after 320 terms the sums are below 2^24 and exact;
// they are read then and added up in one 64-bit integer per element, modulo 2^64,
// which holds the result.  With S the integer sums of the real rows,
//   sum_l conj(q_li) q_lj = S[2i][2j] + S[2i+1][2j+1] + i (S[2i][2j+1] - S[2i+1][2j]),
// two neighbouring lanes of the tile, and it is rounded once, as above: G is bitwise
// the integer kernel's.
//
// Bound: the operand tiles from L2, 72 KB of digits per 128 x 64 x 64 step (62 bytes per
// clock and SM at the full tensor rate), and the reading of the accumulators, which
// is not overlapped.  480 x 480 from 2048 rows on 65 slices: 1.43 ms with its two passes
// over C^H (four digits, 16 products of a real GEMM written to memory and added up from
// there: 4.2 ms); 300 x 300 from 512 rows on 33 slices 0.69 -> 0.15 ms.
// ---------------------------------------------------------------------------
constexpr int GS_D = 3, GS_L = 5;  // digits, levels
constexpr int GS_BM = 128, GS_BN = 64, GS_KB = 64;  // rows of 128 bytes per stage, 128-byte swizzle
constexpr int GS_STAGES = 3;
constexpr int GS_CHUNK = 5;  // stages between two readings of the accumulators (320 terms)
constexpr int GS_A_BYTES = GS_D * GS_BM * GS_KB * 2, GS_B_BYTES = GS_D * GS_BN * GS_KB * 2;
constexpr int GS_STAGE_BYTES = GS_A_BYTES + GS_B_BYTES;
constexpr int GS_SMEM = GS_STAGES * GS_STAGE_BYTES + 1024 + 256;
constexpr int GS_DRAIN = 256;  // threads that read the accumulators (8 warps), then one TMA and one MMA warp
constexpr int GS_THREADS = GS_DRAIN + 64;
constexpr int GS_OUT = GS_BN / 2;  // real columns per draining thread
static_assert(GS_SMEM <= 227 * 1024, "the stages must fit a CTA's shared memory");
static_assert(GS_L * GS_BN <= 512, "the accumulators must fit TMEM");
static_assert(GS_D * GS_BN <= 256, "one instruction takes all digits of the second operand");
static_assert(3 * (1 << 14) * GS_CHUNK * GS_KB < (1 << 24), "the accumulated sums stay exact");

// the BF16 bits of digit s, from y = q + 0x808080 (digit s is byte 2 - s minus 128, the leading one
// with its carry)
__device__ __forceinline__ uint32_t gram_digit(uint32_t y, int s) {
  const uint32_t byte = (y >> (8 * (2 - s))) & (s == 0 ? 0x1ffu : 0xffu);
  return __float_as_uint(__uint_as_float(0x4B000000u | byte) - (8388608.0f + 128.0f)) >> 16;
}

// digit planes D[(b * 3 + s)][2 m][ldd] of the quantized C^H: 64 rows x 32 columns of C^H per
// block, transposed through shared memory so that the rows of D are written along l, two
// entries (one 32-bit word) per thread
__global__ void __launch_bounds__(256) k_gram_digits(const float2* __restrict__ CH, long ldc, long sC, int n2, int m,
                                                     int B, const int* __restrict__ colexp,
                                                     uint32_t* __restrict__ D, long ldd) {
  __shared__ int2 t[64][33];
  const int b = blockIdx.z, i0 = blockIdx.x * 32, l0 = blockIdx.y * 64;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int sh = (i0 + tx < m) ? B - colexp[(long)b * m + i0 + tx] : 0;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int rr = ty + 8 * r, l = l0 + rr, i = i0 + tx;
    int2 q = make_int2(0, 0);
    if (l < n2 && i < m) {
      const float2 x = CH[(long)b * sC + (long)l * ldc + i];
      q = make_int2((int)rintf(ldexpf(x.x, sh)), (int)rintf(ldexpf(x.y, sh)));
    }
    t[rr][tx] = q;
  }
  __syncthreads();
  const int l = l0 + 2 * tx;
  if (l >= n2) return;
  const long w = ldd / 2, plane = 2L * m * w;  // 32-bit words
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int cc = ty + 8 * r, i = i0 + cc;
    if (i >= m) continue;
    const int2 q0 = t[2 * tx][cc], q1 = t[2 * tx + 1][cc];
    uint32_t* dst = D + (long)b * GS_D * plane + 2L * i * w + l / 2;
#pragma unroll
    for (int part = 0; part < 2; ++part) {
      const uint32_t y0 = (uint32_t)(part ? q0.y : q0.x) + 0x808080u, y1 = (uint32_t)(part ? q1.y : q1.x) + 0x808080u;
#pragma unroll
      for (int s = 0; s < GS_D; ++s) dst[s * plane + part * w] = gram_digit(y0, s) | (gram_digit(y1, s) << 16);
    }
  }
}

// v 2^e rounded to nearest, ldexp((double)v, e) in integer arithmetic: those run on the FP64 pipe, which
// took some 7 us of every tile (480 x 480 on 65 slices: 1303 -> 1127 us)
__device__ __forceinline__ double int_to_double(long long v, int e) {
  if (v == 0) return 0.0;
  const bool neg = v < 0;
  unsigned long long a = neg ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int lz = __clzll((long long)a);
  a <<= lz;
  const unsigned rem = (unsigned)a & 0x7ffu;
  unsigned long long m = a >> 11;
  m += (rem > 0x400u || (rem == 0x400u && (m & 1))) ? 1 : 0;
  const int be = 63 - lz + e + 1023;  // biased exponent of the leading bit
  if (be >= 1 && be < 2046) {
    const unsigned long long bits = ((unsigned long long)be << 52) + (m - (1ull << 52));
    return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0)));
  }
  return ldexp((double)v, e);
}

__global__ void __launch_bounds__(GS_THREADS, 1) k_gram_tc(const __grid_constant__ CUtensorMap tmA,
                                                           const __grid_constant__ CUtensorMap tmB,
                                                           const int* __restrict__ colexp, int n2, int m, int B,
                                                           double2* __restrict__ G, long ldg, long sG,
                                                           int* __restrict__ err) {
  extern __shared__ unsigned char gs_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n0 = blockIdx.x * GS_BN, m0 = blockIdx.y * GS_BM, bz = blockIdx.z;
  if (n0 + GS_BN <= m0) return;  // wholly below the diagonal: mirrored from above
  unsigned char* base = (unsigned char*)(((uintptr_t)gs_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(base + GS_STAGES * GS_STAGE_BYTES);  // full[S], empty[S], tfull, tempty
  uint32_t* tslot = (uint32_t*)(bars + 2 * GS_STAGES + 2);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + GS_STAGES);
  const uint32_t tfull = smem_u32(bars + 2 * GS_STAGES), tempty = tfull + 8;
  if (tid == 0) {
    for (int s = 0; s < GS_STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, GS_DRAIN);
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
  const int nk = (n2 + GS_KB - 1) / GS_KB;
  const int chunks = (nk + GS_CHUNK - 1) / GS_CHUNK;

  if (tid == GS_DRAIN) {  // TMA producer
    int issued = 0;
    bool ok = true;
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % GS_STAGES, round = kb / GS_STAGES;
      if (round > 0 && !mbar_wait(empty0 + 8 * s, (round - 1) & 1)) {
        ok = false;
        break;
      }
      const uint32_t dst = smem_u32(base + s * GS_STAGE_BYTES);
      mbar_expect_tx(full0 + 8 * s, GS_STAGE_BYTES);
      tma_load_3d(dst, &tmA, kb * GS_KB, m0, bz * GS_D, full0 + 8 * s);
      tma_load_3d(dst + GS_A_BYTES, &tmB, kb * GS_KB, n0, bz * GS_D, full0 + 8 * s);
      issued = kb + 1;
    }
    if (!ok) {  // copies in flight land before the CTA gives its shared memory back
      for (int kb = (issued > GS_STAGES ? issued - GS_STAGES : 0); kb < issued; ++kb)
        mbar_wait(full0 + 8 * (kb % GS_STAGES), (kb / GS_STAGES) & 1);
    }
  } else if (tid == GS_DRAIN + 32) {  // MMA issuer: digit i of A with the three of B, levels i .. i + 2
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GS_D * GS_BN >> 3) << 17) |
                           ((uint32_t)(GS_BM >> 4) << 24);  // FP32 += BF16 BF16^T
    const uint32_t idesc1 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GS_BN >> 3) << 17) |
                            ((uint32_t)(GS_BM >> 4) << 24);
    bool ok = true;
    for (int c = 0; ok && c < chunks; ++c) {
      if (c > 0 && !mbar_wait(tempty, (c - 1) & 1)) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
      const int k1 = min(nk, (c + 1) * GS_CHUNK);
      for (int kb = c * GS_CHUNK; kb < k1; ++kb) {
        const int s = kb % GS_STAGES;
        if (!mbar_wait(full0 + 8 * s, (kb / GS_STAGES) & 1)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t sa = smem_u32(base + s * GS_STAGE_BYTES), sb = sa + GS_A_BYTES;
#pragma unroll
        for (int kk = 0; kk < GS_KB / 16; ++kk) {
          const uint64_t b0 = smem_desc_sw128(sb) + 2 * kk;
          if (kb == c * GS_CHUNK && kk == 0) {  // the first products of a level overwrite what it held
            mma_issue<true>(tmem, smem_desc_sw128(sa), b0, idesc, 0u);
#pragma unroll
            for (int i = 1; i < GS_D; ++i) {
              const uint64_t ai = smem_desc_sw128(sa + i * (GS_BM * GS_KB * 2));
#pragma unroll
              for (int j = 0; j < GS_D; ++j)
                mma_issue<true>(tmem + (uint32_t)((i + j) * GS_BN), ai,
                                smem_desc_sw128(sb + j * (GS_BN * GS_KB * 2)), idesc1, j == GS_D - 1 ? 0u : 1u);
            }
          } else {
#pragma unroll
            for (int i = 0; i < GS_D; ++i)
              mma_issue<true>(tmem + (uint32_t)(i * GS_BN), smem_desc_sw128(sa + i * (GS_BM * GS_KB * 2)) + 2 * kk, b0,
                              idesc, 1u);
          }
        }
        mma_commit(empty0 + 8 * s);
      }
      if (ok) mma_commit(tfull);
    }
  } else if (warp < GS_DRAIN / 32) {
    const int row = m0 + (warp & 3) * 32 + lane;
    const int col0 = (warp >> 2) * GS_OUT;
    const uint32_t tw = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)col0;
    long long acc[GS_OUT];
#pragma unroll
    for (int q = 0; q < GS_OUT; ++q) acc[q] = 0;
    bool ok = true;
    for (int c = 0; c < chunks; ++c) {
      ok = mbar_wait(tfull, c & 1);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
      for (int q0 = 0; q0 < GS_OUT; q0 += 4) {
        uint32_t r[GS_L][4];
#pragma unroll
        for (int l = 0; l < GS_L; ++l)
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(r[l][0]), "=r"(r[l][1]), "=r"(r[l][2]), "=r"(r[l][3])
                       : "r"(tw + (uint32_t)(l * GS_BN + q0)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          long long h = acc[q0 + u];
#pragma unroll
          for (int l = 0; l < GS_L; ++l)
            h += (long long)__float2int_rn(__uint_as_float(r[l][u])) * (1LL << (8 * (GS_L - 1 - l)));
          acc[q0 + u] = h;
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      mbar_arrive(tempty);
    }
    if (!ok) {
      if (lane == 0) atomicExch(err, 1);
    } else {
      // rows 2i and 2i + 1 are neighbouring lanes; the even one writes G_ij, the odd one G_ji
      const int i = row >> 1;
      const bool odd = row & 1;
      const int ei = i < m ? colexp[(long)bz * m + i] : 0;
      double2* Gb = G + (long)bz * sG;
#pragma unroll
      for (int q = 0; q < GS_OUT; q += 2) {
        const int j = (n0 + col0 + q) >> 1;
        const long long o0 = __shfl_xor_sync(0xffffffffu, acc[q], 1), o1 = __shfl_xor_sync(0xffffffffu, acc[q + 1], 1);
        if (i >= m || j >= m || i > j || (odd && i == j)) continue;
        const long long re = odd ? acc[q + 1] + o0 : acc[q] + o1, im = odd ? o1 - acc[q] : acc[q + 1] - o0;
        const int sc = ei + colexp[(long)bz * m + j] - 2 * B;
        const double2 g = make_double2(int_to_double(re, sc), int_to_double(im, sc));
        if (odd) Gb[(long)j * ldg + i] = make_double2(g.x, -g.y);
        else Gb[(long)i * ldg + j] = g;
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

constexpr int GI_TILE = 64;
constexpr int GI_KC = 16;

// Upper-triangle tiles (ti <= tj) of G per slice; each thread 4 x 4 entries
// with 64-bit accumulators; the tile and its conjugate transpose are written.
__global__ void __launch_bounds__(256) k_gram_int(const int2* __restrict__ Q, const int* __restrict__ colexp, int n2,
                                                  int m, int B, double2* __restrict__ G, long ldg, long sG) {
  __shared__ int2 Qa[GI_KC][GI_TILE];
  __shared__ int2 Qb[GI_KC][GI_TILE];
  const int nt = (m + GI_TILE - 1) / GI_TILE;
  int ti = 0, rem = blockIdx.x;
  while (rem >= nt - ti) {
    rem -= nt - ti;
    ++ti;
  }
  const int tj = ti + rem;
  const int k = blockIdx.y;
  const int i0 = ti * GI_TILE, j0 = tj * GI_TILE;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int2* Qk = Q + (long)k * n2 * m;
  long long re[4][4], im[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) re[a][b] = im[a][b] = 0;
  for (int l0 = 0; l0 < n2; l0 += GI_KC) {
    for (int e = threadIdx.x; e < GI_KC * GI_TILE; e += 256) {
      const int ll = e / GI_TILE, c = e % GI_TILE, l = l0 + ll;
      const bool lok = l < n2;
      Qa[ll][c] = (lok && i0 + c < m) ? Qk[(long)l * m + i0 + c] : make_int2(0, 0);
      Qb[ll][c] = (lok && j0 + c < m) ? Qk[(long)l * m + j0 + c] : make_int2(0, 0);
    }
    __syncthreads();
#pragma unroll 4
    for (int ll = 0; ll < GI_KC; ++ll) {
      int2 a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = Qa[ll][ty + 16 * u];
#pragma unroll
      for (int u = 0; u < 4; ++u) b[u] = Qb[ll][tx + 16 * u];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int nai = -a[u].y;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          // conj(a) b = (ar br + ai bi) + i (ar bi - ai br)
          re[u][v] += (long long)a[u].x * b[v].x;
          re[u][v] += (long long)a[u].y * b[v].y;
          im[u][v] += (long long)a[u].x * b[v].y;
          im[u][v] += (long long)nai * b[v].x;
        }
      }
    }
    __syncthreads();
  }
  const int* ek = colexp + (long)k * m;
  double2* Gk = G + (long)k * sG;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = i0 + ty + 16 * u;
    if (i >= m) continue;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int j = j0 + tx + 16 * v;
      if (j >= m) continue;
      const int sc = ek[i] + ek[j] - 2 * B;
      const double2 g = make_double2(ldexp((double)re[u][v], sc), ldexp((double)im[u][v], sc));
      Gk[(long)i * ldg + j] = g;
      if (ti != tj) Gk[(long)j * ldg + i] = make_double2(g.x, -g.y);
    }
  }
}

int gram_int_fp32(const float2* CH, long ldc, long sC, int n2, int m, int batch, int2* Q, int* colexp, double2* G,
                  long ldg, long sG, cudaStream_t s) {
  if (n2 <= 0 || m <= 0 || batch <= 0) return TSVD_OK;
  if (batch > 65535) return TSVD_ERR_UNSUPPORTED;
  const int B = gram_bits(n2);
  k_gram_quantize<<<dim3(cdiv(m, 32), batch), 256, 0, s>>>(CH, ldc, sC, n2, m, B, Q, colexp);
  TSVD_LAUNCHED();
  const int nt = cdiv(m, GI_TILE);
  k_gram_int<<<dim3(nt * (nt + 1) / 2, batch), 256, 0, s>>>(Q, colexp, n2, m, B, G, ldg, sG);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

// the digit form (n2: 64 rows per block of the grid's second dimension)
bool gram_sliced_ok(int n2, int m) { return n2 >= 1 && n2 <= (1 << 20) && m >= 1 && 2L * m <= 65535; }
static long gram_sliced_ldd(int n2) { return (n2 + 7L) / 8 * 8; }
size_t gram_sliced_bytes(int n2, int m, int batch) {
  return (size_t)batch * GS_D * 2 * m * gram_sliced_ldd(n2) * sizeof(__nv_bfloat16) + 512;
}

static int gram_map(CUtensorMap* tm, const void* ptr, int n2, int rows, long ldd, int planes, int box_rows) {
  auto enc = get_encode();
  if (!enc) return TSVD_ERR_CUDA;
  cuuint64_t dims[3] = {(cuuint64_t)n2, (cuuint64_t)rows, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)(ldd * 2), (cuuint64_t)(ldd * 2 * rows)};
  cuuint32_t box[3] = {(cuuint32_t)GS_KB, (cuuint32_t)box_rows, (cuuint32_t)GS_D};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)ptr, dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? TSVD_OK : TSVD_ERR_UNSUPPORTED;
}

int gram_sliced_fp32(const float2* CH, long ldc, long sC, int n2, int m, int batch, int* colexp, void* ws,
                     double2* G, long ldg, long sG, int* err, cudaStream_t s) {
  if (n2 <= 0 || m <= 0 || batch <= 0) return TSVD_OK;
  if (batch > 65535 || !gram_sliced_ok(n2, m)) return TSVD_ERR_UNSUPPORTED;
  const int B = gram_bits(n2);
  const long ldd = gram_sliced_ldd(n2);
  uint32_t* D = (uint32_t*)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
  k_gram_quantize<<<dim3(cdiv(m, 32), batch), 256, 0, s>>>(CH, ldc, sC, n2, m, B, nullptr, colexp);
  TSVD_LAUNCHED();
  k_gram_digits<<<dim3(cdiv(m, 32), cdiv(n2, 64), batch), 256, 0, s>>>(CH, ldc, sC, n2, m, B, colexp, D, ldd);
  TSVD_LAUNCHED();
  CUtensorMap ma, mb;
  TSVD_TRY(gram_map(&ma, D, n2, 2 * m, ldd, batch * GS_D, GS_BM));
  TSVD_TRY(gram_map(&mb, D, n2, 2 * m, ldd, batch * GS_D, GS_BN));
  if (cudaFuncSetAttribute(k_gram_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, GS_SMEM) != cudaSuccess) {
    cudaGetLastError();
    return TSVD_ERR_CUDA;
  }
  k_gram_tc<<<dim3(cdiv(2 * m, GS_BN), cdiv(2 * m, GS_BM), batch), GS_THREADS, GS_SMEM, s>>>(ma, mb, colexp, n2, m, B,
                                                                                            G, ldg, sG, err);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

}  // namespace tsvd
