// tc_redo.cuh -- the elements that a tensor-core product leaves out, computed directly.
//
// k_dgemm_tc and k_sgemm_tc mark the elements that their form cannot give: a bit for each, a list
// of them as far as it reaches, and their number.  k_redo runs behind the product and computes these from
// the operands as stored, so that the product's pipeline never waits for such sums (a thread of its
// readers took 0.4 ms for 1024 terms, and the waits give up after a second).  Few elements are taken from the
// list, a warp each with its lanes along K, spread over the GPU; where there are more than the list
// holds, the tiles with marks are computed as k_cgemm does.  Without marks it reads one word.
// t-product of 512 x 512 x 512, n3 = 16, against sums by the product's own readers: FP32 (finite data: 106 us) one
// row not finite 695 -> 153 us, every row 6212 -> 748; FP64 (finite: 490) 3412 -> 522 and 14120 -> 8720.
#pragma once

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace tsvd {

// The operands of a complex product as stored: op(A)(i, k) and op(B)(k, j)
template <typename C>
struct DotSrc {
  const C *A, *B;
  long lda, sA, ldb, sB;
  int K;
  bool ah, bh;
  __device__ C a(int b, int i, int k) const {
    const C* p = A + (long)b * sA;
    return ah ? cconj(p[(long)k * lda + i]) : p[(long)i * lda + k];
  }
  __device__ C b(int bi, int k, int j) const {
    const C* p = B + (long)bi * sB;
    return bh ? cconj(p[(long)j * ldb + k]) : p[(long)k * ldb + j];
  }
};

// Words of marks and the elements of a word, as the products come to them:
//   FP64 (k_dgemm_tc reads its accumulators): 32 rows of one column;
//   FP32 (k_sgemm_tc writes its result): 4 rows of 16 columns, the even columns in one word, the odd ones in the next
template <typename C>
struct MarkBits;
template <>
struct MarkBits<double2> {
  static constexpr int LIST = 8;  // the list holds this part of the elements
  __host__ __device__ static long words(int M, int N, long batch) { return batch * ((M + 31) / 32) * N; }
  __device__ static long word(int M, int N, int b, int row, int col) {
    return ((long)b * ((M + 31) / 32) + row / 32) * N + col;
  }
  __device__ static int bit(int row, int) { return row & 31; }
};
template <>
struct MarkBits<float2> {
  static constexpr int LIST = 32;
  __host__ __device__ static long words(int M, int N, long batch) {
    return batch * ((M + 3) / 4) * ((N + 15) / 16) * 2;
  }
  __device__ static long word(int M, int N, int b, int row, int col) {
    return (((long)b * ((M + 3) / 4) + row / 4) * ((N + 15) / 16) + col / 16) * 2 + (col & 1);
  }
  __device__ static int bit(int row, int col) { return (row & 3) * 8 + (col & 15) / 2; }
};

template <typename C>
struct Marks {
  unsigned long long* count;
  long* list;  // (b M + row) N + col
  uint32_t* bits;
  long cap, words;
  static long list_len(int M, int N, long batch) { return (long)M * N * batch / MarkBits<C>::LIST + 1024; }
  static size_t bytes(int M, int N, long batch) {
    return 512 + (size_t)list_len(M, N, batch) * sizeof(long) + (size_t)MarkBits<C>::words(M, N, batch) * sizeof(uint32_t);
  }
  static Marks at(uintptr_t p, int M, int N, long batch) {  // p: 256-byte aligned
    Marks m;
    m.count = (unsigned long long*)p;
    m.list = (long*)(p + 256);
    m.cap = list_len(M, N, batch);
    m.bits = (uint32_t*)(m.list + m.cap);
    m.words = MarkBits<C>::words(M, N, batch);
    return m;
  }
  // by the pass over the operands, before the product: thread i of n
  __device__ void clear(long i, long n) const {
    if (i == 0) *count = 0;
    for (; i < words; i += n) bits[i] = 0;
  }
  // by a whole warp: this lane's element (row, col) of slice b, all in the word of (row0, col0)
  __device__ void put(int M, int N, int b, int row0, int col0, bool mark, int row, int col, int lane) const {
    const uint32_t word = __ballot_sync(0xffffffffu, mark);
    if (word == 0) return;
    unsigned long long at = 0;
    if (lane == 0) {
      bits[MarkBits<C>::word(M, N, b, row0, col0)] = word;
      at = atomicAdd(count, (unsigned long long)__popc(word));
    }
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(word & ((1u << lane) - 1));
    if (mark && (long)at < cap) list[at] = ((long)b * M + row) * N + col;
  }
  __device__ bool get(int M, int N, int b, int row, int col) const {
    return bits[MarkBits<C>::word(M, N, b, row, col)] >> MarkBits<C>::bit(row, col) & 1u;
  }
};

constexpr int REDO_THREADS = 64;
constexpr int REDO_RUN = 16;  // terms added one after another, then the runs: the same sum from the list and by tiles
template <typename C>
constexpr int redo_tile() { return sizeof(C) == 16 ? 16 : 32; }

// upper: a Hermitian product, whose tiles of 128 rows x 32 columns wholly below the diagonal were left out (no marks
// there)
template <typename C>
__global__ void __launch_bounds__(REDO_THREADS, 8) k_redo(const Marks<C> mk, const __grid_constant__ DotSrc<C> src,
                                                       C* __restrict__ Cm, long ldc, long sC, int M, int N, int batch,
                                                       double alpha, int beta, int upper) {
  using R = decltype(C().x);
  const long count = (long)*mk.count;
  if (count == 0) return;
  const int tid = threadIdx.x, lane = tid & 31;
  auto put = [&](int b, int i, int j, C v) {
    C* dst = Cm + (long)b * sC + (long)i * ldc + j;
    v = cscale(v, (R)alpha);
    if (beta) v = cadd(v, *dst);
    *dst = v;
  };
  if (count <= mk.cap) {
    for (long e = (long)blockIdx.x * 2 + (tid >> 5); e < count; e += (long)gridDim.x * 2) {
      const long at = mk.list[e];
      const long r = at / N;
      const int j = (int)(at - r * N), b = (int)(r / M), i = (int)(r - (long)b * M);
      C tot = mkc(R(0), R(0));
      for (int k0 = 0; k0 < src.K; k0 += 32 * REDO_RUN) {  // a run per lane, added in their order
        C acc = mkc(R(0), R(0));
        const int kb = k0 + REDO_RUN * lane;
        const int ke = min(kb + REDO_RUN, src.K);
#pragma unroll
        for (int u = 0; u < REDO_RUN; u += 8) {  // eight terms' loads in flight
          C x[8], y[8];
#pragma unroll
          for (int v = 0; v < 8; ++v) {
            const int k = min(kb + u + v, src.K - 1);
            x[v] = src.a(b, i, k);
            y[v] = src.b(b, k, j);
          }
#pragma unroll
          for (int v = 0; v < 8; ++v)
            if (kb + u + v < ke) cfma(acc, x[v], y[v]);
        }
        const int runs = min(32, (src.K - k0 + REDO_RUN - 1) / REDO_RUN);
        for (int q = 0; q < runs; ++q)
          tot = cadd(tot, mkc(__shfl_sync(0xffffffffu, acc.x, q), __shfl_sync(0xffffffffu, acc.y, q)));
      }
      if (lane == 0) put(b, i, j, tot);
    }
    return;
  }
  constexpr int BT = redo_tile<C>(), BK = REDO_RUN, RT = BT / 8, NS = BT * BK / REDO_THREADS;
  __shared__ __align__(16) C As[BK][BT + 1], Bs[BK][BT + 1];
  const int tx = tid & 7, ty = tid >> 3;
  const long tm = (M + BT - 1) / BT, tn = (N + BT - 1) / BT, tiles = tm * tn * batch;
  for (long t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int n0 = (int)(t % tn) * BT, m0 = (int)(t / tn % tm) * BT, b = (int)(t / tn / tm);
    if (upper && n0 / 32 * 32 + 32 <= m0 / 128 * 128) continue;
    bool mark[RT][RT], some = false;
#pragma unroll
    for (int x = 0; x < RT; ++x)
#pragma unroll
      for (int y = 0; y < RT; ++y) {
        const int i = m0 + ty + 8 * x, j = n0 + tx + 8 * y;
        mark[x][y] = i < M && j < N && mk.get(M, N, b, i, j);
        some |= mark[x][y];
      }
    if (!__syncthreads_or(some)) continue;
    C acc[RT][RT], tot[RT][RT];
#pragma unroll
    for (int x = 0; x < RT; ++x)
#pragma unroll
      for (int y = 0; y < RT; ++y) acc[x][y] = tot[x][y] = mkc(R(0), R(0));
    for (int k0 = 0; k0 < src.K; k0 += BK) {
#pragma unroll
      for (int u = 0; u < NS; ++u) {  // along the contiguous dimension of each operand
        const int e = tid + REDO_THREADS * u;
        const int ka = src.ah ? e / BT : e % BK, ia = src.ah ? e % BT : e / BK;
        const int kb = src.bh ? e % BK : e / BT, jb = src.bh ? e / BK : e % BT;
        As[ka][ia] = (m0 + ia < M && k0 + ka < src.K) ? src.a(b, m0 + ia, k0 + ka) : mkc(R(0), R(0));
        Bs[kb][jb] = (n0 + jb < N && k0 + kb < src.K) ? src.b(b, k0 + kb, n0 + jb) : mkc(R(0), R(0));
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        C a[RT], c[RT];
#pragma unroll
        for (int x = 0; x < RT; ++x) a[x] = As[kk][ty + 8 * x];
#pragma unroll
        for (int y = 0; y < RT; ++y) c[y] = Bs[kk][tx + 8 * y];
#pragma unroll
        for (int x = 0; x < RT; ++x)
#pragma unroll
          for (int y = 0; y < RT; ++y) cfma(acc[x][y], a[x], c[y]);
      }
#pragma unroll
      for (int x = 0; x < RT; ++x)
#pragma unroll
        for (int y = 0; y < RT; ++y) {
          tot[x][y] = cadd(tot[x][y], acc[x][y]);
          acc[x][y] = mkc(R(0), R(0));
        }
      __syncthreads();
    }
#pragma unroll
    for (int x = 0; x < RT; ++x)
#pragma unroll
      for (int y = 0; y < RT; ++y)
        if (mark[x][y]) put(b, m0 + ty + 8 * x, n0 + tx + 8 * y, tot[x][y]);
  }
}

template <typename C>
int redo_marked(const Marks<C>& mk, const DotSrc<C>& src, C* Cm, long ldc, long sC, int M, int N, int batch,
                double alpha, bool beta, bool upper, cudaStream_t s) {
  constexpr int BT = redo_tile<C>();
  const long tiles = (long)cdiv(M, BT) * cdiv(N, BT) * batch;
  k_redo<C><<<(unsigned)std::min<long>(tiles, SMS * 8), REDO_THREADS, 0, s>>>(mk, src, Cm, ldc, sC, M, N, batch, alpha,
                                                                               beta ? 1 : 0, upper ? 1 : 0);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

}  // namespace tsvd
