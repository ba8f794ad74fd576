// cholqr.cu -- block orthonormalisation pieces of the Krylov basis (the T-QR
// step of Alg. 2, per Fourier slice): Cholesky of a Gram matrix (optionally
// shifted), the right triangular solve W <- W R^{-1}, and the replacement of
// numerically dependent columns by fresh orthonormal directions.
//
// The Gram matrix, its Cholesky factorisation and the triangular solve all run
// in the precision of the basis (FP64, or FP32 on the FP32 / mixed paths), as
// in the analysis of shifted CholeskyQR (Fukaya et al.), which takes every step
// in the working precision.
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"

namespace tsvd {

// ---------------------------------------------------------------------------
// Cholesky (upper, right-looking) R^H R = G + s I of one nb x nb Gram matrix
// per CTA, in the Gram's own precision, s = shift_rel * trace(G), followed by
// the inverse M of R-tilde, written dense (zeros below the diagonal):
//   pivot test: shifted pass -> dead iff d_j <= 0; plain pass -> dead iff
//   d_j <= dead_rel * G_jj;
//   R-tilde: R with every dead row and every dead column replaced by the unit
//   vector (so R-tilde = diag(R_live, I) up to a permutation);
//   M: R-tilde^{-1} with the dead columns set to zero, so that W M is
//   W_live R_live^{-1} on the live columns and zero on the dead ones.
// Panels of P rows, two barriers each.  Every thread keeps a T x T tile of the
// upper triangle in registers:
//   factorisation, panel p: the tiles of its rows are published; each warp
//   eliminates the P diagonal columns (its first lanes, redundantly) together with
//   32 - P further columns, one lane per column, the row R(j, .) of the diagonal
//   columns handed round by shuffles; the finished rows are kept in shared
//   memory and every later tile subtracts their rank-P product;
//   inverse, panel from the last to the first (R X = I for all columns at
//   once): the tiles of its rows are published, solved against the panel's
//   triangle with one lane per column, written out as rows of M, and
//   subtracted, times R's columns, from every tile above.
// Bound: the chain of pivots in a panel, and in FP64 its pipe (64 clocks per
// instruction of one warp).  P = 8, T = 4 in FP32; FP64 takes P = 4 and the
// smallest tiles that fit (an instruction costs the same whatever the lanes).
// Against one step and barrier per row, 33 slices: FP32 nb = 25: 23 -> 16 us, 60:
// 59 -> 29, 120: 272 -> 61; FP64 15: 35 -> 28, 60: 271 -> 202, 120: 1910 -> 1240.
// Roots of FP32 pivots by root and division instead of the estimate: + 11 % (60 on 33 slices 24.6 -> 27.4 us, 120 on
// 65 slices 56.5 -> 62.2, as they run in a T-SVD).
// ---------------------------------------------------------------------------

__device__ __forceinline__ float2 shfl_c(float2 v, int l) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}
__device__ __forceinline__ double2 shfl_c(double2 v, int l) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}
// T consecutive complex values of shared memory (16-byte aligned)
template <int T>
__device__ __forceinline__ void load_t(const float2* p, float2* o) {
#pragma unroll
  for (int q = 0; q < T; q += 2) {
    const float4 a = *(const float4*)(p + q);
    o[q] = make_float2(a.x, a.y);
    o[q + 1] = make_float2(a.z, a.w);
  }
}
template <int T>
__device__ __forceinline__ void load_t(const double2* p, double2* o) {
#pragma unroll
  for (int q = 0; q < T; ++q) o[q] = p[q];
}
// acc -= a b and acc -= conj(a) b
template <typename C>
__device__ __forceinline__ void cfms(C& acc, C a, C b) {
  acc.x = fma(-a.x, b.x, acc.x);
  acc.x = fma(a.y, b.y, acc.x);
  acc.y = fma(-a.x, b.y, acc.y);
  acc.y = fma(-a.y, b.x, acc.y);
}
template <typename C>
__device__ __forceinline__ void cfmsc(C& acc, C a, C b) {
  acc.x = fma(-a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(-a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}

// P rows per panel
template <int P>
__host__ __device__ inline int ch_pad(int nb) { return (nb + P - 1) / P * P; }
// panel p's rows in the store of R: P rows of n8 - P p values (columns P p ..)
template <int P>
__host__ __device__ inline int ch_off(int p, int n8) { return P * (n8 * p - P * (p * (p - 1) / 2)); }

// Tiles to threads.  FP32: the triangle's rows one after another.  FP64, whose pipe takes 16 clocks per
// instruction and warp whatever the lanes: a warp holds a block of 4 x 8 tiles, so that the tiles of a
// warp are active in the same steps of the inverse (23 instead of 49 warp-steps at n8 = 64).
template <typename GC>
struct ChMap {  // float2
  static __host__ __device__ int threads(int ntl) { return (ntl * (ntl + 1) / 2 + 31) / 32 * 32; }
  static __device__ void tile(int tid, int ntl, int* ta, int* tb) {
    int a = 0, b = tid;
    while (a < ntl && b >= ntl - a) {
      b -= ntl - a;
      ++a;
    }
    *ta = a;
    *tb = a + b;
  }
};
template <>
struct ChMap<double2> {
  static __host__ __device__ int first(int a) { return a / 2; }  // first block column of block row a
  static __host__ __device__ int threads(int ntl) {
    int n = 0;
    for (int a = 0; 4 * a < ntl; ++a) n += (ntl + 7) / 8 - first(a);
    return 32 * n;
  }
  static __device__ void tile(int tid, int ntl, int* ta, int* tb) {
    int a = 0, w = tid >> 5;
    const int cols = (ntl + 7) / 8, lane = tid & 31;
    while (4 * a < ntl && w >= cols - first(a)) {
      w -= cols - first(a);
      ++a;
    }
    *ta = 4 * a + (lane >> 3);
    *tb = 8 * (first(a) + w) + (lane & 7);
  }
};

template <typename GC, int CH_P, int CH_T, int NT>  // CH_P rows per panel, tiles of edge CH_T; NT: most threads
__global__ void __launch_bounds__(NT, 1) k_chol_inv(const GC* __restrict__ G, long ldg, long sG,
                                                      GC* __restrict__ Mo, long ldm, long sM, int nb,
                                                      double shift_rel, double dead_rel,
                                                      uint32_t* __restrict__ dead_out) {
  using Rt = decltype(GC().x);
  constexpr int TPP = CH_P / CH_T, CH_COLS = 32 - CH_P;  // tile rows per panel; columns a warp eliminates beside the diagonal ones
  extern __shared__ __align__(16) unsigned char chsm[];
  const int n8 = ch_pad<CH_P>(nb), NP = n8 / CH_P, NTL = n8 / CH_T;
  GC* S = (GC*)chsm;           // R by panels
  GC* Raw = S + ch_off<CH_P>(NP, n8);  // [8][n8] published rows
  GC* Xb = Raw + CH_P * n8;      // [8][n8] solved rows of the inverse
  __shared__ Rt thr[128];        // a pivot at or below it is dead
  __shared__ Rt ri[128];         // 1 / R-tilde_jj
  __shared__ int live[128];
  __shared__ double red[NT / 32];
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  G += (long)b * sG;
  Mo += (long)b * sM;
  const GC zero{Rt(0), Rt(0)};
  int ta, tb;  // this thread's tile; none off the upper triangle
  ChMap<GC>::tile(tid, NTL, &ta, &tb);
  const bool own = ta < NTL && tb < NTL && ta <= tb;
  GC v[CH_T][CH_T];
  const Rt gd = tid < nb ? G[(long)tid * ldg + tid].x : Rt(0);
  if (tid < 128) thr[tid] = (shift_rel > 0.0 || tid >= nb) ? Rt(0) : (Rt)dead_rel * gd;
#pragma unroll
  for (int x = 0; x < CH_T; ++x)
#pragma unroll
    for (int y = 0; y < CH_T; ++y) {
      const int i = CH_T * ta + x, k = CH_T * tb + y;
      v[x][y] = (own && i <= k && k < nb) ? G[(long)i * ldg + k] : zero;
      if (i == k && i >= nb) v[x][y].x = Rt(1);  // padding rows: the unit matrix
    }
  __syncthreads();
  const double trace = block_sum((double)gd, red);
  const Rt sft = (shift_rel > 0.0) ? (Rt)(shift_rel * trace) : Rt(0);
  if (own && ta == tb) {
#pragma unroll
    for (int x = 0; x < CH_T; ++x)
      if (CH_T * ta + x < nb) v[x][x].x += sft;
  }
  // publish this thread's tile if it lies in panel p's rows
  auto publish = [&](int p) {
    if (own && ta / TPP == p) {
#pragma unroll
      for (int x = 0; x < CH_T; ++x)
#pragma unroll
        for (int y = 0; y < CH_T; ++y) Raw[(CH_T * (ta % TPP) + x) * n8 + CH_T * tb + y] = v[x][y];
    }
  };

  for (int p = 0; p < NP; ++p) {
    publish(p);
    __syncthreads();
    const int j0 = CH_P * p;
    // columns of this warp: the 8 diagonal ones and 24 of the rest
    const int rest = n8 - j0 - CH_P;
    if (warp == 0 || warp * CH_COLS < rest) {
      const int kc = lane < CH_P ? lane : CH_P + warp * CH_COLS + lane - CH_P;  // column j0 + kc
      const bool in = kc < n8 - j0;
      GC c[CH_P];
#pragma unroll
      for (int r = 0; r < CH_P; ++r) c[r] = in ? Raw[r * n8 + j0 + kc] : zero;
#pragma unroll
      for (int r = 0; r < CH_P; ++r) {
        const Rt d = __shfl_sync(0xffffffffu, c[r].x, r);
        const int j = j0 + r;
        const bool alive = d > thr[j];
        const Rt iv = alive ? inv_sqrt(d) : Rt(0);
        c[r].x *= iv;
        c[r].y *= iv;
        if (lane == r) c[r].y = Rt(0);
        if (warp == 0 && lane == r) {
          live[j] = alive;
          ri[j] = alive ? iv : Rt(1);
        }
#pragma unroll
        for (int i = r + 1; i < CH_P; ++i) cfmsc(c[i], shfl_c(c[r], i), c[r]);
      }
      if (in && (warp == 0 || lane >= CH_P)) {
        GC* o = S + ch_off<CH_P>(p, n8) + kc;
#pragma unroll
        for (int r = 0; r < CH_P; ++r) o[r * (n8 - j0)] = (kc >= r) ? c[r] : zero;
      }
    }
    __syncthreads();
    if (own && ta / TPP > p) {
      const GC* P = S + ch_off<CH_P>(p, n8);
      const int ra = CH_T * ta - j0, rb = CH_T * tb - j0;
#pragma unroll
      for (int r = 0; r < CH_P; ++r) {
        GC x4[CH_T], y4[CH_T];
        load_t<CH_T>(P + r * (n8 - j0) + ra, x4);
        load_t<CH_T>(P + r * (n8 - j0) + rb, y4);
#pragma unroll
        for (int x = 0; x < CH_T; ++x)
#pragma unroll
          for (int y = 0; y < CH_T; ++y) cfmsc(v[x][y], x4[x], y4[y]);
      }
    }
  }
  __syncthreads();
  // R-tilde: dead columns zero (dead rows are already)
  for (int k = warp; k < nb; k += blockDim.x >> 5)
    if (!live[k])
      for (int i = lane; i < k; i += 32) {
        const int q = i / CH_P;
        S[ch_off<CH_P>(q, n8) + (i - CH_P * q) * (n8 - CH_P * q) + k - CH_P * q] = zero;
      }
#pragma unroll
  for (int x = 0; x < CH_T; ++x)
#pragma unroll
    for (int y = 0; y < CH_T; ++y) {
      v[x][y] = zero;
      if (ta == tb && x == y) v[x][y].x = Rt(1);
    }
  for (int p = NP - 1; p >= 0; --p) {
    publish(p);
    __syncthreads();
    const int j0 = CH_P * p, len = n8 - j0;
    const GC* P = S + ch_off<CH_P>(p, n8);
    for (int kc = tid; kc < len; kc += blockDim.x) {
      const int k = j0 + kc;
      GC x[CH_P];
#pragma unroll
      for (int r = 0; r < CH_P; ++r) x[r] = (kc >= r || kc >= CH_P) ? Raw[r * n8 + k] : zero;
#pragma unroll
      for (int r = CH_P - 1; r >= 0; --r) {
#pragma unroll
        for (int q = r + 1; q < CH_P; ++q) cfms(x[r], P[r * len + q], x[q]);
        const Rt s = ri[j0 + r];
        x[r].x *= s;
        x[r].y *= s;
      }
#pragma unroll
      for (int r = 0; r < CH_P; ++r) {
        Xb[r * n8 + k] = x[r];
        if (j0 + r < nb && k < nb && k >= j0 + r) Mo[(long)(j0 + r) * ldm + k] = live[k] ? x[r] : zero;
      }
    }
    __syncthreads();
    if (own && ta / TPP < p && tb / TPP >= p) {
      const int rp = ta / TPP, rl = n8 - CH_P * rp;  // the panel that holds this tile's rows of R
      const GC* A = S + ch_off<CH_P>(rp, n8) + CH_T * (ta % TPP) * rl + j0 - CH_P * rp;
#pragma unroll
      for (int q0 = 0; q0 < CH_P; q0 += CH_T) {
        GC a4[CH_T][CH_T];
#pragma unroll
        for (int x = 0; x < CH_T; ++x) load_t<CH_T>(A + x * rl + q0, a4[x]);
#pragma unroll
        for (int q = 0; q < CH_T; ++q) {
          GC y4[CH_T];
          load_t<CH_T>(Xb + (q0 + q) * n8 + CH_T * tb, y4);
#pragma unroll
          for (int x = 0; x < CH_T; ++x)
#pragma unroll
            for (int y = 0; y < CH_T; ++y) cfms(v[x][y], a4[x][q], y4[y]);
        }
      }
    }
  }
  for (int e = tid; e < nb * nb; e += blockDim.x) {
    const int i = e / nb, k = e - i * nb;
    if (k < i) Mo[(long)i * ldm + k] = zero;
  }
  if (tid < 4) {
    uint32_t msk = 0;
    for (int q = 0; q < 32; ++q) {
      const int jj = tid * 32 + q;
      if (jj < nb && !live[jj]) msk |= 1u << q;
    }
    dead_out[b * 4 + tid] = msk;
  }
}

template <typename GC>
int chol_inv(const GC* G, long ldg, long sG, GC* M, long ldm, long sM, int nb, int batch, double shift_rel,
             double dead_rel, uint32_t* dead, cudaStream_t s) {
  if (nb <= 0 || batch <= 0) return TSVD_OK;
  if (nb > 128) return TSVD_ERR_UNSUPPORTED;
  auto go = [&](auto kern, int n8, int off, int nthr) {
    const size_t smem = ((size_t)off + 2 * (size_t)(n8 % 8 ? 4 : 8) * n8) * sizeof(GC);
    if (smem > 40 * 1024 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
      cudaGetLastError();
      return TSVD_ERR_CUDA;
    }
    kern<<<batch, nthr, smem, s>>>(G, ldg, sG, M, ldm, sM, nb, shift_rel, dead_rel, dead);
    TSVD_LAUNCHED();
    return TSVD_OK;
  };
  // at least 128 threads: one per diagonal entry
  if constexpr (std::is_same<GC, double2>::value) {
    // FP64: panels of 4 (the panel's own elimination is one warp's work, at 64 clocks per FP64
    // instruction of one warp) and the smallest tiles that fit 1024 threads
    const int n4 = ch_pad<4>(nb), t1 = ChMap<GC>::threads(n4), t2 = ChMap<GC>::threads(n4 / 2);
    if (t1 <= 1024) return go(k_chol_inv<GC, 4, 1, 1024>, n4, ch_off<4>(n4 / 4, n4), std::max(128, t1));
    if (t2 <= 1024) return go(k_chol_inv<GC, 4, 2, 1024>, n4, ch_off<4>(n4 / 4, n4), t2);
  }
  const int n8 = ch_pad<8>(nb), off = ch_off<8>(n8 / 8, n8), nthr = std::max(128, ChMap<GC>::threads(n8 / 4));
  // registers: 4 x 4 tiles and a panel's operands take 125 in FP32, 167 in FP64
  if constexpr (std::is_same<GC, float2>::value) {
    if (nthr <= 256) return go(k_chol_inv<GC, 8, 4, 256>, n8, off, nthr);
    if (nthr <= 512) return go(k_chol_inv<GC, 8, 4, 512>, n8, off, nthr);  // n8 <= 120
    return go(k_chol_inv<GC, 8, 4, 544>, n8, off, nthr);                   // 128: 32 * 33 / 2 tiles
  } else {
    if (nthr <= 384) return go(k_chol_inv<GC, 8, 4, 384>, n8, off, nthr);  // n8 <= 96
    return go(k_chol_inv<GC, 8, 4, 640>, n8, off, nthr);                   // 128: 20 blocks
  }
}
template int chol_inv<double2>(const double2*, long, long, double2*, long, long, int, int, double, double, uint32_t*,
                               cudaStream_t);
template int chol_inv<float2>(const float2*, long, long, float2*, long, long, int, int, double, double, uint32_t*,
                              cudaStream_t);

// asynchronous global -> shared copy of one complex element (8 or 16 bytes)
template <typename C>
__device__ __forceinline__ void cp_async_elem(C* dst, const C* src) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(C) == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(src));
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(src));
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// ---------------------------------------------------------------------------
// O <- W M for the n1 x nb block of every slice (M nb x nb, upper
// triangular, dense): a CTA stages TM_ROWS full rows of W and, kchunk rows at
// a time, M in shared memory (all of M at once when it fits); thread
// (ty, tx) accumulates rows ty + 16a (a < 4) and columns tx + 16u in
// registers; column group u takes no terms from rows k >= 16 (u + 1).
// ---------------------------------------------------------------------------
constexpr int TM_ROWS = 64;
template <typename C, int NU>  // NU = ceil(nb / 16) column groups per thread
__global__ void __launch_bounds__(256) k_rmul_block(const C* W, long ldw, long sW, const C* __restrict__ M,
                                                  long ldm, long sM, int n1, int nb, int kchunk, C* O, long ldo,
                                                  long sO) {
  using R = decltype(C().x);
  extern __shared__ __align__(16) unsigned char rmsm[];
  constexpr int MC = 16 * NU;
  C* Ws = (C*)rmsm;                  // [TM_ROWS][nb + 1]
  const int lw = nb + 1;
  C* Ms = Ws + TM_ROWS * lw;         // [kchunk][MC]
  const int b = blockIdx.y, tid = threadIdx.x;
  const int r0 = blockIdx.x * TM_ROWS;
  W += (long)b * sW;
  M += (long)b * sM;
  O += (long)b * sO;
  // asynchronous copies: every element of the rows and of the chunk of M is in flight at once
  for (int r = tid >> 5; r < TM_ROWS; r += 8)
    for (int k = tid & 31; k < nb; k += 32) {
      if (r0 + r < n1) cp_async_elem(Ws + r * lw + k, W + (long)(r0 + r) * ldw + k);
      else Ws[r * lw + k] = C{R(0), R(0)};
    }
  const int ty = tid >> 4, tx = tid & 15;
  C acc[4][NU];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int u = 0; u < NU; ++u) acc[a][u] = C{R(0), R(0)};
  for (int k0 = 0; k0 < nb; k0 += kchunk) {
    const int kc = min(kchunk, nb - k0);
    if (k0 > 0) __syncthreads();  // the previous chunk of M consumed
    for (int e = tid; e < kc * MC; e += 256) {
      const int kk = e / MC, c = e - kk * MC;
      if (c < nb) cp_async_elem(Ms + e, M + (long)(k0 + kk) * ldm + c);
      else Ms[e] = C{R(0), R(0)};
    }
    cp_async_wait_all();
    __syncthreads();
    for (int kk = 0; kk < kc; ++kk) {
      const int k = k0 + kk;
      C a[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) a[q] = Ws[(ty + 16 * q) * lw + k];
      const int u0 = k >> 4;  // M(k, c) = 0 for c < k
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        if (u >= u0) {
          const C mv = Ms[kk * MC + tx + 16 * u];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            acc[q][u].x = fma(a[q].x, mv.x, acc[q][u].x);
            acc[q][u].x = fma(-a[q].y, mv.y, acc[q][u].x);
            acc[q][u].y = fma(a[q].x, mv.y, acc[q][u].y);
            acc[q][u].y = fma(a[q].y, mv.x, acc[q][u].y);
          }
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = r0 + ty + 16 * q;
    if (r < n1) {
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        const int c = tx + 16 * u;
        if (c < nb) O[(long)r * ldo + c] = acc[q][u];
      }
    }
  }
}

template <typename C>
int rmul_block(const C* W, long ldw, long sW, const C* M, long ldm, long sM, int n1, int nb, int batch, C* O, long ldo,
               long sO, cudaStream_t s) {
  if (nb <= 0 || n1 <= 0 || batch <= 0) return TSVD_OK;
  if (nb > 128) return TSVD_ERR_UNSUPPORTED;
  if (batch > 65535) return TSVD_ERR_UNSUPPORTED;
  const int nu = (nb + 15) / 16;
  const size_t wbytes = (size_t)TM_ROWS * (nb + 1) * sizeof(C), mrow = (size_t)16 * nu * sizeof(C);
  int kchunk = nb;
  while (wbytes + kchunk * mrow > 200 * 1024) kchunk = (kchunk + 1) / 2;
  const size_t smem = wbytes + kchunk * mrow;
  const dim3 grid(cdiv(n1, TM_ROWS), batch);
  auto go = [&](auto kern) {
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
      cudaGetLastError();
      return TSVD_ERR_CUDA;
    }
    kern<<<grid, 256, smem, s>>>(W, ldw, sW, M, ldm, sM, n1, nb, kchunk, O, ldo, sO);
    TSVD_LAUNCHED();
    return TSVD_OK;
  };
  switch (nu) {
    case 1: return go(k_rmul_block<C, 1>);
    case 2: return go(k_rmul_block<C, 2>);
    case 3: return go(k_rmul_block<C, 3>);
    case 4: return go(k_rmul_block<C, 4>);
    case 5: return go(k_rmul_block<C, 5>);
    case 6: return go(k_rmul_block<C, 6>);
    case 7: return go(k_rmul_block<C, 7>);
    default: return go(k_rmul_block<C, 8>);
  }
}
template int rmul_block<double2>(const double2*, long, long, const double2*, long, long, int, int, int, double2*, long,
                                 long, cudaStream_t);
template int rmul_block<float2>(const float2*, long, long, const float2*, long, long, int, int, int, float2*, long, long,
                                cudaStream_t);

// ---------------------------------------------------------------------------
// Dependent Krylov columns (exact low rank, zero data): replace column c+j by
// a Philox Gaussian direction (stream 3) projected twice against every other
// live column of the basis, then normalised.  Any orthonormal completion of
// span(K) leaves the Rayleigh-Ritz result of Alg. 2 optimal (Sec. 4: Q (Q^T A)_k is the best rank-k approximation
// within range(Q)).
// ---------------------------------------------------------------------------
template <typename C>
__global__ void __launch_bounds__(256) k_repair_dead(C* __restrict__ Q, long ldq, long sQ, int n1, int c, int nb,
                                                     const uint32_t* __restrict__ dead, uint64_t seed, int block_id,
                                                     int* __restrict__ dead_count, int k0, int nyq) {
  using R = decltype(C().x);
  __shared__ double red[32];
  const int b = blockIdx.x, tid = threadIdx.x;
  uint32_t dm[4];
  int ndead = 0;
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    dm[w] = dead[b * 4 + w];
    ndead += __popc(dm[w]);
  }
  if (ndead == 0) return;
  Q += (long)b * sQ;
  const int k = k0 + b;  // Fourier slice index of this problem
  const bool real_slice = (k == 0) || (k == nyq);
  if (tid == 0) atomicAdd(dead_count, ndead);
  uint32_t pending[4] = {dm[0], dm[1], dm[2], dm[3]};
  for (int j = 0; j < nb; ++j) {
    if (!((dm[j >> 5] >> (j & 31)) & 1u)) continue;
    const int col = c + j;
    for (int attempt = 0; attempt < 4; ++attempt) {
      for (int i = tid; i < n1; i += blockDim.x) {
        const uint4 x = philox10(make_uint4((uint32_t)i, (uint32_t)col | ((uint32_t)attempt << 24),
                                            (uint32_t)block_id, 3u + ((uint32_t)k << 8)),
                                 (uint32_t)seed, (uint32_t)(seed >> 32));
        const double u1 = ((double)x.x + 1.0) * (1.0 / 4294967296.0);
        const double u2 = ((double)x.y + 1.0) * (1.0 / 4294967296.0);
        const double r = sqrt(-2.0 * log(u1));
        double sn, cs;
        sincospi(2.0 * u2, &sn, &cs);
        // the DC slice (and the Nyquist slice of an even-length transform) of a real
        // tensor's spectrum is real: its replacement directions are real too
        C v;
        v.x = (R)(r * cs);
        v.y = real_slice ? (R)0 : (R)(r * sn);
        Q[(long)i * ldq + col] = v;
      }
      __syncthreads();
      for (int pass = 0; pass < 2; ++pass) {
        for (int l = 0; l < c + nb; ++l) {
          if (l == col) continue;
          if (l >= c && ((pending[(l - c) >> 5] >> ((l - c) & 31)) & 1u)) continue;
          double2 part = make_double2(0, 0);
          for (int i = tid; i < n1; i += blockDim.x)
            cfmac(part, to_c64(Q[(long)i * ldq + l]), to_c64(Q[(long)i * ldq + col]));
          const double2 dot = block_sum2(part, red);
          for (int i = tid; i < n1; i += blockDim.x) {
            double2 q = to_c64(Q[(long)i * ldq + col]);
            const double2 ql = to_c64(Q[(long)i * ldq + l]);
            q.x -= dot.x * ql.x - dot.y * ql.y;
            q.y -= dot.x * ql.y + dot.y * ql.x;
            Q[(long)i * ldq + col] = from_c64<C>(q);
          }
          __syncthreads();
        }
      }
      double part = 0;
      for (int i = tid; i < n1; i += blockDim.x) part += cabs2(to_c64(Q[(long)i * ldq + col]));
      const double nrm = sqrt(block_sum(part, red));
      const bool ok = nrm > 1e-3;
      for (int i = tid; i < n1; i += blockDim.x)
        Q[(long)i * ldq + col] = ok ? from_c64<C>(cscale(to_c64(Q[(long)i * ldq + col]), 1.0 / nrm))
                                    : from_c64<C>(make_double2(0, 0));
      __syncthreads();
      if (ok) break;
    }
    pending[j >> 5] &= ~(1u << (j & 31));
  }
}

template <typename C>
int repair_dead(C* Q, long ldq, long sQ, int n1, int c, int nb, const uint32_t* dead, int batch, uint64_t seed,
                int block_id, int* dead_count, int k0, int nyq, cudaStream_t s) {
  if (nb <= 0 || batch <= 0) return TSVD_OK;
  k_repair_dead<C><<<batch, 256, 0, s>>>(Q, ldq, sQ, n1, c, nb, dead, seed, block_id, dead_count, k0, nyq);
  TSVD_LAUNCHED();
  return TSVD_OK;
}
template int repair_dead<double2>(double2*, long, long, int, int, int, const uint32_t*, int, uint64_t, int, int*,
                                  int, int, cudaStream_t);
template int repair_dead<float2>(float2*, long, long, int, int, int, const uint32_t*, int, uint64_t, int, int*, int,
                                 int, cudaStream_t);

// Orthonormalise the nb leading columns of W (n1 x b per slice) against the c
// finished columns of Q and write them to Q columns [c, c+nb), in the
// precision L: shifted CholeskyQR3 (the shift makes the first Cholesky
// succeed for any W; the next two passes restore orthogonality to rounding
// level), each pass preceded by a classical Gram-Schmidt projection against
// Q_{<i}; dependent columns are then replaced.
// The FP32 block step with every product on tcgen05 in split TF32 (FP32-level
// accuracy, tc_gemm.cu): the block Gram W^H W and the coefficients Q^H W as
// real products of de-interleaved columns (K = n1), the update W -= Q (Q^H W)
// and W R^-1 as real(X) E(Y)^T with the small expanded real form E of the
// thin factor.  Q's finished columns are split once per block (hi / lo
// interleaved and de-interleaved rows) and reused by all later projections;
// the update's epilogue writes W's split rows for W R^-1.
// X^H Y (rows x cols complex) from the real product P = X_d Y_d^T of the de-interleaved columns
// (row 2c of X_d the real parts of column c of X, row 2c+1 the imaginary parts; Y_d alike):
//   (X^H Y)_ij = P[2i][2j] + P[2i+1][2j+1] + i (P[2i][2j+1] - P[2i+1][2j])
__global__ void k_complex_from_real(const float* __restrict__ P, long ldp, long sp, int rows, int cols,
                                    float2* __restrict__ G, long ldg, long sG, int batch) {
  const long total = (long)batch * rows * cols;
  for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    const int j = idx % cols;
    const long r = idx / cols;
    const int i = r % rows;
    const int b = r / rows;
    const float* p0 = P + (long)b * sp + (long)(2 * i) * ldp + 2 * j;
    const float* p1 = p0 + ldp;
    G[(long)b * sG + (long)i * ldg + j] = make_float2(p0[0] + p1[1], p0[1] - p1[0]);
  }
}

static int complex_from_real(const float* P, long ldp, long sp, int rows, int cols, float2* G, long ldg, long sG,
                             int batch, cudaStream_t s) {
  const long total = (long)batch * rows * cols;
  if (total <= 0) return TSVD_OK;
  k_complex_from_real<<<(unsigned)std::min<long>(cdiv(total, 256), 4096), 256, 0, s>>>(P, ldp, sp, rows, cols, G,
                                                                                      ldg, sG, batch);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

static int orth_block_tc(int n1, int b, int m, int h, const OrthWs& w, int c, int nb, int block_id, uint64_t seed,
                         cudaStream_t s) {
  const OrthTc& t = *w.tc;
  float2* Q = (float2*)w.Q;
  float2* W = (float2*)w.W;
  float2* P = (float2*)w.P;
  float2* Gs = (float2*)w.G;
  float2* Mi = (float2*)w.Minv;
  const long sQ = (long)n1 * m, sW = (long)n1 * b, sP = (long)m * b, sG = (long)b * b;
  const long sWT = (long)b * t.ldq2, sWr = (long)n1 * t.ldw2, sE = 2L * b * t.ldq2;
  const long ldd = t.ldq2 / 2;  // de-interleaved rows: >= n1, a multiple of 4 (16-byte rows)
  // wr: the split rows of the current W (Whi / Wlo) exist, written by the epilogue of the GEMM that
  // produced W (its de-interleaved rows too, transposed there, gave 10.58 + 0.48 ms of products and
  // passes at 2048 x 120, m = 480 on 65 slices, the separate pass 9.70 + 1.49)
  bool wr = false;
  TcSplitOut rows;
  rows.Rhi = t.Whi;
  rows.Rlo = t.Wlo;
  rows.ldr = t.ldw2;
  rows.sr = sWr;
  for (int pass = 0; pass < 3; ++pass) {
    if (c > 0) {
      // the projection on tcgen05 against the cached split operands of Q's finished columns:
      // Q^H W from the real product Q_d W_d^T (K = n1), then W -= Q (Q^H W) with Q's
      // interleaved rows (K = 2c) against the expanded coefficients
      TSVD_STAGE("orth_cgs", s);
      TSVD_TRY(split_deinterleave(W, n1, nb, b, sW, h, t.WThi, t.WTlo, ldd, sWT, s));
      TSVD_TRY(tc_gemm_split(t.Qdhi, t.Qdlo, ldd, 2L * m * ldd, 2 * c, t.WThi, t.WTlo, ldd, sWT, 2 * nb, n1, t.Elo,
                             2L * b, 4L * m * b, h, t.err, s));
      TSVD_TRY(complex_from_real(t.Elo, 2L * b, 4L * m * b, c, nb, P, nb, sP, h, s));
      const long sEq = 2L * b * t.ldqi;
      TSVD_TRY(expand_thin_split(P, nb, sP, c, nb, t.Ehi, t.Elo, t.ldqi, sEq, h, 0, s));
      TSVD_TRY(tc_gemm_split(t.Qhi, t.Qlo, t.ldqi, (long)n1 * t.ldqi, n1, t.Ehi, t.Elo, t.ldqi, sEq, 2 * nb, 2 * c,
                             (float*)W, 2L * b, 2L * sW, h, t.err, s, -1.0f, 1.0f, &rows));
      wr = true;
    }
    {
      // G = W^H W through the real Gram of W's de-interleaved columns (K = n1; 2 nb x 2 nb outputs,
      // kept in Elo until the Cholesky has read G)
      TSVD_STAGE("orth_gram", s);
      float* Pr = t.Elo;
      TSVD_TRY(split_deinterleave(W, n1, nb, b, sW, h, t.WThi, t.WTlo, ldd, sWT, s));
      TSVD_TRY(tc_gemm_split(t.WThi, t.WTlo, ldd, sWT, 2 * nb, t.WThi, t.WTlo, ldd, sWT, 2 * nb, n1, Pr, 2L * b,
                             4L * b * b, h, t.err, s));
      TSVD_TRY(complex_from_real(Pr, 2L * b, 4L * b * b, nb, nb, Gs, b, sG, h, s));
    }
    {
      TSVD_STAGE("orth_chol", s);
      TSVD_TRY(chol_inv<float2>(Gs, b, sG, Mi, b, sG, nb, h, pass == 0 ? 1e-5 : 0.0, 1e-7, w.dead, s));
    }
    {
      TSVD_STAGE("orth_trsm", s);  // W R^-1, the last pass straight into its columns of Q
      if (!wr) TSVD_TRY(split_rows((const float*)W, 2L * b, t.Whi, t.Wlo, t.ldw2, 2 * nb, (long)h * n1, s));
      TSVD_TRY(expand_thin_split(Mi, b, sG, nb, nb, t.Ehi, t.Elo, t.ldw2, sE, h, 0, s));
      float* out = (pass < 2) ? (float*)W : (float*)(Q + c);
      TSVD_TRY(tc_gemm_split(t.Whi, t.Wlo, t.ldw2, sWr, n1, t.Ehi, t.Elo, t.ldw2, sE, 2 * nb, 2 * nb, out,
                             pass < 2 ? 2L * b : 2L * m, pass < 2 ? 2L * sW : 2L * sQ, h, t.err, s));
      wr = false;
    }
  }
  {
    TSVD_STAGE("orth_repair", s);
    TSVD_TRY(repair_dead<float2>(Q, m, sQ, n1, c, nb, w.dead, h, seed, block_id, w.dead_count, w.k0, w.nyq, s));
  }
  // the finished columns' split operands for the projections of the later blocks
  TSVD_STAGE("orth_cgs", s);
  TSVD_TRY(split_block((const float*)(Q + c), 2L * m, t.Qhi + 2L * c, t.Qlo + 2L * c, t.ldqi, 2 * nb, (long)h * n1,
                       s));
  return split_deinterleave(Q + c, n1, nb, m, sQ, h, t.Qdhi + 2L * c * ldd, t.Qdlo + 2L * c * ldd, ldd,
                            2L * m * ldd, s);
}

template <typename L>
int orth_block_cols(int n1, int b, int m, int h, const OrthWs& w, int c, int nb, int block_id, uint64_t seed,
                    cudaStream_t s) {
  using CL = cx_t<L>;
  if constexpr (std::is_same<L, float>::value) {
    if (w.tc) return orth_block_tc(n1, b, m, h, w, c, nb, block_id, seed, s);
  }
  const long sQ = (long)n1 * m, sW = (long)n1 * b, sP = (long)m * b, sG = (long)b * b;
  CL* Q = (CL*)w.Q;
  CL* W = (CL*)w.W;
  CL* P = (CL*)w.P;
  CL* Gs = (CL*)w.G;
  const size_t sk = std::is_same<L, double>::value ? w.splitk_elems : 2 * w.splitk_elems;
  // FP64: Fukaya et al.'s shift 11 (n nb + nb (nb+1)) u ||W||^2 (trace as the norm
  // bound); FP32: 1e-5 trace(G), above the FP32 Gram error ~ sqrt(n) u ||W||^2
  const double shift = std::is_same<L, double>::value
                           ? 11.0 * ((double)n1 * nb + (double)nb * (nb + 1)) * 1.1102230246251565e-16
                           : 1e-5;
  const double dead_rel = std::is_same<L, double>::value ? 1e-12 : 1e-7;
  // the block goes from W to its columns of Q, back, and again: no product writes over its operand
  CL* Qc = Q + c;
  for (int pass = 0; pass < 3; ++pass) {
    CL *X = pass == 1 ? Qc : W, *Y = pass == 1 ? W : Qc;
    const long ldx = pass == 1 ? m : b, sX = pass == 1 ? sQ : sW, ldy = pass == 1 ? b : m, sY = pass == 1 ? sW : sQ;
    // a Gram-Schmidt projection before every pass: without the third, blocks
    // whose new directions are tiny next to the old ones (exact low rank in
    // FP32, the fast-decaying spectra of Sec. 5 Ex. 1 in FP64) lose accuracy
    if (c > 0) {
      TSVD_STAGE("orth_cgs", s);
      TSVD_TRY(cgemm<CL>(gemm('H', 'N', c, nb, n1, 1.0, Q, m, sQ, X, ldx, sX, 0.0, P, nb, sP, h), w.splitk, sk, s, w.st));
      TSVD_TRY(cgemm<CL>(gemm('N', 'N', n1, nb, c, -1.0, Q, m, sQ, P, nb, sP, 1.0, X, ldx, sX, h), w.splitk, sk, s, w.st));
    }
    {
      TSVD_STAGE("orth_gram", s);
      TSVD_TRY(cgemm<CL>(gemm('H', 'N', nb, nb, n1, 1.0, X, ldx, sX, X, ldx, sX, 0.0, Gs, b, sG, h), w.splitk, sk, s, w.st));
    }
    CL* Mi = (CL*)w.Minv;  // R-tilde^{-1}, nb x nb per slice (leading dimension b)
    {
      TSVD_STAGE("orth_chol", s);
      TSVD_TRY(chol_inv<CL>(Gs, b, sG, Mi, b, sG, nb, h, pass == 0 ? shift : 0.0, dead_rel, w.dead, s));
    }
    {
      TSVD_STAGE("orth_trsm", s);
      const GemmArgs g = gemm('N', 'N', n1, nb, nb, 1.0, X, ldx, sX, Mi, b, sG, 0.0, Y, ldy, sY, h);
      if (std::is_same<L, double>::value && !w.st.simt && dgemm_tc_better(g, sk * sizeof(CL)))
        TSVD_TRY(dgemm_tc(g, w.splitk, sk * sizeof(CL), s, false, w.st));
      else if (std::is_same<L, float>::value && !w.st.simt && sgemm_tc_better(g, sk * sizeof(CL)))
        TSVD_TRY(sgemm_tc(g, w.splitk, sk * sizeof(CL), s, w.st));
      else
        TSVD_TRY(rmul_block<CL>(X, ldx, sX, Mi, b, sG, n1, nb, h, Y, ldy, sY, s));
    }
  }
  {
    TSVD_STAGE("orth_repair", s);
    TSVD_TRY(repair_dead<CL>(Q, m, sQ, n1, c, nb, w.dead, h, seed, block_id, w.dead_count, w.k0, w.nyq, s));
  }
  if (w.Qt) {
    TSVD_STAGE("convert", s);
    TSVD_TRY(convert_c64_to_c32((const double2*)Q + c, m, sQ, (float2*)w.Qt + c, m, sQ, n1, nb, h, s));
  }
  return TSVD_OK;
}

template int orth_block_cols<double>(int, int, int, int, const OrthWs&, int, int, int, uint64_t, cudaStream_t);
template int orth_block_cols<float>(int, int, int, int, const OrthWs&, int, int, int, uint64_t, cudaStream_t);

}  // namespace tsvd
