// fft.cu -- mode-3 transforms and the Gaussian test tensor.
//
// rFFT along mode 3 (Sec. 2, Definition of F_n: omega = exp(-2 pi i/n3),
// unnormalised) keeping the h = floor(n3/2)+1 non-redundant slices (Alg. TP),
// and its inverse from the half spectrum (the conjugate mirror of Alg. TP
// followed by F^{-1} = F^*/n3; the imaginary parts of the DC and Nyquist
// slices are ignored, i.e. the real part of the mirrored inverse).
//
// Layout: the plane index e = i*n2 + j runs fastest, so neighbouring threads own
// neighbouring tubes and every load and store is a contiguous run.  Which kernel:
//   n3 = 2, 4, .., 128      one thread (FP64, 128: two) per tube, in registers;
//   other n3 <= 160         folded direct products (FP64: where they take fewer
//                           operations than mixed-radix passes, rdft_better);
//   the rest                mixed-radix passes out of shared memory, and a direct
//                           sum for tubes too long for those.
#include "common.cuh"
#include "kernels.cuh"
#include "unit_circle.cuh"

namespace tsvd {

// omega^p with omega = exp(sign * 2 pi i / n); exact on the axes so that the DC
// and Nyquist slices of a real tensor come out exactly real.
template <typename T>
__device__ __forceinline__ cx_t<T> twiddle(int p, int n, int sign) {
  p %= n;
  if (p == 0) return mkc(T(1), T(0));
  if (2 * p == n) return mkc(T(-1), T(0));
  if (4 * p == n) return mkc(T(0), T(sign));
  if (4 * p == 3 * n) return mkc(T(0), T(-sign));
  if (sizeof(T) == sizeof(float)) {
    float s, c;
    sincospif(2.0f * (float)p / (float)n, &s, &c);
    return mkc((T)c, (T)(sign * s));
  }
  double s, c;
  sincospi(2.0 * (double)p / (double)n, &s, &c);
  return mkc((T)c, (T)(sign * s));
}

template <typename T>
__global__ void __launch_bounds__(256) k_rfft3(const T* __restrict__ X, cx_t<T>* __restrict__ Xh, long plane,
                                               int n3, int te) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using C = cx_t<T>;
  C* tw = (C*)smem_raw;          // [n3]
  T* xs = (T*)(tw + n3);         // [n3][te]
  const long e0 = (long)blockIdx.x * te;
  for (int p = threadIdx.x; p < n3; p += blockDim.x) tw[p] = twiddle<T>(p, n3, -1);
  for (int idx = threadIdx.x; idx < n3 * te; idx += blockDim.x) {
    const int t = idx / te, e = idx - t * te;
    const long ge = e0 + e;
    xs[idx] = (ge < plane) ? __ldg(X + (long)t * plane + ge) : T(0);
  }
  __syncthreads();
  const int h = n3 / 2 + 1;
  const int e = threadIdx.x % te, kg = threadIdx.x / te, nkg = blockDim.x / te;
  const long ge = e0 + e;
  for (int k = kg; k < h; k += nkg) {
    T re = 0, im = 0;
    int p = 0;
    for (int t = 0; t < n3; ++t) {
      const T x = xs[t * te + e];
      const C w = tw[p];
      re = fma(x, w.x, re);
      im = fma(x, w.y, im);
      p += k;
      if (p >= n3) p -= n3;
    }
    if (ge < plane) Xh[(long)k * plane + ge] = mkc(re, im);
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_irfft3(const cx_t<T>* __restrict__ Xh, T* __restrict__ X, long plane,
                                                int n3, int te) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using C = cx_t<T>;
  const int h = n3 / 2 + 1;
  C* tw = (C*)smem_raw;  // [n3]
  C* xs = tw + n3;       // [h][te]
  const long e0 = (long)blockIdx.x * te;
  for (int p = threadIdx.x; p < n3; p += blockDim.x) tw[p] = twiddle<T>(p, n3, +1);
  for (int idx = threadIdx.x; idx < h * te; idx += blockDim.x) {
    const int k = idx / te, e = idx - k * te;
    const long ge = e0 + e;
    xs[idx] = (ge < plane) ? Xh[(long)k * plane + ge] : mkc(T(0), T(0));
  }
  __syncthreads();
  const bool even = (n3 % 2) == 0;
  const int kint = even ? h - 1 : h;  // interior slices 1..kint-1 appear twice in the full spectrum
  const T inv = T(1) / T(n3);
  const int e = threadIdx.x % te, tg = threadIdx.x / te, ntg = blockDim.x / te;
  const long ge = e0 + e;
  for (int t = tg; t < n3; t += ntg) {
    T acc = xs[e].x;  // DC
    int p = t;
    for (int k = 1; k < kint; ++k) {
      const C x = xs[k * te + e];
      const C w = tw[p];
      acc = fma(T(2) * x.x, w.x, acc);
      acc = fma(T(-2) * x.y, w.y, acc);
      p += t;
      if (p >= n3) p -= n3;
    }
    if (even) {
      const T xn = xs[(h - 1) * te + e].x;
      acc += (t & 1) ? -xn : xn;
    }
    if (ge < plane) X[(long)t * plane + ge] = acc * inv;
  }
}

static int tile_e(int n3, size_t elem, size_t celem, bool inverse) {
  // largest power-of-two tile (<= 128, >= 32) whose shared footprint stays under 96 KB
  const int h = n3 / 2 + 1;
  for (int te = 128; te >= 32; te >>= 1) {
    size_t bytes = (size_t)n3 * celem + (size_t)(inverse ? h * celem : n3 * elem) * te;
    if (bytes <= 96 * 1024) return te;
  }
  return 32;
}

// ---------------------------------------------------------------------------
// Mixed-radix FFT of the tubes for the lengths above 160 and the smooth FP64 ones
// (Stockham autosort, radices 4, 2, 3, 5 and any remaining prime).  A CTA owns a tile of FFT_TUBES consecutive tubes;
// two real tubes are packed into one complex sequence z = x + i y and each warp
// transforms whole sequences in shared memory (lane-parallel butterflies,
// warp barriers between passes).  The half spectra are separated as
// X_k = (Z_k + conj Z_{n-k}) / 2, Y_k = (Z_k - conj Z_{n-k}) / (2i); the inverse
// packs Z = X + i Y over the full (Hermitian) spectrum.  Global reads and writes
// run along the plane index, so they stay coalesced.
// ---------------------------------------------------------------------------
constexpr int FFT_WARPS = 8;
constexpr int FFT_LOADS = 8;
constexpr int FFT_MAXR = 24;
// sequences a warp transforms together
constexpr int fft_seqs(int n) { return n < 1 ? 1 : (256 / n < 1 ? 1 : (256 / n > 4 ? 4 : 256 / n)); }
struct FftPlan {
  int n, nr, tubes;
  int seqs;  // sequences a warp transforms together (every pass has seqs * n / R independent butterflies)
  int radix[FFT_MAXR];
};

static bool make_plan(int n, FftPlan* p) {
  p->n = n;
  p->nr = 0;
  p->seqs = fft_seqs(n);
  int m = n;
  while (m % 4 == 0) { p->radix[p->nr++] = 4; m /= 4; }
  while (m % 2 == 0) { p->radix[p->nr++] = 2; m /= 2; }
  for (int f = 3; m > 1; f += 2) {
    while (m % f == 0) {
      if (p->nr >= FFT_MAXR) return false;
      p->radix[p->nr++] = f;
      m /= f;
    }
  }
  return true;
}

// one Stockham pass of radix R (sign of the exponent in tw): in -> out
template <typename C, int R>
__device__ __forceinline__ void fft_pass_fixed(const C* __restrict__ in0, C* __restrict__ out0,
                                               const C* __restrict__ tw, int n, int Ns, int lane, int nseq) {
  const int nR = n / R, tstep = n / (Ns * R);
  for (int jj = lane; jj < nseq * nR; jj += 32) {
    const int sq = jj / nR, j = jj - sq * nR;
    const C* __restrict__ in = in0 + sq * n;
    C* __restrict__ out = out0 + sq * n;
    const int k = j % Ns;
    C v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      v[r] = in[j + r * nR];
      if (r > 0) v[r] = cmul(v[r], tw[(r * k * tstep) % n]);
    }
    C o[R];
    if (R == 2) {
      o[0] = cadd(v[0], v[1]);
      o[1] = csub(v[0], v[1]);
    } else if (R == 4) {
      // omega_4 = tw[n/4] is exactly +-i
      const C w = tw[n / 4];
      const C a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
      const C c = cadd(v[1], v[3]), d = cmul(csub(v[1], v[3]), w);
      o[0] = cadd(a, c);
      o[2] = csub(a, c);
      o[1] = cadd(b, d);
      o[3] = csub(b, d);
    } else {
#pragma unroll
      for (int q = 0; q < R; ++q) {
        C acc = v[0];
#pragma unroll
        for (int r = 1; r < R; ++r) acc = cadd(acc, cmul(v[r], tw[((q * r) % R) * (n / R)]));
        o[q] = acc;
      }
    }
    const int idxD = (j / Ns) * Ns * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) out[idxD + r * Ns] = o[r];
  }
}

template <typename C>
__device__ void fft_pass_generic(const C* __restrict__ in0, C* __restrict__ out0, const C* __restrict__ tw, int n,
                                 int Ns, int R, int lane, int nseq) {
  const int nR = n / R, tstep = n / (Ns * R);
  for (int jj = lane; jj < nseq * nR; jj += 32) {
    const int sq = jj / nR, j = jj - sq * nR;
    const C* __restrict__ in = in0 + sq * n;
    C* __restrict__ out = out0 + sq * n;
    const int k = j % Ns;
    const int idxD = (j / Ns) * Ns * R + k;
    for (int q = 0; q < R; ++q) {
      C acc = in[j];
      for (int r = 1; r < R; ++r) {
        const C vr = cmul(in[j + r * nR], tw[(r * k * tstep) % n]);
        acc = cadd(acc, cmul(vr, tw[((q * r) % R) * (n / R)]));
      }
      out[idxD + q * Ns] = acc;
    }
  }
}

// in-place (ping-pong) FFT of nseq length-n sequences (stride n) in a / b;
// returns the buffer holding the result
template <typename C>
__device__ C* fft_run(C* a, C* b, const C* tw, const FftPlan& P, int lane, int nseq) {
  int Ns = 1;
  for (int s = 0; s < P.nr; ++s) {
    const int R = P.radix[s];
    if (R == 4) fft_pass_fixed<C, 4>(a, b, tw, P.n, Ns, lane, nseq);
    else if (R == 2) fft_pass_fixed<C, 2>(a, b, tw, P.n, Ns, lane, nseq);
    else if (R == 3) fft_pass_fixed<C, 3>(a, b, tw, P.n, Ns, lane, nseq);
    else if (R == 5) fft_pass_fixed<C, 5>(a, b, tw, P.n, Ns, lane, nseq);
    else fft_pass_generic<C>(a, b, tw, P.n, Ns, R, lane, nseq);
    __syncwarp();
    C* t = a;
    a = b;
    b = t;
    Ns *= R;
  }
  return a;
}

// tubes per CTA of the mixed-radix kernels: the widest tile that leaves room for three CTAs per
// SM, else the widest within 110 KB
constexpr size_t FFT_SMEM_3 = 72 * 1024, FFT_SMEM_MAX = 110 * 1024;
constexpr int fft_pick_tt(size_t s64, size_t s32, size_t s16) {
  return s64 <= FFT_SMEM_3 ? 64 : s32 <= FFT_SMEM_3 ? 32 : s16 <= FFT_SMEM_3 ? 16 :
         s64 <= FFT_SMEM_MAX ? 64 : s32 <= FFT_SMEM_MAX ? 32 : s16 <= FFT_SMEM_MAX ? 16 : 0;
}
template <typename T>
__global__ void __launch_bounds__(FFT_WARPS * 32) k_rfft3_fft(const T* __restrict__ X, cx_t<T>* __restrict__ Xh,
                                                              long plane, FftPlan P) {
  using C = cx_t<T>;
  extern __shared__ __align__(16) unsigned char fsm[];
  const int n = P.n, h = n / 2 + 1, TT = P.tubes;
  C* tw = (C*)fsm;                                  // [n]
  C* zb = tw + n;                                   // [FFT_WARPS][2][seqs][n]
  const int LD = TT + 1;                            // padded row stride: conflict-free column walks
  C* otile = zb + (size_t)FFT_WARPS * 2 * P.seqs * n;  // [h][LD] complex
  T* itile = (T*)(otile + (size_t)h * LD);          // [n][LD] real
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long e0 = (long)blockIdx.x * TT;
  for (int p = threadIdx.x; p < n; p += blockDim.x) tw[p] = twiddle<T>(p, n, -1);
  if (sizeof(T) == 4 && (plane & 3) == 0 && ((uintptr_t)X & 15) == 0 && e0 + TT <= plane) {
    // whole tile, FP32: 16-byte loads of four consecutive tubes, FFT_LOADS in flight per thread
    const int q4 = TT / 4, total = n * q4;
    for (int base = threadIdx.x; base < total; base += FFT_LOADS * blockDim.x) {
      float4 v[FFT_LOADS];
#pragma unroll
      for (int u = 0; u < FFT_LOADS; ++u) {
        const int idx = base + u * blockDim.x;
        const int t = idx / q4, e = 4 * (idx - t * q4);
        v[u] = (idx < total) ? __ldg((const float4*)(X + (long)t * plane + e0 + e)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < FFT_LOADS; ++u) {
        const int idx = base + u * blockDim.x;
        if (idx < total) {
          const int t = idx / q4, e = 4 * (idx - t * q4);
          T* d = itile + t * LD + e;
          d[0] = (T)v[u].x;
          d[1] = (T)v[u].y;
          d[2] = (T)v[u].z;
          d[3] = (T)v[u].w;
        }
      }
    }
  } else {
    // FFT_LOADS independent loads in flight per thread (memory-level parallelism)
    const int total = n * TT;
    for (int base = threadIdx.x; base < total; base += FFT_LOADS * blockDim.x) {
      T v[FFT_LOADS];
#pragma unroll
      for (int u = 0; u < FFT_LOADS; ++u) {
        const int idx = base + u * blockDim.x;
        const int t = idx / TT, e = idx - t * TT;
        const long ge = e0 + e;
        v[u] = (idx < total && ge < plane) ? __ldg(X + (long)t * plane + ge) : T(0);
      }
#pragma unroll
      for (int u = 0; u < FFT_LOADS; ++u) {
        const int idx = base + u * blockDim.x;
        if (idx < total) itile[(idx / TT) * LD + idx % TT] = v[u];
      }
    }
  }
  __syncthreads();
  const int B = P.seqs;
  C* za = zb + (size_t)warp * 2 * B * n;
  C* zc = za + (size_t)B * n;
  const T hf = T(0.5);
  for (int s0 = warp * B; s0 < TT / 2; s0 += FFT_WARPS * B) {
    const int nseq = min(B, TT / 2 - s0);
    for (int q = lane; q < nseq * n; q += 32) {
      const int sq = q / n, t = q - sq * n, s = s0 + sq;
      za[q] = mkc(itile[t * LD + 2 * s], itile[t * LD + 2 * s + 1]);
    }
    __syncwarp();
    const C* Z = fft_run<C>(za, zc, tw, P, lane, nseq);
    for (int q = lane; q < nseq * h; q += 32) {
      const int sq = q / h, k = q - sq * h, s = s0 + sq;
      const C zk = Z[sq * n + k], zn = Z[sq * n + (n - k) % n];
      otile[k * LD + 2 * s] = mkc(hf * (zk.x + zn.x), hf * (zk.y - zn.y));      // X_k
      otile[k * LD + 2 * s + 1] = mkc(hf * (zk.y + zn.y), hf * (zn.x - zk.x));  // Y_k
    }
    __syncwarp();
  }
  __syncthreads();
  if (sizeof(T) == 4 && (plane & 1) == 0 && ((uintptr_t)Xh & 15) == 0 && e0 + TT <= plane) {
    // whole tile, FP32: 16-byte stores of two consecutive complex values
    const int q2 = TT / 2;
    for (int idx = threadIdx.x; idx < h * q2; idx += blockDim.x) {
      const int k = idx / q2, e = 2 * (idx - k * q2);
      const C a = otile[k * LD + e], c = otile[k * LD + e + 1];
      *(float4*)(Xh + (long)k * plane + e0 + e) = make_float4((float)a.x, (float)a.y, (float)c.x, (float)c.y);
    }
  } else {
    for (int idx = threadIdx.x; idx < h * TT; idx += blockDim.x) {
      const int k = idx / TT, e = idx - k * TT;
      const long ge = e0 + e;
      if (ge < plane) Xh[(long)k * plane + ge] = otile[k * LD + e];
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(FFT_WARPS * 32) k_irfft3_fft(const cx_t<T>* __restrict__ Xh, T* __restrict__ X,
                                                               long plane, FftPlan P) {
  using C = cx_t<T>;
  extern __shared__ __align__(16) unsigned char fsm[];
  const int n = P.n, h = n / 2 + 1, TT = P.tubes;
  C* tw = (C*)fsm;                                  // [n]
  C* zb = tw + n;                                   // [FFT_WARPS][2][seqs][n]
  const int LD = TT + 1;                            // padded row stride: conflict-free column walks
  C* itile = zb + (size_t)FFT_WARPS * 2 * P.seqs * n;  // [h][LD] complex
  T* otile = (T*)(itile + (size_t)h * LD);          // [n][LD] real
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long e0 = (long)blockIdx.x * TT;
  for (int p = threadIdx.x; p < n; p += blockDim.x) tw[p] = twiddle<T>(p, n, +1);
  {
    const int total = h * TT;
    for (int base = threadIdx.x; base < total; base += FFT_LOADS * blockDim.x) {
      C v[FFT_LOADS];
#pragma unroll
      for (int u = 0; u < FFT_LOADS; ++u) {
        const int idx = base + u * blockDim.x;
        const int k = idx / TT, e = idx - k * TT;
        const long ge = e0 + e;
        v[u] = mkc(T(0), T(0));
        if (idx < total && ge < plane) v[u] = Xh[(long)k * plane + ge];
        if (k == 0 || 2 * k == n) v[u].y = T(0);  // c2r: the DC and Nyquist slices are real
      }
#pragma unroll
      for (int u = 0; u < FFT_LOADS; ++u) {
        const int idx = base + u * blockDim.x;
        if (idx < total) itile[(idx / TT) * LD + idx % TT] = v[u];
      }
    }
  }
  __syncthreads();
  const int B = P.seqs;
  C* za = zb + (size_t)warp * 2 * B * n;
  C* zc = za + (size_t)B * n;
  const T inv = T(1) / T(n);
  for (int s0 = warp * B; s0 < TT / 2; s0 += FFT_WARPS * B) {
    const int nseq = min(B, TT / 2 - s0);
    for (int q = lane; q < nseq * n; q += 32) {
      const int sq = q / n, k = q - sq * n, s = s0 + sq;
      C x, y;
      if (k < h) {
        x = itile[k * LD + 2 * s];
        y = itile[k * LD + 2 * s + 1];
      } else {
        x = cconj(itile[(n - k) * LD + 2 * s]);
        y = cconj(itile[(n - k) * LD + 2 * s + 1]);
      }
      za[q] = mkc(x.x - y.y, x.y + y.x);  // Z = X + i Y
    }
    __syncwarp();
    const C* z = fft_run<C>(za, zc, tw, P, lane, nseq);
    for (int q = lane; q < nseq * n; q += 32) {
      const int sq = q / n, t = q - sq * n, s = s0 + sq;
      otile[t * LD + 2 * s] = z[q].x * inv;
      otile[t * LD + 2 * s + 1] = z[q].y * inv;
    }
    __syncwarp();
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < n * TT; idx += blockDim.x) {
    const int t = idx / TT, e = idx - t * TT;
    const long ge = e0 + e;
    if (ge < plane) X[(long)t * plane + ge] = otile[t * LD + e];
  }
}

// ---------------------------------------------------------------------------
// Powers of two up to 64 (FP32: 128): one thread transforms one tube in its
// registers.  The n = 2 M real samples are the complex sequence
// z_j = x_2j + i x_2j+1; its M-point transform (radix 4, then 2, decimation in
// frequency, every index and twiddle a compile-time constant) is separated into
// the half spectrum with one rotation per pair of frequencies.  Neighbouring
// threads hold neighbouring tubes, so every load and store of a warp is one
// contiguous run and a thread has its n loads in flight together; nothing goes
// through shared memory, whose butterfly passes bounded the earlier kernel.
// Bound: the bytes in FP32 (n = 128, 512 x 512 plane: 110 -> 55 us forward, 147 ->
// 54 inverse, 40 us at the copy rate; 64: 56 -> 25, 73 -> 23, 20), the FP64 pipe
// in FP64 (64: 539 -> 341 us).
// ---------------------------------------------------------------------------
namespace ct {
// position of frequency k in the output of dif_fft<., M, .>
constexpr int pos(int k, int len) { return len <= 2 ? k : (k % 4) * (len / 4) + pos(k / 4, len / 4); }
}  // namespace ct

template <int V>
struct IntC {
  static constexpr int value = V;
};
template <int B, int E, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (B < E) {
    f(IntC<B>());
    static_for<B + 1, E>(static_cast<F&&>(f));
  }
}

// v <- v * exp(SGN 2 pi i p / n)
template <typename T, int SGN, int P, int N>
__device__ __forceinline__ cx_t<T> rot(cx_t<T> v) {
  if constexpr (P % N == 0) {
    return v;
  } else {
    constexpr T c = (T)ct::cos2pi(P, N), sn = (T)(SGN * ct::sin2pi(P, N));
    return mkc(v.x * c - v.y * sn, v.x * sn + v.y * c);
  }
}

template <typename T, int SGN, int M, int LEN = M>
__device__ __forceinline__ void dif_fft(cx_t<T> (&v)[M]) {
  using C = cx_t<T>;
  if constexpr (LEN >= 4) {
    constexpr int Q = LEN / 4;
    static_for<0, M / LEN>([&](auto b_) {
      static_for<0, Q>([&](auto j_) {
        constexpr int j = decltype(j_)::value, i0 = decltype(b_)::value * LEN + j;
        const C a = cadd(v[i0], v[i0 + 2 * Q]), b = csub(v[i0], v[i0 + 2 * Q]);
        const C c = cadd(v[i0 + Q], v[i0 + 3 * Q]), d = csub(v[i0 + Q], v[i0 + 3 * Q]);
        const C di = SGN < 0 ? mkc(d.y, -d.x) : mkc(-d.y, d.x);
        v[i0] = cadd(a, c);
        v[i0 + Q] = rot<T, SGN, j, LEN>(cadd(b, di));
        v[i0 + 2 * Q] = rot<T, SGN, 2 * j, LEN>(csub(a, c));
        v[i0 + 3 * Q] = rot<T, SGN, 3 * j, LEN>(csub(b, di));
      });
    });
    dif_fft<T, SGN, M, Q>(v);
  } else if constexpr (LEN == 2) {
    static_for<0, M / 2>([&](auto b_) {
      constexpr int i0 = 2 * decltype(b_)::value;
      const C a = v[i0], b = v[i0 + 1];
      v[i0] = cadd(a, b);
      v[i0 + 1] = csub(a, b);
    });
  }
}

template <typename T, int N>
__global__ void __launch_bounds__(128) k_rfft3_reg(const T* __restrict__ X, cx_t<T>* __restrict__ Xh, long plane) {
  using C = cx_t<T>;
  constexpr int M = N / 2;
  const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= plane) return;
  X += e;
  Xh += e;
  C v[M];
  static_for<0, M>([&](auto j_) {
    constexpr int j = decltype(j_)::value;
    v[j] = mkc(__ldg(X + (2 * j) * plane), __ldg(X + (2 * j + 1) * plane));
  });
  dif_fft<T, -1, M>(v);
  Xh[0] = mkc(v[0].x + v[0].y, T(0));
  Xh[M * plane] = mkc(v[0].x - v[0].y, T(0));
  static_for<1, M / 2 + 1>([&](auto k_) {
    constexpr int k = decltype(k_)::value;
    const C z = v[ct::pos(k, M)];
    if constexpr (2 * k == M) {
      Xh[k * plane] = mkc(z.x, -z.y);
    } else if constexpr (2 * k < M) {
      const C y = v[ct::pos(M - k, M)];
      const T hf = T(0.5);
      const C ev = mkc(hf * (z.x + y.x), hf * (z.y - y.y));
      const C od = rot<T, -1, k, N>(mkc(hf * (z.y + y.y), hf * (y.x - z.x)));
      Xh[k * plane] = cadd(ev, od);
      Xh[(M - k) * plane] = mkc(ev.x - od.x, od.y - ev.y);
    }
  });
}

template <typename T, int N>
__global__ void __launch_bounds__(128) k_irfft3_reg(const cx_t<T>* __restrict__ Xh, T* __restrict__ X, long plane) {
  using C = cx_t<T>;
  constexpr int M = N / 2;
  const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= plane) return;
  X += e;
  Xh += e;
  C v[M];
  {
    const T a = Xh[0].x, b = Xh[M * plane].x;  // the DC and Nyquist slices are real
    v[0] = mkc(a + b, a - b);
  }
  static_for<1, M / 2 + 1>([&](auto k_) {
    constexpr int k = decltype(k_)::value;
    const C x = Xh[k * plane];
    if constexpr (2 * k == M) {
      v[k] = mkc(T(2) * x.x, T(-2) * x.y);
    } else if constexpr (2 * k < M) {
      const C y = Xh[(M - k) * plane];
      const C ev = mkc(x.x + y.x, x.y - y.y);
      const C od = rot<T, +1, k, N>(mkc(x.x - y.x, x.y + y.y));
      v[k] = mkc(ev.x - od.y, ev.y + od.x);
      v[M - k] = mkc(ev.x + od.y, od.x - ev.y);
    }
  });
  dif_fft<T, +1, M>(v);
  constexpr T inv = T(1) / T(N);
  static_for<0, M>([&](auto j_) {
    constexpr int j = decltype(j_)::value;
    const C z = v[ct::pos(j, M)];
    X[(2 * j) * plane] = z.x * inv;
    X[(2 * j + 1) * plane] = z.y * inv;
  });
}

// FP64, n = 128: two threads per tube (16 lanes apart), each with the 64-point transform of every
// second sample in its registers (the whole tube would not fit): X_k = E_k + omega^k O_k and
// X_n/2-k = conj(E_k - omega^k O_k), E of the even and O of the odd samples, exchanged by shuffles.
template <typename T, int N>
__global__ void __launch_bounds__(128) k_rfft3_reg2(const T* __restrict__ X, cx_t<T>* __restrict__ Xh, long plane) {
  using C = cx_t<T>;
  constexpr int M = N / 4;  // complex points per thread
  const int odd = (threadIdx.x >> 4) & 1;
  const long e = ((long)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / 2 + (threadIdx.x & 15);
  const bool live = e < plane;
  X += (live ? e : 0) + odd * plane;
  Xh += live ? e : 0;
  C v[M];
  static_for<0, M>([&](auto j_) {
    constexpr int j = decltype(j_)::value;
    v[j] = mkc(__ldg(X + (4 * j) * plane), __ldg(X + (4 * j + 2) * plane));
  });
  dif_fft<T, -1, M>(v);
  // this thread's spectrum value f of frequency k: combined with its partner's, stored
  auto emit = [&](auto k_, C f) {
    constexpr int k = decltype(k_)::value;
    const C own = odd ? rot<T, -1, k, N>(f) : f;
    const C other = mkc(__shfl_xor_sync(0xffffffffu, own.x, 16), __shfl_xor_sync(0xffffffffu, own.y, 16));
    if (!live) return;
    if (!odd) Xh[k * plane] = mkc(own.x + other.x, k == 0 ? T(0) : own.y + other.y);
    else if constexpr (4 * k != N) Xh[(N / 2 - k) * plane] = mkc(other.x - own.x, k == 0 ? T(0) : own.y - other.y);
  };
  emit(IntC<0>(), mkc(v[0].x + v[0].y, T(0)));
  emit(IntC<M>(), mkc(v[0].x - v[0].y, T(0)));
  static_for<1, M / 2 + 1>([&](auto k_) {
    constexpr int k = decltype(k_)::value;
    const C z = v[ct::pos(k, M)];
    if constexpr (2 * k == M) {
      emit(k_, mkc(z.x, -z.y));
    } else if constexpr (2 * k < M) {
      const C y = v[ct::pos(M - k, M)];
      const T hf = T(0.5);
      const C ev = mkc(hf * (z.x + y.x), hf * (z.y - y.y));
      const C od = rot<T, -1, k, 2 * M>(mkc(hf * (z.y + y.y), hf * (y.x - z.x)));
      emit(k_, cadd(ev, od));
      emit(IntC<M - k>(), mkc(ev.x - od.x, od.y - ev.y));
    }
  });
}

template <typename T, int N>
__global__ void __launch_bounds__(128) k_irfft3_reg2(const cx_t<T>* __restrict__ Xh, T* __restrict__ X, long plane) {
  using C = cx_t<T>;
  constexpr int M = N / 4;
  const int odd = (threadIdx.x >> 4) & 1;
  const long e = ((long)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / 2 + (threadIdx.x & 15);
  if (e >= plane) return;
  Xh += e;
  X += e + odd * plane;
  // twice the spectrum of this thread's samples: X_k + conj X_n/2-k, or omega^-k (X_k - conj X_n/2-k)
  auto part = [&](auto k_) {
    constexpr int k = decltype(k_)::value;
    C a = Xh[k * plane], b = Xh[(N / 2 - k) * plane];
    if constexpr (k == 0) a.y = b.y = T(0);  // the DC and Nyquist slices are real
    const C od = rot<T, +1, k, N>(mkc(a.x - b.x, a.y + b.y));
    return odd ? od : mkc(a.x + b.x, a.y - b.y);
  };
  C v[M];
  {
    const T a = part(IntC<0>()).x, b = part(IntC<M>()).x;
    v[0] = mkc(a + b, a - b);
  }
  static_for<1, M / 2 + 1>([&](auto k_) {
    constexpr int k = decltype(k_)::value;
    const C x = part(k_);
    if constexpr (2 * k == M) {
      v[k] = mkc(T(2) * x.x, T(-2) * x.y);
    } else if constexpr (2 * k < M) {
      const C y = part(IntC<M - k>());
      const C ev = mkc(x.x + y.x, x.y - y.y);
      const C od = rot<T, +1, k, 2 * M>(mkc(x.x - y.x, x.y + y.y));
      v[k] = mkc(ev.x - od.y, ev.y + od.x);
      v[M - k] = mkc(ev.x + od.y, od.x - ev.y);
    }
  });
  dif_fft<T, +1, M>(v);
  constexpr T inv = T(1) / T(N);
  static_for<0, M>([&](auto j_) {
    constexpr int j = decltype(j_)::value;
    const C z = v[ct::pos(j, M)];
    X[(4 * j) * plane] = z.x * inv;
    X[(4 * j + 2) * plane] = z.y * inv;
  });
}

// ---------------------------------------------------------------------------
// Any other length up to RDFT_MAX: the half spectrum as a small real matrix
// product.  The samples are folded by symmetry while they are staged: for odd n
//   Re X_k = x_0 + sum_j P_j cos(j k tau/n),  Im X_k = -sum_j Q_j sin(j k tau/n),
//   P_j = x_j + x_n-j, Q_j = x_j - x_n-j, j = 1 .. (n-1)/2;
// for even n = 2m the even and the odd frequencies first separate into the sums
// s_j = x_j + x_j+m and differences d_j = x_j - x_j+m, each folded again (odd
// frequencies: P_j = d_j - d_m-j, Q_j = d_j + d_m-j), which halves the products:
// n/2 (odd n) or n/4 (even n) multiply-adds per sample, inside the time the
// bytes take in FP32.  The inverse runs the same table the other way: for each
// t the sums over even and odd k give the samples t, m-t, m+t and n-t.
// A thread holds KB frequencies of a vector of neighbouring tubes; each operand
// pair read from shared memory feeds 2 KB V multiply-adds.  Sums are taken in
// runs of 8 terms (their rounding then stays below a mixed-radix transform's).
// 512 x 512 plane, against the mixed-radix passes: FP32 n = 33 235 -> 23 us, 100
// 199 -> 81, 31 1446 -> 20 (prime radices ran serially), FP64 33 2304 -> 371;
// FP32 is bound by shared-memory reads (bytes alone: 31 us at n = 100), FP64 by its
// multiply-adds (1130 of 1480 us at n = 100).  The staging keeps eight 16-byte (or
// sixteen 4-byte) loads of a thread in flight: with eight of 4 bytes it took a
// third of the time (n = 33: 36 us, 100: 122).  Tubes 32 apart instead of
// neighbours, for planes whose rows are not aligned, gave no more (33: 44 -> 49).
// ---------------------------------------------------------------------------
constexpr int RDFT_MAX = 160;
template <typename T>
struct RVec;
// (64 tubes x 8 frequencies per warp and 256 threads measured slower: 121 -> 140 us at n = 100 with the former loads)
template <>
struct RVec<float> {
  using type = float4;
  static constexpr int V = 4, KB = 4, THREADS = 128;
};
template <>
struct RVec<double> {
  using type = double2;
  static constexpr int V = 2, KB = 4, THREADS = 128;
};
__device__ __forceinline__ void unpack(float4 v, float* o) { o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w; }
__device__ __forceinline__ void unpack(double2 v, double* o) { o[0] = v.x; o[1] = v.y; }

// KB consecutive twiddles (16-byte aligned) in 16-byte loads
template <int KB>
__device__ __forceinline__ void load_row(const float2* p, float2* o) {
#pragma unroll
  for (int q = 0; q < KB; q += 2) {
    const float4 v = *(const float4*)(p + q);
    o[q] = make_float2(v.x, v.y);
    o[q + 1] = make_float2(v.z, v.w);
  }
}
template <int KB>
__device__ __forceinline__ void load_row(const double2* p, double2* o) {
#pragma unroll
  for (int q = 0; q < KB; ++q) o[q] = p[q];
}

// the two halves of the folded problem (one for odd n)
struct RdftDims {
  int n, types, m, J, half, hc[2], hp[2], HP;
};
__host__ __device__ inline RdftDims rdft_dims(int n, int KB) {
  RdftDims d;
  d.n = n;
  d.types = (n % 2 == 0) ? 2 : 1;
  d.m = n / d.types;
  d.J = (d.m - 1) / 2;
  d.half = (d.m % 2 == 0) ? 1 : 0;  // a middle sample (only for even n)
  const int h = n / 2 + 1;
  d.hc[0] = d.types == 2 ? (h + 1) / 2 : h;
  d.hc[1] = d.types == 2 ? h / 2 : 0;
  for (int t = 0; t < 2; ++t) d.hp[t] = (d.hc[t] + KB - 1) / KB * KB;
  d.HP = d.hp[0] + d.hp[1];
  return d;
}

template <typename T>
__global__ void __launch_bounds__(RVec<T>::THREADS, 4) k_rdft3(const T* __restrict__ X, cx_t<T>* __restrict__ Xh, long plane,
                                                        int n, int lgE) {
  using C = cx_t<T>;
  using VT = typename RVec<T>::type;
  constexpr int V = RVec<T>::V, KB = RVec<T>::KB, THR = RVec<T>::THREADS;
  extern __shared__ __align__(16) unsigned char fsm[];
  const RdftDims d = rdft_dims(n, KB);
  const int J = d.J, m = d.m, rows = 2 * J + 2;  // per half: P_1..P_J, Q_1..Q_J, first, middle
  T* dat = (T*)fsm;                              // [types][rows][E]
  C* tab = (C*)(dat + ((size_t)d.types * rows << lgE));  // [J][HP]
  C* tw = tab + (size_t)J * d.HP;                   // [n]
  const int tid = threadIdx.x, E = 1 << lgE;
  for (int p = tid; p < n; p += THR) tw[p] = twiddle<T>(p, n, +1);
  __syncthreads();
  for (int i = tid; i < J * d.HP; i += THR) {
    const int j = i / d.HP + 1, c = i - (j - 1) * d.HP;
    const int t = c >= d.hp[0], q = c - (t ? d.hp[0] : 0);
    tab[i] = tw[(j * (d.types == 2 ? 2 * q + t : q)) % n];
  }
  // persistent CTAs: the table is made once for all the tiles a CTA takes
  for (long tile = blockIdx.x; (tile << lgE) < plane; tile += gridDim.x) {
    const long e0 = tile << lgE;
    __syncthreads();  // the previous tile's samples have been read
    auto ld = [&](int j, long ge) { return ge < plane ? __ldg(X + (long)j * plane + ge) : T(0); };
    // 16 bytes per load where the planes are aligned (W tubes), else one sample; 8 or 16 loads in flight
    auto fold = [&](auto w_) {
      constexpr int W = decltype(w_)::value;
      using VW = typename std::conditional<W == 1, T, VT>::type;
      constexpr int UB = W == 1 ? 8 : 4;  // items of two loads at a time
      const int lgW = lgE - (W == 4 ? 2 : W == 2 ? 1 : 0), items = J << lgW;
      auto get = [&](int j, long ge, T* o) {
        if (ge < plane) {
          const VW x = __ldg((const VW*)(X + (long)j * plane + ge));
          if constexpr (W == 1) o[0] = x;
          else unpack(x, o);
        } else {
#pragma unroll
          for (int q = 0; q < W; ++q) o[q] = T(0);
        }
      };
      auto put = [&](T* dst, const T* v) {
        if constexpr (W == 4) *(float4*)dst = make_float4(v[0], v[1], v[2], v[3]);
        else if constexpr (W == 2) *(double2*)dst = make_double2(v[0], v[1]);
        else dst[0] = v[0];
      };
      if (d.types == 1) {
        for (int i0 = tid; i0 < items; i0 += UB * THR) {
          T x[UB][2][W];
#pragma unroll
          for (int u = 0; u < UB; ++u) {
            const int i = min(i0 + u * THR, items - 1), j = (i >> lgW) + 1;
            const long ge = e0 + (i & ((1 << lgW) - 1)) * W;
            get(j, ge, x[u][0]);
            get(n - j, ge, x[u][1]);
          }
#pragma unroll
          for (int u = 0; u < UB; ++u) {
            const int i = i0 + u * THR;
            if (i >= items) break;
            T p[W], q[W];
#pragma unroll
            for (int k = 0; k < W; ++k) {
              p[k] = x[u][0][k] + x[u][1][k];
              q[k] = x[u][0][k] - x[u][1][k];
            }
            put(dat + (long)i * W, p);
            put(dat + J * E + (long)i * W, q);
          }
        }
      } else {
        T* o = dat + (size_t)rows * E;
        for (int i0 = tid; i0 < items; i0 += UB / 2 * THR) {
          T x[UB / 2][4][W];
#pragma unroll
          for (int u = 0; u < UB / 2; ++u) {
            const int i = min(i0 + u * THR, items - 1), j = (i >> lgW) + 1;
            const long ge = e0 + (i & ((1 << lgW) - 1)) * W;
            get(j, ge, x[u][0]);
            get(m - j, ge, x[u][1]);
            get(m + j, ge, x[u][2]);
            get(n - j, ge, x[u][3]);
          }
#pragma unroll
          for (int u = 0; u < UB / 2; ++u) {
            const int i = i0 + u * THR;
            if (i >= items) break;
            T p0[W], q0[W], p1[W], q1[W];
#pragma unroll
            for (int k = 0; k < W; ++k) {
              const T s0 = x[u][0][k] + x[u][2][k], s1 = x[u][1][k] + x[u][3][k];
              const T d0 = x[u][0][k] - x[u][2][k], d1 = x[u][1][k] - x[u][3][k];
              p0[k] = s0 + s1;
              q0[k] = s0 - s1;
              p1[k] = d0 - d1;
              q1[k] = d0 + d1;
            }
            put(dat + (long)i * W, p0);
            put(dat + J * E + (long)i * W, q0);
            put(o + (long)i * W, p1);
            put(o + J * E + (long)i * W, q1);
          }
        }
      }
    };
    if (plane % V == 0 && ((uintptr_t)X & 15) == 0) fold(IntC<V>());
    else fold(IntC<1>());
    for (int e = tid; e < E; e += THR) {
      const long ge = e0 + e;
      T* f0 = dat + 2 * J * E + e;
      if (d.types == 1) {
        f0[0] = ld(0, ge);
      } else {
        const T a = ld(0, ge), b = ld(m, ge);
        T* f1 = f0 + (size_t)rows * E;
        f0[0] = a + b;
        f1[0] = a - b;
        if (d.half) {
          const T c = ld(m / 2, ge), f = ld(m / 2 + m, ge);
          f0[E] = c + f;
          f1[E] = c - f;
        }
      }
    }
    __syncthreads();
    const int L = E / V, items = d.HP / KB * L;
    for (int it = tid; it < items; it += THR) {
      const int lane = it % L, c0 = it / L * KB;
      const int t = c0 >= d.hp[0];
      const T* P = dat + (size_t)t * rows * E + lane * V;
      const T* Q = P + J * E;
      T re[KB][V], im[KB][V];
      {
        T f[V], g[V];
        unpack(*(const VT*)(P + 2 * J * E), f);
#pragma unroll
        for (int u = 0; u < V; ++u) g[u] = T(0);
        if (d.half) unpack(*(const VT*)(P + (2 * J + 1) * E), g);
#pragma unroll
        for (int q = 0; q < KB; ++q) {
          // the middle sample: (-1)^k' on the real part (even frequencies) or on -Im (odd ones)
          const T sg = ((c0 - (t ? d.hp[0] : 0) + q) & 1) ? T(-1) : T(1);
#pragma unroll
          for (int u = 0; u < V; ++u) {
            re[q][u] = t ? f[u] : f[u] + sg * g[u];
            im[q][u] = t ? sg * g[u] : T(0);
          }
        }
      }
      const C* w = tab + c0;
      for (int j0 = 0; j0 < J; j0 += 8) {
        T sr[KB][V], si[KB][V];
#pragma unroll
        for (int q = 0; q < KB; ++q)
#pragma unroll
          for (int u = 0; u < V; ++u) sr[q][u] = si[q][u] = T(0);
        const int j1 = min(J, j0 + 8);
#pragma unroll 4
        for (int j = j0; j < j1; ++j) {
          T pv[V], qv[V];
          unpack(*(const VT*)(P + j * E), pv);
          unpack(*(const VT*)(Q + j * E), qv);
          C c[KB];
          load_row<KB>(w + (size_t)j * d.HP, c);
#pragma unroll
          for (int q = 0; q < KB; ++q)
#pragma unroll
            for (int u = 0; u < V; ++u) {
              sr[q][u] = fma(pv[u], c[q].x, sr[q][u]);
              si[q][u] = fma(qv[u], c[q].y, si[q][u]);
            }
        }
#pragma unroll
        for (int q = 0; q < KB; ++q)
#pragma unroll
          for (int u = 0; u < V; ++u) {
            re[q][u] += sr[q][u];
            im[q][u] += si[q][u];
          }
      }
      const int q0 = c0 - (t ? d.hp[0] : 0);
#pragma unroll
      for (int q = 0; q < KB; ++q) {
        if (q0 + q >= d.hc[t]) continue;
        const int k = d.types == 2 ? 2 * (q0 + q) + t : q0 + q;
        const long ge = e0 + lane * V;
        C* dst = Xh + (long)k * plane + ge;
        if (sizeof(T) == 4 && ge + V <= plane && ((uintptr_t)dst & 15) == 0) {
#pragma unroll
          for (int u = 0; u < V; u += 2)
            *(float4*)(dst + u) = make_float4((float)re[q][u], (float)-im[q][u], (float)re[q][u + 1],
                                              (float)-im[q][u + 1]);
        } else {
#pragma unroll
          for (int u = 0; u < V; ++u)
            if (ge + u < plane) dst[u] = mkc(re[q][u], -im[q][u]);
        }
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(RVec<T>::THREADS, 3) k_irdft3(const cx_t<T>* __restrict__ Xh, T* __restrict__ X,
                                                         long plane, int n, int lgE) {
  using C = cx_t<T>;
  using VT = typename RVec<T>::type;
  constexpr int V = RVec<T>::V, KB = RVec<T>::KB, THR = RVec<T>::THREADS;
  extern __shared__ __align__(16) unsigned char fsm[];
  const int types = (n % 2 == 0) ? 2 : 1, m = n / types;
  const int K = (n - 1) / 2;                       // interior frequencies 1 .. K
  const int K0 = types == 2 ? K / 2 : K;           // even ones (2, 4, ..) first, then the odd ones
  const int tc = m / 2 + 1, HP = (tc + KB - 1) / KB * KB;  // t = 0 .. m/2
  const int tid = threadIdx.x, E = 1 << lgE;
  T* dr = (T*)fsm;                                 // [K + 2][E] 2 Re X_k, then Re X_0, Re X_n/2
  T* di = dr + (size_t)(K + 2) * E;                // [K][E] 2 Im X_k
  C* tab = (C*)(di + (size_t)K * E);               // [K][HP]
  C* tw = tab + (size_t)K * HP;                    // [n]
  for (int p = tid; p < n; p += THR) tw[p] = twiddle<T>(p, n, +1);
  auto freq = [&](int r) { return types == 1 ? r + 1 : r < K0 ? 2 * r + 2 : 2 * (r - K0) + 1; };
  __syncthreads();
  for (int i = tid; i < K * HP; i += THR) {
    const int r = i / HP, t = i - r * HP;
    tab[i] = tw[(freq(r) * t) % n];
  }
  for (long tile = blockIdx.x; (tile << lgE) < plane; tile += gridDim.x) {
    const long e0 = tile << lgE;
    __syncthreads();  // the previous tile's samples have been read
    // FP32: two tubes per load where the planes are aligned; 8 loads in flight
    auto stage = [&](auto w_) {
      constexpr int W = decltype(w_)::value, UB = 8;
      const int lgW = lgE - (W == 2 ? 1 : 0), cnt = K << lgW;
      for (int i0 = tid; i0 < cnt; i0 += UB * THR) {
        C x[UB][W];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
          const int i = min(i0 + u * THR, cnt - 1);
          const long ge = e0 + (i & ((1 << lgW) - 1)) * W;
          const C* src = Xh + (long)freq(i >> lgW) * plane + ge;
          if constexpr (W == 2) {
            const float4 y = ge < plane ? *(const float4*)src : make_float4(0.f, 0.f, 0.f, 0.f);
            x[u][0] = mkc(T(y.x), T(y.y));
            x[u][1] = mkc(T(y.z), T(y.w));
          } else {
            x[u][0] = ge < plane ? *src : mkc(T(0), T(0));
          }
        }
#pragma unroll
        for (int u = 0; u < UB; ++u) {
          const int i = i0 + u * THR;
          if (i >= cnt) break;
#pragma unroll
          for (int k = 0; k < W; ++k) {
            dr[i * W + k] = T(2) * x[u][k].x;
            di[i * W + k] = T(2) * x[u][k].y;
          }
        }
      }
    };
    if (sizeof(T) == 4 && plane % 2 == 0 && ((uintptr_t)Xh & 15) == 0) stage(IntC<sizeof(T) == 4 ? 2 : 1>());
    else stage(IntC<1>());
    for (int e = tid; e < E; e += THR) {
      const long ge = e0 + e;
      dr[K * E + e] = ge < plane ? Xh[ge].x : T(0);
      dr[(K + 1) * E + e] = (types == 2 && ge < plane) ? Xh[(long)m * plane + ge].x : T(0);
    }
    __syncthreads();
    const T inv = T(1) / T(n);
    const int L = E / V, items = HP / KB * L;
    for (int it = tid; it < items; it += THR) {
      const int lane = it % L, t0 = it / L * KB;
      T a[2][KB][V], b[2][KB][V];  // sums over the even and the odd frequencies
      {
        T f[V], g[V];
        unpack(*(const VT*)(dr + (size_t)K * E + lane * V), f);
        unpack(*(const VT*)(dr + (size_t)(K + 1) * E + lane * V), g);
#pragma unroll
        for (int q = 0; q < KB; ++q) {
          const T sg = ((t0 + q) & 1) ? T(-1) : T(1);  // Nyquist: (-1)^t, with the frequencies of m's parity
#pragma unroll
          for (int u = 0; u < V; ++u) {
            a[0][q][u] = (m & 1) ? f[u] : f[u] + sg * g[u];
            a[1][q][u] = (m & 1) ? sg * g[u] : T(0);
            b[0][q][u] = b[1][q][u] = T(0);
          }
        }
      }
#pragma unroll
      for (int ty = 0; ty < 2; ++ty) {
        const int rb = ty ? K0 : 0, re = ty ? K : K0;
        for (int r0 = rb; r0 < re; r0 += 8) {
          T sr[KB][V], si[KB][V];
#pragma unroll
          for (int q = 0; q < KB; ++q)
#pragma unroll
            for (int u = 0; u < V; ++u) sr[q][u] = si[q][u] = T(0);
          const int r1 = min(re, r0 + 8);
#pragma unroll 4
          for (int r = r0; r < r1; ++r) {
            T pv[V], qv[V];
            unpack(*(const VT*)(dr + (size_t)r * E + lane * V), pv);
            unpack(*(const VT*)(di + (size_t)r * E + lane * V), qv);
            C c[KB];
            load_row<KB>(tab + (size_t)r * HP + t0, c);
#pragma unroll
            for (int q = 0; q < KB; ++q)
#pragma unroll
              for (int u = 0; u < V; ++u) {
                sr[q][u] = fma(pv[u], c[q].x, sr[q][u]);
                si[q][u] = fma(qv[u], c[q].y, si[q][u]);
              }
          }
#pragma unroll
          for (int q = 0; q < KB; ++q)
#pragma unroll
            for (int u = 0; u < V; ++u) {
              a[ty][q][u] += sr[q][u];
              b[ty][q][u] += si[q][u];
            }
        }
      }
      const long ge = e0 + lane * V;
      auto put = [&](int t, const T* v) {
        T* dst = X + (long)t * plane + ge;
        if (ge + V <= plane && ((uintptr_t)dst & (sizeof(VT) - 1)) == 0) {
          if constexpr (V == 4) *(float4*)dst = make_float4(v[0], v[1], v[2], v[3]);
          else *(double2*)dst = make_double2(v[0], v[1]);
        } else {
#pragma unroll
          for (int u = 0; u < V; ++u)
            if (ge + u < plane) dst[u] = v[u];
        }
      };
#pragma unroll
      for (int q = 0; q < KB; ++q) {
        const int t = t0 + q;
        if (t >= tc) continue;
        T v[V];
        if (types == 1) {
#pragma unroll
          for (int u = 0; u < V; ++u) v[u] = (a[0][q][u] - b[0][q][u]) * inv;
          put(t, v);
          if (t > 0) {
#pragma unroll
            for (int u = 0; u < V; ++u) v[u] = (a[0][q][u] + b[0][q][u]) * inv;
            put(n - t, v);
          }
          continue;
        }
#pragma unroll
        for (int u = 0; u < V; ++u) v[u] = ((a[0][q][u] + a[1][q][u]) - (b[0][q][u] + b[1][q][u])) * inv;
        put(t, v);
        if (2 * t < m) {
#pragma unroll
          for (int u = 0; u < V; ++u) v[u] = ((a[0][q][u] - a[1][q][u]) + (b[0][q][u] - b[1][q][u])) * inv;
          put(m - t, v);
        }
        if (t > 0) {
#pragma unroll
          for (int u = 0; u < V; ++u) v[u] = ((a[0][q][u] + a[1][q][u]) + (b[0][q][u] + b[1][q][u])) * inv;
          put(n - t, v);
          if (2 * t < m) {
#pragma unroll
            for (int u = 0; u < V; ++u) v[u] = ((a[0][q][u] - a[1][q][u]) - (b[0][q][u] - b[1][q][u])) * inv;
            put(m + t, v);
          }
        }
      }
    }
  }
}

// log2 of the tubes per tile: about 32 KB of samples, fewer where that would leave SMs idle (down to 32 tubes)
template <typename T>
static int rdft_tile(int n, long plane) {
  int lg = 9;
  while (lg > 6 && ((size_t)n * sizeof(T) << lg) > 34 * 1024) --lg;
  while (lg > 5 && cdiv(plane, 1 << lg) < 2 * SMS) --lg;
  return lg;
}
// persistent CTAs: as many per SM as registers (the launch bounds) and shared memory allow
static unsigned rdft_grid(long plane, int lgE, size_t smem, bool inverse) {
  const unsigned fit = std::max<unsigned>(1, 227 * 1024 / (unsigned)(smem + 1024));
  return std::min<unsigned>(cdiv(plane, 1L << lgE), SMS * std::min(fit, inverse ? 3u : 4u));
}
// FP64 arithmetic runs at 1/64 of FP32's rate, so there the operation count decides: picoseconds per
// sample of the two forms as measured on a 512 x 512 plane (the mixed-radix passes by radix; the
// folded product by n, and 100 = 4 5 5: 96 against 58, 128: 36 against 73).  In FP32 the folded
// product is the faster one at every length that is not a power of two (97: 106 us against 27 ms,
// 100: 81 against 199, 160: 163 against 346).
template <typename T>
static bool rdft_better(int n) {
  if (n < 3 || n > RDFT_MAX) return false;
  if (sizeof(T) == 4) return true;
  double passes = 0;
  int m = n;
  while (m % 4 == 0) { passes += 9; m /= 4; }
  while (m % 2 == 0) { passes += 8; m /= 2; }
  while (m % 3 == 0) { passes += 18; m /= 3; }
  while (m % 5 == 0) { passes += 42; m /= 5; }
  if (m > 1) return true;
  return n <= 128 && (n % 2 ? 1.13 : 0.57) * n < passes;
}
template <typename T>
static size_t rdft_smem(int n, int E, bool inverse) {
  constexpr int KB = RVec<T>::KB;
  const RdftDims d = rdft_dims(n, KB);
  if (!inverse)
    return sizeof(T) * (size_t)d.types * (2 * d.J + 2) * E + sizeof(cx_t<T>) * ((size_t)d.J * d.HP + n);
  const int K = (n - 1) / 2, HP = (d.m / 2 + KB) / KB * KB;
  return sizeof(T) * (size_t)(2 * K + 2) * E + sizeof(cx_t<T>) * ((size_t)K * HP + n);
}

// shared bytes of the FFT kernels for tile width tt (0 when the plan does not exist)
template <typename T>
static size_t fft_smem(int n, int tt, int seqs) {
  const int h = n / 2 + 1;
  return sizeof(cx_t<T>) * ((size_t)n + (size_t)FFT_WARPS * 2 * seqs * n + (size_t)h * (tt + 1)) +
         sizeof(T) * (size_t)n * (tt + 1);
}

template <typename T>
static bool fft_setup(int n, FftPlan* P, size_t* smem) {
  if (!make_plan(n, P)) return false;
  const int tt = fft_pick_tt(fft_smem<T>(n, 64, P->seqs), fft_smem<T>(n, 32, P->seqs), fft_smem<T>(n, 16, P->seqs));
  if (tt == 0) return false;
  P->tubes = tt;
  *smem = fft_smem<T>(n, tt, P->seqs);
  return true;
}

// threads per CTA of the register kernels: fewer where the plane would leave SMs idle
static int reg_fft_threads(long plane) { return cdiv(plane, 128) >= SMS ? 128 : cdiv(plane, 64) >= SMS ? 64 : 32; }

template <typename T>
int launch_rfft3(const T* X, cx_t<T>* Xh, long plane, int n3, cudaStream_t s) {
  if (plane <= 0) return TSVD_OK;
  {  // powers of two in registers
    auto go = [&](auto kern, int per_tube = 1) {
      const int thr = reg_fft_threads(plane);
      kern<<<cdiv(per_tube * plane, thr), thr, 0, s>>>(X, Xh, plane);
      TSVD_LAUNCHED();
      return TSVD_OK;
    };
    switch (n3) {
      case 2: return go(k_rfft3_reg<T, 2>);
      case 4: return go(k_rfft3_reg<T, 4>);
      case 8: return go(k_rfft3_reg<T, 8>);
      case 16: return go(k_rfft3_reg<T, 16>);
      case 32: return go(k_rfft3_reg<T, 32>);
      case 64: return go(k_rfft3_reg<T, 64>);
      case 128:
        if constexpr (sizeof(T) == 4) return go(k_rfft3_reg<T, 128>);
        else return go(k_rfft3_reg2<T, 128>, 2);
      default: break;
    }
  }
  if (rdft_better<T>(n3)) {
    const int lg = rdft_tile<T>(n3, plane);
    const size_t sm = rdft_smem<T>(n3, 1 << lg, false);
    if (sm > 48 * 1024) cudaFuncSetAttribute(k_rdft3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k_rdft3<T><<<rdft_grid(plane, lg, sm, false), RVec<T>::THREADS, sm, s>>>(X, Xh, plane, n3, lg);
    TSVD_LAUNCHED();
    return TSVD_OK;
  }
  FftPlan P;
  size_t smem;
  if (fft_setup<T>(n3, &P, &smem)) {
    if (smem > 48 * 1024) cudaFuncSetAttribute(k_rfft3_fft<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_rfft3_fft<T><<<cdiv(plane, P.tubes), FFT_WARPS * 32, smem, s>>>(X, Xh, plane, P);
    TSVD_LAUNCHED();
    return TSVD_OK;
  }
  // very long tubes: direct transform
  const int te = tile_e(n3, sizeof(T), sizeof(cx_t<T>), false);
  const size_t sm = (size_t)n3 * sizeof(cx_t<T>) + (size_t)n3 * te * sizeof(T);
  if (sm > 227 * 1024) return TSVD_ERR_UNSUPPORTED;
  if (sm > 48 * 1024) cudaFuncSetAttribute(k_rfft3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_rfft3<T><<<cdiv(plane, te), 256, sm, s>>>(X, Xh, plane, n3, te);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

template <typename T>
int launch_irfft3(const cx_t<T>* Xh, T* X, long plane, int n3, cudaStream_t s) {
  if (plane <= 0) return TSVD_OK;
  {
    auto go = [&](auto kern, int per_tube = 1) {
      const int thr = reg_fft_threads(plane);
      kern<<<cdiv(per_tube * plane, thr), thr, 0, s>>>(Xh, X, plane);
      TSVD_LAUNCHED();
      return TSVD_OK;
    };
    switch (n3) {
      case 2: return go(k_irfft3_reg<T, 2>);
      case 4: return go(k_irfft3_reg<T, 4>);
      case 8: return go(k_irfft3_reg<T, 8>);
      case 16: return go(k_irfft3_reg<T, 16>);
      case 32: return go(k_irfft3_reg<T, 32>);
      case 64: return go(k_irfft3_reg<T, 64>);
      case 128:
        if constexpr (sizeof(T) == 4) return go(k_irfft3_reg<T, 128>);
        else return go(k_irfft3_reg2<T, 128>, 2);
      default: break;
    }
  }
  if (rdft_better<T>(n3)) {
    const int lg = rdft_tile<T>(n3, plane);
    const size_t sm = rdft_smem<T>(n3, 1 << lg, true);
    if (sm > 48 * 1024) cudaFuncSetAttribute(k_irdft3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k_irdft3<T><<<rdft_grid(plane, lg, sm, true), RVec<T>::THREADS, sm, s>>>(Xh, X, plane, n3, lg);
    TSVD_LAUNCHED();
    return TSVD_OK;
  }
  FftPlan P;
  size_t smem;
  if (fft_setup<T>(n3, &P, &smem)) {
    if (smem > 48 * 1024) cudaFuncSetAttribute(k_irfft3_fft<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_irfft3_fft<T><<<cdiv(plane, P.tubes), FFT_WARPS * 32, smem, s>>>(Xh, X, plane, P);
    TSVD_LAUNCHED();
    return TSVD_OK;
  }
  const int h = n3 / 2 + 1;
  const int te = tile_e(n3, sizeof(T), sizeof(cx_t<T>), true);
  const size_t sm = (size_t)n3 * sizeof(cx_t<T>) + (size_t)h * te * sizeof(cx_t<T>);
  if (sm > 227 * 1024) return TSVD_ERR_UNSUPPORTED;
  if (sm > 48 * 1024) cudaFuncSetAttribute(k_irfft3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_irfft3<T><<<cdiv(plane, te), 256, sm, s>>>(Xh, X, plane, n3, te);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

template <typename T>
int load_transforms() {
  int rc = TSVD_OK;
  auto load = [&](auto forward, auto inverse) {
    if (rc == TSVD_OK) rc = load_kernel(forward);
    if (rc == TSVD_OK) rc = load_kernel(inverse);
  };
  load(k_rfft3_reg<T, 2>, k_irfft3_reg<T, 2>);
  load(k_rfft3_reg<T, 4>, k_irfft3_reg<T, 4>);
  load(k_rfft3_reg<T, 8>, k_irfft3_reg<T, 8>);
  load(k_rfft3_reg<T, 16>, k_irfft3_reg<T, 16>);
  load(k_rfft3_reg<T, 32>, k_irfft3_reg<T, 32>);
  load(k_rfft3_reg<T, 64>, k_irfft3_reg<T, 64>);
  if constexpr (sizeof(T) == 4) load(k_rfft3_reg<T, 128>, k_irfft3_reg<T, 128>);
  else load(k_rfft3_reg2<T, 128>, k_irfft3_reg2<T, 128>);
  load(k_rdft3<T>, k_irdft3<T>);
  load(k_rfft3_fft<T>, k_irfft3_fft<T>);
  load(k_rfft3<T>, k_irfft3<T>);
  return rc;
}
template int load_transforms<double>();
template int load_transforms<float>();

template int launch_rfft3<double>(const double*, double2*, long, int, cudaStream_t);
template int launch_rfft3<float>(const float*, float2*, long, int, cudaStream_t);
template int launch_irfft3<double>(const double2*, double*, long, int, cudaStream_t);
template int launch_irfft3<float>(const float2*, float*, long, int, cudaStream_t);

// Element e of stream (seed, stream_id, tensor_id) is Box-Muller output e%4 of
// Philox call e/4; the two uniforms of a pair are (x + 1) 2^-32 in (0, 1].
template <typename T>
__global__ void k_gaussian(uint64_t seed, uint32_t stream_id, uint32_t tensor_id, long n, T* __restrict__ out) {
  const long call = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (4 * call >= n) return;
  const uint4 x = philox10(make_uint4((uint32_t)call, (uint32_t)((unsigned long long)call >> 32), stream_id, tensor_id),
                           (uint32_t)seed, (uint32_t)(seed >> 32));
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
  for (int pair = 0; pair < 2; ++pair) {
    const long e = 4 * call + 2 * pair;
    T g0, g1;
    if constexpr (sizeof(T) == sizeof(float)) {
      // FP32 stream: the same definition evaluated in FP32 (its values are FP32 anyway; FP64
      // transcendentals run at 1/64 of the FP32 rate here)
      const float u1 = fmaf((float)w[2 * pair], 0x1p-32f, 0x1p-32f);
      const float u2 = fmaf((float)w[2 * pair + 1], 0x1p-32f, 0x1p-32f);
      const float r = sqrtf(-2.0f * logf(u1));
      float sn, cs;
      sincospif(2.0f * u2, &sn, &cs);
      g0 = r * cs;
      g1 = r * sn;
    } else {
      const double inv32 = 1.0 / 4294967296.0;
      const double u1 = ((double)w[2 * pair] + 1.0) * inv32;
      const double u2 = ((double)w[2 * pair + 1] + 1.0) * inv32;
      const double r = sqrt(-2.0 * log(u1));
      const double th = 2.0 * 3.141592653589793 * u2;
      g0 = (T)(r * cos(th));
      g1 = (T)(r * sin(th));
    }
    if (e < n) out[e] = g0;
    if (e + 1 < n) out[e + 1] = g1;
  }
}

__global__ void k_philox_words(uint32_t k0, uint32_t k1, uint32_t c1, uint32_t c2, uint32_t c3, long n,
                               uint32_t* __restrict__ out) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 x = philox10(make_uint4((uint32_t)i, c1, c2, c3), k0, k1);
  out[4 * i + 0] = x.x;
  out[4 * i + 1] = x.y;
  out[4 * i + 2] = x.z;
  out[4 * i + 3] = x.w;
}

template <typename T>
int launch_gaussian(uint64_t seed, uint32_t stream_id, uint32_t tensor_id, long n, T* out, cudaStream_t s) {
  if (n <= 0) return TSVD_OK;
  const long calls = (n + 3) / 4;
  k_gaussian<T><<<cdiv(calls, 256), 256, 0, s>>>(seed, stream_id, tensor_id, n, out);
  TSVD_LAUNCHED();
  return TSVD_OK;
}
template int launch_gaussian<double>(uint64_t, uint32_t, uint32_t, long, double*, cudaStream_t);
template int launch_gaussian<float>(uint64_t, uint32_t, uint32_t, long, float*, cudaStream_t);

}  // namespace tsvd

extern "C" int tsvd_gaussian(uint64_t seed, uint32_t stream_id, uint32_t tensor_id, long n, double* out,
                             void* stream) {
  if (n < 0 || (n > 0 && !out)) return TSVD_ERR_INVALID_ARG;
  return tsvd::launch_gaussian<double>(seed, stream_id, tensor_id, n, out, (cudaStream_t)stream);
}

extern "C" int tsvd_philox_words(const uint32_t key[2], uint32_t ctr1, uint32_t ctr2, uint32_t ctr3, long n,
                                 uint32_t* out, void* stream) {
  if (!key || n < 0 || (n > 0 && !out)) return TSVD_ERR_INVALID_ARG;
  if (n == 0) return TSVD_OK;
  tsvd::k_philox_words<<<tsvd::cdiv(n, 256), 256, 0, (cudaStream_t)stream>>>(key[0], key[1], ctr1, ctr2, ctr3, n, out);
  TSVD_LAUNCHED();
  return TSVD_OK;
}

// The mode-3 transforms on their own (Sec. 2, Def. of F_n; Alg. TP first and
// last lines), for callers that move Fourier slices between devices.
extern "C" int tsvd_rfft3(const void* X, long plane, int n3, int precision, void* Xhat, void* stream) {
  if (!X || !Xhat || plane < 1 || n3 < 1) return TSVD_ERR_INVALID_ARG;
  if (precision == TSVD_FP64)
    return tsvd::launch_rfft3<double>((const double*)X, (double2*)Xhat, plane, n3, (cudaStream_t)stream);
  if (precision == TSVD_FP32)
    return tsvd::launch_rfft3<float>((const float*)X, (float2*)Xhat, plane, n3, (cudaStream_t)stream);
  return TSVD_ERR_INVALID_ARG;
}

extern "C" int tsvd_irfft3(const void* Xhat, long plane, int n3, int precision, void* X, void* stream) {
  if (!X || !Xhat || plane < 1 || n3 < 1) return TSVD_ERR_INVALID_ARG;
  if (precision == TSVD_FP64)
    return tsvd::launch_irfft3<double>((const double2*)Xhat, (double*)X, plane, n3, (cudaStream_t)stream);
  if (precision == TSVD_FP32)
    return tsvd::launch_irfft3<float>((const float2*)Xhat, (float*)X, plane, n3, (cudaStream_t)stream);
  return TSVD_ERR_INVALID_ARG;
}
