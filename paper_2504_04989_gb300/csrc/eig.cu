// eig.cu -- the Hermitian eigen-solve behind the small SVD of Alg. 2
// ([U_c, S_c, V_c] = T-SVD(C) with C = Q^H X per Fourier slice): with
// G = C C^H = U_c S_c^2 U_c^H, the R largest eigenpairs of the m x m G give
// sigma_i = sqrt(lambda_i) and U_c(:, 1:R).
//
//   1. Householder reduction to tridiagonal form, T' = H_{m-2}..H_0 G H_0..H_{m-2};
//      a cluster of CTAs shares each slice's rows (FP64 is the bound, so the
//      work of one slice is spread over several SMs).
//   2. T = D^H T' D real symmetric (D diagonal unitary); bisection on Sturm
//      counts (a division-free three-term recurrence) for the R largest
//      eigenvalues, inverse iteration with a partially pivoted LU for the
//      vectors, two classical Gram-Schmidt passes inside clusters of close
//      eigenvalues.
//   3. u_r = H_0 .. H_{m-2} D z_r.
#include <cooperative_groups.h>
#include <float.h>

#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace tsvd {

struct EigScratch {
  double* d;       // [batch][m] diagonal of T
  double* f;       // [batch][m] off-diagonal |alpha_j|
  double2* alpha;  // [batch][m] complex off-diagonals of T'
  double2* delta;  // [batch][m] phases making T real
  double2* Hv;     // [batch][m][m] Householder vectors (row j, columns j+1..m-1)
  double* Z;       // [batch][R][m] real eigenvectors of T (vector-contiguous)
  double* lu;      // [batch][5][m][R] inverse-iteration LU factors
  double* tnorm;   // [batch]
  double2* Sg;     // packed own rows of the cluster reduction when they do not fit in shared memory
  double2* Cp;     // the warps' partials of p where they do not
};

// ---------------------------------------------------------------------------
// Householder tridiagonalisation: a cluster of CL CTAs (one per SM) holds the
// lower triangle of one slice, row g in CTA g mod CL.
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ int hs_own_rows(int m, int c, int CL) { return (c < m) ? (m - 1 - c) / CL + 1 : 0; }
__host__ __device__ __forceinline__ int hs_rowbase(int q, int c, int CL) { return q * (c + 1) + CL * q * (q - 1) / 2; }
// first own row index q with c + CL q > j
__host__ __device__ __forceinline__ int hs_qfirst(int j, int c, int CL) { return (j < c) ? 0 : (j - c) / CL + 1; }

static size_t hetrd_row_elems(int m, int CL) {  // packed own rows of the CTA that has most
  int mx = 0;
  for (int c = 0; c < CL; ++c) mx = std::max(mx, hs_rowbase(hs_own_rows(m, c, CL), c, CL));
  return (size_t)mx;
}

// ---------------------------------------------------------------------------
// Double-float arithmetic of the FP32 path's eigen-solver: unevaluated pairs
// (hi, lo) of floats (about 48 significant bits) built from the error-free
// transformations TwoSum (Knuth) and TwoProduct via FMA (Dekker).  GB300
// issues FP32 at 64x its FP64 rate, so a multiply-add of about 15 FP32
// instructions replaces one DFMA at 1/64 of the rate.  G is first scaled by a
// power of two so its entries stay far inside the FP32 exponent range; the
// rounding level (about 2^-47 ||G|| per operation) is far below what the FP32
// path's accuracy needs.
// ---------------------------------------------------------------------------
struct __align__(8) dfl {
  float hi, lo;
};
struct __align__(16) cdf {  // complex double-float, 16 bytes like double2 (one 16-byte access)
  float rh, rl, ih, il;
};

__device__ __forceinline__ dfl df_two_sum(float a, float b) {
  const float s = a + b, bb = s - a;
  return dfl{s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ dfl df_fast_two_sum(float a, float b) {  // |a| >= |b| or a == 0
  const float s = a + b;
  return dfl{s, b - (s - a)};
}
// a + x y
__device__ __forceinline__ dfl df_fma(dfl a, dfl x, dfl y) {
  const float p = x.hi * y.hi;
  float e = fmaf(x.hi, y.hi, -p);
  e = fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, e));
  const dfl s = df_two_sum(a.hi, p);
  return df_fast_two_sum(s.hi, s.lo + (a.lo + e));
}
__device__ __forceinline__ dfl df_add(dfl a, dfl b) {
  const dfl s = df_two_sum(a.hi, b.hi);
  return df_fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}
__device__ __forceinline__ dfl df_neg(dfl a) { return dfl{-a.hi, -a.lo}; }
__device__ __forceinline__ dfl df_mul(dfl a, dfl b) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  return df_fast_two_sum(p, e);
}
// square root: correctly rounded FP32 root, then one correction with the
// exactly computed residual a - x^2 (about 46 correct bits)
__device__ __forceinline__ dfl df_sqrt(dfl a) {
  if (!(a.hi > 0.f)) return dfl{0.f, 0.f};
  const float x = sqrtf(a.hi);
  const float p = x * x, pe = fmaf(x, x, -p);
  const float r = ((a.hi - p) - pe) + a.lo;
  return df_fast_two_sum(x, r / (2.f * x));
}
// Reciprocal square root and square root without a division: the correctly
// rounded FP32 reciprocal square root y, then one Newton correction with the
// residual formed in double-float (y (1 + e/2), e = 1 - a y^2; for the root,
// x = a_hi y and x + y (a - x^2) / 2 with a - x^2 exact by FMA).  About 46
// correct bits from a 24-bit start.  a > 0.
__device__ __forceinline__ dfl df_rsqrt(dfl a) {
  const float y = __frsqrt_rn(a.hi);
  const float p = y * y, pe = fmaf(y, y, -p);  // y^2 = p + pe exactly
  const dfl ay2 = df_mul(a, dfl{p, pe});
  const float e = (1.0f - ay2.hi) - ay2.lo;    // 1 - a y^2 (1 - ay2.hi exact: ay2.hi is within 2^-22 of 1)
  return df_fast_two_sum(y, 0.5f * y * e);
}
__device__ __forceinline__ dfl df_sqrt_nodiv(dfl a) {
  if (!(a.hi > 0.f)) return dfl{0.f, 0.f};
  const float y = __frsqrt_rn(a.hi);
  const float x = a.hi * y;
  const float r = (fmaf(-x, x, a.hi)) + a.lo;  // a - x^2 (the high part exact by FMA)
  return df_fast_two_sum(x, 0.5f * y * r);
}
__device__ __forceinline__ dfl df_from(double x) {
  const float h = (float)x;
  return dfl{h, (float)(x - (double)h)};
}
__device__ __forceinline__ double df_to(dfl a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ dfl cre(cdf a) { return dfl{a.rh, a.rl}; }
__device__ __forceinline__ dfl cim(cdf a) { return dfl{a.ih, a.il}; }
__device__ __forceinline__ cdf cdf_make(dfl r, dfl i) { return cdf{r.hi, r.lo, i.hi, i.lo}; }
__device__ __forceinline__ cdf cdf_from(double2 x) { return cdf_make(df_from(x.x), df_from(x.y)); }
__device__ __forceinline__ cdf cdf_zero() { return cdf{0.f, 0.f, 0.f, 0.f}; }
__device__ __forceinline__ cdf cdf_add(cdf a, cdf b) { return cdf_make(df_add(cre(a), cre(b)), df_add(cim(a), cim(b))); }
// acc += a b
// a + sum_i x_i y_i with one renormalisation at the end: each exact product
// (TwoProduct by FMA plus the two cross terms) is added to the running high
// part by TwoSum and every rounding error goes to one low accumulator (the
// compensated dot product of Ogita, Rump and Oishi in double-float form).
template <int N>
__device__ __forceinline__ dfl df_dot(dfl a, const dfl (&x)[N], const dfl (&y)[N]) {
  float s = a.hi, e = a.lo;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float p = x[i].hi * y[i].hi;
    float pe = fmaf(x[i].hi, y[i].hi, -p);
    pe = fmaf(x[i].hi, y[i].lo, fmaf(x[i].lo, y[i].hi, pe));
    const float t = s + p, bb = t - s;
    e += ((s - (t - bb)) + (p - bb)) + pe;
    s = t;
  }
  return df_fast_two_sum(s, e);
}
// acc += a b and acc += conj(a) b with acc kept unnormalised: the high words
// carry the running sums, the low words every rounding error (the loop of
// df_dot without its final renormalisation, which cdf_add does later)
__device__ __forceinline__ void df_acc(float& s, float& e, float xh, float xl, float yh, float yl) {
  const float p = xh * yh;
  float pe = fmaf(xh, yh, -p);
  pe = fmaf(xh, yl, fmaf(xl, yh, pe));
  const float t = s + p, bb = t - s;
  e += ((s - (t - bb)) + (p - bb)) + pe;
  s = t;
}
__device__ __forceinline__ void cdf_fma_acc(cdf& acc, cdf a, cdf b) {
  df_acc(acc.rh, acc.rl, a.rh, a.rl, b.rh, b.rl);
  df_acc(acc.rh, acc.rl, -a.ih, -a.il, b.ih, b.il);
  df_acc(acc.ih, acc.il, a.rh, a.rl, b.ih, b.il);
  df_acc(acc.ih, acc.il, a.ih, a.il, b.rh, b.rl);
}
__device__ __forceinline__ void cdf_fmac_acc(cdf& acc, cdf a, cdf b) {
  df_acc(acc.rh, acc.rl, a.rh, a.rl, b.rh, b.rl);
  df_acc(acc.rh, acc.rl, a.ih, a.il, b.ih, b.il);
  df_acc(acc.ih, acc.il, a.rh, a.rl, b.ih, b.il);
  df_acc(acc.ih, acc.il, -a.ih, -a.il, b.rh, b.rl);
}
// a - vg conj(wk) - wg conj(vk)
__device__ __forceinline__ cdf cdf_lag(cdf a, cdf vg, cdf wg, cdf vk, cdf wk) {
  const dfl xr[4] = {df_neg(cre(vg)), df_neg(cim(vg)), df_neg(cre(wg)), df_neg(cim(wg))};
  const dfl yr[4] = {cre(wk), cim(wk), cre(vk), cim(vk)};
  const dfl xi[4] = {df_neg(cim(vg)), cre(vg), df_neg(cim(wg)), cre(wg)};
  const dfl yi[4] = {cre(wk), cim(wk), cre(vk), cim(vk)};
  return cdf_make(df_dot<4>(cre(a), xr, yr), df_dot<4>(cim(a), xi, yi));
}
// x * s for a real double-float s
__device__ __forceinline__ cdf cdf_scale(cdf x, dfl s) {
  const dfl z{0.f, 0.f};
  return cdf_make(df_fma(z, cre(x), s), df_fma(z, cim(x), s));
}
__device__ __forceinline__ dfl df_shfl_xor(dfl a, int o) {
  return dfl{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}
__device__ __forceinline__ cdf cdf_shfl_xor(cdf a, int o) {
  return cdf{__shfl_xor_sync(0xffffffffu, a.rh, o), __shfl_xor_sync(0xffffffffu, a.rl, o),
             __shfl_xor_sync(0xffffffffu, a.ih, o), __shfl_xor_sync(0xffffffffu, a.il, o)};
}
// ---------------------------------------------------------------------------
// The reduction, for cdf (double-float, FP32 path) and double2 (FP64 path).
// Step j (A^(j) = the matrix after j reflectors; the stored rows S lag one
// update behind, S = A^(j-1) on the trailing block; v', w' of step j-1):
//   w' = p' - K v',  K = Re(v'^H p')
//   x = S(:,j) - v' conj(w'_j) - w' conj(v'_j)
//   alpha = -e^{i arg x_0} ||x||,  v = (x - alpha e_1) / ||x - alpha e_1||
//   S(g,k) <- S(g,k) - v'_g conj(w'_k) - w'_g conj(v'_k)   (k <= g, both > j)
//   p = 2 A^(j) v from the lower triangle: row part sum_k S(g,k) v_k and
//       column part sum_g conj(S(g,k)) v_g
// One sweep per step does the update, the store and both parts, and sends the
// updated column j+1 to every CTA of the cluster, so that after the one
// cluster barrier of the step each CTA has the parts of p and the next column
// and goes on alone (the same sums in the same order in every CTA).
//
// Warp w takes every NW-th own row from the last but w on, in strips of HF_SR
// and 32 columns at a time with lane l on column k0 + l: every load is one
// contiguous 512-byte run, the row sums stay in the lane until the strip's
// end, the column sums go to a partial of p private to the warp.  Every sum
// has one order, so reruns agree bitwise.  Rows sit in shared memory where
// they fit, else in a private part of a global array (L2), read 32 columns
// ahead; the warps' partials likewise (`cp_global`).
//
// Bound: in double-float its instructions (about 200 of FP32 per element and
// step) and, per step, a chain of two block sums, the reflector's scalars and a
// cluster barrier (7 to 9 of 14 us at m = 300 in the three-sweep form this
// replaces, about 4 of 11 here); in FP64 its pipe (16 multiply-adds per element
// and step).  Two rows' chains interleave without branches on the lane (all
// eight in turn: 3692 us at m = 300, two at a time 3405, four 3400).  Against
// the former kernels, us: double-float m = 45 on 9 slices 350 -> 215, 135 on 33
// 1420 -> 816, 300 on 33 4363 -> 3405, 480 on 65 (rows in L2) 17330 -> 16500;
// FP64 45 on 9 623 -> 346, 300 on 33 9318 -> 8090, 480 on 9 34880 -> 15650.
// ---------------------------------------------------------------------------

constexpr int HETRD_NT = 256;  // threads (m = 300 on 33 slices in double-float: 512 threads 3764 us, 256 3405)

// operations the kernel takes from its arithmetic
__device__ __forceinline__ dfl r_zero(dfl) { return dfl{0.f, 0.f}; }
__device__ __forceinline__ double r_zero(double) { return 0.0; }
__device__ __forceinline__ cdf c_zero(cdf) { return cdf_zero(); }
__device__ __forceinline__ double2 c_zero(double2) { return make_double2(0.0, 0.0); }
__device__ __forceinline__ cdf c_one(cdf) { return cdf{1.f, 0.f, 0.f, 0.f}; }
__device__ __forceinline__ double2 c_one(double2) { return make_double2(1.0, 0.0); }
__device__ __forceinline__ dfl r_add(dfl a, dfl b) { return df_add(a, b); }
__device__ __forceinline__ double r_add(double a, double b) { return a + b; }
__device__ __forceinline__ dfl r_neg(dfl a) { return df_neg(a); }
__device__ __forceinline__ double r_neg(double a) { return -a; }
__device__ __forceinline__ dfl r_fma(dfl a, dfl x, dfl y) { return df_fma(a, x, y); }
__device__ __forceinline__ double r_fma(double a, double x, double y) { return fma(x, y, a); }
__device__ __forceinline__ dfl r_mul(dfl a, dfl b) { return df_mul(a, b); }
__device__ __forceinline__ double r_mul(double a, double b) { return a * b; }
__device__ __forceinline__ bool r_pos(dfl a) { return a.hi > 0.f; }
__device__ __forceinline__ bool r_pos(double a) { return a > 0.0; }
__device__ __forceinline__ dfl r_rsqrt(dfl a) { return df_rsqrt(a); }
__device__ __forceinline__ double r_rsqrt(double a) { return inv_sqrt(a); }
__device__ __forceinline__ dfl r_sqrt(dfl a) { return df_sqrt_nodiv(a); }
__device__ __forceinline__ double r_sqrt(double a) { return a * inv_sqrt(a); }
__device__ __forceinline__ dfl r_shfl(dfl a, int o) { return df_shfl_xor(a, o); }
__device__ __forceinline__ double r_shfl(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ double r_double(dfl a) { return df_to(a); }
__device__ __forceinline__ double r_double(double a) { return a; }
__device__ __forceinline__ double cre(double2 a) { return a.x; }
__device__ __forceinline__ double cim(double2 a) { return a.y; }
__device__ __forceinline__ cdf c_make(dfl r, dfl i) { return cdf_make(r, i); }
__device__ __forceinline__ double2 c_make(double r, double i) { return make_double2(r, i); }
__device__ __forceinline__ cdf c_add(cdf a, cdf b) { return cdf_add(a, b); }
__device__ __forceinline__ double2 c_add(double2 a, double2 b) { return cadd(a, b); }
__device__ __forceinline__ cdf c_twice(cdf a) { return cdf{2.f * a.rh, 2.f * a.rl, 2.f * a.ih, 2.f * a.il}; }
__device__ __forceinline__ double2 c_twice(double2 a) { return make_double2(2.0 * a.x, 2.0 * a.y); }
__device__ __forceinline__ void c_real(cdf& a) { a.ih = a.il = 0.f; }
__device__ __forceinline__ void c_real(double2& a) { a.y = 0.0; }
__device__ __forceinline__ cdf c_shfl(cdf a, int o) { return cdf_shfl_xor(a, o); }
__device__ __forceinline__ double2 c_shfl(double2 a, int o) {
  return make_double2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
}
__device__ __forceinline__ cdf c_scale_r(cdf a, dfl s) { return cdf_scale(a, s); }
__device__ __forceinline__ double2 c_scale_r(double2 a, double s) { return cscale(a, s); }
__device__ __forceinline__ cdf c_lag(cdf a, cdf vg, cdf wg, cdf vk, cdf wk) { return cdf_lag(a, vg, wg, vk, wk); }
__device__ __forceinline__ double2 c_lag(double2 a, double2 vg, double2 wg, double2 vk, double2 wk) {
  a.x = fma(-vg.x, wk.x, a.x);
  a.x = fma(-vg.y, wk.y, a.x);
  a.x = fma(-wg.x, vk.x, a.x);
  a.x = fma(-wg.y, vk.y, a.x);
  a.y = fma(-vg.y, wk.x, a.y);
  a.y = fma(vg.x, wk.y, a.y);
  a.y = fma(-wg.y, vk.x, a.y);
  a.y = fma(wg.x, vk.y, a.y);
  return a;
}
__device__ __forceinline__ void c_fma_acc(cdf& s, cdf a, cdf b) { cdf_fma_acc(s, a, b); }
__device__ __forceinline__ void c_fma_acc(double2& s, double2 a, double2 b) { cfma(s, a, b); }
__device__ __forceinline__ void c_fmac_acc(cdf& s, cdf a, cdf b) { cdf_fmac_acc(s, a, b); }
__device__ __forceinline__ void c_fmac_acc(double2& s, double2 a, double2 b) { cfmac(s, a, b); }
__device__ __forceinline__ cdf c_from(cdf, double2 x, int ex) {
  return cdf_from(make_double2(ldexp(x.x, -ex), ldexp(x.y, -ex)));
}
__device__ __forceinline__ double2 c_from(double2, double2 x, int) { return x; }
// the Householder vector as the back-transformation reads it (FP32 path: evict-first, so the row
// store keeps the L2)
__device__ __forceinline__ void put_hv(void* Hv, long i, cdf v) { __stcs((float2*)Hv + i, make_float2(v.rh, v.ih)); }
__device__ __forceinline__ void put_hv(void* Hv, long i, double2 v) { ((double2*)Hv)[i] = v; }

// Sum over the block in a fixed order, the result on every thread.  Double-float: every warp adds the
// warps' sums (one barrier).  FP64: one warp adds them (two barriers), since an FP64 instruction of
// every warp costs 64 clocks times the warps of a scheduler.
template <int NW>
__device__ __forceinline__ dfl hf_block_sum(dfl v, dfl* red, int lane, int warp) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = df_add(v, df_shfl_xor(v, o));
  if (lane == 0) red[warp] = v;
  __syncthreads();
  v = red[lane & (NW - 1)];
#pragma unroll
  for (int o = NW / 2; o > 0; o >>= 1) v = df_add(v, df_shfl_xor(v, o));
  return v;
}
template <int NW>
__device__ __forceinline__ double hf_block_sum(double v, double* red, int lane, int warp) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < NW ? red[lane] : 0.0;
#pragma unroll
    for (int o = NW / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[NW] = v;
  }
  __syncthreads();
  return red[NW];
}

template <typename C, int CL, bool GS>
__global__ void __launch_bounds__(HETRD_NT, 1) k_hetrd(const double2* __restrict__ G, long ldg, long sG, int m, int s_elems,
                                                 EigScratch e, int cp_global) {
  using R = decltype(cre(C()));
  constexpr bool DF = std::is_same<C, cdf>::value;
  constexpr int NT = HETRD_NT, NW = NT / 32, IPT = 512 / NT;  // indices of a vector per thread (m <= 512)
  constexpr int HF_SR = DF && !GS ? 8 : 4;       // rows per strip
  constexpr int RP = DF ? 2 : 1;                 // of which interleaved
  extern __shared__ __align__(16) unsigned char hfsm[];
  C* S = GS ? (C*)e.Sg + (long)blockIdx.x * s_elems : (C*)hfsm;  // own rows, packed, private to this CTA
  C* bufV = GS ? (C*)hfsm : S + s_elems;  // [2][m] v of this and of the previous step
  C* w = bufV + 2 * m;                    // [m] w of the previous step
  C* bufP = w + m;                        // [2][m] this CTA's part of p, by step parity (read by the partners)
  C* bufX = bufP + 2 * m;                 // [2][m] the next column before its update, by step parity
  C* cpart = cp_global ? (C*)e.Cp + (long)blockIdx.x * NW * m : bufX + 2 * m;  // [NW][m] column parts of p
  __shared__ R redK[NW + 1], redN[NW + 1];
  __shared__ C s_p2[2], s_ph, s_am;  // p of the entries j and j + 1; the phase of x_0; -alpha
  __shared__ R s_ax0, s_vinv;
  __shared__ int s_exp, s_glast[NW];
  cg::cluster_group cluster = cg::this_cluster();
  const int c = (CL > 1) ? (int)cluster.block_rank() : 0;
  const int b = (int)blockIdx.x / CL;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  G += (long)b * sG;
  void* Hv = DF ? (void*)((float2*)e.Hv + (long)b * m * m) : (void*)(e.Hv + (long)b * m * m);
  const int nq = hs_own_rows(m, c, CL);
  const int qlast = nq - 1 - warp;  // this warp's last own row: qlast, qlast - NW, ..
  const C z = c_zero(C());

  // double-float: power-of-two scale from the largest diagonal entry (identical in every CTA)
  if (tid == 0) s_exp = 0;
  if (lane == 0) s_glast[warp] = qlast >= 0 ? c + CL * qlast : -1;
  if constexpr (DF) {
    __shared__ double wmx[NW];
    double mx = 0;
    for (int i = tid; i < m; i += NT) mx = fmax(mx, fabs(__ldcg(G + (long)i * ldg + i).x));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) wmx[warp] = mx;
    __syncthreads();
    if (tid == 0) {
      double t = 0;
      for (int q = 0; q < NW; ++q) t = fmax(t, wmx[q]);
      int ex = 0;
      if (t > 0 && isfinite(t)) frexp(t, &ex);
      s_exp = ex;
    }
  }
  __syncthreads();
  const int ex = s_exp;
  for (int q = warp; q < nq; q += NW) {
    const int g = c + CL * q;
    const double2* src = G + (long)g * ldg;
    C* dst = S + hs_rowbase(q, c, CL);
    for (int k = lane; k <= g; k += 32) dst[k] = c_from(C(), __ldcg(src + k), ex);
  }
  for (int i = tid; i < m; i += NT) {
    bufX[i] = c_from(C(), __ldcg(G + (long)i * ldg), ex);
    // no update is pending in the first step; entries a vector never gets multiply zeros: finite
    bufV[i] = bufV[m + i] = w[i] = z;
  }
  if (CL > 1) cluster.sync();
  else __syncthreads();

  for (int j = 0; j < m; ++j) {
    const int cur = j & 1;
    C* v = bufV + cur * m;
    const C* vp = bufV + (cur ^ 1) * m;
    const C* xr = bufX + cur * m;
    const bool lag = j > 0;
    // w of step j-1 and the column j of A^(j); indices i = tid + NT u
    C x[IPT], x0 = (j + 1 < m) ? xr[j + 1] : z;
    if (lag) {
      C pi[IPT], vi[IPT];
      R kp = r_zero(R());
#pragma unroll
      for (int u = 0; u < IPT; ++u) {
        const int i = tid + NT * u;
        pi[u] = vi[u] = z;
        if (i >= j && i < m) {
          const C* part = bufP + (cur ^ 1) * m + i;
#pragma unroll
          for (int rr = 0; rr < CL; ++rr) {
            const C* src = (CL > 1) ? cluster.map_shared_rank(part, rr) : part;
            pi[u] = rr == 0 ? *src : c_add(pi[u], *src);
          }
          pi[u] = c_twice(pi[u]);
          vi[u] = vp[i];
          kp = r_fma(kp, cre(vi[u]), cre(pi[u]));
          kp = r_fma(kp, cim(vi[u]), cim(pi[u]));
          if (i - j < 2) s_p2[i - j] = pi[u];
        }
      }
      const R nK = r_neg(hf_block_sum<NW>(kp, redK, lane, warp));
      const C vj = vp[j], pj = s_p2[0];
      const C wj = c_make(r_fma(cre(pj), cre(vj), nK), r_fma(cim(pj), cim(vj), nK));
      if (warp == NW - 1 && j + 1 < m) {  // x_0 once more, for its phase
        const C v1 = vp[j + 1], p1 = s_p2[1];
        const C w1 = c_make(r_fma(cre(p1), cre(v1), nK), r_fma(cim(p1), cim(v1), nK));
        x0 = c_lag(x0, v1, w1, vj, wj);
      }
#pragma unroll
      for (int u = 0; u < IPT; ++u) {
        const int i = tid + NT * u;
        x[u] = z;
        if (i >= j && i < m) {
          const C wi = c_make(r_fma(cre(pi[u]), cre(vi[u]), nK), r_fma(cim(pi[u]), cim(vi[u]), nK));
          w[i] = wi;
          x[u] = c_lag(xr[i], vi[u], wi, vj, wj);
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < IPT; ++u) x[u] = (tid + NT * u < m) ? xr[tid + NT * u] : z;
    }
    if (c == 0) {
#pragma unroll
      for (int u = 0; u < IPT; ++u)
        if (tid + NT * u == j) e.d[(long)b * m + j] = DF ? ldexp(r_double(cre(x[u])), ex) : r_double(cre(x[u]));
    }
    if (j == m - 1) break;
    // the reflector
    {
      R t = r_zero(R());
#pragma unroll
      for (int u = 0; u < IPT; ++u) {
        const int i = tid + NT * u;
        if (i > j && i < m) {
          t = r_fma(t, cre(x[u]), cre(x[u]));
          t = r_fma(t, cim(x[u]), cim(x[u]));
        }
      }
      if (warp == NW - 1) {  // |x_0| and e^{i arg x_0}, beside the norm
        const R ax2 = r_fma(r_fma(r_zero(R()), cre(x0), cre(x0)), cim(x0), cim(x0));
        R ax0 = r_zero(R());
        C phase = c_one(C());
        if (r_pos(ax2)) {
          const R iax = r_rsqrt(ax2);
          ax0 = r_mul(ax2, iax);
          phase = c_make(r_mul(cre(x0), iax), r_mul(cim(x0), iax));
        }
        if (lane == 0) {
          s_ax0 = ax0;
          s_ph = phase;
        }
      }
      const R nrm2 = hf_block_sum<NW>(t, redN, lane, warp);
      C am = z;  // -alpha = e^{i arg x0} |x|
      R vinv = r_zero(R());
      if (DF || warp == 0) {  // FP64: by one warp (one more barrier)
        if (r_pos(nrm2)) {
          const R nrm = r_sqrt(nrm2);
          vinv = r_rsqrt(r_mul(r_add(nrm, nrm), r_add(nrm, s_ax0)));
          am = c_make(r_mul(cre(s_ph), nrm), r_mul(cim(s_ph), nrm));
        }
        if (!DF && lane == 0) {
          s_am = am;
          s_vinv = vinv;
        }
        if (tid == 0 && c == 0) {
          double2 al = make_double2(-r_double(cre(am)), -r_double(cim(am)));
          if (DF) al = make_double2(ldexp(al.x, ex), ldexp(al.y, ex));
          e.alpha[(long)b * m + j] = al;
        }
      }
      if constexpr (!DF) {
        __syncthreads();
        am = s_am;
        vinv = s_vinv;
      }
#pragma unroll
      for (int u = 0; u < IPT; ++u) {
        const int i = tid + NT * u;
        if (i > j && i < m) {
          C vi = x[u];
          if (i == j + 1) vi = c_add(vi, am);
          vi = c_scale_r(vi, vinv);
          v[i] = vi;
          if (c == 0) put_hv(Hv, (long)j * m + i, vi);
        }
      }
    }
    __syncthreads();

    // the sweep
    {
      const int q0 = hs_qfirst(j, c, CL);
      const int nr = qlast >= q0 ? (qlast - q0) / NW + 1 : 0;  // own rows of this warp
      const int nst = (nr + HF_SR - 1) / HF_SR;
      const int per = nst > 0 ? (nr + nst - 1) / nst : 0;      // rows per strip, evenly
      C* cp = cpart + warp * m;
      C* xn = bufX + (cur ^ 1) * m;
      C* pv = bufP + cur * m;
      for (int st = 0; st < nst; ++st) {
        const int r0 = st * per, rn = min(per, nr - r0);
        int gr[HF_SR], off[HF_SR];
#pragma unroll
        for (int r = 0; r < HF_SR; ++r) {
          const int q = max(qlast - NW * (r0 + r), 0);
          gr[r] = r < rn ? c + CL * q : -1;  // -1: no row
          off[r] = hs_rowbase(q, c, CL);
        }
        const int glast = gr[0];
        C racc[HF_SR];
#pragma unroll
        for (int r = 0; r < HF_SR; ++r) racc[r] = z;
        C next[GS ? HF_SR : 1];  // rows in L2: the next 32 columns, on their way during this one's arithmetic
        if constexpr (GS) {
#pragma unroll
          for (int r = 0; r < HF_SR; ++r) next[r] = (j + 1 + lane <= gr[r]) ? S[off[r] + j + 1 + lane] : z;
        }
        for (int k0 = j + 1; k0 <= glast; k0 += 32) {
          const int k = k0 + lane, kc = min(k, glast);
          C a[GS ? HF_SR : 1];
          if constexpr (GS) {
#pragma unroll
            for (int r = 0; r < HF_SR; ++r) {
              a[r] = next[r];
              next[r] = (k + 32 <= gr[r]) ? S[off[r] + k + 32] : z;
            }
          }
          const C vk = v[kc], vpk = vp[kc], wpk = w[kc];
          C cacc[RP];
#pragma unroll
          for (int u = 0; u < RP; ++u) cacc[u] = z;
          // RP rows at a time, without branches on the lane: the chains of the two interleave; lanes
          // past a row's end carry zeros
#pragma unroll
          for (int r = 0; r < HF_SR; r += RP) {
            if (k0 > gr[r]) break;  // rows get shorter
            C y[RP];
#pragma unroll
            for (int u = 0; u < RP; ++u) {
              if constexpr (GS) y[u] = a[r + u];
              else y[u] = (k <= gr[r + u]) ? S[off[r + u] + k] : z;
            }
#pragma unroll
            for (int u = 0; u < RP; ++u) {
              const int g = max(gr[r + u], 0);
              y[u] = c_lag(y[u], vp[g], w[g], vpk, wpk);
              if (k > gr[r + u]) y[u] = z;
              if (k == gr[r + u]) c_real(y[u]);
            }
#pragma unroll
            for (int u = 0; u < RP; ++u)
              if (k <= gr[r + u]) S[off[r + u] + k] = y[u];
            if (k == j + 1) {  // the next column, to every CTA
#pragma unroll
              for (int u = 0; u < RP; ++u)
                if (gr[r + u] >= 0) {
#pragma unroll
                  for (int rr = 0; rr < CL; ++rr) {
                    C* dst = (CL > 1) ? cluster.map_shared_rank(xn, rr) : xn;
                    dst[gr[r + u]] = y[u];
                  }
                }
            }
#pragma unroll
            for (int u = 0; u < RP; ++u) {
              c_fma_acc(racc[r + u], y[u], vk);
              c_fmac_acc(cacc[u], (k < gr[r + u]) ? y[u] : z, v[max(gr[r + u], 0)]);
            }
          }
          // the first strip has the warp's last row, hence all its columns
          if (k < glast) {
            const C cs = RP == 2 ? c_add(cacc[0], cacc[RP - 1]) : cacc[0];
            cp[k] = st == 0 ? cs : c_add(cp[k], cs);
          }
        }
        // row sums across the lanes: halve the rows (the lanes with the bit set keep the upper half)
        // until one is left, then a butterfly; lane l ends with row l SR / 32
        int o = 16;
#pragma unroll
        for (int h = HF_SR / 2; h > 0; h >>= 1, o >>= 1) {
          const bool up = (lane & o) != 0;
#pragma unroll
          for (int i = 0; i < h; ++i) {
            const C keep = up ? racc[h + i] : racc[i], send = up ? racc[i] : racc[h + i];
            racc[i] = c_add(keep, c_shfl(send, o));
          }
        }
#pragma unroll
        for (; o > 0; o >>= 1) racc[0] = c_add(racc[0], c_shfl(racc[0], o));
        constexpr int LR = 32 / HF_SR;  // lanes per row
        if (lane % LR == 0 && lane / LR < rn) pv[c + CL * (qlast - NW * (r0 + lane / LR))] = racc[0];
      }
    }
    __syncthreads();
    // this CTA's part of p: its rows' row parts plus the warps' column parts (a warp has them for the
    // columns before its last row), all loads first, then a pairwise sum
    {
      C* pv = bufP + cur * m;
#pragma unroll
      for (int u = 0; u < IPT; ++u) {
        const int k = tid + NT * u;
        if (k > j && k < m) {
          C part[NW];
#pragma unroll
          for (int q = 0; q < NW; ++q) part[q] = k < s_glast[q] ? cpart[q * m + k] : z;
#pragma unroll
          for (int h = NW / 2; h > 0; h >>= 1)
#pragma unroll
            for (int q = 0; q < h; ++q) part[q] = c_add(part[q], part[q + h]);
          pv[k] = (k % CL == c) ? c_add(pv[k], part[0]) : part[0];
        }
      }
    }
    if (CL > 1) cluster.sync();
    else __syncthreads();
  }
  if (CL > 1) cluster.sync();  // the partners' last reads of this CTA's part of p
  else __syncthreads();
  if (c != 0) return;
  // |alpha_j|, the phases that make T real (running products of alpha_j / |alpha_j|) and a bound of
  // its norm
  double2* ph = (double2*)bufV;
  __syncthreads();
  for (int i = tid; i < m - 1; i += NT) {
    const double2 a = __ldcg(e.alpha + (long)b * m + i);
    const double aa = sqrt(cabs2(a));
    e.f[(long)b * m + i] = aa;
    ph[i] = aa > 0 ? cscale(a, 1.0 / aa) : make_double2(1.0, 0.0);
  }
  __syncthreads();
  if (warp == 0) {
    const int per = (m - 1 + 31) / 32, i0 = min(lane * per, m - 1), i1 = min(i0 + per, m - 1);
    double2 t = make_double2(1.0, 0.0);
    for (int i = i0; i < i1; ++i) t = cmul(t, ph[i]);
    double2 run = t;  // inclusive products of the lanes' own
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double2 up = make_double2(__shfl_up_sync(0xffffffffu, run.x, o), __shfl_up_sync(0xffffffffu, run.y, o));
      if (lane >= o) run = cmul(up, run);
    }
    double2 dl = make_double2(__shfl_up_sync(0xffffffffu, run.x, 1), __shfl_up_sync(0xffffffffu, run.y, 1));
    if (lane == 0) {
      dl = make_double2(1.0, 0.0);
      e.delta[(long)b * m] = dl;
    }
    for (int i = i0; i < i1; ++i) {
      dl = cmul(dl, ph[i]);
      e.delta[(long)b * m + i + 1] = dl;
    }
  } else if (warp == 1) {
    double tn = 0;
    for (int i = lane; i < m; i += 32) {
      const double fl = (i > 0) ? e.f[(long)b * m + i - 1] : 0.0, fr = (i < m - 1) ? e.f[(long)b * m + i] : 0.0;
      tn = fmax(tn, fabs(e.d[(long)b * m + i]) + fl + fr);
    }
    for (int o = 16; o > 0; o >>= 1) tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
    if (lane == 0) e.tnorm[b] = tn;
  }
}

// Number of eigenvalues below x of the symmetric tridiagonal (d, f) (scaled
// to norm ~1): sign changes of the Sturm sequence P_0 = 1, P_1 = d_0 - x,
// P_i = (d_{i-1} - x) P_{i-1} - f_{i-2}^2 P_{i-2}, i.e. negative ratios
// q_i = P_i / P_{i-1}; a zero ratio is replaced by -pivmin.  The pair
// (P_i, P_{i-1}) is rescaled by powers of two to stay in range.
__device__ __forceinline__ int sturm_count(const double* d, const double* f2, int m, double x, double pivmin) {
  double pm = 1.0, p = d[0] - x;
  if (p == 0.0) p = -pivmin;
  int cnt = (int)((unsigned long long)__double_as_longlong(p) >> 63);
  for (int i = 1; i < m; ++i) {
    double pn = fma(d[i] - x, p, -f2[i - 1] * pm);
    long long bn = __double_as_longlong(pn);
    if ((bn << 1) == 0) {  // zero ratio
      pn = -pivmin * p;
      bn = __double_as_longlong(pn);
    }
    cnt += (int)((unsigned long long)(bn ^ __double_as_longlong(p)) >> 63);
    pm = p;
    p = pn;
    // keep the pair in range: rescale both by a power of two when the exponent of p leaves +-600
    const int ex = (int)((bn >> 52) & 0x7ff) - 1023;
    if (ex > 600 || ex < -600) {
      const double sc = __longlong_as_double((long long)(1023 - ex) << 52);
      p *= sc;
      pm *= sc;
    }
  }
  return cnt;
}

// The reduced-precision counts below clamp every ratio q_i of magnitude
// below 2^-64 to -2^-64 (a perturbation of d_{i-1} by at most 2^-63 ||T||)
// and rescale the pair by a power of two whenever |P_i| leaves
// [2^-32, 2^32].  The clamp bounds |P_{i-1} / P_i| by 2^64, so neither member
// of the pair can overflow or become subnormal.
constexpr float kSturmPiv = 0x1p-64f;

// FP32 count.  df[i] = (d_i, f_{i-1}^2) with f_{-1} = 0.  A computed count is
// the exact count of a tridiagonal whose d_i - x and f^2 moved by a few units
// in the last place (the recurrence is backward stable), i.e. of one within
// about 5e-7 ||T|| of the given one, so a bracket from FP32 counts holds the
// eigenvalue once widened by a margin above that.
__device__ __forceinline__ int sturm_count_f32(const float2* __restrict__ df, int m, float x) {
  float p = 1.0f, pm = 0.0f;
  int cnt = 0;
#pragma unroll 4
  for (int i = 0; i < m; ++i) {
    const float2 v = df[i];
    float pn = fmaf(v.x - x, p, -v.y * pm);
    if (fabsf(pn) < kSturmPiv * fabsf(p)) pn = -kSturmPiv * p;
    cnt += (int)((__float_as_uint(pn) ^ __float_as_uint(p)) >> 31);
    pm = p;
    p = pn;
    const float an = fabsf(pn);
    if (an > 0x1p32f || an < 0x1p-32f) {
      const int ex = (int)((__float_as_uint(pn) >> 23) & 0xffu) - 127;
      const float sc = __uint_as_float((unsigned)(127 - ex) << 23);
      p *= sc;
      pm *= sc;
    }
  }
  return cnt;
}

// The same count in double-float arithmetic (each value hi + lo, two FP32
// numbers, about 48 significant bits) on the FP32 pipe, which on GB300 issues
// 64 times the FP64 rate.  v[i] = (d_i hi, d_i lo, f_{i-1}^2 hi, f_{i-1}^2 lo).
// Per step: d_i - x by TwoSum of the high parts plus the low parts; the two
// products by TwoProduct (FMA) of the high parts plus the cross terms; their
// difference by TwoSum and one renormalisation.  Every operation is exact up
// to about 2^-47 of its operands, so a computed count is the exact count of a
// tridiagonal within about 1e-14 ||T|| of the given one.
__device__ __forceinline__ int sturm_count_df(const float4* __restrict__ v, int m, dfl x) {
  float ph = 1.0f, pl = 0.0f, qh = 0.0f, ql = 0.0f;  // P_i, P_{i-1}
  int cnt = 0;
#pragma unroll 2
  for (int i = 0; i < m; ++i) {
    const float4 c = v[i];
    const float th = c.x - x.hi;  // t = d_i - x, not renormalised
    const float tb = th - c.x;
    const float tl = ((c.x - (th - tb)) + (-x.hi - tb)) + (c.y - x.lo);
    const float a = th * ph;  // t P_i
    const float ae = fmaf(tl, ph, fmaf(th, pl, fmaf(th, ph, -a)));
    const float b = c.z * qh;  // f^2 P_{i-1}
    const float be = fmaf(c.w, qh, fmaf(c.z, ql, fmaf(c.z, qh, -b)));
    const float sh = a - b;
    const float sb = sh - a;
    const float sl = ((a - (sh - sb)) + (-b - sb)) + (ae - be);
    float nh = sh + sl;
    float nl = sl - (nh - sh);
    if (fabsf(nh) < kSturmPiv * fabsf(ph)) {
      nh = -kSturmPiv * ph;
      nl = -kSturmPiv * pl;
    }
    cnt += (int)((__float_as_uint(nh) ^ __float_as_uint(ph)) >> 31);
    qh = ph;
    ql = pl;
    ph = nh;
    pl = nl;
    const float an = fabsf(nh);
    if (an > 0x1p32f || an < 0x1p-32f) {
      const int ex = (int)((__float_as_uint(nh) >> 23) & 0xffu) - 127;
      const float sc = __uint_as_float((unsigned)(127 - ex) << 23);
      ph *= sc;
      pl *= sc;
      qh *= sc;
      ql *= sc;
    }
  }
  return cnt;
}

// Multisection: one warp per wanted eigenvalue (the (r+1)-th largest of the
// slice's scaled T); per step the 32 lanes count at 32 interior points of the
// bracket, so the bracket shrinks 33-fold per step.
//
// BIS_F32_ROUNDS rounds of FP32 counts, the bracket widened by BIS_F32_MARGIN
// on both sides (about seven times the FP32 count's backward error bound), then
// double-float counts until the bracket is at most abs_tol wide (FP32 path).
// abs_tol = 0 (FP64 path): until it is 2^-40 ||T|| wide, widened again by
// BIS_DF_MARGIN (eleven times the double-float count's bound), and from there on
// FP64 counts until it is within two units in the last place of the eigenvalue:
// an FP64 count is bound by the FP64 pipe and takes some twenty times a
// double-float one, and 3 rounds of it remain of 11 (m = 300, 50 eigenvalues on 33
// slices: 3.15 -> 1.49 ms).  Each round moves an
// end only to a point whose count was taken, at that point's value in the
// precision of the count.
constexpr int BIS_WARPS = 4;
constexpr int BIS_F32_ROUNDS = 4;
constexpr double BIS_F32_MARGIN = 0x1p-18;
constexpr double BIS_DF_MARGIN = 0x1p-43;
__global__ void __launch_bounds__(BIS_WARPS * 32) k_bisect(int m, int R, EigScratch e, double* __restrict__ lam_out,
                                                          double abs_tol) {
  extern __shared__ __align__(16) double bsm[];
  double* d = bsm;                        // [m] scaled diagonal
  double* f2 = bsm + m;                   // [m] scaled squared off-diagonal
  float4* v4 = (float4*)(bsm + 2 * m);    // [m] double-float (d_i, f_{i-1}^2)
  float2* v2 = (float2*)(v4 + m);         // [m] FP32 (d_i, f_{i-1}^2)
  __shared__ double s_scale, s_lo[BIS_WARPS], s_hi[BIS_WARPS];
  const int b = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = blockIdx.x * BIS_WARPS + warp;
  if (threadIdx.x == 0) {
    const double tn = e.tnorm[b];
    s_scale = (tn > 0.0 && isfinite(tn)) ? 1.0 / tn : 1.0;
  }
  __syncthreads();
  const double sc = s_scale;
  const double* ed = e.d + (long)b * m;
  const double* ef = e.f + (long)b * m;
  double glo = DBL_MAX, ghi = -DBL_MAX;  // Gershgorin bracket of the scaled T
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const double di = ed[i] * sc;
    const double fr = (i < m - 1) ? ef[i] * sc : 0.0;
    const double fl = (i > 0) ? ef[i - 1] * sc : 0.0;
    d[i] = di;
    f2[i] = fr * fr;
    const double fl2 = fl * fl;
    const dfl dh = df_from(di), fh = df_from(fl2);
    v4[i] = make_float4(dh.hi, dh.lo, fh.hi, fh.lo);
    v2[i] = make_float2((float)di, (float)fl2);
    glo = fmin(glo, di - fabs(fl) - fabs(fr));
    ghi = fmax(ghi, di + fabs(fl) + fabs(fr));
  }
  for (int o = 16; o > 0; o >>= 1) {
    glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
    ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
  }
  if (lane == 0) {
    s_lo[warp] = glo;
    s_hi[warp] = ghi;
  }
  __syncthreads();
  if (r >= R) return;
  if (!(e.tnorm[b] > 0.0)) {  // T = 0 (zero data): every eigenvalue is 0
    if (lane == 0) lam_out[(long)b * R + r] = 0.0;
    return;
  }
  double g_lo = s_lo[0], g_hi = s_hi[0];
  for (int w = 1; w < BIS_WARPS; ++w) {
    g_lo = fmin(g_lo, s_lo[w]);
    g_hi = fmax(g_hi, s_hi[w]);
  }
  const double tn = fmax(fabs(g_lo), fabs(g_hi));
  const double pivmin = DBL_MIN * 0x1p+64;
  double lo = g_lo - (4.0 * DBL_EPSILON * tn + pivmin);
  double hi = g_hi + (4.0 * DBL_EPSILON * tn + pivmin);
  const int idx = m - 1 - r;  // ascending index of the wanted eigenvalue
  const double wide_lo = lo, wide_hi = hi;
  {
    for (int it = 0; it < BIS_F32_ROUNDS; ++it) {
      const double w = hi - lo;
      const float x = (float)(lo + w * ((double)(lane + 1) / 33.0));
      const unsigned above = __ballot_sync(0xffffffffu, sturm_count_f32(v2, m, x) > idx);
      const int first = above ? __ffs(above) - 1 : 32;
      const double nlo = (first == 0) ? lo : (double)(float)(lo + w * ((double)first / 33.0));
      const double nhi = (first == 32) ? hi : (double)(float)(lo + w * ((double)(first + 1) / 33.0));
      lo = nlo;
      hi = nhi;
    }
    lo = fmax(lo - BIS_F32_MARGIN * tn, wide_lo);
    hi = fmin(hi + BIS_F32_MARGIN * tn, wide_hi);
    const double df_tol = abs_tol > 0.0 ? abs_tol : 0x1p-40 * tn;
    for (int it = 0; it < 16; ++it) {
      const double w = hi - lo;
      if (w <= df_tol) break;
      const dfl x = df_from(lo + w * ((double)(lane + 1) / 33.0));
      const unsigned above = __ballot_sync(0xffffffffu, sturm_count_df(v4, m, x) > idx);
      const int first = above ? __ffs(above) - 1 : 32;
      const double nlo = (first == 0) ? lo : df_to(df_from(lo + w * ((double)first / 33.0)));
      const double nhi = (first == 32) ? hi : df_to(df_from(lo + w * ((double)(first + 1) / 33.0)));
      if (nlo == lo && nhi == hi) break;
      lo = nlo;
      hi = nhi;
    }
  }
  if (abs_tol == 0.0) {
    lo = fmax(lo - BIS_DF_MARGIN * tn, wide_lo);
    hi = fmin(hi + BIS_DF_MARGIN * tn, wide_hi);
    for (int it = 0; it < 64; ++it) {
      const double w = hi - lo;
      // relative to the eigenvalue
      if (w <= 2.0 * DBL_EPSILON * (fabs(lo) + fabs(hi)) + pivmin) break;
      const double x = lo + w * ((double)(lane + 1) / 33.0);
      const unsigned above = __ballot_sync(0xffffffffu, sturm_count(d, f2, m, x, pivmin) > idx);
      const int first = above ? __ffs(above) - 1 : 32;  // lowest point with more than idx values below it
      const double nlo = (first == 0) ? lo : lo + w * ((double)first / 33.0);
      const double nhi = (first == 32) ? hi : lo + w * ((double)(first + 1) / 33.0);
      if (nlo == lo && nhi == hi) break;
      lo = nlo;
      hi = nhi;
    }
  }
  if (lane == 0) lam_out[(long)b * R + r] = 0.5 * (lo + hi) / sc;
}

// One thread per wanted eigenpair r (the (r+1)-th largest), TP_THREADS pairs
// per CTA: inverse iteration (three solves, two on the FP32 path) with a partially pivoted LU of
// T - lam I for the eigenvalue found by k_bisect.  The LU factors stream
// from global memory (coalesced across the CTA's threads); the iterate lives
// in shared memory, so the dependent chain of each solve never waits on L2.
constexpr int TP_THREADS = 32;

__global__ void __launch_bounds__(TP_THREADS) k_tridiag_pairs(int m, int R, EigScratch e,
                                                              const double* __restrict__ lam_out, int iters) {
  extern __shared__ __align__(16) double tsm[];
  double* d = tsm;      // [m] scaled diagonal
  double* f = tsm + m;  // [m] scaled off-diagonal
  double* f2 = f + m;   // [m] squares
  double* xs = f2 + m;  // [m][TP_THREADS] iterates
  __shared__ double s_scale;
  const int b = blockIdx.y, t = threadIdx.x, r = blockIdx.x * TP_THREADS + t;
  if (t == 0) {
    const double tn = e.tnorm[b];
    s_scale = (tn > 0.0 && isfinite(tn)) ? 1.0 / tn : 1.0;
  }
  __syncthreads();
  const double sc = s_scale;
  for (int i = t; i < m; i += blockDim.x) {
    d[i] = e.d[(long)b * m + i] * sc;
    const double fi = (i < m - 1) ? e.f[(long)b * m + i] * sc : 0.0;
    f[i] = fi;
    f2[i] = fi * fi;
  }
  __syncthreads();
  if (r >= R) return;
  double* Z = e.Z + ((long)b * R + r) * m;  // vector r, contiguous
  if (!(e.tnorm[b] > 0.0)) {  // T = 0 (zero data): vectors e_r
    for (int i = 0; i < m; ++i) Z[i] = (i == r) ? 1.0 : 0.0;
    return;
  }
  double tn = 0;
  for (int i = 0; i < m; ++i) tn = fmax(tn, fabs(d[i]) + ((i > 0) ? f[i - 1] : 0.0) + f[i]);
  const double lam = lam_out[(long)b * R + r] * sc;

  // factor element i of array a at lu[((b*5 + a)*m + i)*R + r] (coalesced over r)
  // a: 0 multiplier, 1 reciprocal U diagonal, 2 U first super, 3 U second super, 4 row swap (0 / 1)
  double* base = e.lu + (long)b * 5 * m * R + r;
#define LU(a, i) base[((long)(a) * m + (i)) * R]
  double* x = xs + t;
#define X(i) x[(long)(i) * TP_THREADS]
  const double tiny = DBL_EPSILON * fmax(tn, 1e-200);
  double dcur = d[0] - lam, ucur = f[0];
  for (int i = 0; i < m - 1; ++i) {
    const double sub = f[i];
    const double dn = d[i + 1] - lam, un = (i < m - 2) ? f[i + 1] : 0.0;
    if (fabs(dcur) >= fabs(sub)) {
      const double piv = (fabs(dcur) < tiny) ? copysign(tiny, dcur) : dcur;
      const double rp = 1.0 / piv;  // one division per step
      const double l = sub * rp;
      LU(0, i) = l;
      LU(1, i) = rp;
      LU(2, i) = ucur;
      LU(3, i) = 0.0;
      LU(4, i) = 0.0;
      dcur = dn - l * ucur;
      ucur = un;
    } else {
      // swap rows i and i+1: the new row i is (sub, dn, un); the old row i is eliminated
      const double sb = (fabs(sub) < tiny) ? copysign(tiny, sub) : sub;
      const double rs = 1.0 / sb;
      const double l = dcur * rs;
      LU(0, i) = l;
      LU(1, i) = rs;
      LU(2, i) = dn;
      LU(3, i) = un;
      LU(4, i) = 1.0;
      const double nd = ucur - l * dn;
      ucur = -l * un;
      dcur = nd;
    }
  }
  LU(1, m - 1) = 1.0 / ((fabs(dcur) < tiny) ? copysign(tiny, dcur) : dcur);
  LU(2, m - 1) = 0.0;
  LU(3, m - 1) = 0.0;
  for (int i = 0; i < m; ++i) {  // starting vector: Philox uniforms in (-1, 1)
    const uint4 w = philox10(make_uint4((uint32_t)i, (uint32_t)r, (uint32_t)b, 0x1e16u), 0x2504u, 0x4989u);
    X(i) = ((double)w.x + 0.5) * (2.0 / 4294967296.0) - 1.0;
  }
  for (int iter = 0; iter < iters; ++iter) {
    double xi = X(0);
    for (int i = 0; i < m - 1; ++i) {  // row interchanges and multipliers: L^{-1} P
      double xn = X(i + 1);
      if (LU(4, i) != 0.0) {
        const double tmp = xi;
        xi = xn;
        xn = tmp;
      }
      X(i) = xi;
      xi = xn - LU(0, i) * xi;
    }
    X(m - 1) = xi;
    double mx = 0, x1 = 0, x2 = 0;
    for (int i = m - 1; i >= 0; --i) {  // back substitution with U
      const double s = (X(i) - LU(2, i) * x1 - LU(3, i) * x2) * LU(1, i);
      X(i) = s;
      x2 = x1;
      x1 = s;
      mx = fmax(mx, fabs(s));
    }
    if (!(mx > 0) || !isfinite(mx)) mx = 1.0;
    const double imx = 1.0 / mx;
    double nrm2 = 0;
    for (int i = 0; i < m; ++i) {
      const double v = X(i) * imx;
      X(i) = v;
      nrm2 += v * v;
    }
    const double inv = 1.0 / sqrt(nrm2);
    for (int i = 0; i < m; ++i) X(i) *= inv;
  }
  for (int i = 0; i < m; ++i) Z[i] = X(i);
#undef X
#undef LU
}

// Reciprocal: correctly rounded FP32 reciprocal, then one Newton correction
// with the residual 1 - b r formed exactly (FMA) plus the low part's term.
__device__ __forceinline__ dfl df_rcp(dfl b) {
  const float r = __frcp_rn(b.hi);
  const float p = b.hi * r, pe = fmaf(b.hi, r, -p);
  const float res = ((1.0f - p) - pe) - b.lo * r;
  return df_fast_two_sum(r, r * res);
}

// The inverse iteration of k_tridiag_pairs in double-float arithmetic (FP32
// path): the LU of T - lam I, the solves and the normalisation carry hi + lo
// pairs (about 48 significant bits, far below the FP32 accuracy this path
// returns) on the FP32 pipe, so each step's dependent chain is a few FP32
// operations rather than FP64 ones at 1/64 of the rate.  Pivots below 2^-47
// ||T|| are raised to that size.  Factors per step (coalesced over r):
// multiplier, reciprocal pivot and the two U super-diagonals as (hi, lo)
// pairs, the row swaps as bits of one word per 32 steps.  NTH pairs per CTA;
// SMF: the factors of all NTH pairs stay in shared memory (16 pairs at
// m = 300: 197 KB), so the solves never wait on L2; otherwise they live in
// global memory and the solves fetch them TP_CHUNK steps at a time, ahead of
// the dependent chain.
constexpr int TP_CHUNK = 8;
template <bool SMF>
__device__ __forceinline__ float2 tp_ld(const float2* p) {
  if constexpr (SMF) return *p;
  else return __ldcg(p);
}
template <bool SMF>
__device__ __forceinline__ unsigned tp_ld(const unsigned* p) {
  if constexpr (SMF) return *p;
  else return __ldcg(p);
}
static size_t tp_df_smem(int m, int nth, bool smf) {
  size_t bytes = (size_t)m * (sizeof(float4) + nth * sizeof(float2));
  if (smf) bytes += (size_t)m * nth * 4 * sizeof(float2) + (size_t)cdiv(m, 32) * nth * sizeof(unsigned);
  return bytes;
}
template <int NTH, bool SMF>
__global__ void __launch_bounds__(NTH) k_tridiag_pairs_df(int m, int R, EigScratch e,
                                                          const double* __restrict__ lam_out, int iters) {
  extern __shared__ __align__(16) double tsm[];
  float4* T4 = (float4*)tsm;         // [m] (d_i hi, lo, f_i hi, lo), f_{m-1} = 0
  float2* xs = (float2*)(T4 + m);    // [m][NTH] iterates
  __shared__ double s_scale;
  const int b = blockIdx.y, t = threadIdx.x, r = blockIdx.x * NTH + t;
  if (t == 0) {
    const double tn = e.tnorm[b];
    s_scale = (tn > 0.0 && isfinite(tn)) ? 1.0 / tn : 1.0;
  }
  __syncthreads();
  const double sc = s_scale;
  for (int i = t; i < m; i += blockDim.x) {
    const dfl dd = df_from(e.d[(long)b * m + i] * sc);
    const dfl ff = df_from((i < m - 1) ? e.f[(long)b * m + i] * sc : 0.0);
    T4[i] = make_float4(dd.hi, dd.lo, ff.hi, ff.lo);
  }
  __syncthreads();
  if (r >= R) return;
  double* Z = e.Z + ((long)b * R + r) * m;  // vector r, contiguous
  if (!(e.tnorm[b] > 0.0)) {  // T = 0 (zero data): vectors e_r
    for (int i = 0; i < m; ++i) Z[i] = (i == r) ? 1.0 : 0.0;
    return;
  }
  const dfl nlam = df_neg(df_from(lam_out[(long)b * R + r] * sc));
  // factor arrays, element i of this pair at [i * ls + lo]: shared memory [m][NTH] (SMF), else
  // this slice's part of e.lu, [m][R]
  const long ls = SMF ? NTH : R;
  float2* L0 = SMF ? (float2*)(xs + (long)m * NTH) : (float2*)(e.lu + (long)b * 5 * m * R);  // multiplier
  float2* L1 = L0 + (long)m * ls;                      // reciprocal pivot
  float2* L2 = L1 + (long)m * ls;                      // U first super-diagonal
  float2* L3 = L2 + (long)m * ls;                      // U second super-diagonal
  unsigned* FL = (unsigned*)(L3 + (long)m * ls);       // row swaps, [cdiv(m, 32)][ls]
  L0 += SMF ? t : r;
  L1 += SMF ? t : r;
  L2 += SMF ? t : r;
  L3 += SMF ? t : r;
  FL += SMF ? t : r;
  float2* x = xs + t;
#define X(i) x[(long)(i) * NTH]
  const float tiny = 0x1p-47f;
  dfl dcur = df_add(dfl{T4[0].x, T4[0].y}, nlam), ucur = dfl{T4[0].z, T4[0].w};
  unsigned flags = 0;
  for (int i = 0; i < m - 1; ++i) {
    const float4 c0 = T4[i], c1 = T4[i + 1];
    const dfl sub = dfl{c0.z, c0.w};
    const dfl dn = df_add(dfl{c1.x, c1.y}, nlam), un = dfl{c1.z, c1.w};
    // partial pivoting without a branch (lanes would diverge on the swaps): with a swap the new
    // row i is (sub, dn, un) and the old one is eliminated; both cases are one reciprocal, one
    // multiply and one multiply-add on selected operands
    const bool sw = !(fabsf(dcur.hi) >= fabsf(sub.hi));
    const dfl pv = sw ? sub : dcur, nm = sw ? dcur : sub;
    const dfl rp = df_rcp((fabsf(pv.hi) < tiny) ? dfl{copysignf(tiny, pv.hi), 0.0f} : pv);
    const dfl l = df_mul(nm, rp);
    const dfl u1 = sw ? dn : ucur, u2 = sw ? un : dfl{0.0f, 0.0f};
    const dfl ua = sw ? ucur : dn, ub = sw ? dn : ucur;
    const dfl lu = df_mul(df_neg(l), un);
    dcur = df_fma(ua, df_neg(l), ub);  // dn - l ucur, or ucur - l dn after a swap
    ucur = sw ? lu : un;
    flags |= (sw ? 1u : 0u) << (i & 31);
    const long o = (long)i * ls;
    L0[o] = make_float2(l.hi, l.lo);
    L1[o] = make_float2(rp.hi, rp.lo);
    L2[o] = make_float2(u1.hi, u1.lo);
    L3[o] = make_float2(u2.hi, u2.lo);
    if ((i & 31) == 31 || i == m - 2) {
      FL[(long)(i >> 5) * ls] = flags;
      flags = 0;
    }
  }
  {
    const dfl rp = df_rcp((fabsf(dcur.hi) < tiny) ? dfl{copysignf(tiny, dcur.hi), 0.0f} : dcur);
    const long o = (long)(m - 1) * ls;
    L1[o] = make_float2(rp.hi, rp.lo);
    L2[o] = make_float2(0.0f, 0.0f);
    L3[o] = make_float2(0.0f, 0.0f);
  }
  for (int i = 0; i < m; ++i) {  // starting vector: Philox uniforms in (-1, 1)
    const uint4 w = philox10(make_uint4((uint32_t)i, (uint32_t)r, (uint32_t)b, 0x1e16u), 0x2504u, 0x4989u);
    const dfl v = df_from(((double)w.x + 0.5) * (2.0 / 4294967296.0) - 1.0);
    X(i) = make_float2(v.hi, v.lo);
  }
  for (int iter = 0; iter < iters; ++iter) {
    // row interchanges and multipliers: L^{-1} P
    dfl xi = dfl{X(0).x, X(0).y};
    unsigned fw = 0;
    for (int i0 = 0; i0 < m - 1; i0 += TP_CHUNK) {
      float2 lc[TP_CHUNK];
#pragma unroll
      for (int k = 0; k < TP_CHUNK; ++k)
        lc[k] = (i0 + k < m - 1) ? tp_ld<SMF>(L0 + (long)(i0 + k) * ls) : make_float2(0.0f, 0.0f);
      if ((i0 & 31) == 0) fw = tp_ld<SMF>(FL + (long)(i0 >> 5) * ls);
#pragma unroll
      for (int k = 0; k < TP_CHUNK; ++k) {
        const int i = i0 + k;
        if (i < m - 1) {
          const float2 xv = X(i + 1);
          dfl xn = dfl{xv.x, xv.y};
          if ((fw >> (i & 31)) & 1u) {
            const dfl tmp = xi;
            xi = xn;
            xn = tmp;
          }
          X(i) = make_float2(xi.hi, xi.lo);
          xi = df_fma(xn, dfl{-lc[k].x, -lc[k].y}, xi);
        }
      }
    }
    X(m - 1) = make_float2(xi.hi, xi.lo);
    // back substitution with U
    dfl x1 = dfl{0.0f, 0.0f}, x2 = dfl{0.0f, 0.0f};
    float mx = 0.0f;
    for (int i0 = m - 1; i0 >= 0; i0 -= TP_CHUNK) {
      float2 pc[TP_CHUNK], ac[TP_CHUNK], bc[TP_CHUNK];
#pragma unroll
      for (int k = 0; k < TP_CHUNK; ++k) {
        const int i = i0 - k;
        const bool ok = i >= 0;
        const long o = (long)(ok ? i : 0) * ls;
        pc[k] = ok ? tp_ld<SMF>(L1 + o) : make_float2(0.0f, 0.0f);
        ac[k] = ok ? tp_ld<SMF>(L2 + o) : make_float2(0.0f, 0.0f);
        bc[k] = ok ? tp_ld<SMF>(L3 + o) : make_float2(0.0f, 0.0f);
      }
#pragma unroll
      for (int k = 0; k < TP_CHUNK; ++k) {
        const int i = i0 - k;
        if (i >= 0) {
          const float2 xv = X(i);
          dfl s = df_fma(dfl{xv.x, xv.y}, dfl{-ac[k].x, -ac[k].y}, x1);
          s = df_fma(s, dfl{-bc[k].x, -bc[k].y}, x2);
          s = df_mul(s, dfl{pc[k].x, pc[k].y});
          X(i) = make_float2(s.hi, s.lo);
          x2 = x1;
          x1 = s;
          mx = fmaxf(mx, fabsf(s.hi));
        }
      }
    }
    // rescale by a power of two (exact) so that the largest component is in [1, 2)
    if (mx > 0.0f && mx <= FLT_MAX) {
      const int ex = (int)((__float_as_uint(mx) >> 23) & 0xffu) - 127;
      const float s2 = ldexpf(1.0f, -ex);
      for (int i = 0; i < m; ++i) {
        const float2 v = X(i);
        X(i) = make_float2(v.x * s2, v.y * s2);
      }
    }
  }
  dfl nrm2 = dfl{0.0f, 0.0f};
  for (int i = 0; i < m; ++i) {
    const dfl v = dfl{X(i).x, X(i).y};
    nrm2 = df_fma(nrm2, v, v);
  }
  const dfl inv = df_rcp(df_sqrt(nrm2));
  for (int i = 0; i < m; ++i) Z[i] = df_to(df_mul(dfl{X(i).x, X(i).y}, inv));
#undef X
}

// Inside clusters of close eigenvalues (gap < 1e-3 ||T||) the vectors are
// made orthonormal.  On the FP32 path (CT = float) a cluster of at most
// CO_BLOCK vectors is orthonormalised as a block by CholeskyQR2: G = Z_c^T Z_c,
// G = R^T R (CTA-wide right-looking factorisation, one barrier per column),
// Z_c <- Z_c R^{-1}, twice -- the basis Gram-Schmidt in eigenvalue order gives,
// in exact arithmetic.  The inverse-iteration vectors of a cluster are close
// to orthonormal already; a pivot below 1e-5 (condition number above about
// 300, beyond what two FP32 passes restore) sends the cluster to two classical
// Gram-Schmidt passes per vector against its earlier members, then
// normalisation, which also serves larger clusters and the FP64 path.
// CT: storage and arithmetic (FP32 on the FP32 path, whose vectors are
// rounded to FP32 right after; FP64 otherwise).  The slice's R vectors are
// staged in shared memory for the whole kernel when they fit.
constexpr int CO_THREADS = 1024;
constexpr int CO_BLOCK = 64;
template <typename CT, bool STAGED>  // !STAGED (vectors too large for shared memory): CT = double, in place in Z
__global__ void __launch_bounds__(CO_THREADS) k_cluster_orth(int m, int R, EigScratch e, const double* __restrict__ lam) {
  extern __shared__ __align__(16) unsigned char cosm[];
  __shared__ double red[32];
  __shared__ CT dots[128], s_inv;
  __shared__ bool starts[128];  // vector r begins a cluster (R <= 128)
  constexpr bool kBlock = std::is_same<CT, float>::value;
  __shared__ float Gs[kBlock ? CO_BLOCK * CO_BLOCK : 1];  // Gram, then R (upper, row-major)
  __shared__ float Rd[kBlock ? CO_BLOCK : 1];             // 1 / R_jj
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  double* Z = e.Z + (long)b * R * m;  // vector r at Z + r*m
  const double* l = lam + (long)b * R;
  const double tol = 1e-3 * e.tnorm[b];
  // only vectors inside a cluster change; find whether there is any
  bool joins = false;
  for (int r = tid; r < R; r += blockDim.x) {
    starts[r] = r == 0 || l[r - 1] - l[r] > tol;
    joins |= !starts[r];
  }
  if (!__syncthreads_or(joins)) return;
  CT* zsm = STAGED ? (CT*)cosm : (CT*)Z;  // [R][m]
  if (STAGED) {
    for (int q = tid; q < R * m; q += blockDim.x) zsm[q] = (CT)Z[q];
    __syncthreads();
  }
  // CholeskyQR2 of vectors [c0, c0 + nc) (FP32); false on a small pivot (vectors as after the
  // last completed pass)
  auto block_qr = [&](int c0, int nc) -> bool {
    float* zc = (float*)zsm + (long)c0 * m;
    for (int pass = 0; pass < 2; ++pass) {
      for (int a = 0; a < nc; ++a)
        for (int bb = a + warp; bb < nc; bb += nwarp) {
          float acc = 0.f;
          for (int i = lane; i < m; i += 32) acc = fmaf(zc[(long)a * m + i], zc[(long)bb * m + i], acc);
          acc = warp_sum(acc);
          if (lane == 0) Gs[a * CO_BLOCK + bb] = acc;
        }
      __syncthreads();
      // G(a, k) -= G(j, a) G(j, k) / d_j for j < a <= k; row j scaled by 1/sqrt(d_j) afterwards
      for (int j = 0; j < nc; ++j) {
        const float d = Gs[j * CO_BLOCK + j];
        if (!(d > 1e-5f)) return false;  // uniform: every thread reads the same pivot
        const float id = 1.0f / d;
        const int k = j + 1 + (tid & 63);
        for (int a = j + 1 + (tid >> 6); a <= k && k < nc; a += CO_THREADS / 64)
          Gs[a * CO_BLOCK + k] -= Gs[j * CO_BLOCK + a] * Gs[j * CO_BLOCK + k] * id;
        __syncthreads();
      }
      if (tid < nc) Rd[tid] = 1.0f / sqrtf(Gs[tid * CO_BLOCK + tid]);
      __syncthreads();
      for (int i = tid; i < m; i += blockDim.x) {  // row i of Z_c: x R = z by forward substitution, in place
        for (int bb = 0; bb < nc; ++bb) {
          float acc = zc[(long)bb * m + i];
          for (int a = 0; a < bb; ++a) acc = fmaf(-zc[(long)a * m + i], Gs[a * CO_BLOCK + bb] * Rd[a], acc);
          zc[(long)bb * m + i] = acc * Rd[bb];
        }
      }
      __syncthreads();
    }
    return true;
  };
  auto cgs2 = [&](int c0, int c1) {
    for (int r = c0 + 1; r < c1; ++r) {
      CT* zr = zsm + (long)r * m;
      for (int pass = 0; pass < 2; ++pass) {
        for (int s2 = c0 + warp; s2 < r; s2 += nwarp) {
          const CT* zs = zsm + (long)s2 * m;
          CT acc = 0;
          for (int i = lane; i < m; i += 32) acc += zs[i] * zr[i];
          acc = warp_sum(acc);
          if (lane == 0) dots[s2 - c0] = acc;
        }
        __syncthreads();
        for (int i = tid; i < m; i += blockDim.x) {
          CT acc = zr[i];
          for (int s2 = c0; s2 < r; ++s2) acc -= dots[s2 - c0] * zsm[(long)s2 * m + i];
          zr[i] = acc;
        }
        __syncthreads();
      }
      double part = 0;
      for (int i = tid; i < m; i += blockDim.x) part += (double)zr[i] * (double)zr[i];
      // the root and the quotient by one warp: all 32 of them on the FP64 pipe took 10 us a vector (100
      // vectors of 480 on 65 slices, clusters up to 69: 903 -> 443 us; FP64 50 of 300 on 33: 764 -> 520)
      if (32 * warp < m) part = warp_sum(part);
      if (lane == 0) red[warp] = part;
      __syncthreads();
      if (warp == 0) {
        const double t = warp_sum(lane < nwarp ? red[lane] : 0.0);
        if (lane == 0) s_inv = (CT)(1.0 / sqrt(t));
      }
      __syncthreads();
      const CT inv = s_inv;
      for (int i = tid; i < m; i += blockDim.x) zr[i] *= inv;
      __syncthreads();
    }
  };
  int c0 = 0;
  for (int r = 1; r <= R; ++r) {
    if (r < R && !starts[r]) continue;  // r extends the cluster starting at c0
    const int nc = r - c0;
    bool done = nc < 2;
    if constexpr (kBlock) done = done || (nc <= CO_BLOCK && block_qr(c0, nc));
    if (!done) cgs2(c0, r);
    c0 = r;
  }
  if (STAGED)
    for (int q = tid; q < R * m; q += blockDim.x) Z[q] = (double)zsm[q];
}

// u_r = H_0 H_1 .. H_{m-2} D z_r in the precision of the output (the FP32
// path rounds U_c to FP32 for its GEMMs anyway): one warp per eigenvector, the
// vector in the warp's registers (entry i in lane i % 32, slot i / 32).  The
// reflectors (VT: float2 copies from the double-float reduction, else double2)
// are taken in pairs, v1 = v_{2k+1} first, then v0 = v_{2k}: with c = v0^H v1,
//   a1 = 2 v1^H u,  a0 = 2 (v0^H u - c a1),  u -= v1 a1 + v0 a0,
// so both products with u come from the same u and their four sums across the
// warp are halved together (six exchanges a pair instead of twenty).  The pairs
// are staged in shared memory by asynchronous copies one pair ahead, three
// buffers deep (one barrier a pair), and read by all the CTA's warps; slots wholly
// at or above row 2k are skipped.  Bound: FP64 by its pipe (8 multiply-adds per
// entry and reflector), FP32 by the exchanges and the barrier.  m = 300, 50
// vectors on 33 slices: FP64 5.53 -> 1.54 ms (one reflector at a time, 16 vectors in every CTA
// before).
constexpr int BT_VPC = 16;
__device__ __forceinline__ void bt_copy(float2* dst, const float2* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void bt_copy(double2* dst, const double2* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}

// c = v_{2k}^H v_{2k+1} of every pair, one warp each, to the unused place (2k+1, 2k) of the
// reflectors' array, and zero to (2k+1, 2k+1), where v_{2k+1} has no entry but v_{2k} has (reflector j
// lies in row j, columns j + 1 on; row m - 1, of an even m, has none)
template <typename VT>
__global__ void __launch_bounds__(256) k_reflector_pairs(int m, EigScratch e) {
  using Rt = decltype(VT().x);
  const int k = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int j0 = 2 * k, j1 = j0 + 1;
  if (j1 >= m) return;
  VT* Hs = (VT*)e.Hv + (long)blockIdx.y * m * m;
  const VT *v0 = Hs + (long)j0 * m, *v1 = Hs + (long)j1 * m;
  Rt cx = Rt(0), cy = Rt(0);
  for (int i = j1 + 1 + lane; i < m; i += 32) {
    const VT a = v0[i], b = v1[i];
    cx = fma(a.x, b.x, cx);
    cx = fma(a.y, b.y, cx);
    cy = fma(a.x, b.y, cy);
    cy = fma(-a.y, b.x, cy);
  }
  cx = warp_sum(cx);
  cy = warp_sum(cy);
  if (lane == 0) {
    Hs[(long)j1 * m + j0] = VT{cx, cy};
    Hs[(long)j1 * m + j1] = VT{Rt(0), Rt(0)};
  }
}

template <typename C, typename VT, int NPL>  // NPL >= ceil(m / 32); C and VT of one precision
__global__ void __launch_bounds__(BT_VPC * 32) k_backtransform(int m, int R, EigScratch e, C* __restrict__ U,
                                                               long ldu, long sU) {
  using Rt = decltype(C().x);
  extern __shared__ __align__(16) unsigned char bts[];
  VT* vb = (VT*)bts;  // [3][2][m]: v1 (from its c on), v0
  const int b = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r = blockIdx.x * (blockDim.x >> 5) + warp;
  const bool active = r < R;
  const VT* Hs = (const VT*)e.Hv + (long)b * m * m;  // reflector j at Hs + j m + j + 1
  C u[NPL];
#pragma unroll
  for (int t = 0; t < NPL; ++t) {
    const int i = lane + 32 * t;
    u[t] = C{Rt(0), Rt(0)};
    if (active && i < m) u[t] = from_c64<C>(cscale(e.delta[(long)b * m + i], e.Z[((long)b * R + r) * m + i]));
  }
  auto stage = [&](int k, int buf) {
    const int j0 = 2 * k;
    const VT* src = Hs + (long)(j0 + 1) * m;
    VT* dst = vb + buf * 2 * m;
    for (int i = j0 + tid; i < m; i += blockDim.x) bt_copy(dst + i, src + i);
    for (int i = j0 + 1 + tid; i < m; i += blockDim.x) bt_copy(dst + m + i, src - m + i);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  const int pairs = m / 2;  // of an even m the first has a reflector without entries
  int buf = 0;
  if (pairs > 0) stage(pairs - 1, 0);
  for (int k = pairs - 1; k >= 0; --k) {
    const int nbuf = buf == 2 ? 0 : buf + 1;
    if (k > 0) {
      stage(k - 1, nbuf);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();  // pair k visible; the buffer staged next was last read two pairs ago
    if (active) {
      const int j0 = 2 * k;
      const VT *v1 = vb + buf * 2 * m, *v0 = v1 + m;
      Rt s1x = Rt(0), s1y = Rt(0), s0x = Rt(0), s0y = Rt(0);
#pragma unroll
      for (int t = 0; t < NPL; ++t) {
        if (32 * t + 31 > j0) {
          const int i = lane + 32 * t;
          if (i > j0 && i < m) {
            const VT a = v1[i], d = v0[i];
            s1x = fma(a.x, u[t].x, s1x);  // conj(v_i) u_i
            s1y = fma(a.x, u[t].y, s1y);
            s0x = fma(d.x, u[t].x, s0x);
            s0y = fma(d.x, u[t].y, s0y);
            s1x = fma(a.y, u[t].y, s1x);
            s1y = fma(-a.y, u[t].x, s1y);
            s0x = fma(d.y, u[t].y, s0x);
            s0y = fma(-d.y, u[t].x, s0y);
          }
        }
      }
      // lanes with bit 4 keep v0's sums, those with bit 3 the imaginary parts
      const bool h4 = lane & 16, h3 = lane & 8;
      Rt px = (h4 ? s0x : s1x) + __shfl_xor_sync(0xffffffffu, h4 ? s1x : s0x, 16);
      Rt py = (h4 ? s0y : s1y) + __shfl_xor_sync(0xffffffffu, h4 ? s1y : s0y, 16);
      Rt p = (h3 ? py : px) + __shfl_xor_sync(0xffffffffu, h3 ? px : py, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
      p *= Rt(2);
      const Rt a1x = __shfl_sync(0xffffffffu, p, 0), a1y = __shfl_sync(0xffffffffu, p, 8);
      Rt a0x = __shfl_sync(0xffffffffu, p, 16), a0y = __shfl_sync(0xffffffffu, p, 24);
      const VT c = v1[j0];
      const Rt cx = Rt(-2) * c.x, cy = Rt(-2) * c.y;
      a0x = fma(cx, a1x, a0x);
      a0x = fma(-cy, a1y, a0x);
      a0y = fma(cx, a1y, a0y);
      a0y = fma(cy, a1x, a0y);
#pragma unroll
      for (int t = 0; t < NPL; ++t) {
        if (32 * t + 31 > j0) {
          const int i = lane + 32 * t;
          if (i > j0 && i < m) {
            const VT a = v1[i], d = v0[i];
            Rt x = u[t].x, y = u[t].y;
            x = fma(-a.x, a1x, x);
            y = fma(-a.x, a1y, y);
            x = fma(a.y, a1y, x);
            y = fma(-a.y, a1x, y);
            x = fma(-d.x, a0x, x);
            y = fma(-d.x, a0y, y);
            u[t].x = fma(d.y, a0y, x);
            u[t].y = fma(-d.y, a0x, y);
          }
        }
      }
    }
    buf = nbuf;
  }
  if (!active) return;
  C* Ub = U + (long)b * sU;
#pragma unroll
  for (int t = 0; t < NPL; ++t) {
    const int i = lane + 32 * t;
    if (i < m) Ub[(long)i * ldu + r] = u[t];
  }
}

template <typename C, typename VT>
static int launch_backtransform(int m, int R, int batch, const EigScratch& e, C* U, long ldu, long sU,
                                cudaStream_t s) {
  if (m >= 2) {
    k_reflector_pairs<VT><<<dim3(cdiv(m / 2, 8), batch), 256, 0, s>>>(m, e);
    TSVD_LAUNCHED();
  }
  const size_t smem = 6 * (size_t)m * sizeof(VT);
  // eigenvectors per CTA: the parts of R that leave the fewest on the busiest SM (each CTA stages all
  // reflectors for itself, so no fewer than 4, and of equal choices the largest)
  int parts = cdiv(R, BT_VPC);
  long best = -1;
  for (int p = parts; p <= std::max<int>(parts, cdiv(R, 4)); ++p) {
    const long load = (long)cdiv((long)p * batch, SMS) * cdiv(R, p);
    if (best < 0 || load < best) {
      best = load;
      parts = p;
    }
  }
  const int vpc = cdiv(R, parts);
  const dim3 grid(cdiv(R, vpc), batch);
  auto go = [&](auto kern) {
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
      cudaGetLastError();
      return TSVD_ERR_CUDA;
    }
    kern<<<grid, vpc * 32, smem, s>>>(m, R, e, U, ldu, sU);
    TSVD_LAUNCHED();
    return TSVD_OK;
  };
  const int npl = cdiv(m, 32);
  if (npl <= 4) return go(k_backtransform<C, VT, 4>);
  if (npl <= 8) return go(k_backtransform<C, VT, 8>);
  if (npl <= 12) return go(k_backtransform<C, VT, 12>);
  if (npl <= 16) return go(k_backtransform<C, VT, 16>);
  if (npl <= 24) return go(k_backtransform<C, VT, 24>);
  return TSVD_ERR_UNSUPPORTED;
}

static int device_attr(cudaDeviceAttr a, int fallback) {
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, a, dev) != cudaSuccess || v <= 0) {
    cudaGetLastError();
    return fallback;
  }
  return v;
}

// Clusters of CL CTAs of k_hetrd that the device holds at once, one CTA per SM (clusters stay inside a
// group of SMs, so 8 x 15 and 4 x 36 of the 152 SMs here); a cluster more would wait for a whole
// reduction to end.  A property of the device, looked up once per size.
static int hetrd_clusters(int CL) {
  static std::mutex mu;
  static int known[64][9];
  int dev = 0;
  const bool have = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64;
  const int guess = std::max(1, device_attr(cudaDevAttrMultiProcessorCount, 148) - 4 * (CL - 1)) / CL;
  if (!have || CL == 1) {
    cudaGetLastError();
    return guess;
  }
  std::lock_guard<std::mutex> lk(mu);
  int& n = known[dev][CL];
  if (n == 0) {
    auto kern = CL == 8 ? k_hetrd<cdf, 8, false> : CL == 4 ? k_hetrd<cdf, 4, false>
                                                                     : k_hetrd<cdf, 2, false>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(64 * CL);
    cfg.blockDim = dim3(HETRD_NT);
    cfg.dynamicSmemBytes = 200 * 1024;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      n = guess;
    }
  }
  return n;
}

// How a batch of m x m reductions is laid out (k_hetrd): the largest cluster in {8, 4, 2, 1} whose CTAs are
// all resident at once, with at least 20 rows each while they take a quarter of the SMs (m = 90 on 9
// slices: 604 us on clusters of 1, 508 on 2, 455 on 4), else 32 (a CTA keeps its SM: in a batch of 24
// tensors, 32 rows throughout gave 9.4 ms, 20 rows 10.3), and whose packed rows fit in shared memory beside the
// vectors, with the warps' partials there too or, where only those do not fit, in L2; else rows in L2.
struct HetrdPlan {
  int CL;
  bool global_rows, cp_global;
  size_t smem;
};
static HetrdPlan hetrd_plan(int m, int batch) {
  // the kernel's static arrays (about 1 KB) share the per-block limit with the dynamic part
  const size_t smax = (size_t)device_attr(cudaDevAttrMaxSharedMemoryPerBlockOptin, 232448) - 2048;
  const size_t el = sizeof(double2), vec = 7 * (size_t)m * el, part = (size_t)(HETRD_NT / 32) * m * el;
  int most = 1;
  for (int CL = 8; CL >= 1; CL >>= 1) {
    if (CL > 1 && (m / CL < (4 * batch * CL <= SMS ? 20 : 32) || batch > hetrd_clusters(CL))) continue;
    most = std::max(most, CL);
    const size_t rows = hetrd_row_elems(m, CL) * el;
    if (rows + vec + part <= smax) return HetrdPlan{CL, false, false, rows + vec + part};
    if (rows + vec <= smax) return HetrdPlan{CL, false, true, rows + vec};
  }
  return HetrdPlan{most, true, false, vec + part};
}

static EigScratch carve_eig(void* base, int m, int R, int batch, size_t* bytes) {
  Carver cv(base);
  EigScratch e;
  e.d = cv.take<double>((size_t)batch * m);
  e.f = cv.take<double>((size_t)batch * m);
  e.alpha = cv.take<double2>((size_t)batch * m);
  e.delta = cv.take<double2>((size_t)batch * m);
  e.Hv = cv.take<double2>((size_t)batch * m * m);
  e.Z = cv.take<double>((size_t)batch * m * R);
  e.lu = cv.take<double>((size_t)batch * 5 * m * R);
  e.tnorm = cv.take<double>((size_t)batch);
  e.Sg = e.Cp = nullptr;
  const HetrdPlan pl = hetrd_plan(m, batch);
  // CL CTAs of a slice own at most m(m+1)/2 + CL m packed elements together (CL <= 8)
  if (pl.global_rows) e.Sg = cv.take<double2>((size_t)batch * ((size_t)m * (m + 1) / 2 + 8 * (size_t)m));
  if (pl.cp_global) e.Cp = cv.take<double2>((size_t)batch * pl.CL * (HETRD_NT / 32) * m);
  if (bytes) *bytes = cv.bytes();
  return e;
}

size_t eig_scratch_bytes(int m, int R, int batch) {
  size_t b = 0;
  carve_eig(nullptr, m, R, batch, &b);
  return b;
}

template <typename C, int CL, bool GS>
static int launch_hetrd_t(const double2* G, long ldg, long sG, int m, int batch, const EigScratch& e,
                          const HetrdPlan& pl, cudaStream_t s) {
  auto kern = k_hetrd<C, CL, GS>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem) != cudaSuccess) {
    cudaGetLastError();
    return TSVD_ERR_CUDA;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(batch * CL);
  cfg.blockDim = dim3(HETRD_NT);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, kern, G, ldg, sG, m, (int)hetrd_row_elems(m, CL), e, pl.cp_global ? 1 : 0) !=
      cudaSuccess) {
    cudaGetLastError();
    return TSVD_ERR_CUDA;
  }
  TSVD_LAUNCHED();
  return TSVD_OK;
}

template <typename C, bool GS>
static int launch_hetrd(const double2* G, long ldg, long sG, int m, int batch, const EigScratch& e,
                        const HetrdPlan& pl, cudaStream_t s) {
  switch (pl.CL) {
    case 8: return launch_hetrd_t<C, 8, GS>(G, ldg, sG, m, batch, e, pl, s);
    case 4: return launch_hetrd_t<C, 4, GS>(G, ldg, sG, m, batch, e, pl, s);
    case 2: return launch_hetrd_t<C, 2, GS>(G, ldg, sG, m, batch, e, pl, s);
    default: return launch_hetrd_t<C, 1, GS>(G, ldg, sG, m, batch, e, pl, s);
  }
}

template <typename C>
int herm_eig_topR(double2* G, long ldg, long sG, int m, int R, int batch, double* lam, C* U, long ldu, long sU,
                  void* scratch, int* status, cudaStream_t s) {
  (void)status;
  if (m <= 0 || R <= 0 || batch <= 0) return TSVD_OK;
  if (R > m || R > 128 || m > 512) return TSVD_ERR_UNSUPPORTED;  // one or two vector entries per thread of k_hetrd
  EigScratch e = carve_eig(scratch, m, R, batch, nullptr);
  // FP32 path (C = float2): double-float reduction; FP64 path: FP64
  constexpr bool kDoubleFloat = std::is_same<C, float2>::value;
  {
    TSVD_STAGE("eig_hetrd", s);
    const HetrdPlan pl = hetrd_plan(m, batch);
    using T = typename std::conditional<kDoubleFloat, cdf, double2>::type;
    if (pl.global_rows) TSVD_TRY((launch_hetrd<T, true>(G, ldg, sG, m, batch, e, pl, s)));
    else TSVD_TRY((launch_hetrd<T, false>(G, ldg, sG, m, batch, e, pl, s)));
  }
  {
    TSVD_STAGE("eig_bisect", s);
    const size_t smem_b = (size_t)m * (2 * sizeof(double) + sizeof(float4) + sizeof(float2));
    // FP32 path: eigenvalues to 3e-13 of ||T|| (the vectors and the outputs are FP32; the
    // smallest kept sigma^2 is far above that); FP64 path: to the eigenvalue's own precision
    const double abs_tol = kDoubleFloat ? 3e-13 : 0.0;
    k_bisect<<<dim3(cdiv(R, BIS_WARPS), batch), BIS_WARPS * 32, smem_b, s>>>(m, R, e, lam, abs_tol);
    TSVD_LAUNCHED();
  }
  {
    TSVD_STAGE("eig_invit", s);
    const size_t smem_tp = (3 + (size_t)TP_THREADS) * m * sizeof(double);
    if (smem_tp > 48 * 1024)
      cudaFuncSetAttribute(k_tridiag_pairs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_tp);
    // solves: 3 (FP64 path), 2 on the FP32 path (eigenvalues to 3e-13 ||T|| already make one solve
    // amplify the wanted direction by gap / 3e-13; the vectors end in FP32)
    if (kDoubleFloat) {
      auto go = [&](auto kern, int nth, bool smf) {
        const size_t smem_df = tp_df_smem(m, nth, smf);
        if (smem_df > 40 * 1024 &&
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_df) != cudaSuccess) {
          cudaGetLastError();
          return TSVD_ERR_CUDA;
        }
        kern<<<dim3(cdiv(R, nth), batch), nth, smem_df, s>>>(m, R, e, lam, 2);
        return TSVD_OK;
      };
      if (tp_df_smem(m, 16, true) <= 200 * 1024) TSVD_TRY(go(k_tridiag_pairs_df<16, true>, 16, true));
      else TSVD_TRY(go(k_tridiag_pairs_df<TP_THREADS, false>, TP_THREADS, false));
    } else {
      k_tridiag_pairs<<<dim3(cdiv(R, TP_THREADS), batch), TP_THREADS, smem_tp, s>>>(m, R, e, lam, 3);
    }
    TSVD_LAUNCHED();
  }
  {
    TSVD_STAGE("eig_cluster", s);
    size_t smem_co = (size_t)R * m * (kDoubleFloat ? sizeof(float) : sizeof(double));
    using CoKernel = void (*)(int, int, EigScratch, const double*);
    CoKernel co = kDoubleFloat ? (CoKernel)k_cluster_orth<float, true> : (CoKernel)k_cluster_orth<double, true>;
    // the kernel's static arrays (the cluster Gram and its reductions) take about 17 KB of the
    // per-block limit
    const size_t smax_co = (size_t)device_attr(cudaDevAttrMaxSharedMemoryPerBlockOptin, 232448) - 20 * 1024;
    if (smem_co > smax_co) {  // vectors stay in global memory
      co = k_cluster_orth<double, false>;
      smem_co = 0;
    }
    // the kernel's static shared memory (the cluster Gram, 16 KB) counts against the same 48 KB default
    if (smem_co > 0 && cudaFuncSetAttribute(co, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_co) !=
                           cudaSuccess) {
      cudaGetLastError();
      return TSVD_ERR_CUDA;
    }
    co<<<batch, CO_THREADS, smem_co, s>>>(m, R, e, lam);
    TSVD_LAUNCHED();
  }
  TSVD_STAGE("eig_backtransform", s);
  using VT = typename std::conditional<kDoubleFloat, float2, double2>::type;  // the Householder vectors as stored
  return launch_backtransform<C, VT>(m, R, batch, e, U, ldu, sU, s);
}
template int herm_eig_topR<double2>(double2*, long, long, int, int, int, double*, double2*, long, long, void*, int*,
                                    cudaStream_t);
template int herm_eig_topR<float2>(double2*, long, long, int, int, int, double*, float2*, long, long, void*, int*,
                                   cudaStream_t);

// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_sigma(const double* __restrict__ lam, int n, double* __restrict__ sig, cx_t<T>* __restrict__ Sh,
                        int* status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double l = lam[i];
  if (!isfinite(l)) atomicExch(status, TSVD_ERR_NOT_CONVERGED);
  const double sg = sqrt(fmax(l, 0.0));
  if (sig) sig[i] = sg;
  Sh[i] = mkc((T)sg, T(0));
}

template <typename T>
int sigma_from_lambda(const double* lam, int R, int batch, double* sig, cx_t<T>* Sh, cudaStream_t s, int* status) {
  const int n = R * batch;
  if (n <= 0) return TSVD_OK;
  k_sigma<T><<<cdiv(n, 256), 256, 0, s>>>(lam, n, sig, Sh, status);
  TSVD_LAUNCHED();
  return TSVD_OK;
}
template int sigma_from_lambda<double>(const double*, int, int, double*, double2*, cudaStream_t, int*);
template int sigma_from_lambda<float>(const double*, int, int, double*, float2*, cudaStream_t, int*);

// 128 rows per CTA: the columns' FP64 roots and quotients once per CTA (2048 x 100 on 65 slices: 390 us
// with one per element, 38 so)
constexpr int SC_ROWS = 128;
template <typename T>
__global__ void __launch_bounds__(256) k_scale_cols(cx_t<T>* __restrict__ V, long ldv, long sV, int rows, int R,
                                                    const double* __restrict__ lam) {
  extern __shared__ __align__(16) unsigned char scsm[];
  T* inv = (T*)scsm;  // [R]
  const int b = blockIdx.y, i0 = blockIdx.x * SC_ROWS;
  for (int r = threadIdx.x; r < R; r += 256) {
    const double sg = sqrt(fmax(lam[(long)b * R + r], 0.0));
    inv[r] = (sg > 0.0) ? (T)(1.0 / sg) : T(0);
  }
  __syncthreads();
  const int total = min(SC_ROWS, rows - i0) * R;
  cx_t<T>* p = V + (long)b * sV + (long)i0 * ldv;
#pragma unroll 4
  for (int e = threadIdx.x; e < total; e += 256) {
    const int i = e / R, r = e - i * R;
    p[(long)i * ldv + r] = cscale(p[(long)i * ldv + r], inv[r]);
  }
}

template <typename T>
int scale_columns_inv(cx_t<T>* V, long ldv, long sV, int rows, int R, const double* lam, int batch, cudaStream_t s) {
  if (rows <= 0 || R <= 0 || batch <= 0) return TSVD_OK;
  k_scale_cols<T><<<dim3(cdiv(rows, SC_ROWS), batch), 256, R * sizeof(T), s>>>(V, ldv, sV, rows, R, lam);
  TSVD_LAUNCHED();
  return TSVD_OK;
}
template int scale_columns_inv<double>(double2*, long, long, int, int, const double*, int, cudaStream_t);
template int scale_columns_inv<float>(float2*, long, long, int, int, const double*, int, cudaStream_t);

}  // namespace tsvd
