// The lowest eigenvalues of batched Hermitian matrices C(k) (Eq.
// (eigenvalueproblem) in standard form) by filtered subspace iteration, for
// the solves that want a few branches of a large matrix.
//
// A reduction to tridiagonal form spends (16/3) n^3 flops per matrix on all n
// eigenvalues, in n or n/8 dependent steps.  The lowest nb <= 24 need one
// factorisation and a few dozen products with 32-column blocks:
//
//  1. FP32: the LDL^dagger of W (C/s + I) W (s of the size of the wanted
//     eigenvalues, W = diag(C/s + 1)^-1/2), its triangular inverse, and so
//     B = W L^-dagger D^-1 L^-1 W = (C/s + I)^-1 to FP32 accuracy, stored as two
//     BF16 terms (2^-17).  The wanted eigenvalues are the largest of B.
//  2. Rounds: an FP64 Rayleigh-Ritz step on the block X (32 vectors, the
//     wanted ones and guards) gives theta, X, and the FP64 residual
//     R = C X - X Theta; then X is filtered by a Chebyshev polynomial T_m of B
//     that is at most 1 on the unwanted part of the spectrum.  Written for
//     the change E of X instead of X itself,
//       T_j(l(B)) x = tau_j (x + E_j),   B x = mu (x - B r / s),  mu = s / (theta + s),
//     every term is a product of B (on the tensor cores) with the residual: the operator only
//     multiplies R, so its error shrinks with R and the rounds converge to
//     the eigenvectors of the FP64 matrix, not of B.
//  3. Certificate: theta_i is an upper bound of lambda_i; with rho a lower
//     bound of lambda_{m+1}, Lehmann's bound in its trace form (the residual
//     Gram matrix replaced by its trace) gives
//       lambda_i >= theta_i - sum_{c <= m} ||r_c||^2 / (rho - theta_c),  i <= m.
//     A matrix passes when that sum, and what the small eigenproblem may have
//     left of the Ritz values, are at most 64 eps64 max_r C_rr (the
//     backward error of a reduction to tridiagonal form and its bisection is
//     of that size; the sum overestimates the error, whose own gap is that to
//     the eigenvalues outside the block).  That rho is such a bound, so that
//     no eigenvalue was skipped, is shown by an FP32 Cholesky factorisation:
//     C + X_m T X_m^dagger, T >= 0, has rank m more than C, so if it is above sigma
//     then lambda_{m+1} is, whatever X_m and T are; see filt_cert_kernel for what the
//     rounding errors of the factorisation take from sigma.
//  4. Matrices that do not pass are reduced by the FP64 Householder reduction
//     and bisected (tridiag.cu, bisect.cu) in one launch each that returns at
//     once when there are none; nothing waits for the host.
//
// Measured (one GB300, whole FP64 solve with its assembly, the reduction to
// tridiagonal form before -> this): n = 882, 90 matrices, 18 branches
// 171 -> 26.2 ms; n = 1029, 30 matrices, 12 branches 136 -> 18.4 ms; n = 242,
// 70 matrices, 18 branches 16.9 -> 4.2 ms; n = 98, 30 matrices, 8 branches
// 3.86 -> 2.42 ms.  What bounds it at n = 882 is the FP32 factorisations (their
// pipe is 58 % busy at most) and the FP64 pipe in the Rayleigh-Ritz steps (32-column
// products at 2 FMA per clock and SM).
//
// What enters a result: C X, an exact-slice product of FP64 operands; the Gram
// matrices, FP64; the Ritz values, Rayleigh quotients in 48 bits with a bound; the
// rotated block and its residuals, 48 bits.
#include <float.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "bs_internal.h"

namespace {

constexpr int FB = BS_FILT_BLOCK;   // columns of the block (32)
constexpr int TB = 64;              // tile edge of the FP32 factorisation
constexpr int LDS = TB + 1;         // row stride of the diagonal blocks in shared memory
constexpr float TINY_PIVOT = 1e-6f; // of the scaled unit diagonal
constexpr int NS = BS_FILT_START;   // plane waves in the starting vectors
constexpr int GR = 64;              // rows per CTA of the Gram and rotation kernels
constexpr int STEER_DIGITS = 5;     // of C X in the steps that only steer (34 bits),
constexpr int LAST_STEER_DIGITS = 6;// and in the step before the first that can certify (41)

// ---------------------------------------------------------------- set-up
// Per matrix: the indices of the NS smallest diagonal entries (the plane waves
// of the starting vectors, filt_start_kernel), the shift s, the row scales
// w_r = (s / (C_rr + s))^1/2 and the largest diagonal entry.
__global__ void __launch_bounds__(256) filt_prep_kernel(const zd* __restrict__ C, int n, int np,
                                                        int nb, double sfac,
                                                        double* __restrict__ shift,
                                                        double* __restrict__ cmax,
                                                        int* __restrict__ ord,
                                                        float* __restrict__ w,
                                                        int* __restrict__ fail,
                                                        int* __restrict__ done) {
  extern __shared__ double dg[];
  const long long* key = reinterpret_cast<const long long*>(dg);
  __shared__ int so[NS];
  __shared__ double red[8];
  const int k = blockIdx.x, tid = threadIdx.x;
  const zd* ck = C + (size_t)k * n * n;
  double cm = 0.0;
  for (int r = tid; r < n; r += 256) {
    const double v = ck[(size_t)r * (n + 1)].x;
    dg[r] = v;
    cm = fmax(cm, fabs(v));
  }
  for (int o = 16; o > 0; o >>= 1) cm = fmax(cm, __shfl_xor_sync(0xffffffffu, cm, o));
  if ((tid & 31) == 0) red[tid >> 5] = cm;
  __syncthreads();
  for (int r = tid; r < n; r += 256) {
    // the diagonal is not negative, so its bit patterns order as its values do
    const long long v = key[r];
    int rank = 0;
    for (int c = 0; c < n; ++c) rank += key[c] < v || (key[c] == v && c < r);
    if (rank < NS) so[rank] = r;
  }
  __syncthreads();
  // (of the eighth entry at least: a shift far below the block's eigenvalues lets
  // the filters grow the lowest branches beyond what a Gram matrix can separate)
  double s = sfac * dg[so[max(nb, 8) - 1]];
  // a zero or non-finite diagonal: any scale will do, the certificate decides
  if (!(s > 1e-250) || !(s < 1e250)) s = 1.0;   // (to_float takes |es| < 897)
  if (tid < min(n, NS)) ord[(size_t)k * NS + tid] = so[tid];
  if (tid == 0) {
    double v = 0.0;
    for (int q = 0; q < 8; ++q) v = fmax(v, red[q]);
    shift[k] = s;
    cmax[k] = v;
    fail[k] = 0;
    done[k] = 0;
  }
  const double is = 1.0 / s;
  for (int r = tid; r < np; r += 256)
    w[(size_t)k * np + r] = r < n ? rsqrtf(fmaxf((float)(dg[r] * is + 1.0), 1e-30f)) : 0.f;
}

// (bi, bk), bi >= bk, of the l-th lower-triangular tile (row-major order)
__device__ __forceinline__ void tile_of(int l, int& bi, int& bk) {
  int r = (int)((sqrtf(8.0f * (float)l + 1.0f) - 1.0f) * 0.5f);
  while ((r + 1) * (r + 2) / 2 <= l) ++r;
  while (r * (r + 1) / 2 > l) --r;
  bi = r;
  bk = l - r * (r + 1) / 2;
}

// (float)x by integer arithmetic (round half up; below the FP32 normal range
// 0): the FP64 to FP32 conversion runs on the FP64 pipe, 2 per clock and SM
// (the scaling of 90 matrices of n = 882: 456 us with it, 158 us without).
// es: (float)(x 2^-es).  Everything in FP32 is held in units of 2^es, es the
// exponent of the matrix's shift, so that no unit of length or mass takes the
// entries, or the squares of Ritz values that the Jacobi sums, out of its range.
__device__ __forceinline__ float to_float(double x, int es = 0) {
  const long long b = __double_as_longlong(x);
  const int e = ((int)(b >> 52) & 0x7ff) - es;
  if ((unsigned)(e - (1023 - 126)) > 252u) {
    if (e - 1023 < 127 && e + es < 0x7ff) return 0.f;
    return e + es == 0x7ff ? (float)x : x < 0.0 ? -INFINITY : INFINITY;
  }
  const unsigned m = (unsigned)((b + (1LL << 28)) >> 29) - ((unsigned)(1023 - 127 + es) << 23);
  return __uint_as_float((m & 0x7fffffffu) | ((unsigned)(b >> 32) & 0x80000000u));
}
// exponent of a positive normal number, and 2^e
__device__ __forceinline__ int exponent(double s) {
  return ((__double2hiint(s) >> 20) & 0x7ff) - 1023;
}
__device__ __forceinline__ double exp2i(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// A <- W (C / s + I) W, lower 64-tiles, FP32, identity in the padding
__global__ void __launch_bounds__(256) filt_scale_kernel(const zd* __restrict__ C, int n, int np,
                                                         const double* __restrict__ shift,
                                                         const float* __restrict__ w,
                                                         zf* __restrict__ A, int* __restrict__ neg,
                                                         int* __restrict__ flag) {
  int bi, bk;
  tile_of(blockIdx.x, bi, bk);
  const int k = blockIdx.y, tid = threadIdx.x;
  const zd* ck = C + (size_t)k * n * n;
  const float* wk = w + (size_t)k * np;
  zf* ak = A + (size_t)k * np * np;
  const double is = 1.0 / shift[k];
  const int es = exponent(shift[k]);
  const float fs = (float)(is * exp2i(es));
  if (blockIdx.x == 0 && tid == 0) {
    neg[k] = 0;
    flag[k] = 0;
  }
  const int r = bi * TB + (tid & 63);
  const float wr = r < n ? wk[r] : 0.f;
#pragma unroll 4
  for (int q = tid >> 6; q < TB; q += 4) {
    const int c = bk * TB + q;
    zf v = make_float2(r == c ? 1.f : 0.f, 0.f);
    if (r < n && c < n) {
      const zd z = ck[(size_t)c * n + r];
      const float f = wr * wk[c];
      if (r == c) {
        v = make_float2((float)(z.x * is + 1.0) * f, 0.f);
      } else {
        v = make_float2(to_float(z.x, es) * fs * f, to_float(z.y, es) * fs * f);
      }
    }
    ak[(size_t)c * np + r] = v;
  }
}

// ---------------------------------------------------------------- FP32 LDL^dagger
// Blocked right-looking factorisation, panels of 64 columns, for a batch of
// matrices padded to a multiple of 64.  As in the other factorisations of the
// library each diagonal block is factored and stored by exactly one CTA, in
// a launch whose other CTAs do not read it: the first by ldl64_diag_kernel,
// block j + 1 by the CTA of ldl64_update_kernel(j) that has just updated it.
// That CTA also inverts the unit lower factor (stored in the diagonal block
// of X), so the block rows below become plain 64 x 64 x 64 products.

// 1 / p by the hardware approximation and, in FP64, one cubic correction
// (1 + e + e^2, e = 1 - p r below 2^-22; plain division outside the FP32 range)
__device__ __forceinline__ float quick_rcp(float p) { return __fdividef(1.f, p); }
__device__ __forceinline__ double quick_rcp(double p) {
  if (!(p > 1e-36 && p < 1e36)) return 1.0 / p;
  float rf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"((float)p));
  const double r = (double)rf, e = fma(-p, r, 1.0);
  return fma(fma(e, e, e), r, r);
}

// LDL^dagger of the 32 x 32 lower triangle S and its inverse unit factor X (row
// strides LD; X's strict upper part is not written), 256 threads: on return
// L D below the diagonal of S, the pivots on it and 1 / pivot in pinv.  ok(p, c)
// passes a pivot or replaces it.  Thread t owns up to three entries (r, s) of
// the lower triangle: step c < s updates S[r][s] -= l conj(S[s][c]), step
// c >= s X[r][s] -= l X[c][s] (kept in a register until row r is next), so the
// three are independent, loads need no branches, and rows that are done leave
// the pipe (FP64 issues a warp in 16 cycles).  One barrier per step; the
// thread that finishes a pivot inverts it, so no other issues a division.
template <typename R, int LD, typename Ok>
__device__ __forceinline__ void ldl32_inverse(typename Cplx<R>::T* S, typename Cplx<R>::T* X,
                                              R* pinv, Ok ok) {
  typedef typename Cplx<R>::T T;
  const int tid = threadIdx.x;
  int er[3], es[3];
  T x[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int e = tid + 256 * q;
    int r = 0, c = 0;   // (0, 0) is never updated
    if (e < 32 * 33 / 2) tile_of(e, r, c);
    er[q] = r;
    es[q] = c;
    x[q] = Cplx<R>::make(r == c ? (R)1 : (R)0, (R)0);
    X[r * LD + c] = x[q];
  }
  if (tid == 0) {
    const R p = ok(S[0].x, 0);
    S[0] = Cplx<R>::make(p, (R)0);
    pinv[0] = quick_rcp(p);
  }
  __syncthreads();
  for (int c = 0; c < 32; ++c) {
    T l[3], u[3], v[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int r = er[q], s = es[q];
      const bool f = s > c;
      l[q] = S[r * LD + c];
      const T* up = f ? S + s * LD + c : X + c * LD + s;
      u[q] = *up;
      const T sv = S[r * LD + s];
      v[q] = f ? sv : x[q];
      u[q].y = f ? -u[q].y : u[q].y;
    }
    const R inv = pinv[c];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int r = er[q], s = es[q];
      if (r <= c) continue;
      T w = zfnma(zscale(l[q], inv), u[q], v[q]);
      if (s > c) {
        if (s == c + 1 && r == s) {
          const R p = ok(w.x, r);
          w = Cplx<R>::make(p, (R)0);
          pinv[r] = quick_rcp(p);
        }
        S[r * LD + s] = w;
      } else {
        x[q] = w;
        if (r == c + 1) X[r * LD + s] = w;   // the row is final: the next steps read it
      }
    }
    __syncthreads();
  }
}

// The 32 x 32 diagonal block at b0 of the 64 x 64 block: see ldl32_inverse
__device__ __forceinline__ void ldl32_block(zf* S, zf* Xs, float* d, float* pinv, int b0, int* bad) {
  ldl32_inverse<float, LDS>(S + b0 * (LDS + 1), Xs + b0 * (LDS + 1), pinv + b0,
                       [&](float p, int c) {
                         if (!(fabsf(p) >= TINY_PIVOT)) {
                           *bad = 1;
                           p = p < 0.f ? -TINY_PIVOT : TINY_PIVOT;
                         }
                         d[b0 + c] = p;
                         return p;
                       });
}

// S: the 64 x 64 lower triangle (row-major, stride LDS); on return L D below
// the diagonal and D on it.  Xs: its inverse unit factor.  Two 32 x 32 blocks
// and 32 x 32 x 32 products between them: 64 dependent steps over the whole
// block took 62 us per launch, this 39 us, and this chain is what every panel waits for.
__device__ __forceinline__ void ldl64_block(zf* S, zf* Xs, float* d, int* bad) {
  __shared__ float pinv[TB];
  const int tid = threadIdx.x, r = tid & 31, w = tid >> 5;
  ldl32_block(S, Xs, d, pinv, 0, bad);
  zf* S21 = S + 32 * LDS;
  zf v[4];
  // L21 D1 = A21 X11^dagger
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = w + 8 * j;
    v[j] = make_float2(0.f, 0.f);
    for (int t = 0; t <= c; ++t) v[j] = zfmac(S21[r * LDS + t], Xs[c * LDS + t], v[j]);
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 4; ++j) S21[r * LDS + w + 8 * j] = v[j];
  __syncthreads();
  // A22 -= (L21 D1) D1^-1 (L21 D1)^dagger, and M = L21 X11 into the unused
  // block of S above the diagonal
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = w + 8 * j;
    zf a = make_float2(0.f, 0.f), m = a;
#pragma unroll 4
    for (int t = 0; t < 32; ++t) {
      const zf l = zscale(S21[r * LDS + t], pinv[t]);
      a = zfmac(l, S21[c * LDS + t], a);
      if (t >= c) m = zfma(l, Xs[t * LDS + c], m);
    }
    if (c <= r) S21[r * LDS + 32 + c] = zsub(S21[r * LDS + 32 + c], a);
    S[r * LDS + 32 + c] = m;
  }
  __syncthreads();
  ldl32_block(S, Xs, d, pinv, 32, bad);
  // X21 = -X22 M, X12 = 0
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = w + 8 * j;
    zf x = make_float2(0.f, 0.f);
    for (int t = 0; t <= r; ++t) x = zfnma(Xs[(32 + r) * LDS + 32 + t], S[t * LDS + 32 + c], x);
    Xs[(32 + r) * LDS + c] = x;
    Xs[r * LDS + 32 + c] = make_float2(0.f, 0.f);
  }
  __syncthreads();
}

// factor the diagonal block at j0 held in S and store L (unit), D, X
__device__ __forceinline__ void ldl64_diag(zf* a, zf* x, float* dk, int np, int j0, int k, zf* S, zf* Xs, float* d,
                           int* bad, int* neg, int* flag) {
  const int tid = threadIdx.x, r = tid & 63;
  if (tid == 0) *bad = 0;
  __syncthreads();
  ldl64_block(S, Xs, d, bad);
  for (int c = tid >> 6; c < TB; c += 4) {
    zf v = make_float2(0.f, 0.f);
    if (r > c) v = zscale(S[r * LDS + c], 1.f / d[c]);
    if (r == c) v.x = d[c];
    if (r >= c) a[(size_t)(j0 + c) * np + j0 + r] = v;
    x[(size_t)(j0 + c) * np + j0 + r] = r >= c ? Xs[r * LDS + c] : make_float2(0.f, 0.f);
  }
  if (tid < TB) dk[j0 + tid] = d[tid];
  if (tid == 0) {
    int cnt = 0;
    for (int c = 0; c < TB; ++c) cnt += d[c] < 0.f;
    neg[k] += cnt;   // one CTA per matrix and launch, launches in order
    if (*bad) flag[k] = 1;
  }
}

__global__ void __launch_bounds__(256) ldl64_diag_kernel(zf* __restrict__ A, zf* __restrict__ X,
                                                         int np, float* __restrict__ dv,
                                                         int* __restrict__ neg,
                                                         int* __restrict__ flag,
                                                         const int* __restrict__ skip) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ float d[TB];
  __shared__ int bad;
  if (skip && skip[blockIdx.x]) return;
  zf* S = reinterpret_cast<zf*>(dsm);
  zf* Xs = S + TB * LDS;
  const int k = blockIdx.x, tid = threadIdx.x, r = tid & 63;
  zf* a = A + (size_t)k * np * np;
  for (int c = tid >> 6; c < TB; c += 4)
    if (r >= c) S[r * LDS + c] = a[(size_t)c * np + r];
  __syncthreads();
  ldl64_diag(a, X + (size_t)k * np * np, dv + (size_t)k * np, np, 0, k, S, Xs, d, &bad, neg, flag);
}

// 64 x 64 x K product on 256 threads, 4 x 4 complex per thread:
// acc[i][j] += sum_t As[t][row(i)] op(Bs[t][col(j)]), rows 2 tx + {0, 1, 32, 33} and
// columns 2 ty + {0, 1, 32, 33}, so that two 16-byte loads fetch each operand
// (eight 8-byte ones kept the shared-memory pipe half busy: 205 -> 183 us per
// update launch of 90 x 896^2).  Rows t of the tiles are LA, LB apart.
__device__ __forceinline__ int own(int x, int i) { return 2 * x + (i & 1) + 32 * (i >> 1); }

template <bool CONJB, int LA = TB, int LB = TB, int K = TB>
__device__ __forceinline__ void mm64(const zf* __restrict__ As, const zf* __restrict__ Bs,
                                     zf (&acc)[4][4]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const float4* A4 = reinterpret_cast<const float4*>(As) + tx;
  const float4* B4 = reinterpret_cast<const float4*>(Bs) + ty;
#pragma unroll 8
  for (int t = 0; t < K; ++t) {
    const float4 a0 = A4[t * (LA / 2)], a1 = A4[t * (LA / 2) + 16];
    const float4 b0 = B4[t * (LB / 2)], b1 = B4[t * (LB / 2) + 16];
    const zf a[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w), make_float2(a1.x, a1.y),
                     make_float2(a1.z, a1.w)};
    const zf b[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y),
                     make_float2(b1.z, b1.w)};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = CONJB ? zfmac(a[i], b[j], acc[i][j])
                                                    : zfma(a[i], b[j], acc[i][j]);
  }
}

// a 64 x 64 tile of a column-major matrix into dst[t * 64 + r] (t = column)
__device__ __forceinline__ void load_tile(zf* dst, const zf* src, int np) {
  float4* d4 = reinterpret_cast<float4*>(dst);
  for (int e = threadIdx.x; e < TB * TB / 2; e += 256) {
    const int t = e >> 5, r2 = e & 31;
    d4[t * 32 + r2] = *reinterpret_cast<const float4*>(src + (size_t)t * np + 2 * r2);
  }
}

// the transpose of a 64 x 64 tile: dst[t * LDT + c] = src[t + c np], scaled by
// sc[t] (optional).  A warp takes eight columns of eight rows t: 64-byte segments
// of global memory, two-way conflicts in shared memory.
constexpr int LDT = TB + 4;
__device__ __forceinline__ void load_tile_t(zf* dst, const zf* src, int np,
                                            const float* sc = nullptr) {
  const int tid = threadIdx.x, t2 = (tid & 3) * 2, c0 = tid >> 2;   // 64 columns, 8 rows a pass
#pragma unroll 4
  for (int t0 = 0; t0 < TB; t0 += 8) {
    const int t = t0 + t2;
    const float4 v = *reinterpret_cast<const float4*>(src + (size_t)c0 * np + t);
    const float f0 = sc ? sc[t] : 1.f, f1 = sc ? sc[t + 1] : 1.f;
    dst[t * LDT + c0] = make_float2(v.x * f0, v.y * f0);
    dst[(t + 1) * LDT + c0] = make_float2(v.z * f1, v.w * f1);
  }
}

// block row i = j + 1 + blockIdx.x: L_i1 = A_i1 L11^-dagger D1^-1
__global__ void __launch_bounds__(256) ldl64_panel_kernel(zf* __restrict__ A,
                                                          const zf* __restrict__ X, int np,
                                                          int j0, const int* __restrict__ skip) {
  if (skip && skip[blockIdx.y]) return;
  extern __shared__ __align__(16) unsigned char dsm[];
  zf* As = reinterpret_cast<zf*>(dsm);
  zf* Bs = As + TB * TB;
  __shared__ float di[TB];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  zf* a = A + (size_t)blockIdx.y * np * np;
  const int i0 = j0 + TB * (blockIdx.x + 1);
  zf* ai = a + (size_t)j0 * np + i0;
  load_tile(As, ai, np);
  load_tile(Bs, X + (size_t)blockIdx.y * np * np + (size_t)j0 * np + j0, np);
  if (tid < TB) di[tid] = 1.f / a[(size_t)(j0 + tid) * (np + 1)].x;
  __syncthreads();
  zf acc[4][4] = {};
  mm64<true>(As, Bs, acc);   // Y[r][c] = sum_t A[r][t] conj(L11^-1[c][t])
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = own(ty, j);
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      const zf u = zscale(acc[i][j], di[c]), v = zscale(acc[i + 1][j], di[c]);
      *reinterpret_cast<float4*>(ai + (size_t)c * np + own(tx, i)) = make_float4(u.x, u.y, v.x, v.y);
    }
  }
}

// trailing update A_ik -= L_i1 D1 L_k1^dagger; the first tile's CTA factors
// the next diagonal block
__global__ void __launch_bounds__(256) ldl64_update_kernel(zf* __restrict__ A, zf* __restrict__ X,
                                                           int np, int j0, float* __restrict__ dv,
                                                           int* __restrict__ neg,
                                                           int* __restrict__ flag,
                                                           const int* __restrict__ skip) {
  if (skip && skip[blockIdx.y]) return;
  extern __shared__ __align__(16) unsigned char dsm[];
  zf* As = reinterpret_cast<zf*>(dsm);
  zf* Bs = As + TB * LDS;
  __shared__ float d[TB];
  __shared__ int bad;
  int bi, bk;
  tile_of(blockIdx.x, bi, bk);
  zf* a = A + (size_t)blockIdx.y * np * np;
  const int i0 = j0 + TB * (bi + 1), k0 = j0 + TB * (bk + 1);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  if (tid < TB) d[tid] = a[(size_t)(j0 + tid) * (np + 1)].x;
  load_tile(Bs, a + (size_t)j0 * np + k0, np);
  __syncthreads();
  {
    float4* d4 = reinterpret_cast<float4*>(As);
    const zf* src = a + (size_t)j0 * np + i0;
    for (int e = tid; e < TB * TB / 2; e += 256) {
      const int t = e >> 5, r2 = e & 31;
      float4 v = *reinterpret_cast<const float4*>(src + (size_t)t * np + 2 * r2);
      const float dt = d[t];
      v.x *= dt;
      v.y *= dt;
      v.z *= dt;
      v.w *= dt;
      d4[t * 32 + r2] = v;
    }
  }
  __syncthreads();
  zf acc[4][4] = {};
  mm64<true>(As, Bs, acc);
  const bool first = blockIdx.x == 0;
  if (first) __syncthreads();   // As is reused for the block below
  // (entries above the diagonal of a diagonal tile are written too: nothing reads them)
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = own(ty, j);
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      const int r = own(tx, i);
      float4* o = reinterpret_cast<float4*>(a + (size_t)(k0 + c) * np + i0 + r);
      float4 v = *o;
      v.x -= acc[i][j].x;
      v.y -= acc[i][j].y;
      v.z -= acc[i + 1][j].x;
      v.w -= acc[i + 1][j].y;
      if (first) {
        As[r * LDS + c] = make_float2(v.x, v.y);
        As[(r + 1) * LDS + c] = make_float2(v.z, v.w);
      } else {
        *o = v;
      }
    }
  }
  if (first) {
    __syncthreads();
    ldl64_diag(a, X + (size_t)blockIdx.y * np * np, dv + (size_t)blockIdx.y * np, np, i0, blockIdx.y, As, Bs, d, &bad, neg, flag);
  }
}

// X_ij = -X_ii sum_{k=j}^{i-1} L_ik X_kj for block diagonal i - j = dd
__global__ void __launch_bounds__(256) trinv64_kernel(const zf* __restrict__ A, zf* __restrict__ X,
                                                      int np, int dd) {
  extern __shared__ __align__(16) unsigned char dsm[];
  zf* As = reinterpret_cast<zf*>(dsm);
  zf* Bs = As + TB * TB;   // [t][col], stride LDT
  const int bj = blockIdx.x, bi = bj + dd;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const zf* l = A + (size_t)blockIdx.y * np * np;
  zf* x = X + (size_t)blockIdx.y * np * np;
  zf acc[4][4] = {};
  for (int bk = bj; bk < bi; ++bk) {
    __syncthreads();
    load_tile(As, l + (size_t)bk * TB * np + bi * TB, np);
    load_tile_t(Bs, x + (size_t)bj * TB * np + bk * TB, np);
    __syncthreads();
    mm64<false, TB, LDT>(As, Bs, acc);
  }
  __syncthreads();
  load_tile(As, x + (size_t)bi * TB * np + bi * TB, np);
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      Bs[own(tx, i) * LDT + own(ty, j)] = acc[i][j];
      acc[i][j] = make_float2(0.f, 0.f);
    }
  __syncthreads();
  mm64<false, TB, LDT>(As, Bs, acc);
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 4; i += 2)
      *reinterpret_cast<float4*>(x + (size_t)(bj * TB + own(ty, j)) * np + bi * TB + own(tx, i)) =
          make_float4(-acc[i][j].x, -acc[i][j].y, -acc[i + 1][j].x, -acc[i + 1][j].y);
}

__device__ __forceinline__ float fsqrt(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// B = W X^dagger D^-1 X W (X = L^-1), 64-tiles (bi, bk) and their mirrors,
// straight to the BF16 split [Re | Im] hi, [Re | Im] lo of rows of 4 np.  The
// tile sums over the block rows t >= bi; the longest sums come first.  rsum (block
// column, row): the tile's part of the row sums of |X^dagger D^-1 X|, for
// filt_kappa_kernel.
__global__ void __launch_bounds__(256) filt_operator_kernel(const zf* __restrict__ X,
                                                            const float* __restrict__ d, int np,
                                                            const float* __restrict__ w,
                                                            uint16_t* __restrict__ Bp,
                                                            float* __restrict__ rsum) {
  extern __shared__ __align__(16) unsigned char dsm[];
  zf* As = reinterpret_cast<zf*>(dsm);   // [t][column], stride LDT
  zf* Bs = As + TB * LDT;
  __shared__ float di[TB];
  int bi, bk;
  tile_of(blockIdx.x, bi, bk);
  const int k = blockIdx.y, tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const zf* x = X + (size_t)k * np * np;
  const float* dk = d + (size_t)k * np;
  const float* wk = w + (size_t)k * np;
  zf acc[4][4] = {};   // conj(B_rc): the columns' conjugates times the rows
  for (int t0 = bi * TB; t0 < np; t0 += TB) {
    __syncthreads();
    if (tid < TB) di[tid] = 1.f / dk[t0 + tid];
    load_tile_t(Bs, x + (size_t)bk * TB * np + t0, np);
    __syncthreads();
    load_tile_t(As, x + (size_t)bi * TB * np + t0, np, di);
    __syncthreads();
    mm64<true, LDT, LDT>(As, Bs, acc);   // sum_t x_tr conj(x_tc) / d_t
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float wc = wk[bk * TB + own(ty, j)];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      As[own(tx, i) * LDS + own(ty, j)] =
          zscale(zconj(acc[i][j]), wk[bi * TB + own(tx, i)] * wc);
  }
  // row sums of |tile| and of its mirror (the padding, an identity, adds rows of sum 1)
  float rp[4] = {}, cp[4] = {};
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float a = fsqrt(fmaf(acc[i][j].x, acc[i][j].x, acc[i][j].y * acc[i][j].y));
      rp[i] += a;
      cp[j] += a;
    }
  float(*red)[TB] = reinterpret_cast<float(*)[TB]>(Bs);   // [ty][row]
  float* rs = rsum + (size_t)k * (np / TB) * np;
#pragma unroll
  for (int i = 0; i < 4; ++i) red[ty][own(tx, i)] = rp[i];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) cp[j] += __shfl_xor_sync(0xffffffffu, cp[j], o);
    if (tx == 0 && bi != bk) rs[(size_t)bi * np + bk * TB + own(ty, j)] = cp[j];
  }
  __syncthreads();
  if (tid < TB) {
    float v = 0.f;
#pragma unroll
    for (int q = 0; q < 16; ++q) v += red[q][tid];
    rs[(size_t)bk * np + bi * TB + tid] = v;
  }
  uint16_t* b = Bp + (size_t)k * np * 4 * np;
  for (int h = 0; h < (bi == bk ? 1 : 2); ++h) {
    // h = 0: rows of bi, columns of bk; h = 1: the conjugate mirror
    const int r0 = (h ? bk : bi) * TB, c0 = (h ? bi : bk) * TB;
    for (int e = tid; e < TB * TB / 2; e += 256) {
      const int r = e >> 5, c = (e & 31) * 2;
      uint32_t v[4];
      uint16_t q[2][4];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const zf y = h ? zconj(As[(c + u) * LDS + r]) : As[r * LDS + c + u];
        bs_bf16_split(y.x, q[u][0], q[u][2]);
        bs_bf16_split(y.y, q[u][1], q[u][3]);
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) v[m] = (uint32_t)q[0][m] | ((uint32_t)q[1][m] << 16);
      uint16_t* o = b + (size_t)(r0 + r) * 4 * np + c0 + c;
#pragma unroll
      for (int m = 0; m < 4; ++m) *reinterpret_cast<uint32_t*>(o + (size_t)m * np) = v[m];
    }
  }
}

// kappa = the largest row sum of |A^-1|, A = W (C / s + I) W: an upper bound of
// its norm, so that s / w^2 = diag(C) + s <= kappa (C + s) as quadratic forms.
// Infinite where the factorisation met a pivot that is not positive.
__global__ void __launch_bounds__(256) filt_kappa_kernel(const float* __restrict__ rsum, int np,
                                                         const int* __restrict__ neg,
                                                         const int* __restrict__ flag,
                                                         double* __restrict__ kappa) {
  __shared__ float red[8];
  const int k = blockIdx.x, tid = threadIdx.x, nt = np / TB;
  const float* rs = rsum + (size_t)k * nt * np;
  float m = 0.f;
  for (int r = tid; r < np; r += 256) {
    float v = 0.f;
#pragma unroll 4
    for (int q = 0; q < nt; ++q) v += rs[(size_t)q * np + r];
    if (!(v <= m)) m = v == v ? v : INFINITY;
  }
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((tid & 31) == 0) red[tid >> 5] = m;
  __syncthreads();
  if (tid == 0) {
    for (int q = 0; q < 8; ++q) m = fmaxf(m, red[q]);
    kappa[k] = neg[k] || flag[k] ? INFINITY : (double)m;
  }
}

// A <- W (C / s - sigma / s I) W + Z Z^dagger, z_i = ((level - theta_i) / s)^1/2 W x_i for the
// first m = expect[k] Ritz vectors, which lifts each to the level of the next
// Ritz value (no higher, so that the diagonal stays near 1), lower 64-tiles,
// FP32, identity in the padding: the matrix whose factorisation shows that
// nothing was skipped.  m = 0: the matrix is not certified and is left out.
__global__ void __launch_bounds__(256) filt_lift_kernel(const zd* __restrict__ C, int n, int np,
                                                        const double* __restrict__ shift,
                                                        const double* __restrict__ sigma,
                                                        const double* __restrict__ level,
                                                        const double* __restrict__ theta,
                                                        const zd* __restrict__ X,
                                                        const int* __restrict__ expect,
                                                        const float* __restrict__ w,
                                                        zf* __restrict__ A, int* __restrict__ neg,
                                                        int* __restrict__ flag) {
  __shared__ __align__(16) zf Zr[FB * TB], Zc[FB * TB];   // [vector][row]
  __shared__ float q[FB];
  const int k = blockIdx.y, m = expect[k], tid = threadIdx.x;
  if (m <= 0) return;
  int bi, bk;
  tile_of(blockIdx.x, bi, bk);
  const zd* ck = C + (size_t)k * n * n;
  const zd* xk = X + (size_t)k * FB * n;
  const float* wk = w + (size_t)k * np;
  zf* ak = A + (size_t)k * np * np;
  const double is = 1.0 / shift[k], beta = sigma[k] * is;
  const int es = exponent(shift[k]);
  const float fs = (float)(is * exp2i(es));
  if (tid < FB) q[tid] = sqrtf((float)((level[k] - theta[(size_t)k * FB + tid]) * is));
  __syncthreads();
  if (blockIdx.x == 0 && tid == 0) {
    neg[k] = 0;
    flag[k] = 0;
  }
  const int m8 = (m + 7) / 8 * 8;   // at most FB
  for (int h = 0; h < 2; ++h)
    for (int e = tid; e < m8 * TB; e += 256) {
      const int t = e / TB, r = (h ? bk : bi) * TB + e % TB;
      zf z = make_float2(0.f, 0.f);
      if (t < m && r < n) {
        const zd x = xk[(size_t)t * n + r];
        const float f = wk[r] * q[t];
        z = make_float2(to_float(x.x) * f, to_float(x.y) * f);
      }
      (h ? Zc : Zr)[e] = z;
    }
  __syncthreads();
  const int tx = tid & 15, ty = tid >> 4;
  zf acc[4][4] = {};
  for (int t = 0; t < m8; t += 8) mm64<true, TB, TB, 8>(Zr + t * TB, Zc + t * TB, acc);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = bk * TB + own(ty, j);
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      const int r = bi * TB + own(tx, i);
      zf v[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        v[u] = make_float2(r + u == c ? 1.f : 0.f, 0.f);
        if (r + u < n && c < n) {
          const zd z = ck[(size_t)c * n + r + u];
          const float f = wk[r + u] * wk[c];
          if (r + u == c) v[u] = make_float2((float)(z.x * is - beta) * f, 0.f);
          else v[u] = make_float2(to_float(z.x, es) * fs * f, to_float(z.y, es) * fs * f);
          v[u] = zadd(v[u], acc[i + u][j]);
        }
      }
      *reinterpret_cast<float4*>(ak + (size_t)c * np + r) =
          make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    }
  }
}

// ---------------------------------------------------------------- Rayleigh-Ritz
// X_i = the unit vector of the i-th smallest diagonal entry (a plane wave in the
// reduced basis) and 0.1 times three others, one of each 32 that follow; CX from
// the columns of C (full Hermitian storage).  The others matter where C falls
// apart into blocks (a layered cell, a supercell, a homogeneous one): products
// with C or B keep a vector in the blocks it started in, so 32 unit vectors
// alone never reach an eigenvector of a block that has fewer of them than
// wanted eigenvalues (bilayer, n = 242, 18 branches: 22 of 30 matrices were
// reduced; with them none).  Elsewhere the rounds stay as many (90 solves of
// ordinary cells, of 4 to 720 matrices: no matrix needs a fifth round with
// 0.1, 47 with 0.3, 1 without).
__global__ void filt_start_kernel(const zd* __restrict__ C, int n, const int* __restrict__ ord,
                                  zd* __restrict__ X, zd* __restrict__ CX) {
  const int k = blockIdx.z, i = blockIdx.y, r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
  const int* ok = ord + (size_t)k * NS;
  const zd* ck = C + (size_t)k * n * n;
  zd x = zmake(r == ok[i] ? 1.0 : 0.0, 0.0), cx = ck[(size_t)ok[i] * n + r];
#pragma unroll
  for (int g = 1; g < NS / FB; ++g) {
    const int j = g * FB + ((23 * i + 5 * g) & (FB - 1));   // 23: neighbours go to distant vectors
    if (j >= n) continue;
    const double f = g & 1 ? 0.1 : -0.1;
    const zd c = ck[(size_t)ok[j] * n + r];
    if (r == ok[j]) x.x += f;
    cx = zmake(fma(f, c.x, cx.x), fma(f, c.y, cx.y));
  }
  const size_t q = ((size_t)k * FB + i) * n + r;
  X[q] = x;
  CX[q] = cx;
}

// X += E
__global__ void filt_add_kernel(zd* __restrict__ X, const zf* __restrict__ E, int n, int np,
                                const int* __restrict__ done) {
  const int k = blockIdx.z, i = blockIdx.y, r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n || done[k]) return;
  zd* x = X + ((size_t)k * FB + i) * n + r;
  const zf e = E[((size_t)k * FB + i) * np + r];
  *x = zmake(x->x + (double)e.x, x->y + (double)e.y);
}

template <typename R>
struct RrSmem {   // rows of X and C X (FP32: in units of 2^es) in the arithmetic of the step
  typename Cplx<R>::T X[GR][FB + 1], Y[GR][FB + 1];
};

template <typename R>
__device__ __forceinline__ void rr_load(RrSmem<R>& sm, const zd* X, const zd* CX, int n, int r0,
                                        int nthreads, int es) {
  typedef typename Cplx<R>::T T;
  for (int e = threadIdx.x; e < GR * FB; e += nthreads) {
    const int c = e / GR, r = e % GR;
    T x = Cplx<R>::make((R)0, (R)0), y = x;
    if (r0 + r < n) {
      const zd a = X[(size_t)c * n + r0 + r], b = CX[(size_t)c * n + r0 + r];
      if constexpr (sizeof(R) == 8) {
        x = a;
        y = b;
      } else {
        x = make_float2(to_float(a.x), to_float(a.y));
        y = make_float2(to_float(b.x, es), to_float(b.y, es));
      }
    }
    sm.X[r][c] = x;
    sm.Y[r][c] = y;
  }
}

// Partial Gram matrices over 64 rows: G = X^dagger X and H = X^dagger C X, lower
// triangle in 2 x 2 blocks, one per thread (2 x 136 of 288 threads).
constexpr int GT = 288;
template <typename R>
__global__ void __launch_bounds__(GT) filt_gram_kernel(const zd* __restrict__ X,
                                                       const zd* __restrict__ CX, int n,
                                                       const double* __restrict__ shift,
                                                       zd* __restrict__ part,
                                                       const int* __restrict__ done) {
  const int es = exponent(shift[blockIdx.y]);
  if (done[blockIdx.y]) return;
  extern __shared__ __align__(16) unsigned char dsm[];
  typedef typename Cplx<R>::T T;
  RrSmem<R>& sm = *reinterpret_cast<RrSmem<R>*>(dsm);
  const int k = blockIdx.y, ch = blockIdx.x, tid = threadIdx.x;
  const int mat = tid >= 136;
  int bi, bj;
  tile_of(mat ? min(tid - 136, 135) : tid, bi, bj);
  T acc[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[i][j] = Cplx<R>::make((R)0, (R)0);
  const int r0 = ch * GR, rows = min(GR, n - r0);
  rr_load(sm, X + (size_t)k * FB * n, CX + (size_t)k * FB * n, n, r0, GT, es);
  __syncthreads();
  if (tid >= 272) return;
#pragma unroll 4
  for (int r = 0; r < rows; ++r) {
    const T a0 = sm.X[r][2 * bi], a1 = sm.X[r][2 * bi + 1];
    const T b0 = mat ? sm.Y[r][2 * bj] : sm.X[r][2 * bj];
    const T b1 = mat ? sm.Y[r][2 * bj + 1] : sm.X[r][2 * bj + 1];
    acc[0][0] = zfmac(b0, a0, acc[0][0]);   // conj(a) b
    acc[0][1] = zfmac(b1, a0, acc[0][1]);
    acc[1][0] = zfmac(b0, a1, acc[1][0]);
    acc[1][1] = zfmac(b1, a1, acc[1][1]);
  }
  zd* p = part + (((size_t)k * gridDim.x + ch) * 2 + mat) * FB * FB;
  // H in units of 2^es (FP32: its operand is)
  const double unit = sizeof(R) == 8 && mat ? exp2i(-es) : 1.0;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
      p[(2 * bi + i) * FB + 2 * bj + j] =
          zmake((double)acc[i][j].x * unit, (double)acc[i][j].y * unit);
}

// A real number as two FP32 terms, and acc += a b with it: the product's high
// part exactly (one FMA gives its rounding), the cross terms, a two-sum.  48
// bits at 11 FP32 operations, where an FP64 FMA costs 64 times an FP32 one.
struct df {
  float h, l;
};
// the upper 24 bits of the mantissa are an FP32 number as they stand, so one
// FP64 subtraction is all that the split takes from the FP64 pipe
__device__ __forceinline__ df df_of(double x, int es = 0) {
  const double xh = __longlong_as_double(__double_as_longlong(x) & ~0x1FFFFFFFLL);
  return {to_float(xh, es), to_float(x - xh, es)};
}
__device__ __forceinline__ void df_fma(df a, df b, df& acc) {
  const float p = a.h * b.h;
  const float e = fmaf(a.h, b.h, -p);
  const float s = acc.h + p, bb = s - acc.h;
  const float t = (acc.h - (s - bb)) + (p - bb);
  acc.h = s;
  acc.l += fmaf(a.h, b.l, fmaf(a.l, b.h, e + t));
}
// a + b in two terms, exactly
__device__ __forceinline__ df df_sum(float a, float b) {
  const float s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
__device__ __forceinline__ df df_neg(df a) { return {-a.h, -a.l}; }

// operands of the rotation: FP32, or two FP32 terms (re, im) high, (re, im) low
template <typename R> struct RotSmem;
template <> struct RotSmem<float> {
  zf W[FB][FB], X[FB][GR], Y[FB][GR];
  static __device__ __forceinline__ void put(zf& o, zd v, int es = 0) {
    o = make_float2(to_float(v.x, es), to_float(v.y, es));
  }
};
template <> struct RotSmem<double> {
  float4 W[FB][FB], X[FB][GR], Y[FB][GR];
  static __device__ __forceinline__ void put(float4& o, zd v, int es = 0) {
    const df a = df_of(v.x, es), b = df_of(v.y, es);
    o = make_float4(a.h, b.h, a.l, b.l);
  }
};

// X <- X W, the split of R / s = (C X W - X W Theta) / s (zero in the padding) and
// the sums of its squares per column (one partial per warp of rows).  R =
// float: FP32 products; double: products in two FP32 terms (48 bits), which
// leave 1e-14 of C X in a residual that is compared with 1e-12 of it; the
// Ritz values themselves come from the FP64 Gram matrices.  (90 matrices of
// n = 882: 1.19 ms in FP64, 0.43 ms so.)  A thread owns a row and eight columns.
template <typename R>
__global__ void __launch_bounds__(256) filt_rotate_kernel(zd* __restrict__ X,
                                                          const zd* __restrict__ CX, int n, int np,
                                                          const zd* __restrict__ W,
                                                          const double* __restrict__ theta,
                                                          const double* __restrict__ shift,
                                                          uint16_t* __restrict__ Rs,
                                                          float* __restrict__ rpart,
                                                          const int* __restrict__ done) {
  const double sh = shift[blockIdx.y];   // (beside the load of done)
  const int es = exponent(sh);
  if (done[blockIdx.y]) return;
  constexpr bool D = sizeof(R) == 8;
  extern __shared__ __align__(16) unsigned char dsm[];
  RotSmem<R>& sm = *reinterpret_cast<RotSmem<R>*>(dsm);
  const int k = blockIdx.y, ch = blockIdx.x, tid = threadIdx.x;
  zd* xk = X + (size_t)k * FB * n;
  const zd* yk = CX + (size_t)k * FB * n;
  for (int e = tid; e < FB * FB; e += 256)   // column-major: l + c FB
    RotSmem<R>::put(sm.W[e % FB][e / FB], W[(size_t)k * FB * FB + e]);
  for (int e = tid; e < GR * FB; e += 256) {
    const int l = e / GR, r = e % GR, row = ch * GR + r;
    const bool ok = row < n;
    RotSmem<R>::put(sm.X[l][r], ok ? xk[(size_t)l * n + row] : zmake(0.0, 0.0));
    RotSmem<R>::put(sm.Y[l][r], ok ? yk[(size_t)l * n + row] : zmake(0.0, 0.0), es);
  }
  __syncthreads();
  const int r = tid & 63, c0 = (tid >> 6) * 8;
  const int row = ch * GR + r;
  const bool live = row < n;
  df xr[8], xi[8], yr[8], yi[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) xr[j] = xi[j] = yr[j] = yi[j] = {0.f, 0.f};
#pragma unroll 2
  for (int l = 0; l < FB; ++l) {
    if constexpr (D) {
      const float4 xv = sm.X[l][r], yv = sm.Y[l][r];
      const df ax = {xv.x, xv.z}, bx = {xv.y, xv.w}, ay = {yv.x, yv.z}, by = {yv.y, yv.w};
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 w4 = sm.W[l][c0 + j];
        const df wr = {w4.x, w4.z}, wi = {w4.y, w4.w};
        df_fma(ax, wr, xr[j]);
        df_fma(df_neg(bx), wi, xr[j]);
        df_fma(ax, wi, xi[j]);
        df_fma(bx, wr, xi[j]);
        df_fma(ay, wr, yr[j]);
        df_fma(df_neg(by), wi, yr[j]);
        df_fma(ay, wi, yi[j]);
        df_fma(by, wr, yi[j]);
      }
    } else {
      const zf xv = sm.X[l][r], yv = sm.Y[l][r];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const zf w = sm.W[l][c0 + j];
        xr[j].h = fmaf(xv.x, w.x, fmaf(-xv.y, w.y, xr[j].h));
        xi[j].h = fmaf(xv.x, w.y, fmaf(xv.y, w.x, xi[j].h));
        yr[j].h = fmaf(yv.x, w.x, fmaf(-yv.y, w.y, yr[j].h));
        yi[j].h = fmaf(yv.x, w.y, fmaf(yv.y, w.x, yi[j].h));
      }
    }
  }
  const double is = exp2i(es) / sh, unit = exp2i(-es);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int c = c0 + j;
    const double t = theta[(size_t)k * FB + c] * unit;
    zf rv = make_float2(0.f, 0.f);
    if (live) {
      const zd x = zmake((double)xr[j].h + (double)xr[j].l, (double)xi[j].h + (double)xi[j].l);
      const zd y = zmake((double)yr[j].h + (double)yr[j].l, (double)yi[j].h + (double)yi[j].l);
      xk[(size_t)c * n + row] = x;
      rv = make_float2((float)(fma(-t, x.x, y.x) * is), (float)(fma(-t, x.y, y.y) * is));
    }
    if (row < np)
      bs_store_block_split(Rs + ((size_t)k * 2 * FB + 2 * c) * 4 * np + row, np, rv);
    float q = rv.x * rv.x + rv.y * rv.y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    if ((tid & 31) == 0)
      rpart[(((size_t)k * gridDim.x + ch) * 2 + ((tid >> 5) & 1)) * FB + c] = q;
  }
}

// Cyclic Jacobi of a 32 x 32 Hermitian matrix with the round-robin pairing,
// 256 threads.  The off-diagonal entries and the vectors are FP32, the
// diagonal is a sum hi + lo of two FP32 numbers (48 bits): the rotations take
// differences of the diagonal and shifts t |c| of it, both exact to FP32
// relative to the off-diagonal entry c, so the error left is FP32 rounding of
// the off-diagonal part alone (1e-7 of what the block is away from diagonal
// when the step begins, squared in the Ritz values).  A full FP64 sweep is
// bound by the SM's FP64 pipe (31 rounds of 8 us); the FP64 step's kernel took
// 1120 us with FP64 sweeps alone, 560 us with one behind FP32 ones, 270 us so
// (90 matrices of n = 882).  Thread (u, v) applies both
// sides' rotations to the 2 x 2 block of the index pairs u, v (the blocks
// partition the matrix) from one copy of A to the other and rotates V's
// columns of pair v in rows u and u + 16: one barrier per round, a lane
// computes the rotation of its v and takes that of its u from the lane with
// that v.
struct JacobiSmem {
  zf A[2][FB][FB + 1], V[FB][FB + 1];
  float2 D[2][FB];   // diagonal, hi + lo
  float red[16];
};

// (hi, lo) + x, renormalised
__device__ __forceinline__ float2 dd_add(float2 a, float x) {
  const float s = a.x + x, b = s - a.x;
  const float e = (a.x - (s - b)) + (x - b) + a.y;
  const float h = s + e;
  return make_float2(h, e - (h - s));
}

__device__ __forceinline__ float frsqrt(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float frcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// rotation of the pair with off-diagonal entry c and diagonal difference
// dq - dp: cs, sn, the phase c / |c| and the shift t |c|
__device__ __forceinline__ void rotation(zf c, float diff, float skip, float& cs, float& sn, zf& ph,
                                         float& shift) {
  const float c2 = c.x * c.x + c.y * c.y;
  cs = 1.f;
  sn = shift = 0.f;
  ph = make_float2(1.f, 0.f);
  const float ica = frsqrt(c2), ca = c2 * ica;
  // t = 1 / (|zeta| + sqrt(1 + zeta^2)) is the tangent: cs^2 = (1 + |zeta| r) / 2
  // and sn = r / (2 cs) with r = 1 / sqrt(1 + zeta^2), three dependent
  // approximations instead of four
  const float zeta = 0.5f * diff * ica, az = fminf(fabsf(zeta), 1e18f);
  const float r = frsqrt(fmaf(az, az, 1.f));
  const float cs2 = fmaf(0.5f * az, r, 0.5f), ic = frsqrt(cs2);
  const float s1 = copysignf(0.5f * r * ic, zeta);
  if (c2 > skip) {
    ph = make_float2(c.x * ica, c.y * ica);
    cs = cs2 * ic;
    sn = s1;
    shift = s1 * ic * ca;
  }
}

// returns the copy of D that holds the result
__device__ __forceinline__ int jacobi32(JacobiSmem& sm, float offtol, int maxsweep) {
  const int tid = threadIdx.x, u = tid >> 4, v = tid & 15;
  int cur = 0;
  for (int sweep = 0; sweep < maxsweep; ++sweep) {
    float o = 0.f, t = 0.f;
    for (int e = tid; e < FB * FB; e += 256) {
      const int r = e >> 5, c = e & 31;
      const zf a = sm.A[cur][r][c];
      if (r != c) o += a.x * a.x + a.y * a.y;
      else t += sm.D[cur][r].x * sm.D[cur][r].x;
    }
    for (int sh = 16; sh > 0; sh >>= 1) {
      o += __shfl_xor_sync(0xffffffffu, o, sh);
      t += __shfl_xor_sync(0xffffffffu, t, sh);
    }
    if ((tid & 31) == 0) {
      sm.red[2 * (tid >> 5)] = o;
      sm.red[2 * (tid >> 5) + 1] = t;
    }
    __syncthreads();
    float so = 0.f, st = 0.f;
    for (int q = 0; q < 8; ++q) {
      so += sm.red[2 * q];
      st += sm.red[2 * q + 1];
    }
    st += so;
    if (!(so > offtol * st)) break;   // also ends on NaN
    const float skip = 0.25f * offtol * st / (FB * FB);   // below the stopping size
    for (int rd = 0; rd < FB - 1; ++rd) {
      auto pair = [&](int m, int& p, int& q) {
        p = rd + m;
        if (p >= FB - 1) p -= FB - 1;
        q = rd - m;
        if (q < 0) q += FB - 1;
        if (m == 0) q = FB - 1;
        const int lo = min(p, q);
        q = max(p, q);
        p = lo;
      };
      int pu, qu, pv, qv;
      pair(u, pu, qu);
      pair(v, pv, qv);
      const zf(*A)[FB + 1] = sm.A[cur];
      zf(*B)[FB + 1] = sm.A[cur ^ 1];
      // everything the round reads, before its stores
      const zf apq = A[pv][qv];
      const float2 dp = sm.D[cur][pv], dq = sm.D[cur][qv];
      const zf a00 = A[pu][pv], a01 = A[pu][qv], a10 = A[qu][pv], a11 = A[qu][qv];
      const zf v0p = sm.V[u][pv], v0q = sm.V[u][qv], v1p = sm.V[u + 16][pv], v1q = sm.V[u + 16][qv];
      float cv, sv, shv;
      zf fv;
      rotation(apq, (dq.x - dp.x) + (dq.y - dp.y), skip, cv, sv, fv, shv);
      // the rotation of pair u is that of the lane whose v is u
      const float cu = __shfl_sync(0xffffffffu, cv, u), su = __shfl_sync(0xffffffffu, sv, u);
      const zf fu = make_float2(__shfl_sync(0xffffffffu, fv.x, u), __shfl_sync(0xffffffffu, fv.y, u));
      fv = zconj(fv);
      // J = [[cs, sn], [-sn conj(ph), cs conj(ph)]] on columns (p, q); A <- J_u^dagger A J_v
      const zf w0 = zmul(v0q, fv), w1 = zmul(v1q, fv);
      sm.V[u][pv] = zsub(zscale(v0p, cv), zscale(w0, sv));
      sm.V[u][qv] = zadd(zscale(v0p, sv), zscale(w0, cv));
      sm.V[u + 16][pv] = zsub(zscale(v1p, cv), zscale(w1, sv));
      sm.V[u + 16][qv] = zadd(zscale(v1p, sv), zscale(w1, cv));
      if (u == v) {
        // the pair itself: the shifted diagonal and a zero (or the skipped entry)
        sm.D[cur ^ 1][pv] = dd_add(dp, -shv);
        sm.D[cur ^ 1][qv] = dd_add(dq, shv);
        const zf c = sv != 0.f ? make_float2(0.f, 0.f) : apq;
        B[pv][qv] = c;
        B[qv][pv] = zconj(c);
      } else {
        const zf c01 = zmul(a01, fv), c10 = zmul(a10, fu), c11 = zmul(zmul(a11, fv), fu);
        const zf b00 = zsub(zscale(a00, cv), zscale(c01, sv));
        const zf b01 = zadd(zscale(a00, sv), zscale(c01, cv));
        const zf b10 = zsub(zscale(c10, cv), zscale(c11, sv));
        const zf b11 = zadd(zscale(c10, sv), zscale(c11, cv));
        B[pu][pv] = zsub(zscale(b00, cu), zscale(b10, su));
        B[pu][qv] = zsub(zscale(b01, cu), zscale(b11, su));
        B[qu][pv] = zadd(zscale(b00, su), zscale(b10, cu));
        B[qu][qv] = zadd(zscale(b01, su), zscale(b11, cu));
      }
      cur ^= 1;
      __syncthreads();
    }
  }
  return cur;
}

// H w = theta G w per matrix from the Gram partials: Cholesky of the
// unit-diagonal G and its inverse factor (one barrier per column, as
// ldl64_block), A = L^-1 H L^-dagger, Jacobi, W = S L^-dagger V, all but the
// Jacobi in R (FP64 but in the steps that only steer).  In the FP64 steps a
// Newton-Schulz step makes the FP32 vectors orthonormal to 1e-12, their norms
// are divided out and W is formed in two FP32 terms: one SM's FP64 pipe, two
// multiply-adds a clock, bounds a matrix otherwise (with the products in FP64
// 210 us per step of one matrix, 155 us so).  fail: G not
// positive definite.
//
// CHECK (the steps that can certify): the Ritz values are replaced by v^dagger A v of
// the corrected vectors, and rerr gets what they may still be off by.  Jacobi's
// FP32 entries leave errors of 6e-8 of what they begin with, which in a step
// whose block was far from diagonal (an ill-conditioned Gram matrix before it)
// made Ritz values wrong by 1e4 eps64 ||C|| that no residual shows.  With
// S = V^dagger A V, a Ritz value is within sum_j min(|S_ij|, 2 |S_ij|^2 / |S_ii - S_jj|) of
// S_ii, and A itself within eps64 max C_rr / (smallest pivot of G), as C X errs by
// eps64 of C's largest entries.  The products
// take 48 bits, the off-diagonal part from U = A V - V diag(S) in FP32: 7 us.
template <typename R>
struct EigSmem {
  typename Cplx<R>::T G[FB][FB + 1], H[FB][FB + 1], Li[FB][FB + 1];
  JacobiSmem J;
};
struct EigCheckSmem : EigSmem<double> {
  float4 A[FB][FB + 1];   // two terms
};

template <typename R, bool CHECK>
__global__ void __launch_bounds__(256) filt_eig_kernel(const zd* __restrict__ part, int nch,
                                                       const double* __restrict__ shift,
                                                       const double* __restrict__ cmax,
                                                       double* __restrict__ theta,
                                                       zd* __restrict__ W,
                                                       int* __restrict__ fail,
                                                       double* __restrict__ rerr,
                                                       const int* __restrict__ done) {
  if (done[blockIdx.x]) return;
  extern __shared__ __align__(16) unsigned char dsm[];
  typedef typename Cplx<R>::T T;
  EigSmem<R>& sm = *reinterpret_cast<EigSmem<R>*>(dsm);
  __shared__ double ev[FB];
  __shared__ float re_max[FB];
  __shared__ R sc[FB], pinv[FB], sc_top;
  __shared__ int rank[FB], bad, out[FB];
  // a pivot of the unit-diagonal G below the rounding of its entries
  constexpr R kTiny = sizeof(R) == 8 ? (R)1e-13 : (R)1e-5;
  const T zero = Cplx<R>::make((R)0, (R)0);
  const int k = blockIdx.x, tid = threadIdx.x;
  if (tid == 0) bad = 0;
  constexpr int NT2 = FB * (FB + 1) / 2;   // entries of a lower triangle
  for (int e = tid; e < NT2; e += 256) {
    int r, c;
    tile_of(e, r, c);
    zd g = zmake(0.0, 0.0), h = g;
    const zd* p = part + (size_t)k * nch * 2 * FB * FB + r * FB + c;
#pragma unroll 4
    for (int q = 0; q < nch; ++q) {
      g = zadd(g, p[(size_t)q * 2 * FB * FB]);
      h = zadd(h, p[(size_t)(q * 2 + 1) * FB * FB]);
    }
    if (r == c) g.y = h.y = 0.0;
    sm.G[r][c] = Cplx<R>::make((R)g.x, (R)g.y);
    sm.H[r][c] = Cplx<R>::make((R)h.x, (R)h.y);
    if (r == c) {
      sc[r] = g.x > 0.0 ? (R)rsqrt((R)g.x) : (R)0;
      out[r] = 0;
    }
  }
  __syncthreads();
  for (int e = tid; e < NT2; e += 256) {
    int r, c;
    tile_of(e, r, c);
    const R f = sc[r] * sc[c];
    sm.G[r][c] = zscale(sm.G[r][c], f);
    const T h = zscale(sm.H[r][c], f);
    sm.H[r][c] = h;
    sm.H[c][r] = zconj(h);
  }
  for (int e = tid; e < FB * FB; e += 256)
    sm.J.V[e / FB][e % FB] = make_float2(e / FB == e % FB ? 1.f : 0.f, 0.f);
  __syncthreads();
  // unit L and pivots: G = L D L^dagger, Li = L^-1, then scaled to the Cholesky factor's
  ldl32_inverse<R, FB + 1>(&sm.G[0][0], &sm.Li[0][0], pinv, [&](R p, int c) {
    if (!(p > kTiny)) {
      bad = 1;
      out[c] = 1;
      p = (R)1;
    }
    return p;
  });
  if (tid == 0) fail[k] = bad;
  if (tid < FB) pinv[tid] = sqrt(pinv[tid]);
  __syncthreads();
  for (int e = tid; e < NT2; e += 256) {
    int r, c;
    tile_of(e, r, c);
    sm.Li[r][c] = zscale(sm.Li[r][c], pinv[r]);
  }
  __syncthreads();
  // G <- Li H, then H <- (Li H) Li^dagger (lower triangle, mirrored)
  for (int e = tid; e < FB * FB; e += 256) {
    const int r = e / FB, c = e % FB;
    T s = zero;
    for (int t = 0; t <= r; ++t) s = zfma(sm.Li[r][t], sm.H[t][c], s);
    sm.G[r][c] = s;
  }
  __syncthreads();
  for (int e = tid; e < NT2; e += 256) {
    int r, c;
    tile_of(e, r, c);
    T s = zero;
    for (int t = 0; t <= c; ++t) s = zfmac(sm.G[r][t], sm.Li[c][t], s);
    if (r == c) s.y = (R)0;
    sm.H[r][c] = s;
  }
  __syncthreads();
  if (bad && tid < 32) {
    // vectors that depend on the others: decoupled, at the top of the spectrum
    R m = out[tid] ? (R)0 : sm.H[tid][tid].x;
    for (int o = 16; o > 0; o >>= 1) {
      const R x = __shfl_xor_sync(0xffffffffu, m, o);
      m = x > m ? x : m;
    }
    if (tid == 0) sc_top = m;
  }
  __syncthreads();
  for (int e = tid; e < FB * FB; e += 256) {
    const int r = e / FB, c = e % FB;
    if (r < c) continue;
    T s = sm.H[r][c];
    if (bad && (out[r] || out[c])) s = Cplx<R>::make(r == c ? sc_top : (R)0, (R)0);
    if constexpr (CHECK) {
        float4(*A4)[FB + 1] = reinterpret_cast<EigCheckSmem&>(sm).A;
        const df x = df_of(s.x), y = df_of(s.y);
        A4[r][c] = make_float4(x.h, y.h, x.l, y.l);
        if (r != c) A4[c][r] = make_float4(x.h, -y.h, x.l, -y.l);
      }
    if (r == c) {
      const float h = (float)s.x;
      sm.J.D[0][r] = make_float2(h, (float)(s.x - (R)h));
      sm.J.A[0][r][r] = make_float2(0.f, 0.f);
      sm.J.A[1][r][r] = make_float2(0.f, 0.f);
    } else {
      sm.J.A[0][r][c] = make_float2((float)s.x, (float)s.y);
      sm.J.A[0][c][r] = make_float2((float)s.x, (float)-s.y);
    }
  }
  __syncthreads();
  // off-diagonal norm below 3e-10 of the whole (3e-7 in the steps that steer)
  const int cur = jacobi32(sm.J, sizeof(R) == 8 ? 1e-19f : 1e-13f, 10);
  if (tid < FB) ev[tid] = (double)sm.J.D[cur][tid].x + (double)sm.J.D[cur][tid].y;
  __syncthreads();
  float4(*V4)[FB + 1] = reinterpret_cast<float4(*)[FB + 1]>(&sm.G[0][0]);   // vectors, two terms
  float4(*L4)[FB + 1] = reinterpret_cast<float4(*)[FB + 1]>(&sm.H[0][0]);   // Li, two terms
  if constexpr (sizeof(R) == 8) {
    // V <- V + V F, F = (I - V^dagger V) / 2, columns to unit length.  F is 1e-6
    // and needs no more than FP32; V^dagger V is summed in two FP32 terms.  The sum is
    // split anew: a low term of 1e-6 instead of 6e-8 of the high one, whose products
    // with low terms df_fma leaves out, made Ritz values wrong by 1e-13 of
    // themselves (up to 1e3 eps64 ||C|| in one of 1000 matrices of n = 98)
    zf(*F)[FB + 1] = sm.J.A[0];
    for (int e = tid; e < NT2; e += 256) {
      int r, c;
      tile_of(e, r, c);
      df re = {0.f, 0.f}, im = {0.f, 0.f};
#pragma unroll 4
      for (int t = 0; t < FB; ++t) {   // conj(V_tr) V_tc
        const zf a = sm.J.V[t][r], b = sm.J.V[t][c];
        df_fma({a.x, 0.f}, {b.x, 0.f}, re);
        df_fma({a.y, 0.f}, {b.y, 0.f}, re);
        df_fma({a.x, 0.f}, {b.y, 0.f}, im);
        df_fma({-a.y, 0.f}, {b.x, 0.f}, im);
      }
      const zf f = make_float2(-0.5f * ((re.h - (r == c ? 1.f : 0.f)) + re.l),
                               r == c ? 0.f : -0.5f * (im.h + im.l));
      F[r][c] = f;
      F[c][r] = zconj(f);
    }
    for (int e = tid; e < FB * FB; e += 256) {
      const int r = e / FB, c = e % FB;
      zd l = r >= c ? sm.Li[r][c] : zmake(0.0, 0.0);
      const df x = df_of(l.x), y = df_of(l.y);
      L4[r][c] = make_float4(x.h, y.h, x.l, y.l);
    }
    __syncthreads();
    for (int e = tid; e < FB * FB; e += 256) {
      const int r = e / FB, c = e % FB;
      zf d = make_float2(0.f, 0.f);
#pragma unroll 8
      for (int t = 0; t < FB; ++t) d = zfma(sm.J.V[r][t], F[t][c], d);
      const zf v = sm.J.V[r][c];
      const df x = df_sum(v.x, d.x), y = df_sum(v.y, d.y);
      V4[r][c] = make_float4(x.h, y.h, x.l, y.l);
    }
    __syncthreads();
    const int c = tid >> 3, q = tid & 7;
    R v2 = (R)0;
    for (int r = q; r < FB; r += 8) {
      const float4 f = V4[r][c];
      const R x = (R)f.x + (R)f.z, y = (R)f.y + (R)f.w;
      v2 += x * x + y * y;
    }
    for (int o = 4; o > 0; o >>= 1) v2 += __shfl_xor_sync(0xffffffffu, v2, o);
    const float iv = (float)(rsqrt(v2) - 1.0);
    for (int r = q; r < FB; r += 8) {
      V4[r][c].z = fmaf(iv, V4[r][c].x, V4[r][c].z);
      V4[r][c].w = fmaf(iv, V4[r][c].y, V4[r][c].w);
    }
    __syncthreads();
    if constexpr (CHECK) {
      float4(*A4)[FB + 1] = reinterpret_cast<EigCheckSmem&>(sm).A;
      zf(*U)[FB + 1] = sm.J.A[0];
      float(*S)[FB + 1] = reinterpret_cast<float(*)[FB + 1]>(&sm.J.A[1][0][0]);
      // (A V)_rc, thread: column c = tid % 32, rows tid / 32 + 8 j
      const int col = tid & 31, row = tid >> 5;
      df re[4], im[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) re[j] = im[j] = {0.f, 0.f};
#pragma unroll 2
      for (int t = 0; t < FB; ++t) {
        const float4 v = V4[t][col];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 a = A4[row + 8 * j][t];
          df_fma({a.x, a.z}, {v.x, v.z}, re[j]);
          df_fma({a.x, a.z}, {v.y, v.w}, im[j]);
          df_fma({-a.y, -a.w}, {v.y, v.w}, re[j]);
          df_fma({a.y, a.w}, {v.x, v.z}, im[j]);
        }
      }
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 4; ++j)
        A4[row + 8 * j][col] = make_float4(re[j].h, im[j].h, re[j].l, im[j].l);
      __syncthreads();
      {   // S_cc = Re v_c^dagger (A v_c), eight lanes per column
        df d = {0.f, 0.f};
        for (int r = q; r < FB; r += 8) {
          const float4 v = V4[r][c], a = A4[r][c];
          df_fma({v.x, v.z}, {a.x, a.z}, d);
          df_fma({v.y, v.w}, {a.y, a.w}, d);
        }
        double x = (double)d.h + (double)d.l;
        for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (q == 0) ev[c] = x;
      }
      __syncthreads();
      const df sc2 = df_of(-ev[col]);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 v = V4[row + 8 * j][col];
        df_fma(sc2, {v.x, v.z}, re[j]);
        df_fma(sc2, {v.y, v.w}, im[j]);
        U[row + 8 * j][col] = make_float2(re[j].h + re[j].l, im[j].h + im[j].l);
      }
      __syncthreads();
      zf d[4] = {};
#pragma unroll 4
      for (int t = 0; t < FB; ++t) {
        const zf u = U[t][col];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 v = V4[t][row + 8 * j];
          d[j] = zfmac(u, make_float2(v.x, v.y), d[j]);
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)   // |S_rc|, r != c
        S[row + 8 * j][col] = fsqrt(fmaf(d[j].x, d[j].x, d[j].y * d[j].y));
      __syncthreads();
      {   // the bound of Ritz value c from its row of S, eight lanes per value
        float e = 0.f, ip = 0.f;
        for (int r = q; r < FB; r += 8) {
          ip = fmaxf(ip, (float)pinv[r]);
          const float a = fmaxf(S[r][c], S[c][r]), g = fabsf((float)(ev[r] - ev[c]));
          if (r != c) e += 2.f * a < g ? 2.f * a * __fdividef(a, g) : a;
        }
        for (int o = 4; o > 0; o >>= 1) {
          e += __shfl_xor_sync(0xffffffffu, e, o);
          ip = fmaxf(ip, __shfl_xor_sync(0xffffffffu, ip, o));
        }
        e += (float)DBL_EPSILON * to_float(cmax[k], exponent(shift[k])) * ip * ip;
        if (q == 0) re_max[c] = e == e ? e : INFINITY;
      }
      __syncthreads();
    }
  }
  const double unit = exp2i(exponent(shift[k]));   // of H and the Ritz values
  if (tid < FB) {
    const double x = ev[tid];
    int rk = 0;
    for (int c = 0; c < FB; ++c) rk += ev[c] < x || (ev[c] == x && c < tid);
    if (!(x == x)) rk = tid;
    rank[tid] = rk;
    if constexpr (CHECK) rerr[(size_t)k * FB + rk] = (double)re_max[tid] * unit;
  }
  __syncthreads();
  for (int e = tid; e < FB * FB; e += 256) {
    const int r = e / FB, c = e % FB;   // W[r][rank(c)] = sc_r sum_t conj(Li[t][r]) V[t][c]
    zd o;
    if constexpr (sizeof(R) == 8) {
      // 48 bits, as the rotation of the block takes them
      df re = {0.f, 0.f}, im = {0.f, 0.f};
      for (int t = r; t < FB; ++t) {
        const float4 l = L4[t][r], v = V4[t][c];
        df_fma({l.x, l.z}, {v.x, v.z}, re);
        df_fma({l.y, l.w}, {v.y, v.w}, re);
        df_fma({l.x, l.z}, {v.y, v.w}, im);
        df_fma({-l.y, -l.w}, {v.x, v.z}, im);
      }
      o = zmake(((double)re.h + (double)re.l) * sc[r], ((double)im.h + (double)im.l) * sc[r]);
    } else {
      zf x = make_float2(0.f, 0.f);
      for (int t = r; t < FB; ++t) x = zfmac(sm.J.V[t][c], sm.Li[t][r], x);
      x = zscale(x, sc[r]);
      o = zmake((double)x.x, (double)x.y);
    }
    W[(size_t)k * FB * FB + r + (size_t)rank[c] * FB] = o;
    if (r == 0) theta[(size_t)k * FB + rank[c]] = ev[c] * unit;
  }
}

// After a Rayleigh-Ritz step, one warp per matrix, lane c = column c: the
// residual norms and the coefficients of a degree-m filter.  The polynomial
// is T_j(l(mu)), l(mu) = 2 mu / mu_cut - 1 with mu_cut that of the last guard
// vector, so l >= 1 on the block.  A column stops at the last degree whose
// growth relative to it, tau_j(l_0) / tau_j(l_c) (the lowest branch grows
// most), times what the residual holds of the other branches stays below
// `allow`: 4e-6 of itself (the split operands), `couple` of the column's Ritz
// value (the rounding of the Rayleigh-Ritz step, and what its Jacobi sweeps
// left, of the largest one) and the rounding of C X.  Beyond, the column
// would turn into the lowest branches; allow is what the Gram matrix of the
// next step can separate again (3 in FP32, 100 in FP64, 1 before the last).
__global__ void __launch_bounds__(128) filt_coef_kernel(const double* __restrict__ theta,
                                                        const float* __restrict__ rpart, int nch,
                                                        const double* __restrict__ shift, int kb,
                                                        const double* __restrict__ cmax,
                                                        double couple, double allow, int m,
                                                        float* __restrict__ coef,
                                                        const int* __restrict__ done) {
  const int k = blockIdx.x * 4 + (threadIdx.x >> 5), c = threadIdx.x & 31;
  if (k >= kb || done[k]) return;
  float rn = 0.f;
  for (int q = 0; q < 2 * nch; ++q) rn += rpart[((size_t)k * 2 * nch + q) * FB + c];
  const double t = fmax(theta[(size_t)k * FB + c] / shift[k], 0.0);
  const double cut = __shfl_sync(0xffffffffu, t, 31);
  const double mu = 1.0 / (t + 1.0), imuc = cut + 1.0;
  const double l = fmax(2.0 * mu * imuc - 1.0, 1.0), f = 2.0 * mu * imuc;
  const double lim = allow / (4e-6 * (double)sqrtf(rn) + couple * (t + 0.1 * cut) +
                              4.0 * DBL_EPSILON * cmax[k] / shift[k]);
  float* cf = coef + (size_t)k * BS_FILT_MAXDEG * 4 * FB + c;
  double t0 = 1.0, t1 = l;   // tau_{j-1}, tau_j
  bool stop = __shfl_sync(0xffffffffu, t1, 0) > lim * t1;
  // step 0 (from g): E_1 = -(f / tau_1) g
  cf[0] = cf[FB] = cf[2 * FB] = 0.f;
  cf[3 * FB] = stop ? 0.f : (float)(-f / t1);
  for (int j = 1; j < m; ++j) {
    const double t2 = 2.0 * l * t1 - t0;
    const double g2 = __shfl_sync(0xffffffffu, t2, 0);
    stop = stop || g2 > lim * t2;
    const double s1 = t1 / t2, s0 = t0 / t2;
    cf += 4 * FB;
    cf[0] = stop ? 0.f : (float)(4.0 * imuc * s1);
    cf[FB] = stop ? 1.f : (float)(-2.0 * s1);
    cf[2 * FB] = stop || j == 1 ? 0.f : (float)(-s0);   // E_0 = 0
    cf[3 * FB] = stop ? 0.f : (float)(-2.0 * s1 * f);
    t0 = t1;
    t1 = t2;
  }
}

// Certificate of a Rayleigh-Ritz step, one warp per matrix: omega, and a cut
// above a Ritz value i >= nb - 1 whose error sum is small: m = i + 1 in expect
// (0: there is none) with sigma and the level for filt_lift_kernel.
//
// sigma lies halfway between theta_i and the next eigenvalue as far as the block
// knows it (theta_{i+1} less its residual norm).  If the factorisation of
// A + E, A = W (C - sigma + X T X^dagger) W / s and E its rounding errors, has
// positive pivots only, then for some x in the span of the lowest m + 1
// eigenvectors with X^dagger x = 0
//   0 < x^dagger (C - sigma) x + s ||E|| x^dagger W^-2 x
//    <= lambda_{m+1} - sigma + ||E|| kappa (lambda_{m+1} + s),
// so lambda_{m+1} > rho = (sigma - e kappa s) / (1 + e kappa) for any e >= ||E||.
// No pivot grows in a definite matrix (|L| |D| |L^dagger| has A's diagonal), so E is
// what roundings of either sign add up to: a numpy model of the kernels over 1600
// cells of n = 98 .. 882, with stiffnesses up to 1e3 and densities up to 1e2
// apart, has at most 57 u in the spectral norm, u = 2^-24, 18 u in 95 of 100, and no
// growth with n; e = (128 + 4 sqrt(n)) u is taken.  (The inertia of the indefinite
// C - sigma has no such bound: its pivots grow by 10 to 2000 there, and E with them.)
__global__ void __launch_bounds__(128) filt_cert_kernel(
    const double* __restrict__ theta, const double* __restrict__ rerr,
    const float* __restrict__ rpart, int nch, const double* __restrict__ shift,
    const double* __restrict__ cmax, const double* __restrict__ kappa, int n, int kb, int nb, const int* __restrict__ fail,
    double* __restrict__ omega, double* __restrict__ sigma, double* __restrict__ level,
    int* __restrict__ expect, int* __restrict__ skip, int* __restrict__ done) {
  const int k = blockIdx.x * 4 + (threadIdx.x >> 5), c = threadIdx.x & 31;
  if (k >= kb || done[k]) return;
  const double s = shift[k], ek = (128.0 + 4.0 * sqrt((double)n)) / 16777216.0 * kappa[k];
  float q32 = 0.f;
  for (int q = 0; q < 2 * nch; ++q) q32 += rpart[((size_t)k * 2 * nch + q) * FB + c];
  const double t = theta[(size_t)k * FB + c];
  q32 *= 1.001f;   // (residual / s)^2; 0.1 % for the FP32 sums
  const double tn = __shfl_down_sync(0xffffffffu, t, 1);
  const double rn = s * (double)sqrtf(__shfl_down_sync(0xffffffffu, q32, 1));
  // lane i: the cut above Ritz value i
  const double gap = tn - t, at = fmax(t, 1e-3 * s);
  const double sig = t + 0.5 * fmax(gap - rn, fmin(gap, 0.02 * at));
  const double rho = (sig - ek * s) / (1.0 + ek);
  // the error sum over s, in FP32 but for the differences
  const double is = 1.0 / s;
  float err = 0.f;
  for (int i = 0; i < FB; ++i) {
    const double ti = __shfl_sync(0xffffffffu, t, i);
    const float qi = __shfl_sync(0xffffffffu, q32, i);
    if (i <= c) err += __fdividef(qi, (float)((rho - ti) * is));
  }
  double re = rerr[(size_t)k * FB + c];   // the most of Ritz values 0 .. c
  for (int o = 1; o < FB; o <<= 1) {
    const double x = __shfl_up_sync(0xffffffffu, re, o);
    if (c >= o) re = fmax(re, x);
  }
  // of the cuts whose sum is small enough the one with the most room below rho
  const bool usable = c >= nb - 1 && c < FB - 1 && rho > t && err >= 0.f &&
                      (double)err * s + re <= 64.0 * DBL_EPSILON * cmax[k];
  double best = usable ? (rho - t) / at : -1.0;
  int at_i = c;
  for (int o = 16; o > 0; o >>= 1) {
    const double b2 = __shfl_xor_sync(0xffffffffu, best, o);
    const int i2 = __shfl_xor_sync(0xffffffffu, at_i, o);
    if (b2 > best || (b2 == best && i2 < at_i)) {
      best = b2;
      at_i = i2;
    }
  }
  const double sg = __shfl_sync(0xffffffffu, sig, at_i), tg = __shfl_sync(0xffffffffu, tn, at_i);
  const bool ok = best > 0.0 && !fail[k];
  if (c < nb) omega[(size_t)k * nb + c] = sqrt(fmax(t, 0.0));
  if (c == 0) {
    done[k] = ok;
    skip[k] = !ok;
    sigma[k] = sg;
    level[k] = tg;
    expect[k] = ok ? at_i + 1 : 0;
  }
}

// the matrices that did not pass (no cut, or a pivot that is not positive), in
// order; one CTA
__global__ void __launch_bounds__(1024) filt_decide_kernel(const int* __restrict__ neg,
                                                           const int* __restrict__ flag,
                                                           const int* __restrict__ expect, int kb,
                                                           int* __restrict__ stat,
                                                           int* __restrict__ list,
                                                           int* __restrict__ nlist,
                                                           int* __restrict__ nred, bool first,
                                                           int* __restrict__ reduced) {
  __shared__ int cnt[32], base;
  const int tid = threadIdx.x;
  if (tid == 0) base = 0;
  for (int k0 = 0; k0 < kb; k0 += 1024) {
    const int k = k0 + tid;
    const bool bad = k < kb && (expect[k] <= 0 || flag[k] || neg[k] > 0);
    const unsigned m = __ballot_sync(0xffffffffu, bad);
    if ((tid & 31) == 0) cnt[tid >> 5] = __popc(m);
    __syncthreads();
    int off = base;
    for (int w = 0; w < (tid >> 5); ++w) off += cnt[w];
    if (bad) list[off + __popc(m & ((1u << (tid & 31)) - 1u))] = k;
    if (k < kb) stat[k] = 0;
    if (k < kb && reduced) reduced[k] = bad;
    __syncthreads();
    if (tid == 0)
      for (int w = 0; w < 32; ++w) base += cnt[w];
    __syncthreads();
  }
  if (tid == 0) {
    *nlist = base;
    *nred = (first ? 0 : *nred) + base;
  }
}

}  // namespace

// ---------------------------------------------------------------- host side
// Largest number of branches, and the sizes, that the filtered iteration
// takes: at least 10 guard vectors beside the wanted ones, diagonals that fit
// the set-up kernel's shared memory, and an order from which its some 200
// launches take less than the reduction's n dependent steps also for a
// single matrix (ms of one solve, iteration / reduction, 1 and 64 matrices:
// n = 50 1.7 / 1.2 and 1.9 / 1.5, n = 98 1.9 / 2.4 and 2.2 / 3.6,
// n = 162 2.2 / 4.1 and 2.9 / 7.5, n = 338 2.8 / 9.2 and 5.2 / 28.5).
bool bs_filter_fits(int n, int nbands) {
  return nbands >= 1 && nbands <= BS_FILT_MAX_BANDS && n >= BS_FILT_MIN_N && n <= 2048;
}

void bs_filter_ws_free(FilterWs* w) {
  void* p[] = {w->A, w->X, w->pA, w->pB, w->pD, w->eA, w->eB, w->Xb, w->CX, w->vec, w->vs, w->d, w->part,
               w->rpart, w->theta, w->rerr, w->W, w->coef, w->shift, w->cmax, w->sigma, w->kappa, w->rsum, w->ord, w->w,
               w->iw, w->nred};
  for (void* q : p) cudaFree(q);
  *w = FilterWs();
}

// bytes of workspace per matrix (the digit planes of C and the two FP32
// factors are most of it)
static size_t filter_bytes(int n) {
  const size_t np = (n + TB - 1) / TB * TB, Kp = (2 * (size_t)n + 63) / 64 * 64;
  return 2 * np * np * sizeof(zf) + (size_t)n * 8 * Kp * 2 + 2 * FB * 8 * Kp * 2 +
         (size_t)24 * 2 * FB * n * 4 + 2 * (size_t)FB * n * sizeof(zd) +
         7 * FB * np * sizeof(zf) + np / TB * np * sizeof(float) + 65536;
}

int bs_filter_ws_alloc(FilterWs* w, int n, int kb) {
  // chunks of at most about 8 GB of workspace, and of the slab launches' grid limit
  const int cap = (int)std::max<size_t>(1, std::min<size_t>(1000, ((size_t)8 << 30) / filter_bytes(n)));
  const int want = std::min(kb, cap);
  if (w->n == n && w->want >= want) return BS_OK;
  bs_filter_ws_free(w);
  const size_t np = (n + TB - 1) / TB * TB, Kp = (2 * (size_t)n + 63) / 64 * 64;
  const size_t nch = (n + GR - 1) / GR;
  struct Item { void** p; size_t bytes; };
  auto buffers = [&](int kf) {
    const size_t k = kf;
    return std::vector<Item>{
        {(void**)&w->A, k * np * np * sizeof(zf)},
        {(void**)&w->X, k * np * np * sizeof(zf)},
        {(void**)&w->pA, k * n * 8 * Kp * 2},
        {(void**)&w->pB, k * 2 * FB * 8 * Kp * 2},
        // fewer digits can be cut into more slabs: room for either
        {(void**)&w->pD, std::max(bs_slice_planes(8, (int)Kp, n, 2 * FB, kf),
                                  std::max(bs_slice_planes(STEER_DIGITS, (int)Kp, n, 2 * FB, kf),
                                           bs_slice_planes(LAST_STEER_DIGITS, (int)Kp, n, 2 * FB, kf))) *
                             n * 2 * FB * sizeof(float)},
        {(void**)&w->eA, k * n * sizeof(int)},
        {(void**)&w->eB, k * FB * sizeof(int)},
        {(void**)&w->Xb, k * FB * n * sizeof(zd)},
        {(void**)&w->CX, k * FB * n * sizeof(zd)},
        {(void**)&w->vec, 3 * k * FB * np * sizeof(zf)},
        {(void**)&w->vs, 2 * k * 2 * FB * 4 * np * sizeof(uint16_t)},
        {(void**)&w->d, k * np * sizeof(float)},
        {(void**)&w->part, k * nch * 2 * FB * FB * sizeof(zd)},
        {(void**)&w->rpart, k * nch * 2 * FB * sizeof(float)},
        {(void**)&w->theta, k * FB * sizeof(double)},
        {(void**)&w->rerr, k * FB * sizeof(double)},
        {(void**)&w->W, k * FB * FB * sizeof(zd)},
        {(void**)&w->coef, k * BS_FILT_MAXDEG * 4 * FB * sizeof(float)},
        {(void**)&w->shift, k * sizeof(double)},
        {(void**)&w->cmax, k * sizeof(double)},
        {(void**)&w->sigma, 2 * k * sizeof(double)},
        {(void**)&w->kappa, k * sizeof(double)},
        {(void**)&w->rsum, k * (np / TB) * np * sizeof(float)},
        {(void**)&w->ord, k * NS * sizeof(int)},
        {(void**)&w->w, k * np * sizeof(float)},
        {(void**)&w->iw, (7 * k + 1) * sizeof(int)},
        {(void**)&w->nred, sizeof(int)},
    };
  };
  // with less memory free, smaller chunks; no allocation is tried in vain
  size_t room = 0, all = 0;
  if (cudaMemGetInfo(&room, &all) != cudaSuccess) {
    cudaGetLastError();
    room = 0;
  }
  int kf = want;
  for (;; kf /= 2) {
    if (kf < 1) {
      bs_set_error("out of device memory (filtered iteration, %zu bytes free)", room);
      return BS_ENOMEM;
    }
    size_t total = 0;
    for (const Item& it : buffers(kf)) total += (it.bytes + (2 << 20)) >> 21 << 21;   // 2 MB pages
    if (total <= room) break;
  }
  for (const Item& it : buffers(kf)) {
    if (cudaMalloc(it.p, it.bytes) != cudaSuccess) {
      cudaGetLastError();
      bs_filter_ws_free(w);
      bs_set_error("out of device memory (filtered iteration, %zu bytes)", it.bytes);
      return BS_ENOMEM;
    }
  }
  w->n = n;
  w->kf = kf;
  w->want = want;
  return BS_OK;
}

int bs_filter_read_counts(const FilterWs* w, int counts[2]) {
  counts[0] = w ? w->taken : 0;
  counts[1] = 0;
  if (!counts[0]) return BS_OK;
  cudaError_t e = cudaDeviceSynchronize();   // the solve may be on any stream
  if (e == cudaSuccess) e = cudaMemcpy(counts + 1, w->nred, sizeof(int), cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? BS_OK : bs_cuda_status(e, "filtered iteration counts");
}

// shared-memory opt-ins, per device
static int filter_attrs() {
  static std::atomic<bool> attr[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (attr[dev].load(std::memory_order_acquire)) return BS_OK;
  struct { const void* f; int bytes; } fs[] = {
      {(const void*)ldl64_diag_kernel, 2 * TB * LDS * (int)sizeof(zf)},
      {(const void*)ldl64_panel_kernel, 2 * TB * TB * (int)sizeof(zf)},
      {(const void*)ldl64_update_kernel, 2 * TB * LDS * (int)sizeof(zf)},
      {(const void*)trinv64_kernel, (TB * TB + TB * LDT) * (int)sizeof(zf)},
      {(const void*)filt_operator_kernel, 2 * TB * LDT * (int)sizeof(zf)},
      {(const void*)filt_gram_kernel<double>, (int)sizeof(RrSmem<double>)},
      {(const void*)filt_gram_kernel<float>, (int)sizeof(RrSmem<float>)},
      {(const void*)filt_rotate_kernel<double>, (int)sizeof(RotSmem<double>)},
      {(const void*)filt_rotate_kernel<float>, (int)sizeof(RotSmem<float>)},
      {(const void*)filt_eig_kernel<double, true>, (int)sizeof(EigCheckSmem)},
      {(const void*)filt_eig_kernel<double, false>, (int)sizeof(EigSmem<double>)},
      {(const void*)filt_eig_kernel<float, false>, (int)sizeof(EigSmem<float>)},
  };
  for (auto& f : fs) {
    const cudaError_t e =
        cudaFuncSetAttribute(f.f, cudaFuncAttributeMaxDynamicSharedMemorySize, f.bytes);
    if (e != cudaSuccess) return bs_cuda_status(e, "filtered iteration smem");
  }
  attr[dev].store(true, std::memory_order_release);
  return BS_OK;
}

// factor A (kf matrices); inverse: then the operator B, whose split replaces A
static int filter_factor(FilterWs& w, int np, int kf, bool inverse, cudaStream_t s,
                         const int* skip = nullptr) {
  const int nt = np / TB;
  int* neg = w.iw;
  int* flag = w.iw + w.kf;
  ldl64_diag_kernel<<<kf, 256, 2 * TB * LDS * sizeof(zf), s>>>(w.A, w.X, np, w.d, neg,
                                                                   flag, skip);
  BS_CHECK_LAUNCH("ldl64_diag_kernel");
  for (int j = 0; j + 1 < nt; ++j) {
    const int rem = nt - j - 1;
    ldl64_panel_kernel<<<dim3(rem, kf), 256, 2 * TB * TB * sizeof(zf), s>>>(w.A, w.X, np, j * TB,
                                                                                skip);
    BS_CHECK_LAUNCH("ldl64_panel_kernel");
    ldl64_update_kernel<<<dim3(rem * (rem + 1) / 2, kf), 256, 2 * TB * LDS * sizeof(zf), s>>>(
        w.A, w.X, np, j * TB, w.d, neg, flag, skip);
    BS_CHECK_LAUNCH("ldl64_update_kernel");
  }
  if (!inverse) return BS_OK;
  for (int d = 1; d < nt; ++d) {
    trinv64_kernel<<<dim3(nt - d, kf), 256, (TB * TB + TB * LDT) * sizeof(zf), s>>>(w.A, w.X, np, d);
    BS_CHECK_LAUNCH("trinv64_kernel");
  }
  filt_operator_kernel<<<dim3(nt * (nt + 1) / 2, kf), 256, 2 * TB * LDT * sizeof(zf), s>>>(
      w.X, w.d, np, w.w, reinterpret_cast<uint16_t*>(w.A), w.rsum);
  BS_CHECK_LAUNCH("filt_operator_kernel");
  filt_kappa_kernel<<<kf, 256, 0, s>>>(w.rsum, np, neg, flag, w.kappa);
  BS_CHECK_LAUNCH("filt_kappa_kernel");
  return BS_OK;
}

// CHECK: a step that can certify, whose Ritz values come with their error bound
template <typename R, bool CHECK>
static int filter_ritz(FilterWs& w, int n, int np, int kf, cudaStream_t s) {
  const int nch = (n + GR - 1) / GR;
  int *fail = w.iw + 4 * w.kf + 1, *done = fail + w.kf;
  filt_gram_kernel<R><<<dim3(nch, kf), GT, sizeof(RrSmem<R>), s>>>(w.Xb, w.CX, n, w.shift, w.part,
                                                                  done);
  BS_CHECK_LAUNCH("filt_gram_kernel");
  filt_eig_kernel<R, CHECK><<<kf, 256, CHECK ? sizeof(EigCheckSmem) : sizeof(EigSmem<R>), s>>>(
      w.part, nch, w.shift, w.cmax, w.theta, w.W, fail, w.rerr, done);
  BS_CHECK_LAUNCH("filt_eig_kernel");
  // the rotation covers the padded rows as well (np <= nch GR)
  filt_rotate_kernel<R><<<dim3(nch, kf), 256, sizeof(RotSmem<R>), s>>>(w.Xb, w.CX, n, np, w.W, w.theta, w.shift,
                                                       w.vs, w.rpart, done);
  BS_CHECK_LAUNCH("filt_rotate_kernel");
  return BS_OK;
}

int bs_launch_eig_filter(zd* C, int n, int kb, int nbands, FilterWs& w, const FilterFallback& fb,
                         double* omega, int* stat, int* err, int rounds, cudaStream_t s,
                         int* reduced) {
  static_assert(TB == GR, "padded rows are covered by the row chunks");
  // filter degrees of the rounds: the first Ritz values come from plane
  // waves and misplace the cut, so the first filters are short; the later ones
  // are long because a Rayleigh-Ritz step costs as much as several products.
  // Matrices certified after the fourth round skip the others.
  static const int degs[BS_FILT_ROUNDS] = {4, 6, 8, 8, 8, 8, 8, 8, 8, 8, 8, 8};
  constexpr int base = 4;
  rounds = std::max(base, std::min(rounds, BS_FILT_ROUNDS));
  if (w.n != n || w.kf < 1 || !bs_filter_fits(n, nbands)) {
    bs_set_error("filtered iteration: workspace for n = %d not set up", n);
    return BS_EINVAL;
  }
  TRY_LAUNCH(filter_attrs());
  const bool first = w.taken == 0;
  w.taken += kb;
  const int np = (n + TB - 1) / TB * TB, nt = np / TB, nch = (n + GR - 1) / GR;
  for (int k0 = 0; k0 < kb; k0 += w.kf) {
    const int kf = std::min(w.kf, kb - k0);
    zd* Ck = C + (size_t)k0 * n * n;
    int *neg = w.iw, *flag = w.iw + w.kf, *expect = w.iw + 2 * w.kf, *list = w.iw + 3 * w.kf,
        *nlist = w.iw + 4 * w.kf, *fail = nlist + 1, *done = fail + w.kf, *skip = done + w.kf;
    double *sigma = w.sigma, *level = w.sigma + w.kf;
    filt_prep_kernel<<<kf, 256, n * sizeof(double), s>>>(Ck, n, np, nbands, 0.2, w.shift, w.cmax,
                                                         w.ord, w.w, fail, done);
    BS_CHECK_LAUNCH("filt_prep_kernel");
    filt_scale_kernel<<<dim3(nt * (nt + 1) / 2, kf), 256, 0, s>>>(Ck, n, np, w.shift, w.w, w.A, neg,
                                                                  flag);
    BS_CHECK_LAUNCH("filt_scale_kernel");
    TRY_LAUNCH(filter_factor(w, np, kf, true, s));
    TRY_LAUNCH(bs_launch_band_pack_trail(Ck, n, 0, n, kf, w.pA, w.eA, s));
    const dim3 cg((n + 255) / 256, FB, kf);
    filt_start_kernel<<<cg, 256, 0, s>>>(Ck, n, w.ord, w.Xb, w.CX);
    BS_CHECK_LAUNCH("filt_start_kernel");
    const size_t vb = (size_t)w.kf * FB * np;
    zf *g = w.vec, *E[2] = {w.vec + vb, w.vec + 2 * vb};
    // the split of the residual and of even terms, and of odd terms
    uint16_t* vs[2] = {w.vs, w.vs + 8 * vb};
    const uint16_t* Bp = reinterpret_cast<const uint16_t*>(w.A);
    const int cstride = BS_FILT_MAXDEG * 4 * FB;
    for (int rd = 0; rd <= rounds; ++rd) {
      // the first three steps only steer the iteration: FP32 products of the block
      if (rd < 3) TRY_LAUNCH((filter_ritz<float, false>(w, n, np, kf, s)));
      else if (rd < base) TRY_LAUNCH((filter_ritz<double, false>(w, n, np, kf, s)));
      else TRY_LAUNCH((filter_ritz<double, true>(w, n, np, kf, s)));
      if (rd >= base) {
        filt_cert_kernel<<<(kf + 3) / 4, 128, 0, s>>>(w.theta, w.rerr, w.rpart, nch, w.shift,
                                                      w.cmax, w.kappa, n, kf, nbands, fail,
                                                      omega + (size_t)k0 * nbands, sigma, level,
                                                      expect, skip, done);
        BS_CHECK_LAUNCH("filt_cert_kernel");
      }
      if (rd == rounds) break;
      const int m = degs[rd];
      filt_coef_kernel<<<(kf + 3) / 4, 128, 0, s>>>(w.theta, w.rpart, nch, w.shift, kf, w.cmax,
                                                    rd < 3 ? 3e-7 : 1e-9,
                                                    rd < 2 ? 3.0 : rd == 2 ? 100.0 : 1.0, m, w.coef, done);
      BS_CHECK_LAUNCH("filt_coef_kernel");
      for (int j = 0; j < m; ++j)
        // j = 0: g = B R, E_1; then E_{j+1} from E_j and E_{j-1}
        TRY_LAUNCH(bs_launch_filter_product(Bp, vs[j & 1], np, kf, w.coef + (size_t)j * 4 * FB,
                                            cstride, j == 0 ? nullptr : E[(j - 1) & 1], E[j & 1], g,
                                            vs[(j + 1) & 1], done, err, s));
      filt_add_kernel<<<cg, 256, 0, s>>>(w.Xb, E[(m - 1) & 1], n, np, done);
      BS_CHECK_LAUNCH("filt_add_kernel");
      TRY_LAUNCH(bs_launch_band_av(n, w.Xb, n, (long)FB * n, FB, kf, rd < 2 ? STEER_DIGITS : rd == 2 ? LAST_STEER_DIGITS : 8,
                                   w.pA, w.pB, w.pD, w.eA,
                                   w.eB, w.CX, n, (long)FB * n, err, s, done));
    }
    filt_lift_kernel<<<dim3(nt * (nt + 1) / 2, kf), 256, 0, s>>>(
        Ck, n, np, w.shift, sigma, level, w.theta, w.Xb, expect, w.w, w.A, neg, flag);
    BS_CHECK_LAUNCH("filt_lift_kernel");
    TRY_LAUNCH(filter_factor(w, np, kf, false, s, skip));
    filt_decide_kernel<<<1, 1024, 0, s>>>(neg, flag, expect, kf, stat + k0, list, nlist, w.nred,
                                          first && k0 == 0,
                                          reduced ? reduced + k0 : nullptr);
    BS_CHECK_LAUNCH("filt_decide_kernel");
    TRY_LAUNCH(bs_launch_tridiag_list(Ck, n, fb.vec + (size_t)k0 * bs_tridiag_vec_elems(n),
                                      fb.part + (size_t)k0 * bs_tridiag_part_elems(n),
                                      fb.de + (size_t)k0 * 2 * n, fb.tau + (size_t)k0 * n,
                                      fb.beta + (size_t)k0 * n, fb.count + k0, list, nlist, s));
    TRY_LAUNCH(bs_launch_bisect_list(fb.de + (size_t)k0 * 2 * n, n, kf, nbands,
                                     omega + (size_t)k0 * nbands, stat + k0, list, nlist, s));
  }
  return BS_OK;
}

extern "C" int bs_lowest_eigenvalues(const double* C, int n, int batch, int nbands,
                                     double* omega_out, int* reduced_out, void* stream) {
  if (!C || !omega_out || batch < 1 || !bs_filter_fits(n, nbands)) {
    bs_set_error("bs_lowest_eigenvalues: need non-NULL arrays, batch >= 1, %d <= n <= 2048 and "
                 "1 <= nbands <= %d", BS_FILT_MIN_N, BS_FILT_MAX_BANDS);
    return BS_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const size_t K = batch, mat = K * n * n * sizeof(zd);
  void* p[11] = {};
  const size_t bytes[11] = {mat, K * bs_tridiag_vec_elems(n) * sizeof(zd),
                            K * bs_tridiag_part_elems(n) * sizeof(zd), K * 2 * n * sizeof(double),
                            K * n * sizeof(double), K * n * sizeof(zd), K * sizeof(unsigned),
                            K * nbands * sizeof(double), K * sizeof(int), K * sizeof(int),
                            sizeof(int)};
  FilterWs w;
  int r = BS_OK, late = 0;
  for (int i = 0; !r && i < 11; ++i)
    if (cudaMalloc(&p[i], bytes[i]) != cudaSuccess) {
      cudaGetLastError();
      bs_set_error("bs_lowest_eigenvalues: out of device memory (%zu bytes)", bytes[i]);
      r = BS_ENOMEM;
    }
  if (!r) r = bs_filter_ws_alloc(&w, n, batch);
  if (!r) {
    int* err = (int*)p[10];
    const FilterFallback fb{(zd*)p[1], (zd*)p[2], (double*)p[3], (double*)p[4], (zd*)p[5],
                            (unsigned*)p[6]};
    cudaError_t e = cudaMemcpyAsync(p[0], C, mat, cudaMemcpyDefault, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, sizeof(int), s);
    if (e == cudaSuccess)
      r = bs_launch_eig_filter((zd*)p[0], n, batch, nbands, w, fb, (double*)p[7], (int*)p[8], err,
                               BS_FILT_ROUNDS, s, (int*)p[9]);
    if (e == cudaSuccess) e = cudaMemcpyAsync(omega_out, p[7], bytes[7], cudaMemcpyDefault, s);
    if (e == cudaSuccess && reduced_out)
      e = cudaMemcpyAsync(reduced_out, p[9], bytes[9], cudaMemcpyDefault, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&late, err, sizeof(int), cudaMemcpyDeviceToHost, s);
    const cudaError_t es = cudaStreamSynchronize(s);   // the scratch is freed below
    if (!r && (e != cudaSuccess || es != cudaSuccess))
      r = bs_cuda_status(e != cudaSuccess ? e : es, "bs_lowest_eigenvalues");
    if (!r && late) {
      bs_set_error("a tensor-core pipeline wait reached its limit");
      r = BS_ECUDA;
    }
  }
  bs_filter_ws_free(&w);
  for (void* q : p) cudaFree(q);
  return r;
}
