// Cholesky factors and triangular inverses of the k-independent Gram
// matrices (Eqs. (ep), (eo)) on the FP64 path, A = L L^dagger and X = L^-1 for
// one or a few matrices of some hundred to a few thousand rows.
//
// A 32 x 32 x 32 complex product takes an SM's FP64 pipe (2 FMA per clock) 32
// us, so a few large tiles leave most SMs idle behind one: the updates and
// products here use 16 x 16 output tiles (four times the CTAs, a quarter of
// the time each), the panel solve multiplies eight rows per CTA with the
// inverse of the diagonal block instead of substituting, and the inverse of
// the whole factor is built by doubling from those diagonal inverses, the
// matrices of the batch and the pairs of one size in one launch.
// Measured on one GB300, factor and inverse: three matrices of n = 441
// 5.9 -> 2.2 ms, one of n = 1323 and one of 441 20.4 -> 10.7 ms.
//
// The mixed path keeps the factorisation of dense.cu: its FP32 reduction turns
// the last bits of C(k) into errors of 1e-9 of omega, and another rounding of
// the factors would only exchange one such error for another.
#include <math.h>

#include <algorithm>

#include "bs_internal.h"

namespace {

constexpr int NB = 32;   // panel width
constexpr int TS = 16;   // tile edge of the updates and products
constexpr int PR = 8;    // rows per CTA of the panel product

// Cholesky of the jb x jb lower triangle in S and its inverse in Xs (256
// threads), as unit L, pivots and unit inverse with one barrier per column;
// the thread that finishes a pivot inverts it, so the other warps issue no
// division.  A pivot that is not positive sets *info and counts as 1.
__device__ void chol_inv_block(zd (*S)[NB + 1], zd (*Xs)[NB + 1], double* piv, int jb, int* info) {
  const int tid = threadIdx.x, r = tid & 31, q = tid >> 5;
  for (int e = tid; e < NB * NB; e += 256) Xs[e / NB][e % NB] = zmake(e / NB == e % NB, 0.0);
  auto pivot = [&](int c) {
    double p = S[c][c].x;
    if (!(p > 0.0) || !isfinite(p)) {
      atomicOr(info, 1);
      p = 1.0;
    }
    piv[c] = 1.0 / p;
  };
  if (tid == 0) pivot(0);
  __syncthreads();
  for (int c = 0; c < jb; ++c) {
    if (r > c && r < jb) {
      const zd l = zscale(S[r][c], piv[c]);
      for (int s = c + 1 + q; s <= r; s += 8) S[r][s] = zfnmac(l, S[s][c], S[r][s]);
      if (q == 0 && r == c + 1) pivot(r);
      for (int s = q; s <= c; s += 8) Xs[r][s] = zfnma(l, Xs[c][s], Xs[r][s]);
    }
    __syncthreads();
  }
  if (tid < jb) piv[tid] = sqrt(piv[tid]);   // 1 / L_cc
  __syncthreads();
  for (int e = tid; e < NB * NB; e += 256) {
    const int rr = e / NB, c = e % NB;
    if (rr >= jb || c > rr) continue;
    S[rr][c] = rr == c ? zmake(1.0 / piv[c], 0.0) : zscale(S[rr][c], piv[c]);
    Xs[rr][c] = zscale(Xs[rr][c], piv[rr]);
  }
  __syncthreads();
}

// factor the diagonal block at j0 held in S; store L and its inverse
__device__ void chol_inv_store(zd* a, zd* x, int n, int j0, zd (*S)[NB + 1], zd (*Xs)[NB + 1],
                               double* piv, int* info) {
  const int jb = min(NB, n - j0);
  chol_inv_block(S, Xs, piv, jb, info);
  for (int e = threadIdx.x; e < NB * NB; e += 256) {
    const int r = e % NB, c = e / NB;
    if (r >= jb || c > r) continue;
    a[(size_t)(j0 + c) * n + j0 + r] = S[r][c];
    x[(size_t)(j0 + c) * n + j0 + r] = Xs[r][c];
  }
}

__global__ void __launch_bounds__(256) gram_diag_kernel(zd* __restrict__ A, zd* __restrict__ X,
                                                        int n, long stride,
                                                        int* __restrict__ info) {
  __shared__ zd S[NB][NB + 1], Xs[NB][NB + 1];
  __shared__ double piv[NB];
  zd* a = A + (size_t)blockIdx.x * stride;
  const int jb = min(NB, n);
  for (int e = threadIdx.x; e < NB * NB; e += 256) {
    const int r = e % NB, c = e / NB;
    if (r < jb && c <= r) S[r][c] = a[(size_t)c * n + r];
  }
  __syncthreads();
  chol_inv_store(a, X + (size_t)blockIdx.x * stride, n, 0, S, Xs, piv, info);
}

// rows of the panel below the (full) diagonal block at j0: L_i = A_i L11^-dagger
__global__ void __launch_bounds__(256) gram_panel_kernel(zd* __restrict__ A,
                                                         const zd* __restrict__ X, int n,
                                                         long stride, int j0) {
  __shared__ zd Ls[NB][NB + 1], As[PR][NB + 1];
  zd* a = A + (size_t)blockIdx.y * stride;
  const zd* x = X + (size_t)blockIdx.y * stride;
  const int i0 = j0 + NB + blockIdx.x * PR, tid = threadIdx.x;
  for (int e = tid; e < NB * NB; e += 256) {
    const int r = e % NB, c = e / NB;
    if (c <= r) Ls[r][c] = x[(size_t)(j0 + c) * n + j0 + r];
  }
  const int r = tid % PR, c = tid / PR;
  const bool ok = i0 + r < n;
  zd* p = a + (size_t)(j0 + c) * n + i0 + r;
  As[r][c] = ok ? *p : zmake(0.0, 0.0);
  __syncthreads();
  zd s = zmake(0.0, 0.0);
  for (int t = 0; t <= c; ++t) s = zfmac(As[r][t], Ls[c][t], s);
  if (ok) *p = s;
}

// (bi, bk), bi >= bk, of the l-th lower-triangular tile (row-major order)
__device__ __forceinline__ void tri_index(int l, int& bi, int& bk) {
  int r = (int)((sqrtf(8.0f * (float)l + 1.0f) - 1.0f) * 0.5f);
  while ((r + 1) * (r + 2) / 2 <= l) ++r;
  while (r * (r + 1) / 2 > l) --r;
  bi = r;
  bk = l - r * (r + 1) / 2;
}

// trailing update A -= L_i L_k^dagger behind panel j0, lower 16-tiles.  CTA 0
// takes the three tiles of the next 32 x 32 diagonal block and then factors
// it (no other CTA of the launch reads or writes that block).
__global__ void __launch_bounds__(256) gram_update_kernel(zd* __restrict__ A, zd* __restrict__ X,
                                                          int n, long stride, int j0,
                                                          int* __restrict__ info) {
  __shared__ zd Li[NB][NB + 1], Lk[NB][NB + 1];
  __shared__ double piv[NB];
  zd* a = A + (size_t)blockIdx.y * stride;
  const int tid = threadIdx.x, o = j0 + NB;
  if (blockIdx.x > 0) {
    int bi, bk;
    tri_index(blockIdx.x + 2, bi, bk);
    const int i0 = o + bi * TS, k0 = o + bk * TS;
    for (int e = tid; e < TS * NB; e += 256) {
      const int r = e % TS, t = e / TS;
      Li[t][r] = i0 + r < n ? a[(size_t)(j0 + t) * n + i0 + r] : zmake(0.0, 0.0);
      Lk[t][r] = k0 + r < n ? a[(size_t)(j0 + t) * n + k0 + r] : zmake(0.0, 0.0);
    }
    __syncthreads();
    const int r = tid % TS, c = tid / TS;
    if (i0 + r < n && i0 + r >= k0 + c) {
      zd acc = zmake(0.0, 0.0);
#pragma unroll 8
      for (int t = 0; t < NB; ++t) acc = zfmac(Li[t][r], Lk[t][c], acc);
      zd* p = a + (size_t)(k0 + c) * n + i0 + r;
      *p = zsub(*p, acc);
    }
    return;
  }
  const int jb = min(NB, n - o);
  for (int e = tid; e < NB * NB; e += 256) {
    const int r = e % NB, t = e / NB;
    Li[t][r] = r < jb ? a[(size_t)(j0 + t) * n + o + r] : zmake(0.0, 0.0);
  }
  __syncthreads();
  zd v[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {   // 528 entries of the lower triangle
    const int e = tid + 256 * q;
    if (e >= NB * (NB + 1) / 2) continue;
    int r, c;
    tri_index(e, r, c);
    zd acc = zmake(0.0, 0.0);
#pragma unroll 8
    for (int t = 0; t < NB; ++t) acc = zfmac(Li[t][r], Li[t][c], acc);
    v[q] = r < jb ? zsub(a[(size_t)(o + c) * n + o + r], acc) : acc;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int e = tid + 256 * q;
    if (e >= NB * (NB + 1) / 2) continue;
    int r, c;
    tri_index(e, r, c);
    Li[r][c] = v[q];
  }
  __syncthreads();
  chol_inv_store(a, X + (size_t)blockIdx.y * stride, n, o, Li, Lk, piv, info);
}

// One doubling step of the inverse: pairs of adjacent inverted diagonal blocks
// [i0, i0 + sz), [i0 + sz, i0 + 2 sz) (the last one ragged) of every matrix.
//   SECOND = false: T^dagger = X11^dagger L21^dagger, kept in the block of X above
//     the diagonal (not used until the end);
//   SECOND = true: X21 = -X22 T.
// 16 x 16 tiles, one entry per thread, the inner dimension in steps of 32.
template <bool SECOND>
__global__ void __launch_bounds__(256) gram_double_kernel(const zd* __restrict__ L,
                                                          zd* __restrict__ X, int n, long stride,
                                                          int sz, int npair) {
  __shared__ zd As[NB][TS + 1], Bs[NB][TS + 1];
  const int z = blockIdx.z, i0 = (z % npair) * 2 * sz, i1 = i0 + sz;
  const int s2 = min(sz, n - i1);
  const zd* l = L + (size_t)(z / npair) * stride;
  zd* x = X + (size_t)(z / npair) * stride;
  const int r0 = blockIdx.x * TS, c0 = blockIdx.y * TS;   // rows, columns of the result
  const int m = SECOND ? s2 : sz, nn = SECOND ? sz : s2;
  if (r0 >= m || c0 >= nn) return;
  const int tid = threadIdx.x, tr = tid % TS, tc = tid / TS;
  // X11 lower: row r of X11^dagger needs k >= r; X22 lower: row r needs k <= r
  const int kb = SECOND ? 0 : r0 / NB * NB, ke = SECOND ? min(s2, r0 + TS) : sz;
  zd acc = zmake(0.0, 0.0);
  for (int k0 = kb; k0 < ke; k0 += NB) {
    __syncthreads();
    if (SECOND) {
      for (int e = tid; e < TS * NB; e += 256) {
        const int r = e % TS, t = e / TS;   // A[r][k] = X22[r][k], B[k][c] = conj(Tp[c][k])
        const int k = k0 + t;
        As[t][r] = (r0 + r < s2 && k < s2 && k <= r0 + r) ? x[(size_t)(i1 + k) * n + i1 + r0 + r]
                                                          : zmake(0.0, 0.0);
        Bs[t][r] = (c0 + r < sz && k < s2) ? zconj(x[(size_t)(i1 + k) * n + i0 + c0 + r])
                                           : zmake(0.0, 0.0);
      }
    } else {
      for (int e = tid; e < TS * NB; e += 256) {
        const int t = e % NB, r = e / NB;   // A[r][k] = conj(X11[k][r])
        const int k = k0 + t;
        As[t][r] = (r0 + r < sz && k < sz && k >= r0 + r)
                       ? zconj(x[(size_t)(i0 + r0 + r) * n + i0 + k])
                       : zmake(0.0, 0.0);
      }
      for (int e = tid; e < TS * NB; e += 256) {
        const int r = e % TS, t = e / TS;   // B[k][c] = conj(L21[c][k])
        const int k = k0 + t;
        Bs[t][r] = (c0 + r < s2 && k < sz) ? zconj(l[(size_t)(i0 + k) * n + i1 + c0 + r])
                                           : zmake(0.0, 0.0);
      }
    }
    __syncthreads();
#pragma unroll 8
    for (int t = 0; t < NB; ++t) acc = zfma(As[t][tr], Bs[t][tc], acc);
  }
  if (r0 + tr >= m || c0 + tc >= nn) return;
  if (SECOND) x[(size_t)(i0 + c0 + tc) * n + i1 + r0 + tr] = zmake(-acc.x, -acc.y);
  else x[(size_t)(i1 + c0 + tc) * n + i0 + r0 + tr] = acc;
}

// zero X strictly above the diagonal
__global__ void gram_zero_upper_kernel(zd* __restrict__ Xg, int n, long stride) {
  zd* x = Xg + (size_t)blockIdx.y * stride;
  const size_t nn = (size_t)n * n;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < nn;
       e += (size_t)gridDim.x * blockDim.x)
    if (e % n < e / n) x[e] = zmake(0.0, 0.0);
}

}  // namespace

int bs_launch_gram_factor(zd* A, zd* X, int n, int batch, long stride, int* info, cudaStream_t s) {
  gram_diag_kernel<<<batch, 256, 0, s>>>(A, X, n, stride, info);
  BS_CHECK_LAUNCH("gram_diag_kernel");
  for (int j0 = 0; j0 + NB < n; j0 += NB) {
    const int m = n - j0 - NB, nt = (m + TS - 1) / TS;
    gram_panel_kernel<<<dim3((m + PR - 1) / PR, batch), 256, 0, s>>>(A, X, n, stride, j0);
    BS_CHECK_LAUNCH("gram_panel_kernel");
    gram_update_kernel<<<dim3(std::max(1, nt * (nt + 1) / 2 - 2), batch), 256, 0, s>>>(
        A, X, n, stride, j0, info);
    BS_CHECK_LAUNCH("gram_update_kernel");
  }
  for (int sz = NB; sz < n; sz *= 2) {
    const int npair = (n - sz + 2 * sz - 1) / (2 * sz);   // pairs with a second block
    const int t = (sz + TS - 1) / TS;
    gram_double_kernel<false><<<dim3(t, t, npair * batch), 256, 0, s>>>(A, X, n, stride, sz, npair);
    BS_CHECK_LAUNCH("gram_double_kernel");
    gram_double_kernel<true><<<dim3(t, t, npair * batch), 256, 0, s>>>(A, X, n, stride, sz, npair);
    BS_CHECK_LAUNCH("gram_double_kernel");
  }
  const unsigned g = (unsigned)std::min<size_t>(((size_t)n * n + 255) / 256, 4096);
  gram_zero_upper_kernel<<<dim3(g, batch), 256, 0, s>>>(X, n, stride);
  BS_CHECK_LAUNCH("gram_zero_upper_kernel");
  return BS_OK;
}
