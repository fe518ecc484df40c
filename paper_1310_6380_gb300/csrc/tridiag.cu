// Batched Householder reduction of Hermitian matrices to tridiagonal form
// (the first stage of the eigensolve of Eq. (eigenvalueproblem) once the
// pencil is reduced to standard form), in FP64 (the plain path) or FP32
// (the reduction of the mixed path, refined afterwards in FP64).
//
// Step j (j = 0 .. n-2) with reflector H_j = I - tau v v^dagger (tau real,
// v[j+1] = 1) needs p = tau B v on the trailing block B = A[j+1:, j+1:],
// w = p - (tau/2)(v^dagger p) v and the rank-2 update B -= v w^dagger + w v^dagger.
// One launch per step does, for every matrix of the batch, the rank-2
// update of step j-1 fused with p of step j over 64 x 64 tiles of the
// lower triangle (each element is read and written once per step), and
// the last tile of each matrix to finish (an arrival counter, no waiting)
// reduces the tile partials, forms w, applies the update to column j+1
// and builds the next reflector.  In FP64 the loop is bound by the FP64
// pipe of GB300, so it is written for FP64 issue: 16 FMAs per element and
// one shared-memory reduction of the row and column partials per tile.
#include <cooperative_groups.h>

#include <algorithm>

#include "bs_internal.h"
#include "shrink_grid.h"

namespace {

constexpr int TSMAX = 64;  // largest tile edge (the default)
constexpr int TSMIN = 32;  // smallest tile edge (sizes the partial-sum buffer)
constexpr int NT = 256;    // threads per CTA (8 warps), a 16 x 16 thread grid

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ double block_sum(double v, double* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  if (warp == 0) {
    double t = lane < NT / 32 ? sh[lane] : 0.0;
    t = warp_sum(t);
    if (lane == 0) sh[NT / 32] = t;
  }
  __syncthreads();
  return sh[NT / 32];
}

template <typename C>
__device__ __forceinline__ C ldg_cg(const C* p) { return __ldcg(p); }

// tau, 1 / (x0 - beta) and beta of the reflector of (alpha = x0, ...), aa = |x0|, nu = ||x||
__device__ __forceinline__ void reflector(zd alpha, double aa, double nu, double& tau, zd& scale,
                                          zd& beta) {
  if (nu > 0.0) {
    beta = aa > 0.0 ? zscale(alpha, -nu / aa) : zmake(-nu, 0.0);
    tau = (aa + nu) / nu;
    const zd den = zsub(alpha, beta);
    const double d2 = den.x * den.x + den.y * den.y;
    scale = zmake(den.x / d2, -den.y / d2);
  }
}

// Reflector of column c below the diagonal, x = A[c+1:n, c]: H x = beta e1
// with beta = -(x0/|x0|) ||x||, tau = (|x0| + ||x||)/||x||, v = x / (x0 - beta).
// The scalars are formed in FP64 for both precisions.  Writes v to the
// vector buffer and to A[c+2:n, c], tau_j, beta_j and |beta_j|.
template <typename R>
__device__ void householder(typename Cplx<R>::T* a, int n, int c, typename Cplx<R>::T* v,
                            double* tau_out, zd* beta_out, double* e_out, double* sh) {
  typedef typename Cplx<R>::T C;
  const int tid = threadIdx.x, r0 = c + 1;
  double s = 0.0;
  for (int r = r0 + 1 + tid; r < n; r += NT) {
    const C x = ldg_cg(a + r + (size_t)c * n);
    s = fma((double)x.x, (double)x.x, fma((double)x.y, (double)x.y, s));
  }
  s = block_sum(s, sh);
  const C al = ldg_cg(a + r0 + (size_t)c * n);
  const zd alpha = zmake(al.x, al.y);
  const double aa = hypot(alpha.x, alpha.y);
  const double nu = sqrt(fma(aa, aa, s));
  double tau = 0.0;
  zd scale = zmake(0.0, 0.0), beta = zmake(0.0, 0.0);
  reflector(alpha, aa, nu, tau, scale, beta);
  for (int r = r0 + 1 + tid; r < n; r += NT) {
    C* ap = a + r + (size_t)c * n;
    const C x = ldg_cg(ap);
    const zd y = zmul(zmake(x.x, x.y), scale);
    const C vr = Cplx<R>::make((R)y.x, (R)y.y);
    v[r] = vr;
    *ap = vr;
  }
  if (tid == 0) {
    v[r0] = Cplx<R>::make((R)1, (R)0);
    *tau_out = tau;
    *beta_out = beta;
    *e_out = nu;
  }
}

template <typename R>
__device__ void tridiag_begin(typename Cplx<R>::T* __restrict__ A, int n,
                              typename Cplx<R>::T* __restrict__ vec, double* __restrict__ de,
                              double* __restrict__ tau, zd* __restrict__ beta,
                              unsigned* __restrict__ count, int b) {
  typedef typename Cplx<R>::T C;
  __shared__ double sh[NT / 32 + 1];
  C* a = A + (size_t)b * n * n;
  C* vb = vec + (size_t)b * 3 * n;
  for (int r = threadIdx.x; r < 3 * n; r += NT) vb[r] = Cplx<R>::make((R)0, (R)0);
  __syncthreads();
  double* d = de + (size_t)b * 2 * n;
  if (threadIdx.x == 0) {
    d[0] = a[0].x;
    count[b] = 0u;
    tau[(size_t)b * n] = 0.0;
    beta[(size_t)b * n] = zmake(0.0, 0.0);
  }
  if (n > 1) householder<R>(a, n, 0, vb, tau + (size_t)b * n, beta + (size_t)b * n, d + n, sh);
}

template <typename R>
__global__ void __launch_bounds__(NT) tridiag_init_kernel(typename Cplx<R>::T* __restrict__ A,
                                                          int n,
                                                          typename Cplx<R>::T* __restrict__ vec,
                                                          double* __restrict__ de,
                                                          double* __restrict__ tau,
                                                          zd* __restrict__ beta,
                                                          unsigned* __restrict__ count) {
  tridiag_begin<R>(A, n, vec, de, tau, beta, count, blockIdx.x);
}

// (bi, bk) with bi >= bk of the l-th lower-triangular tile, row-major;
// FP32 square root (FP64 square root is a long sequence on GB300), then
// exact integer correction
__device__ __forceinline__ void tri_index(int l, int& bi, int& bk) {
  int r = (int)((sqrtf(8.0f * (float)l + 1.0f) - 1.0f) * 0.5f);
  while ((r + 1) * (r + 2) / 2 <= l) ++r;
  while (r * (r + 1) / 2 > l) --r;
  bi = r;
  bk = l - r * (r + 1) / 2;
}

// What the last CTA of a matrix does after step j - 1's tiles, r0 = j + 1 and
// n - r0 <= EPR NT rows: w from the tile partials, the update of column r0 and
// its reflector.  A chain that nothing overlaps within a matrix, so the rows stay
// in registers, the column in shared memory (col, n - r0 entries), and the
// partials of four tiles are loaded together (instead of through global memory
// at every stage: 1.2 us less per step at n = 882, mixed solve of 8 wavevectors
// 44.6 -> 43.6 ms, of 90 77.0 -> 75.3 ms).  The sums take the same terms in the
// same order as the general form in tridiag_tile, which FP64 keeps: there this
// one is slower (n = 50, 98, 242, 338 with 60, 30, 70, 30 matrices: 1.66, 3.42, 16.6
// and 20.4 ms against 1.49, 2.98, 15.2 and 18.4).
constexpr int EPR = 4;
template <typename R>
__device__ __forceinline__ void column_step(typename Cplx<R>::T* a, int n, int r0,
                                            const typename Cplx<R>::T* vcur,
                                            typename Cplx<R>::T* w, typename Cplx<R>::T* vnext,
                                            const typename Cplx<R>::T* pt, int t0, int nt,
                                            double* d, const double* tau, double* tau_out,
                                            zd* beta_out, typename Cplx<R>::T* col, double* sh) {
  typedef typename Cplx<R>::T C;
  __shared__ C first[2];
  const int tid = threadIdx.x;
  const C zero = Cplx<R>::make((R)0, (R)0);
  C p[EPR], v[EPR], x[EPR];
#pragma unroll
  for (int i = 0; i < EPR; ++i) {
    const int rr = r0 + tid + i * NT;
    p[i] = zero;
    v[i] = rr < n ? vcur[rr] : zero;
    x[i] = rr < n ? ldg_cg(a + rr + (size_t)r0 * n) : zero;
  }
  const R tj = (R)*tau;
  for (int t = t0; t < nt; t += 4) {
    C q[EPR][4];
#pragma unroll
    for (int i = 0; i < EPR; ++i)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int rr = r0 + tid + i * NT;
        q[i][u] = rr < n && t + u < nt ? ldg_cg(pt + (size_t)(t + u) * n + rr) : zero;
      }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (t + u < nt) {
#pragma unroll
        for (int i = 0; i < EPR; ++i) p[i] = zadd(p[i], q[i][u]);
      }
  }
  double kp = 0.0;
#pragma unroll
  for (int i = 0; i < EPR; ++i) {
    // (not contracted with the subtraction of K v below)
    if constexpr (sizeof(R) == 4) p[i] = make_float2(__fmul_rn(p[i].x, tj), __fmul_rn(p[i].y, tj));
    else p[i] = zmake(__dmul_rn(p[i].x, tj), __dmul_rn(p[i].y, tj));
    if (r0 + tid + i * NT < n)
      kp = fma((double)v[i].x, (double)p[i].x, fma((double)v[i].y, (double)p[i].y, kp));
  }
  const R K = (R)(0.5 * (double)tj * block_sum(kp, sh));
#pragma unroll
  for (int i = 0; i < EPR; ++i) {
    const int rr = r0 + tid + i * NT;
    p[i] = zsub(p[i], zscale(v[i], K));   // w
    if (rr < n) w[rr] = p[i];
  }
  if (tid == 0) {
    first[0] = p[0];
    first[1] = v[0];
  }
  __syncthreads();
  const C wj = first[0], vj = first[1];
#pragma unroll
  for (int i = 0; i < EPR; ++i) {
    const int rr = r0 + tid + i * NT;
    if (rr >= n) continue;
    x[i] = zfnmac(v[i], wj, x[i]);
    x[i] = zfnmac(p[i], vj, x[i]);
    if (rr == r0) x[i].y = (R)0;
    col[rr - r0] = x[i];
    if (rr <= r0 + 1) a[rr + (size_t)r0 * n] = x[i];   // the rows below become the reflector
  }
  if (tid == 0) d[r0] = (double)x[0].x;
  if (r0 + 1 >= n) return;
  __syncthreads();
  double s = 0.0;
  for (int r = 2 + tid; r < n - r0; r += NT) {
    const C y = col[r];
    s = fma((double)y.x, (double)y.x, fma((double)y.y, (double)y.y, s));
  }
  s = block_sum(s, sh);
  const zd alpha = zmake(col[1].x, col[1].y);
  const double aa = hypot(alpha.x, alpha.y);
  const double nu = sqrt(fma(aa, aa, s));
  double tn = 0.0;
  zd scale = zmake(0.0, 0.0), beta = zmake(0.0, 0.0);
  reflector(alpha, aa, nu, tn, scale, beta);
  for (int r = 2 + tid; r < n - r0; r += NT) {
    const C z = col[r];
    const zd y = zmul(zmake(z.x, z.y), scale);
    const C vr = Cplx<R>::make((R)y.x, (R)y.y);
    vnext[r0 + r] = vr;
    a[r0 + r + (size_t)r0 * n] = vr;
  }
  if (tid == 0) {
    vnext[r0 + 1] = Cplx<R>::make((R)1, (R)0);
    *tau_out = tn;
    *beta_out = beta;
    d[n + r0] = nu;
  }
}

// One tile of step j of matrix b (tile: its index among the ntl lower tiles).
template <typename R, int TS>
__device__ __forceinline__ void tridiag_tile(typename Cplx<R>::T* __restrict__ A, int n, int j,
                                             typename Cplx<R>::T* __restrict__ vec,
                                             typename Cplx<R>::T* __restrict__ part,
                                             double* __restrict__ de, double* __restrict__ tau,
                                             zd* __restrict__ beta, unsigned* __restrict__ count,
                                             int ntl, int b, int tile) {
  typedef typename Cplx<R>::T C;
  // Thread (tx, ty) owns rows R*TS + tx + 16v and columns S*TS + ty + 16u,
  // u, v < EPT: its EPT^2 elements give EPT row and EPT column partials of p,
  // reduced once per tile through shared memory.
  constexpr int EPT = TS / 16;
  __shared__ C vpS[TS], wpS[TS], vcS[TS];
  __shared__ C red[2][16][TS];
  C(*rowred)[TS] = red[0];       // [ty][row]
  C(*colred)[TS] = red[1];       // [tx][col]
  __shared__ double sh[NT / 32 + 1];
  __shared__ int is_last;

  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;
  const int nt = (n + TS - 1) / TS, t0 = (j + 1) / TS, r0 = j + 1;   // TS: template
  const C zero = Cplx<R>::make((R)0, (R)0);
  C* a = A + (size_t)b * n * n;
  C* vb = vec + (size_t)b * 3 * n;
  C* vcur = vb + (size_t)(j & 1) * n;
  C* vprev = vb + (size_t)((j + 1) & 1) * n;
  C* w = vb + 2 * (size_t)n;
  C* pt = part + (size_t)b * nt * n;

  int bi, bk;
  tri_index(tile, bi, bk);
  const int Rt = t0 + bi, St = t0 + bk;
  const int rbase = Rt * TS, sbase = St * TS;

  if (tid < TS) {
    const int s = sbase + tid;
    const bool ok = s < n && s >= r0;
    vpS[tid] = ok ? vprev[s] : zero;
    wpS[tid] = ok ? w[s] : zero;
    vcS[tid] = ok ? vcur[s] : zero;
  }
  C vpr[EPT], wpr[EPT], vcr[EPT], racc[EPT];
#pragma unroll
  for (int v = 0; v < EPT; ++v) {
    const int r = rbase + tx + 16 * v;
    const bool ok = r < n && r >= r0;
    vpr[v] = ok ? vprev[r] : zero;
    wpr[v] = ok ? w[r] : zero;
    vcr[v] = ok ? vcur[r] : zero;
    racc[v] = zero;
  }
  __syncthreads();

  // FP32: all 16 loads first (the stores below could alias them as far as
  // the compiler knows, which would serialise one load latency per element
  // in a loop that is otherwise light).  FP64: interleaved, the FP64 pipe
  // hides the latency and the registers are needed for the accumulators.
  constexpr bool kHoist = sizeof(R) == 4;
  C xs[EPT][EPT];
  if constexpr (kHoist) {
#pragma unroll
    for (int u = 0; u < EPT; ++u) {
      const int s = sbase + ty + 16 * u;
#pragma unroll
      for (int v = 0; v < EPT; ++v) {
        const int r = rbase + tx + 16 * v;
        xs[u][v] = (s >= r0 && r < n && r >= s) ? a[r + (size_t)s * n] : zero;
      }
    }
  }
#pragma unroll
  for (int u = 0; u < EPT; ++u) {
    const int sl = ty + 16 * u, s = sbase + sl;
    const C vps = vpS[sl], wps = wpS[sl], vcs = vcS[sl];
    C cacc = zero;
    const bool sok = s >= r0;
#pragma unroll
    for (int v = 0; v < EPT; ++v) {
      const int r = rbase + tx + 16 * v;
      if (sok && r < n && r >= s) {
        C x;
        if constexpr (kHoist) x = xs[u][v];
        else x = a[r + (size_t)s * n];
        x = zfnmac(vpr[v], wps, x);
        x = zfnmac(wpr[v], vps, x);
        if (r == s) x.y = (R)0;
        a[r + (size_t)s * n] = x;
        racc[v] = zfma(x, vcs, racc[v]);
        if (r != s) cacc = zfma(zconj(x), vcr[v], cacc);
      }
    }
    colred[tx][sl] = cacc;
  }
#pragma unroll
  for (int v = 0; v < EPT; ++v) rowred[ty][tx + 16 * v] = racc[v];
  __syncthreads();
  if (tid < 2 * TS) {
    const bool isrow = tid < TS;
    const int l = isrow ? tid : tid - TS;
    C acc = zero;
#pragma unroll
    for (int q = 0; q < 16; ++q) acc = zadd(acc, isrow ? rowred[q][l] : colred[q][l]);
    if (Rt == St) {
      // diagonal tile: row and column partials of the same index meet here
      if (isrow) rowred[0][l] = acc;
      else colred[0][l] = acc;
    } else if (isrow) {
      if (rbase + l < n) pt[(size_t)St * n + rbase + l] = acc;
    } else {
      pt[(size_t)Rt * n + sbase + l] = acc;
    }
  }
  if (Rt == St) {
    __syncthreads();
    if (tid < TS && rbase + tid < n)
      pt[(size_t)Rt * n + rbase + tid] = zadd(rowred[0][tid], colred[0][tid]);
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) is_last = (atomicAdd(count + b, 1u) == (unsigned)(ntl - 1));
  __syncthreads();
  if (!is_last) return;
  __threadfence();

  // ---- epilogue: one CTA per matrix
  if constexpr (sizeof(R) == 4) if (n - r0 <= EPR * NT) {
    static_assert(2 * 16 * TS >= EPR * NT, "the column fits the reduction buffers");
    column_step<R>(a, n, r0, vcur, w, vprev, pt, t0, nt, de + (size_t)b * 2 * n,
                   tau + (size_t)b * n + j, tau + (size_t)b * n + r0, beta + (size_t)b * n + r0,
                   &red[0][0][0], sh);
    if (tid == 0) count[b] = 0u;
    return;
  }
  const R tj = (R)tau[(size_t)b * n + j];
  double kp = 0.0;
  for (int rr = r0 + tid; rr < n; rr += NT) {
    C p = zero;
    for (int t = t0; t < nt; ++t) p = zadd(p, ldg_cg(pt + (size_t)t * n + rr));
    p = zscale(p, tj);
    w[rr] = p;
    const C v = vcur[rr];
    kp = fma((double)v.x, (double)p.x, fma((double)v.y, (double)p.y, kp));
  }
  const R K = (R)(0.5 * (double)tj * block_sum(kp, sh));
  for (int rr = r0 + tid; rr < n; rr += NT) {
    const C v = vcur[rr];
    w[rr] = zsub(w[rr], zscale(v, K));
  }
  __syncthreads();
  const C wj = w[r0], vj = vcur[r0];
  for (int rr = r0 + tid; rr < n; rr += NT) {
    C* ap = a + rr + (size_t)r0 * n;
    C x = ldg_cg(ap);
    x = zfnmac(vcur[rr], wj, x);
    x = zfnmac(w[rr], vj, x);
    if (rr == r0) x.y = (R)0;
    *ap = x;
  }
  __syncthreads();
  double* d = de + (size_t)b * 2 * n;
  if (tid == 0) {
    d[r0] = (double)a[r0 + (size_t)r0 * n].x;
    count[b] = 0u;
  }
  if (r0 + 1 < n)
    householder<R>(a, n, r0, vprev, tau + (size_t)b * n + r0, beta + (size_t)b * n + r0,
                   d + n + r0, sh);
}

// FP32: 3 CTAs per SM (memory latency needs warps); FP64: 2 (its pipe is the limit).
// TS = 64 (4 x 4 elements per thread) or 32 (2 x 2): the tile edge is tuned per n.
template <typename R, int TS>
__global__ void __launch_bounds__(NT, sizeof(R) == 4 ? 3 : 2)
    tridiag_step_kernel(typename Cplx<R>::T* __restrict__ A, int n, int j,
                        typename Cplx<R>::T* __restrict__ vec,
                        typename Cplx<R>::T* __restrict__ part, double* __restrict__ de,
                        double* __restrict__ tau, zd* __restrict__ beta,
                        unsigned* __restrict__ count, int ntl) {
  tridiag_tile<R, TS>(A, n, j, vec, part, de, tau, beta, count, ntl, blockIdx.y, blockIdx.x);
}

// The same reduction of the matrices list[0 .. *nlist) of a batch, in one
// cooperative launch: the tiles of a step go round the CTAs, a grid barrier
// separates the steps.  The list is made on the device (the matrices an
// iterative solve did not certify) and is nearly always empty: the launch
// then returns at once, where n step launches would cost their launch gaps.
__global__ void __launch_bounds__(NT, 2)
    tridiag_list_kernel(zd* __restrict__ A, int n, zd* __restrict__ vec, zd* __restrict__ part,
                        double* __restrict__ de, double* __restrict__ tau, zd* __restrict__ beta,
                        unsigned* __restrict__ count, const int* __restrict__ list,
                        const int* __restrict__ nlist) {
  const int nf = *nlist;
  if (nf == 0) return;   // the same for every CTA
  cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  for (int f = blockIdx.x; f < nf; f += gridDim.x) {
    tridiag_begin<double>(A, n, vec, de, tau, beta, count, list[f]);
    __syncthreads();
  }
  grid.sync();
  const int nt = (n + 63) / 64;
  for (int j = 0; j + 1 < n; ++j) {
    const int m = nt - (j + 1) / 64, ntl = m * (m + 1) / 2;
    const long items = (long)nf * ntl;
    for (long it = blockIdx.x; it < items; it += gridDim.x) {
      tridiag_tile<double, 64>(A, n, j, vec, part, de, tau, beta, count, ntl, list[it / ntl],
                               (int)(it % ntl));
      __syncthreads();
    }
    grid.sync();
  }
}

}  // namespace

int bs_launch_tridiag_list(zd* A, int n, zd* vec, zd* part, double* de, double* tau, zd* beta,
                           unsigned* count, const int* list, const int* nlist, cudaStream_t s) {
  int per = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, tridiag_list_kernel, NT, 0);
  if (e != cudaSuccess) return bs_cuda_status(e, "tridiag_list_kernel");
  const int grid = std::max(1, per) * bs_sm_count();
  void* args[] = {&A, &n, &vec, &part, &de, &tau, &beta, &count, (void*)&list, (void*)&nlist};
  // (the tiles and matrices go round whatever blocks there are)
  e = bs_shrink_grid(grid, cudaErrorCooperativeLaunchTooLarge, [&](int g) {
    const cudaError_t l =
        cudaLaunchCooperativeKernel((const void*)tridiag_list_kernel, dim3(g), dim3(NT), args, 0, s);
    if (l == cudaErrorCooperativeLaunchTooLarge) cudaGetLastError();
    return l;
  });
  if (e != cudaSuccess) return bs_cuda_status(e, "tridiag_list_kernel");
  BS_CHECK_LAUNCH("tridiag_list_kernel");
  return BS_OK;
}

size_t bs_tridiag_vec_elems(int n) { return 3 * (size_t)n; }
size_t bs_tridiag_part_elems(int n) { return (size_t)((n + TSMIN - 1) / TSMIN) * n; }

int bs_side_create(SideStreams** out) {
  if (*out) return BS_OK;
  SideStreams* w = new SideStreams();
  cudaError_t e = cudaEventCreateWithFlags(&w->fork, cudaEventDisableTiming);
  for (int h = 0; e == cudaSuccess && h < BS_SIDE; ++h) {
    e = cudaStreamCreateWithFlags(&w->s[h], cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&w->join[h], cudaEventDisableTiming);
  }
  if (e != cudaSuccess) {
    bs_side_free(w);
    return bs_cuda_status(e, "side stream");
  }
  *out = w;
  return BS_OK;
}
void bs_side_free(SideStreams* w) {
  if (!w) return;
  for (int h = 0; h < BS_SIDE; ++h) {
    if (w->s[h]) cudaStreamDestroy(w->s[h]);
    if (w->join[h]) cudaEventDestroy(w->join[h]);
  }
  if (w->fork) cudaEventDestroy(w->fork);
  delete w;
}
int bs_side_fork(const SideStreams* w, int parts, cudaStream_t s) {
  cudaError_t e = parts > 1 ? cudaEventRecord(w->fork, s) : cudaSuccess;
  for (int h = 0; e == cudaSuccess && h + 1 < parts; ++h) e = cudaStreamWaitEvent(w->s[h], w->fork, 0);
  return e == cudaSuccess ? BS_OK : bs_cuda_status(e, "side stream fork");
}
int bs_side_join(const SideStreams* w, int parts, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  for (int h = 0; e == cudaSuccess && h + 1 < parts; ++h) {
    e = cudaEventRecord(w->join[h], w->s[h]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, w->join[h], 0);
  }
  return e == cudaSuccess ? BS_OK : bs_cuda_status(e, "side stream join");
}

// With side streams the batch is cut into parts whose steps run at the same
// time: the last CTA of a matrix goes on alone (partial sums, w, the next
// reflector), and the tiles of the other part fill the SMs meanwhile (90
// matrices of n = 882, FP32: 64 -> 50 ms for the reduction; a third part gains
// 0.5 ms more at 90 and loses 2.6 ms at 16; below 16 matrices the tiles of one
// part do not fill the chip and there is nothing to overlap).  Each matrix sees
// the same operations in the same order.
template <typename R, int TS>
static int launch_steps(typename Cplx<R>::T* A, int n, int batch, typename Cplx<R>::T* vec,
                        typename Cplx<R>::T* part, double* de, double* tau, zd* beta,
                        unsigned* count, cudaStream_t s, const SideStreams* side = nullptr) {
  tridiag_init_kernel<R><<<batch, NT, 0, s>>>(A, n, vec, de, tau, beta, count);
  BS_CHECK_LAUNCH("tridiag_init_kernel");
  const int nt = (n + TS - 1) / TS;
  const int parts = side && batch >= 8 * (BS_SIDE + 1) ? BS_SIDE + 1 : 1;
  TRY_LAUNCH(bs_side_fork(side, parts, s));
  for (int j = 0; j + 1 < n; ++j) {
    const int m = nt - (j + 1) / TS;
    const int ntl = m * (m + 1) / 2;
    for (int h = 0; h < parts; ++h) {
      const size_t b0 = (size_t)batch * h / parts, b1 = (size_t)batch * (h + 1) / parts;
      tridiag_step_kernel<R, TS><<<dim3(ntl, (unsigned)(b1 - b0)), NT, 0, h ? side->s[h - 1] : s>>>(
          A + b0 * n * n, n, j, vec + b0 * 3 * n, part + b0 * nt * n, de + b0 * 2 * n, tau + b0 * n,
          beta + b0 * n, count + b0, ntl);
      BS_CHECK_LAUNCH("tridiag_step_kernel");
    }
  }
  return bs_side_join(side, parts, s);
}

// FP64, n <= 600: 64-tiles while a step has enough of them to fill the GPU,
// then 32-tiles (four times as many CTAs) for the small trailing blocks of
// the last steps.  Each step writes and reduces its own partial sums, so the
// tile edge may change from one step to the next.  Larger matrices keep
// 64-tiles throughout (their tail is a negligible share of the steps).
static int launch_steps_fp64(zd* A, int n, int batch, zd* vec, zd* part, double* de, double* tau,
                             zd* beta, unsigned* count, cudaStream_t s) {
  if (n > 600) return launch_steps<double, 64>(A, n, batch, vec, part, de, tau, beta, count, s);
  tridiag_init_kernel<double><<<batch, NT, 0, s>>>(A, n, vec, de, tau, beta, count);
  BS_CHECK_LAUNCH("tridiag_init_kernel");
  const long fill = 2L * 2 * bs_sm_count();   // two waves of the 64-tile kernel (2 CTAs per SM)
  const int nt64 = (n + 63) / 64, nt32 = (n + 31) / 32;
  for (int j = 0; j + 1 < n; ++j) {
    const int m64 = nt64 - (j + 1) / 64;
    const int ntl64 = m64 * (m64 + 1) / 2;
    if ((long)ntl64 * batch >= fill) {
      tridiag_step_kernel<double, 64><<<dim3(ntl64, batch), NT, 0, s>>>(A, n, j, vec, part, de,
                                                                         tau, beta, count, ntl64);
    } else {
      const int m32 = nt32 - (j + 1) / 32;
      const int ntl32 = m32 * (m32 + 1) / 2;
      tridiag_step_kernel<double, 32><<<dim3(ntl32, batch), NT, 0, s>>>(A, n, j, vec, part, de,
                                                                         tau, beta, count, ntl32);
    }
    BS_CHECK_LAUNCH("tridiag_step_kernel");
  }
  return BS_OK;
}

template <typename R>
int bs_launch_tridiag(typename Cplx<R>::T* A, int n, int batch, typename Cplx<R>::T* vec,
                      typename Cplx<R>::T* part, double* de, double* tau, zd* beta,
                      unsigned* count, cudaStream_t s, int tile, const SideStreams* side) {
  if (tile == 0) tile = 64;
  // The whole batch runs in every step launch.  (Reducing it in L2-sized
  // groups one after another was measured slower for FP32: the per-step
  // launch and epilogue latency then repeats once per group.)
  if (tile == 32)
    return launch_steps<R, 32>(A, n, batch, vec, part, de, tau, beta, count, s, side);
  if constexpr (sizeof(R) == 8)
    return launch_steps_fp64(A, n, batch, vec, part, de, tau, beta, count, s);
  return launch_steps<R, 64>(A, n, batch, vec, part, de, tau, beta, count, s, side);
}

template int bs_launch_tridiag<double>(zd*, int, int, zd*, zd*, double*, double*, zd*, unsigned*,
                                       cudaStream_t, int, const SideStreams*);
template int bs_launch_tridiag<float>(zf*, int, int, zf*, zf*, double*, double*, zd*, unsigned*,
                                      cudaStream_t, int, const SideStreams*);
