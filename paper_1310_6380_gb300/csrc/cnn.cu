// Learned warm start for the block LOBPCG path: a small convolutional
// network that maps a cell's material maps and a wavevector to a starting
// subspace (the low-order plane-wave displacement coefficients of nvec
// vectors), with its own forward and backward kernels and Adam, in FP32.
//
// Architecture (fixed; the parameter layout follows this list):
//   input  3 x 64 x 64: standardised log(lam + 2 mu), log mu, log rho per pixel
//   conv 3x3 (circular padding: the cell is periodic) 3 -> 16, ReLU, 2x2 mean pool -> 32x32
//   conv 16 -> 32, ReLU, pool -> 16x16;  conv 32 -> 32, ReLU, pool -> 8x8
//   conv 32 -> 32, ReLU, pool -> 4x4  => 512 features per cell
//   per (cell, k): [features | 7 wavevector features] -> dense 519 -> 512, ReLU
//                  -> dense 512 -> 512, ReLU -> dense 512 -> nvec * L * 2
//   (L = 2 (2Mp+1)^2 complex coefficients per vector, interleaved re, im).
// The convolutional trunk runs once per cell; the head once per (cell, k).
//
// Loss (basis-invariant): with U the predicted L x nvec block and V the L x nb
// low-order part of the true eigenvectors,
//   loss = (||V||^2 - tr(B^H G^-1 B)) / ||V||^2,  G = U^H U + eps I,  B = U^H V,
// the part of V outside span(U); its gradient is dloss/dU* = -(V - U F) F^H
// / ||V||^2 with F = G^-1 B (so d/dRe U = 2 Re, d/dIm U = 2 Im of that).
#include <math.h>

#include <algorithm>
#include <vector>

#include "bs_internal.h"

namespace {

constexpr int IMG = 64;
constexpr int KF = 7;          // wavevector features
constexpr int FEAT = 512;      // trunk output
constexpr int HID = 512;
constexpr float LOSS_EPS = 1e-4f;
constexpr int NCONV = 4;
const int CIN[NCONV] = {3, 16, 32, 32};
const int COUT[NCONV] = {16, 32, 32, 32};
const int SIDE[NCONV] = {64, 32, 16, 8};   // input side of conv l (output side equal, then pooled)

// ------------------------------------------------------------ convolution (3x3, circular)
// forward: out[b][o][y][x] = relu(bias[o] + sum_i,dy,dx w[o][i][dy][dx] in[b][i][y+dy-1][x+dx-1])
// and its 2 x 2 means; data gradient (the taps reversed, the channels of w exchanged):
// out[b][o][y][x] = sum_i,dy,dx w[i][o][dy][dx] in[b][i][y-dy+1][x-dx+1].
//
// A thread owns a 2 x 2 quad of pixels and CT output channels: 16 loads of the
// input and 9 CT / 4 wide broadcast loads of the weights feed 36 CT multiply-adds
// per input channel, so the FP32 pipe bounds it and not the load unit (one pixel
// and scalar weights per thread took a shared load per multiply-add: 170 -> 84 us
// for the four forward layers of 64 cells, their pooling included, 129 -> 71 us
// for the three data gradients).  Every output sums its terms in the order of
// (i, dy, dx), whatever CT is.  S is a power of two.
template <int CT, bool BWD>
__global__ void __launch_bounds__(128) conv_kernel(const float* __restrict__ in,
                                                   const float* __restrict__ w,
                                                   const float* __restrict__ bias, int ni, int no,
                                                   int S, int lgh, int nquad,
                                                   float* __restrict__ out,
                                                   float* __restrict__ pooled) {
  extern __shared__ __align__(16) float wsh[];   // ni x 9 x CT
  const int o0 = blockIdx.y * CT;
  for (int e = threadIdx.x; e < ni * 9 * CT; e += blockDim.x) {
    const int t = e % CT, d = (e / CT) % 9, i = e / (9 * CT);
    wsh[e] = BWD ? w[((size_t)i * no + o0 + t) * 9 + d] : w[((size_t)(o0 + t) * ni + i) * 9 + d];
  }
  __syncthreads();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nquad) return;
  const int h = S / 2, npix = S * S;
  const int x = 2 * (q & (h - 1)), y = 2 * ((q >> lgh) & (h - 1)), b = q >> (2 * lgh);
  float acc[4][CT];
#pragma unroll
  for (int t = 0; t < CT; ++t) {
    const float v = BWD ? 0.f : bias[o0 + t];
#pragma unroll
    for (int f = 0; f < 4; ++f) acc[f][t] = v;
  }
  const float* ic = in + (size_t)b * ni * npix;
  int ro[4], co[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    ro[r] = ((y + r - 1) & (S - 1)) * S;
    co[r] = (x + r - 1) & (S - 1);
  }
#pragma unroll 2
  for (int i = 0; i < ni; ++i, ic += npix) {
    float P[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) P[r][c] = ic[ro[r] + co[c]];
    const float* wi = wsh + i * 9 * CT;
#pragma unroll
    for (int d = 0; d < 9; ++d) {
      float wt[CT];
#pragma unroll
      for (int t = 0; t < CT; t += 2) {
        if constexpr (CT >= 4) {
          if (t % 4 == 0) {
            const float4 f = *reinterpret_cast<const float4*>(wi + d * CT + t);
            wt[t] = f.x;
            wt[t + 1] = f.y;
            wt[t + 2] = f.z;
            wt[t + 3] = f.w;
          }
        } else {
          const float2 f = *reinterpret_cast<const float2*>(wi + d * CT + t);
          wt[t] = f.x;
          wt[t + 1] = f.y;
        }
      }
      const int dy = BWD ? 2 - d / 3 : d / 3, dx = BWD ? 2 - d % 3 : d % 3;
#pragma unroll
      for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int t = 0; t < CT; ++t)
          acc[f][t] = fmaf(wt[t], P[f / 2 + dy][f % 2 + dx], acc[f][t]);
    }
  }
#pragma unroll
  for (int t = 0; t < CT; ++t) {
    float v[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) v[f] = BWD ? acc[f][t] : fmaxf(acc[f][t], 0.f);
    const size_t plane = (size_t)b * no + o0 + t;
    float* o = out + plane * npix + y * S + x;
    *reinterpret_cast<float2*>(o) = make_float2(v[0], v[1]);
    *reinterpret_cast<float2*>(o + S) = make_float2(v[2], v[3]);
    if (!BWD) pooled[plane * h * h + (q & (h * h - 1))] = 0.25f * (v[0] + v[1] + v[2] + v[3]);
  }
}

// partial weight gradients: part[split][co][ci][9] (+ bias partial at part[split][co][cin][0])
// over the samples b with b % nsplit == split.  A CTA takes one input channel
// (or the bias) and WCO output channels: the nine inputs of a pixel serve WCO
// gradients, 9 WCO multiply-adds for 9 + WCO loads (one output channel per CTA
// was bound by the load unit and index arithmetic: 470 -> 127 us for the four
// layers of 64 cells).  The 72 sums of a warp are reduced by halving, 71
// shuffles instead of 360.
constexpr int WCO = 8;
__global__ void __launch_bounds__(256) conv_bwd_weight_kernel(const float* __restrict__ g,
                                                              const float* __restrict__ in, int B,
                                                              int cin, int cout, int S, int lgpix,
                                                              int nsplit,
                                                              float* __restrict__ part) {
  const int co0 = blockIdx.x / (cin + 1) * WCO, ci = blockIdx.x % (cin + 1), split = blockIdx.y;
  const int npix = S * S, lgS = lgpix / 2;
  float acc[9 * WCO];
#pragma unroll
  for (int e = 0; e < 9 * WCO; ++e) acc[e] = 0.f;
  const int cnt = (B - split + nsplit - 1) / nsplit * npix;   // pixels of this split
  for (int e = threadIdx.x; e < cnt; e += 256) {
    const int b = split + nsplit * (e >> lgpix), p = e & (npix - 1);
    const float* gc = g + ((size_t)b * cout + co0) * npix + p;
    float gv[WCO];
#pragma unroll
    for (int t = 0; t < WCO; ++t) gv[t] = gc[(size_t)t * npix];
    if (ci == cin) {   // bias
#pragma unroll
      for (int t = 0; t < WCO; ++t) acc[9 * t] += gv[t];
      continue;
    }
    const float* ic = in + ((size_t)b * cin + ci) * npix;
    const int y = p >> lgS, x = p & (S - 1);
    float v[9], sum = 0.f;
#pragma unroll
    for (int d = 0; d < 9; ++d) {
      v[d] = ic[((y + d / 3 - 1) & (S - 1)) * S + ((x + d % 3 - 1) & (S - 1))];
      sum += v[d];
    }
    if (isfinite(sum)) {
#pragma unroll
      for (int t = 0; t < WCO; ++t)
#pragma unroll
        for (int d = 0; d < 9; ++d) acc[9 * t + d] = fmaf(gv[t], v[d], acc[9 * t + d]);
    } else {   // a gradient stopped by the ReLU adds nothing, whatever the input is
#pragma unroll
      for (int t = 0; t < WCO; ++t)
#pragma unroll
        for (int d = 0; d < 9; ++d)
          if (gv[t] != 0.f) acc[9 * t + d] = fmaf(gv[t], v[d], acc[9 * t + d]);
    }
  }
  static_assert(WCO == 8, "the reduction is written for 64 + 8 sums");
  __shared__ float red[8][9 * WCO];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < 2 * o; ++i) {   // entries i and i + 2 o of the first 64
      const float keep = up ? acc[i + 2 * o] : acc[i], send = up ? acc[i] : acc[i + 2 * o];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
    if (o >= 4) {
#pragma unroll
      for (int i = 0; i < o / 4; ++i) {   // 64 + i and 64 + i + o / 4
        const float keep = up ? acc[64 + i + o / 4] : acc[64 + i];
        const float send = up ? acc[64 + i] : acc[64 + i + o / 4];
        acc[64 + i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    } else {
      acc[64] += __shfl_xor_sync(0xffffffffu, acc[64], o);
    }
  }
  red[wid][2 * lane] = acc[0];
  red[wid][2 * lane + 1] = acc[1];
  if ((lane & 3) == 0) red[wid][64 + lane / 4] = acc[64];
  __syncthreads();
  if (threadIdx.x < 9 * WCO) {
    float sum = 0.f;
    for (int q = 0; q < 8; ++q) sum += red[q][threadIdx.x];
    const int co = co0 + threadIdx.x / 9;
    part[(((size_t)split * cout + co) * (cin + 1) + ci) * 9 + threadIdx.x % 9] = sum;
  }
}

// sum the partials over splits into gw (cout x cin x 9) and gb (cout)
__global__ void conv_wgrad_reduce_kernel(const float* __restrict__ part, int cin, int cout,
                                         int nsplit, float* __restrict__ gw,
                                         float* __restrict__ gb) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int per = (cin + 1) * 9;
  if (e >= cout * per) return;
  float s = 0.f;
  for (int q = 0; q < nsplit; ++q) s += part[(size_t)q * cout * per + e];
  const int co = e / per, ci = (e / 9) % (cin + 1), d = e % 9;
  if (ci < cin) gw[((size_t)co * cin + ci) * 9 + d] = s;
  else if (d == 0) gb[co] = s;
}

// adjoint of the 2x2 mean pooling, with the ReLU mask of the pooled layer's
// input: zero gradient where that activation is zero; one pooled entry per thread
__global__ void pool_bwd_kernel(const float* __restrict__ gout, const float* __restrict__ act,
                                int S, int lgh, size_t npool, float* __restrict__ gin) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= npool) return;
  const int h = S / 2, x = (int)e & (h - 1), y = (int)(e >> lgh) & (h - 1);
  const size_t o = (e >> (2 * lgh)) * S * S + (size_t)(2 * y) * S + 2 * x;
  const float v = 0.25f * gout[e];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const float2 a = *reinterpret_cast<const float2*>(act + o + r * S);
    *reinterpret_cast<float2*>(gin + o + r * S) =
        make_float2(a.x > 0.f ? v : 0.f, a.y > 0.f ? v : 0.f);
  }
}

// ------------------------------------------------------------ dense layers
// C[m][n] = sum_k A(m,k) B(k,n) (+ bias[n], ReLU; or 0 where mask <= 0): A(m,k) =
// TA ? A[k*lda+m] : A[m*lda+k], B(k,n) = TB ? B[n*ldb+k] : B[k*ldb+n].
//
// BT x BT tiles, 32 terms a step, the next step's loads in flight in registers
// and along the contiguous index of each operand.  The layers have few rows (one
// per wavevector), so what bounds them is latency: 64-wide tiles where they fill
// the chip, 32-wide ones elsewhere, and long sums of the backward pass also split
// over blockIdx.z (the partial blocks are added by sum_parts_kernel).  256 rows,
// 512 / 512 / 2352 columns: forward 218 -> 68 us, the two backward products
// 665 -> 122 us for the three layers.  The terms of an entry are added in
// the order of k for both tiles.
template <bool TA, bool TB, int BT>
__global__ void __launch_bounds__(BT == 64 ? 256 : 128)
sgemm_kernel(int M, int N, int K, const float* __restrict__ A, int lda,
             const float* __restrict__ Bm, int ldb, const float* __restrict__ bias, bool relu,
             const float* __restrict__ mask, float* __restrict__ C, int ldc, int kslice,
             size_t zstride) {
  constexpr int NTH = BT == 64 ? 256 : 128, BK = 32, LDT = BT + 4;
  constexpr int PER = BT * BK / NTH, RM = BT * BT / NTH / 4;   // loads and rows per thread
  __shared__ __align__(16) float As[BK][LDT];
  __shared__ __align__(16) float Bs[BK][LDT];
  const int tid = threadIdx.x, tm = tid / (BT / 4), tn = tid % (BT / 4);
  const int m0 = blockIdx.y * BT, n0 = blockIdx.x * BT;
  const int kbeg = blockIdx.z * kslice, kend = min(K, kbeg + kslice);
  float acc[RM][4] = {}, ra[PER], rb[PER];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int e = tid + i * NTH;
      const int ka = k0 + (TA ? e / BT : e % BK), m = m0 + (TA ? e % BT : e / BK);
      const int kb = k0 + (TB ? e % BK : e / BT), n = n0 + (TB ? e / BK : e % BT);
      ra[i] = m < M && ka < kend ? (TA ? A[(size_t)ka * lda + m] : A[(size_t)m * lda + ka]) : 0.f;
      rb[i] = n < N && kb < kend ? (TB ? Bm[(size_t)n * ldb + kb] : Bm[(size_t)kb * ldb + n]) : 0.f;
    }
  };
  fetch(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int e = tid + i * NTH;
      As[TA ? e / BT : e % BK][TA ? e % BT : e / BK] = ra[i];
      Bs[TB ? e % BK : e / BT][TB ? e / BK : e % BT] = rb[i];
    }
    __syncthreads();
    if (k0 + BK < kend) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[RM];
      const float4 b = *reinterpret_cast<const float4*>(&Bs[kk][tn * 4]);
#pragma unroll
      for (int i = 0; i < RM; i += 2) {
        const float2 f = *reinterpret_cast<const float2*>(&As[kk][tm * RM + i]);
        a[i] = f.x;
        a[i + 1] = f.y;
      }
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        acc[i][0] = fmaf(a[i], b.x, acc[i][0]);
        acc[i][1] = fmaf(a[i], b.y, acc[i][1]);
        acc[i][2] = fmaf(a[i], b.z, acc[i][2]);
        acc[i][3] = fmaf(a[i], b.w, acc[i][3]);
      }
    }
  }
  float* c = C + blockIdx.z * zstride;
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int m = m0 + tm * RM + i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tn * 4 + j;
      if (n >= N) continue;
      float v = acc[i][j] + (bias ? bias[n] : 0.f);
      if (relu) v = fmaxf(v, 0.f);
      if (mask && !(mask[(size_t)m * ldc + n] > 0.f)) v = 0.f;
      c[(size_t)m * ldc + n] = v;
    }
  }
}

// C[e] = sum_z part[z][e], 0 where mask <= 0
__global__ void sum_parts_kernel(const float* __restrict__ part, int nz, size_t n,
                                 const float* __restrict__ mask, float* __restrict__ C) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  float s = 0.f;
#pragma unroll 4
  for (int z = 0; z < nz; ++z) s += part[z * n + e];
  C[e] = mask && !(mask[e] > 0.f) ? 0.f : s;
}

// column sums: out[n] = sum_m A[m*ld + n]; 32 columns and 8 interleaved row
// groups per CTA (one thread per column waited for every row: 52 -> 16 us for
// the three layers of 256 rows)
__global__ void __launch_bounds__(256) colsum_kernel(const float* __restrict__ A, int M, int N,
                                                     int ld, float* __restrict__ out) {
  __shared__ float red[8][32];
  const int c = threadIdx.x & 31, r = threadIdx.x >> 5, n = blockIdx.x * 32 + c;
  float s = 0.f;
  if (n < N) {
#pragma unroll 8
    for (int m = r; m < M; m += 8) s += A[(size_t)m * ld + n];
  }
  red[r][c] = s;
  __syncthreads();
  if (r == 0 && n < N) {
    for (int q = 1; q < 8; ++q) s += red[q][c];
    out[n] = s;
  }
}

// head input: h0[s] = [feat[s / kper] | kf[s]]
__global__ void head_input_kernel(const float* __restrict__ feat, const float* __restrict__ kf,
                                  int ns, int kper, float* __restrict__ h0) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int w = FEAT + KF;
  if (e >= ns * w) return;
  const int s = e / w, j = e % w;
  h0[e] = j < FEAT ? feat[(size_t)(s / kper) * FEAT + j] : kf[(size_t)s * KF + (j - FEAT)];
}

// gfeat[c] = sum over the kper samples of cell c of gh0[s][0..FEAT)
__global__ void feat_grad_kernel(const float* __restrict__ gh0, int nc, int kper,
                                 float* __restrict__ gfeat) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nc * FEAT) return;
  const int c = e / FEAT, j = e % FEAT;
  float s = 0.f;
  for (int t = 0; t < kper; ++t) s += gh0[(size_t)(c * kper + t) * (FEAT + KF) + j];
  gfeat[e] = s;
}

// ------------------------------------------------------------ inputs
// x[c] = standardised log(lam + 2 mu), log mu, log rho of every pixel of cell c
// (phase maps P x P with P = 64, tables lam | mu | rho at table + toff[c]);
// kf[s] = (Q1, Q2, cos 2 pi Q1, sin 2 pi Q1, cos 2 pi Q2, sin 2 pi Q2, hex)
// A CTA first encodes the phases of its cell, then its quarter of the pixels reads
// them: three FP64 logarithms per pixel bound it otherwise (2 FP64 FMA per clock
// and SM; 64 cells: 58 -> 10 us).  Cells of more phases than fit take them per pixel.
constexpr int ENC_PH = 1024;
__device__ __forceinline__ float3 encode_one(const double* t, int np, int p) {
  const double lam = t[p], mu = t[np + p], rho = t[2 * np + p];
  return make_float3((float)((log(lam + 2.0 * mu) - 3.5) / 1.0), (float)((log(mu) - 2.2) / 1.2),
                     (float)((log(rho) - 1.0) / 0.6));
}
__global__ void __launch_bounds__(256) encode_kernel(const uint16_t* __restrict__ phase,
                                                     const double* __restrict__ table,
                                                     const long* __restrict__ toff,
                                                     const int* __restrict__ nph,
                                                     float* __restrict__ x) {
  __shared__ float3 enc[ENC_PH];
  constexpr int NPIX = IMG * IMG;
  const int c = blockIdx.x, np = nph[c];
  const double* t = table + toff[c];
  if (np <= ENC_PH)
    for (int p = threadIdx.x; p < np; p += 256) enc[p] = encode_one(t, np, p);
  __syncthreads();
  float* xc = x + (size_t)c * 3 * NPIX;
  for (int e = blockIdx.y * (NPIX / 4) + threadIdx.x; e < (blockIdx.y + 1) * (NPIX / 4); e += 256) {
    const int p = phase[(size_t)c * NPIX + e];
    const float3 v = np <= ENC_PH && p < np ? enc[p] : encode_one(t, np, p);
    xc[e] = v.x;
    xc[NPIX + e] = v.y;
    xc[2 * NPIX + e] = v.z;
  }
}
__global__ void kfeat_kernel(const double* __restrict__ Q, const int* __restrict__ hex, int ns,
                             int kper, float* __restrict__ kf) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= ns) return;
  const double q1 = Q[2 * s], q2 = Q[2 * s + 1];
  float* o = kf + (size_t)s * KF;
  o[0] = (float)q1;
  o[1] = (float)q2;
  o[2] = (float)cospi(2.0 * q1);
  o[3] = (float)sinpi(2.0 * q1);
  o[4] = (float)cospi(2.0 * q2);
  o[5] = (float)sinpi(2.0 * q2);
  o[6] = hex[s / kper] ? 1.f : 0.f;
}

// ------------------------------------------------------------ subspace loss
// one CTA per sample: U (L x nv, from out), V (L x nb, from tgt), loss[s], gout[s].
// Bound by its chain of dependent steps (the factorisation of G and the
// substitutions), so these run one row per lane and one column per thread and
// the sums over the whole CTA (by one thread: 94 us for 256 samples, 25 us so)
constexpr int LMAX = 2 * 49;   // Mp <= 3
constexpr int NVMAX = 16;
__global__ void __launch_bounds__(288) loss_kernel(const float* __restrict__ out,
                                                   const float* __restrict__ tgt, int L, int nv,
                                                   int nb, float scale, float* __restrict__ loss,
                                                   float* __restrict__ gout) {
  __shared__ float2 U[LMAX][NVMAX + 1], V[LMAX][NVMAX + 1], R[LMAX][NVMAX + 1];
  __shared__ float2 G[NVMAX][NVMAX + 1], Bm[NVMAX][NVMAX + 1], F[NVMAX][NVMAX + 1];
  __shared__ float vn2, sums[9][2];
  __shared__ int bad;
  const int s = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  const float* o = out + (size_t)s * nv * L * 2;
  const float* t = tgt + (size_t)s * nb * L * 2;
  for (int e = tid; e < nv * L; e += nt) {
    const int v = e / L, i = e % L;
    U[i][v] = make_float2(o[2 * e], o[2 * e + 1]);
  }
  for (int e = tid; e < nb * L; e += nt) {
    const int v = e / L, i = e % L;
    V[i][v] = make_float2(t[2 * e], t[2 * e + 1]);
  }
  if (tid == 0) bad = 0;
  __syncthreads();
  // G = U^H U + eps I, B = U^H V
  for (int e = tid; e < nv * (nv + nb); e += nt) {
    const int a = e / (nv + nb), c = e % (nv + nb);
    float2 acc = make_float2(0.f, 0.f);
    for (int i = 0; i < L; ++i) {
      const float2 u = U[i][a], w = c < nv ? U[i][c] : V[i][c - nv];
      acc.x += u.x * w.x + u.y * w.y;
      acc.y += u.x * w.y - u.y * w.x;
    }
    if (c < nv) {
      if (a == c) acc.x += LOSS_EPS;
      G[a][c] = acc;
    } else {
      Bm[a][c - nv] = acc;
    }
  }
  __syncthreads();
  // Cholesky G = C C^H (lower, in place): one row per lane, nv <= 16
  if (tid < 32) {
    const int r = tid;
    for (int c = 0; c < nv; ++c) {
      float2 v = make_float2(0.f, 0.f);
      if (r >= c && r < nv) {
        v = G[r][c];
        for (int k = 0; k < c; ++k) {   // v -= G[r][k] conj(G[c][k])
          const float2 a = G[r][k], b = G[c][k];
          v.x -= a.x * b.x + a.y * b.y;
          v.y -= a.y * b.x - a.x * b.y;
        }
      }
      float p = __shfl_sync(0xffffffffu, v.x, c);
      if (!(p > 0.f)) {
        if (r == c) bad = 1;
        p = 1.f;
      }
      const float d = sqrtf(p);
      __syncwarp();
      if (r == c) G[r][c] = make_float2(d, 0.f);
      else if (r > c && r < nv) G[r][c] = make_float2(v.x / d, v.y / d);
      __syncwarp();
    }
  }
  __syncthreads();
  // F = G^-1 B: one column per thread
  if (tid < nb) {
    const int j = tid;
    for (int r = 0; r < nv; ++r) {   // forward: C y = B
      float2 v = Bm[r][j];
      for (int k = 0; k < r; ++k) {
        const float2 a = G[r][k], y = F[k][j];
        v.x -= a.x * y.x - a.y * y.y;
        v.y -= a.x * y.y + a.y * y.x;
      }
      F[r][j] = make_float2(v.x / G[r][r].x, v.y / G[r][r].x);
    }
    for (int r = nv - 1; r >= 0; --r) {   // backward: C^H f = y
      float2 v = F[r][j];
      for (int k = r + 1; k < nv; ++k) {   // v -= conj(G[k][r]) f_k
        const float2 a = G[k][r], f = F[k][j];
        v.x -= a.x * f.x + a.y * f.y;
        v.y -= a.x * f.y - a.y * f.x;
      }
      F[r][j] = make_float2(v.x / G[r][r].x, v.y / G[r][r].x);
    }
  }
  __syncthreads();
  // R = V - U F, ||V||^2, captured part tr(B^H F)
  float sv = 0.f, sc = 0.f;
  for (int e = tid; e < L * nb; e += nt) {
    const int i = e / nb, j = e % nb;
    float2 v = V[i][j];
    sv += v.x * v.x + v.y * v.y;
    for (int a = 0; a < nv; ++a) {
      const float2 u = U[i][a], f = F[a][j];
      v.x -= u.x * f.x - u.y * f.y;
      v.y -= u.x * f.y + u.y * f.x;
    }
    R[i][j] = v;
  }
  for (int e = tid; e < nv * nb; e += nt) {
    const int a = e / nb, j = e % nb;
    sc += Bm[a][j].x * F[a][j].x + Bm[a][j].y * F[a][j].y;
  }
  for (int w = 16; w > 0; w >>= 1) {
    sv += __shfl_xor_sync(0xffffffffu, sv, w);
    sc += __shfl_xor_sync(0xffffffffu, sc, w);
  }
  if ((tid & 31) == 0) {
    sums[tid >> 5][0] = sv;
    sums[tid >> 5][1] = sc;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < nt / 32; ++w) {
      sv += sums[w][0];
      sc += sums[w][1];
    }
    vn2 = fmaxf(sv, 1e-30f);
    loss[s] = bad ? 1.f : (sv - sc) / vn2;
  }
  __syncthreads();
  // d loss / d(Re, Im) U = 2 (Re, Im) of -(R F^H) / ||V||^2, times scale
  const float f2 = bad ? 0.f : -2.f * scale / vn2;
  float* g = gout + (size_t)s * nv * L * 2;
  for (int e = tid; e < nv * L; e += nt) {
    const int a = e / L, i = e % L;
    float2 acc = make_float2(0.f, 0.f);
    for (int j = 0; j < nb; ++j) {   // R[i][j] conj(F[a][j])
      const float2 r = R[i][j], f = F[a][j];
      acc.x += r.x * f.x + r.y * f.y;
      acc.y += r.y * f.x - r.x * f.y;
    }
    g[2 * e] = f2 * acc.x;
    g[2 * e + 1] = f2 * acc.y;
  }
}

// ------------------------------------------------------------ Adam
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, size_t n, float lr, float b1, float b2,
                            float c1, float c2, float eps) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace

// ------------------------------------------------------------------ the network object
struct bs_cnn {
  int nvec, Mp, L, OUT;
  int cmax, smax;          // capacity: cells and samples per call
  size_t nparam;
  size_t off_w[NCONV], off_b[NCONV], off_dw[3], off_db[3];
  float* d_p;              // parameters
  float* d_g;              // gradients
  float* d_m;              // Adam moments
  float* d_v;
  long step;
  // activations (capacity cmax cells, smax samples)
  float* x;                // cmax x 3 x 64 x 64
  float* z[NCONV];         // conv outputs (post-ReLU), before pooling
  float* pl[NCONV];        // pooled outputs (pl[3] = features)
  float* kf;               // smax x KF
  float* h0;               // smax x (FEAT + KF)
  float* h1;
  float* h2;
  float* out;              // smax x OUT
  // backward scratch
  float* gout;
  float* gh0;
  float* gh1;
  float* gh2;
  float* gpl;              // max pooled plane gradients
  float* gz;               // max conv-output gradients
  float* gtmp;             // partial sums of the dense layers' products
  size_t tmp_cap;
  float* wpart;            // conv weight-gradient partials
  float* loss;             // smax
  // encode inputs
  uint16_t* phase;
  double* table;
  long* toff;
  int* nph;
  int* hex;
  double* Q;
  float* tgt;
  size_t table_cap;
};

namespace {

constexpr int WSPLIT = 32;

template <typename T>
int calloc_dev(T** p, size_t n, const char* what) {
  *p = nullptr;
  if (!n) return BS_OK;
  cudaError_t e = cudaMalloc((void**)p, n * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    bs_set_error("cudaMalloc(%s) failed: %s", what, cudaGetErrorString(e));
    return BS_ENOMEM;
  }
  return BS_OK;
}

#define TRYC(x)            \
  do {                     \
    int r__ = (x);         \
    if (r__) return r__;   \
  } while (0)

int log2i(int v) {
  int l = 0;
  while ((1 << (l + 1)) <= v) ++l;
  return l;
}

// output channels per thread: as many as leave a full wave of threads (256 per
// SM of 152); the layers of 8 x 8 and 16 x 16 pixels have too few quads for eight
template <bool BWD>
int conv(const float* in, const float* w, const float* bias, int ni, int no, int S, int nc,
         float* out, float* pooled, cudaStream_t s) {
  const int nquad = nc * (S / 2) * (S / 2), lgh = log2i(S / 2), bx = (nquad + 127) / 128;
  const long full = 152 * 256;
  if ((long)nquad * (no / 8) >= full)
    conv_kernel<8, BWD><<<dim3(bx, no / 8), 128, ni * 9 * 8 * sizeof(float), s>>>(
        in, w, bias, ni, no, S, lgh, nquad, out, pooled);
  else if ((long)nquad * (no / 4) >= full)
    conv_kernel<4, BWD><<<dim3(bx, no / 4), 128, ni * 9 * 4 * sizeof(float), s>>>(
        in, w, bias, ni, no, S, lgh, nquad, out, pooled);
  else
    conv_kernel<2, BWD><<<dim3(bx, no / 2), 128, ni * 9 * 2 * sizeof(float), s>>>(
        in, w, bias, ni, no, S, lgh, nquad, out, pooled);
  BS_CHECK_LAUNCH("conv_kernel");
  return BS_OK;
}

int conv_forward(bs_cnn* m, int nc, cudaStream_t s) {
  const float* in = m->x;
  for (int l = 0; l < NCONV; ++l) {
    TRYC(conv<false>(in, m->d_p + m->off_w[l], m->d_p + m->off_b[l], CIN[l], COUT[l], SIDE[l], nc,
                     m->z[l], m->pl[l], s));
    in = m->pl[l];
  }
  return BS_OK;
}

template <int BT>
void sgemm_launch(bool ta, bool tb, int nz, int ks, int M, int N, int K, const float* A, int lda,
                  const float* B, int ldb, const float* bias, bool relu, const float* mask,
                  float* C, int ldc, cudaStream_t s) {
  const dim3 grid((N + BT - 1) / BT, (M + BT - 1) / BT, nz);
  const int nt = BT == 64 ? 256 : 128;
  const size_t zs = (size_t)M * N;
  auto k = ta ? sgemm_kernel<true, false, BT>
              : tb ? sgemm_kernel<false, true, BT> : sgemm_kernel<false, false, BT>;
  k<<<grid, nt, 0, s>>>(M, N, K, A, lda, B, ldb, bias, relu, mask, C, ldc, ks, zs);
}

// Not both transposed.  part: scratch of `cap` floats that lets a long sum be split
// (C dense, no bias or ReLU)
int sgemm(bool ta, bool tb, int M, int N, int K, const float* A, int lda, const float* B, int ldb,
          const float* bias, bool relu, const float* mask, float* C, int ldc, cudaStream_t s,
          float* part = nullptr, size_t cap = 0) {
  const long t64 = (long)((N + 63) / 64) * ((M + 63) / 64);
  const long t32 = (long)((N + 31) / 32) * ((M + 31) / 32);
  if (t64 >= 192) {   // 64-wide tiles fill the chip
    sgemm_launch<64>(ta, tb, 1, K, M, N, K, A, lda, B, ldb, bias, relu, mask, C, ldc, s);
  } else {
    // slices of at least 128 terms, until four CTAs per SM (of 128 threads) are busy
    const size_t room = part ? cap / ((size_t)M * N) : 0;
    int nz = (int)std::min<long>({(608 + t32 - 1) / t32, (long)K / 128, (long)std::min<size_t>(room, 64)});
    if (nz > 1) {
      const int ks = ((K + nz - 1) / nz + 31) / 32 * 32;
      nz = (K + ks - 1) / ks;
      sgemm_launch<32>(ta, tb, nz, ks, M, N, K, A, lda, B, ldb, nullptr, false, nullptr, part, N, s);
      BS_CHECK_LAUNCH("sgemm_kernel");
      const size_t n = (size_t)M * N;
      sum_parts_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(part, nz, n, mask, C);
    } else {
      sgemm_launch<32>(ta, tb, 1, K, M, N, K, A, lda, B, ldb, bias, relu, mask, C, ldc, s);
    }
  }
  BS_CHECK_LAUNCH("sgemm_kernel");
  return BS_OK;
}

int head_forward(bs_cnn* m, int nc, int kper, cudaStream_t s) {
  const int ns = nc * kper, W0 = FEAT + KF;
  head_input_kernel<<<(ns * W0 + 255) / 256, 256, 0, s>>>(m->pl[NCONV - 1], m->kf, ns, kper, m->h0);
  BS_CHECK_LAUNCH("head_input_kernel");
  TRYC(sgemm(false, true, ns, HID, W0, m->h0, W0, m->d_p + m->off_dw[0], W0, m->d_p + m->off_db[0],
             true, nullptr, m->h1, HID, s));
  TRYC(sgemm(false, true, ns, HID, HID, m->h1, HID, m->d_p + m->off_dw[1], HID,
             m->d_p + m->off_db[1], true, nullptr, m->h2, HID, s));
  TRYC(sgemm(false, true, ns, m->OUT, HID, m->h2, HID, m->d_p + m->off_dw[2], HID,
             m->d_p + m->off_db[2], false, nullptr, m->out, m->OUT, s));
  return BS_OK;
}

int colsum(const float* A, int M, int N, float* out, cudaStream_t s) {
  colsum_kernel<<<(N + 31) / 32, 256, 0, s>>>(A, M, N, N, out);
  BS_CHECK_LAUNCH("colsum_kernel");
  return BS_OK;
}

// gradients of everything from m->gout (ns x OUT) into m->d_g
int backward(bs_cnn* m, int nc, int kper, cudaStream_t s) {
  const int ns = nc * kper, W0 = FEAT + KF, OUT = m->OUT;
  float* dg = m->d_g;
  const float* p = m->d_p;
  float* pt = m->gtmp;   // partial sums
  const size_t pc = m->tmp_cap;
  // dense 3, 2, 1 (the ReLU mask of a layer's input goes with its gradient)
  TRYC(sgemm(true, false, OUT, HID, ns, m->gout, OUT, m->h2, HID, nullptr, false, nullptr,
             dg + m->off_dw[2], HID, s, pt, pc));
  TRYC(colsum(m->gout, ns, OUT, dg + m->off_db[2], s));
  TRYC(sgemm(false, false, ns, HID, OUT, m->gout, OUT, p + m->off_dw[2], HID, nullptr, false,
             m->h2, m->gh2, HID, s, pt, pc));
  TRYC(sgemm(true, false, HID, HID, ns, m->gh2, HID, m->h1, HID, nullptr, false, nullptr,
             dg + m->off_dw[1], HID, s, pt, pc));
  TRYC(colsum(m->gh2, ns, HID, dg + m->off_db[1], s));
  TRYC(sgemm(false, false, ns, HID, HID, m->gh2, HID, p + m->off_dw[1], HID, nullptr, false, m->h1,
             m->gh1, HID, s, pt, pc));
  TRYC(sgemm(true, false, HID, W0, ns, m->gh1, HID, m->h0, W0, nullptr, false, nullptr,
             dg + m->off_dw[0], W0, s, pt, pc));
  TRYC(colsum(m->gh1, ns, HID, dg + m->off_db[0], s));
  TRYC(sgemm(false, false, ns, W0, HID, m->gh1, HID, p + m->off_dw[0], W0, nullptr, false, nullptr,
             m->gh0, W0, s, pt, pc));
  // features: sum over the samples of each cell
  feat_grad_kernel<<<(nc * FEAT + 255) / 256, 256, 0, s>>>(m->gh0, nc, kper, m->gpl);
  BS_CHECK_LAUNCH("feat_grad_kernel");
  // convolution layers, last to first
  for (int l = NCONV - 1; l >= 0; --l) {
    const int S = SIDE[l], ci = CIN[l], co = COUT[l];
    const size_t npool = (size_t)nc * co * (S / 2) * (S / 2);
    pool_bwd_kernel<<<(unsigned)((npool + 255) / 256), 256, 0, s>>>(m->gpl, m->z[l], S,
                                                                    log2i(S / 2), npool, m->gz);
    BS_CHECK_LAUNCH("pool_bwd_kernel");
    const float* in = l == 0 ? m->x : m->pl[l - 1];
    // sample groups: four CTAs per SM
    const int nb = co / WCO * (ci + 1), split = std::min({(608 + nb - 1) / nb, WSPLIT, nc});
    conv_bwd_weight_kernel<<<dim3(nb, split), 256, 0, s>>>(m->gz, in, nc, ci, co, S, 2 * log2i(S),
                                                           split, m->wpart);
    BS_CHECK_LAUNCH("conv_bwd_weight_kernel");
    conv_wgrad_reduce_kernel<<<(co * (ci + 1) * 9 + 255) / 256, 256, 0, s>>>(
        m->wpart, ci, co, split, dg + m->off_w[l], dg + m->off_b[l]);
    BS_CHECK_LAUNCH("conv_wgrad_reduce_kernel");
    // the gradient of the pooled output of layer l - 1
    if (l > 0)
      TRYC(conv<true>(m->gz, p + m->off_w[l], nullptr, co, ci, S, nc, m->gpl, nullptr, s));
  }
  return BS_OK;
}

int stage_inputs(bs_cnn* m, const uint16_t* phase, const double* table, const long* toff,
                 const int* nph, const int* hex, int nc, const double* Q, int kper,
                 cudaStream_t s) {
  const int ns = nc * kper;
  std::vector<long> to(nc);
  std::vector<int> np(nc);
  cudaError_t e = cudaMemcpy(to.data(), toff, nc * sizeof(long), cudaMemcpyDefault);
  if (e == cudaSuccess) e = cudaMemcpy(np.data(), nph, nc * sizeof(int), cudaMemcpyDefault);
  if (e != cudaSuccess) return bs_cuda_status(e, "cnn table offsets");
  long tot = 0;
  for (int c = 0; c < nc; ++c) {
    if (to[c] < 0 || np[c] < 1) {
      bs_set_error("cnn: cell %d has a negative table offset or no phase", c);
      return BS_EINVAL;
    }
    tot = std::max(tot, to[c] + 3L * np[c]);
  }
  e = cudaMemcpyAsync(m->phase, phase, (size_t)nc * IMG * IMG * 2, cudaMemcpyDefault, s);
  if ((size_t)tot > m->table_cap) {
    bs_set_error("cnn: property tables exceed the capacity (%ld > %zu doubles)", tot, m->table_cap);
    return BS_EINVAL;
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(m->table, table, tot * sizeof(double), cudaMemcpyDefault, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(m->toff, toff, nc * sizeof(long), cudaMemcpyDefault, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(m->nph, nph, nc * sizeof(int), cudaMemcpyDefault, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(m->hex, hex, nc * sizeof(int), cudaMemcpyDefault, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(m->Q, Q, (size_t)ns * 2 * sizeof(double), cudaMemcpyDefault, s);
  if (e != cudaSuccess) return bs_cuda_status(e, "cnn inputs");
  encode_kernel<<<dim3(nc, 4), 256, 0, s>>>(m->phase, m->table, m->toff, m->nph, m->x);
  BS_CHECK_LAUNCH("encode_kernel");
  kfeat_kernel<<<(ns + 255) / 256, 256, 0, s>>>(m->Q, m->hex, ns, kper, m->kf);
  BS_CHECK_LAUNCH("kfeat_kernel");
  // (the copies read the caller's arrays; both entry points end with a
  // synchronisation, so none is needed here and the layers queue up behind)
  return BS_OK;
}

int check_call(const bs_cnn* m, int nc, int kper) {
  if (!m || nc < 1 || kper < 1 || nc > m->cmax || nc * kper > m->smax) {
    bs_set_error("cnn: need 1 <= ncells <= %d and ncells * kper <= %d", m ? m->cmax : 0,
                 m ? m->smax : 0);
    return BS_EINVAL;
  }
  return BS_OK;
}

}  // namespace

extern "C" int bs_cnn_create(int nvec, int Mp, int max_cells, int max_samples, bs_cnn** out) {
  if (!out || nvec < 1 || nvec > NVMAX || Mp < 0 || Mp > 3 || max_cells < 1 ||
      max_samples < max_cells) {
    bs_set_error("bs_cnn_create: need 1 <= nvec <= %d, 0 <= Mp <= 3, max_samples >= max_cells >= 1",
                 NVMAX);
    return BS_EINVAL;
  }
  *out = nullptr;
  bs_cnn* m = new bs_cnn();
  m->nvec = nvec;
  m->Mp = Mp;
  m->L = 2 * (2 * Mp + 1) * (2 * Mp + 1);
  m->OUT = nvec * m->L * 2;
  m->cmax = max_cells;
  m->smax = max_samples;
  size_t o = 0;
  for (int l = 0; l < NCONV; ++l) {
    m->off_w[l] = o;
    o += (size_t)COUT[l] * CIN[l] * 9;
    m->off_b[l] = o;
    o += COUT[l];
  }
  const int din[3] = {FEAT + KF, HID, HID}, dout[3] = {HID, HID, m->OUT};
  for (int l = 0; l < 3; ++l) {
    m->off_dw[l] = o;
    o += (size_t)din[l] * dout[l];
    m->off_db[l] = o;
    o += dout[l];
  }
  m->nparam = o;
  const size_t C = max_cells, Sm = max_samples;
  int r = BS_OK;
  if (!r) r = calloc_dev(&m->d_p, o, "cnn parameters");
  if (!r) r = calloc_dev(&m->d_g, o, "cnn gradients");
  if (!r) r = calloc_dev(&m->d_m, o, "cnn moments");
  if (!r) r = calloc_dev(&m->d_v, o, "cnn moments");
  if (!r) r = calloc_dev(&m->x, C * 3 * IMG * IMG, "cnn input");
  size_t zmax = 0;
  for (int l = 0; !r && l < NCONV; ++l) {
    const size_t zs = C * COUT[l] * SIDE[l] * SIDE[l];
    zmax = std::max(zmax, zs);
    r = calloc_dev(&m->z[l], zs, "cnn activations");
    if (!r) r = calloc_dev(&m->pl[l], zs / 4, "cnn pooled");
  }
  const size_t W0 = FEAT + KF;
  if (!r) r = calloc_dev(&m->kf, Sm * KF, "cnn k features");
  if (!r) r = calloc_dev(&m->h0, Sm * W0, "cnn h0");
  if (!r) r = calloc_dev(&m->h1, Sm * HID, "cnn h1");
  if (!r) r = calloc_dev(&m->h2, Sm * HID, "cnn h2");
  if (!r) r = calloc_dev(&m->out, Sm * m->OUT, "cnn out");
  if (!r) r = calloc_dev(&m->gout, Sm * m->OUT, "cnn gout");
  if (!r) r = calloc_dev(&m->gh0, Sm * W0, "cnn gh0");
  if (!r) r = calloc_dev(&m->gh1, Sm * HID, "cnn gh1");
  if (!r) r = calloc_dev(&m->gh2, Sm * HID, "cnn gh2");
  if (!r) r = calloc_dev(&m->gpl, std::max(zmax / 4, C * FEAT), "cnn pooled gradients");
  if (!r) r = calloc_dev(&m->gz, zmax, "cnn conv gradients");
  m->tmp_cap = zmax;
  if (!r) r = calloc_dev(&m->gtmp, zmax, "cnn scratch");
  if (!r) r = calloc_dev(&m->wpart, (size_t)WSPLIT * 32 * 33 * 9, "cnn weight partials");
  if (!r) r = calloc_dev(&m->loss, Sm, "cnn loss");
  if (!r) r = calloc_dev(&m->phase, C * IMG * IMG, "cnn phase maps");
  m->table_cap = C * 3 * 64;
  if (!r) r = calloc_dev(&m->table, m->table_cap, "cnn tables");
  if (!r) r = calloc_dev(&m->toff, C, "cnn table offsets");
  if (!r) r = calloc_dev(&m->nph, C, "cnn phase counts");
  if (!r) r = calloc_dev(&m->hex, C, "cnn lattice flags");
  if (!r) r = calloc_dev(&m->Q, Sm * 2, "cnn wavevectors");
  if (!r) r = calloc_dev(&m->tgt, Sm * 16 * m->L * 2, "cnn targets");
  if (!r && cudaMemset(m->d_m, 0, o * 4) != cudaSuccess) r = BS_ECUDA;
  if (!r && cudaMemset(m->d_v, 0, o * 4) != cudaSuccess) r = BS_ECUDA;
  if (r) {
    bs_cnn_destroy(m);
    return r;
  }
  *out = m;
  return BS_OK;
}

extern "C" int bs_cnn_destroy(bs_cnn* m) {
  if (!m) return BS_OK;
  void* ps[] = {m->d_p, m->d_g, m->d_m, m->d_v, m->x, m->kf, m->h0, m->h1, m->h2, m->out, m->gout,
                m->gh0, m->gh1, m->gh2, m->gpl, m->gz, m->gtmp, m->wpart, m->loss, m->phase,
                m->table, m->toff, m->nph, m->hex, m->Q, m->tgt};
  for (void* p : ps) cudaFree(p);
  for (int l = 0; l < NCONV; ++l) {
    cudaFree(m->z[l]);
    cudaFree(m->pl[l]);
  }
  delete m;
  return BS_OK;
}

extern "C" int bs_cnn_num_params(const bs_cnn* m, long long* n) {
  if (!m || !n) {
    bs_set_error("bs_cnn_num_params: NULL argument");
    return BS_EINVAL;
  }
  *n = (long long)m->nparam;
  return BS_OK;
}

extern "C" int bs_cnn_set_params(bs_cnn* m, const float* p) {
  if (!m || !p) {
    bs_set_error("bs_cnn_set_params: NULL argument");
    return BS_EINVAL;
  }
  cudaError_t e = cudaMemcpy(m->d_p, p, m->nparam * 4, cudaMemcpyDefault);
  if (e == cudaSuccess) e = cudaMemset(m->d_m, 0, m->nparam * 4);
  if (e == cudaSuccess) e = cudaMemset(m->d_v, 0, m->nparam * 4);
  if (e != cudaSuccess) return bs_cuda_status(e, "bs_cnn_set_params");
  m->step = 0;
  return BS_OK;
}

extern "C" int bs_cnn_get_params(const bs_cnn* m, float* p, float* grad) {
  if (!m || (!p && !grad)) {
    bs_set_error("bs_cnn_get_params: NULL argument");
    return BS_EINVAL;
  }
  cudaError_t e = cudaSuccess;
  if (p) e = cudaMemcpy(p, m->d_p, m->nparam * 4, cudaMemcpyDefault);
  if (e == cudaSuccess && grad) e = cudaMemcpy(grad, m->d_g, m->nparam * 4, cudaMemcpyDefault);
  if (e != cudaSuccess) return bs_cuda_status(e, "bs_cnn_get_params");
  return BS_OK;
}

extern "C" int bs_cnn_forward(bs_cnn* m, const uint16_t* phase, const double* table,
                              const long* toff, const int* nph, const int* hex, int ncells,
                              const double* Q, int kper, float* U_out, void* stream) {
  TRYC(check_call(m, ncells, kper));
  if (!phase || !table || !toff || !nph || !hex || !Q || !U_out) {
    bs_set_error("bs_cnn_forward: NULL argument");
    return BS_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  TRYC(stage_inputs(m, phase, table, toff, nph, hex, ncells, Q, kper, s));
  TRYC(conv_forward(m, ncells, s));
  TRYC(head_forward(m, ncells, kper, s));
  cudaError_t e = cudaMemcpyAsync(U_out, m->out, (size_t)ncells * kper * m->OUT * 4,
                                  cudaMemcpyDefault, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return bs_cuda_status(e, "bs_cnn_forward");
  return BS_OK;
}

extern "C" int bs_cnn_train_step(bs_cnn* m, const uint16_t* phase, const double* table,
                                 const long* toff, const int* nph, const int* hex, int ncells,
                                 const double* Q, int kper, const float* V, int nb, float lr,
                                 float* loss_out, void* stream) {
  TRYC(check_call(m, ncells, kper));
  if (!phase || !table || !toff || !nph || !hex || !Q || !V || nb < 1 || nb > 16) {
    bs_set_error("bs_cnn_train_step: NULL argument or nb outside [1, 16]");
    return BS_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const int ns = ncells * kper;
  TRYC(stage_inputs(m, phase, table, toff, nph, hex, ncells, Q, kper, s));
  cudaError_t e = cudaMemcpyAsync(m->tgt, V, (size_t)ns * nb * m->L * 2 * 4, cudaMemcpyDefault, s);
  if (e != cudaSuccess) return bs_cuda_status(e, "bs_cnn_train_step targets");
  TRYC(conv_forward(m, ncells, s));
  TRYC(head_forward(m, ncells, kper, s));
  loss_kernel<<<ns, 288, 0, s>>>(m->out, m->tgt, m->L, m->nvec, nb, 1.f / ns, m->loss, m->gout);
  BS_CHECK_LAUNCH("loss_kernel");
  TRYC(backward(m, ncells, kper, s));
  if (lr > 0.f) {
    m->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)m->step), c2 = 1.f - powf(b2, (float)m->step);
    adam_kernel<<<(unsigned)((m->nparam + 255) / 256), 256, 0, s>>>(m->d_p, m->d_g, m->d_m, m->d_v,
                                                                    m->nparam, lr, b1, b2, c1, c2,
                                                                    1e-8f);
    BS_CHECK_LAUNCH("adam_kernel");
  }
  if (loss_out) {
    e = cudaMemcpyAsync(loss_out, m->loss, ns * sizeof(float), cudaMemcpyDefault, s);
    if (e != cudaSuccess) return bs_cuda_status(e, "bs_cnn_train_step loss");
  }
  e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return bs_cuda_status(e, "bs_cnn_train_step");
  return BS_OK;
}
