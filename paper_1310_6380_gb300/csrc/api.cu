// C ABI of libbs: validation, device storage of a cell and the host-side
// orchestration of the assembly, per-k build and eigensolve kernels.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "bs_internal.h"

// ------------------------------------------------------------------ errors
static thread_local char g_err[512] = "";

void bs_set_error(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
}

int bs_cuda_status(cudaError_t e, const char* where) {
  bs_set_error("%s: %s", where, cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? BS_ENOMEM : BS_ECUDA;
}

#define CK(call, where)                                    \
  do {                                                     \
    cudaError_t e__ = (call);                              \
    if (e__ != cudaSuccess) return bs_cuda_status(e__, where); \
  } while (0)

#define TRY(expr)          \
  do {                     \
    int r__ = (expr);      \
    if (r__) return r__;   \
  } while (0)

extern "C" const char* bs_last_error(void) { return g_err; }

// ------------------------------------------------------------------ profiling
static std::atomic<long long> g_launches{0};
static std::atomic<int> g_lob_maxit{BS_LOB_MAXIT};
static std::atomic<int> g_bisect_sweeps{128};

int bs_lob_maxit() { return g_lob_maxit.load(std::memory_order_relaxed); }

int bs_sm_count() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return 152;
  }
  int v = cache[dev].load(std::memory_order_relaxed);
  if (v > 0) return v;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) {
    cudaGetLastError();
    return 152;
  }
  cache[dev].store(v, std::memory_order_relaxed);
  return v;
}
int bs_bisect_sweeps() { return g_bisect_sweeps.load(std::memory_order_relaxed); }

static std::atomic<int> g_reduction{BS_REDUCE_AUTO};

// the reduction to tridiagonal form of the FP64 eigensolve for dimension n:
// the two-stage (band) reduction from BS_BAND_AUTO_MIN on, where its
// tensor-core products outrun the one-stage reduction's FP64 pipe
int bs_reduction_mode() { return g_reduction.load(std::memory_order_relaxed); }

bool bs_use_band(int n, int mode) {
  if (!bs_band_supported(n)) return false;
  if (mode == BS_REDUCE_TWOSTAGE) return true;
  if (mode == BS_REDUCE_ONESTAGE) return false;
  return n >= BS_BAND_AUTO_MIN;
}

// The filtered iteration takes the solves of few branches: it does a
// factorisation and some 60 block products where the reductions do n or n/8
// dependent steps.  A lowered bisection cap (a diagnostic) is meant for the
// tridiagonal path, so that one runs.
//
// The spread of the wave speeds (SpeedSpread) says what the iteration meets: the
// further the wanted eigenvalues lie below the diagonal, the more rounds it
// takes, and the more of the gap above them the rounding errors of its
// certificate's factorisation take (with n and the spread).  What it does not
// certify is reduced one-stage behind it, which loses against the reduction
// alone.  Of the matrices of 700 drawn cells of two and more materials (10 k each,
// stiffnesses up to 3e3 apart, densities up to 1e2, one part in 200 to 1 in
// volume, n = 98 .. 882) none is refused in 6 rounds while n spread <= 30000 and none
// in 8 while it is <= 60000; 1 % are in 12 rounds up to 90000, 10 to 55 % above.
// Rounds that no matrix needs cost their launches, which return at once (six of
// them 0.4 ms; n = 98, one wavevector, 1.86 ms without).  90 wavevectors, n = 882, 18
// branches, a circle of 0.01, 100, 0.001 and 1000 times the matrix's moduli: 27.6,
// 26.7, 162 and 162 ms (the last two reduced; with the iteration before the
// reduction 625).
constexpr double kSpreadRounds6 = 28000.0, kSpreadRounds8 = 56000.0, kSpreadMost = 90000.0;
bool bs_use_filter(int n, int nbands, double spread, int mode) {
  return mode == BS_REDUCE_AUTO && bs_bisect_sweeps() == 128 &&
         bs_filter_fits(n, nbands) && n * spread <= kSpreadMost;
}
int bs_filter_rounds(int n, double spread) {
  const double x = n * spread;
  return x <= kSpreadRounds6 ? 6 : x <= kSpreadRounds8 ? 8 : BS_FILT_ROUNDS;
}

extern "C" int bs_set_reduction(int mode) {
  if (mode != BS_REDUCE_AUTO && mode != BS_REDUCE_ONESTAGE && mode != BS_REDUCE_TWOSTAGE) {
    bs_set_error("bs_set_reduction: mode %d is not BS_REDUCE_AUTO, _ONESTAGE or _TWOSTAGE", mode);
    return BS_EINVAL;
  }
  g_reduction.store(mode, std::memory_order_relaxed);
  return BS_OK;
}

extern "C" int bs_set_iteration_limits(int lobpcg_maxit, int bisect_sweeps) {
  if (lobpcg_maxit > 1000 || bisect_sweeps > 128) {
    bs_set_error("bs_set_iteration_limits: need lobpcg_maxit <= 1000 and bisect_sweeps <= 128");
    return BS_EINVAL;
  }
  g_lob_maxit.store(lobpcg_maxit > 0 ? lobpcg_maxit : BS_LOB_MAXIT, std::memory_order_relaxed);
  g_bisect_sweeps.store(bisect_sweeps > 0 ? bisect_sweeps : 128, std::memory_order_relaxed);
  return BS_OK;
}

void bs_count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

extern "C" int bs_launch_count(long long* out) {
  if (!out) {
    bs_set_error("bs_launch_count: NULL argument");
    return BS_EINVAL;
  }
  *out = g_launches.load();
  return BS_OK;
}

void bs_phase_begin(bs_cell* c, int ph, cudaStream_t s) {
  if (c->prof) cudaEventRecord(c->ev[ph][0], s);
}

void bs_phase_end(bs_cell* c, int ph, cudaStream_t s) {
  if (c->prof) {
    cudaEventRecord(c->ev[ph][1], s);
    c->prof_ready[ph] = true;
  }
}

// ------------------------------------------------------------------ helpers
static bool is_device_ptr(const void* p) {
  if (!p) return false;
  cudaPointerAttributes at;
  cudaError_t e = cudaPointerGetAttributes(&at, p);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

template <typename T>
static int dalloc(T** p, size_t count, const char* what) {
  *p = nullptr;
  if (count == 0) return BS_OK;
  cudaError_t e = cudaMalloc((void**)p, count * sizeof(T));
  if (e != cudaSuccess) {
    *p = nullptr;
    cudaGetLastError();
    bs_set_error("cudaMalloc(%s, %zu bytes) failed: %s", what, count * sizeof(T),
                 cudaGetErrorString(e));
    return BS_ENOMEM;
  }
  return BS_OK;
}

// copy `bytes` from a host or device pointer into host memory
static int fetch_to_host(void* dst, const void* src, size_t bytes) {
  if (is_device_ptr(src)) {
    CK(cudaMemcpy(dst, src, bytes, cudaMemcpyDeviceToHost), "fetch");
  } else {
    memcpy(dst, src, bytes);
  }
  return BS_OK;
}

static int copy_in(void* ddst, const void* src, size_t bytes, cudaStream_t s) {
  CK(cudaMemcpyAsync(ddst, src, bytes, is_device_ptr(src) ? cudaMemcpyDeviceToDevice
                                                           : cudaMemcpyHostToDevice, s),
     "copy in");
  return BS_OK;
}

static void free_workspace(bs_cell* c) {
  if (c->band) {
    bs_band_ws_free(c->band);
    delete c->band;
    c->band = nullptr;
  }
  if (c->filt) {
    bs_filter_ws_free(c->filt);
    delete c->filt;
    c->filt = nullptr;
  }
  void* mixed[] = {c->d_C32, c->d_vec32, c->d_part32, c->d_lamT, c->d_scr, c->d_mY, c->d_mphase,
                   c->d_X32, c->d_X64, c->d_CX, c->d_mG, c->d_H, c->d_W, c->d_theta, c->d_beta,
                   c->d_cxA, c->d_cxB, c->d_cxD, c->d_cxeA, c->d_cxeB};
  for (void* p : mixed) cudaFree(p);
  c->d_cxA = c->d_cxB = nullptr;
  c->d_cxD = nullptr;
  c->d_cxeA = c->d_cxeB = nullptr;
  c->d_C32 = c->d_vec32 = c->d_part32 = c->d_X32 = nullptr;
  c->d_lamT = c->d_scr = c->d_mY = c->d_theta = nullptr;
  c->d_mphase = c->d_X64 = c->d_CX = c->d_mG = c->d_H = c->d_W = c->d_beta = nullptr;
  c->bcap = 0;
  cudaFree(c->d_C);
  cudaFree(c->d_vec);
  cudaFree(c->d_part);
  cudaFree(c->d_de);
  cudaFree(c->d_tau);
  cudaFree(c->d_count);
  cudaFree(c->d_Q);
  cudaFree(c->d_w);
  cudaFree(c->d_stat);
  c->d_C = nullptr;
  c->d_vec = c->d_part = nullptr;
  c->d_de = c->d_tau = c->d_Q = c->d_w = nullptr;
  c->d_count = nullptr;
  c->d_stat = nullptr;
  c->kcap = 0;
  c->wcap = 0;
}

static void free_lob_workspace(bs_cell* c) {
  void* p[] = {c->d_lS, c->d_lCS, c->d_lA, c->d_lpart, c->d_lZ, c->d_lY, c->d_lst, c->d_lX0,
               c->d_lndone, c->d_liters, c->d_lvec, c->d_lsig, c->d_lsc, c->d_liw};
  for (void* q : p) cudaFree(q);
  c->d_lS = c->d_lCS = c->d_lA = c->d_lpart = c->d_lZ = c->d_lY = c->d_lX0 = nullptr;
  c->d_lst = nullptr;
  c->d_lndone = c->d_liters = nullptr;
  c->d_lvec = nullptr;
  c->d_lsig = c->d_lsc = nullptr;
  c->d_liw = nullptr;
  c->lcap = 0;
  c->lbcap = 0;
}

// LOBPCG workspace for `kb` wavevectors and block size `b`
static int ensure_lob_workspace(bs_cell* c, int kb, int b) {
  if (kb <= c->lcap && b <= c->lbcap) return BS_OK;
  kb = std::max(kb, c->lcap);
  b = std::max(b, c->lbcap);
  free_lob_workspace(c);
  const size_t n = c->n, coef = (size_t)BS_LOB_MAX_BLOCK * 3 * BS_LOB_MAX_BLOCK;
  TRY(dalloc(&c->d_lS, 2 * (size_t)kb * 3 * b * n, "LOBPCG basis"));
  TRY(dalloc(&c->d_lCS, 2 * (size_t)kb * 3 * b * n, "LOBPCG C basis"));
  TRY(dalloc(&c->d_lA, (size_t)kb * bs_lob_small_elems(), "LOBPCG Gram"));
  TRY(dalloc(&c->d_lpart, (size_t)kb * bs_lob_part_elems(c->n), "LOBPCG partial Gram"));
  TRY(dalloc(&c->d_lZ, (size_t)kb * coef, "LOBPCG Ritz coefficients"));
  TRY(dalloc(&c->d_lY, (size_t)kb * coef, "LOBPCG P coefficients"));
  TRY(dalloc(&c->d_lst, (size_t)kb, "LOBPCG state"));
  TRY(dalloc(&c->d_lX0, (size_t)kb * b * n, "LOBPCG starting block"));
  TRY(dalloc(&c->d_lndone, 1, "LOBPCG counter"));
  TRY(dalloc(&c->d_liters, (size_t)kb, "LOBPCG iterations"));
  TRY(dalloc(&c->d_lvec, (size_t)kb * b * n, "LOBPCG vectors"));
  TRY(dalloc(&c->d_lsig, (size_t)kb, "inertia shifts"));
  TRY(dalloc(&c->d_lsc, (size_t)kb * n, "inertia scales"));
  TRY(dalloc(&c->d_liw, 3 * (size_t)kb, "inertia counters"));
  c->lcap = kb;
  c->lbcap = b;
  return BS_OK;
}

// per-k workspace for `kb` matrices and `nb` bands
static int ensure_workspace(bs_cell* c, int kb, int nb) {
  if (kb <= c->kcap && nb <= c->wcap) return BS_OK;
  kb = std::max(kb, c->kcap);
  nb = std::max(nb, c->wcap);
  free_workspace(c);
  const int n = c->n;
  TRY(dalloc(&c->d_C, (size_t)kb * n * n, "C(k)"));
  TRY(dalloc(&c->d_vec, (size_t)kb * bs_tridiag_vec_elems(n), "tridiag vectors"));
  TRY(dalloc(&c->d_part, (size_t)kb * bs_tridiag_part_elems(n), "tridiag partials"));
  TRY(dalloc(&c->d_de, (size_t)kb * 2 * n, "tridiagonal"));
  TRY(dalloc(&c->d_tau, (size_t)kb * n, "tau"));
  TRY(dalloc(&c->d_beta, (size_t)kb * n, "beta"));
  TRY(dalloc(&c->d_count, (size_t)kb, "counters"));
  TRY(dalloc(&c->d_Q, (size_t)kb * 2, "Q"));
  TRY(dalloc(&c->d_w, (size_t)kb * nb, "omega"));
  TRY(dalloc(&c->d_stat, (size_t)kb, "status"));
  if (c->precision == BS_PREC_MIXED) {
    const int b = bs_mixed_guard(nb, n);
    TRY(bs_side_create(&c->side));
    TRY(dalloc(&c->d_C32, (size_t)kb * n * n, "C32"));
    TRY(dalloc(&c->d_vec32, (size_t)kb * bs_tridiag_vec_elems(n), "vec32"));
    TRY(dalloc(&c->d_part32, (size_t)kb * bs_tridiag_part_elems(n), "part32"));
    TRY(dalloc(&c->d_lamT, (size_t)kb * (b + 1), "lamT"));
    TRY(dalloc(&c->d_scr, (size_t)kb * b * 5 * n, "inverse iteration"));
    TRY(dalloc(&c->d_mY, (size_t)kb * b * n, "Y"));
    TRY(dalloc(&c->d_mphase, (size_t)kb * n, "phase"));
    TRY(dalloc(&c->d_X32, (size_t)kb * b * n, "X32"));
    TRY(dalloc(&c->d_X64, (size_t)kb * b * n, "X64"));
    TRY(dalloc(&c->d_CX, (size_t)kb * b * n, "CX"));
    TRY(dalloc(&c->d_mG, (size_t)kb * b * b, "G"));
    TRY(dalloc(&c->d_H, (size_t)kb * b * b, "H"));
    TRY(dalloc(&c->d_W, (size_t)kb * b * b, "W"));
    TRY(dalloc(&c->d_theta, (size_t)kb * b, "theta"));
    size_t ca = 0, cb = 0, cd = 0;
    bs_cx_tc_elems(n, b, kb, &ca, &cb, &cd);
    TRY(dalloc(&c->d_cxA, ca, "C digit planes"));
    TRY(dalloc(&c->d_cxB, cb, "X digit planes"));
    TRY(dalloc(&c->d_cxD, cd, "C X digit-pair products"));
    TRY(dalloc(&c->d_cxeA, (size_t)kb * n, "C exponents"));
    TRY(dalloc(&c->d_cxeB, (size_t)kb * b, "X exponents"));
    c->bcap = b;
  }
  c->kcap = kb;
  c->wcap = nb;
  return BS_OK;
}

// largest k batch whose C(k) workspace stays under ~4 GiB
static int k_batch_cap(const bs_cell* c) {
  const size_t per = (size_t)c->n * c->n * sizeof(zd);
  size_t cap = ((size_t)4 << 30) / per;
  return (int)std::max<size_t>(1, std::min<size_t>(cap, 4096));
}

static double omega_floor2(const bs_cell* c);

// ------------------------------------------------------------------ create
// Device storage of a validated cell (pixel map when cen == nullptr, else a
// mesh of nel elements with fractional centroids cen and areas area).
static int create_common(const double h1[2], const double h2[2], double det, int P, int nel, int M,
                         int np, int precision, const std::vector<double>& raw,
                         const std::vector<uint16_t>& ph, const std::vector<double>* cen,
                         const std::vector<double>* area, bs_cell** out) {
  bs_cell* c = new bs_cell;
  memset(c, 0, sizeof(*c));
  c->P = P;
  c->mesh = cen != nullptr;
  c->nel = nel;
  c->M = M;
  c->N = (2 * M + 1) * (2 * M + 1);
  c->n = 2 * c->N;
  c->D = 4 * M + 1;
  c->nphase = np;
  c->nf = 3;
  c->precision = precision;
  for (int i = 0; i < 2; ++i) {
    c->h1[i] = h1[i];
    c->h2[i] = h2[i];
  }
  c->V = fabs(det);
  // reciprocal basis of Eq. (1) in 2-D: q^1 = 2 pi (h2y, -h2x)/det, q^2 = 2 pi (-h1y, h1x)/det
  c->q1[0] = 2.0 * M_PI * h2[1] / det;
  c->q1[1] = -2.0 * M_PI * h2[0] / det;
  c->q2[0] = -2.0 * M_PI * h1[1] / det;
  c->q2[1] = 2.0 * M_PI * h1[0] / det;

  const size_t NN = (size_t)c->N * c->N, nn = (size_t)c->n * c->n;
  int r = BS_OK;
  if (!r) r = dalloc(&c->d_phase, ph.size(), "phase");
  if (!r) r = dalloc(&c->d_table, 6 * (size_t)np, "table");
  if (!r) r = dalloc(&c->d_E, (size_t)c->D * P, "E");
  if (!r) r = dalloc(&c->d_Y, 3 * (size_t)P * c->D, "Y");
  if (!r) r = dalloc(&c->d_ghat, (c->mesh ? 4 : 3) * (size_t)c->D * c->D, "ghat");
  if (!r && c->mesh) r = dalloc(&c->d_cen, 2 * (size_t)nel, "mesh centroids");
  if (!r && c->mesh) r = dalloc(&c->d_area, (size_t)nel, "mesh areas");
  if (!r && c->mesh) r = dalloc(&c->d_I1, NN, "mesh Gram matrix of the plane waves");
  if (!r && c->mesh) r = dalloc(&c->d_mpart, bs_mesh_partial_elems(M, nel, 4), "mesh partials");
  if (!r) r = dalloc(&c->d_T, 3 * NN, "T");
  if (!r) r = dalloc(&c->d_Linv, 3 * NN, "Linv");
  if (!r) r = dalloc(&c->d_G, 2 * (size_t)c->N, "G");
  if (!r) r = dalloc(&c->d_F, 6 * NN, "F");
  if (!r) r = dalloc(&c->d_Pp, 12 * NN, "P");
  if (!r) r = dalloc(&c->d_Cm, 6 * nn, "Cm");
  if (!r) r = dalloc(&c->d_info, 4, "info");
  size_t sa = 0, sb = 0, sd = 0;
  bs_fields_tc_elems(P, c->D, 3, &sa, &sb, &sd);
  if (!r) r = dalloc(&c->d_sliceA, sa, "field digit planes");
  if (!r) r = dalloc(&c->d_sliceB, sb, "exponential digit planes");
  if (!r) r = dalloc(&c->d_sliceD, sd, "digit-pair products");
  if (!r) r = dalloc(&c->d_expA, 3 * (size_t)P, "field exponents");
  if (!r) r = dalloc(&c->d_expB, 2 * (size_t)c->D, "table exponents");
  size_t ma = 0, mb = 0, md = 0;
  bs_zgemm_tc_elems(c->N, 2, &ma, &mb, &md);
  if (!r) r = dalloc(&c->d_mA, ma, "monomial digit planes A");
  if (!r) r = dalloc(&c->d_mB, mb, "monomial digit planes B");
  if (!r) r = dalloc(&c->d_mD, md, "monomial digit-pair products");
  if (!r) r = dalloc(&c->d_meA, 2 * (size_t)c->N, "monomial exponents A");
  if (!r) r = dalloc(&c->d_meB, 2 * (size_t)c->N, "monomial exponents B");
  if (!r) r = dalloc(&c->d_LinvR2, 2 * NN, "L_R^-1 pair");
  if (r) {
    bs_destroy_cell(c);
    return r;
  }
  std::vector<double> G(2 * (size_t)c->N);
  for (int a = 0; a < c->N; ++a) {
    const int al = a / (2 * M + 1) - M, be = a % (2 * M + 1) - M;
    G[a] = al * c->q1[0] + be * c->q2[0];
    G[c->N + a] = al * c->q1[1] + be * c->q2[1];
  }
  cudaError_t e = cudaMemcpy(c->d_phase, ph.data(), ph.size() * 2, cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(c->d_table + 3 * np, raw.data(), raw.size() * 8, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(c->d_G, G.data(), G.size() * 8, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(c->d_info, 0, 4 * sizeof(int));
  if (e == cudaSuccess && c->mesh)
    e = cudaMemcpy(c->d_cen, cen->data(), cen->size() * 8, cudaMemcpyHostToDevice);
  if (e == cudaSuccess && c->mesh)
    e = cudaMemcpy(c->d_area, area->data(), area->size() * 8, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    r = bs_cuda_status(e, "bs_create_cell upload");
    bs_destroy_cell(c);
    return r;
  }
  c->tol = 1e-6;
  c->floor2 = omega_floor2(c);
  std::vector<double> vol(np, 0.0);   // of every phase
  for (size_t i = 0; i < ph.size(); ++i) vol[ph[i]] += area ? (*area)[i] : 1.0;
  SpeedSpread sp;
  for (int i = 0; i < np; ++i) {
    const double b = 2.0 * (raw[i] + raw[np + i]), g = 2.0 * raw[np + i];
    if (vol[i] > 0.0) sp.add(vol[i], std::min(b, g), std::max(b, g), raw[2 * np + i]);
  }
  c->spread = sp.value();
  *out = c;
  return BS_OK;
}

extern "C" int bs_create_cell(const bs_cell_desc* d, bs_cell** out) {
  if (!d || !out) {
    bs_set_error("bs_create_cell: NULL argument");
    return BS_EINVAL;
  }
  *out = nullptr;
  const int P = d->P, M = d->M, np = d->nphase;
  if (P < 1 || P > 4096 || M < 0 || M > 15 || 2 * M + 1 > P || np < 1 || np > 65536 ||
      !d->phase || !d->lam || !d->mu || !d->rho) {
    bs_set_error("bs_create_cell: need 1 <= P <= 4096, 0 <= M <= 15, 2M+1 <= P, 1 <= nphase "
                 "<= 65536 and non-NULL arrays (P=%d M=%d nphase=%d)", P, M, np);
    return BS_EINVAL;
  }
  if (d->precision != BS_PREC_FP64 && d->precision != BS_PREC_MIXED) {
    bs_set_error("bs_create_cell: unknown precision %d", d->precision);
    return BS_EINVAL;
  }
  const double det = d->h1[0] * d->h2[1] - d->h1[1] * d->h2[0];
  if (!(fabs(det) > 0.0) || !isfinite(det)) {
    bs_set_error("bs_create_cell: h1, h2 are not a basis");
    return BS_EINVAL;
  }
  std::vector<double> raw(3 * (size_t)np);
  TRY(fetch_to_host(raw.data(), d->lam, np * sizeof(double)));
  TRY(fetch_to_host(raw.data() + np, d->mu, np * sizeof(double)));
  TRY(fetch_to_host(raw.data() + 2 * np, d->rho, np * sizeof(double)));
  for (int i = 0; i < np; ++i) {
    const double lam = raw[i], mu = raw[np + i], rho = raw[2 * np + i];
    if (!isfinite(lam) || !isfinite(mu) || !isfinite(rho) || !(mu > 0.0) || !(lam + mu > 0.0) ||
        !(rho > 0.0)) {
      bs_set_error("bs_create_cell: phase %d has lam=%g mu=%g rho=%g (need mu > 0, "
                   "lam + mu > 0, rho > 0, finite)", i, lam, mu, rho);
      return BS_EINVAL;
    }
  }
  std::vector<uint16_t> ph((size_t)P * P);
  TRY(fetch_to_host(ph.data(), d->phase, ph.size() * sizeof(uint16_t)));
  for (size_t i = 0; i < ph.size(); ++i)
    if (ph[i] >= np) {
      bs_set_error("bs_create_cell: pixel %zu has phase %u >= nphase %d", i, ph[i], np);
      return BS_EINVAL;
    }

  return create_common(d->h1, d->h2, det, P, P * P, M, np, d->precision, raw, ph, nullptr, nullptr,
                       out);
}

extern "C" int bs_create_cell_mesh(const bs_mesh_desc* d, bs_cell** out) {
  if (!d || !out) {
    bs_set_error("bs_create_cell_mesh: NULL argument");
    return BS_EINVAL;
  }
  *out = nullptr;
  const int nel = d->nel, M = d->M, np = d->nphase;
  const long N = (2L * M + 1) * (2L * M + 1);
  if (M < 0 || M > 15 || nel < N || nel > (1 << 26) || np < 1 || np > 65536 || !d->centroid ||
      !d->area || !d->phase || !d->lam || !d->mu || !d->rho) {
    bs_set_error("bs_create_cell_mesh: need 0 <= M <= 15, (2M+1)^2 <= nel <= 2^26, 1 <= nphase "
                 "<= 65536 and non-NULL arrays (nel=%d M=%d nphase=%d)", nel, M, np);
    return BS_EINVAL;
  }
  if (d->precision != BS_PREC_FP64 && d->precision != BS_PREC_MIXED) {
    bs_set_error("bs_create_cell_mesh: unknown precision %d", d->precision);
    return BS_EINVAL;
  }
  const double det = d->h1[0] * d->h2[1] - d->h1[1] * d->h2[0];
  if (!(fabs(det) > 0.0) || !isfinite(det)) {
    bs_set_error("bs_create_cell_mesh: h1, h2 are not a basis");
    return BS_EINVAL;
  }
  std::vector<double> raw(3 * (size_t)np);
  TRY(fetch_to_host(raw.data(), d->lam, np * sizeof(double)));
  TRY(fetch_to_host(raw.data() + np, d->mu, np * sizeof(double)));
  TRY(fetch_to_host(raw.data() + 2 * np, d->rho, np * sizeof(double)));
  for (int i = 0; i < np; ++i) {
    const double lam = raw[i], mu = raw[np + i], rho = raw[2 * np + i];
    if (!isfinite(lam) || !isfinite(mu) || !isfinite(rho) || !(mu > 0.0) || !(lam + mu > 0.0) ||
        !(rho > 0.0)) {
      bs_set_error("bs_create_cell_mesh: phase %d has lam=%g mu=%g rho=%g (need mu > 0, "
                   "lam + mu > 0, rho > 0, finite)", i, lam, mu, rho);
      return BS_EINVAL;
    }
  }
  std::vector<uint16_t> ph((size_t)nel);
  std::vector<double> cen(2 * (size_t)nel), area((size_t)nel);
  TRY(fetch_to_host(ph.data(), d->phase, ph.size() * sizeof(uint16_t)));
  TRY(fetch_to_host(cen.data(), d->centroid, cen.size() * sizeof(double)));
  TRY(fetch_to_host(area.data(), d->area, area.size() * sizeof(double)));
  for (int i = 0; i < nel; ++i) {
    if (ph[i] >= np || !(area[i] > 0.0) || !isfinite(area[i]) || !isfinite(cen[2 * i]) ||
        !isfinite(cen[2 * i + 1])) {
      bs_set_error("bs_create_cell_mesh: element %d has phase %u (nphase %d), area %g, "
                   "centroid (%g, %g) (need phase < nphase, area > 0, finite)", i, ph[i], np,
                   area[i], cen[2 * i], cen[2 * i + 1]);
      return BS_EINVAL;
    }
  }
  return create_common(d->h1, d->h2, det, 0, nel, M, np, d->precision, raw, ph, &cen, &area, out);
}


// Re-size the field-dependent storage of a cell for nf material fields.
static int realloc_fields(bs_cell* c, int nf) {
  const size_t NN = (size_t)c->N * c->N, D2 = (size_t)c->D * c->D;
  const int P = c->P, np = c->nphase;
  std::vector<double> raw(3 * (size_t)np);
  CK(cudaMemcpy(raw.data(), c->d_table + (size_t)c->nf * np, raw.size() * 8,
                cudaMemcpyDeviceToHost), "bs_set_stiffness raw");
  zd** zbufs[] = {&c->d_Y, &c->d_ghat, &c->d_T, &c->d_mpart, &c->d_Phi, &c->d_LPhi, &c->d_Yw,
                  &c->d_Wk, &c->d_Pab};
  for (zd** b : zbufs) {
    cudaFree(*b);
    *b = nullptr;
  }
  cudaFree(c->d_table);
  cudaFree(c->d_sliceA);
  cudaFree(c->d_sliceD);
  cudaFree(c->d_expA);
  c->d_table = nullptr;
  c->d_sliceA = nullptr;
  c->d_sliceD = nullptr;
  c->d_expA = nullptr;
  int r = BS_OK;
  if (!r) r = dalloc(&c->d_table, (size_t)(nf + 3) * np, "table");
  if (!r) r = dalloc(&c->d_Y, (size_t)nf * P * c->D, "Y");
  if (!r) r = dalloc(&c->d_ghat, (size_t)(nf + (c->mesh ? 1 : 0)) * D2, "ghat");
  if (!r) r = dalloc(&c->d_T, (size_t)nf * NN, "T");
  if (!r && c->mesh)
    r = dalloc(&c->d_mpart, bs_mesh_partial_elems(c->M, c->nel, nf + 1), "mesh partials");
  size_t sa = 0, sb = 0, sd = 0;
  bs_fields_tc_elems(P, c->D, nf, &sa, &sb, &sd);
  if (!r) r = dalloc(&c->d_sliceA, sa, "field digit planes");
  if (!r) r = dalloc(&c->d_sliceD, sd, "digit-pair products");
  if (!r) r = dalloc(&c->d_expA, (size_t)nf * P, "field exponents");
  if (!r) r = dalloc(&c->d_Phi, 9 * NN, "Phi");
  if (!r) r = dalloc(&c->d_LPhi, 9 * NN, "Phi inverse factor");
  if (!r) r = dalloc(&c->d_Yw, 18 * NN, "H_i Z");
  if (!r) r = dalloc(&c->d_Wk, 18 * NN, "W_i");
  if (!r) r = dalloc(&c->d_Pab, 24 * NN, "W_a W_b^dagger");
  if (!r && nf == 7 && bs_zgemm_tc_fits(3 * c->N)) {
    // the exact-slice workspace grows to the anisotropic products: W_t (N x 3N
    // over K = N, two halves) and the monomials (2N x 2N over K = 3N)
    size_t ma = 0, mb = 0, md = 0, a1 = 0, b1 = 0, d1 = 0;
    bs_zgemm_tc_elems(c->N, 2, &ma, &mb, &md);
    bs_zgemm_tc_rect_elems(c->N, 3 * c->N, c->N, 2, &a1, &b1, &d1);
    ma = std::max(ma, a1), mb = std::max(mb, b1), md = std::max(md, d1);
    bs_zgemm_tc_rect_elems(2 * c->N, 2 * c->N, 3 * c->N, 1, &a1, &b1, &d1);
    ma = std::max(ma, a1), mb = std::max(mb, b1), md = std::max(md, d1);
    cudaFree(c->d_mA);
    cudaFree(c->d_mB);
    cudaFree(c->d_mD);
    cudaFree(c->d_meB);
    c->d_mA = nullptr;
    c->d_mB = nullptr;
    c->d_mD = nullptr;
    c->d_meB = nullptr;
    r = dalloc(&c->d_mA, ma, "monomial digit planes A");
    if (!r) r = dalloc(&c->d_mB, mb, "monomial digit planes B");
    if (!r) r = dalloc(&c->d_mD, md, "monomial digit-pair products");
    if (!r) r = dalloc(&c->d_meB, 6 * (size_t)c->N, "monomial exponents B");
  }
  if (r) return r;
  CK(cudaMemcpy(c->d_table + (size_t)nf * np, raw.data(), raw.size() * 8, cudaMemcpyHostToDevice),
     "bs_set_stiffness raw");
  c->nf = nf;
  return BS_OK;
}

extern "C" int bs_set_stiffness(bs_cell* c, const double* C6) {
  if (!c || !C6) {
    bs_set_error("bs_set_stiffness: NULL argument");
    return BS_EINVAL;
  }
  const int np = c->nphase;
  std::vector<double> cv(6 * (size_t)np);
  TRY(fetch_to_host(cv.data(), C6, cv.size() * sizeof(double)));
  std::vector<double> raw(3 * (size_t)np);
  CK(cudaMemcpy(raw.data(), c->d_table + (size_t)c->nf * np, raw.size() * 8,
                cudaMemcpyDeviceToHost), "bs_set_stiffness raw");
  // derived rows: S11, S22, rho, S12, S13, S23, S33 of S = C^-1 (Voigt)
  std::vector<double> tab(7 * (size_t)np);
  // volume of every phase, for the spread of the wave speeds
  std::vector<uint16_t> ph((size_t)c->nel);
  std::vector<double> area(c->mesh ? c->nel : 0), vol(np, 0.0);
  CK(cudaMemcpy(ph.data(), c->d_phase, ph.size() * 2, cudaMemcpyDeviceToHost),
     "bs_set_stiffness phases");
  if (c->mesh)
    CK(cudaMemcpy(area.data(), c->d_area, area.size() * 8, cudaMemcpyDeviceToHost),
       "bs_set_stiffness areas");
  for (size_t i = 0; i < ph.size(); ++i) vol[ph[i]] += c->mesh ? area[i] : 1.0;
  SpeedSpread sp;
  double c2min = 1e300;
  for (int i = 0; i < np; ++i) {
    const double* v = &cv[6 * (size_t)i];
    const double C[3][3] = {{v[0], v[2], v[3]}, {v[2], v[1], v[4]}, {v[3], v[4], v[5]}};
    // positive definite by its leading minors; inverse by cofactors
    const double m1 = C[0][0], m2 = C[0][0] * C[1][1] - C[0][1] * C[1][0];
    const double co00 = C[1][1] * C[2][2] - C[1][2] * C[2][1];
    const double co01 = -(C[1][0] * C[2][2] - C[1][2] * C[2][0]);
    const double co02 = C[1][0] * C[2][1] - C[1][1] * C[2][0];
    const double det = C[0][0] * co00 + C[0][1] * co01 + C[0][2] * co02;
    bool ok = true;
    for (int k = 0; k < 6; ++k) ok = ok && isfinite(v[k]);
    if (!ok || !(m1 > 0.0) || !(m2 > 0.0) || !(det > 0.0)) {
      bs_set_error("bs_set_stiffness: phase %d stiffness is not symmetric positive definite", i);
      return BS_EINVAL;
    }
    const double S00 = co00 / det, S01 = co01 / det, S02 = co02 / det;
    const double S11 = (C[0][0] * C[2][2] - C[0][2] * C[2][0]) / det;
    const double S12 = -(C[0][0] * C[2][1] - C[0][1] * C[2][0]) / det;
    const double S22 = m2 / det;
    const double rho = raw[2 * (size_t)np + i];
    const double row[7] = {S00, S11, rho, S01, S02, S12, S22};
    for (int f = 0; f < 7; ++f) tab[(size_t)f * np + i] = row[f];
    // smallest eigenvalue of C by bisection on "C - x I is positive definite"
    // (leading minors), a monotone test on [0, min diagonal]; the slowest
    // shear-like speed squared of the phase is taken as lo / rho
    double lo = 0.0, hi = std::min(std::min(C[0][0], C[1][1]), C[2][2]);
    auto pd = [&](double x) {
      const double a = C[0][0] - x, b = C[1][1] - x, e = C[2][2] - x;
      const double d3 = a * (b * e - C[1][2] * C[2][1]) - C[0][1] * (C[1][0] * e - C[1][2] * C[2][0]) +
                        C[0][2] * (C[1][0] * C[2][1] - b * C[2][0]);
      return a > 0.0 && a * b - C[0][1] * C[1][0] > 0.0 && d3 > 0.0;
    };
    for (int it = 0; it < 200; ++it) {
      const double mid = 0.5 * (lo + hi);
      if (pd(mid)) lo = mid; else hi = mid;
    }
    c2min = std::min(c2min, lo / rho);
    if (vol[i] > 0.0) {
      // extreme eigenvalues of the tensor (third row and column by sqrt 2), to a
      // percent, by the signs of the leading minors of t (C - x I), t = +1 or -1
      const double q = sqrt(2.0);
      auto extreme = [&](double t, double x0, double x1) {
        for (int it = 0; it < 40 && x1 > 1.01 * x0; ++it) {
          const double x = x0 > 0.0 ? sqrt(x0 * x1) : 0.01 * x1;
          const double a = t * (C[0][0] - x), b = t * (C[1][1] - x), e = t * (2.0 * C[2][2] - x);
          const double f = t * C[0][1], g = t * q * C[0][2], h = t * q * C[1][2];
          const double d3 = a * (b * e - h * h) - f * (f * e - h * g) + g * (f * h - b * g);
          const bool definite = a > 0.0 && a * b - f * f > 0.0 && d3 > 0.0;
          if (definite == (t > 0.0)) x0 = x; else x1 = x;
        }
        return t > 0.0 ? x0 : x1;
      };
      const double tr = C[0][0] + C[1][1] + 2.0 * C[2][2];
      const double big = extreme(-1.0, tr / 3.0, tr);
      sp.add(vol[i], std::max(extreme(1.0, 0.0, tr / 3.0), 1e-12 * tr), big, rho);
    }
  }
  if (!c->aniso) TRY(realloc_fields(c, 7));
  c->aniso = true;
  CK(cudaMemcpy(c->d_table, tab.data(), tab.size() * 8, cudaMemcpyHostToDevice),
     "bs_set_stiffness table");
  const double q2 = std::min(c->q1[0] * c->q1[0] + c->q1[1] * c->q1[1],
                             c->q2[0] * c->q2[0] + c->q2[1] * c->q2[1]);
  c->floor2 = c2min * q2 / 4.0;
  c->spread = sp.value();
  c->assembled = false;
  return BS_OK;
}

extern "C" int bs_destroy_cell(bs_cell* c) {
  if (!c) return BS_OK;
  bs_set_profiling(c, 0);
  free_workspace(c);
  bs_free_mode_workspace(c);
  free_lob_workspace(c);
  bs_side_free(c->side);
  cudaFree(c->d_phase);
  cudaFree(c->d_table);
  cudaFree(c->d_E);
  cudaFree(c->d_Y);
  cudaFree(c->d_ghat);
  cudaFree(c->d_T);
  cudaFree(c->d_Linv);
  cudaFree(c->d_G);
  cudaFree(c->d_F);
  cudaFree(c->d_Pp);
  cudaFree(c->d_Cm);
  cudaFree(c->d_info);
  cudaFree(c->d_sliceA);
  cudaFree(c->d_sliceB);
  cudaFree(c->d_sliceD);
  cudaFree(c->d_expA);
  cudaFree(c->d_expB);
  cudaFree(c->d_mA);
  cudaFree(c->d_mB);
  cudaFree(c->d_mD);
  cudaFree(c->d_meA);
  cudaFree(c->d_meB);
  cudaFree(c->d_LinvR2);
  cudaFree(c->d_cen);
  cudaFree(c->d_area);
  cudaFree(c->d_I1);
  cudaFree(c->d_mpart);
  cudaFree(c->d_Phi);
  cudaFree(c->d_LPhi);
  cudaFree(c->d_Yw);
  cudaFree(c->d_Wk);
  cudaFree(c->d_Pab);
  delete c;
  return BS_OK;
}

extern "C" int bs_cell_dims(const bs_cell* c, int* N, int* n) {
  if (!c) {
    bs_set_error("bs_cell_dims: NULL cell");
    return BS_EINVAL;
  }
  if (N) *N = c->N;
  if (n) *n = c->n;
  return BS_OK;
}

// ------------------------------------------------------------------ assemble
extern "C" int bs_assemble(bs_cell* c, void* stream) {
  if (!c) {
    bs_set_error("bs_assemble: NULL cell");
    return BS_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const size_t NN = (size_t)c->N * c->N;
  CK(cudaMemsetAsync(c->d_info, 0, 3 * sizeof(int), s), "bs_assemble");
  for (int i = 0; i < PH_COUNT; ++i) c->prof_ready[i] = false;
  bs_phase_begin(c, PH_ASM, s);
  if (c->mesh)
    TRY(bs_launch_mesh_assembly(c, s));                            // a1 + a2 on mesh elements
  else
    TRY(bs_launch_assembly(c, s));                                 // a1 + a2
  bs_phase_end(c, PH_ASM, s);
  bs_phase_begin(c, PH_GRAM, s);
  TRY(bs_launch_toeplitz(c, s));                                   // a3 expansion
  if (c->aniso) {
    TRY(bs_launch_gram_aniso(c, s));                               // R and the full Phi
  } else if (c->precision == BS_PREC_FP64) {
    TRY(bs_launch_gram_factor(c->d_T, c->d_Linv, c->N, 3, (long)NN, c->d_info, s));
  } else {
    TRY(bs_launch_cholesky(c->d_T, c->N, 3, (long)NN, c->d_info, s)); // a3 factors
    TRY(bs_launch_trinv(c->d_T, c->d_Linv, c->N, 3, (long)NN, s));
  }
  bs_phase_end(c, PH_GRAM, s);
  bs_phase_begin(c, PH_MONO, s);
  if (c->aniso)
    TRY(bs_launch_monomials_aniso(c, s));
  else
    TRY(bs_launch_monomials(c, s));                                // a3/a4 coefficients
  bs_phase_end(c, PH_MONO, s);
  c->assembled = true;
  return BS_OK;
}

// stress: also a wait of the last bs_stress_coefficients
static int check_info(bs_cell* c, cudaStream_t s, bool stress = false) {
  int info[3] = {0, 0, 0};
  CK(cudaMemcpyAsync(info, c->d_info, 3 * sizeof(int), cudaMemcpyDeviceToHost, s), "info");
  CK(cudaStreamSynchronize(s), "sync");
  if (info[0]) {
    bs_set_error("Cholesky of a Gram matrix failed (not positive definite)");
    return BS_ENOTPD;
  }
  if (info[1] || (stress && info[2])) {
    bs_set_error("a tensor-core pipeline wait reached its limit");
    return BS_ECUDA;
  }
  return BS_OK;
}

extern "C" int bs_filter_counts(const bs_cell* c, int counts[2]) {
  if (!c || !counts) {
    bs_set_error("bs_filter_counts: NULL argument");
    return BS_EINVAL;
  }
  return bs_filter_read_counts(c->filt, counts);
}

extern "C" int bs_sync(bs_cell* c, void* stream) {
  if (!c) {
    bs_set_error("bs_sync: NULL cell");
    return BS_EINVAL;
  }
  return check_info(c, (cudaStream_t)stream, true);
}

// ------------------------------------------------------------------ solve
// Solve a chunk of kb wavevectors already in c->d_Q; results in c->d_w / d_stat.
// omega_floor^2 = (c_T,min |q|_min / 2)^2: below it frequencies are compared
// in absolute terms (the acoustic branches vanish at Gamma)
static double omega_floor2(const bs_cell* c) {
  std::vector<double> raw(3 * (size_t)c->nphase);
  cudaMemcpy(raw.data(), c->d_table + (size_t)c->nf * c->nphase, raw.size() * 8,
             cudaMemcpyDeviceToHost);
  double ct2 = 1e300;
  for (int i = 0; i < c->nphase; ++i) ct2 = std::min(ct2, raw[c->nphase + i] / raw[2 * c->nphase + i]);
  const double q2 = std::min(c->q1[0] * c->q1[0] + c->q1[1] * c->q1[1],
                             c->q2[0] * c->q2[0] + c->q2[1] * c->q2[1]);
  return ct2 * q2 / 4.0;
}

static int solve_chunk_mixed(bs_cell* c, int kb, int nbands, cudaStream_t s) {
  const int n = c->n, b = bs_mixed_guard(nbands, n);
  bs_phase_begin(c, PH_BUILD, s);
  TRY(bs_launch_builder_mixed(c->d_Cm, n, c->d_Q, kb, c->q1[0], c->q1[1], c->q2[0], c->q2[1],
                              c->d_C, c->d_C32, s));
  bs_phase_end(c, PH_BUILD, s);
  bs_phase_begin(c, PH_TRID, s);
  TRY(bs_launch_tridiag<float>(c->d_C32, n, kb, c->d_vec32, c->d_part32, c->d_de, c->d_tau,
                               c->d_beta, c->d_count, s, 64, c->side));
  bs_phase_end(c, PH_TRID, s);
  bs_phase_begin(c, PH_BISECT, s);
  TRY(bs_launch_bisect(c->d_de, n, kb, std::min(b + 1, n), c->d_lamT, nullptr, s, false, 1e-9));
  bs_phase_end(c, PH_BISECT, s);
  bs_phase_begin(c, PH_REFINE, s);
  MixedWs w;
  w.C64 = c->d_C; w.C32 = c->d_C32; w.de = c->d_de; w.tau = c->d_tau; w.beta = c->d_beta;
  w.lamT = c->d_lamT; w.scratch = c->d_scr; w.Y = c->d_mY; w.phase = c->d_mphase;
  w.X32 = c->d_X32; w.X64 = c->d_X64; w.CX = c->d_CX; w.G = c->d_mG; w.H = c->d_H; w.W = c->d_W;
  w.theta = c->d_theta;
  w.cxA = c->d_cxA; w.cxB = c->d_cxB; w.cxD = c->d_cxD; w.cxeA = c->d_cxeA; w.cxeB = c->d_cxeB;
  w.err = c->d_info + 1;
  TRY(bs_launch_mixed_refine(w, n, kb, nbands, b, c->tol, c->floor2, c->d_w, c->d_stat, s));
  bs_phase_end(c, PH_REFINE, s);
  return BS_OK;
}

// first: the first chunk of a solve
static int solve_chunk(bs_cell* c, int kb, int nbands, bool first, cudaStream_t s) {
  if (c->precision == BS_PREC_MIXED) return solve_chunk_mixed(c, kb, nbands, s);
  const int mode = bs_reduction_mode();   // once: the build and the solve have to agree
  const bool filt = bs_use_filter(c->n, nbands, c->spread, mode);
  bs_phase_begin(c, PH_BUILD, s);
  TRY(bs_launch_builder(c->d_Cm, c->n, c->d_Q, kb, c->q1[0], c->q1[1], c->q2[0], c->q2[1], c->d_C,
                        s, filt));
  bs_phase_end(c, PH_BUILD, s);
  bs_phase_begin(c, PH_TRID, s);
  if (filt && !c->filt) c->filt = new FilterWs();
  if (c->filt && first) c->filt->taken = 0;
  // no memory for its workspace: the reductions below need less
  if (filt && bs_filter_ws_alloc(c->filt, c->n, c->kcap) == BS_OK) {
    const FilterFallback fb{c->d_vec, c->d_part, c->d_de, c->d_tau, c->d_beta, c->d_count};
    TRY(bs_launch_eig_filter(c->d_C, c->n, kb, nbands, *c->filt, fb, c->d_w, c->d_stat,
                             c->d_info + 1, bs_filter_rounds(c->n, c->spread), s));
    c->band_used = false;
    bs_phase_end(c, PH_TRID, s);
    c->prof_ready[PH_BISECT] = false;
    return BS_OK;
  }
  if (bs_use_band(c->n, mode)) {
    if (!c->band) c->band = new BandWs();
    TRY(bs_band_ws_alloc(c->band, c->n, c->kcap, BS_SLICES_BAND));
    c->band->prof = c->prof;
    // the bisection of each part runs inside the reduction, behind its
    // bulge chase (the bisect phase is then part of the tridiag phase)
    BandBisect bis{nbands, c->d_w, c->d_stat};
    TRY(bs_launch_eig_band(c->d_C, c->n, kb, *c->band, c->d_de, c->d_info + 1, s, &bis));
    c->band_used = true;
    bs_phase_end(c, PH_TRID, s);
    c->prof_ready[PH_BISECT] = false;
    return BS_OK;
  }
  TRY(bs_launch_tridiag<double>(c->d_C, c->n, kb, c->d_vec, c->d_part, c->d_de, c->d_tau,
                                c->d_beta, c->d_count, s));
  c->band_used = false;
  bs_phase_end(c, PH_TRID, s);
  bs_phase_begin(c, PH_BISECT, s);
  TRY(bs_launch_bisect(c->d_de, c->n, kb, nbands, c->d_w, c->d_stat, s));
  bs_phase_end(c, PH_BISECT, s);
  return BS_OK;
}

extern "C" int bs_solve_k(bs_cell* c, const double* Q, int nk, int nbands, double* omega_out,
                          int* status_out, void* stream) {
  if (!c || !Q || !omega_out || nk < 0) {
    bs_set_error("bs_solve_k: NULL argument or nk < 0");
    return BS_EINVAL;
  }
  if (!c->assembled) {
    bs_set_error("bs_solve_k: call bs_assemble first");
    return BS_ESTATE;
  }
  if (nbands < 1 || nbands > c->n) {
    bs_set_error("bs_solve_k: nbands=%d outside [1, %d]", nbands, c->n);
    return BS_EINVAL;
  }
  if (c->precision == BS_PREC_MIXED &&
      (nbands > BS_MIXED_MAX_BANDS || nbands + 2 > c->n || c->n > 2048)) {
    bs_set_error("bs_solve_k: the mixed path needs nbands <= %d, nbands + 2 <= n and n <= 2048 "
                 "(n = %d)", BS_MIXED_MAX_BANDS, c->n);
    return BS_EINVAL;
  }
  if (nk == 0) return BS_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const bool q_dev = is_device_ptr(Q), w_dev = is_device_ptr(omega_out);
  const bool st_dev = status_out && is_device_ptr(status_out);
  const int cap = k_batch_cap(c);
  TRY(ensure_workspace(c, std::min(nk, cap), nbands));
  // synchronous call without a status array: the statuses still decide the return code
  std::vector<int> hst(!w_dev && !status_out ? nk : 0);
  for (int k0 = 0; k0 < nk; k0 += cap) {
    const int kb = std::min(cap, nk - k0);
    CK(cudaMemcpyAsync(c->d_Q, Q + 2 * (size_t)k0, 2 * kb * sizeof(double),
                       q_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s),
       "bs_solve_k Q");
    TRY(solve_chunk(c, kb, nbands, k0 == 0, s));
    if (!hst.empty())
      CK(cudaMemcpyAsync(hst.data() + k0, c->d_stat, kb * sizeof(int), cudaMemcpyDeviceToHost, s),
         "bs_solve_k status");
    CK(cudaMemcpyAsync(omega_out + (size_t)k0 * nbands, c->d_w, (size_t)kb * nbands * sizeof(double),
                       w_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s),
       "bs_solve_k omega");
    if (status_out)
      CK(cudaMemcpyAsync(status_out + k0, c->d_stat, kb * sizeof(int),
                         st_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s),
         "bs_solve_k status");
  }
  if (!w_dev || (status_out && !st_dev)) {
    TRY(check_info(c, s));
    const int* hs = status_out && !st_dev ? status_out : (hst.empty() ? nullptr : hst.data());
    if (hs)
      for (int k = 0; k < nk; ++k)
        if (hs[k]) {
          bs_set_error("bs_solve_k: wavevector %d did not converge", k);
          return BS_ENOCONV;
        }
  }
  return BS_OK;
}

// ------------------------------------------------------------------ LOBPCG
// One chunk of kb wavevectors (in c->d_Q): FP32 LOBPCG from the starting
// block, FP64 Rayleigh-Ritz tail; omega / status in c->d_w / c->d_stat,
// iterations in c->d_liters, vectors (optional) in c->d_lvec.
static int solve_chunk_lobpcg(bs_cell* c, int kb, int nbands, int b, const float* X0, bool x0_dev,
                              int nvec, bool want_vec, cudaStream_t s) {
  const int n = c->n, N = c->N;
  bs_phase_begin(c, PH_BUILD, s);
  TRY(bs_launch_builder_mixed(c->d_Cm, n, c->d_Q, kb, c->q1[0], c->q1[1], c->q2[0], c->q2[1],
                              c->d_C, c->d_C32, s, true));
  if (nvec > 0) {
    // starting vectors in displacement coefficients -> reduced basis y = L_R^dagger u
    CK(cudaMemcpyAsync(c->d_lvec, X0, (size_t)kb * nvec * n * sizeof(float2),
                       x0_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s),
       "LOBPCG starting vectors");
    TRY(bs_launch_lob_to_reduced(c->d_lvec, c->d_T + 2 * (size_t)N * N, N, c->M, -1, kb, nvec,
                                 c->d_lX0, s));
  }
  bs_phase_end(c, PH_BUILD, s);
  bs_phase_begin(c, PH_TRID, s);
  LobWs w;
  w.C32 = c->d_C32;
  w.S = c->d_lS;
  w.CS = c->d_lCS;
  w.Axp = c->d_lA;
  w.part = c->d_lpart;
  w.Z = c->d_lZ;
  w.Y = c->d_lY;
  w.st = c->d_lst;
  w.X0 = nvec > 0 ? c->d_lX0 : nullptr;
  w.nvec = nvec;
  w.ndone = c->d_lndone;
  const float tol32 = (float)std::max(sqrt(c->tol), 3e-4);
  TRY(bs_launch_lobpcg(w, n, kb, b, nbands, bs_lob_maxit(), tol32, (float)c->tol, (float)c->floor2,
                       4, s));
  TRY(bs_launch_lob_export(w, n, kb, b, c->d_X64, c->d_liters, s));
  bs_phase_end(c, PH_TRID, s);
  bs_phase_begin(c, PH_REFINE, s);
  MixedWs m;
  memset(&m, 0, sizeof(m));
  m.C64 = c->d_C;
  m.X64 = c->d_X64;
  m.CX = c->d_CX;
  m.G = c->d_mG;
  m.H = c->d_H;
  m.W = c->d_W;
  m.theta = c->d_theta;
  m.lamT = nullptr;
  m.cxA = c->d_cxA;
  m.cxB = c->d_cxB;
  m.cxD = c->d_cxD;
  m.cxeA = c->d_cxeA;
  m.cxeB = c->d_cxeB;
  m.err = c->d_info + 1;
  m.csig = c->d_lsig;         // the count check's shift and expected count
  m.cexp = c->d_liw + kb;
  CK(cudaMemsetAsync(c->d_stat, 0, kb * sizeof(int), s), "status");
  TRY(bs_launch_rr_tail(m, n, kb, nbands, b, c->tol, c->floor2, c->d_w, c->d_stat, s));
  // no eigenvalue skipped below the wanted ones (C32 is free after the iterations)
  TRY(bs_launch_inertia_check(c->d_C32, n, kb, c->d_theta, b, nbands, c->floor2, c->d_lsig,
                              c->d_lsc, c->d_liw, c->d_stat, nullptr, s, true));
  if (want_vec)
    TRY(bs_launch_lob_vectors(c->d_X64, c->d_W, c->d_Linv + 2 * (size_t)N * N, 0, kb, N, c->M, -1,
                              b, nbands, kb, nullptr, c->d_lvec, s));
  bs_phase_end(c, PH_REFINE, s);
  return BS_OK;
}

// dense FP64 solve of the wavevectors Q (host, nf x 2) on an assembled cell:
// omega (host, nf x nbands) and status (host, nf)
int bs_cell_dense_fp64(bs_cell* c, const double* Q, int nf, int nbands, double* om, int* st,
                       cudaStream_t s) {
  if (nf <= 0) return BS_OK;
  TRY(ensure_workspace(c, std::min(nf, std::min(k_batch_cap(c), 256)), nbands));
  const int cap = c->kcap;
  for (int k0 = 0; k0 < nf; k0 += cap) {
    const int kb = std::min(cap, nf - k0);
    CK(cudaMemcpyAsync(c->d_Q, Q + 2 * (size_t)k0, 2 * kb * sizeof(double),
                       cudaMemcpyHostToDevice, s), "fallback Q");
    TRY(bs_launch_builder(c->d_Cm, c->n, c->d_Q, kb, c->q1[0], c->q1[1], c->q2[0], c->q2[1],
                          c->d_C, s));
    TRY(bs_launch_tridiag<double>(c->d_C, c->n, kb, c->d_vec, c->d_part, c->d_de, c->d_tau,
                                  c->d_beta, c->d_count, s));
    TRY(bs_launch_bisect(c->d_de, c->n, kb, nbands, c->d_w, c->d_stat, s));
    CK(cudaMemcpyAsync(om + (size_t)k0 * nbands, c->d_w, (size_t)kb * nbands * 8,
                       cudaMemcpyDeviceToHost, s), "fallback omega");
    CK(cudaMemcpyAsync(st + k0, c->d_stat, kb * sizeof(int), cudaMemcpyDeviceToHost, s),
       "fallback status");
    CK(cudaStreamSynchronize(s), "fallback sync");
  }
  return BS_OK;
}

extern "C" int bs_solve_k_lobpcg(bs_cell* c, const double* Q, int nk, int nbands,
                                 const float* X0, int nvec, double* omega_out, int* status_out,
                                 int* iters_out, int* fallback_out, float* vec_out,
                                 void* stream) {
  if (!c || !Q || !omega_out || nk < 0) {
    bs_set_error("bs_solve_k_lobpcg: NULL argument or nk < 0");
    return BS_EINVAL;
  }
  if (!c->assembled) {
    bs_set_error("bs_solve_k_lobpcg: call bs_assemble first");
    return BS_ESTATE;
  }
  if (c->precision != BS_PREC_MIXED) {
    bs_set_error("bs_solve_k_lobpcg: the cell must be created with BS_PREC_MIXED");
    return BS_EINVAL;
  }
  if (nbands < 1 || nbands > BS_LOB_MAX_BANDS || nbands + 5 > c->n || c->n > 2048) {
    bs_set_error("bs_solve_k_lobpcg: need 1 <= nbands <= %d, nbands + 5 <= n and n <= 2048 "
                 "(nbands = %d, n = %d)", BS_LOB_MAX_BANDS, nbands, c->n);
    return BS_EINVAL;
  }
  const int b = bs_lob_block(nbands, c->n);
  if (nvec < 0 || nvec > b || (nvec > 0 && !X0)) {
    bs_set_error("bs_solve_k_lobpcg: nvec = %d outside [0, %d] or X0 NULL", nvec, b);
    return BS_EINVAL;
  }
  if (nk == 0) return BS_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const int n = c->n;
  const bool q_dev = is_device_ptr(Q), w_dev = is_device_ptr(omega_out);
  const bool st_dev = status_out && is_device_ptr(status_out);
  const bool it_dev = iters_out && is_device_ptr(iters_out);
  const bool fb_dev = fallback_out && is_device_ptr(fallback_out);
  const bool v_dev = vec_out && is_device_ptr(vec_out);
  const bool x0_dev = X0 && is_device_ptr(X0);
  const int cap = std::min(k_batch_cap(c), 1024);
  TRY(ensure_workspace(c, std::min(nk, cap), nbands));
  TRY(ensure_lob_workspace(c, std::min(nk, cap), b));
  std::vector<double> Qh(2 * (size_t)nk);
  TRY(fetch_to_host(Qh.data(), Q, Qh.size() * sizeof(double)));
  std::vector<int> fb(nk, 0);
  for (int k0 = 0; k0 < nk; k0 += cap) {
    const int kb = std::min(cap, nk - k0);
    CK(cudaMemcpyAsync(c->d_Q, Qh.data() + 2 * (size_t)k0, 2 * kb * sizeof(double),
                       cudaMemcpyHostToDevice, s), "bs_solve_k_lobpcg Q");
    TRY(solve_chunk_lobpcg(c, kb, nbands, b, X0 ? X0 + (size_t)k0 * nvec * n * 2 : nullptr, x0_dev,
                           nvec, vec_out != nullptr, s));
    CK(cudaMemcpyAsync(omega_out + (size_t)k0 * nbands, c->d_w, (size_t)kb * nbands * sizeof(double),
                       w_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s),
       "bs_solve_k_lobpcg omega");
    if (iters_out)
      CK(cudaMemcpyAsync(iters_out + k0, c->d_liters, kb * sizeof(int),
                         it_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s),
         "bs_solve_k_lobpcg iterations");
    if (vec_out)
      CK(cudaMemcpyAsync(vec_out + (size_t)k0 * nbands * n * 2, c->d_lvec,
                         (size_t)kb * nbands * n * sizeof(float2),
                         v_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s),
         "bs_solve_k_lobpcg vectors");
    std::vector<int> sth(kb);
    CK(cudaMemcpyAsync(sth.data(), c->d_stat, kb * sizeof(int), cudaMemcpyDeviceToHost, s),
       "bs_solve_k_lobpcg status");
    TRY(check_info(c, s));
    for (int k = 0; k < kb; ++k) fb[k0 + k] = sth[k] != 0;
  }
  // dense FP64 fallback for the wavevectors the residual bound did not certify
  std::vector<double> Qf;
  std::vector<int> idx;
  for (int k = 0; k < nk; ++k)
    if (fb[k]) {
      idx.push_back(k);
      Qf.push_back(Qh[2 * (size_t)k]);
      Qf.push_back(Qh[2 * (size_t)k + 1]);
    }
  std::vector<int> stk(nk, 0);
  if (!idx.empty()) {
    bs_phase_begin(c, PH_BISECT, s);
    std::vector<double> om(idx.size() * nbands);
    std::vector<int> st(idx.size());
    TRY(bs_cell_dense_fp64(c, Qf.data(), (int)idx.size(), nbands, om.data(), st.data(), s));
    bs_phase_end(c, PH_BISECT, s);
    const std::vector<float> nanv((size_t)nbands * n * 2, NAN);
    for (size_t t = 0; t < idx.size(); ++t) {
      const int k = idx[t];
      stk[k] = st[t];
      CK(cudaMemcpyAsync(omega_out + (size_t)k * nbands, om.data() + t * nbands, nbands * 8,
                         w_dev ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost, s),
         "fallback scatter");
      if (vec_out)
        CK(cudaMemcpyAsync(vec_out + (size_t)k * nbands * n * 2, nanv.data(), nanv.size() * 4,
                           v_dev ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost, s),
           "fallback vectors");
    }
    CK(cudaStreamSynchronize(s), "fallback sync");
  }
  if (status_out)
    CK(cudaMemcpyAsync(status_out, stk.data(), nk * sizeof(int),
                       st_dev ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost, s), "status out");
  if (fallback_out)
    CK(cudaMemcpyAsync(fallback_out, fb.data(), nk * sizeof(int),
                       fb_dev ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost, s), "fallback out");
  CK(cudaStreamSynchronize(s), "bs_solve_k_lobpcg sync");
  for (int k = 0; k < nk; ++k)
    if (stk[k] && !status_out) {
      bs_set_error("bs_solve_k_lobpcg: wavevector %d did not converge", k);
      return BS_ENOCONV;
    }
  return BS_OK;
}

// IBZ boundary path, uniform in Cartesian arc length
static int make_path(const bs_cell* c, int path, int nk, std::vector<double>& Q) {
  static const double sq[4][2] = {{0, 0}, {0.5, 0}, {0.5, 0.5}, {0, 0}};
  static const double hx[4][2] = {{0, 0}, {0.5, 0}, {2.0 / 3.0, 1.0 / 3.0}, {0, 0}};
  const double(*pc)[2];
  if (path == BS_PATH_SQUARE_GXMG) pc = sq;
  else if (path == BS_PATH_HEX_GMKG) pc = hx;
  else {
    bs_set_error("bs_bands: unknown path %d", path);
    return BS_EINVAL;
  }
  double seg[3], cum[4] = {0, 0, 0, 0};
  for (int i = 0; i < 3; ++i) {
    const double dq1 = pc[i + 1][0] - pc[i][0], dq2 = pc[i + 1][1] - pc[i][1];
    const double kx = dq1 * c->q1[0] + dq2 * c->q2[0], ky = dq1 * c->q1[1] + dq2 * c->q2[1];
    seg[i] = sqrt(kx * kx + ky * ky);
    cum[i + 1] = cum[i] + seg[i];
  }
  Q.resize(2 * (size_t)nk);
  for (int i = 0; i < nk; ++i) {
    const double sarc = cum[3] * i / (nk - 1);
    int j = 0;
    while (j < 2 && sarc >= cum[j + 1]) ++j;
    double t = seg[j] == 0 ? 0.0 : (sarc - cum[j]) / seg[j];
    t = std::min(std::max(t, 0.0), 1.0);
    Q[2 * i] = pc[j][0] + t * (pc[j + 1][0] - pc[j][0]);
    Q[2 * i + 1] = pc[j][1] + t * (pc[j + 1][1] - pc[j][1]);
  }
  return BS_OK;
}

extern "C" int bs_bands(bs_cell* c, int path, int nk, int nbands, double* Q_out,
                        double* omega_out, void* stream) {
  if (!c || !omega_out || nk < 2) {
    bs_set_error("bs_bands: NULL argument or nk < 2");
    return BS_EINVAL;
  }
  std::vector<double> Q;
  TRY(make_path(c, path, nk, Q));
  cudaStream_t s = (cudaStream_t)stream;
  if (Q_out) {
    CK(cudaMemcpyAsync(Q_out, Q.data(), Q.size() * sizeof(double),
                       is_device_ptr(Q_out) ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost, s),
       "bs_bands Q_out");
  }
  int r = bs_solve_k(c, Q.data(), nk, nbands, omega_out, nullptr, stream);
  if (r) return r;
  CK(cudaStreamSynchronize(s), "bs_bands sync");   // Q lives on this host stack
  return BS_OK;
}

extern "C" int bs_set_profiling(bs_cell* c, int on) {
  if (!c) {
    bs_set_error("bs_set_profiling: NULL cell");
    return BS_EINVAL;
  }
  if (on && !c->prof) {
    for (int i = 0; i < PH_COUNT; ++i)
      for (int j = 0; j < 2; ++j) CK(cudaEventCreate(&c->ev[i][j]), "bs_set_profiling");
  }
  if (!on && c->prof) {
    for (int i = 0; i < PH_COUNT; ++i)
      for (int j = 0; j < 2; ++j) cudaEventDestroy(c->ev[i][j]);
  }
  c->prof = on != 0;
  for (int i = 0; i < PH_COUNT; ++i) c->prof_ready[i] = false;
  return BS_OK;
}

extern "C" int bs_phase_times(bs_cell* c, double ms[8]) {
  if (!c || !ms) {
    bs_set_error("bs_phase_times: NULL argument");
    return BS_EINVAL;
  }
  for (int i = 0; i < PH_COUNT; ++i) {
    ms[i] = 0.0;
    if (!c->prof || !c->prof_ready[i]) continue;
    CK(cudaEventSynchronize(c->ev[i][1]), "bs_phase_times");
    float t = 0.f;
    CK(cudaEventElapsedTime(&t, c->ev[i][0], c->ev[i][1]), "bs_phase_times");
    ms[i] = t;
  }
  return BS_OK;
}

extern "C" int bs_reduction_times(bs_cell* c, double ms[6]) {
  if (!c || !ms) {
    bs_set_error("bs_reduction_times: NULL argument");
    return BS_EINVAL;
  }
  for (int i = 0; i < 6; ++i) ms[i] = 0.0;
  if (!c->prof || !c->band_used || !c->band) return BS_OK;
  TRY(bs_band_times(*c->band, ms));
  ms[5] = c->band->timed;
  return BS_OK;
}

// ------------------------------------------------------------------ diagnostics
namespace {
// 8 independent FMA chains per thread; the sum is stored so that nothing is
// optimised away
__global__ void __launch_bounds__(256) fp64_fma_probe_kernel(int iters, double seed,
                                                             double* __restrict__ out) {
  double a[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = seed + 1e-3 * (threadIdx.x + i);
  const double x = 1.0 - 1e-9, y = 1e-12;
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = fma(a[i], x, y);
  }
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) s += a[i];
  if (s == 12345.678) out[blockIdx.x] = s;   // never true; keeps the chains live
}
}  // namespace

extern "C" int bs_probe_fp64(int blocks_per_sm, int iters, double* tflops, void* stream) {
  if (!tflops || iters < 1 || blocks_per_sm < 1 || blocks_per_sm > 8) {
    bs_set_error("bs_probe_fp64: need tflops, iters >= 1, 1 <= blocks_per_sm <= 8");
    return BS_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const int grid = blocks_per_sm * bs_sm_count();
  double* out = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e = cudaMalloc((void**)&out, grid * sizeof(double));
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  float ms = 0.f;
  if (e == cudaSuccess) {
    fp64_fma_probe_kernel<<<grid, 256, 0, s>>>(iters, 1.0, out);   // warm-up
    g_launches.fetch_add(1, std::memory_order_relaxed);
    e = cudaEventRecord(e0, s);
  }
  if (e == cudaSuccess) {
    fp64_fma_probe_kernel<<<grid, 256, 0, s>>>(iters, 2.0, out);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaEventRecord(e1, s);
  if (e == cudaSuccess) e = cudaEventSynchronize(e1);
  if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaFree(out);
  if (e != cudaSuccess) return bs_cuda_status(e, "bs_probe_fp64");
  *tflops = 2.0 * 8.0 * iters * (double)grid * 256.0 / (ms * 1e-3) / 1e12;
  return BS_OK;
}

extern "C" int bs_gemm_bf16(const uint16_t* A, const uint16_t* B, float* D, int M, int N, int K,
                            int batch, void* stream) {
  if (!A || !B || !D || M < 1 || N < 1 || K < 8 || K % 8 || K > 4096 || batch < 1 ||
      batch > 65535) {
    bs_set_error("bs_gemm_bf16: need non-NULL arrays, M, N >= 1, 8 <= K <= 4096, K %% 8 == 0, "
                 "1 <= batch <= 65535");
    return BS_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const size_t na = (size_t)batch * M * K, nb = (size_t)batch * N * K, nd = (size_t)batch * M * N;
  uint16_t *dA = nullptr, *dB = nullptr;
  float* dD = nullptr;
  int* err = nullptr;
  const bool ad = is_device_ptr(A), bd = is_device_ptr(B), dd = is_device_ptr(D);
  int r = BS_OK;
  if (!ad) r = dalloc(&dA, na, "A");
  if (!r && !bd) r = dalloc(&dB, nb, "B");
  if (!r && !dd) r = dalloc(&dD, nd, "D");
  if (!r) r = dalloc(&err, 1, "err");
  cudaError_t ce = cudaSuccess;
  if (!r) ce = cudaMemsetAsync(err, 0, sizeof(int), s);
  if (!r && ce == cudaSuccess && !ad) ce = cudaMemcpyAsync(dA, A, na * 2, cudaMemcpyHostToDevice, s);
  if (!r && ce == cudaSuccess && !bd) ce = cudaMemcpyAsync(dB, B, nb * 2, cudaMemcpyHostToDevice, s);
  if (!r && ce != cudaSuccess) r = bs_cuda_status(ce, "bs_gemm_bf16 copy");
  if (!r)
    r = bs_launch_slice_gemm(ad ? A : dA, bd ? B : dB, dd ? D : dD, M, N, K, batch, (long)M * K,
                             (long)N * K, M, (long)M * N, err, s);
  int herr = 0;
  if (!r && !dd) {
    ce = cudaMemcpyAsync(D, dD, nd * 4, cudaMemcpyDeviceToHost, s);
    if (ce != cudaSuccess) r = bs_cuda_status(ce, "bs_gemm_bf16 copy out");
  }
  if (!r) {
    ce = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) r = bs_cuda_status(ce, "bs_gemm_bf16 sync");
    else if (herr) {
      bs_set_error("bs_gemm_bf16: a tensor-core pipeline wait reached its limit");
      r = BS_ECUDA;
    }
  } else {
    cudaStreamSynchronize(s);
  }
  cudaFree(dA);
  cudaFree(dB);
  cudaFree(dD);
  cudaFree(err);
  return r;
}

extern "C" int bs_tridiag_eigenvalues(const double* d, const double* e, int n, int batch,
                                      int nbands, double* lam_out, void* stream) {
  if (!d || (!e && n > 1) || !lam_out || n < 1 || batch < 1 || nbands < 1 || nbands > n ||
      n > 100000) {
    bs_set_error("bs_tridiag_eigenvalues: need non-NULL arrays, n >= 1, batch >= 1, "
                 "1 <= nbands <= n");
    return BS_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  double* de = nullptr;
  double* out = nullptr;
  int* st = nullptr;
  int r = dalloc(&de, (size_t)batch * 2 * n, "tridiagonals");
  const bool odev = is_device_ptr(lam_out);
  if (!r && !odev) r = dalloc(&out, (size_t)batch * nbands, "eigenvalues");
  if (!r) r = dalloc(&st, (size_t)batch, "status");
  auto kind = [](const void* p) {
    return is_device_ptr(p) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  };
  cudaError_t ce = cudaSuccess;
  if (!r) ce = cudaMemset2DAsync(de + n, 2 * n * sizeof(double), 0, n * sizeof(double), batch, s);
  if (!r && ce == cudaSuccess)
    ce = cudaMemcpy2DAsync(de, 2 * n * sizeof(double), d, n * sizeof(double), n * sizeof(double),
                           batch, kind(d), s);
  if (!r && ce == cudaSuccess && n > 1)
    ce = cudaMemcpy2DAsync(de + n, 2 * n * sizeof(double), e, (n - 1) * sizeof(double),
                           (n - 1) * sizeof(double), batch, kind(e), s);
  if (!r && ce != cudaSuccess) r = bs_cuda_status(ce, "bs_tridiag_eigenvalues copy");
  if (!r) r = bs_launch_bisect(de, n, batch, nbands, odev ? lam_out : out, st, s, false);
  if (!r && !odev) {
    ce = cudaMemcpyAsync(lam_out, out, (size_t)batch * nbands * sizeof(double),
                         cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) r = bs_cuda_status(ce, "bs_tridiag_eigenvalues copy out");
  }
  if (odev) cudaStreamSynchronize(s);   // the scratch below is freed on return
  cudaFree(de);
  cudaFree(out);
  cudaFree(st);
  return r;
}

extern "C" int bs_form_factors(bs_cell* c, double* out, void* stream) {
  if (!c || !out) {
    bs_set_error("bs_form_factors: NULL argument");
    return BS_EINVAL;
  }
  if (!c->assembled) {
    bs_set_error("bs_form_factors: call bs_assemble first");
    return BS_ESTATE;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const bool dev = is_device_ptr(out);
  CK(cudaMemcpyAsync(out, c->d_ghat, (size_t)c->nf * c->D * c->D * sizeof(zd),
                     dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s),
     "bs_form_factors");
  if (!dev) CK(cudaStreamSynchronize(s), "bs_form_factors sync");
  return BS_OK;
}

extern "C" int bs_reduced_matrix(bs_cell* c, const double* Q, double* out, void* stream) {
  if (!c || !Q || !out) {
    bs_set_error("bs_reduced_matrix: NULL argument");
    return BS_EINVAL;
  }
  if (!c->assembled) {
    bs_set_error("bs_reduced_matrix: call bs_assemble first");
    return BS_ESTATE;
  }
  cudaStream_t s = (cudaStream_t)stream;
  TRY(ensure_workspace(c, 1, 1));
  TRY(copy_in(c->d_Q, Q, 2 * sizeof(double), s));
  TRY(bs_launch_builder(c->d_Cm, c->n, c->d_Q, 1, c->q1[0], c->q1[1], c->q2[0], c->q2[1], c->d_C, s));
  const bool dev = is_device_ptr(out);
  CK(cudaMemcpyAsync(out, c->d_C, (size_t)c->n * c->n * sizeof(zd),
                     dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s),
     "bs_reduced_matrix");
  if (!dev) TRY(check_info(c, s));
  return BS_OK;
}
