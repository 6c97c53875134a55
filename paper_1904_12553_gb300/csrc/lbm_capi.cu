// C ABI of the N-phase phase-field lattice Boltzmann solver: parameter
// validation, derived constants, workspace layout, and the host driver of
// the kernels. The arithmetic of a time step lives in lbm_kernels.cuh.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <new>

#include "lbm_internal.h"
#include "lbm_nphase.h"

using lbm::Consts;
using lbm::Grid;
using lbm::Outputs;

namespace {

constexpr double CS2 = 1.0 / 3.0;

bool finite_pos(double v) { return isfinite(v) && v > 0.0; }

// Coefficient of lambda_ij in the equation of pair (k, l): Eq. N15 (l = N)
// and Eq. N16 (l < N), 0-based phases.
double Lcoef(const lbm_nphase_params *p, int i, int k, int l) {
  const int n = p->N - 1;
  const double rN = p->rho[n];
  if (l == n) return i == k ? 1.0 : rN / (p->rho[i] + rN);
  if (i == k) return p->rho[k] / (p->rho[k] + rN);
  if (i == l) return -p->rho[l] / (p->rho[l] + rN);
  return 0.0;
}

// Least-squares-free square solve A x = b by Householder QR (m <= 10).
// Returns false if R has a (relatively) vanishing diagonal entry.
bool householder_solve(int m, double A[10][10], double b[10], double x[10]) {
  double amax = 0.0;
  for (int r = 0; r < m; ++r)
    for (int c = 0; c < m; ++c) amax = fmax(amax, fabs(A[r][c]));
  if (amax == 0.0) return false;
  for (int c = 0; c < m; ++c) {
    double nrm = 0.0;
    for (int r = c; r < m; ++r) nrm += A[r][c] * A[r][c];
    nrm = sqrt(nrm);
    if (nrm <= 1e-13 * amax) return false;
    const double alpha = A[c][c] > 0 ? -nrm : nrm;
    double v[10];
    for (int r = 0; r < m; ++r) v[r] = r < c ? 0.0 : A[r][c];
    v[c] -= alpha;
    double vv = 0.0;
    for (int r = c; r < m; ++r) vv += v[r] * v[r];
    if (vv == 0.0) continue;
    for (int cc = c; cc < m; ++cc) {
      double d = 0.0;
      for (int r = c; r < m; ++r) d += v[r] * A[r][cc];
      d = 2.0 * d / vv;
      for (int r = c; r < m; ++r) A[r][cc] -= d * v[r];
    }
    double d = 0.0;
    for (int r = c; r < m; ++r) d += v[r] * b[r];
    d = 2.0 * d / vv;
    for (int r = c; r < m; ++r) b[r] -= d * v[r];
  }
  for (int r = m - 1; r >= 0; --r) {
    double s = b[r];
    for (int c = r + 1; c < m; ++c) s -= A[r][c] * x[c];
    x[r] = s / A[r][r];
  }
  return true;
}

// Extreme eigenvalues of a symmetric n x n matrix (n <= 4), cyclic Jacobi.
void sym_eig_range(int n, const double M[4][4], double *lo, double *hi) {
  double a[4][4];
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) a[i][j] = M[i][j];
  for (int sweep = 0; sweep < 100; ++sweep) {
    double off = 0.0;
    for (int i = 0; i < n; ++i)
      for (int j = i + 1; j < n; ++j) off += a[i][j] * a[i][j];
    if (off < 1e-40) break;
    for (int p = 0; p < n; ++p)
      for (int q = p + 1; q < n; ++q) {
        if (a[p][q] == 0.0) continue;
        const double th = 0.5 * atan2(2.0 * a[p][q], a[q][q] - a[p][p]);
        const double c = cos(th), s = sin(th);
        for (int r = 0; r < n; ++r) {
          const double arp = a[r][p], arq = a[r][q];
          a[r][p] = c * arp - s * arq;
          a[r][q] = s * arp + c * arq;
        }
        for (int r = 0; r < n; ++r) {
          const double apr = a[p][r], aqr = a[q][r];
          a[p][r] = c * apr - s * aqr;
          a[q][r] = s * apr + c * aqr;
        }
      }
  }
  *lo = a[0][0];
  *hi = a[0][0];
  for (int i = 1; i < n; ++i) {
    *lo = fmin(*lo, a[i][i]);
    *hi = fmax(*hi, a[i][i]);
  }
}

bool cholesky_ok(int n, const double M[4][4]) {
  double L[4][4] = {{0}};
  for (int j = 0; j < n; ++j) {
    double d = M[j][j];
    for (int k = 0; k < j; ++k) d -= L[j][k] * L[j][k];
    if (!(d > 0.0)) return false;
    L[j][j] = sqrt(d);
    for (int i = j + 1; i < n; ++i) {
      double s = M[i][j];
      for (int k = 0; k < j; ++k) s -= L[i][k] * L[j][k];
      L[i][j] = s / L[j][j];
    }
  }
  return true;
}

lbm_status validate(const lbm_nphase_params *p) {
  if (!p) return LBM_EINVAL;
  if (p->N < 2 || p->N > LBM_MAX_N) return LBM_EINVAL;
  if (p->nx < 1 || p->ny < 1 || p->nx > (1 << 20) || p->ny > (1 << 20))
    return LBM_EINVAL;
  if (p->lattice != 0 && p->lattice != 1) return LBM_EINVAL;
  if (p->lattice == 0 && p->nz != 0 && p->nz != 1) return LBM_EINVAL;
  if (p->lattice == 1 && (p->nz < 1 || p->nz > (1 << 20) || p->grad_scheme != 0))
    return LBM_EINVAL;
  // The generic kernels launch one CTA per tile on a 2-D (D2Q9: 32 x 8
  // tiles) or 3-D (D3Q15: 32 x 4 x 2 tiles) grid, at most 65535 tiles along
  // y and z.
  if (p->lattice == 0 && lbm::tiles_y(p->ny) > 65535) return LBM_EINVAL;
  if (p->lattice == 1 &&
      (lbm::tiles3_y(p->ny) > 65535 || lbm::tiles3_z(p->nz) > 65535))
    return LBM_EINVAL;
  if ((double)p->nx * (double)p->ny * (double)(p->nz > 1 ? p->nz : 1) >
      17179869184.0)
    return LBM_EINVAL;
  if (p->wall_y != 0 && p->wall_y != 1) return LBM_EINVAL;
  if (p->precision < LBM_FP64 || p->precision > LBM_MIX_FP16) return LBM_EINVAL;
  if (p->grad_scheme != 0 && p->grad_scheme != 1) return LBM_EINVAL;
  for (int k = 0; k < p->N; ++k)
    if (!finite_pos(p->rho[k])) return LBM_EINVAL;
  for (int k = 0; k < p->N; ++k)
    for (int l = k + 1; l < p->N; ++l) {
      const double a = p->sigma[k][l], b = p->sigma[l][k];
      if (!finite_pos(a) || !finite_pos(b)) return LBM_EINVAL;
      if (fabs(a - b) > 1e-12 * fmax(a, b)) return LBM_EINVAL;
    }
  if (!finite_pos(p->eta)) return LBM_EINVAL;
  if (!isfinite(p->beta)) return LBM_EINVAL;
  if (!(isfinite(p->tau_g) && p->tau_g > 0.5)) return LBM_EINVAL;
  for (int i = 0; i < p->N - 1; ++i) {
    if (!(isfinite(p->tau[i]) && p->tau[i] > 0.5)) return LBM_EINVAL;
    if (!finite_pos(p->mobility[i])) return LBM_EINVAL;
  }
  if (!isfinite(p->gravity[0]) || !isfinite(p->gravity[1]) ||
      !isfinite(p->gravity[2]) || !isfinite(p->rho0))
    return LBM_EINVAL;
  if (p->lattice == 0 && p->gravity[2] != 0.0) return LBM_EINVAL;
  return LBM_OK;
}

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// LBM_NPHASE_KERNEL: "generic" selects the generic tile kernels everywhere,
// "pipelined" the TMA kernels at every size; else the rules below.
bool kernel_env(const char *name) {
  const char *v = getenv("LBM_NPHASE_KERNEL");
  return v && strcmp(v, name) == 0;
}
bool tma_allowed() { return !kernel_env("generic"); }

struct Layout {
  size_t h0, hm, gm, phi_prev, u_prev, stage, red, red_out, err, total;
};

// Lattice shape: moving directions Q - 1 and velocity components D.
int moving_dirs(const lbm_nphase_params *p) { return p->lattice == 1 ? 14 : 8; }
int dims(const lbm_nphase_params *p) { return p->lattice == 1 ? 3 : 2; }
int depth(const lbm_nphase_params *p) { return p->lattice == 1 ? p->nz : 1; }
// Planes of the u(t-1) buffers: the D velocity components, and for the
// 16-bit forms p(t-1), which their g storage is relative to.
int uplanes(const lbm_nphase_params *p) {
  return dims(p) + (p->precision == LBM_MIX_BF16 || p->precision == LBM_MIX_FP16 ? 1 : 0);
}

// Row pitch of the state's planes: FP32 D2Q9 grids that the pipelined kernel
// serves have their rows padded to a multiple of 8 nodes for its TMA loads.
// The others stay dense: a padded row costs the generic kernel up to a quarter
// (33 x 40000, N = 5 172 -> 216 us per step) and a narrow grid its memory.
int pitch(const lbm_nphase_params *p, bool pad) {
  if (!pad || !tma_allowed() || p->lattice != 0 || p->precision != LBM_FP32 || p->grad_scheme != 0) return p->nx;
  for (int k = 1; k < p->N; ++k)
    if (p->rho[k] != p->rho[0]) return p->nx;
  if (!lbm::tma_pays(p->N, p->nx, p->ny) && !kernel_env("pipelined")) return p->nx;
  return (p->nx + 7) / 8 * 8;
}

Layout layout(const lbm_nphase_params *p, int px) {
  const size_t Vd = (size_t)p->nx * p->ny * depth(p);
  const size_t V = (size_t)px * p->ny * depth(p);
  const int NP = p->N - 1, QM = moving_dirs(p), D = dims(p), UP = uplanes(p);
  const size_t sT = p->precision == LBM_FP64 ? 8 : 4;
  const size_t sS = p->precision == LBM_FP64 ? 8 : (p->precision == LBM_FP32 ? 4 : 2);
  const size_t tiles = lbm::tiles_total(p->lattice, p->nx, p->ny, depth(p));
  Layout L;
  size_t off = 0;
  L.h0 = off;       off += 2 * align256(NP * V * sT);
  L.hm = off;       off += 2 * align256(NP * QM * V * sS);
  L.gm = off;       off += 2 * align256(QM * V * sS);
  L.phi_prev = off; off += 2 * align256(NP * V * sT);
  L.u_prev = off;   off += 2 * align256(UP * V * sT);
  L.stage = off;    off += align256((p->N + D) * Vd * 8);
  L.red = off;      off += align256(tiles * (p->N + 2) * 8);
  L.red_out = off;  off += align256(8 * 8);
  L.err = off;      off += align256(sizeof(int));
  L.total = off;
  return L;
}

bool is_device_ptr(const void *ptr) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, ptr) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

lbm_status cuda_fail(lbm_nphase_t *h, cudaError_t e) {
  h->cuda_err = (int)e;
  return LBM_ECUDA;
}

// cuTensorMapEncodeTiled from the driver, looked up through the runtime.
lbm::EncodeTiledFn tensor_map_encoder() {
  static lbm::EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                         cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (lbm::EncodeTiledFn)p;
    else
      cudaGetLastError();
  }
  return fn;
}

// Device error word: read and clear. Returns LBM_ETIMEOUT if a kernel's
// bounded wait gave up since the last check.
lbm_status check_err(lbm_nphase_t *h) {
  int v = 0;
  cudaError_t e = cudaMemcpyAsync(&v, h->g.err, sizeof(int),
                                  cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  if (v != 0) {
    cudaMemsetAsync(h->g.err, 0, sizeof(int), h->stream);
    h->unstable = true;
    return LBM_ETIMEOUT;
  }
  return LBM_OK;
}

}  // namespace

// --------------------------------------------------------------------------
// Deterministic second pass of the diagnostics reduction.
// --------------------------------------------------------------------------
__global__ void reduce_partials_kernel(const double *__restrict__ part,
                                       int nparts, int nvals,
                                       double *__restrict__ out) {
  __shared__ double s[256];
  const int t = threadIdx.x;
  for (int j = 0; j < nvals; ++j) {
    const bool is_max = j == nvals - 1;
    double v = is_max ? 0.0 : 0.0;
    for (int b = t; b < nparts; b += 256) {
      const double x = part[(size_t)b * nvals + j];
      v = is_max ? fmax(v, x) : v + x;
    }
    s[t] = v;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
      if (t < w) s[t] = is_max ? fmax(s[t], s[t + w]) : s[t] + s[t + w];
      __syncthreads();
    }
    if (t == 0) out[j] = s[0];
    __syncthreads();
  }
}

namespace lbm {

cudaError_t launch_tile(int prec, const Consts &k, const Grid &g, int cur,
                        int mode, const Outputs &o, bool nonunif, bool wall,
                        cudaStream_t s) {
  if (g.lattice == 1) {
    switch (prec) {
      case LBM_FP64: return launch_tile3_f64(k, g, cur, mode, o, nonunif, wall, s);
      case LBM_FP32: return launch_tile3_f32(k, g, cur, mode, o, nonunif, wall, s);
      case LBM_MIX_BF16: return launch_tile3_bf16(k, g, cur, mode, o, nonunif, wall, s);
      case LBM_MIX_FP16: return launch_tile3_f16(k, g, cur, mode, o, nonunif, wall, s);
    }
    return cudaErrorInvalidValue;
  }
  switch (prec) {
    case LBM_FP64: return launch_tile_f64(k, g, cur, mode, o, nonunif, wall, s);
    case LBM_FP32: return launch_tile_f32(k, g, cur, mode, o, nonunif, wall, s);
    case LBM_MIX_BF16: return launch_tile_bf16(k, g, cur, mode, o, nonunif, wall, s);
    case LBM_MIX_FP16: return launch_tile_f16(k, g, cur, mode, o, nonunif, wall, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_init(int prec, const Consts &k, const Grid &g, int cur,
                        const double *c, const double *u, double p0, bool wall,
                        cudaStream_t s) {
  if (g.lattice == 1) {
    switch (prec) {
      case LBM_FP64: return launch_init3_f64(k, g, cur, c, u, p0, wall, s);
      case LBM_FP32: return launch_init3_f32(k, g, cur, c, u, p0, wall, s);
      case LBM_MIX_BF16: return launch_init3_bf16(k, g, cur, c, u, p0, wall, s);
      case LBM_MIX_FP16: return launch_init3_f16(k, g, cur, c, u, p0, wall, s);
    }
    return cudaErrorInvalidValue;
  }
  switch (prec) {
    case LBM_FP64: return launch_init_f64(k, g, cur, c, u, p0, wall, s);
    case LBM_FP32: return launch_init_f32(k, g, cur, c, u, p0, wall, s);
    case LBM_MIX_BF16: return launch_init_bf16(k, g, cur, c, u, p0, wall, s);
    case LBM_MIX_FP16: return launch_init_f16(k, g, cur, c, u, p0, wall, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_reduce(const Grid &g, int nparts, int nvals, cudaStream_t s) {
  reduce_partials_kernel<<<1, 256, 0, s>>>(g.red, nparts, nvals, g.red_out);
  return cudaGetLastError();
}

}  // namespace lbm

// --------------------------------------------------------------------------
// Public API
// --------------------------------------------------------------------------
extern "C" {

const char *lbm_nphase_strerror(lbm_status s) {
  switch (s) {
    case LBM_OK: return "success";
    case LBM_EINVAL: return "invalid argument or parameter set";
    case LBM_ENOMEM: return "workspace too small";
    case LBM_ECUDA: return "CUDA error";
    case LBM_ETIMEOUT: return "bounded device wait timed out";
    case LBM_EUNSTABLE: return "non-finite mass or kinetic energy";
    case LBM_ESTATE: return "call not valid in the current handle state";
  }
  return "unknown status";
}

lbm_status lbm_nphase_derive(const lbm_nphase_params *p, lbm_nphase_model *out) {
  lbm_status st = validate(p);
  if (st != LBM_OK) return st;
  lbm_nphase_model m;
  memset(&m, 0, sizeof(m));
  const int N = p->N, n = N - 1;
  double smin = INFINITY;
  for (int k = 0; k < N; ++k)
    for (int l = k + 1; l < N; ++l) smin = fmin(smin, p->sigma[k][l]);
  m.beta = p->beta > 0.0 ? p->beta : sqrt(3.0 * sqrt(2.0) * smin * p->eta);
  // Eq. N14: unknowns lambda_ij (i <= j), one equation per pair k < l.
  int ui[10], uj[10], M = 0;
  for (int i = 0; i < n; ++i)
    for (int j = i; j < n; ++j) {
      ui[M] = i;
      uj[M] = j;
      ++M;
    }
  double A[10][10], b[10], x[10];
  int row = 0;
  const double rhs = 4.5 * p->eta * p->eta / (m.beta * m.beta);
  for (int k = 0; k < N; ++k)
    for (int l = k + 1; l < N; ++l) {
      for (int c = 0; c < M; ++c) {
        const double Li = Lcoef(p, ui[c], k, l), Lj = Lcoef(p, uj[c], k, l);
        A[row][c] = ui[c] == uj[c] ? Li * Li : 2.0 * Li * Lj;
      }
      b[row] = rhs * p->sigma[k][l] * p->sigma[k][l];
      ++row;
    }
  if (!householder_solve(M, A, b, x)) return LBM_EINVAL;
  for (int c = 0; c < M; ++c) {
    m.lambda[ui[c]][uj[c]] = x[c];
    m.lambda[uj[c]][ui[c]] = x[c];
  }
  double lam4[4][4] = {{0}};
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) lam4[i][j] = m.lambda[i][j];
  if (!cholesky_ok(n, lam4)) return LBM_EINVAL;
  sym_eig_range(n, lam4, &m.lambda_eig_min, &m.lambda_eig_max);
  m.Gamma = 0.0;
  for (int k = 0; k < N; ++k) m.Gamma += 1.0 / p->rho[k];
  for (int i = 0; i < n; ++i) m.a[i] = p->mobility[i] / (CS2 * (p->tau[i] - 0.5));
  m.nu = CS2 * (p->tau_g - 0.5);
  m.uniform_density = 1;
  for (int k = 1; k < N; ++k)
    if (p->rho[k] != p->rho[0]) m.uniform_density = 0;
  if (out) *out = m;
  return LBM_OK;
}

size_t lbm_nphase_workspace_bytes(const lbm_nphase_params *p) {
  return lbm::workspace_bytes(p, true);
}

lbm_status lbm_nphase_create(const lbm_nphase_params *p, void *ws,
                             size_t bytes, void *stream, lbm_nphase_t **out) {
  return lbm::create(p, ws, bytes, stream, true, out);
}

}  // extern "C"

size_t lbm::workspace_bytes(const lbm_nphase_params *p, bool pad) {
  return validate(p) == LBM_OK ? layout(p, pitch(p, pad)).total : 0;
}

lbm_status lbm::create(const lbm_nphase_params *p, void *ws, size_t bytes, void *stream, bool pad,
                       lbm_nphase_t **out) {
  if (!out) return LBM_EINVAL;
  *out = nullptr;
  lbm_nphase_model m;
  lbm_status st = lbm_nphase_derive(p, &m);
  if (st != LBM_OK) return st;
  if (!ws || ((uintptr_t)ws & 255u)) return LBM_EINVAL;
  // a workspace that holds the dense state only is served too (generic kernel)
  int px = pitch(p, pad);
  if (bytes < layout(p, px).total) px = p->nx;
  const Layout L = layout(p, px);
  if (bytes < L.total) return LBM_ENOMEM;
  lbm_nphase_t *h = new (std::nothrow) lbm_nphase_t;
  if (!h) return LBM_ENOMEM;
  memset((void *)h, 0, sizeof(*h));
  h->prm = *p;
  h->mdl = m;
  h->prec = p->precision;
  h->wall = p->wall_y != 0;
  h->nonunif = !m.uniform_density;
  h->stream = (cudaStream_t)stream;
  if (cudaGetDevice(&h->device) != cudaSuccess) {
    delete h;
    return LBM_ECUDA;
  }
  const int N = p->N, n = N - 1;
  Consts &k = h->k;
  memset(&k, 0, sizeof(k));
  k.N = N;
  k.NP = n;
  const double Gam = m.Gamma;
  double gam[5];
  for (int q = 0; q < N; ++q) gam[q] = 1.0 / p->rho[q];
  for (int i = 0; i < n; ++i) {
    for (int j = 0; j < n; ++j) k.lam[i][j] = m.lambda[i][j];
    k.a[i] = m.a[i];
    k.tau_inv[i] = 1.0 / p->tau[i];
    k.src[i] = 1.0 - 1.0 / (2.0 * p->tau[i]);
    k.off[i] = 0.5 * (p->rho[i] - p->rho[n]);
    k.mul[i] = 0.5 * (p->rho[i] + p->rho[n]);
    k.K[i] = 1.0 - N * gam[i] / Gam;
    k.kap[i] = k.K[i] * k.mul[i];
    k.kmob[i] = k.kap[i] * p->mobility[i];
  }
  for (int q = 0; q < N; ++q) {
    k.c0[q] = gam[q] / Gam;
    for (int j = 0; j < n; ++j)
      k.Q[q][j] = (q == j ? gam[q] : 0.0) - gam[q] * gam[j] / Gam;
    k.rho_t[q] = p->rho[q];
  }
  k.bulk = m.beta * m.beta / (p->eta * p->eta);
  k.tg_inv = 1.0 / p->tau_g;
  k.ffac = 1.0 - 1.0 / (2.0 * p->tau_g);
  k.jfac = 1.0 / (p->tau_g - 0.5);
  k.grav[0] = p->gravity[0];
  k.grav[1] = p->gravity[1];
  k.grav[2] = p->gravity[2];
  k.rho_base = N / Gam;
  // 16-bit storage: h_k / w_k and g_k / w_k are O(1e-4 .. 1e-1) for the
  // model's parameter ranges; 2^12 keeps them in FP16's normal range.
  k.sh = 4096.0;
  k.sg = 4096.0;
  Grid &g = h->g;
  g.nx = p->nx;
  g.ny = p->ny;
  g.nz = depth(p);
  g.lattice = p->lattice;
  g.px = px;
  g.V = (size_t)g.px * p->ny * g.nz;
  char *base = (char *)ws;
  const size_t sT = h->prec == LBM_FP64 ? 8 : 4;
  const size_t sS = h->prec == LBM_FP64 ? 8 : (h->prec == LBM_FP32 ? 4 : 2);
  const int QM = moving_dirs(p);
  const size_t h0b = align256(n * g.V * sT), hmb = align256(n * QM * g.V * sS),
               gmb = align256(QM * g.V * sS);
  for (int b = 0; b < 2; ++b) {
    g.h0[b] = base + L.h0 + b * h0b;
    g.hm[b] = base + L.hm + b * hmb;
    g.gm[b] = base + L.gm + b * gmb;
  }
  const size_t ppb = align256(n * g.V * sT);
  g.phi_prev[0] = base + L.phi_prev;
  g.phi_prev[1] = base + L.phi_prev + ppb;
  const size_t upb = align256((size_t)uplanes(p) * g.V * sT);
  g.u_prev[0] = base + L.u_prev;
  g.u_prev[1] = base + L.u_prev + upb;
  h->stage = (double *)(base + L.stage);
  g.scratch = h->stage;
  g.red = (double *)(base + L.red);
  g.red_out = (double *)(base + L.red_out);
  g.err = (int *)(base + L.err);
  g.grad_scheme = p->grad_scheme;
  g.use_tma = false;
  g.step64 = tma_allowed() && h->prec == LBM_FP64 && p->lattice == 0;
  // these kernels address a plane's nodes with 32-bit byte offsets
  g.split3 = tma_allowed() && p->lattice == 1 &&
             (size_t)p->nx * p->ny * sT < ((size_t)1 << 32);
  g.march3 = g.split3 && !h->nonunif;
  g.ring_warps = tma_allowed();
  g.tma_all = kernel_env("pipelined");
  g.tma3 = g.march3 && h->prec == LBM_FP32 &&
           lbm::encode_tma3_f32(k, g, tensor_map_encoder());
  if (tma_allowed() && !h->nonunif && p->grad_scheme == 0 && p->lattice == 0) {
    lbm::EncodeTiledFn enc = tensor_map_encoder();
    switch (h->prec) {
      case LBM_FP32: g.use_tma = lbm::encode_tma_f32(k, g, enc); break;
      case LBM_MIX_BF16: g.use_tma = lbm::encode_tma_bf16(k, g, enc); break;
      case LBM_MIX_FP16: g.use_tma = lbm::encode_tma_f16(k, g, enc); break;
      default: break;
    }
  }
  *out = h;
  return LBM_OK;
}

extern "C" {

lbm_status lbm_nphase_init(lbm_nphase_t *h, const double *c, const double *u,
                           double p0) {
  return lbm::init_at(h, c, u, p0, 0);
}

}  // extern "C"

lbm_status lbm::init_at(lbm_nphase_t *h, const double *c, const double *u,
                        double p0, int cur) {
  if (!h || !c || !isfinite(p0) || (cur != 0 && cur != 1)) return LBM_EINVAL;
  const size_t V = (size_t)h->g.nx * h->g.ny * h->g.nz;
  const int N = h->prm.N;
  const double *dc = c, *du = u;
  cudaError_t e;
  if (!is_device_ptr(c)) {
    e = cudaMemcpyAsync(h->stage, c, N * V * sizeof(double),
                        cudaMemcpyHostToDevice, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e);
    dc = h->stage;
  }
  if (u && !is_device_ptr(u)) {
    e = cudaMemcpyAsync(h->stage + N * V, u, dims(&h->prm) * V * sizeof(double),
                        cudaMemcpyHostToDevice, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e);
    du = h->stage + N * V;
  }
  e = cudaMemsetAsync(h->g.err, 0, sizeof(int), h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  e = lbm::launch_init(h->prec, h->k, h->g, cur, dc, du, p0, h->wall, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  h->cur = cur;
  h->steps = 0;
  h->initialized = true;
  h->unstable = false;
  return LBM_OK;
}

extern "C" {

static cudaError_t step_once(lbm_nphase_t *h, cudaStream_t s, int cur) {
  const Outputs none = {nullptr, nullptr, nullptr, nullptr, nullptr};
  return lbm::launch_tile(h->prec, h->k, h->g, cur, lbm::MODE_STEP, none,
                          h->nonunif, h->wall, s);
}

// Steps per graph: a pair, and a chain for long runs. Back to back, graphs
// start at multiples of about 2 us on GB300, kernels inside one graph follow
// each other at once (0.55 us for empty ones), so a chain saves 1 to 1.6 us per
// step (pairs / chain: FP32 64^2 N = 3 4.11 / 3.02, 512^2 N = 5 21.5 / 20.1,
// 2048^2 268.2 / 266.7; chains of 8, 16, 64 within 2% of 32). Its capture and
// instantiation take about 100 us, so it is built once a handle has run, or is
// about to run, kChainPays steps from the same buffer.
constexpr int kChainPays = 128;
constexpr int kChain[2] = {2, 32};

// kChain[l] steps from buffer p (an even number: back to p) as a graph.
static cudaError_t capture_steps(lbm_nphase_t *h, int l, int p) {
  cudaError_t e = cudaSuccess;
  if (!h->cap) e = cudaStreamCreateWithFlags(&h->cap, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaStreamBeginCapture(h->cap, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return e;
  cudaGraph_t graph = nullptr;
  cudaError_t es = cudaSuccess;
  for (int t = 0; t < kChain[l] && es == cudaSuccess; ++t) es = step_once(h, h->cap, p ^ (t & 1));
  e = cudaStreamEndCapture(h->cap, &graph);
  if (e == cudaSuccess) e = es;
  if (e == cudaSuccess) e = cudaGraphInstantiate(&h->gexec[l][p], graph, 0);
  if (graph) cudaGraphDestroy(graph);
  return e;
}

// The same, as a part of lbm_nphase_step that a caller does not see: in relaxed
// mode, so that a capture under way on another stream, of this thread or of
// another one, stays valid.
static cudaError_t build_step_graph(lbm_nphase_t *h, int l, int p) {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  cudaThreadExchangeStreamCaptureMode(&mode);
  const cudaError_t e = capture_steps(h, l, p);
  cudaThreadExchangeStreamCaptureMode(&mode);
  return e;
}

// Whether a chain from the current buffer is there, built now if `left` steps
// repay it. Not while the caller captures the handle's stream: such calls
// replay pairs.
static bool have_chain(lbm_nphase_t *h, int64_t left) {
  if (h->gexec[1][h->cur]) return true;
  if (h->paired[h->cur] + left < kChainPays) return false;
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (h->no_chain || cudaStreamIsCapturing(h->stream, &st) != cudaSuccess ||
      st != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return false;
  }
  if (build_step_graph(h, 1, h->cur) == cudaSuccess) return true;
  cudaGetLastError();
  h->no_chain = true;
  return false;
}

lbm_status lbm_nphase_step(lbm_nphase_t *h, int64_t nsteps) {
  if (!h || nsteps < 0) return LBM_EINVAL;
  if (!h->initialized || h->unstable) return LBM_ESTATE;
  int64_t t = 0;
  if (nsteps >= 4 && !h->gexec[0][0]) {
    // two steps launched directly first: the launchers' one-time setup
    // (shared-memory attributes, occupancy) then runs outside the capture, and
    // runs of even length start from the same buffer in the first call as later
    cudaError_t e = cudaSuccess;
    for (; t < 2; ++t) {
      e = step_once(h, h->stream, h->cur);
      if (e != cudaSuccess) return cuda_fail(h, e);
      h->cur ^= 1;
      ++h->steps;
    }
    for (int p = 0; p < 2 && e == cudaSuccess; ++p) e = build_step_graph(h, 0, p);
    if (e != cudaSuccess) return cuda_fail(h, e);
  }
  if (h->gexec[0][0])
    for (int l = 1; l >= 0; --l)
      for (; t + kChain[l] <= nsteps && (l == 0 || have_chain(h, nsteps - t));
           t += kChain[l]) {
        cudaError_t e = cudaGraphLaunch(h->gexec[l][h->cur], h->stream);
        if (e != cudaSuccess) return cuda_fail(h, e);
        h->steps += kChain[l];
        if (l == 0) h->paired[h->cur] += kChain[l];
      }
  for (; t < nsteps; ++t) {
    cudaError_t e = step_once(h, h->stream, h->cur);
    if (e != cudaSuccess) return cuda_fail(h, e);
    h->cur ^= 1;
    ++h->steps;
  }
  return LBM_OK;
}

// --------------------------------------------------------------------------
// Checkpoint / resume: the state at the current time as one blob.
// --------------------------------------------------------------------------
namespace {
struct StateHeader {
  char magic[8];  // "LBMNPHS2"
  int32_t N, nx, ny, precision, wall_y, grad_scheme;
  int64_t steps;
  uint64_t payload;  // bytes after the header
  int32_t nz, lattice;
  uint8_t pad[8];
};
static_assert(sizeof(StateHeader) == 64, "state header");

struct Part {
  void *dev;
  size_t planes, es;  // planes of ny nz rows of nx values of es bytes
};

int state_parts(const lbm_nphase_t *h, Part out[5]) {
  const size_t n = h->prm.N - 1;
  const size_t sT = h->prec == LBM_FP64 ? 8 : 4;
  const size_t sS = h->prec == LBM_FP64 ? 8 : (h->prec == LBM_FP32 ? 4 : 2);
  const int c = h->cur;
  const size_t QM = moving_dirs(&h->prm), UP = uplanes(&h->prm);
  out[0] = {h->g.h0[c], n, sT};
  out[1] = {h->g.hm[c], n * QM, sS};
  out[2] = {h->g.gm[c], QM, sS};
  out[3] = {h->g.phi_prev[c], n, sT};
  out[4] = {h->g.u_prev[c], UP, sT};
  return 5;
}

// n dense values (rows of nx) to or from rows of pitch px, value by value in
// dense order, eight loads of a thread in flight. n < 2^32.
__global__ void __launch_bounds__(256) copy_rows_kernel(float *dense, float *rows, unsigned nx,
                                                        unsigned px, unsigned n, bool pack) {
  const size_t base = (size_t)blockIdx.x * 2048 + threadIdx.x;
  float v[8];
  size_t at[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const size_t i = base + k * 256;
    const unsigned r = (unsigned)i / nx;
    at[k] = (size_t)r * px + ((unsigned)i - r * nx);
    if (i < n) v[k] = pack ? rows[at[k]] : dense[i];
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const size_t i = base + k * 256;
    if (i < n) (pack ? dense[i] : rows[at[k]]) = v[k];
  }
}

size_t part_bytes(const lbm_nphase_t *h, const Part &p) {
  return p.planes * h->g.nx * h->g.ny * h->g.nz * p.es;
}

// Copies a part to or from the blob's dense rows. Padded rows (FP32) are packed
// and unpacked by a kernel, through the staging area for a blob in host memory:
// as a 2-D copy, row by row, set_state took up to 40 times as long (from host
// memory, us: 101 x 5000, N = 3 4906 -> 454, 1501 x 997, N = 4 2443 -> 1450), and
// get_state six times on short rows (874 -> 460; long ones go as fast as dense).
// Blobs that a kernel cannot address (another GPU's memory, addresses that are
// no multiple of 4) take the staging area too.
cudaError_t copy_part(const lbm_nphase_t *h, const Part &p, void *blob, bool to_blob,
                      cudaMemcpyKind kind) {
  const size_t nx = h->g.nx, px = h->g.px;
  if (nx == px)
    return to_blob ? cudaMemcpyAsync(blob, p.dev, part_bytes(h, p), kind, h->stream)
                   : cudaMemcpyAsync(p.dev, blob, part_bytes(h, p), kind, h->stream);
  const size_t rows = p.planes * h->g.ny * h->g.nz;
  if (kind == cudaMemcpyDeviceToHost && nx >= 512)
    return cudaMemcpy2DAsync(blob, nx * 4, p.dev, px * 4, nx * 4, rows, kind, h->stream);
  const size_t Vd = nx * h->g.ny * h->g.nz;
  cudaPointerAttributes at;
  bool dev = false;
  if (((uintptr_t)blob & 3u) == 0 && cudaPointerGetAttributes(&at, blob) == cudaSuccess)
    dev = at.type == cudaMemoryTypeDevice && at.device == h->device;
  cudaGetLastError();
  // rows at a time: what the staging area holds, and fewer than 2^31 values
  size_t fit = dev ? rows : (h->prm.N + dims(&h->prm)) * Vd * 8 / (nx * 4);
  if (fit > ((size_t)1 << 31) / px) fit = ((size_t)1 << 31) / px;
  cudaError_t e = cudaSuccess;
  for (size_t r = 0; r < rows && e == cudaSuccess; r += fit) {
    const size_t n = (rows - r < fit ? rows - r : fit) * nx;
    float *state = (float *)p.dev + r * px, *user = (float *)blob + r * nx;
    float *dense = dev ? user : (float *)h->stage;
    if (!dev && !to_blob) e = cudaMemcpyAsync(dense, user, n * 4, kind, h->stream);
    if (e != cudaSuccess) return e;
    copy_rows_kernel<<<(unsigned)((n + 2047) / 2048), 256, 0, h->stream>>>(
        dense, state, (unsigned)nx, (unsigned)px, (unsigned)n, to_blob);
    e = cudaGetLastError();
    if (e == cudaSuccess && !dev && to_blob) e = cudaMemcpyAsync(user, dense, n * 4, kind, h->stream);
  }
  return e;
}
}  // namespace

size_t lbm_nphase_state_bytes(const lbm_nphase_t *h) {
  if (!h) return 0;
  Part parts[5];
  size_t b = sizeof(StateHeader);
  const int np = state_parts(h, parts);
  for (int i = 0; i < np; ++i) b += part_bytes(h, parts[i]);
  return b;
}

lbm_status lbm_nphase_get_state(lbm_nphase_t *h, void *dst, size_t bytes) {
  if (!h || !dst) return LBM_EINVAL;
  if (!h->initialized) return LBM_ESTATE;
  if (bytes < lbm_nphase_state_bytes(h)) return LBM_ENOMEM;
  StateHeader hd;
  memset(&hd, 0, sizeof(hd));
  memcpy(hd.magic, "LBMNPHS2", 8);
  hd.N = h->prm.N;
  hd.nx = h->prm.nx;
  hd.ny = h->prm.ny;
  hd.precision = h->prm.precision;
  hd.wall_y = h->prm.wall_y;
  hd.grad_scheme = h->prm.grad_scheme;
  hd.nz = depth(&h->prm);
  hd.lattice = h->prm.lattice;
  hd.steps = h->steps;
  hd.payload = lbm_nphase_state_bytes(h) - sizeof(hd);
  const bool dev = is_device_ptr(dst);
  cudaError_t e = cudaMemcpyAsync(dst, &hd, sizeof(hd),
                                  dev ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost,
                                  h->stream);
  Part parts[5];
  char *p = (char *)dst + sizeof(hd);
  const int np = state_parts(h, parts);
  for (int i = 0; i < np && e == cudaSuccess; ++i) {
    e = copy_part(h, parts[i], p, true, dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost);
    p += part_bytes(h, parts[i]);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  return LBM_OK;
}

lbm_status lbm_nphase_set_state(lbm_nphase_t *h, const void *src, size_t bytes) {
  if (!h || !src) return LBM_EINVAL;
  if (bytes < lbm_nphase_state_bytes(h)) return LBM_EINVAL;
  const bool dev = is_device_ptr(src);
  StateHeader hd;
  cudaError_t e = cudaMemcpy(&hd, src, sizeof(hd),
                             dev ? cudaMemcpyDeviceToHost : cudaMemcpyHostToHost);
  if (e != cudaSuccess) return cuda_fail(h, e);
  if (memcmp(hd.magic, "LBMNPHS2", 8) != 0 || hd.N != h->prm.N ||
      hd.nx != h->prm.nx || hd.ny != h->prm.ny || hd.nz != depth(&h->prm) ||
      hd.lattice != h->prm.lattice ||
      hd.precision != h->prm.precision || hd.wall_y != h->prm.wall_y ||
      hd.grad_scheme != h->prm.grad_scheme ||
      hd.payload != lbm_nphase_state_bytes(h) - sizeof(hd))
    return LBM_EINVAL;
  h->cur = 0;
  Part parts[5];
  char *p = (char *)src + sizeof(hd);
  const int np = state_parts(h, parts);
  for (int i = 0; i < np && e == cudaSuccess; ++i) {
    e = copy_part(h, parts[i], p, false, dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice);
    p += part_bytes(h, parts[i]);
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(h->g.err, 0, sizeof(int), h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  h->steps = hd.steps;
  h->initialized = true;
  h->unstable = false;
  return LBM_OK;
}

lbm_status lbm_nphase_moments(lbm_nphase_t *h, double *phi, double *c,
                              double *u, double *p, double *rho) {
  if (!h) return LBM_EINVAL;
  if (!h->initialized) return LBM_ESTATE;
  const size_t V = (size_t)h->g.nx * h->g.ny * h->g.nz;
  const int N = h->prm.N;
  double *ptr[5] = {phi, c, u, p, rho};
  const int nf[5] = {N - 1, N, dims(&h->prm), 1, 1};
  Outputs dev = {nullptr, nullptr, nullptr, nullptr, nullptr};
  double **dslot[5] = {&dev.phi, &dev.c, &dev.u, &dev.p, &dev.rho};
  bool any_dev = false, any_host = false;
  for (int f = 0; f < 5; ++f) {
    if (!ptr[f]) continue;
    if (is_device_ptr(ptr[f])) {
      *dslot[f] = ptr[f];
      any_dev = true;
    } else {
      any_host = true;
    }
  }
  cudaError_t e;
  if (any_dev) {
    e = lbm::launch_tile(h->prec, h->k, h->g, h->cur, lbm::MODE_MOMENTS, dev,
                         h->nonunif, h->wall, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e);
  }
  if (any_host) {
    for (int f = 0; f < 5; ++f) {
      if (!ptr[f] || is_device_ptr(ptr[f])) continue;
      Outputs one = {nullptr, nullptr, nullptr, nullptr, nullptr};
      double **slot[5] = {&one.phi, &one.c, &one.u, &one.p, &one.rho};
      *slot[f] = h->stage;
      e = lbm::launch_tile(h->prec, h->k, h->g, h->cur, lbm::MODE_MOMENTS, one,
                           h->nonunif, h->wall, h->stream);
      if (e != cudaSuccess) return cuda_fail(h, e);
      e = cudaMemcpyAsync(ptr[f], h->stage, nf[f] * V * sizeof(double),
                          cudaMemcpyDeviceToHost, h->stream);
      if (e != cudaSuccess) return cuda_fail(h, e);
      e = cudaStreamSynchronize(h->stream);
      if (e != cudaSuccess) return cuda_fail(h, e);
    }
  }
  return check_err(h);  // synchronises
}

lbm_status lbm_nphase_diagnostics(lbm_nphase_t *h, double *mass, double *ke,
                                  double *umax) {
  if (!h) return LBM_EINVAL;
  if (!h->initialized) return LBM_ESTATE;
  const int N = h->prm.N;
  const Outputs none = {nullptr, nullptr, nullptr, nullptr, nullptr};
  cudaError_t e = lbm::launch_tile(h->prec, h->k, h->g, h->cur, lbm::MODE_DIAG,
                                   none, h->nonunif, h->wall, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  const int nparts = (int)lbm::tiles_total(h->g.lattice, h->g.nx, h->g.ny, h->g.nz);
  e = lbm::launch_reduce(h->g, nparts, N + 2, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  double r[LBM_MAX_N + 2];
  e = cudaMemcpyAsync(r, h->g.red_out, (N + 2) * sizeof(double),
                      cudaMemcpyDeviceToHost, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  bool ok = true;
  for (int j = 0; j < N + 2; ++j) ok = ok && isfinite(r[j]);
  if (mass)
    for (int k = 0; k < N; ++k) mass[k] = r[k];
  if (ke) *ke = r[N];
  if (umax) *umax = r[N + 1];
  const lbm_status es = check_err(h);
  if (es != LBM_OK) return es;
  if (!ok) {
    h->unstable = true;
    return LBM_EUNSTABLE;
  }
  return LBM_OK;
}

int lbm_nphase_uses_pipelined_kernel(const lbm_nphase_t *h) {
  if (!h) return 0;
  return h->g.use_tma ? 1 : (h->g.tma3 ? 3 : (h->g.march3 ? 2 : 0));
}

const char *lbm_nphase_step_kernels(const lbm_nphase_t *h) {
  if (!h) return "";
  switch (lbm::step_path(h->prec, h->prm.N, h->g, h->nonunif)) {
    case lbm::STEP_TILE: return "tile_kernel";
    case lbm::STEP_TILE_RING: return "tile_kernel (ring warps)";
    case lbm::STEP_TMA: return "tile_kernel_tma";
    case lbm::STEP_FP64: return "step64_kernel";
    case lbm::STEP_FP64_SPLIT: return "pot64_kernel + coll64_kernel";
    case lbm::STEP_TILE3: return "tile3_kernel";
    case lbm::STEP_SPLIT3: return "phi3_kernel + step3_kernel";
    case lbm::STEP_SPLIT3_NU: return "phi3_kernel + pot3_kernel + step3_kernel";
    case lbm::STEP_MARCH3: return "march3_tma_kernel";
  }
  return "";
}

int64_t lbm_nphase_steps_taken(const lbm_nphase_t *h) { return h ? h->steps : 0; }

int lbm_nphase_cuda_error(const lbm_nphase_t *h) { return h ? h->cuda_err : 0; }

lbm_status lbm_nphase_destroy(lbm_nphase_t *h) {
  if (!h) return LBM_OK;
  for (int l = 0; l < 2; ++l)
    for (int p = 0; p < 2; ++p)
      if (h->gexec[l][p]) cudaGraphExecDestroy(h->gexec[l][p]);
  if (h->cap) cudaStreamDestroy(h->cap);
  delete h;
  return LBM_OK;
}

}  // extern "C"

// --------------------------------------------------------------------------
// Diagnostics without caller scratch: the per-CTA partials and the reduced
// values live in a file-scope device array instead of the handle workspace.
// --------------------------------------------------------------------------
#include <mutex>

// Largest number of diagnostics partials (one per 32 x 8 tile) the static
// array holds: 16384 tiles, e.g. a 2048 x 2048 grid. Slot width 8 doubles
// (N + 2 <= 7 values), plus 8 doubles for the reduced result: 1 MiB + 64 B,
// held by every GPU that loads the library until the process exits.
#define LBM_STATIC_MAX_PARTIALS 16384
#define LBM_STATIC_SLOT 8
static __device__ __align__(256) double
    lbm_static_scratch[LBM_STATIC_MAX_PARTIALS * LBM_STATIC_SLOT + LBM_STATIC_SLOT];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
double *g_static_ptr[kMaxDevices];  // device address of the array, per device
}  // namespace

extern "C" lbm_status lbm_nphase_diagnostics_static(lbm_nphase_t *h,
                                                    double *mass, double *ke,
                                                    double *umax) {
  if (!h) return LBM_EINVAL;
  if (!h->initialized) return LBM_ESTATE;
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(h, e);
  if (dev != h->device || dev < 0 || dev >= kMaxDevices) return LBM_EINVAL;
  const size_t nparts_z =
      lbm::tiles_total(h->g.lattice, h->g.nx, h->g.ny, h->g.nz);
  if (nparts_z > LBM_STATIC_MAX_PARTIALS) return LBM_EINVAL;
  const int nparts = (int)nparts_z;
  double *base;
  {
    // First call on a device: look up the array's device address with that
    // device current. The name is only a host-side stand-in for it.
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
      void *p = nullptr;
      e = cudaGetSymbolAddress(&p, lbm_static_scratch);
      if (e != cudaSuccess) return cuda_fail(h, e);
      g_static_ptr[dev] = (double *)p;
    }
    base = g_static_ptr[dev];
  }
  const int N = h->prm.N;
  // Every partial slot the reduction reads is written by its CTA first and
  // the result slot is overwritten, so nothing needs clearing between calls.
  lbm::Grid g = h->g;
  g.red = base;
  g.red_out = base + (size_t)LBM_STATIC_MAX_PARTIALS * LBM_STATIC_SLOT;
  const Outputs none = {nullptr, nullptr, nullptr, nullptr, nullptr};
  e = lbm::launch_tile(h->prec, h->k, g, h->cur, lbm::MODE_DIAG, none,
                       h->nonunif, h->wall, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  e = lbm::launch_reduce(g, nparts, N + 2, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  double r[LBM_MAX_N + 2];
  e = cudaMemcpyAsync(r, g.red_out, (N + 2) * sizeof(double),
                      cudaMemcpyDeviceToHost, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e);
  bool ok = true;
  for (int j = 0; j < N + 2; ++j) ok = ok && isfinite(r[j]);
  if (mass)
    for (int k = 0; k < N; ++k) mass[k] = r[k];
  if (ke) *ke = r[N];
  if (umax) *umax = r[N + 1];
  // A bounded device wait that gave up (in a step kernel or here) is
  // reported before the finite check, as lbm_nphase_diagnostics does.
  const lbm_status es = check_err(h);
  if (es != LBM_OK) return es;
  if (!ok) {
    h->unstable = true;
    return LBM_EUNSTABLE;
  }
  return LBM_OK;
}
