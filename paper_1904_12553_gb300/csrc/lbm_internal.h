// Internal interface between the C-ABI host code and the per-precision CUDA
// kernel translation units. Not part of the public API.
#pragma once

#include <cuda.h>  // CUtensorMap and its enums (types only; no driver link)
#include <cuda_runtime.h>
#include <stddef.h>

#include "lbm_nphase.h"

namespace lbm {

constexpr int BX = 32;  // tile width (one warp along x)
constexpr int BY = 8;   // tile height
constexpr int NT = BX * BY;

enum Mode { MODE_STEP = 0, MODE_MOMENTS = 1, MODE_DIAG = 2 };

// Model constants in FP64; each precision unit converts them to its type.
// Index conventions: i, j over the N-1 order parameters; k over N phases.
struct Consts {
  int N, NP;
  double lam[4][4];    // lambda_ij (Eq. N14)
  double bulk;         // beta^2 / eta^2
  double a[4];         // a_i (Eq. N30)
  double tau_inv[4];   // 1 / tau_i
  double src[4];       // 1 - 1/(2 tau_i) (Eq. N26)
  double tg_inv;       // 1 / tau_g
  double ffac;         // 1 - 1/(2 tau_g) (Eq. 24)
  double jfac;         // 1 / (tau_g - 1/2) (Eq. N20_1)
  double grav[3];      // G = rho * grav
  double off[4], mul[4];  // varphi_j = off_j + mul_j phi_j (Eq. N12)
  double c0[5];        // gamma~_k / Gamma (Eq. N18)
  double Q[5][4];      // gamma~_k delta_kj - gamma~_k gamma~_j / Gamma
  double rho_base;     // N / Gamma (Eq. N29)
  double K[4];         // 1 - N gamma~_i / Gamma
  double kap[4];       // K_i mul_i: grad rho = sum kap_i grad phi_i
  double kmob[4];      // kap_i m_i: J~ = -sum kmob_i grad C_i
  double rho_t[5];     // rho~_k (initialisation)
  double sh, sg;       // 16-bit storage scales of h_k / w_k and g_k / w_k
};

// TMA descriptors of one state buffer for the pipelined step kernel.
struct TmaMaps {
  CUtensorMap hm, h0, pp, gm, up;
  // FP32 pipelined kernel: the halo column and row that wrap around a
  // periodic grid (boxes of 16 bytes x the box height, and one row x the
  // box width, of the h, d_0 and phi(t-1) arrays)
  CUtensorMap hmx, h0x, ppx, hmy, h0y, ppy;
};

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType,
                                  cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

// Device state of one grid. Buffers [0] and [1] alternate every step.
struct Grid {
  int nx, ny, nz;   // nz = 1 for D2Q9
  int lattice;      // 0 D2Q9, 1 D3Q15
  int px;           // row pitch in nodes (nx, or rounded up to 8: see pitch())
  size_t V;         // plane stride px * ny * nz
  void *h0[2];      // rest slots: h^i_0 (FP64) or h^i_0 - phi_i(t-1): [N-1][V]
  void *hm[2];      // moving populations h^i_k, k = 1..8: [N-1][8][V]
  void *gm[2];      // NS populations g_k, k = 1..8: [8][V]
  void *phi_prev[2];  // phi_i(t-1): [N-1][V]
  void *u_prev[2];  // u(t-1): [D][V] (16-bit forms: [D + 1][V], p(t-1) last),
                    // ping-pong like phi_prev
  double *red;      // per-block partial sums of the diagnostics
  double *red_out;  // N + 2 reduced diagnostics
  int *err;         // device error word (1: a bounded wait gave up)
  double *scratch;  // FP64 staging of host inputs and outputs ([N + D][V]);
                    // initialisation keeps phi_i there ([N-1][V])
  int grad_scheme;  // 0: central (Eq. N31a), 1: mixed (Eq. N40)
  bool use_tma;     // pipelined kernel prepared (tma[] encoded): see step_path
  bool step64;      // D2Q9 step by the FP64 kernels (lbm_step64.cuh)
  bool split3;      // D3Q15 step by the split or z-marching kernels
  bool march3;      // ... with equal densities
  bool tma3;        // ... FP32 z-marching kernel prepared (tma[] holds 4-D maps)
  bool ring_warps;  // halo-ring warps on grids of one wave (not "generic")
  bool tma_all;     // TMA kernels at every size (LBM_NPHASE_KERNEL=pipelined)
  TmaMaps tma[2];   // its descriptors, input buffer 0 or 1
};

struct Outputs {
  double *phi, *c, *u, *p, *rho;
};

// Launchers, one set per precision (lbm_fp64.cu, lbm_fp32.cu, lbm_mixed.cu).
// prec is an lbm_precision value; `cur` selects the input buffer.
cudaError_t launch_tile(int prec, const Consts &k, const Grid &g, int cur,
                        int mode, const Outputs &o, bool nonunif, bool wall,
                        cudaStream_t s);
cudaError_t launch_init(int prec, const Consts &k, const Grid &g, int cur,
                        const double *c, const double *u, double p0, bool wall,
                        cudaStream_t s);
cudaError_t launch_reduce(const Grid &g, int nparts, int nvals, cudaStream_t s);

#define LBM_DECLARE_PREC(SUFFIX)                                              \
  cudaError_t launch_tile_##SUFFIX(const Consts &, const Grid &, int, int,    \
                                   const Outputs &, bool, bool, cudaStream_t);\
  cudaError_t launch_init_##SUFFIX(const Consts &, const Grid &, int,         \
                                   const double *, const double *, double,    \
                                   bool, cudaStream_t);                       \
  bool encode_tma_##SUFFIX(const Consts &, Grid &, EncodeTiledFn);           \
  bool encode_tma3_##SUFFIX(const Consts &, Grid &, EncodeTiledFn);          \
  cudaError_t launch_tile3_##SUFFIX(const Consts &, const Grid &, int, int,   \
                                    const Outputs &, bool, bool, cudaStream_t);\
  cudaError_t launch_init3_##SUFFIX(const Consts &, const Grid &, int,        \
                                    const double *, const double *, double,   \
                                    bool, cudaStream_t);
LBM_DECLARE_PREC(f64)
LBM_DECLARE_PREC(f32)
LBM_DECLARE_PREC(bf16)
LBM_DECLARE_PREC(f16)
#undef LBM_DECLARE_PREC

inline int tiles_x(int nx) { return (nx + BX - 1) / BX; }
inline int tiles_y(int ny) { return (ny + BY - 1) / BY; }
// D3Q15 tiles: 32 x 4 x 2 nodes
inline int tiles3_x(int nx) { return (nx + 31) / 32; }
inline int tiles3_y(int ny) { return (ny + 3) / 4; }
inline int tiles3_z(int nz) { return (nz + 1) / 2; }
inline long long tiles_of(int nx, int ny) { return (long long)tiles_x(nx) * tiles_y(ny); }
// FP32 D2Q9 grids (equal densities, central scheme): the pipelined kernel, or
// the generic one, whose CTAs start their loads at once and overlap on an SM
// where the pipelined kernel's single CTA fetches its tensor maps and fills its
// stages first. The line lies at six to eight waves of tiles on 152 SMs, by
// phases (pipelined / generic, us per step, chains of steps):
//   N = 2: 513^2 (1105 tiles) 9.6 / 9.0, 640 x 512 (1280) 10.0 / 10.8
//   N = 3: 512 x 400 (800) 10.4 / 9.6, 512^2 (1024) 11.6 / 11.8
//   N = 4: 512^2 16.7 / 15.6, 640 x 480 (1200) 17.8 / 18.8
//   N = 5: 512 x 400 17.4 / 16.3, 512^2 20.0 / 21.6
// and 2048^2 109 / 135, 161 / 211, 221 / 260, 265 / 360 at N = 2..5. Tiles
// with idle lanes fill a whole stage all the same: grids up to 63 wide (57 x
// 40000, N = 5 267 / 244; 8 x 40000, N = 3 78 / 37) or with fewer than 60% of
// the lanes in use stay on the generic kernel; N = 4, whose pipelined step gains
// least, counts live lanes only (20001 x 12, 75% 19.8 / 15.2; 65 x 5000, 68% 29.7 /
// 26.5).
inline bool tma_pays(int N, int nx, int ny) {
  const long long t = tiles_of(nx, ny), nodes = (long long)nx * ny;
  if (N == 4) return nx >= 64 && nodes > 1140 * 256 && nodes * 100 >= t * 256 * 70;
  return nx >= 64 && t > (N == 2 ? 1216 : 912) && nodes * 100 >= t * 256 * 60;
}
// N = 3: three stages of 49 KB and one CTA per SM where the state is far beyond
// L2, else two and two CTAs (216 KB, which leave L1 little for the stores, but
// twice the warps). us per step, 3 x 1 / 2 x 2: 256 x 1600 (1600 tiles) 21.1 /
// 16.5, 768^2 (2304) 28.0 / 24.0, 1200 x 900 (4294) 55.1 / 48.4, 1501 x 997
// (5875) 61.8 / 65.0, 96 x 40000 163 / 190, 2048^2 161 / 206; narrow rows of
// whole 32 bytes keep two longer: 64 x 40000 115 / 107, 72 x 40000 168 / 147
// (73 x 40000 173 / 203). 2 x 1 and 4 x 1 are slower than both at 2048^2.
inline bool tma_three_stages(int nx, int ny) {
  return tiles_of(nx, ny) > 33 * 152 && (nx >= 96 || nx % 8 != 0);
}
// FP32 grids whose tiles are all resident at once, ring_ctas per SM, take the
// generic kernel with halo-ring warps (see there).
constexpr int ring_ctas(int NP, bool NU, bool G40) {
  return NP <= (NU && G40 ? 0 : NU || G40 ? 2 : 3) ? 2 : 1;
}
// Whether the TMA-staged z-marching kernel beats the split step: it reads h
// once, but needs columns enough to fill the GPU and few idle lanes in them.
// us per step, march / split, N = 3: 64^3 29.8 / 23.8, 96^3 86.5 / 87.2, 128^3
// 184 / 199, 160^3 329 / 384, 256^3 1290 / 1538, 40 x 200 x 120 (62% of the
// columns' lanes) 152 / 114; N = 2: 128^3 133 / 124, 192 x 192 x 200 401 / 424.
inline bool march3_pays(const Grid &g, int NP) {
  if (!g.tma3) return false;
  if (g.tma_all) return true;
  const long long cols = (long long)tiles_x(g.nx) * 32 * ((g.ny + 7) / 8) * 8;
  return g.V >= ((size_t)1 << (NP >= 2 ? 20 : 22)) && (long long)g.nx * g.ny * 5 >= cols * 4;
}
// The kernels of one step: what the launchers run and lbm_nphase_step_kernels
// reports.
enum StepPath {
  STEP_TILE,        // tile_kernel
  STEP_TILE_RING,   // ... with halo-ring warps
  STEP_TMA,         // tile_kernel_tma
  STEP_FP64,        // step64_kernel
  STEP_FP64_SPLIT,  // pot64_kernel, coll64_kernel
  STEP_TILE3,       // tile3_kernel
  STEP_SPLIT3,      // phi3_kernel, step3_kernel
  STEP_SPLIT3_NU,   // phi3_kernel, pot3_kernel, step3_kernel
  STEP_MARCH3       // march3_tma_kernel
};
inline StepPath step_path(int prec, int N, const Grid &g, bool nonunif) {
  const bool g40 = g.grad_scheme == 1;
  if (g.lattice == 1) {
    if (!g.split3) return STEP_TILE3;
    if (march3_pays(g, N - 1)) return STEP_MARCH3;
    return nonunif ? STEP_SPLIT3_NU : STEP_SPLIT3;
  }
  if (g.step64) return nonunif || g40 ? STEP_FP64_SPLIT : STEP_FP64;
  if (g.use_tma && (prec != LBM_FP32 || g.tma_all || tma_pays(N, g.nx, g.ny))) return STEP_TMA;
  if (prec == LBM_FP32 && g.ring_warps &&
      tiles_of(g.nx, g.ny) <= 152 * ring_ctas(N - 1, nonunif, g40))
    return STEP_TILE_RING;
  return STEP_TILE;
}
// CTAs of the generic step / moments / diagnostics kernel of a grid
inline size_t tiles_total(int lattice, int nx, int ny, int nz) {
  return lattice == 1 ? (size_t)tiles3_x(nx) * tiles3_y(ny) * tiles3_z(nz)
                      : (size_t)tiles_x(nx) * tiles_y(ny);
}

}  // namespace lbm

// One grid's handle (the opaque type of the C ABI).
struct lbm_nphase_t {
  lbm_nphase_params prm;
  lbm_nphase_model mdl;
  lbm::Consts k;
  lbm::Grid g;
  int prec;
  bool nonunif, wall;
  cudaStream_t stream;
  int device;
  double *stage;  // (N + 2) * V doubles: host <-> device staging
  int cur;        // buffer holding the state at the current time
  bool initialized, unstable;
  int64_t steps;
  int cuda_err;
  cudaStream_t cap;            // private stream for graph capture
  cudaGraphExec_t gexec[2][2]; // a pair, a chain of steps from buffer 0 / 1
  int64_t paired[2];           // steps replayed in pairs from buffer 0 / 1
  bool no_chain;               // the chain's capture failed: pairs only
};

namespace lbm {
// lbm_nphase_init with the start state written into buffer `cur` (0 or 1),
// so that grids stepped together keep the same buffer parity.
lbm_status init_at(lbm_nphase_t *h, const double *c, const double *u,
                   double p0, int cur);
// lbm_nphase_create, with rows padded to a multiple of 8 nodes where the
// pipelined kernels use that (single grids), or dense (the cases of a batch).
lbm_status create(const lbm_nphase_params *p, void *ws, size_t bytes, void *stream, bool pad,
                  lbm_nphase_t **out);
size_t workspace_bytes(const lbm_nphase_params *p, bool pad);
}  // namespace lbm
