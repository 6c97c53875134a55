// The D2Q9 time step in FP64. GB300 has two FP64 units per SM, each shared by
// two of its quarters: a warp issues one FP64 instruction per 64 cycles, an SM
// one per 16 at best, so the step is bound by the number of FP64 instructions
// per node, whatever else it does (memory runs at 17% of its rate beside it).
// These kernels are written for that number:
//  - every constant factor of the model is folded on the host (Cst64), the
//    stencil denominators into the coefficients that use them; with equal
//    densities rho and 1/rho are constants, and p, which the next step does
//    not need, is folded into A0 of the NS collision;
//  - opposite directions k, k' share their even and odd parts: with
//    E = w (A0 + (c.u) (B2 c.u + c.H)) and O = w (B1 c.u + C1 c.F),
//    g*_k = (1 - 1/tau) g_k + E + O and g*_k' = ... + E - O, and the same for
//    h^i; the diagonal directions' odd parts are sums of the axes';
//  - Eq. N40's gradient by antisymmetry: sum_k w_k c_k (6 z(x + c_k)
//    - z(x + 2 c_k)) / (4 c_s^2), two central differences;
//  - nothing is computed twice where the halo is wide: unequal densities and
//    Eq. N40 take two kernels, phi and C_i of every node to memory first
//    (pot64_kernel), then the collision from their stencils (coll64_kernel);
//    equal densities with the central scheme need phi on a ring of one node
//    only and take one kernel (step64_kernel);
//  - the form of the instructions: a DFMA of three vector registers takes 16
//    cycles of the SM, a DADD, a DMUL or a DFMA with an immediate, constant-
//    bank or uniform operand 19 (measured, streams of each from 8 and 12
//    warps). So sums and products are fused multiply-adds with 1 and 0, the
//    same values, and every constant is read from shared memory into
//    registers: 718 us -> 615 us per step at N = 5, 1024^2.
// The populations are read again for the collision (L1 and L2 hits) instead
// of held across the barrier: 110 registers, four CTAs of four warps.
// Measured, us per step, the generic tile kernel -> these: N = 5, 1024^2
// equal densities 1064 -> 615 (494 -> 360 FP64 instructions per node; 592 is
// the FP64 units' time for them); N = 3, 128^2 26.6 -> 11.3; N = 3, 150^2
// unequal densities with walls 35.9 -> 20.5; N = 5, 200 x 320 unequal
// densities, Eq. N40 156 -> 69. Largest error against a run in 80 bits (128^2, 150^2
// unequal densities, 200 x 320 Eq. N40, three starts each): u 11.8e-15 -> 8.9e-15
// of its largest value, p 12.8e-15 -> 9.6e-15, phi the same; both kernels differ
// from a 64-bit model by as much as that model from the 80-bit run.
#pragma once

namespace lbm {

// Constants of the model, staged to shared memory by each CTA.
struct Cst64 {
  double one, zero, two, four, six, half, quarter, w1, w5;
  double invN, bN;     // equal densities: 1/N, bulk/N
  double bulk;
  double lam6[4][4];   // lambda_ij / 6 (the Laplacian's denominator)
  double F0x, F0y, rinv, rinvh;  // equal densities: rho G, 1/rho, 1/(2 rho)
  double grx, gry;     // gravity (unequal densities)
  double gsc;          // denominator of the gradient: 1/12, Eq. N40 1/48
  // unequal densities: varphi_j = off_j + mul_j phi_j, gamma~, 1/Gamma,
  // C_i = cm_i (f_i - sum gamma~ f / Gamma) - ..., rho = r0 + sum kap phi,
  // kapg = kap gsc, kmobg = kap m gsc
  double off[4], mul[4], gam[5], invG, cm[4], r0, kap[4], kapg[4], kmobg[4];
  // NS collision; suffix a: times w of the axes (1/9), d: of the diagonals
  // (1/36). A0 = s18 sum g + s09 u.grad rho + ruu rho u.u - f3 u.(F + jh J),
  // H = D1 F + E1 grad rho + E2 J
  double keep_g, s18, s09, ruu, f3, jh;
  double B1a, B1d, B2a, B2d, C1a, C1d, D1a, E1a, E2a;
  // CH collisions
  double kA[4], kD[4], c1[4], c2[4], keep[4], ti[4], kR[4];
};

struct K64 {
  int nx, ny;
  size_t V;
  const double *h0, *hm, *gm, *pp, *u;
  double *h0o, *hmo, *gmo, *ppo, *uo;
  double *C;           // C_i of the two-kernel step, [N-1][V]
  Cst64 c;
};

inline K64 make_k64(const Consts &c, const Grid &g, int cur) {
  K64 ka;
  ka.nx = g.nx;
  ka.ny = g.ny;
  ka.V = g.V;
  ka.h0 = (const double *)g.h0[cur];
  ka.hm = (const double *)g.hm[cur];
  ka.gm = (const double *)g.gm[cur];
  ka.pp = (const double *)g.phi_prev[cur];
  ka.u = (const double *)g.u_prev[cur];
  ka.h0o = (double *)g.h0[cur ^ 1];
  ka.hmo = (double *)g.hm[cur ^ 1];
  ka.gmo = (double *)g.gm[cur ^ 1];
  ka.ppo = (double *)g.phi_prev[cur ^ 1];
  ka.uo = (double *)g.u_prev[cur ^ 1];
  ka.C = g.scratch;
  // The axes' factors are exactly 4 times the diagonals', and the rest slot's
  // -20 times, each rounded once, so that the collision's sums close as far as
  // rounding lets them.
  const double w5 = 1.0 / 36.0, w1 = 4.0 * w5;
  Cst64 &a = ka.c;
  a.one = 1.0;
  a.zero = 0.0;
  a.two = 2.0;
  a.four = 4.0;
  a.six = 6.0;
  a.half = 0.5;
  a.quarter = 0.25;
  a.w1 = w1;
  a.w5 = w5;
  double Gam = 0.0;
  for (int k = 0; k < c.N; ++k) Gam += 1.0 / c.rho_t[k];
  a.invN = 1.0 / c.N;
  a.bulk = c.bulk;
  a.bN = c.bulk / c.N;
  const double rho = c.rho_base;  // equal densities
  a.rinv = 1.0 / rho;
  a.rinvh = 0.5 / rho;
  a.F0x = rho * c.grav[0];
  a.F0y = rho * c.grav[1];
  a.grx = c.grav[0];
  a.gry = c.grav[1];
  a.gsc = g.grad_scheme == 1 ? 1.0 / 48.0 : 1.0 / 12.0;
  a.invG = 1.0 / Gam;
  a.r0 = c.rho_base;
  for (int k = 0; k < 5; ++k) a.gam[k] = k < c.N ? 1.0 / c.rho_t[k] : 0.0;
  for (int i = 0; i < 4; ++i) {
    const bool in = i < c.NP;
    for (int j = 0; j < 4; ++j) a.lam6[i][j] = c.lam[i][j] / 6.0;
    a.off[i] = c.off[i];
    a.mul[i] = c.mul[i];
    a.cm[i] = in ? c.bulk * c.mul[i] * a.gam[i] : 0.0;
    a.r0 += c.K[i] * c.off[i];
    a.kap[i] = c.kap[i];
    a.kapg[i] = c.kap[i] * a.gsc;
    a.kmobg[i] = c.kmob[i] * a.gsc;
    a.kD[i] = c.tau_inv[i] * c.a[i] / 36.0;
    a.kA[i] = 4.0 * a.kD[i];
    a.c1[i] = (c.tau_inv[i] + c.src[i]) / 3.0;
    a.c2[i] = c.src[i] / 3.0;
    a.keep[i] = 1.0 - c.tau_inv[i];
    a.ti[i] = c.tau_inv[i];
    a.kR[i] = -20.0 * a.kD[i];
  }
  const double tg = c.tg_inv, ff = c.ffac;
  a.keep_g = 1.0 - tg;
  // tg (3 p - 3/2 rho u.u) with p = 3/5 (sum g + u.grad(rho)/2 - 2/3 rho u.u)
  a.s18 = 1.8 * tg;
  a.s09 = 0.9 * tg;
  a.ruu = -2.7 * tg;
  a.f3 = 3.0 * ff;
  a.jh = 0.5 * c.jfac;
  a.B1d = tg / 12.0;
  a.B1a = 4.0 * a.B1d;
  a.B2d = tg / 8.0;
  a.B2a = 4.0 * a.B2d;
  a.C1d = ff / 12.0;
  a.C1a = 4.0 * a.C1d;
  a.D1a = ff;
  a.E1a = ff / 3.0;
  a.E2a = 0.5 * ff * c.jfac;
  return ka;
}

// Sum and product as fused multiply-adds of three registers: the same values
// (a product of zero comes out as +0). See above.
__device__ __forceinline__ double add64(const Cst64 &k, double x, double y) {
  return fma(x, k.one, y);
}
__device__ __forceinline__ double sub64(const Cst64 &k, double x, double y) {
  return fma(-y, k.one, x);
}
__device__ __forceinline__ double mul64(const Cst64 &k, double x, double y) {
  return fma(x, y, k.zero);
}

// The constants to shared memory, all of a thread's reads first (one-warp
// blocks, 150^2 unequal densities: 19.0 -> 18.1 us per step against a loop).
template <int NTH>
__device__ __forceinline__ void stage_cst64(Cst64 &k, const Cst64 &c, int tid) {
  constexpr int N = (int)(sizeof(Cst64) / sizeof(double)), M = (N + NTH - 1) / NTH;
  double v[M];
#pragma unroll
  for (int m = 0; m < M; ++m)
    if (tid + m * NTH < N) v[m] = ((const double *)&c)[tid + m * NTH];
#pragma unroll
  for (int m = 0; m < M; ++m)
    if (tid + m * NTH < N) ((double *)&k)[tid + m * NTH] = v[m];
}
// Sums of Eq. N31 over the eight neighbours, in units of w = 1/36: the
// gradient over 12 (or 6 g1 - g2 over 48, Eq. N40) and the Laplacian over 6.
struct Nine {
  double e, w, n, s, ne, nw, se, sw;
};
__device__ __forceinline__ void grad64(const Cst64 &k, const Nine &v, double &gx, double &gy) {
  const double d1 = sub64(k, v.ne, v.sw), d2 = sub64(k, v.se, v.nw);
  gx = fma(k.four, sub64(k, v.e, v.w), add64(k, d1, d2));
  gy = fma(k.four, sub64(k, v.n, v.s), sub64(k, d1, d2));
}
__device__ __forceinline__ double lap64(const Cst64 &k, const Nine &v, double c) {
  const double a = add64(k, add64(k, v.e, v.w), add64(k, v.n, v.s));
  const double d = add64(k, add64(k, v.ne, v.sw), add64(k, v.se, v.nw));
  return fma(k.four, fma(-k.four, c, a), fma(-k.four, c, d));  // 0 on a uniform field
}
// c (1 - c) (1 - 2 c)
__device__ __forceinline__ double bulk64(const Cst64 &k, double c) {
  return mul64(k, fma(-c, c, c), fma(-k.two, c, k.one));
}

__device__ __forceinline__ double phi64(const K64 &a, const Cst64 &k, int i, size_t q) {
  double s = __ldg(a.h0 + (size_t)i * a.V + q);
#pragma unroll
  for (int m = 0; m < 8; ++m) s = add64(k, s, __ldg(a.hm + (size_t)(i * 8 + m) * a.V + q));
  return s;
}

// Collisions and push streaming of node (x, y) = q from phi, C_i and the force.
// With NU, rho, 1/rho, grad rho and J~ vary; without, they are constants in k.
struct Flow64 {
  double Fx, Fy, rho, rinv, gx, gy, Jx, Jy;
};
template <int NP, bool NU, bool WALL>
__device__ __forceinline__ void collide64(const K64 &a, const Cst64 &k, int x, int y, size_t q,
                                          const double *ph, const double *C,
                                          const Flow64 &f) {
  const int nx = a.nx, ny = a.ny;
  const size_t V = a.V;
  const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
  const size_t r0 = q - x;
  const size_t rm = y == 0 ? (size_t)(ny - 1) * nx : r0 - nx;
  const size_t rp = y == ny - 1 ? 0 : r0 + nx;
  // destination slot (direction, node) of population k
  auto put = [&](double *base, int d_, double v) {
    const int cx = cx_of(d_), cy = cy_of(d_);
    size_t d = (cy == 0 ? r0 : (cy > 0 ? rp : rm)) + (cx == 0 ? x : (cx > 0 ? xp : xm));
    int kk = d_;
    if (WALL && ((cy > 0 && y == ny - 1) || (cy < 0 && y == 0))) {
      d = q;
      kk = opp_of(d_);
    }
    base[(size_t)(kk - 1) * V + d] = v;
  };
  double g[9];
#pragma unroll
  for (int m = 1; m < 9; ++m) g[m] = __ldcg(a.gm + (size_t)(m - 1) * V + q);
  auto add = [&](double u, double v) { return add64(k, u, v); };
  auto sub = [&](double u, double v) { return sub64(k, u, v); };
  const double d57 = sub(g[5], g[7]), d68 = sub(g[6], g[8]);
  const double mx = add(sub(g[1], g[3]), sub(d57, d68));
  const double my = add(sub(g[2], g[4]), add(d57, d68));
  const double sg = add(add(add(g[1], g[3]), add(g[2], g[4])),
                        add(add(g[5], g[7]), add(g[6], g[8])));
  double ux, uy, uu, A0, B1a, B1d, B2a, B2d, Hx, Hy;
  if constexpr (NU) {
    ux = mul64(k, fma(k.half, f.Fx, mx), f.rinv);
    uy = mul64(k, fma(k.half, f.Fy, my), f.rinv);
    uu = fma(ux, ux, mul64(k, uy, uy));
    const double ugr = fma(ux, f.gx, mul64(k, uy, f.gy));
    const double uFJ = fma(ux, fma(k.jh, f.Jx, f.Fx), mul64(k, uy, fma(k.jh, f.Jy, f.Fy)));
    A0 = fma(-k.f3, uFJ, fma(mul64(k, k.ruu, f.rho), uu, fma(k.s09, ugr, mul64(k, k.s18, sg))));
    B1a = mul64(k, k.B1a, f.rho);
    B1d = mul64(k, k.B1d, f.rho);
    B2a = mul64(k, k.B2a, f.rho);
    B2d = mul64(k, k.B2d, f.rho);
    Hx = fma(k.E2a, f.Jx, fma(k.E1a, f.gx, mul64(k, k.D1a, f.Fx)));
    Hy = fma(k.E2a, f.Jy, fma(k.E1a, f.gy, mul64(k, k.D1a, f.Fy)));
  } else {
    ux = fma(k.rinvh, f.Fx, mul64(k, mx, k.rinv));
    uy = fma(k.rinvh, f.Fy, mul64(k, my, k.rinv));
    uu = fma(ux, ux, mul64(k, uy, uy));
    const double uF = fma(ux, f.Fx, mul64(k, uy, f.Fy));
    A0 = fma(-k.f3, uF, fma(k.ruu, uu, mul64(k, k.s18, sg)));  // ruu, B1, B2 hold rho
    B1a = k.B1a;
    B1d = k.B1d;
    B2a = k.B2a;
    B2d = k.B2d;
    Hx = mul64(k, k.D1a, f.Fx);
    Hy = mul64(k, k.D1a, f.Fy);
  }
  const double A0a = mul64(k, A0, k.w1), A0d = mul64(k, A0, k.w5);
  {
    const double us = add(ux, uy), ud = sub(uy, ux);
    const double Fs = add(f.Fx, f.Fy), Fd = sub(f.Fy, f.Fx);
    const double Hs = add(Hx, Hy), Hd = sub(Hy, Hx);
    auto axis = [&](int d, double cu, double cF, double cH) {
      const double E = fma(cu, fma(B2a, cu, cH), A0a), O = fma(B1a, cu, mul64(k, k.C1a, cF));
      const int o = opp_of(d);
      put(a.gmo, d, fma(k.keep_g, g[d], add(E, O)));
      put(a.gmo, o, fma(k.keep_g, g[o], sub(E, O)));
    };
    auto diag = [&](int d, double cu, double cF, double cH) {
      const double E = fma(cu, fma(k.quarter, cH, mul64(k, B2d, cu)), A0d), O = fma(B1d, cu, mul64(k, k.C1d, cF));
      const int o = opp_of(d);
      put(a.gmo, d, fma(k.keep_g, g[d], add(E, O)));
      put(a.gmo, o, fma(k.keep_g, g[o], sub(E, O)));
    };
    axis(1, ux, f.Fx, Hx);
    axis(2, uy, f.Fy, Hy);
    diag(5, us, Fs, Hs);
    diag(6, ud, Fd, Hd);
  }
  const double upx = __ldg(a.u + q), upy = __ldg(a.u + V + q);
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    double *hmo = a.hmo + (size_t)(i * 8) * V;
    double h[9];
    h[0] = __ldcg(a.h0 + (size_t)i * V + q);
#pragma unroll
    for (int m = 1; m < 9; ++m) h[m] = __ldcg(a.hm + (size_t)(i * 8 + m - 1) * V + q);
    const double keep = k.keep[i], Ci = C[i];
    const double ala = mul64(k, k.kA[i], Ci), ald = mul64(k, k.kD[i], Ci);
    const double c1 = mul64(k, k.c1[i], ph[i]), c2 = mul64(k, k.c2[i], __ldg(a.pp + (size_t)i * V + q));
    const double bx = fma(c1, ux, -mul64(k, c2, upx)), by = fma(c1, uy, -mul64(k, c2, upy));
    const double bs = add(bx, by), bd = sub(by, bx);  // of the diagonals, times 4
    auto ax = [&](int d, double b) { put(hmo, d, add(fma(keep, h[d], ala), b)); };
    auto dg = [&](int d, double b, double s) {
      put(hmo, d, fma(s, b, fma(keep, h[d], ald)));
    };
    ax(1, bx);
    ax(2, by);
    ax(3, -bx);
    ax(4, -by);
    dg(5, bs, k.quarter);
    dg(6, bd, k.quarter);
    dg(7, bs, -k.quarter);
    dg(8, bd, -k.quarter);
    a.h0o[(size_t)i * V + q] = fma(k.kR[i], Ci, fma(k.ti[i], ph[i], mul64(k, keep, h[0])));
  }
  a.uo[q] = ux;
  a.uo[V + q] = uy;
}

// phi of a TX x TY tile and its ring of one node into s (stride TX + 2), for
// positions up to one beyond the grid (wrapped, or a wall's ghost row).
template <int NP, bool WALL, int TX, int TY>
__device__ __forceinline__ void tile_phi64(const K64 &a, const Cst64 &k, int x0, int y0, int tid,
                                           double (*s)[(TX + 2) * (TY + 2)],
                                           double *ph) {
  constexpr int SW = TX + 2, NTH = TX * TY, NRING = SW * (TY + 2) - NTH;
  const int nx = a.nx, ny = a.ny;
  const size_t V = a.V;
  auto node = [&](int X, int Y) {
    X = X < 0 ? nx - 1 : (X >= nx ? 0 : X);
    if (WALL) Y = Y < 0 ? 0 : (Y >= ny ? ny - 1 : Y);
    else Y = Y < 0 ? ny - 1 : (Y >= ny ? 0 : Y);
    return (size_t)Y * nx + X;
  };
  const int tx = tid % TX, ty = tid / TX;
  if (x0 + tx <= nx && y0 + ty <= ny) {
    const size_t q = node(x0 + tx, y0 + ty);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      ph[i] = phi64(a, k, i, q);
      s[i][(ty + 1) * SW + tx + 1] = ph[i];
    }
  }
  // ring: top row, bottom row, left column, right column; (phase, position)
  // pairs over all warps, so that no quarter of the SM sums more than another
  for (int e = tid; e < NP * NRING; e += NTH) {
    const int i = e / NRING, r = e % NRING;
    int lx, ly;
    if (r < 2 * SW) {
      ly = r < SW ? 0 : TY + 1;
      lx = r < SW ? r : r - SW;
    } else {
      ly = 1 + (r - 2 * SW) % TY;
      lx = (r - 2 * SW) < TY ? 0 : TX + 1;
    }
    const int X = x0 - 1 + lx, Y = y0 - 1 + ly;
    if (X <= nx && Y <= ny) s[i][ly * SW + lx] = phi64(a, k, i, node(X, Y));
  }
}

template <int SW>
__device__ __forceinline__ Nine nine_at(const double *s, int o) {
  return {s[o + 1],      s[o - 1],      s[o + SW],     s[o - SW],
          s[o + SW + 1], s[o + SW - 1], s[o - SW + 1], s[o - SW - 1]};
}

// Equal densities, central scheme: the whole step in one kernel.
template <int NP, bool WALL, int TX, int TY>
__global__ void __launch_bounds__(TX *TY, 512 / (TX * TY))
    step64_kernel(const __grid_constant__ K64 a, int ntx) {
  constexpr int SW = TX + 2;
  __shared__ double s[NP][SW * (TY + 2)];
  __shared__ Cst64 k;
  const int tid = threadIdx.x;
  const int x0 = (int)(blockIdx.x % ntx) * TX, y0 = (int)(blockIdx.x / ntx) * TY;
  double ph[NP];
  stage_cst64<TX * TY>(k, a.c, tid);
  __syncthreads();
  tile_phi64<NP, WALL, TX, TY>(a, k, x0, y0, tid, s, ph);
  __syncthreads();
  const int x = x0 + tid % TX, y = y0 + tid / TX;
  if (x >= a.nx || y >= a.ny) return;
  const size_t q = (size_t)y * a.nx + x;
  const int o = (tid / TX + 1) * SW + tid % TX + 1;
  // C_i (Eqs. N17, N18) and F = sum C_i grad phi_i + rho G
  double C[NP], gx[NP], gy[NP];
  {
    double lp[NP], S = ph[0];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const Nine v = nine_at<SW>(s[i], o);
      grad64(k, v, gx[i], gy[i]);
      lp[i] = lap64(k, v, ph[i]);
    }
#pragma unroll
    for (int i = 1; i < NP; ++i) S = add64(k, S, ph[i]);
    const double base = fma(-k.invN, S, k.invN);
    double f[NP], sum = bulk64(k, base);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      f[i] = bulk64(k, add64(k, ph[i], base));
      sum = add64(k, sum, f[i]);
    }
    const double mean = -mul64(k, k.bN, sum);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      C[i] = fma(k.bulk, f[i], mean);
#pragma unroll
      for (int j = 0; j < NP; ++j) C[i] = fma(-k.lam6[i][j], lp[j], C[i]);
    }
  }
  Flow64 fl;
  double sx = mul64(k, C[0], gx[0]), sy = mul64(k, C[0], gy[0]);
#pragma unroll
  for (int i = 1; i < NP; ++i) {
    sx = fma(C[i], gx[i], sx);
    sy = fma(C[i], gy[i], sy);
  }
  fl.Fx = fma(k.gsc, sx, k.F0x);
  fl.Fy = fma(k.gsc, sy, k.F0y);
#pragma unroll
  for (int i = 0; i < NP; ++i) a.ppo[(size_t)i * a.V + q] = ph[i];
  collide64<NP, false, WALL>(a, k, x, y, q, ph, C, fl);
}

// phi(t) (to the next step's phi(t-1)) and C_i of every node, general maps
// of Eqs. N12, N17, N18 (their rank-one parts summed once):
// c_k = gamma~_k (varphi_k + (1 - sum_j gamma~_j varphi_j) / Gamma).
template <int NP, bool WALL, int TX, int TY>
__global__ void __launch_bounds__(TX *TY) pot64_kernel(const __grid_constant__ K64 a, int ntx) {
  constexpr int SW = TX + 2;
  __shared__ double s[NP][SW * (TY + 2)];
  __shared__ Cst64 k;
  const int tid = threadIdx.x;
  const int x0 = (int)(blockIdx.x % ntx) * TX, y0 = (int)(blockIdx.x / ntx) * TY;
  double ph[NP];
  stage_cst64<TX * TY>(k, a.c, tid);
  __syncthreads();
  tile_phi64<NP, WALL, TX, TY>(a, k, x0, y0, tid, s, ph);
  __syncthreads();
  const int x = x0 + tid % TX, y = y0 + tid / TX;
  if (x >= a.nx || y >= a.ny) return;
  const size_t q = (size_t)y * a.nx + x;
  const int o = (tid / TX + 1) * SW + tid % TX + 1;
  double lp[NP], vp[NP], f[NP], sv = -1.0;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    lp[i] = lap64(k, nine_at<SW>(s[i], o), ph[i]);
    vp[i] = fma(k.mul[i], ph[i], k.off[i]);
    sv = fma(k.gam[i], vp[i], sv);
  }
  const double t = -mul64(k, sv, k.invG);
  double fs = mul64(k, k.gam[NP], bulk64(k, mul64(k, k.gam[NP], t)));
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    f[i] = bulk64(k, mul64(k, k.gam[i], add64(k, vp[i], t)));
    fs = fma(k.gam[i], f[i], fs);
  }
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    double Ci = mul64(k, k.cm[i], fma(-k.invG, fs, f[i]));
#pragma unroll
    for (int j = 0; j < NP; ++j) Ci = fma(-k.lam6[i][j], lp[j], Ci);
    a.C[(size_t)i * a.V + q] = Ci;
    a.ppo[(size_t)i * a.V + q] = ph[i];
  }
}

// The collision of every node from the stencils of phi and C_i in memory
// (9 or, Eq. N40, 17 points; L1 and L2 hits).
template <int NP, bool NU, bool WALL, bool G40, int NTH>
__global__ void __launch_bounds__(NTH, 512 / NTH > 32 ? 32 : 512 / NTH) coll64_kernel(const __grid_constant__ K64 a) {
  __shared__ Cst64 k;
  stage_cst64<NTH>(k, a.c, threadIdx.x);
  __syncthreads();
  const size_t q = (size_t)blockIdx.x * NTH + threadIdx.x;
  const size_t V = a.V;
  if (q >= V) return;
  const int nx = a.nx, ny = a.ny;
  const int y = V <= 0xffffffffu ? (int)((unsigned)q / (unsigned)nx) : (int)(q / nx);
  const int x = (int)(q - (size_t)y * nx);
  auto xi = [&](int v) { return v < 0 ? v + nx : (v >= nx ? v - nx : v); };
  auto yi = [&](int v) {
    if (WALL) return v < 0 ? 0 : (v >= ny ? ny - 1 : v);
    return v < 0 ? v + ny : (v >= ny ? v - ny : v);
  };
  // columns x - 1, x + 1 and rows y - 1, y + 1; the ones two away from those
  // (grids of one or two nodes wrap more than once)
  const int xa = xi(x - 1), xb = xi(x + 1), xaa = xi(xa - 1), xbb = xi(xb + 1);
  const int ya = yi(y - 1), yb = yi(y + 1);
  const int yaa = yi(WALL ? y - 2 : ya - 1), ybb = yi(WALL ? y + 2 : yb + 1);
  const size_t r0 = (size_t)y * nx, ra = (size_t)ya * nx, rb = (size_t)yb * nx;
  const size_t raa = (size_t)yaa * nx, rbb = (size_t)ybb * nx;
  auto grad = [&](const double *z, double &gx, double &gy) {
    const Nine v = {z[r0 + xb], z[r0 + xa], z[rb + x],  z[ra + x],
                    z[rb + xb], z[rb + xa], z[ra + xb], z[ra + xa]};
    grad64(k, v, gx, gy);
    if constexpr (G40) {
      const Nine v2 = {z[r0 + xbb],  z[r0 + xaa],  z[rbb + x],   z[raa + x],
                       z[rbb + xbb], z[rbb + xaa], z[raa + xbb], z[raa + xaa]};
      double hx, hy;
      grad64(k, v2, hx, hy);
      gx = fma(k.six, gx, -hx);
      gy = fma(k.six, gy, -hy);
    }
  };
  Flow64 f;
  double ph[NP], C[NP];
  double sx = 0.0, sy = 0.0;
  f.gx = f.gy = f.Jx = f.Jy = 0.0;
  f.rho = k.r0;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const double *zp = a.ppo + (size_t)i * V, *zc = a.C + (size_t)i * V;
    double gx, gy;
    ph[i] = zp[q];
    C[i] = zc[q];
    grad(zp, gx, gy);
    sx = fma(C[i], gx, sx);
    sy = fma(C[i], gy, sy);
    if constexpr (NU) {
      double cx, cy;
      grad(zc, cx, cy);
      f.gx = fma(k.kapg[i], gx, f.gx);
      f.gy = fma(k.kapg[i], gy, f.gy);
      f.Jx = fma(-k.kmobg[i], cx, f.Jx);
      f.Jy = fma(-k.kmobg[i], cy, f.Jy);
      f.rho = fma(k.kap[i], ph[i], f.rho);
    }
  }
  if constexpr (NU) {
    f.rinv = 1.0 / f.rho;
    f.Fx = fma(k.gsc, sx, mul64(k, f.rho, k.grx));
    f.Fy = fma(k.gsc, sy, mul64(k, f.rho, k.gry));
  } else {
    f.Fx = fma(k.gsc, sx, k.F0x);
    f.Fy = fma(k.gsc, sy, k.F0y);
  }
  collide64<NP, NU, WALL>(a, k, x, y, q, ph, C, f);
}

// Tile of the phi kernels: 16 x 8 nodes (four warps), or 16 x 4 where half
// the tile lets the 152 SMs finish with fewer warps on the busiest one (small
// grids only: its ring is 44 positions per 64 nodes against 52 per 128; 128^2
// is 128 of the larger tiles, 150^2 190, two on some SMs, or 380, three).
template <int NP, bool NU, bool WALL, bool G40>
cudaError_t launch_step64_t(const K64 &a, cudaStream_t s) {
  const long ntx = (a.nx + 15) / 16;
  const long t8 = ntx * ((a.ny + 7) / 8), t4 = ntx * ((a.ny + 3) / 4);
  const bool half = t8 <= 4 * 152 && (t4 + 151) / 152 * 2 < (t8 + 151) / 152 * 4;
  if constexpr (!NU && !G40) {
    if (half) step64_kernel<NP, WALL, 16, 4><<<(unsigned)t4, 64, 0, s>>>(a, (int)ntx);
    else step64_kernel<NP, WALL, 16, 8><<<(unsigned)t8, 128, 0, s>>>(a, (int)ntx);
  } else {
    if (half) pot64_kernel<NP, WALL, 16, 4><<<(unsigned)t4, 64, 0, s>>>(a, (int)ntx);
    else pot64_kernel<NP, WALL, 16, 8><<<(unsigned)t8, 128, 0, s>>>(a, (int)ntx);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // one-warp blocks spread a small grid evenly; large ones take 128 threads
    if (a.V <= (size_t)152 * 32 * 32)
      coll64_kernel<NP, NU, WALL, G40, 32><<<(unsigned)((a.V + 31) / 32), 32, 0, s>>>(a);
    else
      coll64_kernel<NP, NU, WALL, G40, 128><<<(unsigned)((a.V + 127) / 128), 128, 0, s>>>(a);
  }
  return cudaGetLastError();
}

template <int NP, bool NU, bool WALL>
cudaError_t launch_step64(const Consts &c, const Grid &g, int cur, cudaStream_t s) {
  K64 a = make_k64(c, g, cur);
  if (!NU) {  // rho is constant: into the coefficients
    const double r = c.rho_base;
    a.c.ruu *= r;
    a.c.B1d = r * c.tg_inv / 12.0;
    a.c.B1a = 4.0 * a.c.B1d;
    a.c.B2d = r * c.tg_inv / 8.0;
    a.c.B2a = 4.0 * a.c.B2d;
  }
  return g.grad_scheme == 1 ? launch_step64_t<NP, NU, WALL, true>(a, s)
                            : launch_step64_t<NP, NU, WALL, false>(a, s);
}

}  // namespace lbm
