// Reverse mode of the D2Q9 BGK + exact-difference-forcing step (eq. (1),
// eq. (2), Sec. 3 of Tauzin et al. 2018) and of the box-averaged
// dissipation objective built from the RHS^{E,4} term of eq. (8).  This is
// the differentiation of the forward model; the paper has no counterpart.
//
// Forward step in the public layout (f = pre-collision state):
//   f*_l(x) = (1 - w) f_l + (w - 1) feq_l(rho, j) + feq_l(rho, m'),
//   f_l(x + c_l, n+1) = f*_l(x),
// with w = 1/tau, rho = sum f, j = sum c f, m' = (1 - alpha) j + F_ext
// (= rho (u + F/rho)), and the equilibrium written in momentum form
//   feq_l(rho, m) = t_l [rho + 3 c.m + (4.5 (c.m)^2 - 1.5 |m|^2) / rho].
// Adjoint: mu_l(x) = lambda_l(x + c_l, n+1) (transpose of the push), then
//   lambda_l(x, n) = (1 - w) mu_l + A_rho + c_l . A_j + dJ_n/df_l(x),
//   A_rho = sum_k mu_k [(w - 1) d_rho feq_k(rho, j) + d_rho feq_k(rho, m')],
//   A_j   = sum_k mu_k [(w - 1) d_m feq_k(rho, j) + (1 - alpha) d_m feq_k(rho, m')],
//   dJ/dtau += sum mu_l (f_l - feq_l(rho, j)) / tau^2,
//   dJ/dF0  += sum mu_l d_m feq_l(rho, m') . s,  s = (sin(2 pi kf y/ny), sin(2 pi kf x/nx)).
// Objective term at time n: J_n = weight / L^2 * sum_{x in box} eps(x),
//   eps = -nu rho S_ij G_ij, G_ij = D_j u_i, S_ij = G_ij + G_ji,
//   u = (j + F/2)/rho, F = F_ext - alpha j, nu = (tau - 1/2)/3,
// whose adjoint uses D^T = -D (antisymmetric periodic eq. (18) stencil).
// The step's adjoint is formed in 64-bit fixed point (the FP64 pipe is narrow)
// with FP64 as the fallback, the objective in FP64; reductions are
// block-deterministic.
#include <algorithm>
#include <cmath>

#include "lbm_collide.cuh"

namespace lbm {

namespace {

// Fields of the objective on its region, one set per level of a batch:
// kObjFields planes of region cells.
enum ObjField { A_RHO = 0, A_U, A_V, GAM_XX, GAM_XY, GAM_YY, D_RHO, D_JX, D_JY, D_TOT, kObjFields };
constexpr int kObjLevels = 256;  // levels of one batch at most
struct ObjWeights {
  double cw[kObjLevels];  // weight / L^2 per level, 0: no objective at that level
};

struct AGrid {
  int nx, ny, kf, force;
  double nu, alpha, tau, omega, F0;
  const double *fxt, *fyt;  // F_ext tables (F0 included)
  FixedBgk fixed;           // constants of the fixed-point forms
  long long w1, keep;       // (omega - 1) 2^63, (1 - omega) 2^63
};

__device__ __forceinline__ int wrapn(int i, int n) {
  return i < 0 ? i + n : (i >= n ? i - n : i);
}
__device__ __forceinline__ int wr(int i, int n) { return n >= 4 ? wrapn(i, n) : wrapi(i, n); }

__device__ __forceinline__ void force_dir(const AGrid &g, int x, int y, double &sx, double &sy) {
  if (g.force == 1) {
    sx = sinpi(2.0 * g.kf * (double)y / g.ny);
    sy = sinpi(2.0 * g.kf * (double)x / g.nx);
  } else {
    sx = 0.0;
    sy = 0.0;
  }
}

// The direction s of dF_ext/dF0 per row and column, tabulated once per
// adjoint step (the cell kernel then reads two doubles instead of
// evaluating two FP64 sines, which the FP64 pipe of this part pays for).
__global__ void k_sine_tables(AGrid g, double *tab) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.ny + g.nx;
       i += gridDim.x * blockDim.x) {
    double sx, sy;
    if (i < g.ny) {
      force_dir(g, 0, i, sx, sy);
      tab[i] = sx;
    } else {
      force_dir(g, i - g.ny, 0, sx, sy);
      tab[i] = sy;
    }
  }
}

template <int NQ>
__device__ void block_sums(double (&v)[NQ], double *out, int add = 0) {
  __shared__ double sh[NQ][32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    double a = v[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if (lane == 0) sh[q][wid] = a;
  }
  __syncthreads();
  if (tid < NQ) {
    double a = 0.0;
    for (int k = 0; k < nw; ++k) a += sh[tid][k];
    out[tid] = add ? out[tid] + a : a;
  }
}

#define FOR_CELLS                                                                   \
  const size_t N = (size_t)g.nx * g.ny;                                             \
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < N;             \
       c += (size_t)gridDim.x * blockDim.x)

// The objective touches only the box V0 and the cells within the eq. (18)
// stencil reach (4 cells) of it: the region R = V0 widened by 4 on each
// side (the whole axis where that covers it).  u is needed on R, Gamma on
// V0 and dJ/du = -D^T Gamma on R; every other cell has no objective term.
struct Region {
  int x0, y0, w, h;  // lower-left corner (wrapped) and extent, w <= nx, h <= ny
};

__host__ __device__ inline Region objective_region(int nx, int ny, int bx, int by, int L) {
  Region r;
  if (L + 8 >= nx) { r.x0 = 0; r.w = nx; } else { r.x0 = ((bx - 4) % nx + nx) % nx; r.w = L + 8; }
  if (L + 8 >= ny) { r.y0 = 0; r.h = ny; } else { r.y0 = ((by - 4) % ny + ny) % ny; r.h = L + 8; }
  return r;
}

__device__ __forceinline__ bool in_region(int x, int y, const Region &r, const AGrid &g) {
  return wrapi(x - r.x0, g.nx) < r.w && wrapi(y - r.y0, g.ny) < r.h;
}

// Index of cell (x, y) of the region in its planes.
__device__ __forceinline__ int region_index(int x, int y, const Region &r, const AGrid &g) {
  return wrapi(y - r.y0, g.ny) * r.w + wrapi(x - r.x0, g.nx);
}

// The objective's kernels run over the levels of a batch at once (blockIdx.y):
// they read the recorded states only, so nothing of them has to wait for the
// adjoint.  One launch per level and kernel cost 14.4 us per weighted level of
// 256^2, L = 16, between the adjoint steps.

// rho, j and u = (j + F/2)/rho of the public states f[level][9][ny][nx] on R.
__global__ void k_region_velocity(AGrid g, Region R, const double *states, double *fields,
                                  ObjWeights W) {
  const int q = blockIdx.y, nreg = R.w * R.h;
  if (W.cw[q] == 0.0) return;
  const size_t N = (size_t)g.nx * g.ny;
  const double *f = states + (size_t)q * kQ * N;
  double *F = fields + (size_t)q * kObjFields * nreg;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nreg; i += gridDim.x * blockDim.x) {
    const int x = wrapi(R.x0 + i % R.w, g.nx), y = wrapi(R.y0 + i / R.w, g.ny);
    const size_t c = (size_t)y * g.nx + x;
    double r = 0, a = 0, b = 0;
#pragma unroll
    for (int l = 0; l < kQ; ++l) {
      const double v = f[(size_t)l * N + c];
      r += v;
      if (cx_of(l) != 0) a += cx_of(l) * v;
      if (cy_of(l) != 0) b += cy_of(l) * v;
    }
    const double Fx = g.fxt[y] - g.alpha * a, Fy = g.fyt[x] - g.alpha * b;
    const double ir = 1.0 / r;
    F[A_RHO * nreg + i] = r;
    F[A_U * nreg + i] = (a + 0.5 * Fx) * ir;
    F[A_V * nreg + i] = (b + 0.5 * Fy) * ir;
  }
}

// Four lanes per cell: lanes 4q .. 4q + 3 of a warp share cell q of the
// warp's group of eight, lane part p = lane & 3 evaluates one of the cell's
// four stencil derivatives and the quad exchanges them by shuffles (a
// quarter of the dependent FP64 chain per lane, four times the SMs).  The
// loop runs in whole warps: a lane past the last cell works on the last
// cell and writes nothing, so every shuffle has the full warp.
#define FOR_QUADS(NCELLS)                                                      \
  const int lane = threadIdx.x & 31, p = lane & 3, qb = lane & ~3;             \
  const int wglob = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);       \
  const int nwarps = (int)((gridDim.x * blockDim.x) >> 5);                     \
  for (int i0 = wglob * 8; i0 < (NCELLS); i0 += nwarps * 8)

__device__ __forceinline__ double quad_get(double v, int qb, int k) {
  return __shfl_sync(0xffffffffu, v, qb + k);
}

// The eq. (18) stencil derivative of the region plane A along x (dir 0) or y
// (dir 1) at (x, y), one code path for both directions (no divergence within
// a quad).
__device__ __forceinline__ double D_dir(const double *A, const AGrid &g, const Region &R, int x,
                                        int y, int dir) {
  auto at = [&](int k) {
    return A[dir ? region_index(x, wr(y + k, g.ny), R, g) : region_index(wr(x + k, g.nx), y, R, g)];
  };
  return 0.8 * (at(1) - at(-1)) - 0.2 * (at(2) - at(-2)) + (4.0 / 105.0) * (at(3) - at(-3)) -
         (1.0 / 280.0) * (at(4) - at(-4));
}

// Objective pass 1, over V0: Gamma_ij = dJ/dG_ij = -2 c nu rho S_ij
// (c = weight / L^2); explicit dJ/dtau part -c rho Q / 3 (d nu / d tau = 1/3).
// Four lanes per cell (FOR_QUADS): d/dx u, d/dy u, d/dx v, d/dy v.
__global__ void k_obj_gamma(AGrid g, Region R, double *fields, ObjWeights W, int bx, int by, int L,
                            double *partials) {
  const int q = blockIdx.y, nreg = R.w * R.h;
  const double cw = W.cw[q];
  double *F = fields + (size_t)q * kObjFields * nreg;
  double acc[1] = {0.0};
  const int nc = cw == 0.0 ? 0 : L * L;
  FOR_QUADS(nc) {
    const int iq = i0 + (lane >> 2), i = iq < nc ? iq : nc - 1;
    const int x = wrapi(bx + i % L, g.nx), y = wrapi(by + i / L, g.ny);
    const int c = region_index(x, y, R, g);
    const double d = D_dir(F + (p < 2 ? A_U : A_V) * nreg, g, R, x, y, p & 1);
    const double dxu = quad_get(d, qb, 0), dyu = quad_get(d, qb, 1);
    const double dxv = quad_get(d, qb, 2), dyv = quad_get(d, qb, 3);
    if (iq < nc) {
      const double sxx = 2 * dxu, sxy = dyu + dxv, syy = 2 * dyv;
      const double r = F[A_RHO * nreg + c];
      if (p < 3) {  // Gamma_xx, Gamma_xy, Gamma_yy: one per lane
        const double sp = p == 0 ? sxx : (p == 1 ? sxy : syy);
        F[(GAM_XX + p) * nreg + c] = -2.0 * cw * g.nu * r * sp;
      } else {
        const double Q = sxx * dxu + sxy * dyu + sxy * dxv + syy * dyv;
        F[D_RHO * nreg + c] = -cw * g.nu * Q;
        acc[0] += -cw * r * Q / 3.0;
      }
    }
  }
  block_sums<1>(acc, partials + (size_t)q * gridDim.x + blockIdx.x);
}

// Objective pass 2, over R: dJ/du_i = -sum_j D_j Gamma_ij (D^T = -D), then
// dJ/drho (with the direct part of V0), dJ/dj and the explicit dJ/dF0 part
// through u = ((1 - alpha/2) j + F_ext/2)/rho.  Four lanes per cell
// (FOR_QUADS): D_x Gamma_xx, D_y Gamma_xy, D_x Gamma_xy, D_y Gamma_yy, Gamma
// zero outside V0; then one quotient per lane (dJ/djx, dJ/djy, the velocity
// part of dJ/drho, the dJ/dF0 term) and the force direction s from the
// sine tables.
__global__ void k_obj_velocity_adjoint(AGrid g, Region R, double *fields, ObjWeights W,
                                       const double *sines, int bx, int by, int L,
                                       double *partials) {
  const int q = blockIdx.y, nreg = R.w * R.h;
  double *F = fields + (size_t)q * kObjFields * nreg;
  double acc[1] = {0.0};
  const int nc = W.cw[q] == 0.0 ? 0 : nreg;
  FOR_QUADS(nc) {
    const int iq = i0 + (lane >> 2), i = iq < nc ? iq : nc - 1;
    const int x = wrapi(R.x0 + i % R.w, g.nx), y = wrapi(R.y0 + i / R.w, g.ny);
    // box-relative coordinates: the stencil point k along dir is in V0 when
    // its along coordinate wraps into [0, L) and the cross one already is
    const int rx = wrapi(x - bx, g.nx), ry = wrapi(y - by, g.ny);
    const int dir = p & 1;
    const double *G = F + (p == 0 ? GAM_XX : (p == 3 ? GAM_YY : GAM_XY)) * nreg;
    const int ra = dir ? ry : rx, na = dir ? g.ny : g.nx;
    const bool cross_in = (dir ? rx : ry) < L;
    auto at = [&](int k) {
      if (!(cross_in && wr(ra + k, na) < L)) return 0.0;
      return G[dir ? region_index(x, wr(y + k, g.ny), R, g) : region_index(wr(x + k, g.nx), y, R, g)];
    };
    const double d = 0.8 * (at(1) - at(-1)) - 0.2 * (at(2) - at(-2)) +
                     (4.0 / 105.0) * (at(3) - at(-3)) - (1.0 / 280.0) * (at(4) - at(-4));
    const double Ux = -(quad_get(d, qb, 0) + quad_get(d, qb, 1));
    const double Uy = -(quad_get(d, qb, 2) + quad_get(d, qb, 3));
    const double r = F[A_RHO * nreg + i];
    double num;
    if (p == 0) {
      num = Ux * (1.0 - 0.5 * g.alpha);
    } else if (p == 1) {
      num = Uy * (1.0 - 0.5 * g.alpha);
    } else if (p == 2) {
      num = Ux * F[A_U * nreg + i] + Uy * F[A_V * nreg + i];
    } else {
      num = Ux * sines[y] + Uy * sines[g.ny + x];
    }
    const double qt = num / (p == 3 ? 2.0 * r : r);
    if (iq < nc) {
      if (p < 2) {
        F[(D_JX + p) * nreg + i] = qt;
      } else if (p == 2) {
        const double direct = (rx < L && ry < L) ? F[D_RHO * nreg + i] : 0.0;
        F[D_TOT * nreg + i] = direct - qt;
      } else {
        acc[0] += qt;
      }
    }
  }
  block_sums<1>(acc, partials + (size_t)q * gridDim.x + blockIdx.x);
}

// Adds a batch's objective partials to the sweep's running sums, fixed order.
__global__ void __launch_bounds__(256) k_obj_sum(const double *pt, int nt, const double *pf, int nf,
                                                 double *tau, double *F0) {
  double acc[2] = {0.0, 0.0};
  for (int i = threadIdx.x; i < nt; i += 256) acc[0] += pt[i];
  for (int i = threadIdx.x; i < nf; i += 256) acc[1] += pf[i];
  __shared__ double out[2];
  block_sums<2>(acc, out);
  __syncthreads();
  if (threadIdx.x == 0) {
    *tau += out[0];
    *F0 += out[1];
  }
}

// t_l-weighted sums over the populations of the pulled adjoint mu_l and
// their contractions with the equilibrium's derivatives.  With
//   feq_l(rho, m) = t_l [rho + 3 c.m + (4.5 (c.m)^2 - 1.5 |m|^2) / rho]
// and the moments M0 = sum t mu, M_a = sum t c_a mu, M_ab = sum t c_a c_b mu:
//   sum mu d_rho feq(rho, m) = M0 - (4.5 m.M2.m - 1.5 |m|^2 M0) / rho^2,
//   sum mu d_m   feq(rho, m) = 3 M1 + (9 M2.m - 3 m M0) / rho,
//   sum mu feq(rho, m)       = rho M0 + 3 m.M1 + (4.5 m.M2.m - 1.5 |m|^2 M0) / rho.
struct MuMoments {
  double m0, mx, my, mxx, mxy, myy;
};

__device__ __forceinline__ MuMoments mu_moments(const double (&mu)[kQ]) {
  constexpr double t1 = 1.0 / 9.0, t2 = 1.0 / 36.0;
  // sums and differences of the opposite pairs (1, 3), (2, 4), (5, 7), (6, 8)
  const double s13 = mu[1] + mu[3], d13 = mu[1] - mu[3], s24 = mu[2] + mu[4], d24 = mu[2] - mu[4];
  const double s57 = mu[5] + mu[7], d57 = mu[5] - mu[7], s68 = mu[6] + mu[8], d68 = mu[6] - mu[8];
  const double diag = s57 + s68;
  MuMoments M;
  M.m0 = fma(4.0 / 9.0, mu[0], fma(t1, s13 + s24, t2 * diag));
  M.mx = fma(t1, d13, t2 * (d57 - d68));
  M.my = fma(t1, d24, t2 * (d57 + d68));
  M.mxx = fma(t1, s13, t2 * diag);
  M.myy = fma(t1, s24, t2 * diag);
  M.mxy = t2 * (s57 - s68);
  return M;
}

// One cell of the adjoint of a step in FP64: lambda_out from the state fl, the
// pulled adjoint mu and the objective's (d_rho, d_jx, d_jy); t and (bx, by)
// receive sum mu (f - feq) and the adjoint of m'.
__device__ __forceinline__ void adjoint_cell_f64(const AGrid &g, int x, int y,
                                                 const double (&fl)[kQ], const double (&mu)[kQ],
                                                 double d_rho, double d_jx, double d_jy,
                                                 double (&out)[kQ], double &t, double &bx,
                                                 double &by) {
  // moments from the opposite pairs' sums and differences
  const double d57 = fl[5] - fl[7], d68 = fl[6] - fl[8];
  const double rho = fl[0] + ((fl[1] + fl[3]) + (fl[2] + fl[4])) + ((fl[5] + fl[7]) + (fl[6] + fl[8]));
  const double jx = (fl[1] - fl[3]) + (d57 - d68), jy = (fl[2] - fl[4]) + (d57 + d68);
  const double ir = 1.0 / rho;
  const double mpx = (1.0 - g.alpha) * jx + g.fxt[y];
  const double mpy = (1.0 - g.alpha) * jy + g.fyt[x];
  const MuMoments M = mu_moments(mu);
  // equilibrium at (rho, j): q_a = m.M2.m, p_a = M2.m
  const double pax = M.mxx * jx + M.mxy * jy, pay = M.mxy * jx + M.myy * jy;
  const double qa = (4.5 * (jx * pax + jy * pay) - 1.5 * (jx * jx + jy * jy) * M.m0) * ir;
  // at (rho, m')
  const double pbx = M.mxx * mpx + M.mxy * mpy, pby = M.mxy * mpx + M.myy * mpy;
  const double qb = (4.5 * (mpx * pbx + mpy * pby) - 1.5 * (mpx * mpx + mpy * mpy) * M.m0) * ir;
  const double w1 = g.omega - 1.0;
  const double Sa_rho = M.m0 - qa * ir, Sb_rho = M.m0 - qb * ir;
  // S_a = 3 M_a + 9 p_a / rho - 3 m_a M0 / rho with 9 / rho and 3 M0 / rho
  // formed once
  const double ir9 = 9.0 * ir, k0 = 3.0 * M.m0 * ir, mx3 = 3.0 * M.mx, my3 = 3.0 * M.my;
  const double Sa_x = fma(ir9, pax, fma(-jx, k0, mx3));
  const double Sa_y = fma(ir9, pay, fma(-jy, k0, my3));
  bx = fma(ir9, pbx, fma(-mpx, k0, mx3));
  by = fma(ir9, pby, fma(-mpy, k0, my3));
  const double Arho = w1 * Sa_rho + Sb_rho + d_rho;
  const double Ajx = w1 * Sa_x + (1.0 - g.alpha) * bx + d_jx;
  const double Ajy = w1 * Sa_y + (1.0 - g.alpha) * by + d_jy;
  // sum mu (f - feq(rho, j)) for dJ/dtau
  double muf = 0.0;
#pragma unroll
  for (int l = 0; l < kQ; ++l) muf += mu[l] * fl[l];
  t = muf - (rho * M.m0 + 3.0 * (jx * M.mx + jy * M.my) + qa);
  const double keep = 1.0 - g.omega;
  // lambda_l = keep mu_l + Arho + c_l . A, by opposite pairs (c . A once
  // per pair; a product by c = 0 still costs an FMA under IEEE arithmetic)
  const double cA[4] = {Ajx, Ajy, Ajx + Ajy, Ajy - Ajx};  // c of 1, 2, 5, 6
  out[0] = fma(keep, mu[0], Arho);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int l = k < 2 ? 1 + k : 5 + (k - 2), m = opposite(l);
    out[l] = fma(keep, mu[l], Arho + cA[k]);
    out[m] = fma(keep, mu[m], Arho - cA[k]);
  }
}

// The same in 64-bit fixed point (collide_fixed's reasons and range; 256^2:
// 13.9 us per adjoint step against 22.8).  The populations of the adjoint have no
// scale of their own: they are taken in units of 2^-53 of the exponent of the
// cell's largest one (emax), sums and products with three to six more bits, so
// that the cell's largest values keep FP64's 53 bits.  (A scale per warp loses
// the small adjoints beside a large one: 1e-8 relative at the 99th percentile
// on the rim of the objective's reach, 1e-14 in FP64.)  With u = j / rho and v = m' / rho the terms are
//   S_rho = M0 - Q(u), S = 3 M1 + 9 M2.u - 3 u M0,
//   Q(u) = 4.5 u.M2.u - 1.5 |u|^2 M0,
// (36 M are exact integer sums of the mu), sum mu feq = rho (M0 + 3 u.M1 +
// Q(u)).  Returns false where the cell needs the FP64 form.
__device__ __forceinline__ long long adj_fixed(double v, int emax) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const int e = (int)((hi >> 20) & 0x7ffu), r = emax - e;
  const unsigned long long m =
      (((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << 2;  // 2 x 2^53 .. 2^54
  // to nearest, ties to even: ties are frequent here (r = 2 drops one bit), and
  // rounding them one way would bias every step's adjoint
  const unsigned long long h = m >> (r & 63), odd = (h >> 1) & 1ull;
  const unsigned long long sticky = m & ((1ull << (r & 63)) - 1);
  const long long q = r > 57 || e == 0 ? 0 : (long long)((h + (sticky ? 1ull : odd)) >> 1);
  return (int)hi < 0 ? -q : q;
}
// v 2^(emax - 1023 - 53) to double, to nearest even
__device__ __forceinline__ double adj_double(long long v, int emax) {
  const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int n = __clzll((long long)a);
  const unsigned long long x = a << (n & 63), r = x + 0x3ffull + ((x >> 11) & 1ull);
  const unsigned carry = r < x;
  const unsigned e = (unsigned)(emax - 53 + 63 - 1 - n) << 20;
  const unsigned hi = n == 64 ? 0u : (unsigned)(r >> 43) + e + (carry << 21);
  return __hiloint2double((int)(hi | (v < 0 ? 0x80000000u : 0u)),
                          n == 64 ? 0 : (int)(unsigned)(r >> 11));
}
__device__ __forceinline__ bool adjoint_cell_fixed(const AGrid &g, int x, int y, int emax,
                                                   const double (&fl)[kQ], const double (&mu)[kQ],
                                                   double (&out)[kQ], double &t, double &bx,
                                                   double &by) {
  int bad;
  FixedCell C;
  fixed_cell(fl, g.fixed.k, C, bad);
  long long vx = C.ux, vy = C.uy;
  const Dig al = dig(g.fixed.alpha);
  if (g.fixed.forced) {
    const Dig Fx = dig(small_fixed(g.fxt[y], g.fixed.k, bad) - mulr(C.djx, al));
    const Dig Fy = dig(small_fixed(g.fyt[x], g.fixed.k, bad) - mulr(C.djy, al));
    const long long dx = mulr(Fx, C.ir), dy = mulr(Fy, C.ir);  // in 2^-60
    bad |= (unsigned long long)(dx + (1ll << 57)) > (1ull << 58) ||
           (unsigned long long)(dy + (1ll << 57)) > (1ull << 58);
    vx += dx << 4;
    vy += dy << 4;
  }
  if (bad) return false;
  long long m[kQ];
#pragma unroll
  for (int l = 0; l < kQ; ++l) m[l] = adj_fixed(mu[l], emax);  // |m| < 2^54
  const long long s13 = m[1] + m[3], d13 = m[1] - m[3], s24 = m[2] + m[4], d24 = m[2] - m[4];
  const long long s57 = m[5] + m[7], d57 = m[5] - m[7], s68 = m[6] + m[8], d68 = m[6] - m[8];
  const long long dg = s57 + s68;
  // 36 times the t-weighted moments, below 2^59.2
  const long long m0 = 16 * m[0] + 4 * (s13 + s24) + dg;
  const long long m1x = 4 * d13 + (d57 - d68), m1y = 4 * d24 + (d57 + d68);
  const Dig D0 = dig(m0), Dxx = dig(4 * s13 + dg), Dyy = dig(4 * s24 + dg), Dxy = dig(s57 - s68);
  struct Part {
    long long q2, px, py;  // 2 Q, 9 M2.w - 3 w M0
  };
  auto part = [&](long long wx, long long wy) {
    const Dig ax = dig(wx), ay = dig(wy);
    const long long px = mulr(Dxx, ax) + mulr(Dxy, ay), py = mulr(Dxy, ax) + mulr(Dyy, ay);
    const long long w2 = mulr(ax, ax) + mulr(ay, ay);
    const long long up = mulr(dig(px), ax) + mulr(dig(py), ay);
    Part P;
    P.q2 = 9 * up - 3 * mulr(D0, dig(w2));
    P.px = 9 * px - 3 * mulr(D0, ax);
    P.py = 9 * py - 3 * mulr(D0, ay);
    return P;
  };
  const Part A = part(C.ux, C.uy), B = part(vx, vy);
  const Dig w1 = dig(g.w1);  // omega - 1 in 2^-63
  const long long sbx = 3 * m1x + B.px, sby = 3 * m1y + B.py;
  const long long ar2 = 2 * mulr(dig(2 * m0 - A.q2), w1) + (2 * m0 - B.q2);  // 2 x 36 A_rho
  const long long ax = 2 * mulr(dig(3 * m1x + A.px), w1) + sbx - mulr(dig(sbx), al);
  const long long ay = 2 * mulr(dig(3 * m1y + A.py), w1) + sby - mulr(dig(sby), al);
  // back from 36 times, eight times over for one rounding at the end
  const Dig c836 = dig(4099276460824344804ll), c436 = dig(2049638230412172402ll);  // 2^67, 2^66 / 36
  const Dig kp = dig(g.keep);  // (1 - omega) 2^63
  const long long r = mulr(dig(ar2), c436), cx = mulr(dig(ax), c836), cy = mulr(dig(ay), c836);
  auto put = [&](int l, long long add) {
    out[l] = adj_double(mulr(dig(m[l] << 4), kp) + add, emax - 3);
  };
  put(0, r);
  put(1, r + cx);
  put(3, r - cx);
  put(2, r + cy);
  put(4, r - cy);
  put(5, r + cx + cy);
  put(7, r - cx - cy);
  put(6, r - cx + cy);
  put(8, r + cx - cy);
  // sum mu f - rho (M0 + 3 u.M1 + Q), 64 times over: the difference is a
  // thousandth of its parts
  const Dig c6436 = dig(8198552921648689607ll);  // 2^68 / 36
  long long muf = mulr(dig(m[0] << 6), dig(C.n[0] << 2));
#pragma unroll
  for (int l = 1; l < kQ; ++l) muf += mulr(dig(m[l] << 6), dig(C.n[l]));
  const long long u1 = 3 * (mulr(dig(m1x), dig(C.ux)) + mulr(dig(m1y), dig(C.uy)));
  // rho with the bits that its two quarter sums dropped (one sign: they would
  // add up over the cells)
  const int cut = ((int)(C.n[1] + C.n[2] + C.n[3] + C.n[4]) & 3) +
                  ((int)(C.n[5] + C.n[6] + C.n[7] + C.n[8]) & 3);
  muf -= 2 * mulr(dig(mulr(dig(2 * (2 * (m0 + u1) + A.q2)), c6436)), dig(2 * C.rho + (cut >> 1)));
  t = adj_double(muf, emax + g.fixed.k - 6);
  bx = adj_double(mulr(dig(sbx), c836), emax - 3);
  by = adj_double(mulr(dig(sby), c836), emax - 3);
  return true;
}

// Adjoint of one step (see the header comment).  obj_fields (or NULL) adds
// dJ_n/df on the objective region R.  Each CTA's (dJ/dtau, dJ/dF0) sums are
// added to its slot of `partials` (a sweep's running sums; steps are
// stream-ordered, so a slot has one writer at a time).
__global__ void k_adjoint(AGrid g, Region R, const double *f, const double *lam_in,
                          double *lam_out, const double *sines, const double *obj_fields,
                          double *partials) {
  double acc[2] = {0.0, 0.0};
  FOR_CELLS {
    const int x = (int)(c % g.nx), y = (int)(c / g.nx);
    double fl[kQ], mu[kQ], out[kQ], t, bx, by;
    unsigned emax = 0, ef = 0;
#pragma unroll
    for (int l = 0; l < kQ; ++l) {
      fl[l] = f[(size_t)l * N + c];
      const int xd = wr(x + cx_of(l), g.nx), yd = wr(y + cy_of(l), g.ny);
      mu[l] = lam_in ? lam_in[(size_t)l * N + (size_t)yd * g.nx + xd] : 0.0;
      if (mu[l] != 0.0) emax = max(emax, max(1u, ((unsigned)__double2hiint(mu[l]) >> 20) & 0x7ffu));
      ef = max(ef, ((unsigned)__double2hiint(fl[l]) >> 20) & 0x7ffu);
    }
    const bool obj = obj_fields && in_region(x, y, R, g);
    if (emax == 0 && !obj && ef < 0x7ffu) {  // no adjoint here yet
#pragma unroll
      for (int l = 0; l < kQ; ++l) lam_out[(size_t)l * N + c] = 0.0;
      continue;
    }
    // a common scale for the cell, away from the ends of the exponent range
    if (obj || !g.fixed.ok || emax < 200u || emax > 1800u ||
        !adjoint_cell_fixed(g, x, y, (int)emax, fl, mu, out, t, bx, by)) {
      const int nreg = R.w * R.h, i = obj ? region_index(x, y, R, g) : 0;
      const double *F = obj_fields + i;
      adjoint_cell_f64(g, x, y, fl, mu, obj ? F[D_TOT * nreg] : 0.0, obj ? F[D_JX * nreg] : 0.0,
                       obj ? F[D_JY * nreg] : 0.0, out, t, bx, by);
    }
    const double sx = sines[y], sy = sines[g.ny + x];
    acc[0] += t * g.omega * g.omega;  // / tau^2
    acc[1] += bx * sx + by * sy;
#pragma unroll
    for (int l = 0; l < kQ; ++l) lam_out[(size_t)l * N + c] = out[l];
  }
  block_sums<2>(acc, partials + 2 * blockIdx.x, 1);
}

// Adds every partial into the two accumulators: thread i sums the partials
// i, i + 256, ... in order, then a fixed-order tree in shared memory (the
// same order every call: block-deterministic).
__global__ void __launch_bounds__(256) k_adjoint_final(const double *p_step, int nb,
                                                       const double *p_tau, int nbo,
                                                       const double *p_F0, int nbr, int with_obj,
                                                       double *dJ_dtau, double *dJ_dF0) {
  __shared__ double sa[256], sb[256];
  const int t = threadIdx.x;
  double a = 0.0, b = 0.0;
  for (int i = t; i < nb; i += 256) {
    a += p_step[2 * i];
    b += p_step[2 * i + 1];
  }
  if (with_obj) {
    for (int i = t; i < nbo; i += 256) a += p_tau[i];
    for (int i = t; i < nbr; i += 256) b += p_F0[i];
  }
  sa[t] = a;
  sb[t] = b;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (t < w) {
      sa[t] += sa[t + w];
      sb[t] += sb[t + w];
    }
    __syncthreads();
  }
  if (t == 0) {
    if (dJ_dtau) *dJ_dtau += sa[0];
    if (dJ_dF0) *dJ_dF0 += sb[0];
  }
}

// The forward objective in one launch of many CTAs.  The box is cut into
// TB x TB tiles; for each of its tiles a CTA computes rho and u = (j +
// F/2)/rho from the storage state `state` (the snapshot's moment arithmetic)
// on the tile widened by the 4-cell reach of the eq. (18) stencils (cells of
// the overlaps computed once per tile that needs them), keeps them in shared
// memory and sums the dissipation terms of the tile's box cells.  Each CTA
// writes one partial; the last CTA to finish (the arrival counter `count`,
// zero before the launch and reset by that CTA) sums the partials in a fixed
// order and adds cw times the sum to acc.  Small tiles for small boxes, a
// thread per cell of the widened tile and four lanes per box cell: the FP64
// work spreads over more SMs and its dependent chains stay short (GB300
// issues about 1.7 FP64 FMAs per clock per SM).
template <typename T, int TB, int NT>
__global__ void __launch_bounds__(NT)
    k_obj_tiles(const Member *__restrict__ members, int member, int state, AGrid g, int bx,
                int by, int L, double cw, double *partials, unsigned *count, double *acc) {
  constexpr int W = TB + 8, NC = W * W;
  __shared__ double sr[NC], su[NC], sv[NC];
  __shared__ double sw[NT / 32];
  __shared__ int is_last;
  const Member &M = members[member];
  const T *src = static_cast<const T *>(state_buffer(M, state));
  const int tid = threadIdx.x, ntx = (L + TB - 1) / TB, nt = ntx * ntx;
  double a = 0.0;
  for (int t = blockIdx.x; t < nt; t += gridDim.x) {
    const int ox = (t % ntx) * TB, oy = (t / ntx) * TB;  // tile origin within the box
    __syncthreads();  // the previous tile's reads of shared memory are done
    for (int i = tid; i < NC; i += NT) {
      const int x = wrapi(bx + ox - 4 + i % W, g.nx), y = wrapi(by + oy - 4 + i / W, g.ny);
      T f[kQ];
#pragma unroll
      for (int l = 0; l < kQ; ++l) f[l] = src[pub_index(M, state, l, x, y)];
      double r, jx, jy;
      pub_moments<T>(f, M.rho0, r, jx, jy);
      const double Fx = g.fxt[y] - g.alpha * jx, Fy = g.fyt[x] - g.alpha * jy;
      const double ir = 1.0 / r;
      sr[i] = r;
      su[i] = (jx + 0.5 * Fx) * ir;
      sv[i] = (jy + 0.5 * Fy) * ir;
    }
    __syncthreads();
    // the tile's box cells, four lanes per cell (d/dx u, d/dy u, d/dx v,
    // d/dy v), whole warps per pass so that every shuffle has the full warp
    const int lane = tid & 31, p = lane & 3, qb = lane & ~3;
    for (int i0 = (tid >> 5) * 8; i0 < TB * TB; i0 += (NT / 32) * 8) {
      const int iq = i0 + (lane >> 2), i = iq < TB * TB ? iq : TB * TB - 1;
      const int lx = i % TB, ly = i / TB;
      const int c = (ly + 4) * W + lx + 4, s = (p & 1) ? W : 1;
      const double *A = p < 2 ? su : sv;
      const double d = 0.8 * (A[c + s] - A[c - s]) - 0.2 * (A[c + 2 * s] - A[c - 2 * s]) +
                       (4.0 / 105.0) * (A[c + 3 * s] - A[c - 3 * s]) -
                       (1.0 / 280.0) * (A[c + 4 * s] - A[c - 4 * s]);
      const double dxu = __shfl_sync(0xffffffffu, d, qb), dyu = __shfl_sync(0xffffffffu, d, qb + 1);
      const double dxv = __shfl_sync(0xffffffffu, d, qb + 2), dyv = __shfl_sync(0xffffffffu, d, qb + 3);
      if (p == 0 && iq < TB * TB && ox + lx < L && oy + ly < L) {
        const double sxx = 2 * dxu, sxy = dyu + dxv, syy = 2 * dyv;
        a += -g.nu * sr[c] * (sxx * dxu + sxy * dyu + sxy * dxv + syy * dyv);
      }
    }
  }
  // the CTA's partial: shuffle tree per warp, warps in order
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
  if ((tid & 31) == 0) sw[tid >> 5] = a;
  __syncthreads();
  if (tid == 0) {
    double p = 0.0;
    for (int w = 0; w < NT / 32; ++w) p += sw[w];
    partials[blockIdx.x] = p;
    __threadfence();
    is_last = atomicAdd(count, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  // last CTA: strided fixed-order chains, the same tree
  double b = 0.0;
  for (int k = tid; k < (int)gridDim.x; k += NT) b += __ldcg(partials + k);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) b += __shfl_down_sync(0xffffffffu, b, o);
  __syncthreads();
  if ((tid & 31) == 0) sw[tid >> 5] = b;
  __syncthreads();
  if (tid == 0) {
    double p = 0.0;
    for (int w = 0; w < NT / 32; ++w) p += sw[w];
    *acc += cw * p;
    *count = 0u;
  }
}

template <typename T>
cudaError_t launch_obj_tiles(const Member *d_members, int member, int state, const AGrid &g,
                             int bx, int by, int L, double cw, double *partials,
                             unsigned *count, double *acc, cudaStream_t s) {
  // the largest tile that still gives a CTA to every SM, 4 x 4 at least;
  // a thread per cell of the widened tile ((TB + 8)^2 rounded up to warps)
  // for the latency-bound small tiles, 256 threads for 16 x 16 tiles, whose
  // many CTAs keep the FP64 pipes busy (L = 256 on 256^2: 28.8 us against
  // 30.8 with 576 threads)
  auto tiles = [&](int tb) { return (long long)((L + tb - 1) / tb) * ((L + tb - 1) / tb); };
  const int tb = tiles(16) >= 152 ? 16 : tiles(8) >= 152 ? 8 : 4;
  const int grid = (int)std::min<long long>(tiles(tb), kMaxPartialBlocks);
  if (tb == 16)
    k_obj_tiles<T, 16, 256><<<grid, 256, 0, s>>>(d_members, member, state, g, bx, by, L, cw,
                                                 partials, count, acc);
  else if (tb == 8)
    k_obj_tiles<T, 8, 256><<<grid, 256, 0, s>>>(d_members, member, state, g, bx, by, L, cw,
                                                partials, count, acc);
  else
    k_obj_tiles<T, 4, 160><<<grid, 160, 0, s>>>(d_members, member, state, g, bx, by, L, cw,
                                                partials, count, acc);
  return cudaGetLastError();
}

AGrid agrid(const Member &hm, const FixedBgk &fixed) {
  AGrid g;
  g.nx = hm.nx;
  g.ny = hm.ny;
  g.kf = hm.kf;
  g.force = hm.force_kind;
  g.nu = hm.nu;
  g.alpha = hm.alpha;
  g.tau = hm.tau;
  g.omega = hm.omega;
  g.F0 = hm.F0;
  g.fxt = hm.fx_tab64;
  g.fyt = hm.fy_tab64;
  g.fixed = fixed;
  g.fixed.ok = g.fixed.ok && std::abs(g.fixed.k) < 100 && std::fabs(hm.omega - 1.0) < 1.0 - 1e-9;
  g.w1 = g.fixed.ok ? std::llrint(std::ldexp(hm.omega - 1.0, 63)) : 0;
  g.keep = -g.w1;
  return g;
}

int nblocks_for(size_t N, int threads = 256) {
  size_t b = (N + threads - 1) / threads;
  return (int)(b > (size_t)kMaxPartialBlocks ? kMaxPartialBlocks : (b < 1 ? 1 : b));
}

// CTA size of the objective kernels of an adjoint step: their few hundred
// to few thousand cells of FP64 work spread over as many SMs as possible
// (GB300 issues about 1.7 FP64 FMAs per clock per SM).  A 100-level sweep
// of 256^2 with every other level weighted (L = 16): 42.8 us per level with
// 32-thread CTAs, 44.4 with 256 threads, 52.0 with the three kernels in one
// single-CTA launch.
constexpr int kObjThreads = 32;

// CTA size of k_adjoint: 64 threads below 2^17 cells, so that a small
// grid's FP64 work spreads evenly over the SMs (256^2: 44.3 against 46.2 us
// per adjoint step with 256-thread CTAs in 1.7 waves), 256 above.
int adjoint_threads(size_t N) { return N < ((size_t)1 << 17) ? 64 : 256; }

}  // namespace

cudaError_t adjoint_step(const Member &hm, const FixedBgk &fixed, const double *f_n, const double *lam_in,
                         double *lam_out, double w, int bx, int by, int L, double *dJ_dtau,
                         double *dJ_dF0, const DiagScratch &sc, cudaStream_t s) {
  return adjoint_sweep(hm, fixed, f_n, 1, lam_in, lam_out, nullptr, &w, bx, by, L, dJ_dtau, dJ_dF0, sc, s,
                       nullptr);
}

int adjoint_kernel_count(double w) { return w != 0.0 ? 7 : 3; }

// The adjoint steps of states[nstates - 1] .. states[0] (each [9][ny][nx]),
// the adjoint ping-ponging between lam_out and lam_tmp so that the last
// (state 0) lands in lam_out; weights[k] (host) the objective weight of
// step k.  The objective's fields of a batch of levels (as many as the
// scratch holds) come from three launches before the batch's adjoint steps.
// Each CTA keeps running sums of its (dJ/dtau, dJ/dF0) partials over the
// whole sweep and one reduction at the end adds them into the accumulators;
// the force-direction tables are built once.
cudaError_t adjoint_sweep(const Member &hm, const FixedBgk &fixed, const double *states, int nstates,
                          const double *lam_in, double *lam_out, double *lam_tmp,
                          const double *weights, int bx, int by, int L, double *dJ_dtau,
                          double *dJ_dF0, const DiagScratch &sc, cudaStream_t s,
                          long long *launches) {
  const AGrid g = agrid(hm, fixed);
  const size_t N = (size_t)hm.nx * hm.ny;
  const int tpb = adjoint_threads(N), nb = nblocks_for(N, tpb);
  double *sines = sc.f, *fields = sc.f + (hm.nx + hm.ny);
  double *p_step = sc.partials;                    // [nb][2]
  double *p_tau = p_step + 2 * kMaxPartialBlocks;  // the objective's running sums
  double *p_F0 = p_tau + kMaxPartialBlocks;
  int any_obj = 0;
  for (int k = 0; k < nstates; ++k) any_obj |= weights[k] != 0.0;
  const Region R = any_obj ? objective_region(hm.nx, hm.ny, bx, by, L) : Region{0, 0, 1, 1};
  const size_t nreg = (size_t)R.w * R.h;
  const int nbv = nblocks_for(nreg, kObjThreads);
  const int nbr = any_obj ? nblocks_for(4 * nreg, kObjThreads) : 1;  // four lanes per cell
  const int nbo = any_obj ? nblocks_for(4 * (size_t)L * L, kObjThreads) : 1;
  // per level: the fields and the two passes' partials
  const size_t per = kObjFields * nreg + nbr + nbo;
  const size_t room = (size_t)kDiagFields * sc.N - (hm.nx + hm.ny);
  const int batch = (int)std::min<size_t>({room / per, (size_t)kObjLevels, (size_t)nstates});
  if (any_obj && batch < 1) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(p_step, 0, sizeof(double) * 4 * kMaxPartialBlocks, s);
  if (e != cudaSuccess) return e;
  k_sine_tables<<<(hm.nx + hm.ny + 255) / 256, 256, 0, s>>>(g, sines);
  long long n = 2;
  const double *in = lam_in;
  for (int hi = nstates; hi > 0;) {
    const int lo = any_obj ? std::max(0, hi - batch) : 0, cnt = hi - lo;
    if (any_obj) {
      ObjWeights W{};
      bool some = false;
      for (int q = 0; q < cnt; ++q) {
        W.cw[q] = weights[lo + q] / ((double)L * (double)L);
        some |= W.cw[q] != 0.0;
      }
      if (some) {
        double *pt = fields + (size_t)cnt * kObjFields * nreg, *pf = pt + (size_t)cnt * nbo;
        const double *f0 = states + (size_t)lo * kQ * N;
        k_region_velocity<<<dim3(nbv, cnt), kObjThreads, 0, s>>>(g, R, f0, fields, W);
        k_obj_gamma<<<dim3(nbo, cnt), kObjThreads, 0, s>>>(g, R, fields, W, bx, by, L, pt);
        k_obj_velocity_adjoint<<<dim3(nbr, cnt), kObjThreads, 0, s>>>(g, R, fields, W, sines, bx,
                                                                      by, L, pf);
        k_obj_sum<<<1, 256, 0, s>>>(pt, cnt * nbo, pf, cnt * nbr, p_tau, p_F0);
        n += 4;
      }
    }
    for (int k = hi - 1; k >= lo; --k) {
      double *out = (k % 2 == 0) ? lam_out : lam_tmp;
      k_adjoint<<<nb, tpb, 0, s>>>(g, R, states + (size_t)k * kQ * N, in, out, sines,
                                   weights[k] / ((double)L * (double)L) != 0.0
                                       ? fields + (size_t)(k - lo) * kObjFields * nreg
                                       : nullptr,
                                   p_step);
      n += 1;
      in = out;
    }
    hi = lo;
  }
  k_adjoint_final<<<1, 256, 0, s>>>(p_step, nb, p_tau, 1, p_F0, 1, any_obj, dJ_dtau, dJ_dF0);
  if (launches) *launches += n;
  return cudaGetLastError();
}

// Forward objective of the state in storage `state`: one launch.
cudaError_t objective_tiles(int precision, const Member *d_members, int member,
                            const Member &hm, int state, double w, int bx, int by, int L,
                            double *acc, const DiagScratch &sc, cudaStream_t s) {
  const AGrid g = agrid(hm, FixedBgk{});
  const double cw = w / ((double)L * (double)L);
  if (precision == 32)
    return launch_obj_tiles<float>(d_members, member, state, g, bx, by, L, cw, sc.partials,
                                   sc.count, acc, s);
  return launch_obj_tiles<double>(d_members, member, state, g, bx, by, L, cw, sc.partials,
                                  sc.count, acc, s);
}

}  // namespace lbm
