// physics.cuh -- pointwise physics of the preconditioned Navier-Stokes equations
// (Sections 2.1-2.3) in binary64: fluxes, the preconditioning matrix, and the
// Weiss-Smith/Turkel preconditioned Roe flux in a closed form.  Its tangents for
// the block assembly are in physics_tan.cuh, its double-word form in
// physics_dw.cuh.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace pmg {

struct Phys {
  double gamma;    // ratio of specific heats
  double gm1;      // gamma - 1
  double Cp;       // gamma / (gamma - 1) with R = 1
  double eps_min;  // kappa * Ma_inf when the cut-off is on, 0 otherwise
  double p_ref;    // device states hold p - p_ref (gauge pressure)
  double inv_gamma;  // 1 / gamma
  double inv_gm1;    // 1 / (gamma - 1)
  double inv_Cp;     // (gamma - 1) / gamma
  double mu;         // constant dynamic viscosity (0: Euler)
  double kT;         // heat conductivity mu Cp / Pr
  double nw[5];      // weights 1 / res_scale of the equations in the residual norm
  double qinf[5];    // free stream of far-field faces: (p absolute, u, v, T) in 2D,
                     // (p absolute, u, v, w, T) in 3D
  double wait_ns;    // bound of the bulk-copy waits (< 0: give up at once)
};

// Reciprocal.  On the device, division costs about ten FP64 FMAs on GB300;
// here the hardware approximation (PTX rcp.approx.ftz.f64, about 20 correct
// bits) is refined by two Newton-Raphson steps y <- y + y (1 - x y), each
// doubling the number of correct bits, to full FP64 accuracy (within an ulp
// or two of the correctly rounded quotient; the parity tests bound the
// effect on the residual).  Arguments here are normal numbers (T, p, eps^2,
// c' > 0).
__host__ __device__ inline double s_rcp(double x) {
#ifdef __CUDA_ARCH__
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double e = fma(-x, y, 1.0);
  y = fma(y, e, y);
  e = fma(-x, y, 1.0);
  return fma(y, e, y);
#else
  return 1.0 / x;
#endif
}
#ifdef __CUDACC__
// 1 / sqrt(x) (x normal, positive): the hardware approximation refined by two
// Newton steps, as s_rcp.
__device__ __forceinline__ double s_rsqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double e = fma(-x * y, y, 1.0);
  y = fma(0.5 * y, e, y);
  e = fma(-x * y, y, 1.0);
  return fma(0.5 * y, e, y);
}
#endif
__host__ __device__ inline double s_min(double a, double b) { return a <= b ? a : b; }
__host__ __device__ inline double s_max(double a, double b) { return a >= b ? a : b; }

// ---------------------------------------------------------------------------
// Inviscid fluxes (rho v, rho v v + p I, rho v H), R = 1.
// ---------------------------------------------------------------------------
//
// q holds the absolute pressure; pm is the pressure used in the momentum
// flux.  With gauge storage pm = p - p_ref: the constant p_ref contributes
// p_ref times the discrete metric identity, which vanishes wherever the
// discretisation preserves a uniform flow (straight elements, or curved
// elements with P >= geometry order), and leaving it out keeps the rounding
// of p ~ 1/Ma^2 out of the momentum residual (and, through the velocity
// updates, out of the H-weighted energy residual).
// Cartesian fluxes f (x) and g (y) of quadrilaterals at one point, with the
// density rho = p / T supplied by the caller.
__host__ __device__ inline void flux_xy_rho(const double q[4], double pm, double rho, const Phys& ph, double f[4],
                                            double g[4]) {
  double H = ph.Cp * q[3] + 0.5 * (q[1] * q[1] + q[2] * q[2]);
  double mx = rho * q[1], my = rho * q[2];
  f[0] = mx; f[1] = mx * q[1] + pm; f[2] = mx * q[2]; f[3] = mx * H;
  g[0] = my; g[1] = my * q[1]; g[2] = my * q[2] + pm; g[3] = my * H;
}

__host__ __device__ inline void flux_xy(const double q[4], double pm, const Phys& ph, double f[4], double g[4]) {
  flux_xy_rho(q, pm, q[0] * s_rcp(q[3]), ph, f, g);
}

// Conservative variables (rho, rho u, rho v, rho E).
__host__ __device__ inline void cons(const double q[4], const Phys& ph, double qc[4]) {
  double rho = q[0] / q[3];
  qc[0] = rho;
  qc[1] = rho * q[1];
  qc[2] = rho * q[2];
  qc[3] = rho * (q[3] * ph.inv_gm1 + 0.5 * (q[1] * q[1] + q[2] * q[2]));
}

// eps^2 with eps = min(1, max(eps_min, Ma)) (eq. eps_nonmove; eps_min = 0
// when the cut-off is off).
__host__ __device__ inline double eps2_of(const double q[4], const Phys& ph) {
  double ma2 = (q[1] * q[1] + q[2] * q[2]) / (ph.gamma * q[3]);
  double e2 = s_max(ph.eps_min * ph.eps_min, ma2);
  return s_min(1.0, e2);
}

// ---------------------------------------------------------------------------
// Preconditioned Roe flux (eq. invis_com) through the unit normal n times the
// face area dS, with every matrix at the arithmetic mean of the primitive states.
//
// Closed form used here.  With K = M^-1 Gamma (identity except K_pp = 1/eps^2
// and K_Tp = (1/eps^2 - 1)/(rho Cp)), Gamma = M K and
// Gamma^-1 A_n = K^-1 (M^-1 A_n).  In rotated primitive variables
// (p, u_n, u_t, T) the matrix K^-1 M^-1 A_n is block lower triangular: a 2x2
// acoustic block B on (p, u_n) with eigenvalues u_n' +- c', u_t decoupled
// with eigenvalue u_n, and the T row coupled to (p, u_n) through
// r = (-(1-eps^2) u_n/(rho Cp), eps^2 (gamma-1) T) with eigenvalue u_n.  So
// |B| = a0 I + a1 B (linear interpolation of |lambda| on the two acoustic
// eigenvalues), and the T row of |.| is r (|B| - |u_n|)(B - u_n)^-1 on
// (p, u_n) plus |u_n| on T.  The dissipation is then M K |.| dq_p.  In 3D both
// tangential components are decoupled like u_t, so their part of it is |u_n| times
// the tangential velocity jump, |u_n| (dv - (dv.n) n) in Cartesian form.
// ---------------------------------------------------------------------------
#ifdef __CUDACC__
// D = 2 or 3 dimensions, states (p absolute, velocity, T), dq = qp - qm formed by
// the caller, pgm and pgp the pressures of the momentum fluxes.  An FP64 warp
// instruction takes 64 cycles of its sub-partition on GB300 whatever the
// number of active lanes, so the count of FP64 instructions is the time: half
// the face area is folded into the mass fluxes, 1/T and 1/p come from one
// reciprocal, c' and 1/c' from one inverse square root, e2 (gamma - 1) T is
// Ur2 / Cp, and the velocity part of the dissipation is
// |u_n| dv + (z_u - |u_n| du_n) n (about 180 FP64 instructions in 3D; 215 with
// each reciprocal, root and rotation written out).
template <int D>
__device__ __forceinline__ void roe_jump_d(const double qm[D + 2], const double qp[D + 2], const double dq[D + 2],
                                           double pgm, double pgp, const double n[D], double dS, const Phys& ph,
                                           double out[D + 2]) {
  const double h = 0.5 * dS;
  double unm = qm[1] * n[0], unq = qp[1] * n[0], vvm = qm[1] * qm[1], vvp = qp[1] * qp[1];
#pragma unroll
  for (int c = 1; c < D; ++c) {
    unm = fma(qm[1 + c], n[c], unm);
    unq = fma(qp[1 + c], n[c], unq);
    vvm = fma(qm[1 + c], qm[1 + c], vvm);
    vvp = fma(qp[1 + c], qp[1 + c], vvp);
  }
  const double mm = qm[0] * s_rcp(qm[D + 1]) * (unm * h), mp = qp[0] * s_rcp(qp[D + 1]) * (unq * h);
  const double pn = (pgm + pgp) * h;
  double f[D + 2];
  f[0] = mm + mp;
#pragma unroll
  for (int c = 0; c < D; ++c) f[1 + c] = fma(mm, qm[1 + c], fma(mp, qp[1 + c], pn * n[c]));
  f[D + 1] = fma(mm, fma(ph.Cp, qm[D + 1], 0.5 * vvm), mp * fma(ph.Cp, qp[D + 1], 0.5 * vvp));
  // averaged state, formed from the jump
  const double dp = dq[0], dT = dq[D + 1];
  const double p = fma(0.5, dp, qm[0]), T = fma(0.5, dT, qm[D + 1]);
  double v[D], vv = 0.0, un = 0.0, dun = 0.0;
#pragma unroll
  for (int c = 0; c < D; ++c) {
    v[c] = fma(0.5, dq[1 + c], qm[1 + c]);
    vv = fma(v[c], v[c], vv);
    un = fma(v[c], n[c], un);
    dun = fma(dq[1 + c], n[c], dun);
  }
  const double r = s_rcp(p * T), iT = p * r, irho = T * (T * r), rho = p * iT;
  const double c2 = ph.gamma * T, ic2 = iT * ph.inv_gamma;
  const double e2 = s_min(1.0, s_max(ph.eps_min * ph.eps_min, vv * ic2));
  const double Ur2 = e2 * c2, ie2 = s_rcp(e2), iUr2 = ie2 * ic2;
  const double bun = (1.0 - e2) * un, hun = 0.5 * bun;
  const double x = fma(hun, hun, Ur2), y = s_rsqrt(x), g = x * y, hy = 0.5 * y;
  const double cpr = fma(hy, fma(-g, g, x), g);   // sqrt(x)
  const double uc = un - hun, lp = uc + cpr, lm = uc - cpr;
  const double aun = fabs(un), alp = fabs(lp);
  const double a1 = (alp - fabs(lm)) * hy, a0 = fma(-a1, lp, alp);
  const double rc2 = rho * c2, dpr = dp * irho, a1e = a1 * e2;
  const double zp = fma(a0, dp, a1e * fma(un, dp, rc2 * dun));
  const double zu = fma(a0, dun, a1 * fma(un, dun, dpr));
  const double w0 = rho * dun, w1 = fma(bun, dun, dpr) * iUr2, a0u = a0 - aun;
  const double y0 = fma(a0u, w0, a1e * fma(un, w0, rc2 * w1));
  const double y1 = fma(a0u, w1, a1 * fma(un, w1, dun));
  const double irCp = irho * ph.inv_Cp;
  const double xT = fma(aun, dT, fma(Ur2 * ph.inv_Cp, y1, -(bun * irCp) * y0));
  const double yp = zp * ie2, yT = fma(irCp, yp - zp, xT);
  const double drho = fma(-rho, yT, yp) * iT;
  const double zz = fma(-aun, dun, zu);
  double vx = ph.Cp * yT;
  out[0] = fma(-h, drho, f[0]);
#pragma unroll
  for (int c = 0; c < D; ++c) {
    const double xv = fma(aun, dq[1 + c], zz * n[c]);
    vx = fma(v[c], xv, vx);
    out[1 + c] = fma(-h, fma(v[c], drho, rho * xv), f[1 + c]);
  }
  const double H = fma(ph.Cp, T, 0.5 * vv);
  out[D + 1] = fma(-h, fma(rho, vx, fma(H, drho, -yp)), f[D + 1]);
}
#endif

// Gamma (eq. preconditioning, 2D rows) and M = dq_c/dq_p at one point,
// row-major 4x4.
__host__ __device__ inline void gamma_and_M(const double q[4], const Phys& ph, double G[16], double M[16]) {
  double p = q[0], u = q[1], v = q[2], T = q[3];
  double rho = p / T, rp = 1.0 / T, rT = -rho / T;
  double H = ph.Cp * T + 0.5 * (u * u + v * v);
  double e2 = eps2_of(q, ph);
  double Th = 1.0 / (e2 * ph.gamma * T) - rT / (rho * ph.Cp);
  double c0[4] = {1.0, u, v, H};
  for (int i = 0; i < 4; ++i) {
    G[i * 4 + 0] = Th * c0[i];
    M[i * 4 + 0] = rp * c0[i];
    G[i * 4 + 3] = rT * c0[i];
    M[i * 4 + 3] = rT * c0[i];
    G[i * 4 + 1] = G[i * 4 + 2] = M[i * 4 + 1] = M[i * 4 + 2] = 0.0;
  }
  G[12] -= 1.0; M[12] -= 1.0;
  G[5] = M[5] = rho;
  G[10] = M[10] = rho;
  G[13] = M[13] = rho * u;
  G[14] = M[14] = rho * v;
  G[15] += rho * ph.Cp;
  M[15] += rho * ph.Cp;
}

// Viscous fluxes (Section 2.1, constant mu) in x and y from the velocity and
// the gradients g = (du/dx, dv/dx, dT/dx, du/dy, dv/dy, dT/dy):
// tau_ij = mu (du_i/dx_j + du_j/dx_i) - (2/3) mu div(u) delta_ij, and the
// energy flux u_i tau_ij - K_j with K_j = -kT dT/dx_j.  Mass rows are zero.
__host__ __device__ inline void viscous_flux(double u, double v, const double g[6], const Phys& ph, double fv[4], double gv[4]) {
  const double div3 = (g[0] + g[4]) * (2.0 / 3.0);
  const double txx = ph.mu * (2.0 * g[0] - div3);
  const double tyy = ph.mu * (2.0 * g[4] - div3);
  const double txy = ph.mu * (g[3] + g[1]);
  fv[0] = 0.0;
  fv[1] = txx;
  fv[2] = txy;
  fv[3] = u * txx + v * txy + ph.kT * g[2];
  gv[0] = 0.0;
  gv[1] = txy;
  gv[2] = tyy;
  gv[3] = u * txy + v * tyy + ph.kT * g[5];
}

}  // namespace pmg
