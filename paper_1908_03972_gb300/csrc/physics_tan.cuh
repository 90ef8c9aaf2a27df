// physics_tan.cuh -- exact tangents of the inviscid fluxes for the block
// assembly (Section 2.4, eq. smoothing_element_jacobi), D = 2 or 3 dimensions,
// states (p absolute, velocity, T).
//
// The assembly needs, per face point, D + 2 directional derivatives of the
// preconditioned Roe flux.  Dual numbers pushed through the flux repeat the
// value for every direction and multiply by the zero parts of their seeds;
// here the value's intermediates are formed once (RoeLin) and each direction
// is the hand-written tangent of the same closed form (physics.cuh
// roe_jump_d), about 200 FP64 instructions instead of about 700.
#pragma once
#include "physics.cuh"

namespace pmg {

#ifdef __CUDACC__

// Tangent of the inviscid flux through n at q along t; pm's tangent is t[0]
// (the gauge shift is constant).
template <int D>
__device__ __forceinline__ void flux_tangent(const double q[D + 2], const double n[D], const double t[D + 2],
                                             const Phys& ph, double out[D + 2]) {
  const double iT = s_rcp(q[D + 1]), rho = q[0] * iT;
  double un = 0.0, tun = 0.0, vv = 0.0, vt = 0.0;
#pragma unroll
  for (int c = 0; c < D; ++c) {
    un = fma(q[1 + c], n[c], un);
    tun = fma(t[1 + c], n[c], tun);
    vv = fma(q[1 + c], q[1 + c], vv);
    vt = fma(q[1 + c], t[1 + c], vt);
  }
  const double H = fma(ph.Cp, q[D + 1], 0.5 * vv), tH = fma(ph.Cp, t[D + 1], vt);
  const double trho = fma(-rho, t[D + 1], t[0]) * iT;
  const double mn = rho * un, tmn = fma(rho, tun, trho * un);
  out[0] = tmn;
#pragma unroll
  for (int c = 0; c < D; ++c) out[1 + c] = fma(tmn, q[1 + c], fma(mn, t[1 + c], t[0] * n[c]));
  out[D + 1] = fma(tmn, H, mn * tH);
}

// Intermediates of the Roe dissipation at the mean state (roe_jump_d).
template <int D>
struct RoeLin {
  double n[D], v[D], dv[D];
  double dp, dT, T, un, dun, iT, irho, rho, c2, ic2, vv, e2, ie2, Ur2, iUr2, bun, hun, y, lp, lm, a1, a0, rc2, dpr,
      a1e, s1, s2, w0, s3, w1, a0u, s4, y0, s5, y1, irCp, t1, UrC, yz, yT, drho, xv[D], vx, H, zp, aun, sun;
  bool act;   // eps^2 follows the local Mach number

  __device__ __forceinline__ void init(const double qm[D + 2], const double qp[D + 2], const double nn[D],
                                       const Phys& ph) {
    dp = qp[0] - qm[0];
    dT = qp[D + 1] - qm[D + 1];
    const double p = fma(0.5, dp, qm[0]);
    T = fma(0.5, dT, qm[D + 1]);
    vv = un = dun = 0.0;
#pragma unroll
    for (int c = 0; c < D; ++c) {
      n[c] = nn[c];
      dv[c] = qp[1 + c] - qm[1 + c];
      v[c] = fma(0.5, dv[c], qm[1 + c]);
      vv = fma(v[c], v[c], vv);
      un = fma(v[c], n[c], un);
      dun = fma(dv[c], n[c], dun);
    }
    const double r = s_rcp(p * T);
    iT = p * r;
    irho = T * (T * r);
    rho = p * iT;
    c2 = ph.gamma * T;
    ic2 = iT * ph.inv_gamma;
    const double m2 = vv * ic2, em = ph.eps_min * ph.eps_min;
    const double mx = s_max(em, m2);
    e2 = s_min(1.0, mx);
    act = !(em >= m2) && !(1.0 <= mx);   // the branch s_max and s_min take
    Ur2 = e2 * c2;
    ie2 = s_rcp(e2);
    iUr2 = ie2 * ic2;
    bun = (1.0 - e2) * un;
    hun = 0.5 * bun;
    const double x = fma(hun, hun, Ur2);
    y = s_rsqrt(x);
    const double g = x * y, cpr = fma(0.5 * y, fma(-g, g, x), g), uc = un - hun;
    lp = uc + cpr;
    lm = uc - cpr;
    aun = fabs(un);
    sun = un < 0.0 ? -1.0 : 1.0;
    const double alp = fabs(lp);
    a1 = (alp - fabs(lm)) * (0.5 * y);
    a0 = fma(-a1, lp, alp);
    rc2 = rho * c2;
    dpr = dp * irho;
    a1e = a1 * e2;
    s1 = fma(un, dp, rc2 * dun);
    zp = fma(a0, dp, a1e * s1);
    s2 = fma(un, dun, dpr);
    const double zu = fma(a0, dun, a1 * s2);
    w0 = rho * dun;
    s3 = fma(bun, dun, dpr);
    w1 = s3 * iUr2;
    a0u = a0 - aun;
    s4 = fma(un, w0, rc2 * w1);
    y0 = fma(a0u, w0, a1e * s4);
    s5 = fma(un, w1, dun);
    y1 = fma(a0u, w1, a1 * s5);
    irCp = irho * ph.inv_Cp;
    t1 = bun * irCp;
    UrC = Ur2 * ph.inv_Cp;
    const double xT = fma(aun, dT, fma(UrC, y1, -t1 * y0));
    const double yp = zp * ie2;
    yz = yp - zp;
    yT = fma(irCp, yz, xT);
    drho = fma(-rho, yT, yp) * iT;
    const double zz = fma(-aun, dun, zu);
    vx = ph.Cp * yT;
#pragma unroll
    for (int c = 0; c < D; ++c) {
      xv[c] = fma(aun, dv[c], zz * n[c]);
      vx = fma(v[c], xv[c], vx);
    }
    H = fma(ph.Cp, T, 0.5 * vv);
  }

  // Tangent of the dissipation M K |.| dq along tq (mean state: p, velocity,
  // T) and jq (jump).
  __device__ __forceinline__ void tangent(const double tq[D + 2], const double jq[D + 2], const Phys& ph,
                                          double out[D + 2]) const {
    const double tp = tq[0], tT = tq[D + 1], jp = jq[0], jT = jq[D + 1];
    double tvv = 0.0, tun = 0.0, jun = 0.0;
#pragma unroll
    for (int c = 0; c < D; ++c) {
      tvv = fma(v[c], tq[1 + c], tvv);
      tun = fma(n[c], tq[1 + c], tun);
      jun = fma(n[c], jq[1 + c], jun);
    }
    tvv *= 2.0;
    const double trho = fma(-rho, tT, tp) * iT, tiT = -(iT * iT) * tT;
    const double tirho = -(irho * irho) * trho, tc2 = ph.gamma * tT;
    const double te2 = act ? fma(tvv, ic2, vv * (tiT * ph.inv_gamma)) : 0.0;
    const double tUr2 = fma(te2, c2, e2 * tc2);
    const double tbun = fma(1.0 - e2, tun, -te2 * un), thun = 0.5 * tbun;
    const double tcpr = (0.5 * y) * fma(2.0 * hun, thun, tUr2);
    const double tuc = tun - thun, tlp = tuc + tcpr, tlm = tuc - tcpr;
    const double talp = lp < 0.0 ? -tlp : tlp, talm = lm < 0.0 ? -tlm : tlm, taun = sun * tun;
    const double ta1 = y * fma(0.5, talp - talm, -a1 * tcpr);
    const double ta0 = fma(-ta1, lp, fma(-a1, tlp, talp));
    const double trc2 = fma(trho, c2, rho * tc2), tdpr = fma(jp, irho, dp * tirho);
    const double ta1e = fma(ta1, e2, a1 * te2);
    const double ts1 = fma(tun, dp, fma(un, jp, fma(trc2, dun, rc2 * jun)));
    const double tzp = fma(ta0, dp, fma(a0, jp, fma(ta1e, s1, a1e * ts1)));
    const double ts2 = fma(tun, dun, fma(un, jun, tdpr));
    const double tzu = fma(ta0, dun, fma(a0, jun, fma(ta1, s2, a1 * ts2)));
    const double tw0 = fma(trho, dun, rho * jun);
    const double ts3 = fma(tbun, dun, fma(bun, jun, tdpr));
    const double tw1 = iUr2 * fma(-w1, tUr2, ts3);
    const double ta0u = ta0 - taun;
    const double ts4 = fma(tun, w0, fma(un, tw0, fma(trc2, w1, rc2 * tw1)));
    const double ty0 = fma(ta0u, w0, fma(a0u, tw0, fma(ta1e, s4, a1e * ts4)));
    const double ts5 = fma(tun, w1, fma(un, tw1, jun));
    const double ty1 = fma(ta0u, w1, fma(a0u, tw1, fma(ta1, s5, a1 * ts5)));
    const double tirCp = tirho * ph.inv_Cp, tt1 = fma(tbun, irCp, bun * tirCp);
    const double txT = fma(taun, dT, fma(aun, jT, fma(tUr2 * ph.inv_Cp, y1, fma(UrC, ty1, -fma(tt1, y0, t1 * ty0)))));
    const double typ = ie2 * fma(-(zp * ie2), te2, tzp);
    const double tyT = fma(tirCp, yz, fma(irCp, typ - tzp, txT));
    const double tdrho = iT * fma(-drho, tT, fma(-trho, yT, fma(-rho, tyT, typ)));
    const double tzz = fma(-taun, dun, fma(-aun, jun, tzu));
    double tvx = ph.Cp * tyT;
    out[0] = tdrho;
#pragma unroll
    for (int c = 0; c < D; ++c) {
      const double txv = fma(taun, dv[c], fma(aun, jq[1 + c], tzz * n[c]));
      tvx = fma(tq[1 + c], xv[c], fma(v[c], txv, tvx));
      out[1 + c] = fma(tq[1 + c], drho, fma(v[c], tdrho, fma(trho, xv[c], rho * txv)));
    }
    const double tH = fma(ph.Cp, tT, 0.5 * tvv);
    out[D + 1] = fma(tH, drho, fma(H, tdrho, fma(trho, vx, fma(rho, tvx, -typ))));
  }
};
#endif  // __CUDACC__

}  // namespace pmg
