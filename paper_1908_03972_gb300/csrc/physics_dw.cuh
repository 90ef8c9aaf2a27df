// physics_dw.cuh -- the preconditioned Roe flux of physics.cuh (eq. invis_com, the
// same closed form in the arrangement of roe_jump_d) in double-word arithmetic
// (dword.cuh), for the residual kernels.  GB300's FP64 rate (2 lanes per
// clock per SM) bounds the face-flux and sweep kernels; the same flux on the
// FP32 pipes runs several times faster at ~2^-46 relative rounding.
//
// The jumps dq arrive already formed in binary64 relative to a common
// reference (see line_trace in k_residual.cu): their double-word copies keep
// the low-Mach cancellation p+ - p- out of this arithmetic entirely.
#pragma once
#include "dword.cuh"
#include "physics.cuh"

namespace pmg {

// Double-word copies of the gas constants (filled on the host).
struct PhysW {
  dw gamma, Cp, inv_gamma, inv_Cp, eps_min2;
  dw p_ref;     // gauge reference pressure of the device states
  dw inv_gm1;   // 1 / (gamma - 1)
  double wait_ns;   // bound of the bulk-copy waits (< 0: give up at once)
};

// Double-word copies of a level's 1D operators (see OpTab).
struct OpTabW {
  dw Dt[6][6];            // D - gL lm^T - gR lp^T
  dw gL[6], gR[6];
};

inline PhysW make_physw(const Phys& ph) {
  PhysW k;
  k.gamma = dw_const(ph.gamma);
  k.Cp = dw_const(ph.Cp);
  k.inv_gamma = dw_const(ph.inv_gamma);
  k.inv_Cp = dw_const(1.0 / ph.Cp);
  k.eps_min2 = dw_const(ph.eps_min * ph.eps_min);
  k.p_ref = dw_const(ph.p_ref);
  k.inv_gm1 = dw_const(ph.inv_gm1);
  k.wait_ns = ph.wait_ns;
  return k;
}

#ifdef __CUDACC__
__device__ __forceinline__ dw half(dw x) { return scale2(x, 0.5f); }
__device__ __forceinline__ dw one_minus(dw x) { return dw{1.0f, 0.0f} - x; }

// roe_jump_d<2> of physics.cuh in double-word, without the pressure part
// (pm^- + pm^+)/2 n dS of the central momentum flux: qm, qp hold absolute
// pressure, dq = qp - qm (formed by the caller), (nx, ny) is the unit normal
// and dS the face area.  The pressure part is the one large term of the
// momentum rows (p ~ 1/(gamma Ma^2) when the absolute pressure is stored);
// the caller adds it.  The arrangement is roe_jump_d's (half the area in the
// mass fluxes) with sums of products renormalised once: about 1100 FP32
// operations, 1400 as separate products and sums.  64 elements (one GB300,
// launches of one warp's latency): the fused P = 0 sweep 7.6 -> 5.4 us, the P = 1
// face and update launches 5.2 -> 4.3 and 6.4 -> 4.7 us, with the geometry kept in
// double-word and the states formed on the FP32 pipes.
__device__ __forceinline__ void roe_flux_jump_dw(const dw qm[4], const dw qp[4], const dw dq[4], dw nx, dw ny,
                                                 dw dS, const PhysW& k, dw out[4]) {
  const dw h = half(dS);
  const dw mm = (qm[0] * rcp(qm[3])) * (dot2(qm[1], nx, qm[2], ny) * h);
  const dw mp = (qp[0] * rcp(qp[3])) * (dot2(qp[1], nx, qp[2], ny) * h);
  const dw Hm = mul_add(k.Cp, qm[3], half(dot2(qm[1], qm[1], qm[2], qm[2])));
  const dw Hp = mul_add(k.Cp, qp[3], half(dot2(qp[1], qp[1], qp[2], qp[2])));
  const dw f[4] = {mm + mp, dot2(mm, qm[1], mp, qp[1]), dot2(mm, qm[2], mp, qp[2]), dot2(mm, Hm, mp, Hp)};
  const dw dp = dq[0], du = dq[1], dv = dq[2], dT = dq[3];
  const dw p = qm[0] + half(dp);
  const dw u = qm[1] + half(du);
  const dw v = qm[2] + half(dv);
  const dw T = qm[3] + half(dT);
  const dw iT = rcp(T), irho = T * rcp(p), rho = p * iT;   // not through 1/(p T), which leaves the FP32 range first
  const dw c2 = k.gamma * T, ic2 = iT * k.inv_gamma;
  const dw vv = dot2(u, u, v, v);
  const dw e2 = min_dw(dw{1.0f, 0.0f}, max_dw(k.eps_min2, vv * ic2));
  const dw Ur2 = e2 * c2;
  const dw ie2 = rcp(e2), iUr2 = ie2 * ic2;
  const dw un = dot2(u, nx, v, ny);
  const dw dun = dot2(du, nx, dv, ny);
  const dw bun = one_minus(e2) * un, hun = half(bun);
  const dw cpr = sqrt_dw(mul_add(hun, hun, Ur2));
  const dw uc = un - hun;
  const dw lp = uc + cpr, lm = uc - cpr;
  const dw alp = abs_dw(lp), aun = abs_dw(un);
  const dw a1 = (alp - abs_dw(lm)) * half(rcp(cpr));
  const dw a0 = mul_add(-a1, lp, alp);
  const dw rc2 = rho * c2, dpr = dp * irho, a1e = a1 * e2;
  // |B| (dp, dun)
  const dw zp = dot2(a0, dp, a1e, dot2(un, dp, rc2, dun));
  const dw zu = dot2(a0, dun, a1, mul_add(un, dun, dpr));
  // w = (B - u_n)^-1 (dp, dun), y = (|B| - |u_n|) w
  const dw w0 = rho * dun, w1 = mul_add(bun, dun, dpr) * iUr2;
  const dw a0u = a0 - aun;
  const dw y0 = dot2(a0u, w0, a1e, dot2(un, w0, rc2, w1));
  const dw y1 = dot2(a0u, w1, a1, mul_add(un, w1, dun));
  const dw irCp = irho * k.inv_Cp;
  const dw xT = dot3(aun, dT, Ur2 * k.inv_Cp, y1, -(bun * irCp), y0);
  // K then M
  const dw yp = zp * ie2;
  const dw yT = mul_add(irCp, yp - zp, xT);
  const dw drho = mul_add(-rho, yT, yp) * iT;
  const dw zz = mul_add(-aun, dun, zu);
  const dw xu = dot2(aun, du, zz, nx), xv = dot2(aun, dv, zz, ny);
  const dw H = mul_add(k.Cp, T, half(vv));
  const dw vx = dot3(u, xu, v, xv, k.Cp, yT);
  out[0] = mul_add(-h, drho, f[0]);
  out[1] = mul_add(-h, dot2(u, drho, rho, xu), f[1]);
  out[2] = mul_add(-h, dot2(v, drho, rho, xv), f[2]);
  out[3] = mul_add(-h, dot2_add(H, drho, rho, vx, -yp), f[3]);
}

// States of one face point in double-word from its binary64 parts: the own
// trace sm and the jump dq, both relative to the reference state (ref: p and T;
// the velocity's reference is zero).  The sums run on the FP32 pipes: an FP64
// instruction takes as long as 16 of theirs.  pg receives the gauge pressures'
// sum p^- + p^+.
__device__ __forceinline__ void face_states_dw(double ref_p, double ref_T, const double sm[4], const double dq[4],
                                               const PhysW& k, dw Qm[4], dw Qp[4], dw DQ[4], dw& pg) {
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    Qm[v] = dw_from_double(sm[v]);
    DQ[v] = dw_from_double(dq[v]);
  }
  const dw P = dw_from_double(ref_p) + Qm[0];
  Qm[3] = dw_from_double(ref_T) + Qm[3];
  pg = scale2(P, 2.0f) + DQ[0];
  Qm[0] = P + k.p_ref;
#pragma unroll
  for (int v = 0; v < 4; ++v) Qp[v] = Qm[v] + DQ[v];
}

// Common Roe flux of one face point from binary64 traces; DWF selects the
// double-word evaluation (above; the central pressure term in binary64)
// over the binary64 one.  ref, sm, dq as in face_states_dw; sp = sm + dq.
template <bool DWF>
__device__ __forceinline__ void face_roe(const double ref[4], const double sm[4], const double sp[4],
                                         const double dq[4], double nx, double ny, double dS, const Phys& ph,
                                         const PhysW& phw, double out[4]) {
  if (DWF) {
    dw Qm[4], Qp[4], DQ[4], o[4], pg;
    face_states_dw(ref[0], ref[3], sm, dq, phw, Qm, Qp, DQ, pg);
    roe_flux_jump_dw(Qm, Qp, DQ, dw_from_double(nx), dw_from_double(ny), dw_from_double(dS), phw, o);
    const double pc = ((ref[0] + sm[0]) + (ref[0] + sp[0])) * (0.5 * dS);
    out[0] = dw_to_double(o[0]);
    out[1] = fma(pc, nx, dw_to_double(o[1]));
    out[2] = fma(pc, ny, dw_to_double(o[2]));
    out[3] = dw_to_double(o[3]);
  } else {
    double qm[4], qp[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      qm[v] = ref[v] + sm[v];
      qp[v] = ref[v] + sp[v];
    }
    const double pgm = qm[0], pgp = qp[0], n[2] = {nx, ny};   // gauge pressures for the momentum fluxes
    qm[0] += ph.p_ref;   // absolute pressure for the averaged state and rho
    qp[0] += ph.p_ref;
    roe_jump_d<2>(qm, qp, dq, pgm, pgp, n, dS, ph, out);
  }
}
// The double-word face flux left in double-word, the central pressure term
// included (gauge storage, p - p_ref in the momentum rows).  (nx, ny, dS): the
// double-word face geometry; g, with PC64: the same in binary64, in which the
// pressure term is then formed and added, as face_roe does.  Where the pressure
// dominates the momentum flux its rounding is the row's: the largest error is
// 1.7 times as large in double-word (4.2e-12 against 2.4e-12 of rho u^2 at a
// gauge pressure of 300 rho u^2).  Without PC64 (the one-launch sweeps of P = 0
// levels) the term is double-word.
template <bool PC64>
__device__ __forceinline__ void face_roe_dw(double ref_p, double ref_T, const double sm[4], const double sp[4],
                                            const double dq[4], dw nx, dw ny, dw dS, const double g[3],
                                            const PhysW& phw, dw out[4]) {
  dw Qm[4], Qp[4], DQ[4], pg;
  face_states_dw(ref_p, ref_T, sm, dq, phw, Qm, Qp, DQ, pg);
  roe_flux_jump_dw(Qm, Qp, DQ, nx, ny, dS, phw, out);
  if (PC64) {
    const double pc = ((ref_p + sm[0]) + (ref_p + sp[0])) * (0.5 * g[2]);
    out[1] = dw_from_double(fma(pc, g[0], dw_to_double(out[1])));
    out[2] = dw_from_double(fma(pc, g[1], dw_to_double(out[2])));
  } else {
    const dw pc = half(pg * dS);
    out[1] = mul_add(pc, nx, out[1]);
    out[2] = mul_add(pc, ny, out[2]);
  }
}
#endif  // __CUDACC__

}  // namespace pmg
