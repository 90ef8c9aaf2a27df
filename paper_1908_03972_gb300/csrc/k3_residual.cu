// k3_residual.cu -- FR/CPR residual on hexahedra (Section 2.3 with d = 3),
// binary64.
//
// Same two-launch structure as the quadrilateral kernels (k_residual.cu):
//  * face_flux3: one thread per face point of the face list.  It extrapolates
//    both elements' solution polynomials along the lines normal to the face
//    (the neighbour's face point through the face's orientation code),
//    evaluates the preconditioned Roe flux through the face normal once and
//    writes it with opposite signs into both elements' face slots.  Boundary
//    faces take the ghost state of their type.
//  * volume3: one thread per solution point, EPB3 elements per CTA.  The
//    contravariant fluxes F^i = f . J a^i of the element's points go to
//    shared memory, the common fluxes of its faces by asynchronous copies; a
//    line's divergence is Dt F + gL F_com(-1) + gR F_com(+1), the derivative
//    with the extrapolated part of the correction folded in (OpTab::Dt), then
//    the epilogue of the requested mode, a deterministic per-CTA sum of squares
//    for the norm, and with APPLY the element-Jacobi update
//    q += cs .* D^-1 (rs .* (F - S)).
//
// All three kernels are bound by FP64 issue: a warp instruction takes 64 cycles
// of its sub-partition however many lanes are active, so what counts is FP64
// instructions per warp.  The face jumps are not formed (one extrapolation per
// face point and equation less), the corrected gradient adds only the face
// corrections to the broken gradient the gradient launch wrote (12 planes read
// instead of 36 derivative sums recomputed: 96 bytes against about 100 FP64
// instructions a point), the viscous and inviscid fluxes are joined as
// symmetric Cartesian tensors before the metric terms contract them, and the
// gradient launch subtracts one reference per element, once per value.
// Measured on 3,072 viscous hexahedra at P = 3 (one GB300): gradient 57 -> 38
// us, face flux 136 -> 114 us, residual 165 -> 108 us.
//
// Layout: states q[(v*E + e)*N + pt], v < 5, pt = (k*(P+1) + j)*(P+1) + i;
// metric planes met[c*E*N + e*N + pt], c = 3 i + n for J a^i_n, c = 9 for 1/J;
// face geometry face[((e*6 + f)*NF + fp)*4] = (unit outward normal, area);
// common fluxes Fcom[((v*E + e)*6 + f)*NF + fp], outward for element e.
#include "pmg_internal.h"

namespace pmg {

template <int P>
struct EPB3 {   // elements per CTA of the volume kernel: one or two warps per CTA
  static constexpr int value = P == 0 ? 32 : P == 1 ? 8 : P == 2 ? 2 : 1;
};

// Solution point at position m on the line normal to face f through face
// point (a, b).
template <int P>
__device__ __forceinline__ int line_pt3(int f, int a, int b, int m) {
  constexpr int n1 = P + 1;
  const int d = f >> 1;
  const int i = d == 0 ? m : a;
  const int j = d == 1 ? m : (d == 0 ? a : b);
  const int k = d == 2 ? m : b;
  return (k * n1 + j) * n1 + i;
}

// Trace of the solution polynomial at face point (a, b) of face f, minus ref.
template <int P>
__device__ __forceinline__ void line_trace3(const double* __restrict__ q, size_t plane, int e, int f, int a, int b,
                                            const double* lm, const double* lp, const double ref[5],
                                            double out[5]) {
  constexpr int n1 = P + 1, N = n1 * n1 * n1;
  const double* base = q + (size_t)e * N;
  const bool plus = f & 1;
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    double s = 0.0;
#pragma unroll
    for (int m = 0; m < n1; ++m)
      s = fma(plus ? lp[m] : lm[m], __ldg(base + v * plane + line_pt3<P>(f, a, b, m)) - ref[v], s);
    out[v] = s;
  }
}

// With VISC (mu > 0) the face launch also forms the viscous common flux of
// eq. com_grad_q at q_com: the mean of both sides' broken-gradient traces
// (Gb, extrapolated along each side's normal line; a boundary mirrors the
// element) plus the BR2 lifting pen (1/|J|^- + 1/|J|^+)/4 dS n (q^+ - q^-);
// walls carry no viscous energy flux.  It writes q_com - q_own of
// (u, v, w, T) for both elements (Qj), the jumps the volume launch's
// corrected gradient takes.
template <int P, bool VISC>
__global__ void __launch_bounds__(64) face_flux3_kernel(const int* __restrict__ faces, int n_faces, int E,
                                                        const double* __restrict__ q,
                                                        const double* __restrict__ face,
                                                        double* __restrict__ Fcom, OpTab op, Phys ph,
                                                        const double* __restrict__ Gb,
                                                        const double* __restrict__ fJinv,
                                                        double* __restrict__ Qj) {
  constexpr int n1 = P + 1, N = n1 * n1 * n1, NF = n1 * n1;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= n_faces * NF) return;
  const int fc = tid / NF, fp = tid - fc * NF;
  const int a = fp % n1, b = fp / n1;
  const int* fr = faces + fc * 5;
  const int eL = fr[0], fL = fr[1], eR = fr[2], fR = fr[3], o = fr[4];
  const bool bnd = eR < 0;
  const size_t plane = (size_t)E * N;
  double lm[n1], lp[n1];
#pragma unroll
  for (int m = 0; m < n1; ++m) { lm[m] = op.lm[m]; lp[m] = op.lp[m]; }
  const double ref[5] = {__ldg(q + (size_t)eL * N), 0.0, 0.0, 0.0, __ldg(q + 4 * plane + (size_t)eL * N)};
  const double* g = face + (((size_t)eL * 6 + fL) * NF + fp) * 4;
  const double nrm[3] = {__ldg(g), __ldg(g + 1), __ldg(g + 2)};
  const double dS = __ldg(g + 3);
  double sm[5], sp[5];
  line_trace3<P>(q, plane, eL, fL, a, b, lm, lp, ref, sm);
  int fp2 = fp;
  if (!bnd) {
    const int s = (o & 4) ? b : a, t = (o & 4) ? a : b;
    const int a2 = (o & 1) ? P - s : s, b2 = (o & 2) ? P - t : t;
    fp2 = b2 * n1 + a2;
    line_trace3<P>(q, plane, eR, fR, a2, b2, lm, lp, ref, sp);
  } else if (fR == PMG_BC_FARFIELD) {
    sp[0] = (ph.qinf[0] - ph.p_ref) - ref[0];
    sp[1] = ph.qinf[1];
    sp[2] = ph.qinf[2];
    sp[3] = ph.qinf[3];
    sp[4] = ph.qinf[4] - ref[4];
  } else if (fR == PMG_BC_NOSLIP_WALL) {   // same p and T, velocity reversed
    sp[0] = sm[0];
    sp[4] = sm[4];
#pragma unroll
    for (int c = 0; c < 3; ++c) sp[1 + c] = -sm[1 + c];
  } else {   // slip wall: same p and T, normal velocity reflected
    const double un = sm[1] * nrm[0] + sm[2] * nrm[1] + sm[3] * nrm[2];
    sp[0] = sm[0];
    sp[4] = sm[4];
#pragma unroll
    for (int c = 0; c < 3; ++c) sp[1 + c] = fma(-2.0 * un, nrm[c], sm[1 + c]);
  }
  double qm[5], qp[5], dq[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    qm[v] = ref[v] + sm[v];
    qp[v] = ref[v] + sp[v];
    dq[v] = sp[v] - sm[v];
  }
  const double pgm = qm[0], pgp = qp[0];
  qm[0] += ph.p_ref;
  qp[0] += ph.p_ref;
  double out[5];
  roe_jump_d<3>(qm, qp, dq, pgm, pgp, nrm, dS, ph, out);
  const size_t fplane = (size_t)E * 6 * NF;
  const size_t iL = ((size_t)eL * 6 + fL) * NF + fp;
  if (VISC) {
    // mean of both sides' broken-gradient traces (a boundary mirrors the
    // element), plus the lifting; at P = 0 the broken gradient is zero
    const double iJm = __ldg(fJinv + iL);
    const double iJp = bnd ? iJm : __ldg(fJinv + ((size_t)eR * 6 + fR) * NF + fp2);
    const double wl = 0.25 * op.pen * (iJm + iJp) * dS;
    double gc[12];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int k = 0; k < 4; ++k) gc[c * 4 + k] = (wl * nrm[c]) * dq[k + 1];
    if (P > 0) {
      const int a2 = fp2 % n1, b2 = fp2 / n1;
      const double* bL = Gb + (size_t)eL * N;
      const double* bR = Gb + (size_t)(bnd ? eL : eR) * N;
      const int fo = bnd ? fL : fR, ao = bnd ? a : a2, bo = bnd ? b : b2;
#pragma unroll
      for (int m = 0; m < n1; ++m) {
        const double wL = (fL & 1) ? op.hlp[m] : op.hlm[m], wR = (fo & 1) ? op.hlp[m] : op.hlm[m];
        const int iLp = line_pt3<P>(fL, a, b, m), iRp = line_pt3<P>(fo, ao, bo, m);
#pragma unroll
        for (int c = 0; c < 12; ++c) {
          gc[c] = fma(wL, __ldg(bL + c * plane + iLp), gc[c]);
          gc[c] = fma(wR, __ldg(bR + c * plane + iRp), gc[c]);
        }
      }
    }
    // viscous flux through n dS at q_com: mu (g + g^T) n - 2/3 mu div n, and
    // its work on u_com plus the heat flux
    const double mdS = ph.mu * dS, kdS = ph.kT * dS;
    const double d23 = (gc[0] + gc[5] + gc[10]) * (2.0 / 3.0);
    const double s01 = gc[1] + gc[4], s02 = gc[2] + gc[8], s12 = gc[6] + gc[9];
    double t[3];
    t[0] = fma(2.0 * gc[0] - d23, nrm[0], fma(s01, nrm[1], s02 * nrm[2]));
    t[1] = fma(2.0 * gc[5] - d23, nrm[1], fma(s01, nrm[0], s12 * nrm[2]));
    t[2] = fma(2.0 * gc[10] - d23, nrm[2], fma(s02, nrm[0], s12 * nrm[1]));
    double wk = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      out[1 + c] = fma(-mdS, t[c], out[1 + c]);
      wk = fma(fma(0.5, dq[1 + c], qm[1 + c]), t[c], wk);
    }
    const bool wall = bnd && fR != PMG_BC_FARFIELD;   // walls: no viscous energy flux
    const double ht = fma(gc[3], nrm[0], fma(gc[7], nrm[1], gc[11] * nrm[2]));
    if (!wall) out[4] = fma(-mdS, wk, fma(-kdS, ht, out[4]));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double hj = 0.5 * dq[k + 1];
      Qj[k * fplane + iL] = hj;
      if (!bnd) Qj[k * fplane + ((size_t)eR * 6 + fR) * NF + fp2] = -hj;
    }
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) Fcom[v * fplane + iL] = out[v];
  if (!bnd) {
    const size_t iR = ((size_t)eR * 6 + fR) * NF + fp2;
#pragma unroll
    for (int v = 0; v < 5; ++v) Fcom[v * fplane + iR] = -out[v];
  }
}

// One double by an asynchronous copy (8 bytes: the only alignment every
// caller's buffers have).
__device__ __forceinline__ void async_g2s(double* dst, const double* src) {
  const unsigned int d = (unsigned int)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// With VISC the contravariant fluxes take f_inv - f_vis: the viscous flux at
// each solution point from the corrected gradient, the broken gradient Gb plus
// the DG correction of the face jumps Qj on the two faces of each line through
// the point (eq. com_q), chain rule with the metric terms.
template <int P, class W, bool APPLY, bool VISC>
__global__ void __launch_bounds__(64) volume3_kernel(int E, const double* q, const double* __restrict__ met,
                                                     const double* __restrict__ Fcom, const double* __restrict__ Qj,
                                                     const double* Gb,
                                                     OpTab op, Phys ph,
                                                     double* __restrict__ out, int mode, double inv_odt,
                                                     const double* __restrict__ src, const double* __restrict__ S,
                                                     double* __restrict__ Sout, const double* __restrict__ Pd,
                                                     const double* __restrict__ qn, double* __restrict__ partial,
                                                     double* qw, const W* __restrict__ Dinv,
                                                     const double* __restrict__ rs, const double* __restrict__ cs,
                                                     double* Gnext) {
  // Gnext: leave the broken gradients of the updated state.  It is Gb itself (a
  // point's own entries, read before they are written), which is then neither
  // restricted nor read as constant.
  constexpr bool kGrad = APPLY && VISC && P > 0;
  constexpr int n1 = P + 1, N = n1 * n1 * n1, NF = n1 * n1, EPB = EPB3<P>::value, n = 5 * N;
  using Acc = typename Blk<W>::acc;
  __shared__ double sF[EPB][3][5][N];
  __shared__ double sC[5][EPB * 6 * NF];                        // common fluxes, outward
  __shared__ double sQ[VISC ? 4 : 1][VISC ? EPB * 6 * NF : 1];  // face jumps
  __shared__ Acc sr[APPLY ? EPB : 1][APPLY ? n : 1];
  __shared__ double sD[n1][n1], sgL[n1], sgR[n1];
  __shared__ double sDg[kGrad ? n1 : 1][kGrad ? n1 : 1];   // D
  __shared__ double sred[2];
  const int le = threadIdx.x / N, pt = threadIdx.x - le * N;
  const int e = blockIdx.x * EPB + le;
  const bool active = (le < EPB) && (e < E);
  const size_t plane = (size_t)E * N;
  const size_t fplane = (size_t)E * 6 * NF;
  {
    const int e0 = blockIdx.x * EPB, nf = min(EPB, E - e0) * 6 * NF;
    const size_t f0 = (size_t)e0 * 6 * NF;
    for (int t = threadIdx.x; t < nf; t += blockDim.x) {
      if (VISC)
#pragma unroll
        for (int k = 0; k < 4; ++k) async_g2s(&sQ[VISC ? k : 0][VISC ? t : 0], Qj + k * fplane + f0 + t);
#pragma unroll
      for (int v = 0; v < 5; ++v) async_g2s(&sC[v][t], Fcom + v * fplane + f0 + t);
    }
  }
  if (threadIdx.x < n1 * n1) {
    sD[threadIdx.x / n1][threadIdx.x % n1] = op.Dt[threadIdx.x / n1][threadIdx.x % n1];
    if (kGrad) sDg[kGrad ? threadIdx.x / n1 : 0][kGrad ? threadIdx.x % n1 : 0] = op.D[threadIdx.x / n1][threadIdx.x % n1];
  }
  if (threadIdx.x < n1) {
    sgL[threadIdx.x] = op.gL[threadIdx.x];
    sgR[threadIdx.x] = op.gR[threadIdx.x];
  }
  const size_t gi = (size_t)e * N + pt;
  const int i = pt % n1, j = (pt / n1) % n1, k = pt / (n1 * n1);
  const int fb = le * 6 * NF, fp0 = k * n1 + j, fp1 = k * n1 + i, fp2 = j * n1 + i;   // face points of the three lines
  double qq[5] = {0, 0, 0, 0, 0}, invJ = 0.0, rho_pt = 0.0;
  double ja[3][3], g[12];
  if (active) {
#pragma unroll
    for (int v = 0; v < 5; ++v) qq[v] = q[v * plane + gi];
    invJ = __ldg(met + 9 * plane + gi);
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int c = 0; c < 3; ++c) ja[d][c] = __ldg(met + (3 * d + c) * plane + gi);
    if (VISC && P > 0)
#pragma unroll
      for (int c = 0; c < 12; ++c) g[c] = kGrad ? Gb[c * plane + gi] : __ldg(Gb + c * plane + gi);
  }
  if (VISC) {
    async_wait_all();
    __syncthreads();
  }
  if (active) {
    const double pabs = qq[0] + ph.p_ref;
    rho_pt = pabs * s_rcp(qq[4]);
    if (VISC) {
      double sj[3][3];
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int c = 0; c < 3; ++c) sj[d][c] = invJ * ja[d][c];
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const double* Q = sQ[VISC ? w : 0] + (VISC ? fb : 0);
        const double c0 = fma(sgL[i], Q[fp0], sgR[i] * Q[NF + fp0]);
        const double c1 = fma(sgL[j], Q[2 * NF + fp1], sgR[j] * Q[3 * NF + fp1]);
        const double c2 = fma(sgL[k], Q[4 * NF + fp2], sgR[k] * Q[5 * NF + fp2]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const double t = fma(sj[0][c], c0, fma(sj[1][c], c1, sj[2][c] * c2));
          g[c * 4 + w] = P > 0 ? g[c * 4 + w] + t : t;
        }
      }
      // Cartesian fluxes: momentum T = rho u u + pm I - tau (symmetric),
      // energy rho u H - tau u - kT grad T
      const double H = fma(ph.Cp, qq[4], 0.5 * fma(qq[1], qq[1], fma(qq[2], qq[2], qq[3] * qq[3])));
      const double m2 = -2.0 * ph.mu, l23 = (ph.mu * (2.0 / 3.0)) * (g[0] + g[5] + g[10]);
      double m[3], T[3][3], tt[3][3], en[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        m[c] = rho_pt * qq[1 + c];
        tt[c][c] = fma(m2, g[c * 4 + c], l23);
        T[c][c] = fma(m[c], qq[1 + c], qq[0] + tt[c][c]);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int d = c + 1; d < 3; ++d) {
          tt[c][d] = tt[d][c] = -ph.mu * (g[c * 4 + d] + g[d * 4 + c]);
          T[c][d] = T[d][c] = fma(m[c], qq[1 + d], tt[c][d]);
        }
#pragma unroll
      for (int c = 0; c < 3; ++c)
        en[c] = fma(m[c], H, fma(-ph.kT, g[c * 4 + 3],
                                 fma(qq[1], tt[c][0], fma(qq[2], tt[c][1], qq[3] * tt[c][2]))));
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        sF[le][d][0][pt] = fma(ja[d][0], m[0], fma(ja[d][1], m[1], ja[d][2] * m[2]));
#pragma unroll
        for (int c = 0; c < 3; ++c)
          sF[le][d][1 + c][pt] = fma(ja[d][0], T[0][c], fma(ja[d][1], T[1][c], ja[d][2] * T[2][c]));
        sF[le][d][4][pt] = fma(ja[d][0], en[0], fma(ja[d][1], en[1], ja[d][2] * en[2]));
      }
    } else {
      const double H = fma(ph.Cp, qq[4], 0.5 * fma(qq[1], qq[1], fma(qq[2], qq[2], qq[3] * qq[3])));
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double mn = rho_pt * fma(qq[1], ja[d][0], fma(qq[2], ja[d][1], qq[3] * ja[d][2]));
        sF[le][d][0][pt] = mn;
#pragma unroll
        for (int c = 0; c < 3; ++c) sF[le][d][1 + c][pt] = fma(mn, qq[1 + c], qq[0] * ja[d][c]);
        sF[le][d][4][pt] = mn * H;
      }
    }
  }
  if (!VISC) async_wait_all();
  __syncthreads();
  double ssq = 0.0;
  if (active) {
    const double ninvJ = -invJ;
    double qc[5];
    if (qn) {
      // q_c(q) - q_c(q_ref) with the energy through the pressure difference
      double qo[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) qo[v] = __ldg(qn + v * plane + gi);
      const double rho = rho_pt, rhoo = (qo[0] + ph.p_ref) * s_rcp(qo[4]);
      qc[0] = rho - rhoo;
#pragma unroll
      for (int c = 1; c < 4; ++c) qc[c] = rho * qq[c] - rhoo * qo[c];
      qc[4] = (qq[0] - qo[0]) * ph.inv_gm1 +
              0.5 * (rho * (qq[1] * qq[1] + qq[2] * qq[2] + qq[3] * qq[3]) -
                     rhoo * (qo[1] * qo[1] + qo[2] * qo[2] + qo[3] * qo[3]));
    } else {
      qc[0] = rho_pt;
#pragma unroll
      for (int c = 1; c < 4; ++c) qc[c] = rho_pt * qq[c];
      qc[4] = rho_pt * (qq[4] * ph.inv_gm1 + 0.5 * (qq[1] * qq[1] + qq[2] * qq[2] + qq[3] * qq[3]));
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      double acc = 0.0;
#pragma unroll
      for (int m = 0; m < n1; ++m) {
        acc = fma(sD[i][m], sF[le][0][v][(k * n1 + j) * n1 + m], acc);
        acc = fma(sD[j][m], sF[le][1][v][(k * n1 + m) * n1 + i], acc);
        acc = fma(sD[k][m], sF[le][2][v][(m * n1 + j) * n1 + i], acc);
      }
      const double* C = sC[v] + fb;   // outward: the -1 side's reference-direction flux is its negative
      acc = fma(-sgL[i], C[fp0], acc);
      acc = fma(sgR[i], C[NF + fp0], acc);
      acc = fma(-sgL[j], C[2 * NF + fp1], acc);
      acc = fma(sgR[j], C[3 * NF + fp1], acc);
      acc = fma(-sgL[k], C[4 * NF + fp2], acc);
      acc = fma(sgR[k], C[5 * NF + fp2], acc);
      const double R = acc * ninvJ;
      const size_t o = v * plane + gi;
      if (mode == RES_PURE) {
        out[o] = R;
      } else if (mode == RES_FORCING) {
        const double Fraw = fma(-qc[v], inv_odt, R);
        const double pd = Pd[o];
        Sout[o] = Fraw + pd;
        out[o] = -pd;
        ssq = fma(pd, pd, ssq);
      } else {
        double F = fma(-qc[v], inv_odt, R);
        if (src) F += src[o];
        if (mode == RES_SYSTEM && S) F -= S[o];
        if (APPLY) sr[APPLY ? le : 0][APPLY ? v * N + pt : 0] = scaled_in<W>(F, rs[(size_t)e * n + v * N + pt]);
        else out[o] = F;
        if (partial) {
          const double Fw = F * ph.nw[v];
          ssq = fma(Fw, Fw, ssq);
        }
      }
    }
  }
  if (APPLY) {
    __syncthreads();
    if (active) {
      // thread (le, pt) forms the rows v N + pt (its own point) of D^-1 r;
      // the inverse is column-major, so the threads of an element read each
      // column's rows contiguously
      Acc acc[5] = {0, 0, 0, 0, 0};
      const W* Dm = Dinv + (size_t)e * n * n + pt;
#pragma unroll 10
      for (int kk = 0; kk < n; ++kk) {
        const Acc rk = sr[APPLY ? le : 0][APPLY ? kk : 0];
#pragma unroll
        for (int v = 0; v < 5; ++v) acc[v] = fma(blk_val(__ldg(Dm + (size_t)kk * n + v * N)), rk, acc[v]);
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const size_t o = v * plane + gi;
        qq[v] += scaled_out<W>(acc[v], cs[(size_t)e * n + v * N + pt]);
        qw[o] = qq[v];
      }
    }
    if (kGrad && Gnext) {
      // The operations of grad3_kernel on the updated state, which is here
      // already: 960 elements, sweep of P = 3 (FP32) 118 us with its gradient
      // launch, 108 without; P = 2 40.7 and 37.2, P = 1 19.4 and 17.5, a launch
      // gap less each.
      if (active && pt == 0) {
#pragma unroll
        for (int w = 0; w < 4; ++w) sF[le][0][w][0] = qq[1 + w];
      }
      __syncthreads();
      if (active) {
#pragma unroll
        for (int w = 0; w < 4; ++w) sF[le][1][w][pt] = qq[1 + w] - sF[le][0][w][0];
      }
      __syncthreads();
      if (active) {
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
          for (int c = 0; c < 3; ++c) ja[d][c] *= invJ;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const double* V = sF[le][1][w];
          double dr[3] = {0.0, 0.0, 0.0};
#pragma unroll
          for (int m = 0; m < n1; ++m) {
            dr[0] = fma(sDg[kGrad ? i : 0][kGrad ? m : 0], V[(k * n1 + j) * n1 + m], dr[0]);
            dr[1] = fma(sDg[kGrad ? j : 0][kGrad ? m : 0], V[(k * n1 + m) * n1 + i], dr[1]);
            dr[2] = fma(sDg[kGrad ? k : 0][kGrad ? m : 0], V[(m * n1 + j) * n1 + i], dr[2]);
          }
#pragma unroll
          for (int c = 0; c < 3; ++c)
            Gnext[(c * 4 + w) * plane + gi] = fma(ja[0][c], dr[0], fma(ja[1][c], dr[1], ja[2][c] * dr[2]));
        }
      }
    }
  }
  if (partial) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ssq += __shfl_down_sync(0xffffffffu, ssq, off);
    if ((threadIdx.x & 31) == 0) sred[threadIdx.x >> 5] = ssq;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) s += sred[w];
      partial[blockIdx.x] = s;
    }
  }
}

template <int P>
static int threads3() { return (EPB3<P>::value * (P + 1) * (P + 1) * (P + 1) + 31) / 32 * 32; }

int residual_blocks_for3(int P, int E) {
  int epb;
  switch (P) {
    case 0: epb = EPB3<0>::value; break;
    case 1: epb = EPB3<1>::value; break;
    case 2: epb = EPB3<2>::value; break;
    default: epb = EPB3<3>::value; break;
  }
  return (E + epb - 1) / epb;
}

// Broken gradient of (u, v, w, T) at every solution point of hexahedra:
// Gb[(c*4 + k) * E N + e N + pt], c = x, y, z, by the Lagrange derivative
// along the three lines through the point and the chain rule with J a^i / |J|.
// The derivative is taken of the differences to the element's first value
// (the derivative matrix annihilates constants, which keeps T ~ 1/Ma^2 out of
// the rounding), formed once per value in shared memory.  Not run at P = 0,
// where the gradient is zero.
template <int P>
struct GradEPB3 {
  static constexpr int value = P == 1 ? 16 : P == 2 ? 7 : 2;   // 128, 189 (of 192), 128 points
  static constexpr int threads = (value * (P + 1) * (P + 1) * (P + 1) + 31) / 32 * 32;
};
template <int P>
__global__ void __launch_bounds__(GradEPB3<P>::threads) grad3_kernel(int E, const double* __restrict__ q,
                                                                     const double* __restrict__ met, OpTab op,
                                                                     double* __restrict__ Gb) {
  constexpr int n1 = P + 1, N = n1 * n1 * n1, EPB = GradEPB3<P>::value;
  __shared__ double sV[4][EPB * N];
  __shared__ double sD[n1][n1];
  const int e0 = blockIdx.x * EPB, np = min(EPB, E - e0) * N;
  const size_t plane = (size_t)E * N, g0 = (size_t)e0 * N;
  const int t = threadIdx.x, le = t / N, pt = t - le * N;
  const int i = pt % n1, j = (pt / n1) % n1, k = pt / (n1 * n1);
  const bool active = t < np;
  if (t < n1 * n1) sD[t / n1][t % n1] = op.D[t / n1][t % n1];
  double ja[3][3];
  if (active) {
    const double iJ = __ldg(met + 9 * plane + g0 + t);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const double* V = q + (w + 1) * plane + g0;
      sV[w][t] = __ldg(V + t) - __ldg(V + le * N);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int c = 0; c < 3; ++c) ja[d][c] = iJ * __ldg(met + (3 * d + c) * plane + g0 + t);
  }
  __syncthreads();
  if (!active) return;
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    const double* V = sV[w] + le * N;
    double dr[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int m = 0; m < n1; ++m) {
      dr[0] = fma(sD[i][m], V[(k * n1 + j) * n1 + m], dr[0]);
      dr[1] = fma(sD[j][m], V[(k * n1 + m) * n1 + i], dr[1]);
      dr[2] = fma(sD[k][m], V[(m * n1 + j) * n1 + i], dr[2]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
      Gb[(c * 4 + w) * plane + g0 + t] = fma(ja[0][c], dr[0], fma(ja[1][c], dr[1], ja[2][c] * dr[2]));
  }
}

void launch_grad3(const Ctx& c, const LevelDev& L, const double* q, cudaStream_t s) {
#define PMG_G3(PP)                                                                                            \
  grad3_kernel<PP><<<(c.E + GradEPB3<PP>::value - 1) / GradEPB3<PP>::value, GradEPB3<PP>::threads, 0, s>>>( \
      c.E, q, L.met, L.op, L.Gb)
  switch (L.P) {
    case 0: break;   // zero
    case 1: PMG_G3(1); break;
    case 2: PMG_G3(2); break;
    default: PMG_G3(3); break;
  }
#undef PMG_G3
}

void launch_face_flux3(const Ctx& c, const LevelDev& L, const double* q, cudaStream_t s, bool have_grad) {
  const int total = c.n_faces * L.NF, threads = 64, blocks = (total + threads - 1) / threads;
  const bool visc = c.ph.mu > 0.0;
  if (visc && !have_grad) launch_grad3(c, L, q, s);
#define PMG_F3(PP)                                                                                                \
  if (visc)                                                                                                       \
    face_flux3_kernel<PP, true><<<blocks, threads, 0, s>>>(c.d_faces, c.n_faces, c.E, q, L.face, L.Fcom, L.op,   \
                                                           c.ph, L.Gb, L.fJinv, L.Qj);                           \
  else                                                                                                            \
    face_flux3_kernel<PP, false><<<blocks, threads, 0, s>>>(c.d_faces, c.n_faces, c.E, q, L.face, L.Fcom, L.op,  \
                                                            c.ph, nullptr, nullptr, nullptr)
  switch (L.P) {
    case 0: PMG_F3(0); break;
    case 1: PMG_F3(1); break;
    case 2: PMG_F3(2); break;
    default: PMG_F3(3); break;
  }
#undef PMG_F3
}

void launch_volume3(const Ctx& c, const LevelDev& L, const double* q, double* out, ResMode mode, double inv_odt,
                    const double* src, const double* S, double* Sout, const double* Pd, double* partial,
                    cudaStream_t s, const double* qn) {
  const int blocks = residual_blocks_for3(L.P, c.E);
  const bool visc = c.ph.mu > 0.0;
#define PMG_V3(PP)                                                                                               \
  if (visc)                                                                                                      \
    volume3_kernel<PP, double, false, true><<<blocks, threads3<PP>(), 0, s>>>(                                  \
        c.E, q, L.met, L.Fcom, L.Qj, L.Gb, L.op, c.ph, out, (int)mode, inv_odt, src, S, Sout, Pd, qn, partial, nullptr, \
        nullptr, nullptr, nullptr, nullptr);                                                                              \
  else                                                                                                           \
    volume3_kernel<PP, double, false, false><<<blocks, threads3<PP>(), 0, s>>>(                                 \
        c.E, q, L.met, L.Fcom, nullptr, nullptr, L.op, c.ph, out, (int)mode, inv_odt, src, S, Sout, Pd, qn, partial,      \
        nullptr, nullptr, nullptr, nullptr, nullptr)
  switch (L.P) {
    case 0: PMG_V3(0); break;
    case 1: PMG_V3(1); break;
    case 2: PMG_V3(2); break;
    default: PMG_V3(3); break;
  }
#undef PMG_V3
}

template <class W>
static void volume_apply3_dispatch(const Ctx& c, const LevelDev& L, double* q, double inv_odt, const double* src,
                                   const double* S, const double* qn, double* gnext, cudaStream_t s) {
  const int blocks = residual_blocks_for3(L.P, c.E);
  const W* Dinv = (const W*)L.Dinv;
  const bool visc = c.ph.mu > 0.0;
#define PMG_VA3(PP)                                                                                             \
  if (visc)                                                                                                     \
    volume3_kernel<PP, W, true, true><<<blocks, threads3<PP>(), 0, s>>>(                                       \
        c.E, q, L.met, L.Fcom, L.Qj, L.Gb, L.op, c.ph, nullptr, (int)RES_SYSTEM, inv_odt, src, S, nullptr, nullptr, qn, \
        nullptr, q, Dinv, L.rs, L.cs, gnext);                                                                          \
  else                                                                                                          \
    volume3_kernel<PP, W, true, false><<<blocks, threads3<PP>(), 0, s>>>(                                      \
        c.E, q, L.met, L.Fcom, nullptr, nullptr, L.op, c.ph, nullptr, (int)RES_SYSTEM, inv_odt, src, S, nullptr, nullptr, \
        qn, nullptr, q, Dinv, L.rs, L.cs, nullptr)
  switch (L.P) {
    case 0: PMG_VA3(0); break;
    case 1: PMG_VA3(1); break;
    case 2: PMG_VA3(2); break;
    default: PMG_VA3(3); break;
  }
#undef PMG_VA3
}

void launch_volume_apply3(const Ctx& c, const LevelDev& L, double* q, double inv_odt, const double* src,
                          const double* S, const double* qn, double* gnext, int prec, cudaStream_t s) {
  if (prec == PMG_PREC_FP64) volume_apply3_dispatch<double>(c, L, q, inv_odt, src, S, qn, gnext, s);
  else if (prec == PMG_PREC_BF16R) volume_apply3_dispatch<__nv_bfloat16>(c, L, q, inv_odt, src, S, qn, gnext, s);
  else volume_apply3_dispatch<float>(c, L, q, inv_odt, src, S, qn, gnext, s);
}

}  // namespace pmg
