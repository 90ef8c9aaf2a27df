// k3_fused.cu -- one element-Jacobi sweep of the P = 0 level on hexahedra in
// one launch (Section 2.4, eq. smoothing_element_jacobi, on the level system of
// Section 3), binary64.
//
// At P = 0 an element is one point, its residual the sum of six face fluxes
// (the line operator of the divergence is zero and so is the broken gradient of
// the viscous terms).  A small level does not fill the chip: the split face and
// volume launches each last as long as one warp's chain of FP64 instructions
// (64 cycles each), 10.4 and 12.2 us at 960 elements.  Here a lane takes a face
// of an element, five elements to a warp; every face is evaluated by both of
// its elements, which costs nothing while the warps fit the sub-partitions, and
// the update follows in the same warp, a lane per equation, into the second
// state buffer (Jacobi: every element reads the old state).
// Measured on one GB300, ten P{2-1-0} V-cycles of the viscous ellipse: 22.2 ->
// 20.0 ms at 960 elements, 30.4 -> 28.2 at 1920, 67.1 -> 66.4 at 5760; of the
// inviscid sphere 21.4 -> 20.1 ms at 2304 and equal at 6480.
#include "pmg_internal.h"

namespace pmg {

constexpr int kFused3Elems = 5;   // per warp: 30 lanes

template <class W>
__global__ void __launch_bounds__(32) fused_sweep3_kernel(
    int E, const double* __restrict__ qin, double* __restrict__ qout, const double* __restrict__ met,
    const double* __restrict__ face, const double* __restrict__ fJinv, const int* __restrict__ nbr, double pen, Phys ph,
    double inv_odt, const double* __restrict__ S, const double* __restrict__ qref, const W* __restrict__ Dinv,
    const double* __restrict__ rs, const double* __restrict__ cs) {
  using Acc = typename Blk<W>::acc;
  __shared__ double sC[kFused3Elems][5][6];
  __shared__ Acc sr[kFused3Elems][5];
  const int le = threadIdx.x / 6, f = threadIdx.x - 6 * le, e = blockIdx.x * kFused3Elems + le;
  const bool act = le < kFused3Elems && e < E;
  const size_t plane = E;
  double qm[5] = {0, 0, 0, 0, 0}, qo[5] = {0, 0, 0, 0, 0}, invJ = 0.0, Sv = 0.0, rsv = 0.0, csv = 0.0;
  Acc dv[5] = {0, 0, 0, 0, 0};
  const bool eq = act && f < 5;   // lane f updates equation f
  if (act) {
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      qm[v] = __ldg(qin + v * plane + e);
      if (qref) qo[v] = __ldg(qref + v * plane + e);
    }
    invJ = __ldg(met + 9 * plane + e);
    if (eq) {
      if (S) Sv = __ldg(S + f * plane + e);
      rsv = __ldg(rs + (size_t)e * 5 + f);
      csv = __ldg(cs + (size_t)e * 5 + f);
#pragma unroll
      for (int k = 0; k < 5; ++k) dv[k] = blk_val(__ldg(Dinv + (size_t)e * 25 + k * 5 + f));
    }
    const int* nb = nbr + ((size_t)e * 6 + f) * 3;
    const int en = __ldg(nb), fn = __ldg(nb + 1);
    const bool bnd = en < 0;
    const double* g = face + ((size_t)e * 6 + f) * 4;
    const double nrm[3] = {__ldg(g), __ldg(g + 1), __ldg(g + 2)}, dS = __ldg(g + 3);
    double dq[5], qp[5];
    if (!bnd) {
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        qp[v] = __ldg(qin + v * plane + en);
        dq[v] = qp[v] - qm[v];
      }
    } else if (fn == PMG_BC_FARFIELD) {
      qp[0] = ph.qinf[0] - ph.p_ref;
#pragma unroll
      for (int v = 1; v < 5; ++v) qp[v] = ph.qinf[v];
#pragma unroll
      for (int v = 0; v < 5; ++v) dq[v] = qp[v] - qm[v];
    } else {   // walls: same p and T, velocity reversed (no-slip) or its normal part (slip)
      const double un = qm[1] * nrm[0] + qm[2] * nrm[1] + qm[3] * nrm[2];
      qp[0] = qm[0];
      qp[4] = qm[4];
      dq[0] = dq[4] = 0.0;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dq[1 + c] = fn == PMG_BC_NOSLIP_WALL ? -2.0 * qm[1 + c] : (-2.0 * un) * nrm[c];
        qp[1 + c] = qm[1 + c] + dq[1 + c];
      }
    }
    const double pgm = qm[0], pgp = qp[0];
    double qa[5] = {qm[0] + ph.p_ref, qm[1], qm[2], qm[3], qm[4]}, out[5];
    qp[0] += ph.p_ref;
    roe_jump_d<3>(qa, qp, dq, pgm, pgp, nrm, dS, ph, out);
    if (ph.mu > 0.0) {
      // the common gradient is the lifting alone, wl n dq (k3_residual.cu face_flux3)
      const double iJm = __ldg(fJinv + (size_t)e * 6 + f), iJp = bnd ? iJm : __ldg(fJinv + (size_t)en * 6 + fn);
      const double wl = 0.25 * pen * (iJm + iJp) * dS;
      double dn = 0.0, n2 = 0.0, wk = 0.0;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dn = fma(nrm[c], dq[1 + c], dn);
        n2 = fma(nrm[c], nrm[c], n2);
      }
      // (g + g^T) n - 2/3 div n with g = wl n (x) dv: wl (|n|^2 dv + n (n.dv)/3)
      const double a = ph.mu * dS * wl, an = a * n2, b = a * dn * (1.0 / 3.0);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double t = fma(an, dq[1 + c], b * nrm[c]);
        out[1 + c] -= t;
        wk = fma(fma(0.5, dq[1 + c], qm[1 + c]), t, wk);
      }
      if (!(bnd && fn != PMG_BC_FARFIELD)) out[4] = fma(-(ph.kT * dS * wl * n2), dq[4], out[4] - wk);
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) sC[le][v][f] = out[v];
  }
  __syncwarp();
  double qv = 0.0;
  if (eq) {
    // at P = 0 both correction weights are 1/2: R = -(1/2) sum of outward fluxes / |J|
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 6; ++k) s += sC[le][f][k];
    const double rho = (qm[0] + ph.p_ref) * s_rcp(qm[4]);
    double qc;
    const double uu = fma(qm[1], qm[1], fma(qm[2], qm[2], qm[3] * qm[3]));
    const double um = f == 1 ? qm[1] : f == 2 ? qm[2] : qm[3];
    if (qref) {   // q_c(q) - q_c(q_ref), the energy through the pressure difference
      const double rhoo = (qo[0] + ph.p_ref) * s_rcp(qo[4]);
      const double uo = fma(qo[1], qo[1], fma(qo[2], qo[2], qo[3] * qo[3]));
      const double umo = f == 1 ? qo[1] : f == 2 ? qo[2] : qo[3];
      qc = f == 0 ? rho - rhoo
                  : f < 4 ? rho * um - rhoo * umo : (qm[0] - qo[0]) * ph.inv_gm1 + 0.5 * (rho * uu - rhoo * uo);
    } else {
      qc = f == 0 ? rho : f < 4 ? rho * um : rho * (qm[4] * ph.inv_gm1 + 0.5 * uu);
    }
    const double F = fma(-qc, inv_odt, (-0.5 * s) * invJ) - Sv;
    sr[le][f] = scaled_in<W>(F, rsv);
    qv = f == 0 ? qm[0] : f == 4 ? qm[4] : um;
  }
  __syncwarp();
  if (eq) {
    Acc acc = 0;
#pragma unroll
    for (int k = 0; k < 5; ++k) acc = fma(dv[k], sr[le][k], acc);
    qout[f * plane + e] = qv + scaled_out<W>(acc, csv);
  }
}

// Worth it while the doubled face work stays within about two warps per SM
// sub-partition (8 warps of 5 elements per SM; the figures above cross there).
bool fused3_applies(int P, int E, int sms) { return P == 0 && E <= 40 * sms; }

void launch_fused_sweep3(const Ctx& c, const LevelDev& L, const double* qin, double* qout, double inv_odt,
                         const double* S, const double* qref, int prec, cudaStream_t s) {
  const int blocks = (c.E + kFused3Elems - 1) / kFused3Elems;
  const int* nbr = c.d_faces + 5 * c.n_faces;
#define PMG_FS3(WT)                                                                                          \
  fused_sweep3_kernel<WT><<<blocks, 32, 0, s>>>(c.E, qin, qout, L.met, L.face, L.fJinv, nbr, L.op.pen, c.ph, \
                                                inv_odt, S, qref, (const WT*)L.Dinv, L.rs, L.cs)
  if (prec == PMG_PREC_FP64) PMG_FS3(double);
  else if (prec == PMG_PREC_BF16R) PMG_FS3(__nv_bfloat16);
  else PMG_FS3(float);
#undef PMG_FS3
}

}  // namespace pmg
