// k_assemble.cu -- assembly of the element-Jacobi blocks (Section 2.4, eqs.
// linearized_pseudo_transient_final and smoothing_element_jacobi),
//   D_e = Gamma/dtau + M/(omega dt) - dR_e/dq_e,
// on quadrilaterals (DIM = 2) and hexahedra (DIM = 3), neighbours frozen, in
// binary64.  dR_e/dq_e is exact: closed-form flux Jacobians at the solution
// points, hand-written tangents of the preconditioned Roe flux at the face
// points (physics_tan.cuh; through the averaged state and, on boundary faces,
// the ghost state), and the viscous terms below.
//
// The kernels are bound by FP64 issue (a warp instruction takes 64 cycles of
// its sub-partition, whatever lanes are active), so they work on the pairs
// (r, c) of solution points that are coupled at all, with full warps:
//  * assemble: R couples points of one line.  A pair on a line along d takes
//    Dt[r_d][c_d] A_d(c) + gL[r_d] lm[c_d] C(-1) + gR[r_d] lp[c_d] C(+1) per
//    pair of variables (Dt: the derivative with the extrapolated part of the
//    correction folded in), a lane per pair of variables; the other entries
//    are zeroed without arithmetic.
//  * assemble_visc (mu > 0) adds the viscous part to rows and columns of
//    (velocity, T).  The tangent of the viscous flux is linear in the gradient's:
//    with dg = s Y at a point, X . dtau = mu s Q(X, Y),
//    Q_iw = (X.Y) delta_iw + X_w Y_i - 2/3 X_i Y_w, for any area vector X.  A
//    perturbation at c reaches the gradients on the lines through c only, so a
//    pair of points that differ in two coordinates (d, e) takes one term for
//    (e-line of r, gradient along d) and one for the converse, a pair on a line
//    the sum over the line, and points that differ in three nothing.  Common
//    viscous fluxes enter the same sums with the face's area vector for X:
//    half the broken gradient's tangent (all of it where a boundary mirrors the
//    element) plus the BR2 lifting of the jump, d(q^+ - q^-) = 2 kappa dq^-
//    (kappa = -1/2 on interior and far-field faces, -1 for the velocity and 0
//    for T at no-slip walls).
// Before, every column was pushed through the whole element with dual numbers
// and every block entry evaluated all the lines.  Measured on one GB300, ms:
//                                      inviscid        viscous part
//   960 hexahedra, P = 3 (n = 320)     3.75 -> 0.66    16.7 -> 1.72
//   960 hexahedra, P = 2 (n = 135)     1.20 -> 0.27     3.6 -> 0.53
//   16384 quadrilaterals, P = 4        7.1  -> 1.61    11.8 -> 4.5
//   4096 quadrilaterals, P = 3         1.07 -> 0.27
#include "pmg_internal.h"
#include "physics_tan.cuh"

namespace pmg {

namespace {

// Face f as (direction, side), and its number; quadrilateral faces are
// 0: eta = -1, 1: xi = +1, 2: eta = +1, 3: xi = -1.
template <int DIM> __device__ __forceinline__ int face_dir(int f) { return DIM == 3 ? f >> 1 : 1 - (f & 1); }
template <int DIM> __device__ __forceinline__ bool face_plus(int f) { return DIM == 3 ? f & 1 : f == 1 || f == 2; }
template <int DIM> __device__ __forceinline__ int face_of(int d, int s) {
  return DIM == 3 ? 2 * d + s : d == 0 ? (s ? 1 : 3) : (s ? 2 : 0);
}
// Point m of the d-line through face point fp of a face normal to d.
template <int DIM, int P> __device__ __forceinline__ int line_point(int d, int fp, int m) {
  constexpr int n1 = P + 1;
  if (DIM == 2) return d == 0 ? fp * n1 + m : m * n1 + fp;
  const int a = fp % n1, b = fp / n1;
  const int i = d == 0 ? m : a, j = d == 1 ? m : (d == 0 ? a : b), k = d == 2 ? m : b;
  return (k * n1 + j) * n1 + i;
}
// Coordinate along d of a point, the stride of that coordinate, and the face
// point of its d-line.
template <int DIM, int P> __device__ __forceinline__ int coord(int pt, int d) {
  constexpr int n1 = P + 1;
  return d == 0 ? pt % n1 : d == 1 ? (pt / n1) % n1 : pt / (n1 * n1);
}
template <int P> __device__ __forceinline__ int stride_of(int d) {
  constexpr int n1 = P + 1;
  return d == 0 ? 1 : d == 1 ? n1 : n1 * n1;
}
template <int DIM, int P> __device__ __forceinline__ int face_point(int pt, int d) {
  constexpr int n1 = P + 1;
  if (DIM == 2) return d == 0 ? pt / n1 : pt % n1;
  const int i = pt % n1, j = (pt / n1) % n1, k = pt / (n1 * n1);
  return d == 0 ? k * n1 + j : d == 1 ? k * n1 + i : j * n1 + i;
}
// The neighbour's number of face point fp.
template <int DIM, int P> __device__ __forceinline__ int other_point(int fp, int o) {
  constexpr int n1 = P + 1;
  if (DIM == 2) return o ? P - fp : fp;
  const int a = fp % n1, b = fp / n1, s = (o & 4) ? b : a, t = (o & 4) ? a : b;
  return ((o & 2) ? P - t : t) * n1 + ((o & 1) ? P - s : s);
}

template <int DIM, int P>
struct AsmShape {
  static constexpr int n1 = P + 1, NV = DIM + 2, VV = NV * NV, N = DIM == 3 ? n1 * n1 * n1 : n1 * n1,
                       NF = DIM == 3 ? n1 * n1 : n1, F = 2 * DIM, FP = F * NF, n = NV * N;
  static constexpr int kThreads = 128;
  static constexpr int most = N > FP ? N : FP;
  static constexpr int fit = kThreads / most < 1 ? 1 : kThreads / most;
  static constexpr int EPB = fit > 32 ? 32 : fit;   // elements per CTA: full warps in the point and face phases
  static constexpr size_t per_elem = sizeof(double) * ((size_t)N * (DIM + 1) * VV + (size_t)FP * VV);
  static constexpr size_t smem = per_elem * EPB;
};

}  // namespace

template <int DIM, int P>
__global__ void __launch_bounds__(128) assemble_kernel(int E, const double* __restrict__ q,
                                                       const double* __restrict__ met,
                                                       const double* __restrict__ face,
                                                       const int* __restrict__ nbr, OpTab op, Phys ph,
                                                       const double* __restrict__ d_dtau, double inv_odt,
                                                       double* __restrict__ Dout) {
  using Y = AsmShape<DIM, P>;
  constexpr int n1 = Y::n1, NV = Y::NV, VV = Y::VV, N = Y::N, NF = Y::NF, F = Y::F, FP = Y::FP, n = Y::n,
                EPB = Y::EPB;
  extern __shared__ __align__(16) double dyn[];
  double* sA = dyn;                              // [EPB][N][DIM][VV] d(F^d)/dq at each point
  double* sDiag = sA + (size_t)EPB * N * DIM * VV;   // [EPB][N][VV] Gamma/dtau + M/(omega dt)
  double* sC = sDiag + (size_t)EPB * N * VV;     // [EPB][FP][VV] d(reference-direction common flux)/dq(own trace)
  __shared__ double sq[EPB][NV][N];
  __shared__ double sinvJ[EPB * N];
  __shared__ double sLine[3][n1][n1];            // Dt, gL lm, gR lp
  __shared__ double sl[2][n1];
  const int e0 = blockIdx.x * EPB, ne = min(EPB, E - e0), tid = threadIdx.x;
  const size_t plane = (size_t)E * N;
  for (int t = tid; t < ne * NV * N; t += blockDim.x) {
    const int v = t / (ne * N), r = t - v * ne * N;
    sq[r / N][v][r % N] = q[v * plane + (size_t)e0 * N + r];
  }
  if (tid < n1 * n1) {
    const int i = tid / n1, m = tid % n1;
    sLine[0][i][m] = op.Dt[i][m];
    sLine[1][i][m] = op.gL[i] * op.lm[m];
    sLine[2][i][m] = op.gR[i] * op.lp[m];
  }
  if (tid < n1) {
    sl[0][tid] = op.lm[tid];
    sl[1][tid] = op.lp[tid];
  }
  // the blocks' zeros (the coupled pairs are written after the barriers below)
  {
    double* Db = Dout + (size_t)e0 * n * n;
    const int total = ne * n * n;
#pragma unroll 8
    for (int t = tid; t < total; t += blockDim.x) Db[t] = 0.0;
  }
  __syncthreads();
  // pointwise: flux Jacobians along each J a^d, time terms
  for (int t = tid; t < ne * N; t += blockDim.x) {
    const int le = t / N, pt = t - le * N;
    const size_t gi = (size_t)e0 * N + t;
    sinvJ[t] = met[DIM * DIM * plane + gi];
    double v[DIM], vv = 0.0;
    const double p = sq[le][0][pt] + ph.p_ref, T = sq[le][NV - 1][pt];
#pragma unroll
    for (int c = 0; c < DIM; ++c) {
      v[c] = sq[le][1 + c][pt];
      vv = fma(v[c], v[c], vv);
    }
    const double rp = s_rcp(T), rho = p * rp, rT = -rho * rp, H = fma(ph.Cp, T, 0.5 * vv);
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      double* A = sA + ((size_t)t * DIM + d) * VV;
      double a[DIM], un = 0.0;
#pragma unroll
      for (int c = 0; c < DIM; ++c) {
        a[c] = met[(DIM * d + c) * plane + gi];
        un = fma(v[c], a[c], un);
      }
      const double up = rp * un, mn = rho * un, uT = rT * un;
      A[0] = up;
      A[NV - 1] = uT;
      A[(NV - 1) * NV] = up * H;
      A[(NV - 1) * NV + NV - 1] = fma(uT, H, mn * ph.Cp);
#pragma unroll
      for (int c = 0; c < DIM; ++c) {
        const double ra = rho * a[c];
        A[1 + c] = ra;
        A[(1 + c) * NV] = fma(up, v[c], a[c]);
        A[(1 + c) * NV + NV - 1] = uT * v[c];
        A[(NV - 1) * NV + 1 + c] = fma(ra, H, mn * v[c]);
#pragma unroll
        for (int k = 0; k < DIM; ++k) A[(1 + k) * NV + 1 + c] = k == c ? fma(ra, v[k], mn) : ra * v[k];
      }
    }
    // Gamma/dtau + M/(omega dt): they differ in the pressure column only
    const double idt = 1.0 / *d_dtau, s = idt + inv_odt;
    const double e2 = s_min(1.0, s_max(ph.eps_min * ph.eps_min, vv * (rp * ph.inv_gamma)));
    const double Th = rp * fma(s_rcp(e2), ph.inv_gamma, ph.inv_Cp);   // 1/Ur^2 - rho_T / (rho Cp)
    const double cp = fma(Th, idt, rp * inv_odt), cT = rT * s, rs = rho * s;
    double* G = sDiag + (size_t)t * VV;
    G[0] = cp;
    G[NV - 1] = cT;
    G[(NV - 1) * NV] = fma(cp, H, -s);
    G[(NV - 1) * NV + NV - 1] = fma(cT, H, rs * ph.Cp);
#pragma unroll
    for (int c = 0; c < DIM; ++c) {
      G[1 + c] = 0.0;
      G[(1 + c) * NV] = cp * v[c];
      G[(1 + c) * NV + NV - 1] = cT * v[c];
      G[(NV - 1) * NV + 1 + c] = rs * v[c];
#pragma unroll
      for (int k = 0; k < DIM; ++k) G[(1 + k) * NV + 1 + c] = k == c ? rs : 0.0;
    }
  }
  // own-side derivative of the reference-direction common flux
  for (int t = tid; t < ne * FP; t += blockDim.x) {
    const int le = t / FP, r = t - le * FP, f = r / NF, fp = r - f * NF, d = face_dir<DIM>(f), e = e0 + le;
    const bool plus = face_plus<DIM>(f);
    const int en = nbr[(e * F + f) * 3], fn = nbr[(e * F + f) * 3 + 1], o = nbr[(e * F + f) * 3 + 2];
    double qm[NV], qp[NV], nrm[DIM];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      double s = 0.0;
#pragma unroll
      for (int m = 0; m < n1; ++m) s = fma(sl[plus ? 1 : 0][m], sq[le][v][line_point<DIM, P>(d, fp, m)], s);
      qm[v] = s;
    }
    qm[0] += ph.p_ref;
    const double* g = face + ((size_t)(e * F + f) * NF + fp) * (DIM + 1);
#pragma unroll
    for (int c = 0; c < DIM; ++c) nrm[c] = g[c];
    const double hdS = 0.5 * g[DIM];
    if (en >= 0) {
      const int fp2 = other_point<DIM, P>(fp, o), dn = face_dir<DIM>(fn);
      const bool pn = face_plus<DIM>(fn);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        double s = 0.0;
#pragma unroll
        for (int m = 0; m < n1; ++m)
          s = fma(sl[pn ? 1 : 0][m], q[v * plane + (size_t)en * N + line_point<DIM, P>(dn, fp2, m)], s);
        qp[v] = s;
      }
      qp[0] += ph.p_ref;
    } else if (fn == PMG_BC_FARFIELD) {
#pragma unroll
      for (int v = 0; v < NV; ++v) qp[v] = ph.qinf[v];
    } else {
      double un = 0.0;
#pragma unroll
      for (int c = 0; c < DIM; ++c) un = fma(qm[1 + c], nrm[c], un);
      qp[0] = qm[0];
      qp[NV - 1] = qm[NV - 1];
#pragma unroll
      for (int c = 0; c < DIM; ++c) qp[1 + c] = fn == PMG_BC_NOSLIP_WALL ? -qm[1 + c] : fma(-2.0 * un, nrm[c], qm[1 + c]);
    }
    RoeLin<DIM> R;
    R.init(qm, qp, nrm, ph);
    const bool wall = en < 0 && fn != PMG_BC_FARFIELD;
    const double sg = plus ? hdS : -hdS;
    double* C = sC + (size_t)t * VV;
#pragma unroll 1
    for (int w = 0; w < NV; ++w) {
      double tm[NV], tg[NV], tq[NV], jq[NV], ft[NV], dd[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        tm[v] = v == w ? 1.0 : 0.0;
        tg[v] = wall ? tm[v] : 0.0;   // the ghost of a wall follows the own trace
      }
      if (wall) {
        double tn = 0.0;
#pragma unroll
        for (int c = 0; c < DIM; ++c) tn = fma(tm[1 + c], nrm[c], tn);
#pragma unroll
        for (int c = 0; c < DIM; ++c) tg[1 + c] = fn == PMG_BC_NOSLIP_WALL ? -tm[1 + c] : fma(-2.0 * tn, nrm[c], tm[1 + c]);
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        tq[v] = 0.5 * (tm[v] + tg[v]);
        jq[v] = tg[v] - tm[v];
      }
      flux_tangent<DIM>(qm, nrm, tm, ph, ft);
      if (wall) {
        double fg[NV];
        flux_tangent<DIM>(qp, nrm, tg, ph, fg);
#pragma unroll
        for (int v = 0; v < NV; ++v) ft[v] += fg[v];
      }
      R.tangent(tq, jq, ph, dd);
#pragma unroll
      for (int v = 0; v < NV; ++v) C[v * NV + w] = sg * (ft[v] - dd[v]);
    }
  }
  __syncthreads();
  // the coupled pairs: LP lanes per pair, a lane per pair of variables
  constexpr int LP = DIM == 3 ? 32 : 16, PW = DIM * (n1 - 1) + 1;
  const int vw = tid % LP, v = vw / NV, w = vw - v * NV;
  if (vw >= VV) return;
  for (int t = tid / LP; t < ne * N * PW; t += blockDim.x / LP) {
    const int le = t / (N * PW), u = t - le * N * PW, rp = u / PW, x = u - rp * PW;
    const double* A = sA + (size_t)le * N * DIM * VV + vw;
    const double* C = sC + (size_t)le * FP * VV + vw;
    int cp = rp;
    double s = 0.0;
    if (x > 0) {
      const int d = (x - 1) / (n1 > 1 ? n1 - 1 : 1), m = (x - 1) - d * (n1 - 1), i = coord<DIM, P>(rp, d);
      const int c = m >= i ? m + 1 : m, fp = face_point<DIM, P>(rp, d);
      cp = rp + (c - i) * stride_of<P>(d);
      s = sLine[0][i][c] * A[(cp * DIM + d) * VV];
      s = fma(sLine[1][i][c], C[(face_of<DIM>(d, 0) * NF + fp) * VV], s);
      s = fma(sLine[2][i][c], C[(face_of<DIM>(d, 1) * NF + fp) * VV], s);
    } else {
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
        const int i = coord<DIM, P>(rp, d), fp = face_point<DIM, P>(rp, d);
        s = fma(sLine[0][i][i], A[(cp * DIM + d) * VV], s);
        s = fma(sLine[1][i][i], C[(face_of<DIM>(d, 0) * NF + fp) * VV], s);
        s = fma(sLine[2][i][i], C[(face_of<DIM>(d, 1) * NF + fp) * VV], s);
      }
    }
    s *= sinvJ[le * N + rp];
    if (x == 0) s += sDiag[((size_t)le * N + rp) * VV + vw];
    Dout[(size_t)(e0 + le) * n * n + (size_t)(v * N + rp) * n + w * N + cp] = s;
  }
}

// ------------------------------------------------------------- viscous part
namespace {

template <int DIM, int P>
struct ViscShape {
  static constexpr int n1 = P + 1, N = DIM == 3 ? n1 * n1 * n1 : n1 * n1, NF = DIM == 3 ? n1 * n1 : n1, F = 2 * DIM,
                       FP = F * NF, NW = DIM + 1, n = (DIM + 2) * N;
  static constexpr int kThreads = N >= 64 ? 256 : 128;
  static constexpr int EPB = N == 1 ? 16 : N <= 4 ? 16 : N <= 9 ? 7 : N <= 16 ? 4 : N <= 27 ? 2 : 1;
  static constexpr int KN = DIM * (DIM + 1) / 2 + DIM + 1;   // K_dd: symmetric part, energy row, T
  // doubles per element
  static constexpr int oJa = 0;                     // [N][DIM][DIM] J a^d
  static constexpr int oIJ = oJa + N * DIM * DIM;   // [N]
  static constexpr int oV = oIJ + N;                // [NW][N] velocity, T
  static constexpr int oTau = oV + NW * N;          // [N][DIM][DIM] stress / mu
  static constexpr int oK = oTau + N * DIM * DIM;   // [N][DIM][KN]
  static constexpr int oN = oK + N * DIM * KN;      // [FP][DIM] area vector in the reference direction
  static constexpr int oUc = oN + FP * DIM;         // [FP][DIM] q_com velocity
  static constexpr int oTn = oUc + FP * DIM;        // [FP][DIM] common stress / mu times the area vector
  static constexpr int oLf = oTn + FP * DIM;        // [FP][DIM] lifting vector
  static constexpr int oQj = oLf + FP * DIM;        // [FP][NW] half jump
  static constexpr int oYb = oQj + FP * NW;         // [F][N][DIM] face gradient per perturbation on the face's line
  static constexpr int per_elem = oYb + F * N * DIM;
  static constexpr size_t smem = sizeof(double) * (size_t)per_elem * EPB;
};

// acc += s Q(X, Y) with the energy row u . Q weighted by we.
template <int DIM>
struct ViscAcc {
  double m[DIM][DIM], en[DIM], tt;
  __device__ __forceinline__ void zero() {
    tt = 0.0;
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      en[i] = 0.0;
#pragma unroll
      for (int w = 0; w < DIM; ++w) m[i][w] = 0.0;
    }
  }
  __device__ __forceinline__ void mom(const double X[DIM], const double Y[DIM]) {
    double xy = 0.0, x23[DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c) {
      xy = fma(X[c], Y[c], xy);
      x23[c] = (-2.0 / 3.0) * X[c];
    }
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
      for (int w = 0; w < DIM; ++w) {
        m[i][w] = fma(X[w], Y[i], fma(x23[i], Y[w], m[i][w]));
        if (i == w) m[i][w] += xy;
      }
  }
  // energy row of s Q(X, Y) for the velocity u
  __device__ __forceinline__ void energy(double s, double xy, const double X[DIM], const double Y[DIM],
                                         const double u[DIM]) {
    double uy = 0.0, ux = 0.0;
#pragma unroll
    for (int c = 0; c < DIM; ++c) {
      uy = fma(u[c], Y[c], uy);
      ux = fma(u[c], X[c], ux);
    }
    const double sxy = s * xy, suy = s * uy, sux = (-2.0 / 3.0) * (s * ux);
#pragma unroll
    for (int w = 0; w < DIM; ++w) en[w] = fma(u[w], sxy, fma(X[w], suy, fma(sux, Y[w], en[w])));
  }
};

template <int DIM>
__device__ __forceinline__ double dotv(const double* a, const double* b) {
  double s = 0.0;
#pragma unroll
  for (int c = 0; c < DIM; ++c) s = fma(a[c], b[c], s);
  return s;
}

}  // namespace

template <int DIM, int P>
__global__ void __launch_bounds__(ViscShape<DIM, P>::kThreads)
    assemble_visc_kernel(int E, const double* __restrict__ q, const double* __restrict__ Gb,
                         const double* __restrict__ met, const double* __restrict__ face,
                         const double* __restrict__ fJinv, const int* __restrict__ nbr, OpTab op, Phys ph,
                         double* __restrict__ Dout) {
  using Y_ = ViscShape<DIM, P>;
  constexpr int n1 = Y_::n1, N = Y_::N, NF = Y_::NF, F = Y_::F, FP = Y_::FP, NW = Y_::NW, n = Y_::n, EPB = Y_::EPB,
                KN = Y_::KN;
  extern __shared__ __align__(16) double dyn[];
  __shared__ double sD[n1][n1], sDt[n1][n1], sg[2][n1], sl[2][n1];
  __shared__ double sCd[EPB][DIM][2][n1][n1];   // corrected derivative: velocity, T
  __shared__ double sKap[EPB][F][2], sGf[EPB][F], sWe[EPB][F];
  const int e0 = blockIdx.x * EPB, ne = min(EPB, E - e0), tid = threadIdx.x, nt = blockDim.x;
  const size_t plane = (size_t)E * N;
  auto base = [&](int le) { return dyn + (size_t)le * Y_::per_elem; };
  if (tid < n1 * n1) {
    sD[tid / n1][tid % n1] = op.D[tid / n1][tid % n1];
    sDt[tid / n1][tid % n1] = op.Dt[tid / n1][tid % n1];
  }
  if (tid < n1) {
    sg[0][tid] = op.gL[tid];
    sg[1][tid] = op.gR[tid];
    sl[0][tid] = op.lm[tid];
    sl[1][tid] = op.lp[tid];
  }
  for (int t = tid; t < ne * F; t += nt) {
    const int le = t / F, f = t - le * F, en = nbr[((size_t)(e0 + le) * F + f) * 3],
              bc = nbr[((size_t)(e0 + le) * F + f) * 3 + 1];
    const bool wall = en < 0 && bc != PMG_BC_FARFIELD;
    sKap[le][f][0] = wall ? -1.0 : -0.5;
    sKap[le][f][1] = wall ? 0.0 : -0.5;
    sGf[le][f] = en < 0 ? 1.0 : 0.5;
    sWe[le][f] = wall ? 0.0 : 1.0;   // walls carry no viscous energy flux
  }
  for (int t = tid; t < ne * N; t += nt) {
    const int le = t / N, pt = t - le * N;
    double* B = base(le);
    const size_t gi = (size_t)e0 * N + t;
#pragma unroll
    for (int c = 0; c < DIM * DIM; ++c) B[Y_::oJa + pt * DIM * DIM + c] = met[c * plane + gi];
    B[Y_::oIJ + pt] = met[DIM * DIM * plane + gi];
#pragma unroll
    for (int k = 0; k < NW; ++k) B[Y_::oV + k * N + pt] = q[(k + 1) * plane + gi];
  }
  __syncthreads();
  for (int t = tid; t < ne * DIM * n1 * n1; t += nt) {
    const int le = t / (DIM * n1 * n1), r = t - le * DIM * n1 * n1, d = r / (n1 * n1), i = (r / n1) % n1, c = r % n1;
    const int fL = face_of<DIM>(d, 0), fR = face_of<DIM>(d, 1);
#pragma unroll
    for (int k = 0; k < 2; ++k)
      sCd[le][d][k][i][c] = fma(sg[0][i] * sKap[le][fL][k], sl[0][c], fma(sg[1][i] * sKap[le][fR][k], sl[1][c], sD[i][c]));
  }
  // face points: traces, half jumps, common velocity and stress, lifting
  for (int t = tid; t < ne * FP; t += nt) {
    const int le = t / FP, tf = t - le * FP, f = tf / NF, fp = tf - f * NF, d = face_dir<DIM>(f), e = e0 + le;
    const bool plus = face_plus<DIM>(f);
    double* B = base(le);
    const double* V = B + Y_::oV;
    const int en = nbr[((size_t)e * F + f) * 3], fn = nbr[((size_t)e * F + f) * 3 + 1], o = nbr[((size_t)e * F + f) * 3 + 2];
    const bool bnd = en < 0;
    const int fp2 = bnd ? fp : other_point<DIM, P>(fp, o), dn = bnd ? d : face_dir<DIM>(fn);
    const double* lo = sl[plus ? 1 : 0];
    const double* ln = sl[(bnd ? plus : face_plus<DIM>(fn)) ? 1 : 0];
    double dq[NW], uc[DIM];
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const double ref = V[w * N];
      double sm = 0.0, sp = 0.0;
#pragma unroll
      for (int m = 0; m < n1; ++m) {
        sm = fma(lo[m], V[w * N + line_point<DIM, P>(d, fp, m)] - ref, sm);
        if (!bnd) sp = fma(ln[m], q[(w + 1) * plane + (size_t)en * N + line_point<DIM, P>(dn, fp2, m)] - ref, sp);
      }
      // far field: the free stream; no-slip wall: velocity reversed, same T
      if (bnd) {
        if (fn == PMG_BC_FARFIELD) dq[w] = ph.qinf[w + 1] - (ref + sm);
        else dq[w] = w < DIM ? -2.0 * (ref + sm) : 0.0;
      } else {
        dq[w] = sp - sm;
      }
      if (w < DIM) uc[w < DIM ? w : 0] = fma(0.5, dq[w], ref + sm);
      B[Y_::oQj + tf * NW + w] = 0.5 * dq[w];
    }
    const double* g = face + ((size_t)(e * F + f) * NF + fp) * (DIM + 1);
    double nrm[DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c) nrm[c] = g[c];
    const double dS = g[DIM];
    const double iJm = fJinv[(size_t)(e * F + f) * NF + fp], iJp = bnd ? iJm : fJinv[(size_t)(en * F + fn) * NF + fp2];
    const double wl = 0.25 * op.pen * (iJm + iJp) * dS;
    // common gradient of the velocity
    double gc[DIM][DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c)
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        double s = 0.0, s2 = 0.0;
        if (P > 0)
#pragma unroll
          for (int m = 0; m < n1; ++m) {
            s = fma(lo[m], Gb[(c * NW + k) * plane + (size_t)e * N + line_point<DIM, P>(d, fp, m)], s);
            if (!bnd) s2 = fma(ln[m], Gb[(c * NW + k) * plane + (size_t)en * N + line_point<DIM, P>(dn, fp2, m)], s2);
          }
        gc[c][k] = fma(wl * nrm[c], dq[k], 0.5 * (s + (bnd ? s : s2)));
      }
    double div = 0.0;
#pragma unroll
    for (int c = 0; c < DIM; ++c) div += gc[c][c];
    const double sgn = plus ? dS : -dS;
#pragma unroll
    for (int w = 0; w < DIM; ++w) {
      double tn = (-2.0 / 3.0) * div * nrm[w];
#pragma unroll
      for (int c = 0; c < DIM; ++c) tn = fma(gc[c][w] + gc[w][c], nrm[c], tn);
      B[Y_::oTn + tf * DIM + w] = sgn * tn;
      B[Y_::oN + tf * DIM + w] = sgn * nrm[w];
      B[Y_::oUc + tf * DIM + w] = uc[w];
      B[Y_::oLf + tf * DIM + w] = 2.0 * wl * nrm[w];
    }
  }
  __syncthreads();
  // points: stress of the corrected gradient, the line-diagonal operators K
  for (int t = tid; t < ne * N; t += nt) {
    const int le = t / N, pt = t - le * N;
    double* B = base(le);
    const double iJ = B[Y_::oIJ + pt];
    const double* Ja = B + Y_::oJa + pt * DIM * DIM;
    double gr[DIM][DIM], u[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
      u[k] = B[Y_::oV + k * N + pt];
#pragma unroll
      for (int c = 0; c < DIM; ++c) gr[c][k] = P > 0 ? Gb[(c * NW + k) * plane + (size_t)e0 * N + t] : 0.0;
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
        const int i = coord<DIM, P>(pt, d), fp = face_point<DIM, P>(pt, d);
        const double cor = iJ * fma(sg[0][i], B[Y_::oQj + (face_of<DIM>(d, 0) * NF + fp) * NW + k],
                                    sg[1][i] * B[Y_::oQj + (face_of<DIM>(d, 1) * NF + fp) * NW + k]);
#pragma unroll
        for (int c = 0; c < DIM; ++c) gr[c][k] = fma(Ja[d * DIM + c], cor, gr[c][k]);
      }
    }
    double div = 0.0;
#pragma unroll
    for (int c = 0; c < DIM; ++c) div += gr[c][c];
#pragma unroll
    for (int c = 0; c < DIM; ++c)
#pragma unroll
      for (int w = 0; w < DIM; ++w)
        B[Y_::oTau + (pt * DIM + c) * DIM + w] = gr[c][w] + gr[w][c] - (c == w ? (2.0 / 3.0) * div : 0.0);
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const double* a = Ja + d * DIM;
      const double a2 = iJ * dotv<DIM>(a, a), i3 = iJ * (1.0 / 3.0), ua = dotv<DIM>(u, a);
      double* K = B + Y_::oK + (pt * DIM + d) * KN;
      int x = 0;
#pragma unroll
      for (int i = 0; i < DIM; ++i)
#pragma unroll
        for (int w = i; w < DIM; ++w) K[x++] = fma(i3 * a[i], a[w], i == w ? a2 : 0.0);
#pragma unroll
      for (int w = 0; w < DIM; ++w) K[x++] = fma(i3 * ua, a[w], a2 * u[w]);
      K[x] = a2;
    }
  }
  // face gradient per unit perturbation at a point c of the face's normal line:
  // trace of the broken-gradient tangent (along the line, and at c across it)
  for (int t = tid; t < ne * F * N; t += nt) {
    const int le = t / (F * N), r = t - le * F * N, f = r / N, cp = r - f * N, e = face_dir<DIM>(f);
    double* B = base(le);
    const double* l = sl[face_plus<DIM>(f) ? 1 : 0];
    const int ce = coord<DIM, P>(cp, e), p0 = cp - ce * stride_of<P>(e);
    double y[DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c) y[c] = 0.0;
#pragma unroll
    for (int m = 0; m < n1; ++m) {
      const int pm = p0 + m * stride_of<P>(e);
      const double s = l[m] * sD[m][ce] * B[Y_::oIJ + pm];
#pragma unroll
      for (int c = 0; c < DIM; ++c) y[c] = fma(s, B[Y_::oJa + (pm * DIM + e) * DIM + c], y[c]);
    }
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      if (d == e) continue;
      const int cd = coord<DIM, P>(cp, d);
      const double s = l[ce] * sD[cd][cd] * B[Y_::oIJ + cp];
#pragma unroll
      for (int c = 0; c < DIM; ++c) y[c] = fma(s, B[Y_::oJa + (cp * DIM + d) * DIM + c], y[c]);
    }
#pragma unroll
    for (int c = 0; c < DIM; ++c) B[Y_::oYb + (f * N + cp) * DIM + c] = sGf[le][f] * y[c];
  }
  __syncthreads();

  // contribution of r's e-line when c differs from r in d (and maybe in e):
  // the one point m of that line on c's d-line
  auto off_line = [&](ViscAcc<DIM>& acc, const double* B, int le, int rp, int e, int d, int ce, int cd) {
    const int re = coord<DIM, P>(rp, e), rd = coord<DIM, P>(rp, d), pm = rp + (ce - re) * stride_of<P>(e);
    const double iJ = B[Y_::oIJ + pm];
    double Yv[DIM], X[DIM], u[DIM], X1[DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c) {
      Yv[c] = iJ * B[Y_::oJa + (pm * DIM + d) * DIM + c];
      X1[c] = B[Y_::oJa + (pm * DIM + e) * DIM + c];
      u[c] = B[Y_::oV + c * N + pm];
    }
    const double dt = sDt[re][ce], av = dt * sCd[le][d][0][rd][cd], aT = dt * sCd[le][d][1][rd][cd];
    const double xy = dotv<DIM>(X1, Yv);
    acc.energy(av, xy, X1, Yv, u);
    acc.tt = fma(aT, xy, acc.tt);
#pragma unroll
    for (int c = 0; c < DIM; ++c) X[c] = av * X1[c];
    const int fp = face_point<DIM, P>(rp, e);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int f = face_of<DIM>(e, s), tf = f * NF + fp;
      const double cf = sg[s][re] * sGf[le][f] * sl[s][ce] * sD[rd][cd], we = sWe[le][f] * cf;
      const double* Nf = B + Y_::oN + tf * DIM;
      const double ny = dotv<DIM>(Nf, Yv);
      acc.energy(we, ny, Nf, Yv, B + Y_::oUc + tf * DIM);
      acc.tt = fma(we, ny, acc.tt);
#pragma unroll
      for (int c = 0; c < DIM; ++c) X[c] = fma(cf, Nf[c], X[c]);
    }
    acc.mom(X, Yv);
  };
  // contribution of the e-line that r and c share
  auto on_line = [&](ViscAcc<DIM>& acc, const double* B, int le, int rp, int cp, int e) {
    const int re = coord<DIM, P>(rp, e), ce = coord<DIM, P>(cp, e), p0 = cp - ce * stride_of<P>(e);
#pragma unroll
    for (int m = 0; m < n1; ++m) {
      const double dt = sDt[re][m], av = dt * sCd[le][e][0][m][ce], aT = dt * sCd[le][e][1][m][ce];
      const double* K = B + Y_::oK + ((p0 + m * stride_of<P>(e)) * DIM + e) * KN;
      int x = 0;
#pragma unroll
      for (int i = 0; i < DIM; ++i)
#pragma unroll
        for (int w = i; w < DIM; ++w) {
          acc.m[i][w] = fma(av, K[x], acc.m[i][w]);
          if (w != i) acc.m[w][i] = fma(av, K[x], acc.m[w][i]);
          ++x;
        }
#pragma unroll
      for (int w = 0; w < DIM; ++w) acc.en[w] = fma(av, K[x++], acc.en[w]);
      acc.tt = fma(aT, K[x], acc.tt);
    }
    const double dt = sDt[re][ce], iJ = B[Y_::oIJ + cp];
    const double* Xe = B + Y_::oJa + (cp * DIM + e) * DIM;
    double u[DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c) u[c] = B[Y_::oV + c * N + cp];
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      if (d == e) continue;
      const int cd = coord<DIM, P>(cp, d);
      double Yd[DIM], X[DIM];
      const double av = dt * sCd[le][d][0][cd][cd], aT = dt * sCd[le][d][1][cd][cd];
#pragma unroll
      for (int c = 0; c < DIM; ++c) {
        Yd[c] = iJ * B[Y_::oJa + (cp * DIM + d) * DIM + c];
        X[c] = av * Xe[c];
      }
      const double xy = dotv<DIM>(Xe, Yd);
      acc.mom(X, Yd);
      acc.energy(av, xy, Xe, Yd, u);
      acc.tt = fma(aT, xy, acc.tt);
    }
    // the perturbed velocity's work against the stress
#pragma unroll
    for (int w = 0; w < DIM; ++w) {
      double s = 0.0;
#pragma unroll
      for (int c = 0; c < DIM; ++c) s = fma(Xe[c], B[Y_::oTau + (cp * DIM + c) * DIM + w], s);
      acc.en[w] = fma(dt, s, acc.en[w]);
    }
    const int fp = face_point<DIM, P>(cp, e);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int f = face_of<DIM>(e, s), tf = f * NF + fp;
      const double g = sg[s][re], lc = sl[s][ce], kv = sKap[le][f][0] * lc, kT = sKap[le][f][1] * lc,
                   we = sWe[le][f] * g;
      const double* Nf = B + Y_::oN + tf * DIM;
      double Yv[DIM], X[DIM], ny = 0.0, nyT = 0.0;
#pragma unroll
      for (int c = 0; c < DIM; ++c) {
        const double lf = B[Y_::oLf + tf * DIM + c], yb = B[Y_::oYb + (f * N + cp) * DIM + c];
        Yv[c] = fma(kv, lf, yb);
        ny = fma(Nf[c], Yv[c], ny);
        nyT = fma(Nf[c], fma(kT, lf, yb), nyT);
        X[c] = g * Nf[c];
      }
      acc.mom(X, Yv);
      acc.energy(we, ny, Nf, Yv, B + Y_::oUc + tf * DIM);
      acc.tt = fma(we, nyT, acc.tt);
      const double wt = we * (lc + kv);   // q_com's velocity follows by 1 + kappa
#pragma unroll
      for (int w = 0; w < DIM; ++w) acc.en[w] = fma(wt, B[Y_::oTn + tf * DIM + w], acc.en[w]);
    }
  };
  auto store = [&](const ViscAcc<DIM>& acc, const double* B, int le, int rp, int cp, bool add) {
    const double s = -ph.mu * B[Y_::oIJ + rp], sT = -ph.kT * B[Y_::oIJ + rp];
    double* Db = Dout + (size_t)(e0 + le) * n * n + (size_t)(N + rp) * n + N + cp;
#pragma unroll
    for (int w = 0; w < DIM; ++w) {
#pragma unroll
      for (int i = 0; i < DIM; ++i) {
        double* p = Db + (size_t)i * N * n + w * N;
        *p = add ? fma(s, acc.m[i][w], *p) : s * acc.m[i][w];
      }
      double* p = Db + (size_t)DIM * N * n + w * N;
      *p = add ? fma(s, acc.en[w], *p) : s * acc.en[w];
    }
    double* p = Db + (size_t)DIM * N * n + DIM * N;
    *p = add ? fma(sT, acc.tt, *p) : sT * acc.tt;
  };
  // points that differ in two coordinates (the inviscid block is zero there)
  if (P > 0) {
    constexpr int M = n1 > 1 ? n1 - 1 : 1, PD = DIM == 3 ? 3 : 1, W2 = PD * M * M;
    for (int t = tid; t < ne * N * W2; t += nt) {
      const int le = t / (N * W2), u = t - le * N * W2, rp = u / W2, x = u - rp * W2, pd = x / (M * M), mm = x - pd * M * M;
      const int d = pd == 2 ? 1 : 0, e = pd == 0 ? 1 : 2;
      const int rd = coord<DIM, P>(rp, d), re = coord<DIM, P>(rp, e);
      const int cd = mm % M >= rd ? mm % M + 1 : mm % M, ce = mm / M >= re ? mm / M + 1 : mm / M;
      const double* B = base(le);
      ViscAcc<DIM> acc;
      acc.zero();
      off_line(acc, B, le, rp, e, d, ce, cd);
      off_line(acc, B, le, rp, d, e, cd, ce);
      store(acc, B, le, rp, rp + (cd - rd) * stride_of<P>(d) + (ce - re) * stride_of<P>(e), false);
    }
    // points of one line
    constexpr int W1 = DIM * M;
    for (int t = tid; t < ne * N * W1; t += nt) {
      const int le = t / (N * W1), u = t - le * N * W1, rp = u / W1, x = u - rp * W1, d = x / M, m = x - d * M;
      const int rd = coord<DIM, P>(rp, d), cd = m >= rd ? m + 1 : m, cp = rp + (cd - rd) * stride_of<P>(d);
      const double* B = base(le);
      ViscAcc<DIM> acc;
      acc.zero();
      on_line(acc, B, le, rp, cp, d);
#pragma unroll 1
      for (int k = 1; k < DIM; ++k) {
        const int e = (d + k) % DIM;
        off_line(acc, B, le, rp, e, d, coord<DIM, P>(rp, e), cd);
      }
      store(acc, B, le, rp, cp, true);
    }
  }
  for (int t = tid; t < ne * N; t += nt) {
    const int le = t / N, rp = t - le * N;
    const double* B = base(le);
    ViscAcc<DIM> acc;
    acc.zero();
#pragma unroll 1
    for (int e = 0; e < DIM; ++e) on_line(acc, B, le, rp, rp, e);
    store(acc, B, le, rp, rp, true);
  }
}

namespace {

template <int DIM, int P>
void assemble_call(const Ctx& c, const LevelDev& L, const double* q, const double* d_dtau, double inv_odt,
                   cudaStream_t s) {
  using A = AsmShape<DIM, P>;
  const int* nbr = c.d_faces + 5 * c.n_faces;   // neighbour table stored after the face list
  assemble_kernel<DIM, P><<<(c.E + A::EPB - 1) / A::EPB, A::kThreads, A::smem, s>>>(
      c.E, q, L.met, L.face, nbr, L.op, c.ph, d_dtau, inv_odt, L.Dfull);
  if (c.ph.mu > 0.0) {
    using V = ViscShape<DIM, P>;
    if (DIM == 3) launch_grad3(c, L, q, s);
    else launch_grad(c, L, q, s);
    assemble_visc_kernel<DIM, P><<<(c.E + V::EPB - 1) / V::EPB, V::kThreads, V::smem, s>>>(
        c.E, q, L.Gb, L.met, L.face, L.fJinv, nbr, L.op, c.ph, L.Dfull);
  }
}

template <int DIM, int P>
cudaError_t assemble_prep() {
  const cudaError_t e = cudaFuncSetAttribute(assemble_kernel<DIM, P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)AsmShape<DIM, P>::smem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(assemble_visc_kernel<DIM, P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)ViscShape<DIM, P>::smem);
}

}  // namespace

void launch_assemble(const Ctx& c, const LevelDev& L, const double* q, const double* d_dtau, double inv_odt,
                     cudaStream_t s) {
  if (c.dim == 3) {
    switch (L.P) {
      case 0: assemble_call<3, 0>(c, L, q, d_dtau, inv_odt, s); break;
      case 1: assemble_call<3, 1>(c, L, q, d_dtau, inv_odt, s); break;
      case 2: assemble_call<3, 2>(c, L, q, d_dtau, inv_odt, s); break;
      default: assemble_call<3, 3>(c, L, q, d_dtau, inv_odt, s); break;
    }
    return;
  }
  switch (L.P) {
    case 0: assemble_call<2, 0>(c, L, q, d_dtau, inv_odt, s); break;
    case 1: assemble_call<2, 1>(c, L, q, d_dtau, inv_odt, s); break;
    case 2: assemble_call<2, 2>(c, L, q, d_dtau, inv_odt, s); break;
    case 3: assemble_call<2, 3>(c, L, q, d_dtau, inv_odt, s); break;
    case 4: assemble_call<2, 4>(c, L, q, d_dtau, inv_odt, s); break;
    default: assemble_call<2, 5>(c, L, q, d_dtau, inv_odt, s); break;
  }
}

// Dynamic shared memory of the assembly kernels (once, outside any capture).
cudaError_t prepare_assemble(const Ctx& c) {
  for (int l = 0; l < c.cfg.n_levels; ++l) {
    cudaError_t e;
    if (c.dim == 3) {
      switch (c.lev[l].P) {
        case 0: e = assemble_prep<3, 0>(); break;
        case 1: e = assemble_prep<3, 1>(); break;
        case 2: e = assemble_prep<3, 2>(); break;
        default: e = assemble_prep<3, 3>(); break;
      }
    } else {
      switch (c.lev[l].P) {
        case 0: e = assemble_prep<2, 0>(); break;
        case 1: e = assemble_prep<2, 1>(); break;
        case 2: e = assemble_prep<2, 2>(); break;
        case 3: e = assemble_prep<2, 3>(); break;
        case 4: e = assemble_prep<2, 4>(); break;
        default: e = assemble_prep<2, 5>(); break;
      }
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace pmg
