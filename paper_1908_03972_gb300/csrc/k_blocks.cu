// k_blocks.cu -- element-Jacobi smoother blocks (Section 2.4, eqs.
// linearized_pseudo_transient_final and smoothing_element_jacobi).
//
//  * assemble: one CTA per element builds D_e = Gamma/dtau + M/(omega dt)
//    - dR_e/dq_e in FP64.  dR_e/dq_e is exact: pointwise flux Jacobians and
//    the own-side derivative of the preconditioned Roe flux (including its
//    dependence through the averaged state) come from forward-mode dual
//    numbers pushed through the same flux code as the residual; the FR
//    structure (derivative, extrapolation, correction) is applied in
//    tensor-product form.  Neighbour states are frozen.
//  * factor (k_factor.cu): the block equilibrated with power-of-two row and
//    column scales (exact in any precision) and inverted by Gauss-Jordan
//    elimination with partial pivoting in the working precision (FP64, or FP32
//    for the mixed-precision smoother).  The explicit inverse turns every
//    smoothing sweep into a batched matrix-vector product.  The equilibrated
//    rows have unit size, so a pivot that is not finite or not above n eps of
//    the working precision (the rounding a dependent row leaves after
//    elimination) marks a block that is singular to that precision: the
//    element is flagged for the host (PMG_ESINGULAR).
//  * apply: x = cs .* (inv(D^) (rs .* r)); each thread owns four consecutive
//    rows and streams the column-major inverse with 16-byte (FP32) or
//    2x16-byte (FP64) loads.  This stream is the smoother's HBM/L2 traffic.
#include <cstdint>
#include <algorithm>

#include "pmg_internal.h"

namespace pmg {

// ------------------------------------------------------------------ assemble
template <int P>
__global__ void __launch_bounds__(128) assemble_kernel(int E, const double* __restrict__ q,
                                                       const double* __restrict__ met,
                                                       const double* __restrict__ face,
                                                       const int* __restrict__ nbr, OpTab op, Phys ph,
                                                       const double* __restrict__ d_dtau, double inv_odt,
                                                       double* __restrict__ Dout) {
  constexpr int n1 = P + 1, N = n1 * n1, n = 4 * N;
  __shared__ double sq[4][N];
  __shared__ double sAx[N][16], sAe[N][16], sDiag[N][16];
  __shared__ double sC[4][n1][16];
  __shared__ double sinvJ[N];
  __shared__ double sD[n1][n1], sgL[n1], sgR[n1], slm[n1], slp[n1];
  const int e = blockIdx.x;
  const size_t plane = (size_t)E * N;
  const double dtau = *d_dtau;
  for (int t = threadIdx.x; t < 4 * N; t += blockDim.x) sq[t / N][t % N] = q[(t / N) * plane + (size_t)e * N + t % N];
  if (threadIdx.x < n1 * n1) sD[threadIdx.x / n1][threadIdx.x % n1] = op.D[threadIdx.x / n1][threadIdx.x % n1];
  if (threadIdx.x < n1) {
    sgL[threadIdx.x] = op.gL[threadIdx.x];
    sgR[threadIdx.x] = op.gR[threadIdx.x];
    slm[threadIdx.x] = op.lm[threadIdx.x];
    slp[threadIdx.x] = op.lp[threadIdx.x];
  }
  __syncthreads();
  // pointwise contravariant flux Jacobians and the pseudo/physical time terms
  for (int pt = threadIdx.x; pt < N; pt += blockDim.x) {
    size_t gi = (size_t)e * N + pt;
    double a = met[gi], b = met[plane + gi], c = met[2 * plane + gi], d = met[3 * plane + gi];
    sinvJ[pt] = met[4 * plane + gi];
    double qv[4] = {sq[0][pt] + ph.p_ref, sq[1][pt], sq[2][pt], sq[3][pt]};   // absolute pressure
    for (int w = 0; w < 4; ++w) {
      Dual qd[4];
      for (int k = 0; k < 4; ++k) qd[k] = Dual(qv[k], k == w ? 1.0 : 0.0);
      Dual f[4], g[4];
      flux_xy(qd, qd[0] - ph.p_ref, ph, f, g);
      for (int v = 0; v < 4; ++v) {
        sAx[pt][v * 4 + w] = a * f[v].d + b * g[v].d;
        sAe[pt][v * 4 + w] = c * f[v].d + d * g[v].d;
      }
    }
    double G[16], M[16];
    gamma_and_M(qv, ph, G, M);
    for (int i = 0; i < 16; ++i) sDiag[pt][i] = G[i] / dtau + M[i] * inv_odt;
  }
  // own-side derivative of the reference-direction common flux at each face point
  for (int t = threadIdx.x; t < 4 * n1; t += blockDim.x) {
    int f = t / n1, k = t - f * n1;
    const bool plus = (f == 1 || f == 2);
    const bool eta = (f == 0 || f == 2);
    double qm[4], qp[4] = {0.0, 0.0, 0.0, 0.0};
    for (int v = 0; v < 4; ++v) {
      double s = 0.0;
      for (int m = 0; m < n1; ++m) s += (plus ? slp[m] : slm[m]) * sq[v][eta ? m * n1 + k : k * n1 + m];
      qm[v] = s;
    }
    int en = nbr[(e * 4 + f) * 3 + 0], fn = nbr[(e * 4 + f) * 3 + 1], rev = nbr[(e * 4 + f) * 3 + 2];
    int kn = rev ? P - k : k;
    if (en >= 0) {
      const bool pn = (fn == 1 || fn == 2);
      const bool en_eta = (fn == 0 || fn == 2);
      for (int v = 0; v < 4; ++v) {
        double s = 0.0;
        for (int m = 0; m < n1; ++m)
          s += (pn ? slp[m] : slm[m]) * q[v * plane + (size_t)en * N + (en_eta ? m * n1 + kn : kn * n1 + m)];
        qp[v] = s;
      }
      qp[0] += ph.p_ref;
    }
    qm[0] += ph.p_ref;
    const double* g = face + (((size_t)e * 4 + f) * n1 + k) * 3;
    double sg = plus ? 1.0 : -1.0;
    for (int w = 0; w < 4; ++w) {
      Dual dm[4], dp[4], o[4];
      for (int v = 0; v < 4; ++v) { dm[v] = Dual(qm[v], v == w ? 1.0 : 0.0); dp[v] = Dual(qp[v], 0.0); }
      // a boundary face's ghost state follows the own trace (fn = boundary type)
      if (en < 0) ghost_state(fn, dm, g[0], g[1], ph, dp);
      roe_flux(dm, dp, g[0], g[1], g[2], ph, o);
      for (int v = 0; v < 4; ++v) sC[f][k][v * 4 + w] = sg * o[v].d;
    }
  }
  __syncthreads();
  // fill the block: D = diag terms - dR/dq, with dR/dq = -(1/|J|) d(div + corr)/dq
  double* Db = Dout + (size_t)e * n * n;
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    int row = t / n, col = t - row * n;
    int v = row / N, rp = row - v * N, w = col / N, cp = col - w * N;
    int i = rp % n1, j = rp / n1, k = cp % n1, l = cp / n1;
    int vw = v * 4 + w;
    double s = 0.0;
    if (l == j) {   // same xi line
      double A = sAx[cp][vw];
      s += sD[i][k] * A;
      s += sgL[i] * slm[k] * (sC[3][j][vw] - A);
      s += sgR[i] * slp[k] * (sC[1][j][vw] - A);
    }
    if (k == i) {   // same eta line
      double A = sAe[cp][vw];
      s += sD[j][l] * A;
      s += sgL[j] * slm[l] * (sC[0][i][vw] - A);
      s += sgR[j] * slp[l] * (sC[2][i][vw] - A);
    }
    double val = s * sinvJ[rp];
    if (rp == cp) val += sDiag[rp][vw];
    Db[t] = val;
  }
}

void launch_assemble(const Ctx& c, const LevelDev& L, const double* q, const double* d_dtau, double inv_odt,
                     cudaStream_t s) {
  if (c.dim == 3) { launch_assemble3(c, L, q, d_dtau, inv_odt, s); return; }
  const int* nbr = c.d_faces + 5 * c.n_faces;   // neighbour table stored after the face list
#define PMG_ASM(PP) \
  assemble_kernel<PP><<<c.E, 128, 0, s>>>(c.E, q, L.met, L.face, nbr, L.op, c.ph, d_dtau, inv_odt, L.Dfull)
  switch (L.P) {
    case 0: PMG_ASM(0); break;
    case 1: PMG_ASM(1); break;
    case 2: PMG_ASM(2); break;
    case 3: PMG_ASM(3); break;
    case 4: PMG_ASM(4); break;
    default: PMG_ASM(5); break;
  }
#undef PMG_ASM
  if (c.ph.mu > 0.0) launch_assemble_visc(c, L, q, s);
}

// --------------------------------------------------------------------- apply
template <class W> struct Vec4;
template <> struct Vec4<float> {
  __device__ static inline void load(const float* p, float o[4]) {
    float4 t = __ldg(reinterpret_cast<const float4*>(p));
    o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
  }
};
template <> struct Vec4<__nv_bfloat16> {
  __device__ static inline void load(const __nv_bfloat16* p, float o[4]) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
    const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
    const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
    o[0] = lo.x; o[1] = lo.y; o[2] = hi.x; o[3] = hi.y;
  }
};
template <> struct Vec4<double> {
  __device__ static inline void load(const double* p, double o[4]) {
    double2 a = __ldg(reinterpret_cast<const double2*>(p));
    double2 b = __ldg(reinterpret_cast<const double2*>(p) + 1);
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
  }
};

// One thread per four rows of one element's block; N threads per element.
template <int N>
struct ApplyEPB {   // elements per CTA: 1-2 warps per CTA, enough CTAs for all SMs
  static constexpr int value = N <= 4 ? 32 / N : (64 / N > 0 ? 64 / N : 1);
};

template <class W, int N>
__global__ void __launch_bounds__(64) apply_kernel(int E, const W* __restrict__ Dinv, const double* __restrict__ rs,
                                                   const double* __restrict__ cs, const double* __restrict__ r,
                                                   double* __restrict__ x, int accumulate) {
  constexpr int n = 4 * N;
  constexpr int EPB = ApplyEPB<N>::value;
  using Acc = typename Blk<W>::acc;
  __shared__ Acc sr[EPB][n];
  const int le = threadIdx.x / N, t = threadIdx.x - le * N;
  const int e = blockIdx.x * EPB + le;
  const bool active = (le < EPB) && (e < E);
  const size_t plane = (size_t)E * N;
  if (active) {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      int row = v * N + t;
      sr[le][row] = scaled_in<W>(r[v * plane + (size_t)e * N + t], rs[(size_t)e * n + row]);
    }
  }
  __syncthreads();
  if (!active) return;
  Acc acc[4] = {0, 0, 0, 0};
  const W* Dm = Dinv + (size_t)e * n * n + 4 * t;
#pragma unroll 8
  for (int k = 0; k < n; ++k) {
    Acc d[4];
    Vec4<W>::load(Dm + (size_t)k * n, d);
    Acc rk = sr[le][k];
    acc[0] = fma(d[0], rk, acc[0]);
    acc[1] = fma(d[1], rk, acc[1]);
    acc[2] = fma(d[2], rk, acc[2]);
    acc[3] = fma(d[3], rk, acc[3]);
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    int row = 4 * t + m;
    int v = row / N, pt = row - v * N;
    double xv = scaled_out<W>(acc[m], cs[(size_t)e * n + row]);
    size_t o = v * plane + (size_t)e * N + pt;
    if (accumulate) x[o] += xv;
    else x[o] = xv;
  }
}

template <class W>
static void apply_dispatch(const Ctx& c, const LevelDev& L, const W* Dinv, const double* r, double* x, int acc,
                           cudaStream_t s) {
  int N = L.N;
  int epb = 1;
  switch (N) {
    case 1: epb = ApplyEPB<1>::value; break;
    case 4: epb = ApplyEPB<4>::value; break;
    case 9: epb = ApplyEPB<9>::value; break;
    case 16: epb = ApplyEPB<16>::value; break;
    case 25: epb = ApplyEPB<25>::value; break;
    default: epb = ApplyEPB<36>::value; break;
  }
  int threads = ((epb * N) + 31) / 32 * 32;
  int blocks = (c.E + epb - 1) / epb;
#define PMG_APPLY(NN) apply_kernel<W, NN><<<blocks, threads, 0, s>>>(c.E, Dinv, L.rs, L.cs, r, x, acc)
  switch (N) {
    case 1: PMG_APPLY(1); break;
    case 4: PMG_APPLY(4); break;
    case 9: PMG_APPLY(9); break;
    case 16: PMG_APPLY(16); break;
    case 25: PMG_APPLY(25); break;
    default: PMG_APPLY(36); break;
  }
#undef PMG_APPLY
}

void launch_apply(const Ctx& c, const LevelDev& L, int prec, const double* r, double* x, int accumulate,
                  cudaStream_t s) {
  if (c.dim == 3) { launch_apply3(c, L, prec, r, x, accumulate, s); return; }
  if (prec == PMG_PREC_FP64) apply_dispatch<double>(c, L, (const double*)L.Dinv, r, x, accumulate, s);
  else if (prec == PMG_PREC_BF16R)
    apply_dispatch<__nv_bfloat16>(c, L, (const __nv_bfloat16*)L.Dinv, r, x, accumulate, s);
  else apply_dispatch<float>(c, L, (const float*)L.Dinv, r, x, accumulate, s);
}

}  // namespace pmg
