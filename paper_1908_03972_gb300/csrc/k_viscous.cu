// k_viscous.cu -- broken (uncorrected) gradients of (u, v, T) at every solution
// point of quadrilaterals (Section 2.1 viscous fluxes; Section 2.3, eqs. com_q
// and com_grad_q), by the Lagrange derivative and the chain rule with the metric
// terms.  The face launch extrapolates them to both sides of each face, the
// volume launch adds the face corrections to them, and the block assembly
// (k_assemble.cu) takes them as the values its tangents are linearised at.
#include "pmg_internal.h"

namespace pmg {

// ----------------------------------------------------------------- gradients
// Broken gradient of (u, v, T): Gb[c * 3 + v] planes, c = x, y.  Derivatives
// are taken of the differences to the element's first value (the derivative
// matrix annihilates constants), which keeps T ~ 1/Ma^2 out of the rounding;
// the differences are formed once per value, in shared memory.  Not run at
// P = 0, where the gradient is zero.
template <int P>
struct GradEPB {
  static constexpr int N = (P + 1) * (P + 1);
  static constexpr int value = P == 1 ? 32 : P == 2 ? 14 : P == 3 ? 8 : P == 4 ? 5 : 7;   // at most 4 idle lanes (P = 3: 0)
  static constexpr int threads = (value * N + 31) / 32 * 32;
};
template <int P>
__global__ void __launch_bounds__(GradEPB<P>::threads) grad_kernel(int E, const double* __restrict__ q,
                                                                   const double* __restrict__ met, OpTab op,
                                                                   double* __restrict__ Gb) {
  constexpr int n1 = P + 1, N = n1 * n1, EPB = GradEPB<P>::value;
  __shared__ double sV[3][EPB * N];
  __shared__ double sD[n1][n1];
  const int e0 = blockIdx.x * EPB, np = min(EPB, E - e0) * N;
  const size_t plane = (size_t)E * N, g0 = (size_t)e0 * N;
  const int t = threadIdx.x, le = t / N, pt = t - le * N, i = pt % n1, j = pt / n1;
  const bool active = t < np;
  if (t < n1 * n1) sD[t / n1][t % n1] = op.D[t / n1][t % n1];
  double a = 0.0, b = 0.0, c = 0.0, d = 0.0;
  if (active) {
    const double iJ = __ldg(met + 4 * plane + g0 + t);
    a = iJ * __ldg(met + g0 + t);
    b = iJ * __ldg(met + plane + g0 + t);
    c = iJ * __ldg(met + 2 * plane + g0 + t);
    d = iJ * __ldg(met + 3 * plane + g0 + t);
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      const double* V = q + (v + 1) * plane + g0;
      sV[v][t] = __ldg(V + t) - __ldg(V + le * N);
    }
  }
  __syncthreads();
  if (!active) return;
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    const double* V = sV[v] + le * N;
    double ax = 0.0, ae = 0.0;
#pragma unroll
    for (int m = 0; m < n1; ++m) {
      ax = fma(sD[i][m], V[j * n1 + m], ax);
      ae = fma(sD[j][m], V[m * n1 + i], ae);
    }
    Gb[v * plane + g0 + t] = fma(a, ax, c * ae);
    Gb[(3 + v) * plane + g0 + t] = fma(b, ax, d * ae);
  }
}

void launch_grad(const Ctx& c, const LevelDev& L, const double* q, cudaStream_t s) {
#define PMG_GRAD(PP)                                                                                      \
  grad_kernel<PP><<<(c.E + GradEPB<PP>::value - 1) / GradEPB<PP>::value, GradEPB<PP>::threads, 0, s>>>( \
      c.E, q, L.met, L.op, L.Gb)
  switch (L.P) {
    case 0: break;   // zero
    case 1: PMG_GRAD(1); break;
    case 2: PMG_GRAD(2); break;
    case 3: PMG_GRAD(3); break;
    case 4: PMG_GRAD(4); break;
    default: PMG_GRAD(5); break;
  }
#undef PMG_GRAD
}

}  // namespace pmg
