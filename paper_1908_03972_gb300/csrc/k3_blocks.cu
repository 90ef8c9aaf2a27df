// k3_blocks.cu -- application of the element-Jacobi blocks on hexahedra
// (Section 2.4, eq. smoothing_element_jacobi, d = 3): x = cs .* (D^-1 (rs .* r))
// with the factored inverse (column-major); one thread per solution point forms
// its point's five rows, so the threads of an element read every column
// contiguously.  Bound by the stream of the inverses, so ten columns' loads are
// in flight per thread.
// Assembly and factorisation: k_assemble.cu, k_factor.cu.
#include "pmg_internal.h"
#include "physics3.cuh"

namespace pmg {

template <class W, int P>
__global__ void __launch_bounds__(64) apply3_kernel(int E, const W* __restrict__ Dinv, const double* __restrict__ rs,
                                                    const double* __restrict__ cs, const double* __restrict__ r,
                                                    double* __restrict__ x, int accumulate) {
  constexpr int N = (P + 1) * (P + 1) * (P + 1), n = 5 * N;
  constexpr int EPB = N <= 32 ? 64 / N : 1;
  using Acc = typename Blk<W>::acc;
  __shared__ Acc sr[EPB][n];
  const int le = threadIdx.x / N, pt = threadIdx.x - le * N;
  const int e = blockIdx.x * EPB + le;
  const bool active = (le < EPB) && (e < E);
  const size_t plane = (size_t)E * N;
  if (active) {
#pragma unroll
    for (int v = 0; v < 5; ++v)
      sr[le][v * N + pt] = scaled_in<W>(r[v * plane + (size_t)e * N + pt], rs[(size_t)e * n + v * N + pt]);
  }
  __syncthreads();
  if (!active) return;
  Acc acc[5] = {0, 0, 0, 0, 0};
  const W* Dm = Dinv + (size_t)e * n * n + pt;
#pragma unroll 10
  for (int k = 0; k < n; ++k) {
    const Acc rk = sr[le][k];
#pragma unroll
    for (int v = 0; v < 5; ++v) acc[v] = fma(blk_val(__ldg(Dm + (size_t)k * n + v * N)), rk, acc[v]);
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const double xv = scaled_out<W>(acc[v], cs[(size_t)e * n + v * N + pt]);
    const size_t o = v * plane + (size_t)e * N + pt;
    if (accumulate) x[o] += xv;
    else x[o] = xv;
  }
}

template <class W>
static void apply3_dispatch(const Ctx& c, const LevelDev& L, const double* r, double* x, int acc, cudaStream_t s) {
  const W* Dinv = (const W*)L.Dinv;
  const int N = L.N;
  const int epb = N <= 32 ? 64 / N : 1;
  const int threads = (epb * N + 31) / 32 * 32, blocks = (c.E + epb - 1) / epb;
#define PMG_AP3(PP) apply3_kernel<W, PP><<<blocks, threads, 0, s>>>(c.E, Dinv, L.rs, L.cs, r, x, acc)
  switch (L.P) {
    case 0: PMG_AP3(0); break;
    case 1: PMG_AP3(1); break;
    case 2: PMG_AP3(2); break;
    default: PMG_AP3(3); break;
  }
#undef PMG_AP3
}

void launch_apply3(const Ctx& c, const LevelDev& L, int prec, const double* r, double* x, int accumulate,
                   cudaStream_t s) {
  if (prec == PMG_PREC_FP64) apply3_dispatch<double>(c, L, r, x, accumulate, s);
  else if (prec == PMG_PREC_BF16R) apply3_dispatch<__nv_bfloat16>(c, L, r, x, accumulate, s);
  else apply3_dispatch<float>(c, L, r, x, accumulate, s);
}

}  // namespace pmg
