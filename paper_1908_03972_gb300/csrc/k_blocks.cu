// k_blocks.cu -- element-Jacobi smoother blocks (Section 2.4, eqs.
// linearized_pseudo_transient_final and smoothing_element_jacobi).
//
//  * assemble (k_assemble.cu): D_e = Gamma/dtau + M/(omega dt) - dR_e/dq_e in
//    FP64, exact, neighbour states frozen.
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
