// sweep_common.cuh -- CTA shapes and shared-memory prefetch layout of the
// residual-and-update kernels (binary64 and double-word variants).
#pragma once
#include "pmg_internal.h"

namespace pmg {

// Elements per CTA of the volume kernels.  Their threads are bound by FP64
// issue (binary64: 2 DFMA per clock per SM) or by the latency of their chain
// (double-word), so small CTAs of one or two warps spread even the coarse
// levels (4096 elements) over all 152 SMs.  An FP64 instruction takes its
// 64 cycles whatever the active lanes, so the points should fill their warps:
// at P = 4 five elements (125 of 128 lanes; two filled 50 of 64) take the
// residual of 16384 viscous elements from 136 to 110 us and the BF16 update
// from 231 to 204, although the five inverses no longer fit the prefetch; at
// P = 5 three (108 of 128; one filled 36 of 64) take 1073 elements from 16.2
// to 12.5 us.
// On few elements the updates are bound by the latency of their loads and chain
// instead, and in double-word with FP32 or BF16 blocks, off the FP64 pipe, at any
// size at P = 4: there they take two and one (FewElemsPerBlock).  us a sweep at
// P = 4, five / two elements:
//   binary64 viscous, BF16: 27.0 / 23.9 on 100 elements, 33.3 / 27.9 on 784, 41.2 /
//     44.1 on 1600; FP32: 33.6 / 30.7 on 784, 59.2 / 54.3 on 2304, 102 / 106 on 4096;
//   double-word, BF16: 15.4 / 14.1 on 100, 66.4 / 59.8 on 6400, 138 / 133 on 16384;
//     FP32: 16.0 / 15.3, 79.4 / 76.2, 166 / 168; FP64: 28.5 / 28.3, 147 / 171.
// P = 5, three / one: double-word FP32 17.8 / 16.6 on 100 elements, 19.5 / 19.1 on
// 400, 21.4 / 20.9 on 784, BF16 20.4 / 21.1 there; binary64 FP32 24.0 / 22.9 on 100,
// 24.8 / 25.8 on 400.  The residual alone gains nothing from it.
template <int P>
struct ElemsPerBlock {
  static constexpr int N = (P + 1) * (P + 1);
  static constexpr int value = P == 0 ? 32 : P == 1 ? 8 : P == 2 ? 7 : P == 3 ? 4 : P == 4 ? 5 : 3;
};
template <int P>
struct FewElemsPerBlock {
  static constexpr int value = P == 4 ? 2 : P == 5 ? 1 : ElemsPerBlock<P>::value;
};
inline bool few_elems(int P, int E, int sms, int prec, bool dword) {
  const bool light = dword && prec != PMG_PREC_FP64;
  if (P == 4) return light || E <= (prec == PMG_PREC_FP32 ? 20 : 8) * sms;
  return P == 5 && E <= (light ? 4 : 1) * sms;
}
template <int P, int EPB>
constexpr int elem_threads() { return (EPB * (P + 1) * (P + 1) + 31) / 32 * 32; }

// Prefetch layout of the residual-and-update sweep: the CTA's common face
// fluxes, block scales and (where they fit, VolPrefetch::blocks) block
// inverses are copied to shared memory by bulk asynchronous copies issued at
// entry, and the reference and forcing states are loaded into registers
// there too: the latency of these reads then overlaps the flux arithmetic
// instead of adding one L2 round trip per phase.
template <int P, class W, int EPB>
struct VolPrefetch {
  static constexpr int n1 = P + 1, N = n1 * n1, n = 4 * N;
  static constexpr bool blocks = (size_t)EPB * n * n * sizeof(W) <= 40 * 1024;
  static constexpr size_t dinv_bytes = blocks ? (size_t)EPB * n * n * sizeof(W) : 0;
  static constexpr size_t scale_bytes = (size_t)EPB * n * sizeof(double);   // rs, then cs
  static constexpr size_t flux_bytes = (size_t)EPB * 4 * n1 * sizeof(double);   // per equation
  static constexpr size_t smem = dinv_bytes + 2 * scale_bytes + 4 * flux_bytes;
};

// Loads four consecutive block entries (16-byte aligned for float, 32 for double).
__device__ __forceinline__ void ld4(const float* p, float a[4]) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  a[0] = t.x; a[1] = t.y; a[2] = t.z; a[3] = t.w;
}
__device__ __forceinline__ void ld4(const double* p, double a[4]) {
  const double2 t0 = reinterpret_cast<const double2*>(p)[0], t1 = reinterpret_cast<const double2*>(p)[1];
  a[0] = t0.x; a[1] = t0.y; a[2] = t1.x; a[3] = t1.y;
}
__device__ __forceinline__ void ldg4(const float* p, float a[4]) {
  const float4 t = __ldg(reinterpret_cast<const float4*>(p));
  a[0] = t.x; a[1] = t.y; a[2] = t.z; a[3] = t.w;
}
__device__ __forceinline__ void ldg4(const double* p, double a[4]) {
  const double2 t0 = __ldg(reinterpret_cast<const double2*>(p)), t1 = __ldg(reinterpret_cast<const double2*>(p) + 1);
  a[0] = t0.x; a[1] = t0.y; a[2] = t1.x; a[3] = t1.y;
}
// BF16 entries (8 bytes, 8-byte aligned), widened to FP32.
__device__ __forceinline__ void bf4_to_f(uint2 u, float a[4]) {
  const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  a[0] = lo.x; a[1] = lo.y; a[2] = hi.x; a[3] = hi.y;
}
__device__ __forceinline__ void ld4(const __nv_bfloat16* p, float a[4]) {
  bf4_to_f(*reinterpret_cast<const uint2*>(p), a);
}
__device__ __forceinline__ void ldg4(const __nv_bfloat16* p, float a[4]) {
  bf4_to_f(__ldg(reinterpret_cast<const uint2*>(p)), a);
}

// rs .* F of a double-word F in the block precision W (rs: powers of two).
template <class W>
__device__ __forceinline__ typename Blk<W>::acc scaled_in_dw(dw F, double s);
template <>
__device__ __forceinline__ float scaled_in_dw<float>(dw F, double s) {
  return __fmul_rn(__fadd_rn(F.h, F.l), (float)s);
}
template <>
__device__ __forceinline__ double scaled_in_dw<double>(dw F, double s) {
  return dw_to_double(F) * s;
}
template <>
__device__ __forceinline__ float scaled_in_dw<__nv_bfloat16>(dw F, double s) {
  return __fmul_rn(__fadd_rn(F.h, F.l), (float)s);
}

}  // namespace pmg
