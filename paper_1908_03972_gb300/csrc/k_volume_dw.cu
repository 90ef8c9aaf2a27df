// k_volume_dw.cu -- the residual-and-update of an element-Jacobi sweep
// (volume_kernel with APPLY, k_residual.cu) in double-word arithmetic.
//
// The sweep q += cs .* (D^-1 (rs .* F)) is the smoother, and on the coarse
// levels it only drives the FAS corrections of Section 3; the binary64
// residual of the finest level (a separate evaluation) defines the converged
// state.  Forming F on the FP32 pipes (dword.cuh, ~2^-46 relative rounding)
// instead of in binary64 takes the kernel's longest chain, ~130 FP64
// instructions per thread at one FP64 warp-instruction per ~64 cycles per SM
// sub-partition, off the FP64 pipe.
//
// Same steps and CTA shape as the binary64 kernel: contravariant fluxes of
// the element's points, the divergence of each line Dt F + gL F_com(-1) +
// gR F_com(+1) (the extrapolated part of the DG correction folded into Dt: the
// separate jump stage it replaces was a quarter of the kernel's instructions
// and a barrier), the level-system epilogue F = R - (q_c(q) - q_c(q_ref)) /
// (omega dt) + src - S (q_c(q) itself without q_ref), then the block update.
// The face launch of a sweep leaves its fluxes as double-words, so neither
// side converts them.  4096 elements, FP32 blocks (one GB300): P = 1 7.3 -> 6.1
// us, P = 2 10.5 -> 8.0 us, P = 3 14.7 -> 13.4 us (there the block stream
// bounds it).  The states hold gauge
// pressure; with p_ref = 0 (absolute pressure, p ~ 1/(gamma Ma^2) in the
// momentum flux) the binary64 kernel is used.
#include "sweep_common.cuh"

namespace pmg {

template <int P, class W, int EPB>
__global__ void __launch_bounds__(256, 1) volume_apply_dw_kernel(
    int E, double* q, const dw* __restrict__ met, const dw* __restrict__ Fcom, OpTabW opw, PhysW k,
    double inv_odt, const double* __restrict__ src, const double* __restrict__ S, const double* __restrict__ qref,
    const W* __restrict__ Dinv, const double* __restrict__ rs, const double* __restrict__ cs,
    double* __restrict__ werr) {
  constexpr int n1 = P + 1, N = n1 * n1, n = 4 * N;
  using PF = VolPrefetch<P, W, EPB>;
  extern __shared__ __align__(128) unsigned char dsm[];
  __shared__ __align__(8) unsigned long long mbar[2];   // 0: face fluxes, 1: blocks and scales
  using Acc = typename Blk<W>::acc;
  __shared__ Acc sr[EPB][n];
  __shared__ dw sFt[EPB][4][N];
  __shared__ dw sGt[EPB][4][N];
  __shared__ dw sD[n1][n1], sgL[n1], sgR[n1];   // Dt, -gL (the fluxes are outward), gR

  const int le = threadIdx.x / N, pt = threadIdx.x - le * N;
  const int e = blockIdx.x * EPB + le;
  const bool active = (le < EPB) && (e < E);
  const size_t plane = (size_t)E * N;
  const size_t fplane = (size_t)E * 4 * n1;
  W* sDinv = reinterpret_cast<W*>(dsm);
  double* srs = reinterpret_cast<double*>(dsm + PF::dinv_bytes);
  double* scs = srs + EPB * n;
  dw* sFc = reinterpret_cast<dw*>(scs + EPB * n);   // [v][local element][face][k]
  if (threadIdx.x == 0) {
    const int e0 = blockIdx.x * EPB, ne = min(EPB, E - e0);
    const unsigned bF = (unsigned)(ne * 4 * n1 * sizeof(dw));
    const unsigned bS = (unsigned)(ne * n * sizeof(double));
    const unsigned bD = PF::blocks ? (unsigned)((size_t)ne * n * n * sizeof(W)) : 0u;
    mbar_init(&mbar[0]);
    mbar_init(&mbar[1]);
    mbar_arrive_expect(&mbar[0], 4 * bF);
#pragma unroll
    for (int v = 0; v < 4; ++v)
      bulk_g2s(sFc + v * EPB * 4 * n1, Fcom + v * fplane + (size_t)e0 * 4 * n1, bF, &mbar[0]);
    mbar_arrive_expect(&mbar[1], 2 * bS + bD);
    bulk_g2s(srs, rs + (size_t)e0 * n, bS, &mbar[1]);
    bulk_g2s(scs, cs + (size_t)e0 * n, bS, &mbar[1]);
    if (PF::blocks) bulk_g2s(sDinv, Dinv + (size_t)e0 * n * n, bD, &mbar[1]);
  }
  const size_t gi = (size_t)e * N + pt;
  // Sv: src - S of the epilogue
  double qq[4] = {0, 0, 0, 0}, qo[4] = {0, 0, 0, 0}, Sv[4] = {0, 0, 0, 0};
  dw mt[5] = {};
  if (active) {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      qq[v] = q[v * plane + gi];
      if (qref) qo[v] = __ldg(qref + v * plane + gi);
      if (src) Sv[v] = __ldg(src + v * plane + gi);
      if (S) Sv[v] = src ? Sv[v] - __ldg(S + v * plane + gi) : -__ldg(S + v * plane + gi);
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) mt[c] = met[c * plane + gi];
  }
  if (threadIdx.x < n1 * n1) sD[threadIdx.x / n1][threadIdx.x % n1] = opw.Dt[threadIdx.x / n1][threadIdx.x % n1];
  if (threadIdx.x < n1) {
    sgL[threadIdx.x] = -opw.gL[threadIdx.x];
    sgR[threadIdx.x] = opw.gR[threadIdx.x];
  }

  dw Q[4], rho = {0.0f, 0.0f};
  if (active) {
#pragma unroll
    for (int v = 0; v < 4; ++v) Q[v] = dw_from_double(qq[v]);   // gauge p, u, v, T
    rho = (Q[0] + k.p_ref) * rcp(Q[3]);
    // Cartesian fluxes with the gauge pressure in the momentum rows; at P = 0
    // the line operator Dt is zero and only the face fluxes remain
    if (P > 0) {
      const dw H = mul_add(k.Cp, Q[3], half(dot2(Q[1], Q[1], Q[2], Q[2])));
      const dw mx = rho * Q[1], my = rho * Q[2];
      const dw f[4] = {mx, mul_add(mx, Q[1], Q[0]), mx * Q[2], mx * H};
      const dw g[4] = {my, f[2], mul_add(my, Q[2], Q[0]), my * H};
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        sFt[le][v][pt] = dot2(mt[0], f[v], mt[1], g[v]);
        sGt[le][v][pt] = dot2(mt[2], f[v], mt[3], g[v]);
      }
    }
  }
  __syncthreads();
  const bool okF = mbar_wait0(&mbar[0], k.wait_ns);
  if (!okF) *werr = 1.0;
  const bool okS = mbar_wait0(&mbar[1], k.wait_ns);
  if (!okS) *werr = 1.0;
  if (active) {
    const int i = pt % n1, j = pt / n1;
    dw qc[4];
    if (qref) {
      // q_c(q) - q_c(q_ref), energy through p / (gamma - 1) + rho |v|^2 / 2
      // with the gauge-pressure difference (no p ~ 1/Ma^2 is rounded)
      dw Qo[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) Qo[v] = dw_from_double(qo[v]);
      const dw rhoo = (Qo[0] + k.p_ref) * rcp(Qo[3]);
      qc[0] = rho - rhoo;
      qc[1] = dot2(rho, Q[1], -rhoo, Qo[1]);
      qc[2] = dot2(rho, Q[2], -rhoo, Qo[2]);
      qc[3] = mul_add(Q[0] - Qo[0], k.inv_gm1,
                      half(dot2(rho, dot2(Q[1], Q[1], Q[2], Q[2]), -rhoo, dot2(Qo[1], Qo[1], Qo[2], Qo[2]))));
    } else {
      qc[0] = rho;
      qc[1] = rho * Q[1];
      qc[2] = rho * Q[2];
      qc[3] = rho * (Q[3] * k.inv_gm1 + half(Q[1] * Q[1] + Q[2] * Q[2]));
    }
    const dw ninvJ = -mt[4];
    const dw nodt = dw_from_double(-inv_odt);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      dw_acc acc;
      if (P > 0)
#pragma unroll
        for (int m = 0; m < n1; ++m) {
          acc.add_prod(sD[i][m], sFt[le][v][j * n1 + m]);
          acc.add_prod(sD[j][m], sGt[le][v][m * n1 + i]);
        }
      dw com[4];
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const int kk = (f == 1 || f == 3) ? j : i;
        com[f] = okF ? sFc[((v * EPB + le) * 4 + f) * n1 + kk] : Fcom[v * fplane + ((size_t)e * 4 + f) * n1 + kk];
      }
      acc.add_prod(sgL[i], com[3]);
      acc.add_prod(sgR[i], com[1]);
      acc.add_prod(sgL[j], com[0]);
      acc.add_prod(sgR[j], com[2]);
      // F = -acc / |J| - qc / (omega dt) + src - S
      const dw F = dot2_add(acc.value(), ninvJ, qc[v], nodt, dw_from_double(Sv[v]));
      const int row = v * N + pt;
      sr[le][row] = scaled_in_dw<W>(F, okS ? srs[le * n + row] : rs[(size_t)e * n + row]);
    }
  }
  __syncthreads();
  if (active) {
    // thread (le, pt) owns rows 4 pt .. 4 pt + 3 of its element's block
    Acc acc[4] = {0, 0, 0, 0};
    if (PF::blocks && okS) {
      const W* Dm = sDinv + (size_t)le * n * n + 4 * pt;
#pragma unroll 8
      for (int kk = 0; kk < n; ++kk) {
        const Acc rk = sr[le][kk];
        Acc d[4];
        ld4(Dm + (size_t)kk * n, d);
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[m] = fma(d[m], rk, acc[m]);
      }
    } else {
      const W* Dm = Dinv + (size_t)e * n * n + 4 * pt;
#pragma unroll 8
      for (int kk = 0; kk < n; ++kk) {
        const Acc rk = sr[le][kk];
        Acc d[4];
        ldg4(Dm + (size_t)kk * n, d);
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[m] = fma(d[m], rk, acc[m]);
      }
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int row = 4 * pt + m;
      const int v = row / N, p2 = row - v * N;
      const size_t o = v * plane + (size_t)e * N + p2;
      const double csc = okS ? scs[le * n + row] : cs[(size_t)e * n + row];
      q[o] = q[o] + scaled_out<W>(acc[m], csc);
    }
  }
  // copies still in flight land before the CTA exits
  if (!okF) mbar_drain0(&mbar[0]);
  if (!okS) mbar_drain0(&mbar[1]);
}

template <class W>
static void dw_dispatch(const Ctx& c, const LevelDev& L, double* q, double inv_odt, const double* src,
                        const double* S, const double* qref, cudaStream_t s) {
  const W* Dinv = (const W*)L.Dinv;
#define PMG_VDW_E(PP, EP)                                                                                   \
  do {                                                                                                      \
    constexpr int epb = EP<PP>::value, threads = elem_threads<PP, epb>();                                   \
    volume_apply_dw_kernel<PP, W, epb><<<(c.E + epb - 1) / epb, threads, VolPrefetch<PP, W, epb>::smem, s>>>( \
        c.E, q, L.metW, reinterpret_cast<const dw*>(L.Fcom), L.opw, c.phw, inv_odt, src, S, qref, Dinv, L.rs, \
        L.cs, c.d_scal + 1);                                                                                \
  } while (0)
#define PMG_VDW(PP)                                                \
  if (few_elems(PP, c.E, c.sms, c.cfg.block_prec, true)) PMG_VDW_E(PP, FewElemsPerBlock); \
  else PMG_VDW_E(PP, ElemsPerBlock)
  switch (L.P) {
    case 0: PMG_VDW(0); break;
    case 1: PMG_VDW(1); break;
    case 2: PMG_VDW(2); break;
    case 3: PMG_VDW(3); break;
    case 4: PMG_VDW(4); break;
    default: PMG_VDW(5); break;
  }
#undef PMG_VDW
#undef PMG_VDW_E
}

bool volume_dw_applies(const Ctx& c) {
  return c.dim == 2 && flux_dw_sweep(c) && c.ph.mu == 0.0 && c.ph.p_ref != 0.0;
}

void launch_volume_apply_dw(const Ctx& c, const LevelDev& L, double* q, double inv_odt, const double* src,
                            const double* S, const double* qref, int prec, cudaStream_t s) {
  if (prec == PMG_PREC_FP64) dw_dispatch<double>(c, L, q, inv_odt, src, S, qref, s);
  else if (prec == PMG_PREC_BF16R) dw_dispatch<__nv_bfloat16>(c, L, q, inv_odt, src, S, qref, s);
  else dw_dispatch<float>(c, L, q, inv_odt, src, S, qref, s);
}

template <class W>
static cudaError_t prep_dw(int P, bool few) {
#define PMG_PDW_E(PP, EP)                                                                                  \
  return cudaFuncSetAttribute(volume_apply_dw_kernel<PP, W, EP<PP>::value>,                                \
                              cudaFuncAttributeMaxDynamicSharedMemorySize,                                 \
                              (int)VolPrefetch<PP, W, EP<PP>::value>::smem)
#define PMG_PDW(PP)                        \
  if (few) PMG_PDW_E(PP, FewElemsPerBlock); \
  PMG_PDW_E(PP, ElemsPerBlock)
  switch (P) {
    case 0: PMG_PDW(0);
    case 1: PMG_PDW(1);
    case 2: PMG_PDW(2);
    case 3: PMG_PDW(3);
    case 4: PMG_PDW(4);
    default: PMG_PDW(5);
  }
#undef PMG_PDW
#undef PMG_PDW_E
}

cudaError_t prepare_volume_dw_kernels(const Ctx& c) {
  for (int l = 0; l < c.cfg.n_levels; ++l) {
    const bool few = few_elems(c.lev[l].P, c.E, c.sms, c.cfg.block_prec, true);
    cudaError_t e = c.cfg.block_prec == PMG_PREC_FP64    ? prep_dw<double>(c.lev[l].P, few)
                    : c.cfg.block_prec == PMG_PREC_BF16R ? prep_dw<__nv_bfloat16>(c.lev[l].P, few)
                                                         : prep_dw<float>(c.lev[l].P, few);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace pmg
