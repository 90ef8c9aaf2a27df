// k_transfer.cu -- transfers between P-levels (Section 3): restriction (L2
// projection) and prolongation (interpolation), tensor products of 1D operators
// on quadrilaterals (DIM = 2) and hexahedra (DIM = 3), binary64.
//
// A field of one element goes through one 1D operator per direction in shared
// memory (sum factorisation), all lanes on FP64 work: a P = 3 to 2 restriction
// takes 84 FMAs per field in 2D and 444 in 3D, where forming each output from
// its whole tensor product took 180 and 2268.  The sums run in the same order,
// so the results are the same bit for bit.  The V-cycle restricts the state and
// the defect in one launch.  Measured on one GB300, us (before: one launch per
// field kind): restrict P = 3 to 2 on 4096 quads 14.2 (two
// launches) -> 7.9, prolong 12.9 -> 5.8; 4 to 2 on 16384 quads 68.8 -> 34.0 and
// 69.2 -> 22.2; 3 to 2 on 960 hexes 47.6 -> 10.6 and 43.2 -> 7.3; 2 to 1 on
// 2304 hexes 21.6 -> 8.6 and 15.9 -> 6.0.
#include "pmg_internal.h"

namespace pmg {

namespace {

__host__ __device__ constexpr int ipow(int b, int e) { return e == 0 ? 1 : b * ipow(b, e - 1); }

// Fields (one variable of one element) per CTA: about 256 fine points.
template <int DIM, int PF>
struct Fields {
  static constexpr int Nf = ipow(PF + 1, DIM), value = 256 / Nf < 1 ? 1 : 256 / Nf;
};
constexpr int kXferThreads = 128;

// out[f][r][o][l] = sum_m A[o][m] in[f][r][m][l]: operator A (no x ni) along the
// direction with L points below it and R above it, over nf fields.
template <int no, int ni, int L, int R>
__device__ __forceinline__ void apply_1d(const double (*A)[ni], const double* in, double* out, int nf) {
  for (int t = threadIdx.x; t < nf * R * no * L; t += kXferThreads) {
    const int l = t % L, o = (t / L) % no, fr = t / (L * no);
    double s = 0.0;
#pragma unroll
    for (int m = 0; m < ni; ++m) s = fma(A[o][m], in[(fr * ni + m) * L + l], s);
    out[t] = s;
  }
}

}  // namespace

// blockIdx.y = 0: out = R in (and out2, if any, the same); 1: outd = -R ind.
template <int DIM, int PF, int PC>
__global__ void __launch_bounds__(kXferThreads) restrict_kernel(int nfields, XferTab X, const double* __restrict__ in,
                                                                double* __restrict__ out, double* __restrict__ out2,
                                                                const double* __restrict__ ind,
                                                                double* __restrict__ outd) {
  constexpr int nf = PF + 1, nc = PC + 1, Nf = ipow(nf, DIM), Nc = ipow(nc, DIM), FB = Fields<DIM, PF>::value;
  __shared__ double sR[nc][nf];
  __shared__ double b0[FB * Nf], b1[FB * Nf];
  const int f0 = blockIdx.x * FB, n = min(FB, nfields - f0);
  const bool second = blockIdx.y == 1;
  const double* src = second ? ind : in;
  if (threadIdx.x < nc * nf) sR[threadIdx.x / nf][threadIdx.x % nf] = X.R[threadIdx.x / nf][threadIdx.x % nf];
  for (int t = threadIdx.x; t < n * Nf; t += kXferThreads) b0[t] = __ldg(src + (size_t)f0 * Nf + t);
  __syncthreads();
  apply_1d<nc, nf, 1, Nf / nf>(sR, b0, b1, n);
  __syncthreads();
  apply_1d<nc, nf, nc, Nf / nf / nf>(sR, b1, b0, n);
  __syncthreads();
  if (DIM == 3) {
    apply_1d<nc, nf, nc * nc, 1>(sR, b0, b1, n);
    __syncthreads();
  }
  const double* res = DIM == 3 ? b1 : b0;
  for (int t = threadIdx.x; t < n * Nc; t += kXferThreads) {
    const double s = second ? -res[t] : res[t];
    const size_t o = (size_t)f0 * Nc + t;
    if (second) outd[o] = s;
    else {
      out[o] = s;
      if (out2) out2[o] = s;
    }
  }
}

// qf += I (qc - qcb), or qf = I qc (add = 0, qcb null).
template <int DIM, int PF, int PC>
__global__ void __launch_bounds__(kXferThreads) prolong_kernel(int nfields, XferTab X, const double* __restrict__ qc,
                                                               const double* __restrict__ qcb, double* __restrict__ qf,
                                                               int add) {
  constexpr int nf = PF + 1, nc = PC + 1, Nf = ipow(nf, DIM), Nc = ipow(nc, DIM), FB = Fields<DIM, PF>::value;
  __shared__ double sI[nf][nc];
  __shared__ double b0[FB * Nf], b1[FB * Nf];
  const int f0 = blockIdx.x * FB, n = min(FB, nfields - f0);
  if (threadIdx.x < nf * nc) sI[threadIdx.x / nc][threadIdx.x % nc] = X.I[threadIdx.x / nc][threadIdx.x % nc];
  for (int t = threadIdx.x; t < n * Nc; t += kXferThreads) {
    const size_t o = (size_t)f0 * Nc + t;
    double v = __ldg(qc + o);
    if (qcb) v -= __ldg(qcb + o);
    b0[t] = v;
  }
  __syncthreads();
  apply_1d<nf, nc, 1, Nc / nc>(sI, b0, b1, n);
  __syncthreads();
  apply_1d<nf, nc, nf, Nc / nc / nc>(sI, b1, b0, n);
  __syncthreads();
  if (DIM == 3) {
    apply_1d<nf, nc, nf * nf, 1>(sI, b0, b1, n);
    __syncthreads();
  }
  const double* res = DIM == 3 ? b1 : b0;
  for (int t = threadIdx.x; t < n * Nf; t += kXferThreads) {
    const size_t o = (size_t)f0 * Nf + t;
    if (add) qf[o] += res[t];
    else qf[o] = res[t];
  }
}

#define PMG_PAIRS2(M) M(2, 1, 0) M(2, 2, 0) M(2, 2, 1) M(2, 3, 0) M(2, 3, 1) M(2, 3, 2) M(2, 4, 0) M(2, 4, 1) \
  M(2, 4, 2) M(2, 4, 3) M(2, 5, 0) M(2, 5, 1) M(2, 5, 2) M(2, 5, 3) M(2, 5, 4)
#define PMG_PAIRS3(M) M(3, 1, 0) M(3, 2, 0) M(3, 2, 1) M(3, 3, 0) M(3, 3, 1) M(3, 3, 2)

static void restrict_impl(const Ctx& c, const LevelDev& Lf, const LevelDev& Lc, const XferTab& X, const double* in,
                          double* out, double* out2, const double* ind, double* outd, cudaStream_t s) {
  const int fields = c.nv * c.E;
#define PMG_R(D, A, B)                                                                                         \
  if (c.dim == D && Lf.P == A && Lc.P == B) {                                                                  \
    constexpr int FB = Fields<D, A>::value;                                                                    \
    restrict_kernel<D, A, B><<<dim3((fields + FB - 1) / FB, ind ? 2 : 1), kXferThreads, 0, s>>>(               \
        fields, X, in, out, out2, ind, outd);                                                                  \
    return;                                                                                                    \
  }
  PMG_PAIRS2(PMG_R)
  PMG_PAIRS3(PMG_R)
#undef PMG_R
}

void launch_restrict(const Ctx& c, const LevelDev& Lf, const LevelDev& Lc, const XferTab& X, const double* in,
                     double* out, cudaStream_t s) {
  restrict_impl(c, Lf, Lc, X, in, out, nullptr, nullptr, nullptr, s);
}

void launch_restrict_fas(const Ctx& c, const LevelDev& Lf, const LevelDev& Lc, const XferTab& X, const double* q,
                         double* qc, double* qcb, const double* F, double* Pd, cudaStream_t s) {
  restrict_impl(c, Lf, Lc, X, q, qc, qcb, F, Pd, s);
}

static void prolong_impl(const Ctx& c, const LevelDev& Lf, const LevelDev& Lc, const XferTab& X, const double* qc,
                         const double* qcb, double* qf, int add, cudaStream_t s) {
  const int fields = c.nv * c.E;
#define PMG_P(D, A, B)                                                                                             \
  if (c.dim == D && Lf.P == A && Lc.P == B) {                                                                      \
    constexpr int FB = Fields<D, A>::value;                                                                        \
    prolong_kernel<D, A, B><<<(fields + FB - 1) / FB, kXferThreads, 0, s>>>(fields, X, qc, qcb, qf, add); \
    return;                                                                                                        \
  }
  PMG_PAIRS2(PMG_P)
  PMG_PAIRS3(PMG_P)
#undef PMG_P
}

void launch_prolong_add(const Ctx& c, const LevelDev& Lf, const LevelDev& Lc, const XferTab& X, const double* qc,
                        const double* qcb, double* qf, cudaStream_t s) {
  prolong_impl(c, Lf, Lc, X, qc, qcb, qf, 1, s);
}

void launch_prolong(const Ctx& c, const LevelDev& Lf, const LevelDev& Lc, const XferTab& X, const double* in,
                    double* out, cudaStream_t s) {
  prolong_impl(c, Lf, Lc, X, in, nullptr, out, 0, s);
}

}  // namespace pmg
