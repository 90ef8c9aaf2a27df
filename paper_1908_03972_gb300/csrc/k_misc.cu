// k_misc.cu -- P-level transfers (Section 3) and ESDIRK stage arithmetic
// (Section 2.4, eqs. ESDIRK_ns and ESDIRK_primitive), all FP64 and HBM-bound.
#include "pmg_internal.h"

namespace pmg {

// ------------------------------------------------------------------ stages
__global__ void cons_kernel(size_t plane, Phys ph, const double* __restrict__ q, double* __restrict__ qc) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= plane) return;
  double qq[4] = {q[i], q[plane + i], q[2 * plane + i], q[3 * plane + i]}, o[4];
  cons(qq, ph, o);
  for (int v = 0; v < 4; ++v) qc[v * plane + i] = o[v];
}

struct RPtrs {
  const double* p[6];
  double coef[6];
};

// src = (q_c^n + dt sum_j a_ij R^j) / (omega dt); without q_c^n (split form of
// the stage system, where q_c^n enters through q_c(q) - q_c(q^n)) only the
// R-sum part is formed.
__global__ void stage_src_kernel(size_t tot, const double* __restrict__ qcn, RPtrs R, int nr, double dt,
                                 double inv_odt, double* __restrict__ src) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= tot) return;
  double acc = qcn ? qcn[i] : 0.0;
  for (int j = 0; j < nr; ++j) acc += dt * R.coef[j] * R.p[j][i];
  src[i] = acc * inv_odt;
}

// q_c^{n+1} = q_c^n + dt sum_i b_i R^i, then back to primitive variables.
// Formed as increments of q^n (gauge pressure p - p_ref): the new pressure is
// p^n + (gamma-1) (d(rho E) - d(rho |v|^2 / 2)), so neither rho E ~ 1/Ma^2 nor
// p is rounded on the way.
__global__ void bsum_kernel(size_t plane, Phys ph, const double* __restrict__ qn, RPtrs R, int nr, double dt,
                            double* __restrict__ q) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= plane) return;
  double d[4];
  for (int v = 0; v < 4; ++v) {
    double acc = 0.0;
    for (int j = 0; j < nr; ++j) acc += R.coef[j] * R.p[j][v * plane + i];
    d[v] = dt * acc;
  }
  double pn = qn[i], un = qn[plane + i], vn = qn[2 * plane + i], Tn = qn[3 * plane + i];
  double rhon = (pn + ph.p_ref) / Tn;
  double rho = rhon + d[0];
  double mu = rhon * un + d[1], mv = rhon * vn + d[2];
  double u = mu / rho, w = mv / rho;
  double dke = 0.5 * (mu * u + mv * w) - 0.5 * rhon * (un * un + vn * vn);
  double p = pn + ph.gm1 * (d[3] - dke);
  q[i] = p;
  q[plane + i] = u;
  q[2 * plane + i] = w;
  q[3 * plane + i] = (p + ph.p_ref) / rho;
}

// Gauge conversion of the pressure plane: q[0..plane) += delta.
__global__ void shift_kernel(size_t plane, double delta, double* __restrict__ q) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < plane) q[i] += delta;
}

void launch_shift_pressure(size_t plane, double delta, double* q, cudaStream_t s) {
  if (delta == 0.0) return;
  shift_kernel<<<(unsigned)((plane + 255) / 256), 256, 0, s>>>(plane, delta, q);
}

// out = in with the pressure plane shifted: the gauge conversion of a state
// between device buffers in one launch (a copy and a shift take 6 + 2 us for
// 1.2 MB, this 2).  8-byte accesses, the alignment a caller's buffer has.
__global__ void __launch_bounds__(256) copy_shift_kernel(size_t plane, size_t n, double delta,
                                                         const double* __restrict__ in, double* __restrict__ out) {
  const size_t i0 = (size_t)blockIdx.x * 1024 + threadIdx.x;
  double v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = i0 + 256 * k < n ? __ldg(in + i0 + 256 * k) : 0.0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const size_t i = i0 + 256 * k;
    if (i < n) out[i] = i < plane ? v[k] + delta : v[k];
  }
}

void launch_copy_shift(size_t plane, size_t n, double delta, const double* in, double* out, cudaStream_t s) {
  copy_shift_kernel<<<(unsigned)((n + 1023) / 1024), 256, 0, s>>>(delta == 0.0 ? 0 : plane, n, delta, in, out);
}

void launch_cons(const Ctx& c, int N, const double* q, double* qc, cudaStream_t s) {
  size_t plane = (size_t)c.E * N;
  cons_kernel<<<(unsigned)((plane + 255) / 256), 256, 0, s>>>(plane, c.ph, q, qc);
}

void launch_stage_src(const Ctx& c, int N, const double* qcn, double* const* R, const double* a, int nr,
                      double dt, double inv_odt, double* src, cudaStream_t s) {
  RPtrs rp;
  for (int j = 0; j < 6; ++j) { rp.p[j] = j < nr ? R[j] : nullptr; rp.coef[j] = j < nr ? a[j] : 0.0; }
  size_t tot = (size_t)c.nv * c.E * N;
  stage_src_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(tot, qcn, rp, nr, dt, inv_odt, src);
}

void launch_bsum_update(const Ctx& c, int N, const double* qn, double* const* R, const double* b, int nr,
                        double dt, double* q, cudaStream_t s) {
  if (c.dim == 3) { launch_bsum_update3(c, N, qn, R, b, nr, dt, q, s); return; }
  RPtrs rp;
  for (int j = 0; j < 6; ++j) { rp.p[j] = j < nr ? R[j] : nullptr; rp.coef[j] = j < nr ? b[j] : 0.0; }
  size_t plane = (size_t)c.E * N;
  bsum_kernel<<<(unsigned)((plane + 255) / 256), 256, 0, s>>>(plane, c.ph, qn, rp, nr, dt, q);
}

// dtau_min of the CFL form (Section 2.4) on the finest level: per element
// (dx/(P+1)) / max(c + |v|) and (dx/(P+1))^2 min(rho) / mu, then the minimum
// over all elements (per-block minima, then one block).
__global__ void dtau_elem_kernel(int E, int N, int P, const double* __restrict__ q, const double* __restrict__ dx,
                                 Phys ph, double* __restrict__ partial) {
  __shared__ double red[128];
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  double best = 1e300;
  if (e < E) {
    const size_t plane = (size_t)E * N;
    double smax = 0.0, rmin = 1e300;
    for (int p = 0; p < N; ++p) {
      const size_t i = (size_t)e * N + p;
      const double pr = q[i] + ph.p_ref, u = q[plane + i], v = q[2 * plane + i], T = q[3 * plane + i];
      smax = fmax(smax, sqrt(ph.gamma * T) + sqrt(u * u + v * v));
      rmin = fmin(rmin, pr / T);
    }
    const double hP = dx[e] / (P + 1);
    best = hP / smax;
    if (ph.mu > 0.0) best = fmin(best, hP * hP * rmin / ph.mu);
  }
  red[threadIdx.x] = best;
  __syncthreads();
  for (int w = 64; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] = fmin(red[threadIdx.x], red[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

__global__ void min_final_kernel(const double* __restrict__ partial, int n, double* __restrict__ out) {
  __shared__ double red[256];
  double m = 1e300;
  for (int i = threadIdx.x; i < n; i += 256) m = fmin(m, partial[i]);
  red[threadIdx.x] = m;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] = fmin(red[threadIdx.x], red[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = red[0];
}

void launch_dtau_min(const Ctx& c, double* partial, double* out, cudaStream_t s) {
  const LevelDev& L = c.lev[0];
  const int blocks = (c.E + 127) / 128;
  dtau_elem_kernel<<<blocks, 128, 0, s>>>(c.E, L.N, L.P, L.q, c.d_dx, c.ph, partial);
  min_final_kernel<<<1, 256, 0, s>>>(partial, blocks, out);
}

}  // namespace pmg
