// k3_misc.cu -- ESDIRK stage arithmetic (Section 2.4) on hexahedra, FP64.
#include "pmg_internal.h"

namespace pmg {

// q_c^{n+1} = q_c^n + dt sum_i b_i R^i back to primitive variables, formed as
// increments of q^n (gauge pressure), as in 2D.
struct RPtrs3 {
  const double* p[6];
  double coef[6];
};

__global__ void bsum3_kernel(size_t plane, Phys ph, const double* __restrict__ qn, RPtrs3 R, int nr, double dt,
                             double* __restrict__ q) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= plane) return;
  double d[5];
  for (int v = 0; v < 5; ++v) {
    double acc = 0.0;
    for (int j = 0; j < nr; ++j) acc += R.coef[j] * R.p[j][v * plane + i];
    d[v] = dt * acc;
  }
  const double pn = qn[i], Tn = qn[4 * plane + i];
  const double vn[3] = {qn[plane + i], qn[2 * plane + i], qn[3 * plane + i]};
  const double rhon = (pn + ph.p_ref) / Tn;
  const double rho = rhon + d[0];
  double vel[3], ke_new = 0.0, ke_old = 0.0;
  for (int c = 0; c < 3; ++c) {
    const double m = rhon * vn[c] + d[1 + c];
    vel[c] = m / rho;
    ke_new += m * vel[c];
    ke_old += rhon * vn[c] * vn[c];
  }
  const double p = pn + ph.gm1 * (d[4] - 0.5 * (ke_new - ke_old));
  q[i] = p;
  for (int c = 0; c < 3; ++c) q[(1 + c) * plane + i] = vel[c];
  q[4 * plane + i] = (p + ph.p_ref) / rho;
}

void launch_bsum_update3(const Ctx& c, int N, const double* qn, double* const* R, const double* b, int nr,
                         double dt, double* q, cudaStream_t s) {
  RPtrs3 rp;
  for (int j = 0; j < 6; ++j) { rp.p[j] = j < nr ? R[j] : nullptr; rp.coef[j] = j < nr ? b[j] : 0.0; }
  const size_t plane = (size_t)c.E * N;
  bsum3_kernel<<<(unsigned)((plane + 255) / 256), 256, 0, s>>>(plane, c.ph, qn, rp, nr, dt, q);
}

}  // namespace pmg
