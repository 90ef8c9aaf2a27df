// physics3.cuh -- the preconditioning matrix in three dimensions: primitive
// working variables (p absolute, u, v, w, T), R = 1 (Sections 2.1-2.2 with d = 3).
// The fluxes are those of physics.cuh with D = 3.
#pragma once
#include "physics.cuh"

namespace pmg {

__host__ __device__ inline double eps2_of3(const double q[5], const Phys& ph) {
  double ma2 = (q[1] * q[1] + q[2] * q[2] + q[3] * q[3]) / (ph.gamma * q[4]);
  return s_min(1.0, s_max(ph.eps_min * ph.eps_min, ma2));
}

// Gamma (eq. preconditioning) and M = dq_c/dq_p at one point, row-major 5x5.
__host__ __device__ inline void gamma_and_M3(const double q[5], const Phys& ph, double G[25], double M[25]) {
  double p = q[0], T = q[4];
  double rho = p / T, rp = 1.0 / T, rT = -rho / T;
  double H = ph.Cp * T + 0.5 * (q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
  double e2 = eps2_of3(q, ph);
  double Th = 1.0 / (e2 * ph.gamma * T) - rT / (rho * ph.Cp);
  double c0[5] = {1.0, q[1], q[2], q[3], H};
  for (int i = 0; i < 5; ++i) {
    G[i * 5 + 0] = Th * c0[i];
    M[i * 5 + 0] = rp * c0[i];
    G[i * 5 + 4] = M[i * 5 + 4] = rT * c0[i];
    for (int j = 1; j < 4; ++j) G[i * 5 + j] = M[i * 5 + j] = 0.0;
  }
  G[20] -= 1.0; M[20] -= 1.0;
  for (int c = 1; c < 4; ++c) {
    G[c * 5 + c] = M[c * 5 + c] = rho;
    G[20 + c] = M[20 + c] = rho * q[c];
  }
  G[24] += rho * ph.Cp;
  M[24] += rho * ph.Cp;
}

}  // namespace pmg
