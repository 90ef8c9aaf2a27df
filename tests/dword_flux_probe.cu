// dword_flux_probe.cu -- test driver for the sums of products of dword.cuh and
// the double-word face flux of physics_dw.cuh (built and run by
// tests/test_gpu_dword_flux.py; not part of the library).
//
// Input: n, then gamma, eps_min and p_ref, then n rows of 21 binary64 values
// (raw little-endian): six factors a .. f, the reference p and T, the traces sm
// and sp of both sides (four each), nx, ny, dS.
// Output per row, as (h, l) FP32 words: dw(a) .. dw(f), a b + c, a b + c d,
// a b + c d + e, a b + c d + e f, and the face flux with the pressure term in
// binary64 (four) and in double-word (four).
#include <cstdio>
#include <vector>

#include "../paper_1908_03972_gb300/csrc/physics_dw.cuh"

using pmg::dw;

constexpr int kIn = 21, kOut = 18;

__global__ void probe(int n, pmg::PhysW k, const double* in, dw* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double* x = in + (size_t)i * kIn;
  dw* o = out + (size_t)i * kOut;
  dw a[6];
  for (int j = 0; j < 6; ++j) o[j] = a[j] = pmg::dw_from_double(x[j]);
  o[6] = pmg::mul_add(a[0], a[1], a[2]);
  o[7] = pmg::dot2(a[0], a[1], a[2], a[3]);
  o[8] = pmg::dot2_add(a[0], a[1], a[2], a[3], a[4]);
  o[9] = pmg::dot3(a[0], a[1], a[2], a[3], a[4], a[5]);
  const double *sm = x + 8, *sp = x + 12, *g = x + 16;
  double dq[4];
  for (int v = 0; v < 4; ++v) dq[v] = sp[v] - sm[v];
  const dw nx = pmg::dw_from_double(g[0]), ny = pmg::dw_from_double(g[1]), dS = pmg::dw_from_double(g[2]);
  pmg::face_roe_dw<true>(x[6], x[7], sm, sp, dq, nx, ny, dS, g, k, o + 10);
  pmg::face_roe_dw<false>(x[6], x[7], sm, sp, dq, nx, ny, dS, g, k, o + 14);
}

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  FILE* f = fopen(argv[1], "rb");
  if (!f) return 3;
  int n = 0;
  double c[3];
  if (fread(&n, sizeof(int), 1, f) != 1 || n <= 0 || n > (1 << 20) || fread(c, sizeof(double), 3, f) != 3) return 4;
  std::vector<double> in((size_t)n * kIn);
  if (fread(in.data(), sizeof(double), in.size(), f) != in.size()) return 5;
  fclose(f);
  pmg::Phys ph = {};
  ph.gamma = c[0];
  ph.gm1 = c[0] - 1.0;
  ph.Cp = c[0] / (c[0] - 1.0);
  ph.eps_min = c[1];
  ph.p_ref = c[2];
  ph.inv_gamma = 1.0 / c[0];
  ph.inv_gm1 = 1.0 / (c[0] - 1.0);
  ph.inv_Cp = (c[0] - 1.0) / c[0];
  double* din;
  dw* dout;
  if (cudaMalloc(&din, in.size() * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&dout, (size_t)n * kOut * sizeof(dw)) != cudaSuccess)
    return 6;
  cudaMemcpy(din, in.data(), in.size() * sizeof(double), cudaMemcpyHostToDevice);
  probe<<<(n + 127) / 128, 128>>>(n, pmg::make_physw(ph), din, dout);
  std::vector<dw> out((size_t)n * kOut);
  cudaMemcpy(out.data(), dout, out.size() * sizeof(dw), cudaMemcpyDeviceToHost);
  const cudaError_t e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    fprintf(stderr, "CUDA error: %s\n", cudaGetErrorString(e));
    return 7;
  }
  FILE* o = fopen(argv[2], "wb");
  if (!o) return 8;
  fwrite(out.data(), sizeof(dw), out.size(), o);
  fclose(o);
  return 0;
}
