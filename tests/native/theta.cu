// The theta contraction of complex128 states on its own (test infrastructure).
#include "gate_kernels.cuh"

using namespace mpsv;

// Host arrays: Bl (chi_l, 2, chi_m), Br (chi_m, 2, chi_r), the 4 x 4 gate and C
// (2 chi_l, 2 chi_r), complex128.  Returns a CUDA error code.
extern "C" int theta_c128(int chi_l, int chi_m, int chi_r, const double* Bl, const double* Br, const double* gate,
                          double* C) {
  const size_t nl = (size_t)chi_l * 2 * chi_m, nr = (size_t)chi_m * 2 * chi_r, nc = (size_t)4 * chi_l * chi_r;
  double2* d;
  DevGate* dg;
  int* dchi;
  cudaError_t e = cudaMalloc(&d, (nl + nr + nc) * sizeof(double2));
  if (e == cudaSuccess) e = cudaMalloc(&dg, sizeof(DevGate));
  if (e == cudaSuccess) e = cudaMalloc(&dchi, 3 * sizeof(int));
  if (e != cudaSuccess) return e;
  DevGate g = {};
  g.arity = 2;
  for (int i = 0; i < 16; ++i) g.u[i] = make_double2(gate[2 * i], gate[2 * i + 1]);
  const int chi[3] = {chi_l, chi_m, chi_r};
  cudaMemcpy(d, Bl, nl * sizeof(double2), cudaMemcpyHostToDevice);
  cudaMemcpy(d + nl, Br, nr * sizeof(double2), cudaMemcpyHostToDevice);
  cudaMemcpy(dg, &g, sizeof(g), cudaMemcpyHostToDevice);
  cudaMemcpy(dchi, chi, sizeof(chi), cudaMemcpyHostToDevice);
  theta_kernel<double><<<dim3((chi_r + kTile - 1) / kTile, (chi_l + kTile - 1) / kTile), dim3(kTile, kTile)>>>(
      d, d + nl, dg, dchi, 0, d + nl + nr);
  e = cudaMemcpy(C, d + nl + nr, nc * sizeof(double2), cudaMemcpyDeviceToHost);
  cudaFree(d);
  cudaFree(dg);
  cudaFree(dchi);
  return e;
}
