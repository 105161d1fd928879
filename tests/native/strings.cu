// The kernels that sum string values, on their own (test infrastructure).
#include <vector>

#include "energy_kernels.cuh"

using namespace mpsv;

namespace {
template <typename T> T* up(const T* host, size_t n) {
  T* d = nullptr;
  if (cudaMalloc(&d, n * sizeof(T)) != cudaSuccess) return nullptr;
  cudaMemcpy(d, host, n * sizeof(T), cudaMemcpyHostToDevice);
  return d;
}
}  // namespace

// One leaf with operator op: B (chi_l, 2, chi_r), M (chi_l, 2, chi_r), complex128;
// weight (chi_r, nullable).
extern "C" int leaf_c128(int chi_l, int chi_r, int op, const double* B, const double* M, const double* weight,
                         double* value) {
  const size_t n = (size_t)2 * chi_l * chi_r;
  double2 *dB = up((const double2*)B, n), *dM = up((const double2*)M, n);
  double* dw = weight ? up(weight, chi_r) : nullptr;
  const int4 leaf = make_int4(0, op, 0, 0);
  int4* dl = up(&leaf, 1);
  double* dv = up(value, 1);
  EnvLevel lv = {};
  lv.leaf = dl;
  lv.n_leaves = 1;
  lv.chi_l = chi_l;
  lv.chi_r = chi_r;
  lv.weight = dw;
  env_leaf_kernel<double><<<1, 128>>>(dM, dB, lv, dv);
  const cudaError_t e = cudaMemcpy(value, dv, sizeof(double), cudaMemcpyDeviceToHost);
  for (void* p : {(void*)dB, (void*)dM, (void*)dw, (void*)dl, (void*)dv}) cudaFree(p);
  return e;
}

// n strings of one prefix: L and n matrices R (chi x chi, Hermitian, complex128).
extern "C" int cross_c128(int chi, int n, const double* L, const double* R, double* values) {
  const size_t size = (size_t)chi * chi;
  double2 *dL = up((const double2*)L, size), *dR = up((const double2*)R, n * size);
  std::vector<int2> pair;
  for (int i = 0; i < n; ++i) pair.push_back(make_int2(i, i));
  const int4 item = make_int4(0, 0, n, 0);
  int2* dp = up(pair.data(), n);
  int4* di = up(&item, 1);
  double* dv = up(values, n);
  env_cross_kernel<double><<<1, 128>>>(dL, dR, chi, di, dp, dv);
  const cudaError_t e = cudaMemcpy(values, dv, n * sizeof(double), cudaMemcpyDeviceToHost);
  for (void* p : {(void*)dL, (void*)dR, (void*)dp, (void*)di, (void*)dv}) cudaFree(p);
  return e;
}
