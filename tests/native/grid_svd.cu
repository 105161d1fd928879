// The co-resident-grid SVD launched on its own, with the grid barrier's abort
// flag as the caller sets it (test infrastructure).
#include <vector>

#include "svd_jacobi.cuh"

using namespace mpsv;

// SVD of the n x n theta C (host, row-major complex128) by the double-float
// grid kernel; abort != 0: as if one CTA's wait had already run out.  Returns a
// CUDA error code; out = (tc_error, kept singular values or -1 where untouched).
extern "C" int grid_svd(int n, const double* C, int abort, int* out) {
  const SvdWs<ArDF> ws(n, n, true);
  const int P = std::min(128, (n + 3) / 4);
  double2 *dC, *dB, *dBq;
  double *dl, *dln;
  int* dchi;
  char* dws;
  DevReport* drep;
  const size_t mat = (size_t)n * n * sizeof(double2);
  const size_t sizes[] = {mat, mat, mat, n * sizeof(double), n * sizeof(double), 4 * sizeof(int),
                          ws.total + 256, sizeof(DevReport)};
  void** ptrs[] = {(void**)&dC, (void**)&dB, (void**)&dBq, (void**)&dl, (void**)&dln, (void**)&dchi, (void**)&dws,
                   (void**)&drep};
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 8; ++i) {
    if (e == cudaSuccess) e = cudaMalloc(ptrs[i], sizes[i]);
    if (e == cudaSuccess) e = cudaMemset(*ptrs[i], 0, sizes[i]);
  }
  if (e != cudaSuccess) return e;
  const std::vector<double> ones(n, 1.0);
  const int chi[4] = {n / 2, -1, n / 2, 0};
  GridSync* sync = reinterpret_cast<GridSync*>(dws + ws.total);
  const unsigned flag = abort ? 1u : 0u;
  cudaMemcpy(dC, C, mat, cudaMemcpyHostToDevice);
  cudaMemcpy(dl, ones.data(), n * sizeof(double), cudaMemcpyHostToDevice);
  cudaMemcpy(dchi, chi, sizeof(chi), cudaMemcpyHostToDevice);
  cudaMemcpy(&sync->abort, &flag, sizeof(flag), cudaMemcpyHostToDevice);
  SvdParams p;
  p.chi_max = n;
  p.max_sweeps = 60;
  p.trunc_rel = 0.0;
  p.tol = 0.0;
  const size_t smem = std::min(SvdSmem<ArDF>::bytes(n, n, P, false, true), kSvdSmemLimit);
  e = cudaFuncSetAttribute(svd_grid_kernel<ArDF, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.gridDim = dim3(P);
  cfg.blockDim = dim3(kSvdThreads<ArDF>);
  cfg.dynamicSmemBytes = smem;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, svd_grid_kernel<ArDF, double>, static_cast<const double2*>(dC),
                         static_cast<const double*>(dl), dchi, 0, p, dB, dln, drep, dBq, dws, sync, 8, (unsigned)smem);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  DevReport rep;
  int k[4];
  if (e == cudaSuccess) e = cudaMemcpy(&rep, drep, sizeof(rep), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(k, dchi, sizeof(k), cudaMemcpyDeviceToHost);
  for (void** p2 : ptrs) cudaFree(*p2);
  if (e != cudaSuccess) return e;
  out[0] = rep.tc_error;
  out[1] = k[1];
  return 0;
}
