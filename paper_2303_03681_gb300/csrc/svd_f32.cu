// The FP32 truncation SVD (mps_config.svd_fp64 = 0): launch plan and launches
// of svd_cluster.cuh.
#include <algorithm>
#include <mutex>

#include "internal.h"
#include "svd_cluster.cuh"
#include "svd_launch.cuh"

namespace mpsv {

namespace {

// Launch plan for a theta with up to mcap rows and ncap columns (stacked
// columns [A; V] of length mcap + ncap), or P = 0 when the single-CTA kernel
// is used.  The pair steps are latency-bound: few CTAs (fewer rounds and
// cluster barriers) with 16 warps each, so that concurrent evaluations find
// SMs free.  The stacked columns stay in shared memory when the capacities
// allow; otherwise they live in the global workspace, and the kernel still
// keeps them in shared memory whenever the actual sizes fit.
struct PlanF32 {
  int P = 0;
  size_t smem = 0;
  bool global = false;
};

PlanF32 plan_f32(int mcap, int ncap) {
  PlanF32 pl;
  if (ncap < 96) return pl;
  const size_t lim = (size_t)device_limits().smem - 2048;
  const int P = 4, b = (ncap + 2 * P - 1) / (2 * P);
  pl.P = P;
  ClusterSvdSmem<float> L(b, mcap + ncap, 2 * P * b, kClusterMaxThreads);
  if (L.total <= lim) {
    pl.smem = L.total;
  } else {
    pl.global = true;
    pl.smem = std::min(lim, std::max(ClusterSvdSmem<float>(b, 0, 2 * P * b, kClusterMaxThreads).total,
                                     (size_t)160 * 1024));
  }
  return pl;
}

size_t truncate_smem(int mcap, int ncap, bool use_smem) {
  size_t b = (size_t)ncap * (sizeof(double) + sizeof(int)) + 64;
  if (use_smem) b += ((size_t)mcap * ncap + (size_t)ncap * ncap) * sizeof(float2);
  return b;
}

// Entries of the workspace's first part: the column-major theta of the
// single-CTA kernel or the stacked columns of the cluster kernel.
size_t part_a(int mcap, int ncap) {
  return std::max((size_t)mcap * ncap, cluster_svd_workspace(mcap, ncap));
}

template <typename R> void attrs_f32() {
  static std::mutex mu;
  static uint64_t done = 0;
  int dev = 0;
  cudaGetDevice(&dev);
  const int smem = device_limits().smem;
  std::lock_guard<std::mutex> g(mu);
  if (done & (1ull << (dev & 63))) return;
  cudaFuncSetAttribute(svd_truncate_kernel<float, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem - 1024);
  cudaFuncSetAttribute(svd_cluster_kernel<float, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem - 1024);
  done |= 1ull << (dev & 63);
}

template <typename R> void launch_f32(const SvdJob& j) {
  attrs_f32<R>();
  const PlanF32 pl = plan_f32(j.mcap, j.ncap);
  const cplx<R>* C = static_cast<const cplx<R>*>(j.C);
  cplx<R>* B = static_cast<cplx<R>*>(j.Bnext);
  float2* A = reinterpret_cast<float2*>(j.ws);
  if (pl.P) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.P);
    cfg.blockDim = dim3(kClusterMaxThreads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = j.stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = pl.P;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, svd_cluster_kernel<float, R>, C, j.lam_l, j.chi, j.q, j.p, B, j.lam_next, j.rep,
                       pl.global ? A : (float2*)nullptr, (unsigned)pl.smem);
    return;
  }
  const bool use_smem = truncate_smem(j.mcap, j.ncap, true) + 2048 <= (size_t)device_limits().smem;
  const int warps = std::min(32, std::max(1, j.ncap / 2));
  svd_truncate_kernel<float, R><<<1, 32 * warps, truncate_smem(j.mcap, j.ncap, use_smem), j.stream>>>(
      C, j.lam_l, A, A + part_a(j.mcap, j.ncap), use_smem ? 1 : 0, j.chi, j.q, j.p, B, j.lam_next, j.rep);
}

}  // namespace

size_t svd_workspace_f32(int mcap, int ncap) {
  return (part_a(mcap, ncap) + (size_t)ncap * ncap) * sizeof(float2);
}

void svd_prime_f32() {
  attrs_f32<float>();
  attrs_f32<double>();
}

void svd_launch_f32(const SvdJob& j) {
  if (j.storage32)
    launch_f32<float>(j);
  else
    launch_f32<double>(j);
}

}  // namespace mpsv
