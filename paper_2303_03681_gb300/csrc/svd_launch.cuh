// Host side of the truncation SVD: the launch plan from the bond capacities
// and the launches.  Included by one translation unit per arithmetic
// (svd_df.cu, svd_f32.cu, svd_f64.cu), which compile in parallel.
#pragma once

#include <algorithm>
#include <mutex>

#include "internal.h"
#include "svd_jacobi.cuh"

namespace mpsv {

// Launch plan for a theta of up to mcap x ncap.  One CTA while the capacity is
// within its reach, else 4 CTAs, else 8 (the largest portable cluster); the
// kernel uses as many as the actual sizes need.  Past the shared memory of 8
// CTAs a cooperative grid follows the cluster launch and takes the thetas
// that the cluster left.
template <class A> struct SvdPlan {
  int P = 1;
  size_t smem = 0;
  int grid = 0;  // CTAs of the cooperative launch (0: none)
  size_t grid_smem = 0;
};

struct DeviceLimits {
  int smem = 0, sms = 0;
};
inline DeviceLimits device_limits() {
  static std::mutex mu;
  static DeviceLimits lim[64];
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> g(mu);
  DeviceLimits& l = lim[dev & 63];
  if (!l.smem) {
    cudaDeviceGetAttribute(&l.smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&l.sms, cudaDevAttrMultiProcessorCount, dev);
  }
  return l;
}

template <class A> SvdPlan<A> svd_plan(int mcap, int ncap) {
  const DeviceLimits d = device_limits();
  const size_t lim = kSvdSmemLimit;
  SvdPlan<A> pl;
  pl.P = svd_team_size<A>(mcap, ncap, 8);
  if (pl.P == 1) {
    pl.smem = SvdSmem<A>::bytes_one(mcap, ncap);
    return pl;
  }
  pl.smem = lim;  // smaller thetas may need more per CTA, on fewer CTAs
  if (pl.P) return pl;
  pl.P = 8;
  pl.grid = std::min(std::min(128, d.sms), std::max(2, (std::min(mcap, ncap) + 3) / 4));
  pl.grid_smem = SvdSmem<A>::bytes(mcap, ncap, pl.grid, false, true);
  if (pl.grid_smem > lim) pl.grid_smem = lim;
  return pl;
}

// The kernels' shared-memory opt-in, once per device (before any capture).
template <class A, class R> cudaError_t svd_attrs() {
  static std::mutex mu;
  static uint64_t done = 0;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> g(mu);
  const uint64_t bit = 1ull << (dev & 63);
  if (done & bit) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(svd_kernel<A, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSvdSmemLimit);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(svd_grid_kernel<A, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSvdSmemLimit);
  if (e == cudaSuccess) done |= bit;
  return e;
}

template <class A> size_t svd_workspace_t(int mcap, int ncap) {
  return SvdWs<A>(mcap, ncap, svd_plan<A>(mcap, ncap).grid > 0).total + 256;
}

template <class A, class R> void svd_launch_t(const SvdJob& j) {
  const SvdPlan<A> pl = svd_plan<A>(j.mcap, j.ncap);
  (void)svd_attrs<A, R>();
  const cplx<R>* C = static_cast<const cplx<R>*>(j.C);
  cplx<R>* B = static_cast<cplx<R>*>(j.Bnext);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  cfg.blockDim = dim3(kSvdThreads<A>);
  cfg.stream = j.stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(pl.P);
  cfg.dynamicSmemBytes = pl.smem;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = pl.P;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  if (j.early) {
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
  }
  cudaLaunchKernelEx(&cfg, svd_kernel<A, R>, C, j.lam_l, j.chi, j.q, j.p, B, j.lam_next, j.rep,
                     static_cast<cplx<R>*>(j.Bq), j.ws);
  if (!pl.grid) return;
  GridSync* sync = reinterpret_cast<GridSync*>(j.ws + SvdWs<A>(j.mcap, j.ncap, true).total);
  cudaMemsetAsync(sync, 0, sizeof(GridSync), j.stream);
  cfg.gridDim = dim3(pl.grid);
  cfg.numAttrs = 1;
  cfg.dynamicSmemBytes = pl.grid_smem;
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cudaLaunchKernelEx(&cfg, svd_grid_kernel<A, R>, C, j.lam_l, j.chi, j.q, j.p, B, j.lam_next, j.rep,
                     static_cast<cplx<R>*>(j.Bq), j.ws, sync, pl.P, (unsigned)pl.grid_smem);
}

}  // namespace mpsv
