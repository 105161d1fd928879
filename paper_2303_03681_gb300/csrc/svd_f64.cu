// The truncation SVD in FP64 arithmetic (svd_jacobi.cuh).
#include "svd_launch.cuh"

namespace mpsv {

size_t svd_workspace_f64(int mcap, int ncap) { return svd_workspace_t<ArF64>(mcap, ncap); }

void svd_prime_f64() {
  (void)svd_attrs<ArF64, float>();
  (void)svd_attrs<ArF64, double>();
}

void svd_launch_f64(const SvdJob& j) {
  if (j.storage32)
    svd_launch_t<ArF64, float>(j);
  else
    svd_launch_t<ArF64, double>(j);
}

}  // namespace mpsv
