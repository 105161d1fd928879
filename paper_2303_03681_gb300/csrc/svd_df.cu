// The truncation SVD in double-float arithmetic (svd_jacobi.cuh).
#include "svd_launch.cuh"

namespace mpsv {

size_t svd_workspace_df(int mcap, int ncap) { return svd_workspace_t<ArDF>(mcap, ncap); }

void svd_prime_df() {
  (void)svd_attrs<ArDF, float>();
  (void)svd_attrs<ArDF, double>();
}

void svd_launch_df(const SvdJob& j) {
  if (j.storage32)
    svd_launch_t<ArDF, float>(j);
  else
    svd_launch_t<ArDF, double>(j);
}

}  // namespace mpsv
