// Sets and reads what a timed-out wait leaves behind (test infrastructure).
#include "internal.h"

using namespace mpsv;

// Marks a state as its kernels do when a bounded wait runs out.
extern "C" int set_timeout_flag(mps_state* st) {
  const int one = 1;
  return cudaMemcpy(&st->d_rep->tc_error, &one, sizeof(one), cudaMemcpyHostToDevice);
}

extern "C" int status_of(int tc_error, int not_converged) {
  DevReport r = {};
  r.tc_error = tc_error;
  return svd_status(r, "test", not_converged);
}
