// The rule for feeding a batch's streams (test infrastructure).
#include <algorithm>

#include "internal.h"

extern "C" void gate_by_gate_streams(const int* device, int n, char* out) {
  const std::vector<char> v = mpsv::gate_by_gate_streams(std::vector<int>(device, device + n));
  std::copy(v.begin(), v.end(), out);
}
