// The nu = 3 kernels (ace_nu3.cuh) in FP32; k_ace_nu3_d.cu has them in FP64 (the straight-line
// code takes a minute to compile, and the two units compile side by side).
#include "ace_nu3.cuh"

namespace ap {

template int launch_ace_nu3<float>(ap_ctx*, const AceArgs<float>&, int, cudaStream_t);

// The compiled nu = 3 code must match the host enumeration of the basis.
bool ace_nu3_matches(const AceTables& t) {
  if (t.nu3_key.size() != (size_t)AP_NU3_N) return false;
  for (int k = 0; k < AP_NU3_N; ++k)
    if (t.nu3_key[k] != kNu3Key[k]) return false;
  return true;
}

}  // namespace ap
