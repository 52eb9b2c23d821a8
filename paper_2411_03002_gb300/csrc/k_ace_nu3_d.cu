// The nu = 3 kernels (ace_nu3.cuh) in FP64.
#include "ace_nu3.cuh"

namespace ap {

template int launch_ace_nu3<double>(ap_ctx*, const AceArgs<double>&, int, cudaStream_t);

}  // namespace ap
