// hc_kernels_n12f.cu -- kernels and launchers for N = 4096, folded twiddles (see hc_kernels.cuh).
#include "hc_kernels.cuh"

namespace hc {
template hc_status launch_n<12, true>(const hc_ctx *, int, int, const LaunchArgs &, cudaStream_t);
}  // namespace hc
