// hc_keyswitch_n14.cu -- key-switch kernels for N = 16384 (see hc_keyswitch.cuh).
#include "hc_keyswitch.cuh"

namespace hc {
template hc_status launch_ks_n<14, false>(const KsArgs &, size_t, uint32_t, cudaStream_t);
template hc_status launch_ks_n<14, true>(const KsArgs &, size_t, uint32_t, cudaStream_t);
}  // namespace hc
