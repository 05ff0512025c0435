// Encode kernels for group size 32, 3-word codes.
#include "pvq_encode_impl.cuh"
#include "pvq_encode_lanes.cuh"

namespace pvq {
int launch_encode_n32_w3(BatchArgs& a, int dtype, cudaStream_t s) {
    return launch_encode_any<32, 3>(a, dtype, s);
}
}  // namespace pvq
