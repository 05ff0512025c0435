// Encode kernels for group size 64, 5-word codes.
#include "pvq_encode_impl.cuh"
#include "pvq_encode_lanes.cuh"

namespace pvq {
int launch_encode_n64_w5(BatchArgs& a, int dtype, cudaStream_t s) {
    return launch_encode_any<64, 5>(a, dtype, s);
}
}  // namespace pvq
