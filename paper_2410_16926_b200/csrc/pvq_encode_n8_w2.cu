// Encode kernels for group size 8, 2-word codes.
#include "pvq_encode_impl.cuh"
#include "pvq_encode_lanes.cuh"

namespace pvq {
int launch_encode_n8_w2(BatchArgs& a, int dtype, cudaStream_t s) {
    return launch_encode_any<8, 2>(a, dtype, s);
}
}  // namespace pvq
