// The decoder for wide codes at group size 256.
#include "pvq_decode_window.cuh"

namespace pvq {

int launch_decode_window_256(BatchArgs& a, const WinTables& t, cudaStream_t stream) {
    return launch_window_t<256, 24, 160>(a, t, stream);
}

}  // namespace pvq
