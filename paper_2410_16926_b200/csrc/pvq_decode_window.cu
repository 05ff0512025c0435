// Dispatch of the decoder for wide codes; its kernels are in pvq_decode_window.cuh.
#include "pvq_decode_window.cuh"

namespace pvq {

int launch_decode_window_256(BatchArgs& a, const WinTables& t, cudaStream_t stream);  // pvq_decode_window_n256.cu

namespace {

template <int N, int W>
int launch_window_w(BatchArgs& a, const WinTables& t, cudaStream_t s) {
    if constexpr (N == 64) return t.plane == 96 ? launch_window_t<N, W, 96>(a, t, s) : launch_window_t<N, W, 192>(a, t, s);
    return launch_window_t<N, W, N == 64 ? 192 : 160>(a, t, s);
}

}  // namespace

int launch_decode_window(const BatchArgs& args, int N, int W, cudaStream_t stream) {
    if (!has_window_tables(N, W, args.K)) return PVQ_ERR_UNSUPPORTED;
    const auto t = window_tables(N, args.K, stream);
    if (!t || t->args.blocks_of[W] < 1) return PVQ_ERR_UNSUPPORTED;
    BatchArgs a = args;
    unsigned tiles = 0;
    for (int i = 0; i < a.count; ++i) {
        a.m[i].tile_begin = tiles;
        tiles += static_cast<unsigned>((a.m[i].rows * a.m[i].G + 31) / 32);
        if (a.m[i].rows * a.m[i].ld_out >= (1ll << 35) - 8) return PVQ_ERR_UNSUPPORTED;  // 32 bits number its 16-byte pieces
    }
    a.total_tiles = tiles;
    switch (N * 16 + W) {
        case 64 * 16 + 5: return launch_window_w<64, 5>(a, *t, stream);
        case 64 * 16 + 6: return launch_window_w<64, 6>(a, *t, stream);
        case 64 * 16 + 7: return launch_window_w<64, 7>(a, *t, stream);
        case 64 * 16 + 8: return launch_window_w<64, 8>(a, *t, stream);
        case 128 * 16 + 9: return launch_window_w<128, 9>(a, *t, stream);
        case 128 * 16 + 10: return launch_window_w<128, 10>(a, *t, stream);
        case 128 * 16 + 11: return launch_window_w<128, 11>(a, *t, stream);
        case 128 * 16 + 12: return launch_window_w<128, 12>(a, *t, stream);
        case 256 * 16 + 24: return launch_decode_window_256(a, *t, stream);
        default: break;
    }
    return PVQ_ERR_UNSUPPORTED;
}

}  // namespace pvq
