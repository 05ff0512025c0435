// The fused round trip of activations (pvq_roundtrip, pvq_rotate_roundtrip): encode -> decode in one
// kernel, for every group size and code width.
//
// The Fischer index is a bijection between the points of P(N,K) and [0, N(N,K)) (Sec. 2.4,
// Algorithms 2 and 3): decoding the index of a point gives that point back, whatever the
// table.  What a round trip changes is the direction (to the nearest point) and the amplitude (to its
// quantile level, or binary16), so the kernel quantises both and scales the point; the index
// and its inverse cancel.  No count table is read.
//
// A group lies on L = N / 32 neighbouring lanes (pvq_quant.cuh), so every size loads 64 bytes of bf16 a
// lane and the work per lane is the same from group size 32 up.  A thread block takes whole
// rows, or one row in chunks when it is longer than the block (then the energies are summed in a
// pass of their own, since every group's amplitude needs its row's).
// What bounds it: issue slots and the integer pipe (about 40 instructions a value-quad; see
// profiles/), not the 4 bytes a value moves.
#include <algorithm>

#include <cuda_fp16.h>

#include "pvq_rotate.cuh"
#include "pvq_rows.cuh"

namespace pvq {

namespace {

constexpr int kRoundThreadsMax = 512;

struct RoundArgs {
    const void* x;
    void* out;
    const float* edges;
    const float* levels;
    const float* signs;
    long long rows, cols, ld, ld_out;
    int G, gp;        // groups per row, and that rounded up to a power of two
    int C;            // lanes per row
    int rpt, chunks;  // rows per block; pieces a row longer than the block is taken in
    int K, b;
    int rot_block;
    uint32_t ss_off, levels_off, signs_off, xbuf_off;  // in shared memory, behind the bin edges
    uint32_t* debug_status;
};

// One lane's values of the point, scaled and rounded to bf16.
template <int E, bool BF16, bool WIDE>
__device__ __forceinline__ void emit_lane(const LanePoint<E, WIDE>& pt, const uint32_t (&raw)[kRawWords<E, BF16>], float sc,
                                          __nv_bfloat16* dst) {
    const f32x2 sc2 = pack2(sc, sc);
    const f32x2 off = WIDE ? pack2(-8421376.0f, -8421376.0f) : pack2(-8388736.0f, -8388736.0f);  // -(2^23 + the bias)
    uint32_t o[E / 2];
#pragma unroll
    for (int j = 0; j < E / 4; ++j) {
        const uint32_t neg = pt.has_dir ? chunk_signs4<E, BF16>(raw, j) : 0u;
        float f[4];
        if constexpr (!WIDE) {
            // 128 + y_i in a byte; as the low mantissa bits of 2^23 it becomes a float by one subtraction
            const uint32_t biased = ((kH4 + pt.y[j]) & ~neg) | ((kH4 - pt.y[j]) & neg);
#pragma unroll
            for (int e = 0; e < 4; ++e) f[e] = __uint_as_float(__byte_perm(biased, 0x4B000000u, 0x7540u + 3 - e));
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h) {  // positions 4j + 2h (high half), 4j + 2h + 1
                const uint32_t y = pt.y[2 * j + h], n2 = __byte_perm(neg, 0u, h == 0 ? 0x3322 : 0x1100);
                const uint32_t biased = ((0x80008000u + y) & ~n2) | ((0x80008000u - y) & n2);
                f[2 * h] = __uint_as_float(__byte_perm(biased, 0x4B000000u, 0x7532u));
                f[2 * h + 1] = __uint_as_float(__byte_perm(biased, 0x4B000000u, 0x7510u));
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float lo, hi;
            unpack2(mul2(add2(pack2(f[2 * h], f[2 * h + 1]), off), sc2), lo, hi);
            o[2 * j + h] = pack_bf16x2(lo, hi);
        }
    }
#pragma unroll
    for (int q = 0; q < E / 8; ++q)
        reinterpret_cast<uint4*>(dst)[q] = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
}

template <int E, bool WIDE>
__device__ __forceinline__ int lane_squares(const LanePoint<E, WIDE>& pt) {
    unsigned s = 0u;
    if constexpr (!WIDE) {
#pragma unroll
        for (int j = 0; j < E / 4; ++j) s = __dp4a(pt.y[j], pt.y[j], s);
    } else {
#pragma unroll
        for (int h = 0; h < E / 2; ++h) {
            const unsigned a = pt.y[h] & 0xffffu, b = pt.y[h] >> 16;
            s += a * a + b * b;
        }
    }
    return static_cast<int>(s);
}

template <int E, int L, bool BF16, bool WIDE, bool ROT>
__global__ void __launch_bounds__(kRoundThreadsMax) roundtrip_kernel(const __grid_constant__ RoundArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    constexpr bool WBF16 = BF16 && !ROT;  // the form the kernel works on: packed bf16, or fp32
    float* s_edges = reinterpret_cast<float*>(smem);
    float* s_levels = reinterpret_cast<float*>(smem + a.levels_off);
    float* s_ss = reinterpret_cast<float*>(smem + a.ss_off);
    uint32_t* s_signs = reinterpret_cast<uint32_t*>(smem + a.signs_off);
    float* s_xbuf = reinterpret_cast<float*>(smem + a.xbuf_off);
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
    const int b = a.b;
    const int nedges = b <= 8 ? (1 << b) - 1 : 0;  // 16 bits: the amplitude itself, no codebook
    float rot_scale = 1.0f;
#ifdef PVQ_DEBUG
    debug_begin(0u, 0u, 0u, 0u, 0u, a.debug_status);
#endif
    if constexpr (ROT) {
        pack_signs<E>(s_signs, a.signs, a.rot_block);
        rot_scale = static_cast<float>(1.0 / sqrt(static_cast<double>(a.rot_block)));
    }
    for (int i = tid; i < nedges; i += T) s_edges[i] = a.edges[i];
    for (int i = tid; i <= nedges && nedges > 0; i += T) s_levels[i] = a.levels[i];
    if (ROT) __syncthreads();

    const int rl = a.chunks == 1 ? tid / a.C : 0;
    const int c0 = a.chunks == 1 ? tid - rl * a.C : tid;
    const long long row = static_cast<long long>(blockIdx.x) * a.rpt + rl;
    const bool row_ok = rl < a.rpt && row < a.rows;
    // a row inside a warp: its energy is a sum over lanes, no shared memory
    const bool in_warp = a.C <= 32 && (a.C & (a.C - 1)) == 0;

    auto load = [&](int c, bool active, uint32_t (&w)[kRawWords<E, WBF16>]) {
        const size_t at = static_cast<size_t>(row) * a.ld + static_cast<size_t>(c) * E;
        if constexpr (!ROT) {
#pragma unroll
            for (int i = 0; i < kRawWords<E, WBF16>; ++i) w[i] = 0u;
            if (active) load_chunk<E, BF16>(a.x, at, w);
        } else {
            uint32_t r[kRawWords<E, BF16>];
            float x[E];
#pragma unroll
            for (int i = 0; i < kRawWords<E, BF16>; ++i) r[i] = 0u;
            if (active) load_chunk<E, BF16>(a.x, at, r);
#pragma unroll
            for (int i = 0; i < E; ++i)
                x[i] = BF16 ? __uint_as_float((i & 1) ? (r[i / 2] & 0xffff0000u) : (r[i / 2] << 16)) : __uint_as_float(r[BF16 ? i / 2 : i]);
            rotate_lanes<E>(x, s_signs, a.rot_block, rot_scale, c, s_xbuf);
#pragma unroll
            for (int i = 0; i < E; ++i) w[i] = __float_as_uint(x[i]);
        }
    };

    if (a.chunks > 1) {
        for (int ch = 0; ch < a.chunks; ++ch) {
            const int c = c0 + ch * T;
            const bool active = row_ok && c < a.C;
            uint32_t raw[kRawWords<E, WBF16>];
            float ax[E], l1, ss;
            load(c, active, raw);
            group_norms<E, L, WBF16>(raw, ax, l1, ss);
            if (active && (c & (L - 1)) == 0) s_ss[c / L] = ss;
        }
        for (int g = a.G + tid; g < a.gp; g += T) s_ss[g] = 0.0f;
        __syncthreads();
    }
    float ss_row = 0.0f;
    for (int ch = 0; ch < a.chunks; ++ch) {
        const int c = c0 + ch * T;
        const bool active = row_ok && c < a.C;
        uint32_t raw[kRawWords<E, WBF16>];
        float ss;
        LanePoint<E, WIDE> pt;
        load(c, active, raw);
        {
            float ax[E], l1;
            group_norms<E, L, WBF16>(raw, ax, l1, ss);
            if constexpr (ROT)
                quantize_group<E, L, WIDE>(ax, l1, a.K, FetchRotated{s_xbuf + tid, T}, pt);
            else
                quantize_group<E, L, WIDE>(ax, l1, a.K,
                                           FetchGlobal<BF16>{static_cast<const uint8_t*>(a.x) +
                                                             (static_cast<size_t>(row) * a.ld + static_cast<size_t>(c) * E) * (BF16 ? 2 : 4)},
                                           pt);
        }
        if (in_warp) {
            ss_row = ss;
            for (int o = L; o < a.C; o <<= 1) ss_row = __fadd_rn(ss_row, __shfl_xor_sync(0xffffffffu, ss_row, o));
            if (ch == 0) __syncthreads();  // edges and levels
        } else if (ch == 0) {
            if (a.chunks == 1) {
                if (active && (c & (L - 1)) == 0 && PVQ_DEBUG_INDEX(rl * a.gp + c / L, a.rpt * a.gp, PVQ_DEBUG_SHARED_INDEX))
                    s_ss[rl * a.gp + c / L] = ss;
                if (a.gp != a.G)  // zero padding of the rows' trees
                    for (int j = tid; j < a.rpt * a.gp; j += T)
                        if ((j & (a.gp - 1)) >= a.G) s_ss[j] = 0.0f;
                __syncthreads();
            }
            ss_row = row_energy(s_ss, a.gp, rl, a.rpt, lane);
        }
        float amp;
        if (b == 16) {  // the amplitude as binary16
            amp = __half2float(__float2half_rn(__fsqrt_rn(ss)));
        } else {
            // Step 5: q = floor(CDF(u) 2^b) as the number of bin edges <= u, then the bin's level
            const float u = ss_row > 0.0f ? __fdiv_rn(ss, ss_row) : 0.0f;
            int q = 0;
            for (int step = 1 << (b - 1); step >= 1; step >>= 1)
                if (s_edges[q + step - 1] <= u) q += step;
            amp = __fmul_rn(__fsqrt_rn(ss_row), s_levels[q]);
        }
        const int ssy = group_add<L>(lane_squares<E, WIDE>(pt));
        const float sc = __fdiv_rn(amp, __fsqrt_rn(static_cast<float>(ssy)));
        if (active && PVQ_DEBUG_INDEX(row, a.rows, PVQ_DEBUG_GLOBAL_STORE) &&
            PVQ_DEBUG_INDEX(static_cast<long long>(c + 1) * E - 1, a.cols, PVQ_DEBUG_GLOBAL_STORE))
            emit_lane<E, WBF16, WIDE>(pt, raw, sc,
                                      static_cast<__nv_bfloat16*>(a.out) + static_cast<size_t>(row) * a.ld_out + static_cast<size_t>(c) * E);
    }
}

template <int E, int L, bool BF16, bool WIDE, bool ROT>
int launch_round_t(RoundArgs& a, cudaStream_t stream) {
    DeviceInfo di;
    int st = device_info(&di);
    if (st != PVQ_OK) return st;
    a.C = a.G * L;
    a.gp = 1;
    while (a.gp < a.G) a.gp <<= 1;
    int threads = 0;
    if (a.C > kRoundThreadsMax) {
        // 512 lanes hold whole rotation blocks (at most 16384 values at 32 a lane; for the smaller
        // groups a block of more than 512 lanes is refused)
        if (ROT && a.rot_block / E > kRoundThreadsMax) return PVQ_ERR_UNSUPPORTED;
        threads = kRoundThreadsMax;
        a.rpt = 1;
        a.chunks = (a.C + threads - 1) / threads;
    } else {
        // Whole rows: the block of up to 256 threads (more when a row needs it) that leaves the
        // fewest lanes idle; among equals the largest, or the smallest when the launch would
        // not fill the SMs anyway.
        a.chunks = 1;
        long long best = -1;
        for (int t = std::max(64, (a.C + 31) / 32 * 32); t <= std::max(256, (a.C + 31) / 32 * 32); t += 32) {
            const int rpt = t / a.C;
            const long long tiles = (a.rows + rpt - 1) / rpt, cost = tiles * t;
            const bool few = tiles < 2 * di.sms;
            if (best < 0 || cost < best || (cost == best && !few)) {
                best = cost;
                threads = t;
            }
        }
        a.rpt = threads / a.C;
    }
    const long long tiles = (a.rows + a.rpt - 1) / a.rpt;
    if (tiles > 0x7fffffffLL) return PVQ_ERR_UNSUPPORTED;
    a.levels_off = a.b <= 8 ? 4u << a.b : 0u;
    a.ss_off = 2u * a.levels_off;
    a.ss_off = (a.ss_off + 15u) & ~15u;
    a.signs_off = (a.ss_off + static_cast<uint32_t>(a.rpt * a.gp) * 4u + 15u) & ~15u;
    a.xbuf_off = a.signs_off + (ROT ? (static_cast<uint32_t>(a.rot_block / E) * 4u + 15u) & ~15u : 0u);
    const size_t smem = a.xbuf_off + (ROT ? static_cast<size_t>(threads) * E * 4u : 0u);
    if (smem > static_cast<size_t>(di.smem_max)) return PVQ_ERR_UNSUPPORTED;
    auto kern = roundtrip_kernel<E, L, BF16, WIDE, ROT>;
    int per_sm = 0;
    if ((st = prepare_kernel(reinterpret_cast<const void*>(kern), threads, smem, &per_sm)) != PVQ_OK) return st;
    if (per_sm < 1) return PVQ_ERR_UNSUPPORTED;
    kern<<<static_cast<unsigned>(tiles), threads, smem, stream>>>(a);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PVQ_OK : set_cuda_error(e);
}

template <int E, int L>
int launch_round_n(RoundArgs& a, bool bf16, cudaStream_t s) {
    const bool wide = a.K > 127, rot = a.rot_block != 0;
    if (bf16) {
        if (rot) return wide ? launch_round_t<E, L, true, true, true>(a, s) : launch_round_t<E, L, true, false, true>(a, s);
        return wide ? launch_round_t<E, L, true, true, false>(a, s) : launch_round_t<E, L, true, false, false>(a, s);
    }
    if (rot) return wide ? launch_round_t<E, L, false, true, true>(a, s) : launch_round_t<E, L, false, false, true>(a, s);
    return wide ? launch_round_t<E, L, false, true, false>(a, s) : launch_round_t<E, L, false, false, false>(a, s);
}

}  // namespace

int launch_roundtrip(const MatrixArgs& m, int dtype, int N, int K, int scale_bits, int rot_block, const float* signs,
                     uint32_t* debug_status, cudaStream_t stream) {
    RoundArgs a;
    a.x = m.x;
    a.out = m.out;
    a.edges = m.edges;
    a.levels = m.levels;
    a.signs = signs;
    a.rows = m.rows;
    a.cols = m.cols;
    a.ld = m.ld;
    a.ld_out = m.ld_out;
    a.G = m.G;
    a.K = K;
    a.b = scale_bits;
    a.rot_block = rot_block;
    a.debug_status = debug_status;
    const bool bf16 = dtype == PVQ_DTYPE_BF16;
    switch (N) {
        case 8: return launch_round_n<8, 1>(a, bf16, stream);
        case 16: return launch_round_n<16, 1>(a, bf16, stream);
        case 32: return launch_round_n<32, 1>(a, bf16, stream);
        case 64: return launch_round_n<32, 2>(a, bf16, stream);
        case 128: return launch_round_n<32, 4>(a, bf16, stream);
        case 256: return launch_round_n<32, 8>(a, bf16, stream);
        default: return PVQ_ERR_UNSUPPORTED;
    }
}

}  // namespace pvq
