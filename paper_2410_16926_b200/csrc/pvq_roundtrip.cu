// The fused round trip of activations (pvq_roundtrip, pvq_rotate_roundtrip): encode -> decode in one
// kernel, for every group size and code width.
//
// The Fischer index is a bijection between the points of P(N,K) and [0, N(N,K)) (Sec. 2.4,
// Algorithms 2 and 3): decoding the index of a point gives that point back, whatever the
// table.  What a round trip changes is the direction (to the nearest point) and the amplitude (to its
// quantile level, or binary16), so the kernel quantises both and scales the point; the index
// and its inverse cancel.  No count table is read.
//
// A group lies on L = N / 32 neighbouring lanes (pvq_quant.cuh): the work and the bytes per lane are the
// same from group size 32 up.  What bounds it: issue slots and the half-rate integer pipe (about
// 840 warp instructions per 1024 values), not the 4 bytes a value moves.
#include <algorithm>

#include <cuda_fp16.h>

#include "pvq_rotate.cuh"
#include "pvq_rows.cuh"
#include "pvq_stage.cuh"

namespace pvq {

namespace {

constexpr int kRoundThreadsMax = 512;
constexpr int kCodebookMax = 256;  // levels of an amplitude codebook

struct RoundArgs {
    const void* x;
    void* out;
    const float* edges;
    const float* levels;
    const float* signs;
    long long rows, cols, ld, ld_out;
    int G, gp;        // groups per row, and that rounded up to a power of two
    int C;            // lanes per row
    int rpt, chunks;  // rows per tile; pieces a row longer than the block is taken in
    unsigned tiles;
    int K, b;
    int rot_block;
    float minus_zero;  // -0 (see mul2_rounded)
    uint32_t levels_off, ss_off, signs_off, xbuf_off;  // in shared memory, behind the bin edges
    uint32_t ring_off, tile_bytes;                     // buffers for input and output tiles
    int bufs;                                          // how many (see roundtrip_kernel)
    uint32_t* status;
    uint32_t* debug_status;
};

// Four values of the point (word j of its packing, or two words when WIDE), scaled and rounded to
// bf16.  neg: 0xff in the bytes of negative values.
template <int E, bool WIDE>
__device__ __forceinline__ uint2 scaled_values(const LanePoint<E, WIDE>& pt, int j, uint32_t neg, f32x2 sc2) {
    const f32x2 off = WIDE ? pack2(-8421376.0f, -8421376.0f) : pack2(-8388736.0f, -8388736.0f);  // -(2^23 + the bias)
    float f[4];
    if constexpr (!WIDE) {
        // 128 + y_i in a byte; as the low mantissa bits of 2^23 it becomes a float by one subtraction
        // (128 + y, or 128 + 255 - y - 255: no byte of the sum leaves 1 .. 255)
        const uint32_t biased = (pt.y[j] ^ neg) + kH4 - neg;
#pragma unroll
        for (int e = 0; e < 4; ++e) f[e] = __uint_as_float(__byte_perm(biased, 0x4B000000u, 0x7540u + 3 - e));
    } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // positions 4j + 2h (high half), 4j + 2h + 1
            const uint32_t y = pt.y[2 * j + h], n2 = __byte_perm(neg, 0u, h == 0 ? 0x3322 : 0x1100);
            const uint32_t biased = (y ^ n2) + 0x80008000u - n2;
            f[2 * h] = __uint_as_float(__byte_perm(biased, 0x4B000000u, 0x7532u));
            f[2 * h + 1] = __uint_as_float(__byte_perm(biased, 0x4B000000u, 0x7510u));
        }
    }
    float a, b, c, d;
    unpack2(mul2(add2(pack2(f[0], f[1]), off), sc2), a, b);
    unpack2(mul2(add2(pack2(f[2], f[3]), off), sc2), c, d);
    return make_uint2(pack_bf16x2(a, b), pack_bf16x2(c, d));
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

// The amplitude codebook, edges padded to the 15 or 255 that amplitude() looks at; a barrier follows.
__device__ __forceinline__ void stage_codebook(const RoundArgs& a, float* s_edges, float* s_levels, int tid, int T) {
    if (a.b == 16) return;  // the amplitude itself
    const int levels = 1 << a.b, entries = a.b > 4 ? kCodebookMax : 16;
#pragma unroll 1  // (four at a time: small calls 0.1 to 0.4 us slower)
    for (int i = tid; i < entries; i += T) {
        s_edges[i] = i + 1 < levels ? a.edges[i] : __int_as_float(0x7fffffff);
        if (i < levels) s_levels[i] = a.levels[i];
    }
}

// The group's dequantised amplitude.
__device__ __forceinline__ float amplitude(float ss, float ss_row, int b, const float* s_edges, const float* s_levels) {
    if (b == 16) return __half2float(__float2half_rn(__fsqrt_rn(ss)));  // the amplitude as binary16
    // Step 5: q = floor(CDF(u) 2^b) as the number of bin edges <= u, then the bin's level.  The edges are padded to 255 by NaN, which
    // nothing reaches: four or eight steps without a counter.  (16384 x 4096: 75.2 us with one, 74.3 by a jump to the
    // first step, 72.7 so.)
    const float u = ss_row > 0.0f ? __fdiv_rn(ss, ss_row) : 0.0f;
    int q = 0;
    if (b > 4) {
#pragma unroll
        for (int step = 128; step >= 16; step >>= 1)
            if (s_edges[q + step - 1] <= u) q += step;
    }
#pragma unroll
    for (int step = 8; step >= 1; step >>= 1)
        if (s_edges[q + step - 1] <= u) q += step;
    return __fmul_rn(__fsqrt_rn(ss_row), s_levels[q]);
}

// For bf16 input in rows of up to 512 lanes.  A block stays and takes tile after tile of whole rows.
// Input tiles arrive in shared memory by bulk copy, a tile ahead; the results are written over
// the input in place and leave by bulk copy: no thread waits for global memory, and the copies
// are whole lines whatever the lanes' access pattern (64 bytes a lane, 16 at a time).  Three
// buffers: one worked on, one arriving, one leaving.  One block-wide barrier per tile.
// Rotated, 32 values a lane (DIRECT): every warp writes its results to memory itself, brought into whole lines in its part
// of the rotation's buffer, so a tile's buffer is free once it is read: two buffers, or one where the rotation's
// barriers say so early (blocks that span warps).  4096 columns: 28 KB a row, seven rows an SM.
template <int E, int L, bool WIDE, bool ROT>
__global__ void __launch_bounds__(kRoundThreadsMax, 2) roundtrip_kernel(const __grid_constant__ RoundArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t full[3];
    constexpr int P = E / 8;  // 16-byte pieces a lane
    constexpr bool DIRECT = ROT && E == 32;
    float* s_edges = reinterpret_cast<float*>(smem);
    float* s_levels = reinterpret_cast<float*>(smem + a.levels_off);
    uint32_t* s_signs = reinterpret_cast<uint32_t*>(smem + a.signs_off);
    float* s_xbuf = reinterpret_cast<float*>(smem + a.xbuf_off);
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
    const int b = a.b;
    const uint32_t row_bytes = static_cast<uint32_t>(a.cols) * 2u;
    auto tile_rows = [&](unsigned tile) {
        return static_cast<int>(min(static_cast<long long>(a.rpt), a.rows - static_cast<long long>(tile) * a.rpt));
    };
    const bool withheld = debug_withhold(a.debug_status);
    auto request = [&](unsigned tile, int buf) {  // thread 0
        if (withheld) return;
        const int nr = tile_rows(tile);
        const BulkStage st{shared_addr(full + buf)};
        bulk_stage_expect(st, nr * row_bytes);
        uint8_t* dst = smem + a.ring_off + buf * a.tile_bytes;
        const uint8_t* src = static_cast<const uint8_t*>(a.x) + static_cast<size_t>(tile) * a.rpt * a.ld * 2;
        if (a.ld == a.cols)
            bulk_stage_copy(st, dst, src, nr * row_bytes);
        else
            for (int r = 0; r < nr; ++r) bulk_stage_copy(st, dst + r * row_bytes, src + static_cast<size_t>(r) * a.ld * 2, row_bytes);
    };
    auto deliver = [&](unsigned tile, int buf) {  // thread 0
        const int nr = tile_rows(tile);
        const uint8_t* src = smem + a.ring_off + buf * a.tile_bytes;
        uint8_t* dst = static_cast<uint8_t*>(a.out) + static_cast<size_t>(tile) * a.rpt * a.ld_out * 2;
        if (a.ld_out == a.cols)
            bulk_store(dst, src, nr * row_bytes);
        else
            for (int r = 0; r < nr; ++r) bulk_store(dst + static_cast<size_t>(r) * a.ld_out * 2, src + r * row_bytes, row_bytes);
        bulk_store_commit();
    };

    unsigned tile = blockIdx.x;
    if (tid == 0) {
        for (int i = 0; i < 3; ++i) mbarrier_init_one(full + i);
        mbarrier_init_fence();
    }
    grid_launch_dependents();
    grid_dependency_wait();
    if (tid == 0) request(tile, 0);
    float rot_scale = 1.0f;
    if constexpr (ROT) {
        pack_signs<E>(s_signs, a.signs, a.rot_block);
        rot_scale = static_cast<float>(1.0 / sqrt(static_cast<double>(a.rot_block)));
    }
    stage_codebook(a, s_edges, s_levels, tid, T);
#ifdef PVQ_DEBUG
    debug_begin(0u, 0u, 0u, 0u, 0u, a.debug_status);
#endif
    __syncthreads();  // barriers, codebook, signs

    const int rl = tid / a.C, c = tid - rl * a.C;
    const int rot8 = ROT ? 0 : lane_rotation<E>(lane);
    // a row inside a warp: its energy is a sum over lanes, no shared memory; whole warps: a warp's part of it is, and the parts
    // go through shared memory, `parts` a row (zero padded to a power of two).  The sum over lanes is then made while the group is
    // quantised, not after the barrier: 16384 x 4096 72.8 -> 72.0 us, at N = 128 94.5 -> 92.8.  (Rotated: 23.0 -> 23.2, so not there.)
    const bool in_warp = a.C <= 32 && (a.C & (a.C - 1)) == 0, whole = !ROT && !in_warp && (a.C & 31) == 0;
    const int parts = whole ? a.gp * L / 32 : a.gp, used = whole ? a.C / 32 : a.G;
    if (parts != used)  // the zero padding of the rows' trees, for both tiles at work
        for (int j = tid; j < a.rpt * parts; j += T)
            if ((j & (parts - 1)) >= used) {
                float* p = reinterpret_cast<float*>(smem + a.ss_off) + j;
                p[0] = p[a.rpt * a.gp] = 0.0f;
            }
    const uint32_t lane_off = a.ring_off + static_cast<uint32_t>(tid) * (E * 2);  // rows of a tile follow one another
    int buf = 0, parity = 0;
    for (int i = 0;; ++i) {
        uint8_t* mine = smem + lane_off + buf * a.tile_bytes;
        const bool active = rl < a.rpt && static_cast<long long>(tile) * a.rpt + rl < a.rows;
        float* s_ss = reinterpret_cast<float*>(smem + a.ss_off) + (i & 1) * a.rpt * a.gp;
        // (a thread that gives up works on whatever the buffer holds, as far as the next barrier)
        const bool failed = !mbarrier_wait(shared_addr(full + buf), parity, stream_polls(withheld));
        const unsigned next = tile + gridDim.x;
        const bool have_next = next < a.tiles;
        const int nbuf = buf + 1 == a.bufs ? 0 : buf + 1;
        float ss;
        uint32_t neg[E / 4];
        LanePoint<E, WIDE> pt;
        {
            float ax[E], l1;
            uint32_t raw[E / 2];
#pragma unroll
            for (int v = 0; v < P; ++v) {
                uint4 q = make_uint4(0u, 0u, 0u, 0u);
                if (active) q = reinterpret_cast<const uint4*>(mine)[(v + rot8) & (P - 1)];
                raw[4 * v] = q.x, raw[4 * v + 1] = q.y, raw[4 * v + 2] = q.z, raw[4 * v + 3] = q.w;
            }
            if constexpr (ROT) {
                float x[E];
                uint32_t w[E];
                if constexpr (E == 32) {
                    const int T0 = a.rot_block / E;
                    const uint32_t sb = s_signs[c & (T0 - 1)];
#pragma unroll
                    for (int k = 0; k < E / 2; ++k) raw[k] ^= (sb << k) & 0x80008000u;
#pragma unroll
                    for (int k = 0; k < E; ++k) x[k] = __uint_as_float((k & 1) ? (raw[k / 2] & 0xffff0000u) : (raw[k / 2] << 16));
                    bool asked = a.bufs != 1;
                    rotate_lanes32(x, T0, rot_scale, smem, a.xbuf_off, a.minus_zero, [&]() {
                        __syncthreads();
                        if (!asked && tid == 0 && have_next && !failed) request(next, nbuf);  // the tile has been read
                        asked = true;
                    });
                } else {
#pragma unroll
                    for (int k = 0; k < E; ++k) x[k] = __uint_as_float((k & 1) ? (raw[k / 2] & 0xffff0000u) : (raw[k / 2] << 16));
                    rotate_lanes<E>(x, s_signs, a.rot_block, rot_scale, c, s_xbuf, a.minus_zero);
                }
#pragma unroll
                for (int k = 0; k < E; ++k) w[k] = __float_as_uint(x[k]);
#pragma unroll
                for (int j = 0; j < E / 4; ++j) neg[j] = chunk_signs4<E, false>(w, j);
                group_norms<E, L, false>(w, ax, l1, ss, a.minus_zero);
                quantize_group<E, L, WIDE>(ax, l1, a.K, FetchRotated<E>{smem, a.xbuf_off, rot_scale}, pt, a.minus_zero);
            } else {
#pragma unroll
                for (int j = 0; j < E / 4; ++j) neg[j] = chunk_signs4<E, true>(raw, j);
                group_norms<E, L, true>(raw, ax, l1, ss, a.minus_zero, rot8);
                quantize_group<E, L, WIDE>(ax, l1, a.K, FetchShared{reinterpret_cast<const unsigned short*>(mine)}, pt, a.minus_zero, rot8);
            }
        }
        float part = ss;
        if (whole) {
#pragma unroll
            for (int o = L; o < 32; o <<= 1) part = __fadd_rn(part, __shfl_xor_sync(0xffffffffu, part, o));
            if (active && lane == 0 && PVQ_DEBUG_INDEX(rl * parts + c / 32, a.rpt * a.gp, PVQ_DEBUG_SHARED_INDEX)) s_ss[rl * parts + c / 32] = part;
        } else if (!in_warp) {
            if (active && (c & (L - 1)) == 0 && PVQ_DEBUG_INDEX(rl * a.gp + c / L, a.rpt * a.gp, PVQ_DEBUG_SHARED_INDEX))
                s_ss[rl * a.gp + c / L] = ss;
        }
        // energies are in place, and the tile before this one is complete in its buffer
        if (!DIRECT) bulk_store_fence();
        if (__syncthreads_or(failed)) {  // the copy never arrived: report and leave rather than spin, all threads
            if (a.status && failed) atomicOr(a.status, PVQ_STATUS_STAGING_TIMEOUT);
            if (tid == 0) {
                if (!DIRECT && i > 0) deliver(tile - gridDim.x, buf == 0 ? a.bufs - 1 : buf - 1);
                bulk_store_wait_read<0>();
                // (asked for already: it has to land before the block's memory goes away)
                if (DIRECT && a.bufs == 1 && have_next && !failed) mbarrier_wait(shared_addr(full), parity ^ 1, stream_polls(withheld));
            }
            return;
        }
        if (tid == 0) {
            if (!DIRECT && i > 0) deliver(tile - gridDim.x, buf == 0 ? a.bufs - 1 : buf - 1);
            if (have_next && a.bufs != 1) {
                if (!DIRECT) bulk_store_wait_read<1>();  // what was in the buffer has left it
                request(next, nbuf);
            }
        }
        float ss_row;
        if (in_warp) {
            ss_row = ss;
            for (int o = L; o < a.C; o <<= 1) ss_row = __fadd_rn(ss_row, __shfl_xor_sync(0xffffffffu, ss_row, o));
        } else if (whole && parts == 4) {
            const float4 q = *reinterpret_cast<const float4*>(s_ss + rl * 4);
            ss_row = __fadd_rn(__fadd_rn(q.x, q.y), __fadd_rn(q.z, q.w));
        } else if (whole) {
            ss_row = warp_tree_sum(s_ss + rl * parts, parts, lane);
        } else {
            ss_row = row_energy(s_ss, a.gp, rl, a.rpt, lane);
        }
        const float amp = amplitude(ss, ss_row, b, s_edges, s_levels);
        const int ssy = group_add<L>(lane_squares<E, WIDE>(pt));
        const float sc = __fdiv_rn(amp, __fsqrt_rn(static_cast<float>(ssy)));
        const f32x2 sc2 = pack2(sc, sc);
        if (!pt.has_dir) {  // (K, 0, ..., 0), positive
#pragma unroll
            for (int j = 0; j < E / 4; ++j) neg[j] = 0u;
        }
        auto piece_of = [&](int v) {
            const uint2 lo = scaled_values<E, WIDE>(pt, 2 * v, neg[2 * v], sc2);
            const uint2 hi = scaled_values<E, WIDE>(pt, 2 * v + 1, neg[2 * v + 1], sc2);
            return make_uint4(lo.x, lo.y, hi.x, hi.y);
        };
        if constexpr (DIRECT) {
            // piece p of lane l lies at 4 l + (p ^ (l / 2) % 4): the lanes of an access hit different banks
            uint4* lines = reinterpret_cast<uint4*>(s_xbuf + (tid - lane) * E);
            __syncwarp();  // nobody looks for residuals there any more
#pragma unroll
            for (int v = 0; v < P; ++v) lines[lane * P + (v ^ ((lane >> 1) & 3))] = piece_of(v);
            const long long row = static_cast<long long>(tile) * a.rpt + rl;
            const bool ok = active && PVQ_DEBUG_INDEX(row, a.rows, PVQ_DEBUG_GLOBAL_STORE) &&
                            PVQ_DEBUG_INDEX(static_cast<long long>(c + 1) * E - 1, a.cols, PVQ_DEBUG_GLOBAL_STORE);
            const unsigned long long at =
                ok ? reinterpret_cast<unsigned long long>(static_cast<__nv_bfloat16*>(a.out) + static_cast<size_t>(row) * a.ld_out + static_cast<size_t>(c) * E) : 0ull;
            __syncwarp();
#pragma unroll
            for (int v = 0; v < P; ++v) {
                const int l = v * (32 / P) + lane / P, p = lane % P;
                const unsigned long long dst = __shfl_sync(0xffffffffu, at, l);
                const uint4 q = lines[l * P + (p ^ ((l >> 1) & 3))];
                if (dst != 0ull) reinterpret_cast<uint4*>(dst)[p] = q;
            }
            __syncwarp();  // free for the next tile
        } else if (active) {
#pragma unroll
            for (int v = 0; v < P; ++v) {
                const int piece = (v + rot8) & (P - 1);
                if (PVQ_DEBUG_INDEX(tid * P + piece, a.tile_bytes / 16, PVQ_DEBUG_SHARED_INDEX)) reinterpret_cast<uint4*>(mine)[piece] = piece_of(v);
            }
        }
        if (!have_next) break;
        tile = next;
        buf = nbuf;
        if (buf == 0) parity ^= 1;
    }
    if (DIRECT) return;
    bulk_store_fence();
    __syncthreads();
    if (tid == 0) {
        deliver(tile, buf);
        bulk_store_wait_read<0>();
    }
}

// For fp32 input and for rows longer than a thread block: one tile of whole rows per block, or one row in
// chunks (then the energies are summed in a pass of their own, since every group's amplitude needs
// its row's), loads and stores straight from and to global memory.
template <int E, int L, bool BF16, bool WIDE, bool ROT>
__global__ void __launch_bounds__(kRoundThreadsMax) roundtrip_rows_kernel(const __grid_constant__ RoundArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr bool WBF16 = BF16 && !ROT;  // the form the kernel works on: packed bf16, or fp32
    float* s_edges = reinterpret_cast<float*>(smem);
    float* s_levels = reinterpret_cast<float*>(smem + a.levels_off);
    float* s_ss = reinterpret_cast<float*>(smem + a.ss_off);
    uint32_t* s_signs = reinterpret_cast<uint32_t*>(smem + a.signs_off);
    float* s_xbuf = reinterpret_cast<float*>(smem + a.xbuf_off);
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
    const int b = a.b;
    grid_launch_dependents();
    grid_dependency_wait();
    float rot_scale = 1.0f;
#ifdef PVQ_DEBUG
    debug_begin(0u, 0u, 0u, 0u, 0u, a.debug_status);
#endif
    if constexpr (ROT) {
        pack_signs<E>(s_signs, a.signs, a.rot_block);
        rot_scale = static_cast<float>(1.0 / sqrt(static_cast<double>(a.rot_block)));
    }
    stage_codebook(a, s_edges, s_levels, tid, T);
    if (ROT) __syncthreads();

    const int rl = a.chunks == 1 ? tid / a.C : 0;
    const int c0 = a.chunks == 1 ? tid - rl * a.C : tid;
    const long long row = static_cast<long long>(blockIdx.x) * a.rpt + rl;
    const bool row_ok = rl < a.rpt && row < a.rows;
    // a row inside a warp: its energy is a sum over lanes, no shared memory
    const bool in_warp = a.C <= 32 && (a.C & (a.C - 1)) == 0;

    auto at = [&](int c) { return static_cast<size_t>(row) * a.ld + static_cast<size_t>(c) * E; };  // of a lane's first value
    auto load = [&](int c, bool active, uint32_t (&w)[kRawWords<E, WBF16>]) {
        if constexpr (!ROT) {
#pragma unroll
            for (int i = 0; i < kRawWords<E, WBF16>; ++i) w[i] = 0u;
            if (active) load_chunk<E, BF16>(a.x, at(c), w);
        } else {
            uint32_t r[kRawWords<E, BF16>];
            float x[E];
#pragma unroll
            for (int i = 0; i < kRawWords<E, BF16>; ++i) r[i] = 0u;
            if (active) load_chunk<E, BF16>(a.x, at(c), r);
#pragma unroll
            for (int i = 0; i < E; ++i)
                x[i] = BF16 ? __uint_as_float((i & 1) ? (r[i / 2] & 0xffff0000u) : (r[i / 2] << 16)) : __uint_as_float(r[BF16 ? i / 2 : i]);
            if constexpr (E == 32) {
                const int T0 = a.rot_block / E;
                const uint32_t sb = s_signs[c & (T0 - 1)];
#pragma unroll
                for (int i = 0; i < E; ++i) x[i] = __uint_as_float(__float_as_uint(x[i]) ^ ((sb << (i / 2 + (i & 1 ? 0 : 16))) & 0x80000000u));
                rotate_lanes32(x, T0, rot_scale, smem, a.xbuf_off, a.minus_zero, []() { __syncthreads(); });
            } else {
                rotate_lanes<E>(x, s_signs, a.rot_block, rot_scale, c, s_xbuf, a.minus_zero);
            }
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
            group_norms<E, L, WBF16>(raw, ax, l1, ss, a.minus_zero);
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
            group_norms<E, L, WBF16>(raw, ax, l1, ss, a.minus_zero);
            if constexpr (ROT)
                quantize_group<E, L, WIDE>(ax, l1, a.K, FetchRotated<E>{smem, a.xbuf_off, rot_scale}, pt, a.minus_zero);
            else
                quantize_group<E, L, WIDE>(ax, l1, a.K, FetchGlobal<BF16>{static_cast<const uint8_t*>(a.x) + (active ? at(c) : 0) * (BF16 ? 2 : 4)}, pt,
                                           a.minus_zero);
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
        const float amp = amplitude(ss, ss_row, b, s_edges, s_levels);
        const int ssy = group_add<L>(lane_squares<E, WIDE>(pt));
        const float sc = __fdiv_rn(amp, __fsqrt_rn(static_cast<float>(ssy)));
        const f32x2 sc2 = pack2(sc, sc);
        if (active && PVQ_DEBUG_INDEX(row, a.rows, PVQ_DEBUG_GLOBAL_STORE) &&
            PVQ_DEBUG_INDEX(static_cast<long long>(c + 1) * E - 1, a.cols, PVQ_DEBUG_GLOBAL_STORE)) {
            uint4* dst = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(a.out) + static_cast<size_t>(row) * a.ld_out +
                                                  static_cast<size_t>(c) * E);
#pragma unroll
            for (int q = 0; q < E / 8; ++q) {
                // a group without direction: (K, 0, ..., 0), positive (the sign of a zero does not matter)
                const uint2 lo = scaled_values<E, WIDE>(pt, 2 * q, q > 0 || pt.has_dir ? chunk_signs4<E, WBF16>(raw, 2 * q) : 0u, sc2);
                const uint2 hi = scaled_values<E, WIDE>(pt, 2 * q + 1, chunk_signs4<E, WBF16>(raw, 2 * q + 1), sc2);
                dst[q] = make_uint4(lo.x, lo.y, hi.x, hi.y);
            }
        }
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
    const int T0 = ROT ? a.rot_block / E : 1;
    int threads = 0;
    if (a.C > kRoundThreadsMax) {
        // 512 lanes hold whole rotation blocks (at most 16384 values at 32 a lane; for the smaller
        // groups a block of more than 512 lanes is refused)
        if (ROT && a.rot_block / E > kRoundThreadsMax) return PVQ_ERR_UNSUPPORTED;
        threads = kRoundThreadsMax;
        a.rpt = 1;
        a.chunks = (a.C + threads - 1) / threads;
    } else {
        // Whole rows: the block that leaves the fewest lanes idle; among equals the largest, or the smallest when the launch
        // would not fill the SMs anyway.  Blocks of up to 128 threads, and of up to 256 where such blocks stay and there is work for
        // one of 128 threads an SM: those above 128 are counted 3 % dearer (N = 128, 16384 x 4096: 95.3 us with 128, 97.6 with 256), but
        // for groups on eight lanes (4096 x 4096: 32.9 and 30.8).  (With at most 128, us: 6553 x 2560 at N = 32 26.7 instead
        // of 21.9, 7281 x 2304 at N = 128 36.5 instead of 29.6.  Less work, 100 x 1152 at N = 64, 4.6 with 128, 5.1 with 256.
        // Blocks that take one tile, fp32: 4096 x 1024 at N = 128 11.1 with 128, 13.6 with 256.)  Rotated in blocks that span
        // warps: whole blocks, and no more threads than need be, as they meet often (B = 2048, 8192 rows: 64 threads
        // 41.5, 128 38.2, 256 39.2).
        a.chunks = 1;
        const int need = (a.C + 31) / 32 * 32;
        const bool large = BF16 && a.rows * a.C >= 128ll * di.sms;
        const int most = std::max(need, T0 > 32 ? (BF16 ? 128 : 64) : (large ? 256 : 128));
        double best = -1.0;
        for (int t = std::max(64, need); t <= most; t += 32) {
            if (T0 > 32 && t % T0 != 0) continue;
            const int rpt = t / a.C;
            const long long tiles = (a.rows + rpt - 1) / rpt;
            const double cost = static_cast<double>(tiles * t) * (L < 8 && t > 128 ? 1.03 : 1.0);
            if (best < 0.0 || cost < best || (cost == best && tiles >= 2 * di.sms)) {
                best = cost;
                threads = t;
            }
        }
        a.rpt = threads / a.C;
    }
    const long long tiles = (a.rows + a.rpt - 1) / a.rpt;
    if (tiles > 0x7fffffffLL) return PVQ_ERR_UNSUPPORTED;
    a.tiles = static_cast<unsigned>(tiles);
    a.levels_off = a.b <= 8 ? 4u * kCodebookMax : 0u;
    a.ss_off = 2u * a.levels_off;
    a.signs_off = (a.ss_off + 2u * static_cast<uint32_t>(a.rpt * a.gp) * 4u + 15u) & ~15u;
    a.xbuf_off = (a.signs_off + (ROT ? static_cast<uint32_t>(a.rot_block / E) * 4u : 0u) + 127u) & ~127u;
    a.ring_off = (a.xbuf_off + (ROT ? static_cast<uint32_t>(threads) * E * 4u : 0u) + 127u) & ~127u;
    a.tile_bytes = static_cast<uint32_t>(threads) * E * 2u;
    size_t smem = a.ring_off;
    void (*kern)(RoundArgs) = roundtrip_rows_kernel<E, L, BF16, WIDE, ROT>;
    bool stays = false;  // the block stays and takes tile after tile
    if constexpr (BF16) {
        a.bufs = !ROT || E != 32 ? 3 : (T0 > 32 ? 1 : 2);
        if (a.chunks == 1 && smem + a.bufs * a.tile_bytes <= static_cast<size_t>(di.smem_max)) {
            stays = true;
            smem += a.bufs * a.tile_bytes;
            kern = roundtrip_kernel<E, L, WIDE, ROT>;
        }
    }
    if (smem > static_cast<size_t>(di.smem_max)) return PVQ_ERR_UNSUPPORTED;
    int per_sm = 0;
    if ((st = prepare_kernel(reinterpret_cast<const void*>(kern), threads, smem, &per_sm)) != PVQ_OK) return st;
    if (per_sm < 1) return PVQ_ERR_UNSUPPORTED;
    // A launch of a few blocks an SM asks for the shared memory that keeps more than its share of them off an SM: where calls follow
    // one another, the blocks of one are placed while those of the one before still run, and several came to lie on one SM while
    // others had none.  (us, without and with: 100 x 8192 rotated, B = 8192, 16.5 and 7.7, B = 4096 13.1 and 8.0; 600 x 2048, B = 2048,
    // 15.9 and 8.7; not rotated, N = 128, 256 x 4096 8.2 and 4.7.  From some 2 M values on it makes no difference.)
    const int share = static_cast<int>((tiles + di.sms - 1) / di.sms);
    if (share < per_sm) {
        const size_t sm_bytes = static_cast<size_t>(di.smem_max) + 1280;  // of an SM; 1024 are added for every block
        smem = std::max(smem, (sm_bytes / (share + 1) - 1024 + 255) & ~size_t(127));
        if ((st = prepare_kernel(reinterpret_cast<const void*>(kern), threads, smem, &per_sm)) != PVQ_OK) return st;
    }
    const unsigned grid = stays ? std::min(a.tiles, static_cast<unsigned>(di.sms * per_sm)) : a.tiles;
    return launch_hot(kern, grid, threads, smem, stream, a);
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
                     uint32_t* status, uint32_t* debug_status, cudaStream_t stream) {
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
    a.minus_zero = -0.0f;
    a.status = status;
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
