// The encode kernel for codes of up to four words and up to 127 pulses (Sec. 3.3 Steps 3, 4, 5, 7;
// Algorithms 1 and 2): group sizes 8 to 64, the tables of the Fischer index in shared memory.
//
// What bounds it: issue slots and the half-rate integer pipe.  So:
//   - the last pulses of the direction are found bit by bit in bit planes of the residuals (pvq_quant.cuh),
//     not by a sorting network;
//   - the index is summed from one table entry per position, E(i, m) with m = 2 k' + (y_i > 0), k' the
//     pulses behind position i (the telescoped tables, `cenc` of TableLayout, interleaved).  The
//     k' of four positions are one multiplication (a running sum over the bytes of the packed
//     point), so a position costs a byte extraction, one table read and the addition;
//   - for codes of two and three words M = -E is kept as doubles, 48 bits each (32 of them add up
//     exactly), so that the additions are one or two instructions on the fp64 pipe, which nothing
//     else uses, without carries; positions whose M stays below 2^48 have no upper half to read;
//   - the input arrives in shared memory by asynchronous copies of whole lines, a chunk ahead (or as soon as the
//     chunk before has been read, LaneGeom::in_bufs), each lane's run padded by 16 bytes so that the
//     lanes' 16-byte reads hit different banks.
// Larger groups and wider codes (any group size, up to 32 words, any K): the same kernel with a group on up
// to 8 lanes, the point in 16-bit halves, and Algorithm 2's two terms per position read from the cumulative
// tables in global memory (L1, L2), only as many words as the position's counts have.
// One block per SM shares one copy of the tables; within it, teams of threads take whole rows, in chunks
// of a lane per 32 values, each at its own pace.  A team of one warp needs no barrier and spreads the
// work per row over most chunks; larger teams make more tiles of few rows (LaneGeom's choice in the launcher).
#pragma once
#include <cuda_fp16.h>

#include <algorithm>

#include "pvq_quant.cuh"
#include "pvq_rows.cuh"
#include "pvq_walk.cuh"

namespace pvq {

// threads per block: the wide kernels' accumulators need more registers.  (4096 x 4096, N = 32, 96 bits: 768 threads
// 41.8 us, 896 threads 37.6 us.)
template <int W>
constexpr int kLaneThreads = W <= 4 ? 896 : (W <= 16 ? 768 : 512);
constexpr int kSplitBit = 48;

struct LaneGeom {
    int team, teams;                // threads per team, teams per block
    int in_bufs;                    // 2: the next chunk's input is asked for a chunk ahead; 1: as soon as the chunk's point is there
    uint32_t team_off, team_bytes;  // the teams' areas: [input buffers], then one (a team of one warp) or two each of [energies][LS amplitudes][index words]
    uint32_t in_bytes;              // of one input buffer
    uint32_t ss_off, amp_off, idx_off;  // inside a team's area
    int ss_floats, idx_words;       // per buffer
    int wide_blocks;                // blocks of four positions with entries of 2^48 and more (two and three words)
    float minus_zero;
};

// The staged table: rows by position, RE entries (64, 112, 128 or 256, the first that holds 2 K + 2) of 4, 8 or 16 bytes;
// two and three words: a plane of lower halves, then one of upper halves for the first wide_blocks * 4 positions
// (for all positions where a group has two lanes, both of which run through as many blocks).
template <int W>
constexpr int kLaneEntry = W == 1 ? 4 : (W <= 3 ? 8 : 16);
template <int N>
__host__ __device__ constexpr int lane_upper_rows(int wide_blocks) {
    return N <= 32 ? wide_blocks * 4 : N;
}
template <int N, int W, int RE>
__host__ __device__ constexpr int lane_table_bytes(int wide_blocks) {
    return N * RE * kLaneEntry<W> + (W == 2 || W == 3 ? lane_upper_rows<N>(wide_blocks) * RE * 8 : 0);
}

// bytes from one lane's values in an input buffer to the next lane's
template <int E, bool BF16>
constexpr int kLaneRun = E * (BF16 ? 2 : 4) + (E * (BF16 ? 2 : 4) >= 32 ? 16 : 0);

__device__ __forceinline__ void team_barrier(int id, int threads) {
    if (threads == 32)
        __syncwarp();
    else
        asm volatile("bar.sync %0, %1;" ::"r"(id + 1), "r"(threads) : "memory");
}

__device__ __forceinline__ void copy16_async(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void copy_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

struct FetchSharedF32 {
    const float* p;
    __device__ __forceinline__ float operator()(int i) const { return fabsf(p[i]); }
};

template <typename T>
__device__ __forceinline__ T lane_entry(const uint8_t* p) {
#ifdef PVQ_DEBUG
    if (!debug_table_ok(shared_addr(p), sizeof(T))) return T{};
#endif
    return *reinterpret_cast<const T*>(p);
}

// The block's threads meet once, when the tables are staged: those that go on wait, the others only say that they are done.
__device__ __forceinline__ void tables_done() { asm volatile("bar.arrive 0, %0;" ::"r"(blockDim.x) : "memory"); }
__device__ __forceinline__ void tables_wait() { asm volatile("bar.sync 0, %0;" ::"r"(blockDim.x) : "memory"); }

// Stages the tables, with `threads` threads of which this is the `first`-th: entry (i, m) from the blob's telescoped word planes.
template <int N, int W, int RE>
__device__ __forceinline__ void stage_lane_table(uint8_t* tab, const uint32_t* blob, const TableLayout& L, int K, int wide_blocks, int first, int threads) {
    constexpr int TW = W <= 2 ? W : 4;
    // entry by entry, several loads in flight: a small launch consists mostly of this
#pragma unroll 4
    for (int e = first; e < N * RE; e += threads) {
        const int i = e / RE, m = e - i * RE;
        if (m >= 2 * K + 2) continue;
        const uint32_t* src = blob + ((m & 1) ? L.cenc_off[1] : L.cenc_off[0]) / 4 + static_cast<size_t>(i) * TW * L.crow + (m >> 1);
        uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int j = 0; j < W; ++j) w[j] = __ldg(src + j * L.crow);
        uint8_t* dst = tab + e * kLaneEntry<W>;
        if constexpr (W == 1) {
            *reinterpret_cast<uint32_t*>(dst) = w[0];
        } else if constexpr (W <= 3) {
            // E is never positive: M = -E in 32 W bits, split
            mp<W> zero, v, neg;
            mp_zero(zero);
#pragma unroll
            for (int j = 0; j < W; ++j) v.w[j] = w[j];
            mp_sub_borrow<W>(neg, zero, v);
            const unsigned long long low = static_cast<unsigned long long>(neg.w[0]) | (static_cast<unsigned long long>(neg.w[1]) << 32);
            const unsigned long long up = (low >> kSplitBit) | (static_cast<unsigned long long>(W == 3 ? neg.w[W - 1] : 0u) << (64 - kSplitBit));
            *reinterpret_cast<double*>(dst) = static_cast<double>(low & ((1ull << kSplitBit) - 1ull));
            if (i < lane_upper_rows<N>(wide_blocks)) *reinterpret_cast<double*>(dst + N * RE * 8) = static_cast<double>(up);
        } else {
            *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// The columns of four positions (word j of the packed point): bytes m = 2 k' + (y > 0).
// base: pulses behind the word's positions, updated for the next word.
__device__ __forceinline__ uint32_t lane_columns(uint32_t y, uint32_t neg, uint32_t& base) {
    const uint32_t behind = __byte_perm(y, base, 0x2104);                              // base, then the word's last three
    const uint32_t positive = ((y + 0x7f7f7f7fu) >> 7) & kOne4 & ~neg;                 // |y| <= 127: bit 7 is y != 0
    base = __dp4a(y, kOne4, base);
    return behind * 0x02020202u + positive;
}
__device__ __forceinline__ uint32_t byte_of(uint32_t m4, int b) {
    return b == 3 ? m4 >> 24 : (b == 0 ? m4 & 0xffu : __byte_perm(m4, 0u, 0x4440u + b));
}

// The index of the group's point: K pulses, this lane's positions and signs (0xff: negative).
template <int E, int L, int W, int RE>
__device__ __forceinline__ mp<W> lanes_index(const LanePoint<E, false>& pt, const uint32_t (&neg)[E / 4], int K, const uint8_t* tab,
                                             int wide_blocks, const mp<W>& start) {
    constexpr int J = E / 4, N = E * L, EB = kLaneEntry<W>, ROW = RE * EB;
    const int sub = static_cast<int>(threadIdx.x) & (L - 1);
    uint32_t base = 0u;  // pulses behind the positions that are still to come
    if constexpr (L > 1) {
        static_assert(L == 2, "the pulses of the lanes behind are K minus this lane's");
        uint32_t own = 0u;
#pragma unroll
        for (int j = 0; j < J; ++j) own += pt.y[j];
        base = sub == 0 ? static_cast<uint32_t>(K) - __dp4a(own, kOne4, 0u) : 0u;
        tab += sub * E * ROW;
    }
    mp<W> c = start;
    if constexpr (W == 1) {
        uint32_t sum = 0u;
#pragma unroll
        for (int j = J - 1; j >= 0; --j) {
            const uint32_t m4 = lane_columns(pt.y[j], neg[j], base);
#pragma unroll
            for (int b = 0; b < 4; ++b) sum += lane_entry<uint32_t>(tab + byte_of(m4, b) * EB + (4 * j + 3 - b) * ROW);
        }
        c.w[0] += static_cast<uint32_t>(group_add<L>(static_cast<int>(sum)));
    } else if constexpr (W <= 3) {
        double lo[2] = {0.0, 0.0}, hi[2] = {0.0, 0.0};  // two chains each; together no more than 32 entries
#pragma unroll
        for (int j = J - 1; j >= 0; --j) {
            const uint32_t m4 = lane_columns(pt.y[j], neg[j], base);
            if (j < wide_blocks) {  // the same for all threads
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const uint8_t* p = tab + byte_of(m4, b) * EB + (4 * j + 3 - b) * ROW;
                    lo[b & 1] += lane_entry<double>(p);
                    hi[b & 1] += lane_entry<double>(p + N * ROW);
                }
            } else {
#pragma unroll
                for (int b = 0; b < 4; ++b) lo[b & 1] += lane_entry<double>(tab + byte_of(m4, b) * EB + (4 * j + 3 - b) * ROW);
            }
        }
        unsigned long long l = static_cast<unsigned long long>(lo[0] + lo[1]), h = static_cast<unsigned long long>(hi[0] + hi[1]);
#pragma unroll
        for (int o = 1; o < L; o <<= 1) {
            l += __shfl_xor_sync(kFull, l, o);
            h += __shfl_xor_sync(kFull, h, o);
        }
        const unsigned long long up = h << (kSplitBit - 32);
        mp<W> t, u, d;
        mp_zero(t);
        mp_zero(u);
        t.w[0] = static_cast<uint32_t>(l), t.w[1] = static_cast<uint32_t>(l >> 32);
        u.w[1] = static_cast<uint32_t>(up);
        if constexpr (W == 3) u.w[2] = static_cast<uint32_t>(up >> 32);
        mp_add<W>(t, u);
        mp_sub_borrow<W>(d, c, t);
        c = d;
    } else {
        mp<4> sum;
        mp_zero(sum);
#pragma unroll
        for (int j = J - 1; j >= 0; --j) {
            const uint32_t m4 = lane_columns(pt.y[j], neg[j], base);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const uint4 e = lane_entry<uint4>(tab + byte_of(m4, b) * EB + (4 * j + 3 - b) * ROW);
                const mp<4> m = {{e.x, e.y, e.z, e.w}};
                mp_add<4>(sum, m);
            }
        }
#pragma unroll
        for (int o = 1; o < L; o <<= 1) {
            mp<4> other;
#pragma unroll
            for (int w = 0; w < 4; ++w) other.w[w] = __shfl_xor_sync(kFull, sum.w[w], o);
            mp_add<4>(sum, other);
        }
        mp_add<4>(c, sum);
    }
    return c;
}

// Words [0, W) of a table entry of TW words in global memory, no more than `words` of them (the rest zero).
template <int W>
__device__ __forceinline__ mp<W> global_entry(const uint32_t* p, int TW, int words) {
    mp<W> t;
    if ((TW & 3) == 0) {
#pragma unroll
        for (int v = 0; v < (W + 3) / 4; ++v) {
            uint4 q = make_uint4(0u, 0u, 0u, 0u);
            if (4 * v < words) q = __ldg(reinterpret_cast<const uint4*>(p) + v);
            const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (4 * v + u < W) t.w[4 * v + u] = w[u];
        }
    } else if ((TW & 1) == 0) {
#pragma unroll
        for (int v = 0; v < (W + 1) / 2; ++v) {
            uint2 q = make_uint2(0u, 0u);
            if (2 * v < words) q = __ldg(reinterpret_cast<const uint2*>(p) + v);
            t.w[2 * v] = q.x;
            if (2 * v + 1 < W) t.w[2 * v + 1] = q.y;
        }
    } else {
#pragma unroll
        for (int w = 0; w < W; ++w) t.w[w] = w < words ? __ldg(p + w) : 0u;
    }
    return t;
}

// The index of the group's point from the cumulative tables (Algorithm 2, App. C.2): with k pulses before a
// position and k' behind it, U(n,k) - U(n,k') for y < 0, U(n,k) - 2 V(n,k') for y > 0, nothing
// for y = 0.  s_words: words of the counts at every position.  All lanes of a group get the sum.
template <int E, int L, int W>
__device__ __forceinline__ mp<W> lanes_index_global(const LanePoint<E, true>& pt, const uint32_t (&neg)[E / 4], int K, const uint32_t* tab_u,
                                                    const uint32_t* tab_2v, int TW, const uint8_t* s_words) {
    const int sub = static_cast<int>(threadIdx.x) & (L - 1);
    int behind = 0;  // pulses behind the lane's positions
    if constexpr (L > 1) {
        uint32_t own2 = 0u;
#pragma unroll
        for (int h = 0; h < E / 2; ++h) own2 += pt.y[h];
        const int own = static_cast<int>((own2 & 0xffffu) + (own2 >> 16));
#pragma unroll
        for (int o = 1; o < L; ++o) {
            const int other = __shfl_xor_sync(kFull, own, o);
            if ((sub ^ o) > sub) behind += other;
        }
    }
    mp<W> c;
    mp_zero(c);
    const uint32_t rowlen = static_cast<uint32_t>(K + 2) * TW;
#pragma unroll
    for (int h = E / 2 - 1; h >= 0; --h) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {  // position 2h + 1 (low half), then 2h
            const int pos = 2 * h + 1 - half;
            const int y = static_cast<int>(half ? pt.y[h] >> 16 : pt.y[h] & 0xffffu);
            const bool negative = (neg[pos / 4] >> (8 * (3 - (pos & 3)))) & 1u;
            if (y != 0) {
                const int i = sub * E + pos;
                const int words = s_words[i];
                const uint32_t row = static_cast<uint32_t>(i) * rowlen;
                const mp<W> u = global_entry<W>(tab_u + row + static_cast<uint32_t>(behind + y + 1) * TW, TW, words);
                const mp<W> x = global_entry<W>((negative ? tab_u : tab_2v) + row + static_cast<uint32_t>(behind + 1) * TW, TW, words);
                mp_add<W>(c, u);
                mp<W> d;
                mp_sub_borrow<W>(d, c, x);
                c = d;
                behind += y;
            }
        }
    }
#pragma unroll
    for (int o = 1; o < L; o <<= 1) {
        mp<W> other;
#pragma unroll
        for (int w = 0; w < W; ++w) other.w[w] = __shfl_xor_sync(kFull, c.w[w], o);
        mp_add<W>(c, other);
    }
    return c;
}

// Step 4 as least squares: a = (sum |y_i| |x_i|) / sqrt(sum y_i^2), the rounded products summed by
// the balanced tree.
template <int E, int L, bool BF16, bool WIDE>
__device__ __forceinline__ float least_squares_amplitude(const LanePoint<E, WIDE>& pt, const uint8_t* mine) {
    float t[E];
    unsigned sq = 0u;
#pragma unroll
    for (int j = 0; j < E / 4; ++j) {
        float x[4];
        if constexpr (BF16) {
            const uint2 q = reinterpret_cast<const uint2*>(mine)[j];
            x[0] = __uint_as_float((q.x & 0x7fffu) << 16), x[1] = __uint_as_float(q.x & 0x7fff0000u);
            x[2] = __uint_as_float((q.y & 0x7fffu) << 16), x[3] = __uint_as_float(q.y & 0x7fff0000u);
        } else {
            const float4 q = reinterpret_cast<const float4*>(mine)[j];
            x[0] = fabsf(q.x), x[1] = fabsf(q.y), x[2] = fabsf(q.z), x[3] = fabsf(q.w);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            unsigned y;
            if constexpr (WIDE)
                y = (e & 1) ? pt.y[2 * j + e / 2] & 0xffffu : pt.y[2 * j + e / 2] >> 16;
            else
                y = (pt.y[j] >> (8 * (3 - e))) & 0xffu;
            sq += y * y;
            t[4 * j + e] = __fmul_rn(static_cast<float>(y), x[e]);
        }
    }
    const float dot = group_add<L>(tree_sum<E>(t));
    const int ssy = group_add<L>(static_cast<int>(sq));
    return __fdiv_rn(dot, __fsqrt_rn(static_cast<float>(ssy)));
}

// Where a team works: chunk `ch` of a tile (whole rows that fit the team, or one longer row in chunks).
struct LanePlace {
    unsigned tile;
    int ch, mi, rl, c0;  // matrix; row inside the tile and lane inside the row (of chunk 0) of this thread
};

__device__ __forceinline__ void enter_matrix(const BatchArgs& a, LanePlace& p, int mi, int tid, int L) {
    p.mi = mi;
    const int C = a.m[mi].G * L;
    p.rl = a.m[mi].chunks == 1 ? tid / C : 0;
    p.c0 = a.m[mi].chunks == 1 ? tid - p.rl * C : tid;
}

// Asks for a warp's share of the input of a place.
template <int E, int L, bool BF16>
__device__ __forceinline__ void request_input(const BatchArgs& a, const LanePlace& p, uint32_t dst0, int T, int tid) {
    constexpr int ES = BF16 ? 2 : 4, P = E * ES / 16, RUN = kLaneRun<E, BF16>;
    const int lane = threadIdx.x & 31, wbase = tid & ~31;
    const MatrixArgs& m = a.m[p.mi];
    const int C = m.G * L;
    const long long row0 = static_cast<long long>(p.tile - m.tile_begin) * m.rows_per_tile;
    const int nr = static_cast<int>(min(static_cast<long long>(m.rows_per_tile), m.rows - row0));
    const int valid = m.chunks == 1 ? nr * C : C - p.ch * T;  // lanes that have values
    const uint8_t* src = static_cast<const uint8_t*>(m.x) +
                         (static_cast<size_t>(row0) * m.ld + static_cast<size_t>(p.ch * T + wbase) * E) * ES + lane * 16;
    const long long skip = m.chunks == 1 ? (m.ld - m.cols) * ES : 0;
#pragma unroll
    for (int v = 0; v < P; ++v) {
        const int q = v * 32 + lane;  // 16-byte piece of the warp's run
        const int l = wbase + q / P;  // the lane it belongs to
        if (l < valid) {
            const uint8_t* s = src + v * 512;
            if (skip != 0) s += static_cast<long long>(l / C) * skip;
            copy16_async(dst0 + l * RUN + (q & (P - 1)) * 16, s);
        }
    }
    copy_async_commit();
}

// Index words of a finished tile -> memory; the buffer is cleared for the tile after next.
__device__ __forceinline__ void flush_index_words(const MatrixArgs& m, unsigned tile, uint32_t* s_idx, int T, int tid) {
    const int iw = m.sstride >> 2;
    const long long row0 = static_cast<long long>(tile - m.tile_begin) * m.rows_per_tile;
    for (int i = tid; i < m.rows_per_tile * iw; i += T) {
        const int r2 = m.rows_per_tile == 1 ? 0 : i / iw;
        if (row0 + r2 < m.rows) reinterpret_cast<uint32_t*>(m.scale_idx + static_cast<size_t>(row0 + r2) * m.sstride)[i - r2 * iw] = s_idx[i];
        s_idx[i] = 0u;
    }
}

// RE: entries per row of the staged table (codes of exactly W words); 0: the tables stay in global memory,
// codes of up to W words.  LATE: for small launches, whose staging of the tables it hides.
template <int E, int L, int W, int RE, bool BF16, bool LS, bool LATE>
__global__ void __launch_bounds__(kLaneThreads<W>, 1) encode_lanes_kernel(const __grid_constant__ BatchArgs a,
                                                                           const __grid_constant__ LaneGeom g) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint8_t s_words[RE == 0 ? E * L : 1];
    constexpr int N = E * L;
    constexpr bool GLOBAL = RE == 0;
    constexpr int P = E * (BF16 ? 2 : 4) / 16, RUN = kLaneRun<E, BF16>;
    const int K = a.K, b = a.scale_bits;
    const int Wc = GLOBAL ? a.code_words : W;  // words of a code in memory
    const TableLayout TL = table_layout(N, K, Wc);
    grid_launch_dependents();
    const int T = g.team, team = threadIdx.x / T, tid = threadIdx.x - team * T, lane = threadIdx.x & 31;
    uint8_t* area = smem + g.team_off + team * g.team_bytes;

    LanePlace at;
    at.tile = blockIdx.x + static_cast<unsigned>(team) * gridDim.x;  // the first tiles go to different SMs
    at.ch = 0;
    const unsigned stride = gridDim.x * static_cast<unsigned>(g.teams);
    const bool works = team < g.teams && at.tile < a.total_tiles;
    if (works) {
        enter_matrix(a, at, find_matrix(a, at.tile), tid, L);
        uint32_t* s_idx2 = reinterpret_cast<uint32_t*>(area + g.idx_off);
        for (int i = tid; i < (T == 32 ? 1 : 2) * g.idx_words; i += T) s_idx2[i] = 0u;
    }
    grid_dependency_wait();
    if (works) request_input<E, L, BF16>(a, at, shared_addr(area), T, tid);
    mp<GLOBAL ? 1 : W> start;
    if constexpr (GLOBAL) {
        // words of N(n+1,K) = U(n,K), which no term of the position exceeds (N(N,K) may be a power of two
        // beyond the entry: all words)
        for (int i = threadIdx.x; i < N; i += blockDim.x) {
            const uint32_t* u = a.table + TL.enc_off[0] / 4 + (static_cast<size_t>(i) * (K + 2) + K + 1) * TL.top_words;
            int words = Wc;
            while (i > 0 && words > 1 && __ldg(u + words - 1) == 0u) --words;
            s_words[i] = static_cast<uint8_t>(words);
        }
#ifdef PVQ_DEBUG
        debug_begin(0u, 0u, 0u, 0u, 0u, a.debug_status);
#endif
    } else {
        // LATE: most threads have no values.  They stage the tables while the others quantise, which wait half way through
        // their first chunk.
        const int busy = g.team * static_cast<int>(min(static_cast<unsigned>(g.teams), (a.total_tiles - blockIdx.x + gridDim.x - 1u) / gridDim.x));
        const int skip = LATE ? busy : 0, first = static_cast<int>(threadIdx.x) - skip;
        if (first >= 0) stage_lane_table<N, W, GLOBAL ? 64 : RE>(smem, a.table, TL, K, g.wide_blocks, first, static_cast<int>(blockDim.x) - skip);
#pragma unroll
        for (int w = 0; w < W; ++w) start.w[GLOBAL ? 0 : w] = a.table[TL.start_off / 4 + w];
#ifdef PVQ_DEBUG
        debug_begin(shared_addr(smem), shared_addr(smem) + lane_table_bytes<N, W, GLOBAL ? 64 : RE>(g.wide_blocks), 0u, 0u, 0u, a.debug_status);
#endif
    }
    if constexpr (LATE) {
        if (!works) {
            tables_done();
            return;
        }
    } else {
        __syncthreads();  // the tables; from here on the teams go their own way
        if (!works) return;
    }
    bool tables_here = !LATE;
    const int wide_blocks = g.wide_blocks;

    int in_buf = 0, buf = 0;
    const int in_flip = g.in_bufs - 1;
    int done_mi = -1;  // matrix of the tile before, whose index words are still to be written out
    for (;; in_buf ^= in_flip) {
        copy_async_wait<0>();
        __syncwarp();
        const LanePlace cur = at;
        const MatrixArgs& m = a.m[cur.mi];
        const bool last_chunk = cur.ch + 1 == m.chunks;
        // what comes next, and its input
        bool more = true;
        if (!last_chunk) {
            at.ch = cur.ch + 1;
        } else {
            at.ch = 0;
            at.tile = cur.tile + stride;
            more = at.tile < a.total_tiles;
            if (more && cur.mi + 1 < a.count && at.tile >= a.m[cur.mi + 1].tile_begin) {
                int ni = cur.mi + 1;
                while (ni + 1 < a.count && at.tile >= a.m[ni + 1].tile_begin) ++ni;
                enter_matrix(a, at, ni, tid, L);
            }
        }
        if (more && in_flip != 0) request_input<E, L, BF16>(a, at, shared_addr(area + (in_buf ^ 1) * g.in_bytes), T, tid);

        const int G = m.G, C = G * L, gp = G > 1 ? 1 << (32 - __clz(G - 1)) : 1;
        const long long row = static_cast<long long>(cur.tile - m.tile_begin) * m.rows_per_tile + cur.rl;
        const bool row_ok = cur.rl < m.rows_per_tile && row < m.rows;
        float* s_ss = reinterpret_cast<float*>(area + g.ss_off) + buf * g.ss_floats;
        float* s_amp = reinterpret_cast<float*>(area + g.amp_off) + buf * g.ss_floats;
        {
            const int c = cur.c0 + cur.ch * T;
            const uint8_t* mine = area + in_buf * g.in_bytes + tid * RUN;
            uint32_t neg[E / 4];
            LanePoint<E, GLOBAL> pt;
            float ss;
            {
                // (a lane beyond the values works on whatever is there: any bits are safe)
                uint32_t raw[kRawWords<E, BF16>];
                float ax[E], l1;
#pragma unroll
                for (int v = 0; v < P; ++v) {
                    const uint4 q = reinterpret_cast<const uint4*>(mine)[v];
                    raw[4 * v] = q.x, raw[4 * v + 1] = q.y, raw[4 * v + 2] = q.z, raw[4 * v + 3] = q.w;
                }
#pragma unroll
                for (int j = 0; j < E / 4; ++j) neg[j] = chunk_signs4<E, BF16>(raw, j);
                group_norms<E, L, BF16>(raw, ax, l1, ss, g.minus_zero);
                auto tables = [&]() {
                    if (LATE && !tables_here) {
                        __syncwarp();
                        tables_wait();
                        tables_here = true;
                    }
                };
                if constexpr (BF16)
                    quantize_group<E, L, GLOBAL>(ax, l1, K, FetchShared{reinterpret_cast<const unsigned short*>(mine)}, pt, g.minus_zero, 0, tables);
                else
                    quantize_group<E, L, GLOBAL>(ax, l1, K, FetchSharedF32{reinterpret_cast<const float*>(mine)}, pt, g.minus_zero, 0, tables);
            }
            const bool leader = row_ok && c < C && (c & (L - 1)) == 0;
            const int slot = cur.rl * gp + c / L;
            if (leader && PVQ_DEBUG_INDEX(slot, g.ss_floats, PVQ_DEBUG_SHARED_INDEX)) s_ss[slot] = ss;
            if constexpr (LS) {
                const float ls = least_squares_amplitude<E, L, BF16, GLOBAL>(pt, mine);
                if (leader) s_amp[slot] = ls;
            }
            if (more && in_flip == 0) {
                __syncwarp();  // (the warp's lanes asked for the input, and are through with it)
                request_input<E, L, BF16>(a, at, shared_addr(area), T, tid);
            }
            if (!pt.has_dir) {  // (K, 0, ..., 0), positive
#pragma unroll
                for (int j = 0; j < E / 4; ++j) neg[j] = 0u;
            }
            const long long group = row * G + c / L;
            if constexpr (GLOBAL) {
                const mp<W> code = lanes_index_global<E, L, W>(pt, neg, K, a.table + TL.enc_off[0] / 4, a.table + TL.enc_off[1] / 4, TL.top_words, s_words);
                // the lanes of the group share the stores
                if (row_ok && c < C) {
                    uint32_t* cp = m.codes + static_cast<size_t>(group) * Wc;
                    const bool quads = ((Wc & 3) | (reinterpret_cast<uintptr_t>(m.codes) & 15u)) == 0;
#pragma unroll
                    for (int v = 0; v < (W + 3) / 4; ++v) {
                        if ((v & (L - 1)) != (c & (L - 1)) || 4 * v >= Wc) continue;
                        uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (4 * v + u < W) w[u] = code.w[4 * v + u < W ? 4 * v + u : 0];
                        if (quads) {
                            reinterpret_cast<uint4*>(cp)[v] = make_uint4(w[0], w[1], w[2], w[3]);
                        } else {
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                if (4 * v + u < Wc) cp[4 * v + u] = w[u];
                        }
                    }
                }
            } else {
                const mp<W> code = lanes_index<E, L, W, GLOBAL ? 64 : RE>(pt, neg, K, smem, wide_blocks, start);
                if (leader && PVQ_DEBUG_INDEX(group, m.rows * G, PVQ_DEBUG_GLOBAL_STORE)) {
                    uint32_t* cp = m.codes + static_cast<size_t>(group) * W;
#pragma unroll
                    for (int w = 0; w < W; ++w) cp[w] = code.w[w];
                }
            }
        }
        if (!last_chunk) continue;

        // the tile's rows are complete: their energies, then the amplitude indices
        if (gp != G)  // zero padding of the rows' trees
            for (int j = tid; j < m.rows_per_tile * gp; j += T)
                if ((j & (gp - 1)) >= G && PVQ_DEBUG_INDEX(j, g.ss_floats, PVQ_DEBUG_SHARED_INDEX)) s_ss[j] = 0.0f;
        team_barrier(team, T);  // this tile's energies are in place; the previous tile's index words are complete
        uint32_t* s_idx = reinterpret_cast<uint32_t*>(area + g.idx_off) + buf * g.idx_words;
        if (done_mi >= 0) flush_index_words(a.m[done_mi], cur.tile - stride, reinterpret_cast<uint32_t*>(area + g.idx_off) + (buf ^ 1) * g.idx_words, T, tid);
        const float ss_row = row_energy(s_ss, gp, cur.rl, m.rows_per_tile, lane);
        const float* edges = m.edges;
        for (int c = cur.c0; row_ok && c < C; c += T) {
            if ((c & (L - 1)) != 0) break;
            const int gi = c / L;
            const float ss = s_ss[cur.rl * gp + gi];
            const float ls = LS ? s_amp[cur.rl * gp + gi] : 0.0f;
            int q = 0;
            if (b == 16) {  // the amplitude itself, as binary16
                q = __half_as_ushort(__float2half_rn(LS ? ls : __fsqrt_rn(ss)));
            } else {
                const float u = ss_row > 0.0f ? __fdiv_rn(LS ? __fmul_rn(ls, ls) : ss, ss_row) : 0.0f;
                q = amplitude_bin(u, b, [&](int i) { return __ldg(edges + i); });
            }
            if (gi == 0 && PVQ_DEBUG_INDEX(row, m.rows, PVQ_DEBUG_GLOBAL_STORE)) m.row_norm[row] = __fsqrt_rn(ss_row);
            const unsigned bit = static_cast<unsigned>(gi) * b;
            const unsigned sh = bit & 31u;
            const int word = cur.rl * (m.sstride >> 2) + static_cast<int>(bit >> 5);
            if (!PVQ_DEBUG_INDEX(word + (sh + b > 32u ? 1 : 0), g.idx_words, PVQ_DEBUG_SHARED_INDEX)) continue;
            atomicOr(s_idx + word, static_cast<uint32_t>(q) << sh);
            if (sh + b > 32u) atomicOr(s_idx + word + 1, static_cast<uint32_t>(q) >> (32u - sh));
        }
        if (T == 32) {  // no other warp to wait for: out with the index words, and the same buffers again
            __syncwarp();
            flush_index_words(m, cur.tile, s_idx, T, tid);
            __syncwarp();
            if (!more) break;
            continue;
        }
        done_mi = cur.mi;
        if (!more) {
            team_barrier(team, T);  // the last tile's index words are complete
            flush_index_words(m, cur.tile, s_idx, T, tid);
            break;
        }
        buf ^= 1;
    }
}

// Geometry and launch.  Returns PVQ_ERR_UNSUPPORTED when the case is not this kernel's (the
// caller then takes the general kernel).
template <int E, int L, int W, int RE, bool BF16, bool LS>
static int launch_encode_lanes_t(BatchArgs& a, cudaStream_t stream) {
    constexpr int N = E * L;
    DeviceInfo di;
    int st = device_info(&di);
    if (st != PVQ_OK) return st;
    LaneGeom g;
    g.minus_zero = -0.0f;
    g.wide_blocks = RE != 0 && (W == 2 || W == 3) ? (positions_from(N, a.K, kSplitBit) + 3) / 4 : 0;
    g.team_off = RE == 0 ? 0u : (static_cast<uint32_t>(lane_table_bytes<N, W, RE == 0 ? 64 : RE>(g.wide_blocks)) + 127u) & ~127u;

    // Team size: the one whose rounds of tiles cost least.  A chunk costs about as much as six times
    // what a tile adds (energies, amplitude indices), eight with a barrier between warps; what
    // decides is mostly how full the last round is.
    long long lanes = 0;
    for (int i = 0; i < a.count; ++i) lanes += a.m[i].rows * a.m[i].G * L;
    const bool long_launch = lanes > 8ll * di.sms * kLaneThreads<W>;
    double best = -1.0;
    LaneGeom chosen{};
    for (int t : {32, 64, 96, 128, 160, 192, 224, 256}) {
        LaneGeom c = g;
        c.team = t;
        long long tiles = 0, chunks_all = 0;
        int idx_words = 1, ss_floats = 4;
        for (int i = 0; i < a.count; ++i) {
            const MatrixArgs& m = a.m[i];
            const int C = m.G * L, rpt = C <= t ? t / C : 1, chunks = C <= t ? 1 : (C + t - 1) / t;
            const long long n = (m.rows + rpt - 1) / rpt;
            tiles += n;
            chunks_all += n * chunks;
            int gp = 1;
            while (gp < m.G) gp <<= 1;
            idx_words = std::max(idx_words, rpt * (m.sstride / 4));
            ss_floats = std::max(ss_floats, rpt * gp);
        }
        if (tiles > 0x7fffffffLL) return PVQ_ERR_UNSUPPORTED;
        c.in_bytes = (static_cast<uint32_t>(t) * kLaneRun<E, BF16> + 15u) & ~15u;
        c.ss_floats = (ss_floats + 3) & ~3;
        c.idx_words = idx_words;
        const uint32_t bufs = t == 32 ? 1u : 2u;
        // As many teams as the threads, the shared memory and (larger than a warp) the named barriers hold.  Where the
        // shared memory is what limits them, a long launch makes do with one input buffer a team: the wait for the input is
        // covered by the other warps.  (A decoder layer at N = 32, 96 bits: 23 warps and two buffers 336 us, 28 and one 286.)
        const long long most_teams = std::min(kLaneThreads<W> / t, t == 32 ? 32 : 15);
        auto place = [&](int in_bufs) {  // the team's area, and how many of them fit
            c.in_bufs = in_bufs;
            c.ss_off = static_cast<uint32_t>(in_bufs) * c.in_bytes;
            c.amp_off = c.ss_off + bufs * static_cast<uint32_t>(c.ss_floats) * 4u;
            c.idx_off = c.amp_off + (LS ? bufs * static_cast<uint32_t>(c.ss_floats) * 4u : 0u);
            c.team_bytes = (c.idx_off + bufs * static_cast<uint32_t>(idx_words) * 4u + 127u) & ~127u;
            return std::min(most_teams, (static_cast<long long>(di.smem_max) - c.team_off) / c.team_bytes);
        };
        long long teams = place(2);
        if (long_launch && teams < most_teams) {
            const long long more = place(1);
            teams = more > teams ? more : place(2);
        }
        if (teams < 1) continue;
        const double per_tile = static_cast<double>(chunks_all) / tiles + (t == 32 ? 0.16 : 0.25);
        const double rounds = std::ceil(static_cast<double>(tiles) / (static_cast<double>(teams) * di.sms));
        // In a long launch an SM with fewer warps than it holds runs them faster.  Few rounds take as long with few warps as with
        // many: the latency of tables and barriers, not issue.  (Taken for up to four times shorter, one-warp teams with a row in
        // many chunks won where rows are few: 1024 x 4096 at N = 64, 320 bits, 145 us instead of 84, N = 32, 96 bits 19.4
        // instead of 14.9.  A decoder layer, work for 51 rounds: 402 us, 454 without the factor.)
        const double load = long_launch ? static_cast<double>(teams) * t / kLaneThreads<W> : 1.0;
        const double cost = rounds * per_tile * load;
        if (best < 0.0 || cost < best) {
            best = cost;
            c.teams = static_cast<int>(std::min<long long>(teams, (tiles + di.sms - 1) / di.sms));
            chosen = c;
        }
    }
    if (best < 0.0) return PVQ_ERR_UNSUPPORTED;
    g = chosen;
    unsigned tiles = 0;
    for (int i = 0; i < a.count; ++i) {
        MatrixArgs& m = a.m[i];
        const int C = m.G * L;
        m.chunks = C <= g.team ? 1 : (C + g.team - 1) / g.team;
        m.rows_per_tile = C <= g.team ? g.team / C : 1;
        m.tile_begin = tiles;
        tiles += static_cast<unsigned>((m.rows + m.rows_per_tile - 1) / m.rows_per_tile);
    }
    a.total_tiles = tiles;

    const size_t smem = g.team_off + static_cast<size_t>(g.teams) * g.team_bytes;
    // at least sixteen warps to share the staging of the tables
    const int threads = std::max(g.team * g.teams, RE == 0 ? 64 : 512);
    const unsigned blocks = (tiles + g.teams - 1) / g.teams;
    // (512 x 512 fp32 7.3 -> 6.5 us.  In large launches the wait further on costs: 4096 x 4096 at N = 32 29.8 -> 30.1 us, fp32
    // 38.7 -> 39.4.)
    auto kern = encode_lanes_kernel<E, L, W, RE, BF16, LS, false>;
    if constexpr (RE != 0 && !LS) {
        const unsigned share = std::min<unsigned>(blocks, static_cast<unsigned>(di.sms));  // blocks, one an SM
        const int busy = g.team * static_cast<int>(std::min<unsigned>(static_cast<unsigned>(g.teams), (tiles + share - 1) / share));
        if (threads - busy >= 256) kern = encode_lanes_kernel<E, L, W, RE, BF16, LS, true>;
    }
    int per_sm = 0;
    if ((st = prepare_kernel(reinterpret_cast<const void*>(kern), threads, smem, &per_sm)) != PVQ_OK) return st;
    if (per_sm < 1) return PVQ_ERR_UNSUPPORTED;
    const unsigned grid = std::min<unsigned>(blocks, static_cast<unsigned>(di.sms * per_sm));
    // Tables in global memory: early only where the launch is small and its start counts (4096 groups at N = 16, 128 bits: 12.1 us
    // early, 14.3 in order; 32768 groups at N = 32, 200 bits, not yet a block an SM: 31.6 and 22.6).
    return launch_hot_if(RE != 0 || lanes < 32768, kern, grid, threads, smem, stream, a, g);
}

template <int E, int L, int W, bool BF16>
static int launch_encode_lanes(BatchArgs& a, cudaStream_t s) {
    const TableLayout L0 = table_layout(E * L, a.K, W);
    if (L0.cenc_bytes == 0) return PVQ_ERR_UNSUPPORTED;
    const bool ls = a.amp_mode == 1;
    switch (L0.crow) {
        case 32: return ls ? launch_encode_lanes_t<E, L, W, 64, BF16, true>(a, s) : launch_encode_lanes_t<E, L, W, 64, BF16, false>(a, s);
        case 64:
            if (2 * a.K + 2 <= 112)
                return ls ? launch_encode_lanes_t<E, L, W, 112, BF16, true>(a, s) : launch_encode_lanes_t<E, L, W, 112, BF16, false>(a, s);
            return ls ? launch_encode_lanes_t<E, L, W, 128, BF16, true>(a, s) : launch_encode_lanes_t<E, L, W, 128, BF16, false>(a, s);
        case 128: return ls ? launch_encode_lanes_t<E, L, W, 256, BF16, true>(a, s) : launch_encode_lanes_t<E, L, W, 256, BF16, false>(a, s);
        default: return PVQ_ERR_UNSUPPORTED;
    }
}

// The kernel with the tables in global memory, computing in W words: W and up to the code's width.
template <int N, int W>
static int launch_encode_lanes_global(BatchArgs& a, int dtype, cudaStream_t s) {
    constexpr int E = N <= 32 ? N : 32, L = N / E;
    const bool bf16 = dtype == PVQ_DTYPE_BF16;
    if (a.amp_mode == 1)
        return bf16 ? launch_encode_lanes_t<E, L, W, 0, true, true>(a, s) : launch_encode_lanes_t<E, L, W, 0, false, true>(a, s);
    return bf16 ? launch_encode_lanes_t<E, L, W, 0, true, false>(a, s) : launch_encode_lanes_t<E, L, W, 0, false, false>(a, s);
}

// Entry of the per-(N, W) translation units of the codes the shared-memory kernels are built for:
// everything but the rotation goes to the kernels above, with the tables in shared memory where
// they fit; the rotation to the general one.
template <int N, int W>
static int launch_encode_any(BatchArgs& a, int dtype, cudaStream_t s) {
    if (a.rot_block == 0) {
        BatchArgs b = a;
        if constexpr (W <= 4) {
            constexpr int E = N <= 32 ? N : 32, L = N / E;
            const int st = dtype == PVQ_DTYPE_BF16 ? launch_encode_lanes<E, L, W, true>(b, s) : launch_encode_lanes<E, L, W, false>(b, s);
            if (st != PVQ_ERR_UNSUPPORTED) return st;
        }
        // More than 127 pulses, but cumulative tables that fit shared memory: the general kernel with them, but for large bf16
        // input and the plain amplitude.  (us, general kernel and this one with tables in global memory, fp32: N = 8, 56 bits,
        // 1024 x 4096 24.6, 57.4, 4096 x 4096 79.6, 91.9; N = 16, 90 bits 25.9, 57.6, 78.6, 88.6; bf16: N = 8 2048 x 4096 56.3,
        // 64.9, 4096 x 4096 108.6, 89.2; N = 16 41.0, 55.3, 75.8, 73.8.)
        if constexpr ((N == 8 && W == 2) || (N == 16 && W == 3)) {
            long long values = 0;
            for (int i = 0; i < a.count; ++i) values += a.m[i].rows * a.m[i].cols;
            if (a.K > 127 && (values < (1 << 24) || dtype == PVQ_DTYPE_F32 || a.amp_mode == 1)) {
                b = a;
                const int st = launch_encode_nw<N, W, false>(b, dtype, s);
                if (st != PVQ_ERR_UNSUPPORTED) return st;
            }
        }
        b = a;
        return launch_encode_lanes_global<N, (W <= 4 ? 4 : W)>(b, dtype, s);
    }
    return launch_encode_nw<N, W, true>(a, dtype, s);
}

}  // namespace pvq
