// Encode kernel for wide codes: group size 64 with codes of 5 to 8 words, 128 with 9 to 12 (no rotation).
//
// The lanes kernel (pvq_encode_lanes.cuh) reads two entries of up to 12 words a position from tables in L2, at rows
// that differ between the lanes of a group: at N = 128, 384 bits that was four fifths of its time (4096 x 4096: 181 us).
// Here the index is a second phase with a thread per group.  A block takes a tile of whole rows, up to 28 x 32
// groups.  First its warps quantise the groups, a group on 2 or 4 lanes (pvq_quant.cuh), and leave the
// points in shared memory, a signed byte a value; then the amplitudes, once the rows' energies are complete;
// then every thread sums its group's index from the windowed tables (pvq_window.cuh), one entry of E a position, read
// word plane by word plane from the ring that a feeding warp keeps filled, the last block of rows first.  With q the
// number that the decoder searches, the code is N(N,K) - q: the sum of all E is 1 - q.  Same matrix: 54 us; the two phases
// do not overlap (59% of the issue slots used).
#include <algorithm>
#include <cstring>

#include "pvq_encode_impl.cuh"
#include "pvq_encode_lanes.cuh"
#include "pvq_window.cuh"

namespace pvq {

namespace {

constexpr int kEwWarps = 28, kEwBufs = 6;

struct EwGeom {
    int warps;          // that work (one more feeds)
    int quant_warps;    // of them quantise: as many as have room for their input
    int bufs;
    uint32_t buf_bytes;
    uint32_t slots_off, ss_off, amp_off, idx_off;
    int idx_words;
    float minus_zero;
};

__device__ __forceinline__ void ew_barrier(int threads) { asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); }

// A word of the tables in shared memory; ew_slot_word: of the points.
template <int OFF = 0>
__device__ __forceinline__ uint32_t ew_slot_word(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(OFF));
    return v;
}
template <int OFF = 0>
__device__ __forceinline__ uint32_t ew_load(uint32_t addr) {
#ifdef PVQ_DEBUG
    if (!debug_table_ok(addr + OFF, 4u)) return 0u;
#endif
    return ew_slot_word<OFF>(addr);
}
template <int PW, int PLANE, int FROM, int W = 0>
__device__ __forceinline__ void ew_entry(mp<PW>& e, uint32_t addr) {
    if constexpr (W < PW) {
        e.w[W] = ew_load<(FROM + W) * PLANE * 4>(addr);
        ew_entry<PW, PLANE, FROM, W + 1>(e, addr);
    }
}

// The last four words of a block's head: x (not used here), y delta, z klo, w khi - klo.
__device__ __forceinline__ uint4 ew_head(uint32_t stage) {
    static_assert(kWinDlo4 % 16 == 0 && kWinDelta == kWinDlo4 + 4 && kWinKlo4 == kWinDlo4 + 8 && kWinWidth4 == kWinDlo4 + 12, "one read");
    uint4 v;
#ifdef PVQ_DEBUG
    if (!debug_table_ok(stage + kWinDlo4, 16u)) return make_uint4(0u, 0u, 0u, 0u);
#endif
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4+%5];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(stage), "n"(kWinDlo4));
    return v;
}

// a[0] is the leading word of -q (the words above it are all ones, those below the block's are zero).
template <int W>
struct EwState {
    uint32_t a[W + 1];
    uint32_t delta;   // bits the number is shifted right by when the next block begins
    uint32_t behind;  // pulses behind the positions still to come
    uint32_t flag;    // bit 7 of a byte set: a position was outside its window
};

template <int PW, int PLANE, int W>
__device__ __forceinline__ void ew_block4(EwState<W>& st, uint32_t stage, uint32_t point) {
    mp<PW> v;
    v.w[PW - 1] = __funnelshift_r(st.a[0], 0xffffffffu, st.delta);
#pragma unroll
    for (int j = 1; j < PW; ++j) v.w[PW - 1 - j] = __funnelshift_r(st.a[j], st.a[j - 1], st.delta);
    const uint4 head = ew_head(stage);
    st.delta = head.y;
    // pulses behind each of the four positions: running sums, first position in the highest byte
    const uint32_t mag = point & 0x7f7f7f7fu;
    const uint32_t positive = (((mag + 0x7f7f7f7fu) & ~point) >> 7) & kOne4;
    const uint32_t local = __byte_perm(mag, st.behind, 0x2104) * kOne4 - head.z;
    st.flag |= local | (head.w - local);
    st.behind = __dp4a(mag, kOne4, st.behind);
    const uint32_t m4 = local + local + positive, rows = stage + kWinHead;
    mp<PW> e;
    ew_entry<PW, PLANE, 0>(e, rows + (m4 >> 24) * 4u);
    mp_add<PW>(v, e);
    ew_entry<PW, PLANE, PW>(e, rows + __byte_perm(m4, 0u, 0x4442) * 4u);
    mp_add<PW>(v, e);
    ew_entry<PW, PLANE, 2 * PW>(e, rows + __byte_perm(m4, 0u, 0x4441) * 4u);
    mp_add<PW>(v, e);
    ew_entry<PW, PLANE, 3 * PW>(e, rows + (m4 & 0xffu) * 4u);
    mp_add<PW>(v, e);
#pragma unroll
    for (int j = 0; j < PW; ++j) st.a[j] = v.w[PW - 1 - j];
}

// The blocks, last one first: the narrowest first.
template <int PW, int PLANE, int W, typename Enter, typename Leave>
__device__ __forceinline__ void ew_blocks(EwState<W>& st, const WinArgs& t, int& b, uint32_t slot, Enter&& enter, Leave&& leave) {
#pragma unroll 1
    for (const int end = PW < W ? t.blocks_of[PW + 1] : 0; b >= end; --b) {
        const uint32_t stage = enter();
        ew_block4<PW, PLANE, W>(st, stage, ew_slot_word(slot + static_cast<uint32_t>(b) * 4u));
        leave();
    }
    if constexpr (PW < W) ew_blocks<PW + 1, PLANE, W>(st, t, b, slot, enter, leave);
}

// The index of a point whose path leaves the windows, by Algorithm 2 from the cumulative tables in global memory.
__device__ __noinline__ void ew_index_global(const uint32_t* blob, int N, int K, int Wc, const uint8_t* slot, uint32_t* code) {
    const TableLayout L = table_layout(N, K, Wc);
    uint32_t c[12];
    for (int w = 0; w < Wc; ++w) c[w] = 0u;
    int behind = 0;
    for (int i = N - 1; i >= 0; --i) {
        const uint32_t p = slot[(i & ~3) + 3 - (i & 3)];
        const int y = static_cast<int>(p & 0x7fu);
        if (y == 0) continue;
        const uint32_t* u = blob + L.enc_off[0] / 4 + (static_cast<size_t>(i) * (K + 2) + behind + y + 1) * L.top_words;
        const uint32_t* x = blob + L.enc_off[(p & 0x80u) ? 0 : 1] / 4 + (static_cast<size_t>(i) * (K + 2) + behind + 1) * L.top_words;
        long long carry = 0;
        for (int w = 0; w < Wc; ++w) {
            carry += static_cast<long long>(c[w]) + __ldg(u + w) - __ldg(x + w);
            c[w] = static_cast<uint32_t>(carry);
            carry >>= 32;
        }
        behind += y;
    }
    for (int w = 0; w < Wc; ++w) code[w] = c[w];
}

// What the word behind a slot's point says.
enum : uint32_t { kEwPoint = 0, kEwZero = 1, kEwWritten = 2 };

template <int N, int W, int PLANE, bool BF16>
__global__ void __launch_bounds__((kEwWarps + 1) * 32, 1)
    encode_window_kernel(const __grid_constant__ BatchArgs a, const __grid_constant__ WinArgs t, const __grid_constant__ EwGeom g) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t full[kEwBufs], empty[kEwBufs], go;
    __shared__ int s_failed, s_gave_up;  // s_gave_up: written and read between the working warps' barriers only
    __shared__ uint8_t s_words[N];
    constexpr int E = 32, L = N / E, BLOCKS = N / 4, YS = N + 4, GW = 32 / L;
    constexpr bool LARGE = N == 64 ? W >= 7 : W >= 10;  // K may pass 127 (it is at most 255: a byte holds a coordinate's pulses)
    constexpr int P = E * (BF16 ? 2 : 4) / 16, RUN = kLaneRun<E, BF16>;
    grid_launch_dependents();
    if (threadIdx.x == 0) {
        s_failed = s_gave_up = 0;
        for (int j = 0; j < g.bufs; ++j) {
            mbarrier_init_one(&full[j]);
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(shared_addr(&empty[j])), "r"(g.warps) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(shared_addr(&go)), "r"(g.warps) : "memory");
        mbarrier_init_fence();
    }
    __syncthreads();
    grid_dependency_wait();
#ifdef PVQ_DEBUG
    debug_begin(shared_addr(smem), shared_addr(smem) + g.bufs * g.buf_bytes + (256 - PLANE) * 4, 0u, 0u, 0u, a.debug_status);
#endif
    const int warp = __shfl_sync(kFull, static_cast<int>(threadIdx.x) >> 5, 0), lane = threadIdx.x & 31;
    const int passes = blockIdx.x < a.total_tiles ? static_cast<int>((a.total_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x) : 0;
    const bool withheld = debug_withhold(a.debug_status);
    if (warp == g.warps) {  // feeds the ring; the points' input lies there while a tile is quantised
        if (lane == 0) {
            int j = 0, round = 0, n = 0;
            bool ok = true;
            for (int pass = 0; pass < passes && ok; ++pass) {
                ok = mbarrier_wait(shared_addr(&go), pass & 1, stream_polls(withheld));
                for (int b = BLOCKS - 1; b >= 0 && ok; --b) {
                    if (round > 0 && !mbarrier_wait(shared_addr(&empty[j]), (round - 1) & 1, stream_polls(withheld))) {
                        ok = false;
                        break;
                    }
                    if (!withheld) {
                        const BulkStage st{shared_addr(&full[j])};
                        const uint32_t bytes = win_rows_bytes(t.words[b], PLANE);
                        bulk_stage_expect(st, bytes);
                        bulk_stage_copy(st, smem + j * g.buf_bytes, t.data + t.block_off[b], bytes);
                        ++n;
                    }
                    if (++j == g.bufs) j = 0, ++round;
                }
            }
            if (!ok) atomicExch(&s_failed, 1);
            // what is in flight has to land before the block's memory goes away
            for (int i = n > g.bufs ? n - g.bufs : 0; i < n; ++i) mbarrier_wait(shared_addr(&full[i % g.bufs]), (i / g.bufs) & 1);
        }
        return;
    }
    const int T = g.warps * 32, K = a.K, b = a.scale_bits;
    const TableLayout TL = table_layout(N, K, W);
    for (int i = threadIdx.x; LARGE && i < N; i += T) {  // words of N(n+1,K), which no term of the position exceeds
        const uint32_t* u = a.table + TL.enc_off[0] / 4 + (static_cast<size_t>(i) * (K + 2) + K + 1) * TL.top_words;
        int words = W;
        while (i > 0 && words > 1 && __ldg(u + words - 1) == 0u) --words;
        s_words[i] = static_cast<uint8_t>(words);
    }
    mp<W> bound;
#pragma unroll
    for (int w = 0; w < W; ++w) bound.w[w] = a.table[TL.bound_off / 4 + w];
    float* s_ss = reinterpret_cast<float*>(smem + g.ss_off);
    float* s_amp = reinterpret_cast<float*>(smem + g.amp_off);
    uint32_t* s_idx = reinterpret_cast<uint32_t*>(smem + g.idx_off);
    uint8_t* my_slot = smem + g.slots_off + threadIdx.x * YS;
    uint8_t* in = smem + warp * 32 * RUN;
    const bool ls_mode = a.amp_mode == 1;
    bool failed = false;
    int mi = 0, j = 0, parity = 0;
    for (int pass = 0; pass < passes; ++pass) {
        const unsigned tile = blockIdx.x + pass * gridDim.x;
        while (mi + 1 < a.count && tile >= a.m[mi + 1].tile_begin) ++mi;
        const MatrixArgs& m = a.m[mi];
        const int G = m.G, gp = 1 << (32 - __clz(G - 1)), rpt = m.rows_per_tile;
        // row of a group: i / G as a product, exact as i and G are below 1024 (i * (per_row * G - 2^22) < 2^22)
        const unsigned per_row = (1u << 22) / static_cast<unsigned>(G) + 1u;
        auto row_of = [&](int i) { return static_cast<int>((static_cast<unsigned>(i) * per_row) >> 22); };
        const long long row0 = static_cast<long long>(tile - m.tile_begin) * rpt;
        const int nr = static_cast<int>(min(static_cast<long long>(rpt), m.rows - row0)), groups = nr * G;
        const int idx_words = m.sstride >> 2;
        for (int i = threadIdx.x; i < rpt * gp; i += T) s_ss[i] = 0.0f;
        for (int i = threadIdx.x; i < rpt * idx_words; i += T) s_idx[i] = 0u;
        ew_barrier(T);  // the tile before is done with shared memory

        // the points
        const int g_step = g.quant_warps * GW, g_first = warp < g.quant_warps ? warp * GW : groups;
        auto request = [&](int g0) {
#pragma unroll
            for (int v = 0; v < P; ++v) {
                const int q = v * 32 + lane, l = q / P, gi = g0 + l / L;  // 16-byte piece; the lane and group it belongs to
                if (gi < groups) {
                    const int r = row_of(gi);
                    const size_t off = static_cast<size_t>(row0 + r) * m.ld + static_cast<size_t>(gi - r * G) * N + (l % L) * E;
                    copy16_async(shared_addr(in) + l * RUN + (q & (P - 1)) * 16, static_cast<const uint8_t*>(m.x) + off * (BF16 ? 2 : 4) + (q & (P - 1)) * 16);
                }
            }
            copy_async_commit();
        };
        if (g_first < groups) request(g_first);
        for (int g0 = g_first; g0 < groups; g0 += g_step) {
            copy_async_wait<0>();
            __syncwarp();
            const uint8_t* mine = in + lane * RUN;
            uint32_t neg[E / 4];
            LanePoint<E, false> pt;
            float ss;
            {
                uint32_t raw[kRawWords<E, BF16>];
                float ax[E], l1;
#pragma unroll
                for (int v = 0; v < P; ++v) {
                    const uint4 q = reinterpret_cast<const uint4*>(mine)[v];
                    raw[4 * v] = q.x, raw[4 * v + 1] = q.y, raw[4 * v + 2] = q.z, raw[4 * v + 3] = q.w;
                }
#pragma unroll
                for (int i = 0; i < E / 4; ++i) neg[i] = chunk_signs4<E, BF16>(raw, i);
                group_norms<E, L, BF16>(raw, ax, l1, ss, g.minus_zero);
                if constexpr (BF16)
                    quantize_group<E, L, false>(ax, l1, K, FetchShared{reinterpret_cast<const unsigned short*>(mine)}, pt, g.minus_zero);
                else
                    quantize_group<E, L, false>(ax, l1, K, FetchSharedF32{reinterpret_cast<const float*>(mine)}, pt, g.minus_zero);
            }
            const int gi = g0 + lane / L, sub = lane % L;
            const bool ok = gi < groups, leader = ok && sub == 0;
            const int r = row_of(gi), gr = gi - r * G;
            if (leader && PVQ_DEBUG_INDEX(r * gp + gr, (g.amp_off - g.ss_off) / 4, PVQ_DEBUG_SHARED_INDEX)) s_ss[r * gp + gr] = ss;
            if (ls_mode) {
                const float ls = least_squares_amplitude<E, L, BF16, false>(pt, mine);
                if (leader) s_amp[r * gp + gr] = ls;
            }
            __syncwarp();  // the input buffer is free
            if (g0 + g_step < groups) request(g0 + g_step);
            uint32_t kind = pt.has_dir ? kEwPoint : kEwZero;
            if constexpr (LARGE) {
                uint32_t high = 0u;
#pragma unroll
                for (int i = 0; i < E / 4; ++i) high |= pt.y[i];
                const int lanes_high = group_add<L>((high & kH4) != 0u ? 1 : 0);  // (every lane takes part)
                const bool large = pt.has_dir && ok && lanes_high != 0;
                if (__any_sync(kFull, large)) {  // 128 pulses and more leave no room for a sign in the byte: its index right here
                    LanePoint<E, true> halves;
                    halves.has_dir = pt.has_dir;
#pragma unroll
                    for (int i = 0; i < E / 4; ++i) {
                        halves.y[2 * i] = __byte_perm(pt.y[i], 0u, 0x4342);
                        halves.y[2 * i + 1] = __byte_perm(pt.y[i], 0u, 0x4140);
                    }
                    const mp<W> code = lanes_index_global<E, L, W>(halves, neg, K, a.table + TL.enc_off[0] / 4, a.table + TL.enc_off[1] / 4, TL.top_words, s_words);
                    if (large) kind = kEwWritten;
                    if (large && leader) {
                        uint32_t* cp = m.codes + (static_cast<size_t>(row0 + r) * G + gr) * W;
#pragma unroll
                        for (int w = 0; w < W; ++w) cp[w] = code.w[w];
                    }
                }
            }
            if (ok && PVQ_DEBUG_INDEX(gi, T, PVQ_DEBUG_SLOT_WRITE)) {
                uint32_t* slot = reinterpret_cast<uint32_t*>(smem + g.slots_off + gi * YS) + sub * (E / 4);
#pragma unroll
                for (int i = 0; i < E / 4; ++i) slot[i] = pt.y[i] | (neg[i] & kH4);
                if (sub == L - 1) slot[E / 4] = kind;
            }
        }
        bulk_store_fence();  // the ring's buffers are written by bulk copies next
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(shared_addr(&go)) : "memory");
        ew_barrier(T);

        // the amplitudes
        const int gi = threadIdx.x, rl = row_of(gi), gr = gi - rl * G;
        const bool active = gi < groups;
        const long long row = row0 + rl;
        const float ss_row = row_energy(s_ss, gp, rl, rpt, lane);
        if (active) {
            const float ss = s_ss[rl * gp + gr];
            const float ls = ls_mode ? s_amp[rl * gp + gr] : 0.0f;
            int q = 0;
            if (b == 16) {
                q = __half_as_ushort(__float2half_rn(ls_mode ? ls : __fsqrt_rn(ss)));
            } else {
                // Step 5: q = floor(CDF(u) 2^b) as the number of bin edges <= u
                const float u = ss_row > 0.0f ? __fdiv_rn(ls_mode ? __fmul_rn(ls, ls) : ss, ss_row) : 0.0f;
                for (int step = 1 << (b - 1); step >= 1; step >>= 1)
                    if (__ldg(m.edges + q + step - 1) <= u) q += step;
            }
            if (gr == 0) m.row_norm[row] = __fsqrt_rn(ss_row);
            const unsigned bit = static_cast<unsigned>(gr) * b, sh = bit & 31u;
            const int word = rl * idx_words + static_cast<int>(bit >> 5);
            if (PVQ_DEBUG_INDEX(word + (sh + b > 32u ? 1 : 0), g.idx_words, PVQ_DEBUG_SHARED_INDEX)) {
                atomicOr(s_idx + word, static_cast<uint32_t>(q) << sh);
                if (sh + b > 32u) atomicOr(s_idx + word + 1, static_cast<uint32_t>(q) >> (32u - sh));
            }
        }

        // the indices
        const uint32_t slot = shared_addr(my_slot);
        EwState<W> st;
        st.a[0] = 0xffffffffu << t.up[BLOCKS - 1];  // -q = -1 at the end of the vector
#pragma unroll
        for (int i = 1; i <= W; ++i) st.a[i] = 0u;
        st.delta = 0u;
        st.behind = 0u;
        st.flag = 0u;
        int blk = BLOCKS - 1;
        ew_blocks<1, PLANE, W>(
            st, t, blk, slot,
            [&]() {
                // (a lane that gives up goes on with what is there, inside the buffer, and writes nothing)
                if (!failed && !mbarrier_wait(shared_addr(&full[j]), parity, stream_polls(withheld))) failed = true;
                return shared_addr(smem) + j * g.buf_bytes;
            },
            [&]() {
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(shared_addr(&empty[j])) : "memory");
                if (++j == g.bufs) j = 0, parity ^= 1;
            });
        if (active && !failed && PVQ_DEBUG_INDEX(row, m.rows, PVQ_DEBUG_GLOBAL_STORE)) {
            const uint32_t kind = reinterpret_cast<const uint32_t*>(my_slot)[N / 4];
            uint32_t* cp = m.codes + (static_cast<size_t>(row) * G + gr) * W;
            if (kind == kEwPoint && (st.flag & kH4) != 0u) {
                ew_index_global(a.table, N, K, W, my_slot, cp);
            } else if (kind != kEwWritten) {
                mp<W> code;  // -q, back from the top of the words; (K, 0, ..., 0) has q = 2
                code.w[W - 1] = __funnelshift_r(st.a[0], 0xffffffffu, st.delta);
#pragma unroll
                for (int i = 1; i < W; ++i) code.w[W - 1 - i] = __funnelshift_r(st.a[i], st.a[i - 1], st.delta);
                if (kind == kEwZero) {
#pragma unroll
                    for (int w = 0; w < W; ++w) code.w[w] = w == 0 ? 0xfffffffeu : 0xffffffffu;
                }
                mp_add<W>(code, bound);
#pragma unroll
                for (int w = 0; w < W; ++w) cp[w] = code.w[w];
            }
        }
        if (failed) s_gave_up = 1;
        ew_barrier(T);  // the amplitude indices are complete
        for (int i = threadIdx.x; i < nr * idx_words; i += T) {
            const int r = i / idx_words;
            reinterpret_cast<uint32_t*>(m.scale_idx + static_cast<size_t>(row0 + r) * m.sstride)[i - r * idx_words] = s_idx[i];
        }
        ew_barrier(T);
        if (s_gave_up != 0) break;  // (a copy that comes late would land in the next tile's input)
    }
    if (a.status && (failed || s_failed != 0)) atomicOr(a.status, PVQ_STATUS_STAGING_TIMEOUT);
}

template <int N, int W, int PLANE, bool BF16>
int launch_ew_t(BatchArgs& a, const WinTables& t, cudaStream_t stream) {
    constexpr uint32_t RUN = kLaneRun<32, BF16>;
    DeviceInfo di;
    int st = device_info(&di);
    if (st != PVQ_OK) return st;
    const uint32_t limit = static_cast<uint32_t>(di.smem_max);
    EwGeom best;
    std::memset(&best, 0, sizeof best);
    double best_cost = -1.0;
    size_t best_smem = 0;
    for (int w = kEwWarps; w >= 2; --w) {
        const int T = w * 32;
        EwGeom g;
        std::memset(&g, 0, sizeof g);
        long long tiles = 0;
        uint32_t ss = 4, idx = 1;
        bool fits = true;
        for (int i = 0; i < a.count && fits; ++i) {
            const MatrixArgs& m = a.m[i];
            fits = m.G <= T;
            if (!fits) break;
            const int rpt = static_cast<int>(std::min<long long>(T / m.G, m.rows));
            uint32_t gp = 1;
            while (gp < static_cast<uint32_t>(m.G)) gp <<= 1;
            tiles += (m.rows + rpt - 1) / rpt;
            ss = std::max(ss, rpt * gp);
            idx = std::max(idx, static_cast<uint32_t>(rpt * (m.sstride / 4)));
        }
        if (!fits || tiles > 0x7fffffffLL) continue;
        g.warps = w;
        g.idx_words = static_cast<int>(idx);
        g.buf_bytes = (t.max_rows + 127u) & ~127u;
        // (an index outside its window reads as far as 256 entries from the start of a plane: that much behind the last
        // buffer is not used otherwise; 256 bytes for the alignment of what follows)
        constexpr uint32_t behind = (256u - PLANE) * 4u;
        const uint32_t slots = static_cast<uint32_t>(T) * (N + 4), rest = (2u * ss + idx) * 4u + behind + 256u;
        if (slots + rest + 2u * g.buf_bytes > limit) continue;
        g.bufs = static_cast<int>(std::min<uint32_t>(kEwBufs, (limit - slots - rest) / g.buf_bytes));
        uint32_t ring = g.bufs * g.buf_bytes + behind;
        ring = std::max(ring, std::min(w * 32u * RUN, (limit - slots - rest) & ~127u));
        g.quant_warps = static_cast<int>(std::min<uint32_t>(w, ring / (32u * RUN)));
        g.slots_off = (ring + 127u) & ~127u;
        g.ss_off = (g.slots_off + slots + 127u) & ~127u;
        g.amp_off = g.ss_off + ss * 4u;
        g.idx_off = g.amp_off + ss * 4u;
        const size_t smem = g.idx_off + idx * 4u;
        if (smem > limit || g.quant_warps < 1) continue;
        // a round costs its warps' work and something to fill and drain
        const double cost = static_cast<double>((tiles + di.sms - 1) / di.sms) * (w + 6);
        if (best_cost < 0.0 || cost < best_cost) best_cost = cost, best = g, best_smem = smem;
    }
    if (best_cost < 0.0) return PVQ_ERR_UNSUPPORTED;
    best.minus_zero = -0.0f;
    unsigned tiles = 0;
    for (int i = 0; i < a.count; ++i) {
        MatrixArgs& m = a.m[i];
        m.rows_per_tile = static_cast<int>(std::min<long long>(best.warps * 32 / m.G, m.rows));
        m.tile_begin = tiles;
        tiles += static_cast<unsigned>((m.rows + m.rows_per_tile - 1) / m.rows_per_tile);
    }
    a.total_tiles = tiles;
    auto kern = encode_window_kernel<N, W, PLANE, BF16>;
    const int threads = (best.warps + 1) * 32;
    int per_sm = 0;
    if ((st = prepare_kernel(reinterpret_cast<const void*>(kern), threads, best_smem, &per_sm)) != PVQ_OK) return st;
    if (per_sm < 1) return PVQ_ERR_UNSUPPORTED;
    return launch_hot(kern, std::min<unsigned>(tiles, static_cast<unsigned>(di.sms)), threads, best_smem, stream, a, t.args, best);
}

template <int N, int W>
int launch_ew(BatchArgs& a, int dtype, const WinTables& t, cudaStream_t s) {
    const bool bf16 = dtype == PVQ_DTYPE_BF16;
    if constexpr (N == 64) {
        if (t.plane == 96) return bf16 ? launch_ew_t<N, W, 96, true>(a, t, s) : launch_ew_t<N, W, 96, false>(a, t, s);
        return bf16 ? launch_ew_t<N, W, 192, true>(a, t, s) : launch_ew_t<N, W, 192, false>(a, t, s);
    }
    return bf16 ? launch_ew_t<N, W, N == 64 ? 192 : 160, true>(a, t, s) : launch_ew_t<N, W, N == 64 ? 192 : 160, false>(a, t, s);
}

}  // namespace

int launch_encode_window(const BatchArgs& args, int dtype, int N, int W, cudaStream_t stream) {
    static_assert(!has_window_tables(64, 8, 256) && !has_window_tables(128, 12, 256), "a coordinate's pulses and the sums of four have a byte each");
    if (N == 256 || !has_window_tables(N, W, args.K)) return PVQ_ERR_UNSUPPORTED;
    const auto t = window_tables(N, args.K, stream);
    if (!t || t->args.words[N / 4 - 1] != 1) return PVQ_ERR_UNSUPPORTED;
    BatchArgs a = args;
    switch (N * 16 + W) {
        case 64 * 16 + 5: return launch_ew<64, 5>(a, dtype, *t, stream);
        case 64 * 16 + 6: return launch_ew<64, 6>(a, dtype, *t, stream);
        case 64 * 16 + 7: return launch_ew<64, 7>(a, dtype, *t, stream);
        case 64 * 16 + 8: return launch_ew<64, 8>(a, dtype, *t, stream);
        case 128 * 16 + 9: return launch_ew<128, 9>(a, dtype, *t, stream);
        case 128 * 16 + 10: return launch_ew<128, 10>(a, dtype, *t, stream);
        case 128 * 16 + 11: return launch_ew<128, 11>(a, dtype, *t, stream);
        case 128 * 16 + 12: return launch_ew<128, 12>(a, dtype, *t, stream);
        default: break;
    }
    return PVQ_ERR_UNSUPPORTED;
}

}  // namespace pvq
