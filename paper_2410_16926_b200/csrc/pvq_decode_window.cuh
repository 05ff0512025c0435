// Decode kernel for wide codes: group size 64 with codes of 5 to 8 words, 128 with 9 to 12, 256 with 24.  One thread per group, one
// threshold search per position in windowed tables (pvq_window.cuh), N steps a group where the walk takes
// N + K (160 at N = 64, 192 bits; 315 at N = 128, 384 bits).
//
// What bounds it: shared-memory wavefronts and issue slots.  A position reads a row's record, one bucket and, word plane
// by word plane, the entry of E, as wide as the numbers still are (4 words on average at N = 64, 192 bits): the
// threads of a warp read entries a few apart, mostly different banks.  The searches of a warp are independent
// of each other, so the latency of a position (two dependent reads) is covered by 8 warps per scheduler.
//
// The tables stay in shared memory where they fit beside the output slots (N = 64, 192 bits: 150 KB).  Otherwise
// (N = 128, 384 bits: 760 KB; N = 256: 2.4 MB) they are streamed from L2 through a ring of buffers, block of rows
// after block of rows, all warps of the thread block following the stream; an additional warp feeds it.
//
// Measured, with the walk (pvq_walk.cuh, pvq_big_impl.cuh) and now: 8192 x 28672, N = 64, 192 bits, 774 -> 356 us (77% of the
// issue slots, 88% of the shared-memory wavefronts a cycle); 4096 x 4096, N = 128, 384 bits, 190 -> 47.6 us; N = 256, 768
// bits, 601 -> 155 us.
// (Group size 256 has a translation unit of its own: the functions that are not inlined take the registers of the
// most generous kernel that calls them, and spill in the others.)
#pragma once
#include <algorithm>
#include <cmath>
#include <cstring>

#include <cuda_fp16.h>

#include "pvq_walk.cuh"
#include "pvq_window.cuh"

namespace pvq {

namespace {

struct WinGeom {
    uint32_t slots_off;  // of the output slots in shared memory
    uint32_t buf_bytes;  // streamed: bytes of a buffer
    int bufs;            // streamed: number of buffers
    int warps;           // that decode
};

// A word of the tables in shared memory; win_slot_word: of the output slots.
template <int OFF = 0>
__device__ __forceinline__ uint32_t win_slot_word(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(OFF));
    return v;
}
template <int OFF = 0>
__device__ __forceinline__ uint32_t win_load(uint32_t addr) {
#ifdef PVQ_DEBUG
    if (!debug_table_ok(addr + OFF, 4u)) return 0u;
#endif
    return win_slot_word<OFF>(addr);
}
template <int PW, int PLANE, int FROM, int W = 0>
__device__ __forceinline__ void win_entry(mp<PW>& e, uint32_t addr) {
    if constexpr (W < PW) {
        e.w[W] = win_load<(FROM + W) * PLANE * 4>(addr);
        win_entry<PW, PLANE, FROM, W + 1>(e, addr);
    }
}

// A row's record (WinRow): x base, y last, z shift, w buckets.
__device__ __forceinline__ uint4 win_record(uint32_t addr) {
    uint4 v;
#ifdef PVQ_DEBUG
    if ((addr & 15u) != 0u || !debug_table_ok(addr, 16u)) return make_uint4(0u, 0u, 0u, 0u);
#endif
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}

// Two neighbouring words of a block's head.
template <int OFF>
__device__ __forceinline__ uint2 win_load2(uint32_t addr) {
    uint2 v;
#ifdef PVQ_DEBUG
    if (!debug_table_ok(addr + OFF, 8u)) return make_uint2(0u, 0u);
#endif
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2+%3];" : "=r"(v.x), "=r"(v.y) : "r"(addr), "n"(OFF));
    return v;
}

// The key of q: its KW leading words as an fp32, every step rounded towards zero.
template <int PW, int KW>
__device__ __forceinline__ uint32_t win_key(const mp<PW>& v) {
    float x = __uint2float_rz(v.w[PW - 1]);
    if constexpr (PW > 1) x = __fmaf_rz(x, 4294967296.0f, __uint2float_rz(v.w[PW - 2]));
    if constexpr (PW > 2 && KW > 2) x = __fmaf_rz(x, 4294967296.0f, __uint2float_rz(v.w[PW - 3]));
    return __float_as_uint(x);
}

// Marks pulses left that an index outside the window might pass for: the local index 255 says 127 left, and with 127 or more
// before the position that is no growth.  (A bit that the packed test looks at, above any number of pulses.)
constexpr int kWinFar = 0x800000;

// What the repeated search of a block works on: q (`over`: the word above the block's, for paths above the windows), the
// local pulses left, and what it hands back.
template <int PW>
struct WinExact {
    mp<PW> v;
    uint32_t over;
    int h;
    uint32_t y4, ssy;
    bool lost;
};

// Word w of an entry of one of the blob's tables: zero from Wc on.
__device__ __forceinline__ uint32_t win_count_word(const uint32_t* t, int w, int Wc) { return w < Wc ? __ldg(t + w) : 0u; }

// t < q ?  (t: an entry of Wc words; q: PW + 1 words)
template <int PW>
__device__ __forceinline__ bool win_less(const uint32_t* t, int Wc, const uint32_t (&q)[PW + 1]) {
    long long c = 0;
#pragma unroll
    for (int w = 0; w <= PW; ++w) c = (c + static_cast<long long>(win_count_word(t, w, Wc)) - q[w]) >> 32;
    uint32_t rest = 0u;
    for (int w = PW + 1; w < Wc; ++w) rest |= __ldg(t + w);
    return c < 0 && rest == 0u;
}

// The four positions of block b once more, for the paths that the fast pass cannot decide: key bits the same as a
// threshold's (compared in full), positions outside the window (searched in the whole row, in global memory).
template <int PW, int PLANE, int KW>
__device__ __noinline__ void win_exact4(WinExact<PW>& st, uint32_t acc, uint32_t stage, const WinArgs& t, int b, const uint32_t* blob, int N,
                                        int K, int Wc) {
#pragma unroll 1
    for (int s = 3; s >= 0; --s) {  // back to where the block began
        mp<PW> e, d;
        win_entry<PW, PLANE, 0>(e, stage + kWinHead + static_cast<uint32_t>(s) * (PW * PLANE * 4) + ((acc >> (8 * s)) & 0xffu) * 4u);
        mp_sub_borrow<PW>(d, st.v, e);
        st.v = d;
    }
    const TableLayout L = table_layout(N, K, Wc);
    const int up = t.up[b];
    int k = (b > 0 ? t.klo[4 * b - 1] : K) + (st.h >= kWinFar ? st.h - kWinFar : st.h);  // pulses left before the position
    st.y4 = 0u;
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
        const int i = 4 * b + s, n = N - 1 - i;
        const uint4 r = win_record(stage + 16u * static_cast<uint32_t>(s));
        const uint32_t key = min(win_key<PW, KW>(st.v) - r.x, r.y);
        const uint32_t sum = key + win_load(stage + r.w + ((key >> r.z) << 2));
        int left;
        bool odd;
        if (st.over == 0u && key < r.y) {
            uint32_t m = sum >> 24;
            if ((sum | 0xff000000u) == 0xffffffffu) {
                const uint32_t* thr = reinterpret_cast<const uint32_t*>(t.thr + t.thr_off[b]) + s * PW * PLANE + m;
                mp<PW> th, d;
#pragma unroll
                for (int w = 0; w < PW; ++w) th.w[w] = __ldg(thr + w * PLANE);
                m += mp_sub_borrow<PW>(d, th, st.v) ? 1u : 0u;
            }
            mp<PW> e;
            win_entry<PW, PLANE, 0>(e, stage + kWinHead + static_cast<uint32_t>(s) * (PW * PLANE * 4) + m * 4u);
            mp_add<PW>(st.v, e);
            left = t.klo[i] + static_cast<int>(m >> 1);
            odd = (m & 1u) != 0u;
        } else {
            uint32_t q[PW + 1];
#pragma unroll
            for (int w = 0; w <= PW; ++w) {
                const uint32_t lo = w < PW ? st.v.w[w < PW ? w : 0] : st.over;
                const uint32_t hi = w + 1 < PW ? st.v.w[w + 1 < PW ? w + 1 : 0] : (w + 1 == PW ? st.over : 0u);
                q[w] = __funnelshift_r(lo, hi, up);
            }
            const uint32_t* row_u = blob + L.enc_off[0] / 4 + static_cast<size_t>(i) * (K + 2) * L.top_words;
            const uint32_t* row_v = blob + L.enc_off[1] / 4 + static_cast<size_t>(i) * (K + 2) * L.top_words;
            left = max(min(k, K), 0);
            // 2 V(n, left - 1) < q <= 2 V(n, left)
            while (left > 0 && !win_less<PW>(row_v + static_cast<size_t>(left) * L.top_words, Wc, q)) --left;
            const uint32_t* u = row_u + static_cast<size_t>(left + 1) * L.top_words;
            odd = win_less<PW>(u, Wc, q);
            if (odd) u = row_v + static_cast<size_t>(left + 1) * L.top_words;
            // q -= T - N(n, left)
            const uint32_t* c0 = blob + (static_cast<size_t>(n) * (K + 1) + left) * Wc;
            long long c = 0;
#pragma unroll
            for (int w = 0; w <= PW; ++w) {
                c += static_cast<long long>(q[w]) - win_count_word(u, w, Wc) + win_count_word(c0, w, Wc);
                q[w] = static_cast<uint32_t>(c);
                c >>= 32;
            }
            st.over = __funnelshift_l(q[PW - 1], q[PW], up);
            st.lost = st.lost || (up > 0 && (q[PW] >> (32 - up)) != 0u);
#pragma unroll
            for (int w = PW - 1; w >= 0; --w) st.v.w[w] = __funnelshift_l(w > 0 ? q[w > 0 ? w - 1 : 0] : 0u, q[w], up);
        }
        const int mag = k - left;
        st.lost = st.lost || mag < 0 || mag > 127;
        st.y4 |= (static_cast<uint32_t>(128 + (odd ? mag : -mag)) & 0xffu) << (8 * s);
        st.ssy += static_cast<uint32_t>(mag * mag);
        k = left;
    }
    st.h = k - t.klo[4 * b + 3];
    if (4 * b + 4 < N && k - t.klo[4 * b + 4] >= 127) st.h += kWinFar;  // (only a repeated search can leave so many)
    if (st.over >= 0x10000u) st.lost = true;  // the next block's shift (16 bits at most) would push bits out
    if (st.lost) st.over = 0u, st.h = 0;
}

// State of one thread's search.  a[0] is the leading word; the words a block does not work on are zero.
template <int W>
struct WinState {
    uint32_t a[W + 1];
    uint32_t over;  // the word above a[0]: zero but for paths above the windows
    int h;          // pulses left after the position before, minus its klo (kWinFar added where they are too many)
    uint32_t ssy;   // sum of y^2
    bool lost;      // some |y| has no byte, or q no room: the group is walked
};

// `sum`: all ones but for the top byte where the key bits are the same as the threshold's.
template <int PW, int PLANE, int KW, int S>
__device__ __forceinline__ void win_position(mp<PW>& v, uint32_t& acc, uint32_t& sum, uint32_t stage) {
    const uint4 r = win_record(stage + 16u * S);
    const uint32_t key = min(win_key<PW, KW>(v) - r.x, r.y);
    sum = key + win_load(stage + r.w + ((key >> r.z) << 2));
    acc = __byte_perm(acc, sum, 0x7321);
    mp<PW> e;
    win_entry<PW, PLANE, S * PW>(e, stage + kWinHead + ((sum >> 24) << 2));
    mp_add<PW>(v, e);
}

template <int N, int PW, int PLANE, int KW, int W>
__device__ __forceinline__ void win_block4(WinState<W>& st, uint32_t stage, const BatchArgs& a, const WinArgs& t, int b, uint32_t y) {
    mp<PW> v;
    static_assert(kWinDelta == kWinDlo4 + 4, "one read");
    const uint2 head = win_load2<kWinDlo4>(stage);
    {
        const uint32_t delta = head.y;
        st.over = __funnelshift_l(st.a[0], st.over, delta);
#pragma unroll
        for (int j = 0; j < PW; ++j) v.w[PW - 1 - j] = __funnelshift_l(st.a[j + 1], st.a[j], delta);
        st.a[PW] = 0u;
    }
    uint32_t acc = 0u, sum;
    win_position<PW, PLANE, KW, 0>(v, acc, sum, stage);
    win_position<PW, PLANE, KW, 1>(v, acc, sum, stage);
    win_position<PW, PLANE, KW, 2>(v, acc, sum, stage);
    win_position<PW, PLANE, KW, 3>(v, acc, sum, stage);
    // |y|: pulses left before the position minus those left after it, a byte each: one sum, whose bytes do not
    // touch each other while all of them are 0..127 (else some bit 7 shows, unless the position before was out of the
    // window too: in the block, its own bit 7 shows; in the block before, h shows it); y > 0 where the index is odd
    const uint32_t after = (acc >> 1) & 0x7f7f7f7fu;
    const uint32_t mag = (after << 8) + head.x - after + static_cast<uint32_t>(st.h);
    const uint32_t odd = acc & 0x01010101u, pos = (odd << 8) - odd;
    uint32_t y4 = (mag ^ ~pos) + 0x80808081u + pos;  // 128 + |y|; else 255 - |y| + 128 - 255: no byte of the sum leaves 1 .. 255
    // Key bits the same as a threshold's, and q above it all the same: the index is one short, and q' = T_(n-1)[2k'] + d with d =
    // q - T_n[m] is too large for the k' pulses left.  The next position's index is then 2k' + 1 or more, which no q of a valid code
    // has: y = 0 with an odd index, or pulses that grow.  At the last position, whose next is in another block, the bits are
    // looked at.
    const uint32_t odd_zero = ~((mag | 0x80808080u) - odd);
    if (__any_sync(kFull, (sum | 0xff000000u) == 0xffffffffu || (((mag | odd_zero | static_cast<uint32_t>(st.h)) & 0x80808080u) | st.over) != 0u)) {
        WinExact<PW> x;
        x.v = v;
        x.over = st.over, x.h = st.h, x.ssy = st.ssy, x.lost = st.lost;
        win_exact4<PW, PLANE, KW>(x, acc, stage, t, b, a.table, N, a.K, W);
        v = x.v;
        st.over = x.over, st.h = x.h, st.ssy = x.ssy, st.lost = x.lost;
        y4 = x.y4;
    } else {
        st.h = static_cast<int>(after >> 24);
        st.ssy = __dp4a(mag, mag, st.ssy);
    }
#ifdef PVQ_DEBUG
    if (debug_slot_ok(y, 4u))
#endif
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(y), "r"(y4) : "memory");
#pragma unroll
    for (int j = 0; j < PW; ++j) st.a[j] = v.w[PW - 1 - j];
}

constexpr uint32_t kNoStage = 0xffffffffu;  // no block of tables has arrived: nothing is read

// All blocks from the one that PW words are first enough for: the widest first.
template <bool STREAM, int N, int PW, int PLANE, int KW, int W, typename Enter, typename Leave>
__device__ __forceinline__ void win_blocks(WinState<W>& st, const BatchArgs& a, const WinArgs& t, int& b, uint32_t y, Enter&& enter, Leave&& leave) {
#pragma unroll 1
    for (; b < t.blocks_of[PW]; ++b) {
        const uint32_t stage = enter(b), yb = y + static_cast<uint32_t>(b) * 4u;
        if (!STREAM || stage != kNoStage) win_block4<N, PW, PLANE, KW, W>(st, stage, a, t, b, yb);
        leave(b);
    }
    if constexpr (PW > 1) win_blocks<STREAM, N, PW - 1, PLANE, KW, W>(st, a, t, b, y, enter, leave);
}

// Algorithm 3 step by step for the group at hand, from the count table in global memory: for points with a |y| of 128 or
// more, or with a path far above the windows.  Its point goes to the thread's slot if all |y| < 128; else its values are
// written to `out` right away (the walk done twice), and the result is true.
template <int W>
__device__ __noinline__ bool win_walk(const uint32_t* count, int N, int K, const uint32_t* code, uint8_t* slot, float amp,
                                      __nv_bfloat16* out, uint32_t* ssy_out) {
    float sc = 0.0f;
    bool fits = true;
    uint32_t ssy = 0u;
    for (int pass = 0; pass < 2; ++pass) {
        uint32_t r[W];
        for (int w = 0; w < W; ++w) r[w] = code[w];
        int k = K;
        for (int i = 0; i < N; ++i) {
            int y = 0;
            for (;;) {
                const uint32_t* t = count + (static_cast<size_t>(N - 1 - i) * (K + 1) + k) * W;
                // r against t, and against 2t
                int top = W - 1;
                while (top > 0 && r[top] == __ldg(t + top)) --top;
                if (r[top] < __ldg(t + top)) break;  // nothing more here, and y >= 0
                long long c = 0;
                uint32_t d[W];
                for (int w = 0; w < W; ++w) {
                    c += static_cast<long long>(r[w]) - __ldg(t + w);
                    d[w] = static_cast<uint32_t>(c);
                    c >>= 32;
                }
                if (y > 0) {
                    int t2 = W - 1;
                    while (t2 > 0 && d[t2] == __ldg(t + t2)) --t2;
                    const bool more = d[t2] >= __ldg(t + t2);
                    if (more) {
                        c = 0;
                        for (int w = 0; w < W; ++w) {
                            c += static_cast<long long>(d[w]) - __ldg(t + w);
                            r[w] = static_cast<uint32_t>(c);
                            c >>= 32;
                        }
                    } else {
                        for (int w = 0; w < W; ++w) r[w] = d[w];
                        y = -y;
                        break;
                    }
                } else {
                    for (int w = 0; w < W; ++w) r[w] = d[w];
                }
                if (k == 0) break;  // (no valid code gets here)
                ++y;
                --k;
            }
            if (pass == 0) {
                ssy += static_cast<uint32_t>(y * y);
                fits = fits && y < 128 && y > -128;
                slot[i] = static_cast<uint8_t>(y + 128);
            } else {
                out[i] = __float2bfloat16_rn(__fmul_rn(static_cast<float>(y), sc));
            }
        }
        if (fits) break;
        sc = __fdiv_rn(amp, __fsqrt_rn(static_cast<float>(static_cast<int>(ssy))));
    }
    *ssy_out = ssy;
    return !fits;
}

// One tile: the 32 groups of a warp, from the code to the stored values.  enter(b) gives the shared address of block b,
// or, streamed, kNoStage, to all lanes alike; from then on `failed` is set, and the tile is not written.
template <bool STREAM, int N, int W, int PLANE, typename Enter, typename Leave>
__device__ __forceinline__ void win_tile(const BatchArgs& a, const WinArgs& t, const mp<W>& bound, unsigned tile, int& mi, uint32_t slots,
                                         uint32_t y, uint8_t* slot, bool& bad, const bool& failed, Enter&& enter, Leave&& leave) {
    constexpr int YS = N + 4;
    const int lane = threadIdx.x & 31;
    const unsigned b = a.scale_bits;
    const bool any = tile < a.total_tiles;
    while (mi + 1 < a.count && tile >= a.m[mi + 1].tile_begin) ++mi;
    const MatrixArgs& m = a.m[mi];
    const unsigned G = static_cast<unsigned>(m.G);
    const unsigned ngroups = static_cast<unsigned>(m.rows) * G;
    const unsigned gi = (tile - m.tile_begin) * 32u + lane;
    const bool active = any && gi < ngroups;
    const unsigned row = group_row(m, gi), g = gi - row * G;
    mp<W> c;
    mp_zero(c);
    unsigned sbits = 0u;
    float rnorm = 0.0f;
    bool valid = false;
    const uint32_t* code = m.codes + static_cast<size_t>(gi) * W;
    if (active) {
        c = mp_load<W>(code);
        const uint8_t* srow = m.scale_idx + static_cast<size_t>(row) * m.sstride;
        const unsigned bit = g * b;
        sbits = srow[bit >> 3];
        if ((bit & 7u) + b > 8u) sbits |= static_cast<unsigned>(srow[(bit >> 3) + 1]) << 8;
        if (b != 16u) rnorm = m.row_norm[row];
        mp<W> tmp;
        valid = mp_sub_borrow<W>(tmp, c, bound);
        bad = bad || !valid;
    }
    WinState<W> st;
    bool alone = false;  // the point (K, 0, ..., 0), which a group of zeros has: q = 2
    if (valid) {
        mp<W> q;
        mp_sub_borrow<W>(q, bound, c);  // 1 <= q <= N(N,K)
        uint32_t rest = q.w[0] ^ 2u;
#pragma unroll
        for (int w = 1; w < W; ++w) rest |= q.w[w];
        alone = rest == 0u;
        // (the first block's delta brings it to the top of the words)
#pragma unroll
        for (int j = 0; j < W; ++j) st.a[j] = q.w[W - 1 - j];
    }
    if (!valid || alone) {  // not searched: a path that costs nothing extra in its place
#pragma unroll
        for (int j = 0; j < W; ++j) st.a[j] = t.typical[W - 1 - j];
    }
    st.a[W] = 0u;
    st.over = 0u;
    st.h = 0;
    st.ssy = 0u;
    st.lost = false;
    int blk = 0;
    win_blocks<STREAM, N, W, PLANE, win_key_words(N), W>(st, a, t, blk, y, enter, leave);
    if (STREAM && failed) return;

    float amp = 0.0f;
    __nv_bfloat16* out = static_cast<__nv_bfloat16*>(m.out) + static_cast<size_t>(row) * m.ld_out + static_cast<size_t>(g) * N;
    bool done = !active;
    if (valid) {
        const unsigned qi = (sbits >> ((g * b) & 7u)) & ((1u << b) - 1u);
        // 16 bits: the amplitude itself as binary16; else the quantile level times the row norm
        amp = b == 16u ? __half2float(__ushort_as_half(static_cast<unsigned short>(qi))) : __fmul_rn(rnorm, m.levels[qi]);
    }
    const bool zeros = active && (!valid || (alone && amp == 0.0f));
    const bool single = valid && !zeros && alone && a.K < 128;
    if (zeros || single) {
#pragma unroll 1
        for (int i = 0; i < N / 4; ++i) reinterpret_cast<uint32_t*>(slot)[i] = 0x80808080u;
        if (single) slot[0] = static_cast<uint8_t>(128 + a.K);
        st.ssy = single ? static_cast<uint32_t>(a.K * a.K) : 1u;
    } else if (valid && (st.lost || alone)) {
        uint32_t ssy;
        done = win_walk<W>(a.table, N, a.K, code, slot, amp, out, &ssy);
        st.ssy = ssy;
    }
    const float sc = zeros ? 0.0f : __fdiv_rn(amp, __fsqrt_rn(static_cast<float>(static_cast<int>(st.ssy))));
    // The warp writes the groups one after the other, 16 bytes a lane: whole lines.
    done = done || !PVQ_DEBUG_INDEX(row, m.rows, PVQ_DEBUG_GLOBAL_STORE) ||
           !PVQ_DEBUG_INDEX(static_cast<long long>(g + 1) * N - 1, m.cols, PVQ_DEBUG_GLOBAL_STORE);
    const uint32_t at = done ? 0xffffffffu : static_cast<uint32_t>((static_cast<size_t>(row) * m.ld_out + static_cast<size_t>(g) * N) >> 3);
    uint4* base = static_cast<uint4*>(m.out);
    __syncwarp();
    constexpr int PIECES = N / 8;  // lanes that share a group
    const uint32_t sub = static_cast<uint32_t>(lane) % PIECES;
    uint32_t src = slots + static_cast<uint32_t>(lane / PIECES) * YS + sub * 8u;
#pragma unroll 2
    for (int from = lane / PIECES; from < 32; from += 32 / PIECES, src += 32 / PIECES * YS) {
        const float s = __shfl_sync(kFull, sc, from);
        const uint32_t dst = __shfl_sync(kFull, at, from);
        const uint32_t lo = win_slot_word(src), hi = win_slot_word<4>(src);
        const uint4 v = scale_bytes8(lo, hi, s);
        if (dst != 0xffffffffu) base[dst + sub] = v;
    }
    __syncwarp();  // the slots are free
}

template <int W>
__device__ __forceinline__ mp<W> win_bound(const BatchArgs& a, int N) {
    const TableLayout L = table_layout(N, a.K, W);
    mp<W> bound;
#pragma unroll
    for (int w = 0; w < W; ++w) bound.w[w] = a.table[L.bound_off / 4 + w];
    return bound;
}

template <int N, int W, int PLANE>
__global__ void __launch_bounds__(1024, 1)
    decode_window_kernel(const __grid_constant__ BatchArgs a, const __grid_constant__ WinArgs t, const __grid_constant__ WinGeom g) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t stage_bar;
    grid_launch_dependents();
    const BulkStage stage = bulk_stage_begin(&stage_bar);
    grid_dependency_wait();
    if (threadIdx.x == 0) {
        const uint32_t bytes = t.block_off[N / 4];
        bulk_stage_expect(stage, bytes);
        bulk_stage_copy(stage, smem, t.data, bytes);
    }
    const mp<W> bound = win_bound<W>(a, N);
    if (!__syncthreads_and(bulk_stage_wait(stage))) {  // the tables never arrived: report and leave, all threads
        if (a.status && threadIdx.x == 0) atomicOr(a.status, PVQ_STATUS_STAGING_TIMEOUT);
        return;
    }
    const uint32_t base = shared_addr(smem);
    uint8_t* slot = smem + g.slots_off + threadIdx.x * (N + 4);
    const uint32_t y = shared_addr(slot), slots = y - (threadIdx.x & 31) * (N + 4);
#ifdef PVQ_DEBUG
    debug_begin(base, base + t.block_off[N / 4], shared_addr(smem) + g.slots_off, N + 4, N, a.debug_status);
#endif
    const unsigned warp = __shfl_sync(kFull, threadIdx.x >> 5, 0), total = gridDim.x * g.warps;
    bool bad = false;
    int mi = 0;
    for (unsigned tile = warp * gridDim.x + blockIdx.x; tile < a.total_tiles; tile += total)
        win_tile<false, N, W, PLANE>(a, t, bound, tile, mi, slots, y, slot, bad, false, [&](int b) { return base + t.block_off[b]; }, [](int) {});
    if (bad && a.status) atomicOr(a.status, PVQ_STATUS_INVALID_CODE);
}

constexpr int kWinBufs = 8;  // at most

__device__ __forceinline__ void win_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Streamed tables.  Buffer j holds the blocks n with n % bufs == j, n counted over all passes; full[j] completes when
// a block has arrived, empty[j] when every decoding warp is through with it.  A wait that runs out sets the
// status bit; the warp then goes through the remaining motions without waiting, reading or writing, and leaves (no copy
// is issued into a buffer that was not given back, and the feeding warp waits for what it has issued).
template <int N, int W, int PLANE>
__global__ void __launch_bounds__(N == 256 ? 384 : 928, 1)
    decode_window_stream_kernel(const __grid_constant__ BatchArgs a, const __grid_constant__ WinArgs t, const __grid_constant__ WinGeom g) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t full[kWinBufs], empty[kWinBufs];
    __shared__ int s_failed;
    constexpr int BLOCKS = N / 4;
    grid_launch_dependents();
    if (threadIdx.x == 0) {
        s_failed = 0;
        for (int j = 0; j < g.bufs; ++j) {
            mbarrier_init_one(&full[j]);
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(shared_addr(&empty[j])), "r"(g.warps) : "memory");
        }
        mbarrier_init_fence();
    }
    __syncthreads();
    grid_dependency_wait();
#ifdef PVQ_DEBUG
    debug_begin(shared_addr(smem), shared_addr(smem) + g.bufs * g.buf_bytes, shared_addr(smem) + g.slots_off, N + 4, N, a.debug_status);
#endif
    const unsigned warp = __shfl_sync(kFull, threadIdx.x >> 5, 0), step = gridDim.x * g.warps, first = blockIdx.x;
    const bool withheld = debug_withhold(a.debug_status);
    const int passes = first < a.total_tiles ? static_cast<int>((a.total_tiles - first + step - 1) / step) : 0;
    if (warp == static_cast<unsigned>(g.warps)) {  // feeds the ring
        if ((threadIdx.x & 31) == 0) {
            const int n_all = passes * BLOCKS;
            int j = 0, round = 0, issued = 0;
            for (int n = 0, b = 0; n < n_all; ++n) {
                if (round > 0 && !mbarrier_wait(shared_addr(&empty[j]), (round - 1) & 1, stream_polls(withheld))) {
                    atomicExch(&s_failed, 1);
                    break;
                }
                if (!withheld) {
                    const BulkStage st{shared_addr(&full[j])};
                    const uint32_t bytes = t.block_off[b + 1] - t.block_off[b];
                    bulk_stage_expect(st, bytes);
                    bulk_stage_copy(st, smem + j * g.buf_bytes, t.data + t.block_off[b], bytes);
                    issued = n + 1;
                }
                if (++b == BLOCKS) b = 0;
                if (++j == g.bufs) j = 0, ++round;
            }
            // what is in flight has to land before the block's memory goes away
            for (int n = issued > g.bufs ? issued - g.bufs : 0; n < issued; ++n) mbarrier_wait(shared_addr(&full[n % g.bufs]), (n / g.bufs) & 1);
        }
        return;
    }
    const mp<W> bound = win_bound<W>(a, N);
    const uint32_t base = shared_addr(smem);
    uint8_t* slot = smem + g.slots_off + threadIdx.x * (N + 4);
    const uint32_t y = shared_addr(slot), slots = y - (threadIdx.x & 31) * (N + 4);
    bool bad = false, failed = false;
    int mi = 0, j = 0, parity = 0;
    for (int pass = 0; pass < passes; ++pass) {
        const unsigned tile = pass * step + warp * gridDim.x + blockIdx.x;  // the first tiles go to different SMs
        win_tile<true, N, W, PLANE>(
            a, t, bound, tile, mi, slots, y, slot, bad, failed,
            [&](int) {
                // (the warp as one: its lanes vote with each other further on)
                if (!failed) failed = !__all_sync(kFull, mbarrier_wait(shared_addr(&full[j]), parity, stream_polls(withheld)));
                return failed ? kNoStage : base + j * g.buf_bytes;
            },
            [&](int) {
                __syncwarp();
                if ((threadIdx.x & 31) == 0) win_arrive(shared_addr(&empty[j]));
                if (++j == g.bufs) j = 0, parity ^= 1;
            });
    }
    if (a.status) {
        if (failed || s_failed != 0) atomicOr(a.status, PVQ_STATUS_STAGING_TIMEOUT);
        if (bad) atomicOr(a.status, PVQ_STATUS_INVALID_CODE);
    }
}

template <int N, int W, int PLANE>
int launch_window_t(BatchArgs& a, const WinTables& t, cudaStream_t stream) {
    DeviceInfo di;
    int st = device_info(&di);
    if (st != PVQ_OK) return st;
    const unsigned tiles = a.total_tiles;
    WinGeom g;
    std::memset(&g, 0, sizeof g);
    const uint32_t all = t.args.block_off[N / 4], ys = N + 4;
    const uint32_t limit = static_cast<uint32_t>(di.smem_max);
    const bool resident = N == 64 && PLANE == 96 && all + 512u * ys <= limit;
    const int most = resident ? 32 : (N == 256 ? 11 : 28);
    int warps = 0;
    double best = -1.0;
    for (int w = most; w >= 4; --w) {
        g.bufs = 0;
        uint32_t smem;
        if (resident) {
            smem = all + w * 32u * ys;
        } else {
            smem = (N == 256 ? 2u : 3u) * (t.max_block + 128u) + w * 32u * ys;
        }
        if (smem > limit) continue;
        // every tile costs the same: rounds of one tile per warp, the fullest last round wins, with a preference for
        // more warps; a launch of one round takes the smallest block that still makes it one (more SMs share it)
        const double slots = static_cast<double>(di.sms) * w, rounds = std::ceil(tiles / slots);
        if (rounds > 1.0 && warps > 0 && w < most / 2) break;
        const double score = rounds > 1.0 ? tiles / (rounds * slots) * (1.0 - 0.004 * (most - w)) : 2.0 + (most - w);
        if (score > best) best = score, warps = w;
    }
    if (warps == 0) return PVQ_ERR_UNSUPPORTED;
    g.warps = warps;
    const uint32_t slot_bytes = warps * 32u * ys;
    uint32_t tables;
    if (resident) {
        tables = (all + 127u) & ~127u;
    } else {
        g.buf_bytes = (t.max_block + 127u) & ~127u;
        g.bufs = static_cast<int>(std::min<uint32_t>(kWinBufs, (limit - slot_bytes - 128u) / g.buf_bytes));
        if (g.bufs < 2) return PVQ_ERR_UNSUPPORTED;
        tables = (g.bufs * g.buf_bytes + 127u) & ~127u;
    }
    g.slots_off = tables;
    const size_t smem = tables + slot_bytes;
    if (smem > limit) return PVQ_ERR_UNSUPPORTED;
    const int threads = warps * 32 + (resident ? 0 : 32);
    auto kern = decode_window_stream_kernel<N, W, PLANE>;
    if constexpr (N == 64 && PLANE == 96) {
        if (resident) kern = decode_window_kernel<N, W, PLANE>;
    }
    int per_sm = 0;
    if ((st = prepare_kernel(reinterpret_cast<const void*>(kern), threads, smem, &per_sm)) != PVQ_OK) return st;
    if (per_sm < 1) return PVQ_ERR_UNSUPPORTED;
    const unsigned grid = std::max(1u, std::min<unsigned>(tiles, static_cast<unsigned>(di.sms)));
    return launch_hot(kern, grid, threads, smem, stream, a, t.args, g);
}

}  // namespace

}  // namespace pvq
