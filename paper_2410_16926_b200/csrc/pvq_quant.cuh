// Direction of a group (Sec. 2.5 / Algorithm 1 in the floor + greedy reading) for the kernels
// that spread a group over lanes: the L = 1, 2, 4 or 8 neighbouring lanes of a group hold E = 8,
// 16 or 32 of its N = E * L consecutive values each.
//
//   a_i = |x_i| * (K / l1), f_i = floor(a_i), e_i = a_i - f_i, d = K - sum f_i;
//   the d largest residuals e_i get one more pulse, lowest index first among equals
//   (why this is the greedy loop's result: quantize_direction in pvq_encode_impl.cuh).
//
// Nothing is sorted or counted twice.  The residuals' leading 8 bits, a byte each, are turned into eight bit
// planes (a plane: one bit of every residual of the lane, in one register), and the d-th largest is found
// a bit at a time from the top: the residuals still undecided that have the bit are either all chosen, or
// are the undecided ones from here on.  What no bit of the eight tells apart, two residuals of a group now
// and then, is ranked on the exact fp32 values, fetched again from where the group came from.
// 32 values a lane: 48 instructions for the planes, 56 for the eight steps (a sorting network: 382 min / max at half
// rate; before: about five counting passes of some 45 instructions, and four candidates to rank).  What uses it is
// bound by issue: encoding a decoder layer at N = 32, 96 bits 403 -> 336 us, the round trip of 16384 x 4096 98 -> 77 us at
// N = 32 and 131 -> 97 us at N = 128, encoding 4096 x 4096 at N = 128, 384 bits 66 -> 58 us.
//
// The result is a point packed in bytes: word j holds |y_i| of positions 4j .. 4j+3, last
// position lowest, which is the order in which the Fischer index needs the pulses behind
// a position (a multiplication by 0x01010101 is then the running sum).  K > 127 (WIDE): 16-bit
// halves, word h holds positions 2h (high) and 2h+1 (low).
#pragma once
#include <cuda_bf16.h>

#include "pvq_f32x2.cuh"
#include "pvq_internal.cuh"

namespace pvq {

constexpr uint32_t kH4 = 0x80808080u, kOne4 = 0x01010101u;

// Step 5: q = floor(CDF(u) 2^b) as the number of bin edges <= u, for b <= 8 bits; edge(i): the i-th of 2^b - 1.
// (Unrolled: three or four instructions a step instead of eight with a counter; decoder layer 286 -> 284.5 us, 4096 x 4096 fp32
// 39.5 -> 39.1.)
template <class Edge>
__device__ __forceinline__ int amplitude_bin(float u, int b, const Edge& edge) {
    int q = 0;
    switch (b) {
        case 8: if (edge(127) <= u) q = 128; [[fallthrough]];
        case 7: if (edge(q + 63) <= u) q += 64; [[fallthrough]];
        case 6: if (edge(q + 31) <= u) q += 32; [[fallthrough]];
        case 5: if (edge(q + 15) <= u) q += 16; [[fallthrough]];
        case 4: if (edge(q + 7) <= u) q += 8; [[fallthrough]];
        case 3: if (edge(q + 3) <= u) q += 4; [[fallthrough]];
        case 2: if (edge(q + 1) <= u) q += 2; [[fallthrough]];
        default: if (edge(q) <= u) q += 1;
    }
    return q;
}

// A lane's E values as they sit in memory: E/2 words of two bf16, or E words.
template <int E, bool BF16>
constexpr int kRawWords = BF16 ? E / 2 : E;

template <int E, bool BF16>
__device__ __forceinline__ void load_chunk(const void* base, size_t elem_off, uint32_t (&r)[kRawWords<E, BF16>]) {
    const uint4* p = reinterpret_cast<const uint4*>(static_cast<const uint8_t*>(base) + elem_off * (BF16 ? 2 : 4));
#pragma unroll
    for (int v = 0; v < kRawWords<E, BF16> / 4; ++v) {
        const uint4 q = __ldg(p + v);
        r[4 * v] = q.x, r[4 * v + 1] = q.y, r[4 * v + 2] = q.z, r[4 * v + 3] = q.w;
    }
}

template <int E, bool BF16>
__device__ __forceinline__ float chunk_abs(const uint32_t (&raw)[kRawWords<E, BF16>], int i) {
    if constexpr (BF16)
        return __uint_as_float((i & 1) ? (raw[i / 2] & 0x7fff0000u) : ((raw[i / 2] & 0x7fffu) << 16));
    else
        return fabsf(__uint_as_float(raw[i]));
}

// A tile of bf16 values lies in shared memory as it does in global memory, E values (E / 8 pieces of 16
// bytes) a lane.  For the lanes' 16-byte accesses to hit different banks, lane l starts with
// piece lane_rotation(l) and goes round.
template <int E>
__device__ __forceinline__ int lane_rotation(int lane) {
    return (lane * (E / 8) >> 3) & (E / 8 - 1);
}

// |x_i| one at a time, from where the lane's values came from (global memory)
template <bool BF16>
struct FetchGlobal {
    const void* p;  // the lane's first value
    __device__ __forceinline__ float operator()(int i) const {
        if constexpr (BF16)
            return __uint_as_float(static_cast<uint32_t>(__ldg(static_cast<const unsigned short*>(p) + i) & 0x7fffu) << 16);
        else
            return fabsf(__ldg(static_cast<const float*>(p) + i));
    }
};

// |x_i| of a lane whose values sit in shared memory
struct FetchShared {
    const unsigned short* p;
    __device__ __forceinline__ float operator()(int i) const { return __uint_as_float(static_cast<uint32_t>(p[i] & 0x7fffu) << 16); }
};

// all lanes of a group get the sum over its lanes (contiguous halves: the balanced tree's order)
template <int L>
__device__ __forceinline__ float group_add(float v) {
#pragma unroll
    for (int o = 1; o < L; o <<= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
template <int L>
__device__ __forceinline__ int group_add(int v) {
#pragma unroll
    for (int o = 1; o < L; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The group's norms by the balanced tree over contiguous halves, and the lane's |x_i|.
// Values i and i + E/2 share a register pair: the halves of the tree only meet in its last
// addition.  A lane may hold its values rotated by a number of runs of 8 (see lane_rotation):
// all that changes is which quarters belong together when that number is odd.
template <int E, int L, bool BF16>
__device__ __forceinline__ void group_norms(const uint32_t (&raw)[kRawWords<E, BF16>], float (&ax)[E], float& l1, float& ss,
                                            float minus_zero, int rotation = 0) {
    constexpr int H = E / 2, Q = E / 4;
#pragma unroll
    for (int i = 0; i < E; ++i) ax[i] = chunk_abs<E, BF16>(raw, i);
    f32x2 s[Q], q[Q];
#pragma unroll
    for (int w = 0; w < Q; ++w) {
        const f32x2 a = pack2(ax[2 * w], ax[2 * w + H]), b = pack2(ax[2 * w + 1], ax[2 * w + 1 + H]);
        s[w] = add2(a, b);
        // Each square rounded by itself, for bf16 too: below 2^-67 the square of a bf16 value has bits under the last
        // place of the smallest fp32 number.  (Not merged: 8 instructions more for 32 values; a decoder layer, N = 32,
        // 389 -> 402 us.)
        q[w] = add2(mul2_rounded(a, a, minus_zero), mul2_rounded(b, b, minus_zero));
    }
#pragma unroll
    for (int st = 1; st < Q; st <<= 1) {
        if (E == 32 && 2 * st == Q) {  // quarters 0 | 2 in s[0], 1 | 3 in s[st]
            float a, b;
            unpack2(s[st], a, b);
            s[st] = (rotation & 1) ? pack2(b, a) : pack2(a, b);
            unpack2(q[st], a, b);
            q[st] = (rotation & 1) ? pack2(b, a) : pack2(a, b);
        }
#pragma unroll
        for (int w = 0; w < Q; w += 2 * st) {
            s[w] = add2(s[w], s[w + st]);
            q[w] = add2(q[w], q[w + st]);
        }
    }
    float lo, hi;
    unpack2(s[0], lo, hi);
    l1 = group_add<L>(__fadd_rn(lo, hi));
    unpack2(q[0], lo, hi);
    ss = group_add<L>(__fadd_rn(lo, hi));
}

// prmt with the selectors' top bits in use (the byte's sign, eight times); __byte_perm ignores them
__device__ __forceinline__ uint32_t perm_sign(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// 0xff in the bytes whose value has its sign bit set, in the packed point's order
template <int E, bool BF16>
__device__ __forceinline__ uint32_t chunk_signs4(const uint32_t (&raw)[kRawWords<E, BF16>], int j) {
    if constexpr (BF16)
        return perm_sign(raw[2 * j + 1], raw[2 * j], 0xDF9B);
    else
        return __byte_perm(perm_sign(raw[4 * j + 3], raw[4 * j + 2], 0x00FB), perm_sign(raw[4 * j + 1], raw[4 * j], 0x00FB), 0x5410);
}

// A lane's share of the point.
template <int E, bool WIDE>
struct LanePoint {
    static constexpr int J = E / 4;
    static constexpr int FW = WIDE ? E / 2 : E / 4;
    uint32_t y[FW];  // |y_i|, packed as said at the top
    bool has_dir;    // false: the group's point is (K, 0, ..., 0), its first coordinate positive
};

// Masks of a lane's residuals: bit 8b + j stands for byte b of word j.  The position that a bit belongs to:
__device__ __forceinline__ int mask_bit_position(int bit) { return 4 * (bit & 7) + 3 - (bit >> 3); }

// x[j] holds a byte for each of four residuals.  Afterwards bit 8b + j of (x[p % J] >> (p - p % J)), j < J, is bit p of
// byte b of word j: in every byte the J rows of J bits that lie below one another are transposed.
template <int J>
__device__ __forceinline__ void bit_planes(uint32_t (&x)[J]) {
    static_assert(J == 2 || J == 4 || J == 8, "");
#pragma unroll
    for (int s = J / 2; s >= 1; s >>= 1) {
        const uint32_t low = s == 4 ? 0x0f0f0f0fu : (s == 2 ? 0x33333333u : 0x55555555u);
#pragma unroll
        for (int j = 0; j < J; ++j)
            if ((j & s) == 0) {
                const uint32_t a = x[j], b = x[j + s];
                x[j] = (a & low) | ((b << s) & ~low);
                x[j + s] = ((a >> s) & low) | (b & ~low);
            }
    }
}

// The residuals of the candidates (bits of `cand`), exactly, and which of the group's candidates
// are the r largest, lowest index first among equals.  Returns the chosen bits.  Called by
// all lanes of a warp; a group with nothing to choose comes with cand = 0.
//   Usual (rank_candidates): no lane has more than C candidates; every candidate counts the better ones.
//   Otherwise (many equal or nearly equal residuals): one value class after the other, from the
//   largest down, until r are chosen.
// rotation: position i of the lane is held as position i - 8 * rotation (modulo E).
template <int E, int L, int C, class Fetch>
__device__ __forceinline__ uint32_t rank_candidates(uint32_t cand, int r, float gsc, const Fetch& fetch, int rotation) {
    constexpr float magic = 8388608.0f;  // 2^23
    const int sub = static_cast<int>(threadIdx.x) & (L - 1);
    uint32_t chosen = 0u;
    {
        float e[C];
        int pos[C], better[C];
        uint32_t bit[C];
        uint32_t left = cand;
#pragma unroll
        for (int s = 0; s < C; ++s) {
            const int b = 31 - __clz(static_cast<int>(left));  // -1: no candidate left
            bit[s] = left & (1u << (b & 31));
            left ^= bit[s];
            pos[s] = bit[s] ? (mask_bit_position(b) + 8 * rotation) & (E - 1) : 0;
        }
#pragma unroll
        for (int s = 0; s < C; ++s) e[s] = fetch(pos[s]);
#pragma unroll
        for (int s = 0; s < C; ++s) {
            const float a = __fmul_rn(e[s], gsc);
            e[s] = __fsub_rn(a, __fsub_rn(__fadd_rd(a, magic), magic));
            if (!bit[s]) e[s] = -1.0f;
            better[s] = 0;
        }
#pragma unroll
        for (int s = 0; s < C; ++s) {
#pragma unroll
            for (int u = s + 1; u < C; ++u) {
                const bool second = e[u] > e[s] || (e[u] == e[s] && pos[u] < pos[s]);
                better[s] += second ? 1 : 0;
                better[u] += second ? 0 : 1;
            }
        }
#pragma unroll
        for (int o = 1; o < L; ++o) {
            const bool lower = (sub ^ o) < sub;  // that lane holds lower positions: it wins ties
#pragma unroll
            for (int u = 0; u < C; ++u) {
                const float eo = __shfl_xor_sync(0xffffffffu, e[u], o);
#pragma unroll
                for (int s = 0; s < C; ++s) better[s] += (eo > e[s] || (lower && eo == e[s])) ? 1 : 0;
            }
        }
#pragma unroll
        for (int s = 0; s < C; ++s)
            if (better[s] < r) chosen |= bit[s];
    }
    return chosen;
}

template <int E, int L, class Fetch>
__device__ __forceinline__ uint32_t choose_candidates(uint32_t cand, int r, float gsc, const Fetch& fetch, int rotation) {
    constexpr float magic = 8388608.0f;  // 2^23
    auto residual = [&](int i) {
        const float a = __fmul_rn(fetch(i), gsc);
        return __fsub_rn(a, __fsub_rn(__fadd_rd(a, magic), magic));
    };
    const int sub = static_cast<int>(threadIdx.x) & (L - 1);
    const int mine_all = __popc(cand);
    if (__all_sync(0xffffffffu, mine_all <= 2)) {
        if constexpr (L > 1) return rank_candidates<E, L, 2>(cand, r, gsc, fetch, rotation);
        // two, or none, of which one is chosen
        const uint32_t one = cand & (0u - cand), two = cand ^ one;
        const int i = (mask_bit_position(31 - __clz(static_cast<int>(one))) + 8 * rotation) & (E - 1);
        const int j = (mask_bit_position(31 - __clz(static_cast<int>(two))) + 8 * rotation) & (E - 1);
        const float a = residual(i), b = residual(j);
        return a > b || (a == b && i < j) ? one : two;
    }
    if (__all_sync(0xffffffffu, mine_all <= 4)) return rank_candidates<E, L, 4>(cand, r, gsc, fetch, rotation);
    uint32_t chosen = 0u;
    for (int round = 0; round < E * L; ++round) {
        if (!__any_sync(0xffffffffu, cand != 0u && r > 0)) break;
        float top = -1.0f;  // the group's largest residual left
        for (uint32_t left = cand; left; left &= left - 1u) top = fmaxf(top, residual((mask_bit_position(__ffs(left) - 1) + 8 * rotation) & (E - 1)));
#pragma unroll
        for (int o = 1; o < L; o <<= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
        uint32_t equal = 0u;
        for (uint32_t left = cand; left; left &= left - 1u)
            if (residual((mask_bit_position(__ffs(left) - 1) + 8 * rotation) & (E - 1)) == top) equal |= left & (0u - left);
        const int mine = __popc(equal);
        int before = 0, all = 0;  // of the class: in lower lanes, in the group
#pragma unroll
        for (int o = 0; o < L; ++o) {
            const int n = L == 1 ? mine : __shfl_xor_sync(0xffffffffu, mine, o);
            all += n;
            if ((sub ^ o) < sub) before += n;
        }
        if (all <= r) {
            chosen |= equal;
        } else {  // the lowest positions of the class
            int take = min(max(r - before, 0), mine);
            for (int i = 0; i < E && take > 0; ++i) {
                const int held = (i - 8 * rotation) & (E - 1);
                const uint32_t b = 1u << (8 * (3 - (held & 3)) + (held >> 2));
                if (equal & b) chosen |= b, --take;
            }
        }
        r -= min(all, r);
        cand &= ~equal;
        if (r == 0) cand = 0u;
    }
    return chosen;
}

// One step of the selection: `have`, c in the group, are the undecided residuals with the bit.  All of them are taken if no more
// are needed than that, and those without the bit stay undecided; else those with it do.  (Predicates: a selection
// and an operation each otherwise.)
__device__ __forceinline__ void take_or_keep(int c, uint32_t have, uint32_t plane, uint32_t& sel, int& need, uint32_t& cand) {
    uint32_t rest;
    asm("{\n\t.reg .pred p;\n\t"
        "setp.le.s32 p, %3, %1;\n\t"
        "mov.b32 %2, %4;\n\t"
        "@p lop3.b32 %2, %5, %6, 0, 0x30;\n\t"
        "@p or.b32 %0, %0, %4;\n\t"
        "@p sub.s32 %1, %1, %3;\n\t}"
        : "+r"(sel), "+r"(need), "=&r"(rest)
        : "r"(c), "r"(have), "r"(cand), "r"(plane));
    cand = rest;
}

struct NoHook {
    __device__ __forceinline__ void operator()() const {}
};

// ax: |x_i| of the lane's values; l1: of the whole group.  Points in bytes (not WIDE) hold up to 255 pulses: no coordinate, and no
// sum of the lane's floors over the words, which is an integer of at most K as their sum is below K + 1, leaves its byte.  (What
// reads a sign or a comparison from a byte's top bit has to see to K <= 127 itself.)  `hook` is called by the warp half way, where few registers
// are in use.
template <int E, int L, bool WIDE, class Fetch, class Hook = NoHook>
__device__ __forceinline__ void quantize_group(const float (&ax)[E], float l1, int K, const Fetch& fetch,
                                               LanePoint<E, WIDE>& pt, float minus_zero, int rotation = 0, Hook&& hook = Hook()) {
    constexpr int N = E * L, J = E / 4, H = E / 2;
    const float gsc = __fdiv_rn(static_cast<float>(K), l1);
    // no direction: l1 zero or not finite, or a scale that overflows
    bool has_dir = (l1 > 0.0f) && (l1 <= 3.4028234e38f) && (gsc <= 3.4028234e38f);
    // a + 2^15 rounded down is 2^15 + floor(256 a) / 256: 8 bits of the residual are the lowest byte, the floor
    // begins at the next (a < K + 1 leaves the exponent alone)
    static_assert(kMaxPulses + 1 < 32768, "2^15 + a below 2^16");
    uint32_t t[E];
    {
        const f32x2 g2 = pack2(gsc, gsc), m2 = pack2(32768.0f, 32768.0f);
#pragma unroll
        for (int i = 0; i < H; ++i) {
            float lo, hi;
            unpack2(add2_rd(mul2_rounded(pack2(ax[i], ax[i + H]), g2, minus_zero), m2), lo, hi);
            t[i] = __float_as_uint(lo);
            t[i + H] = __float_as_uint(hi);
        }
    }
    uint32_t x[J];  // leading 8 bits of the residuals, a byte each
    int fsum;
    if constexpr (!WIDE) {
        uint32_t sum4 = 0u;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const uint32_t u = __byte_perm(t[4 * j + 3], t[4 * j + 2], 0x5410), v = __byte_perm(t[4 * j + 1], t[4 * j], 0x5410);
            x[j] = __byte_perm(u, v, 0x6420);
            pt.y[j] = __byte_perm(u, v, 0x7531);  // floors, at most K
            sum4 += pt.y[j];                      // ... as are these
        }
        fsum = static_cast<int>(__dp4a(sum4, kOne4, 0u));
    } else {
        uint32_t sum2 = 0u;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const uint32_t u = __byte_perm(t[4 * j + 3], t[4 * j + 2], 0x0040), v = __byte_perm(t[4 * j + 1], t[4 * j], 0x0040);
            x[j] = __byte_perm(u, v, 0x5410);
            pt.y[2 * j] = __byte_perm(t[4 * j + 1], t[4 * j], 0x6521);
            pt.y[2 * j + 1] = __byte_perm(t[4 * j + 3], t[4 * j + 2], 0x6521);
            sum2 += pt.y[2 * j] + pt.y[2 * j + 1];
        }
        fsum = static_cast<int>((sum2 & 0xffffu) + (sum2 >> 16));
    }
    int d = K - group_add<L>(fsum);
    // 0 <= d <= N for finite input (sum floor(a_i) <= sum a_i < K + 1); anything else is treated
    // as "no direction"
    has_dir = has_dir && d >= 0 && d <= N;
    if (!has_dir) d = 0;

    hook();
    bit_planes<J>(x);
    uint32_t sel = 0u, cand = ((1u << J) - 1u) * kOne4;  // chosen; undecided: the same in all bits so far
    int need = d;                                        // still to be chosen among the undecided ones
#pragma unroll
    for (int p = 7; p >= 0; --p) {
        const uint32_t plane = x[p % J] >> (p - p % J), have = cand & plane;
        const int c = group_add<L>(__popc(have));
        take_or_keep(c, have, plane, sel, need, cand);
    }
    const bool rest = group_add<L>(__popc(cand)) == need;  // (none needed: no matter)
    if (rest) sel |= cand;
    if (rest || need == 0) cand = 0u;
    if (__any_sync(0xffffffffu, cand != 0u)) sel |= choose_candidates<E, L>(cand, need, gsc, fetch, rotation);

    if constexpr (!WIDE) {
#pragma unroll
        for (int j = 0; j < J; ++j) pt.y[j] += (sel >> j) & kOne4;
    } else {
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const uint32_t b4 = (sel >> j) & kOne4;
            pt.y[2 * j] += __byte_perm(b4, 0u, 0x4342);      // positions 4j+1 (low half), 4j
            pt.y[2 * j + 1] += __byte_perm(b4, 0u, 0x4140);  // positions 4j+3, 4j+2
        }
    }
    if (__any_sync(0xffffffffu, !has_dir)) {
        if (!has_dir) {  // (K, 0, ..., 0)
            const int first = (threadIdx.x & (L - 1)) == 0 ? (-8 * rotation) & (E - 1) : -1;  // where position 0 is held
#pragma unroll
            for (int w = 0; w < LanePoint<E, WIDE>::FW; ++w)
                pt.y[w] = (WIDE ? 2 * w : 4 * w) == first ? static_cast<uint32_t>(K) << (WIDE ? 16 : 24) : 0u;
        }
    }
    pt.has_dir = has_dir;
}

}  // namespace pvq
