// Device pieces shared by the builder of the search section (pvq_tables.cu) and the kernel
// that decodes with it (pvq_decode_search.cu); the section is described at SearchLayout.
#pragma once
#include <cstdint>

#include "pvq_walk.cuh"

namespace pvq {

// Key of a W-word integer q >= 1: q truncated to its leading 24 bits, as the bits of an fp32.
// Every conversion and every multiply-add rounds towards zero, and a truncation of a
// truncation is the truncation, so the result is exact whatever the width; it never
// decreases when q grows, which is all the bucket tables need.
__device__ __forceinline__ uint32_t search_key(const uint32_t* q, int W) {
    float x = 0.0f;
    for (int w = W - 1; w >= 0; --w) x = __fmaf_rz(x, 4294967296.0f, __uint2float_rz(q[w]));
    return __float_as_uint(x);
}

template <int W>
__device__ __forceinline__ uint32_t search_key(const uint32_t (&q)[W]) {
    float x = __uint2float_rz(q[W - 1]);
#pragma unroll
    for (int w = W - 2; w >= 0; --w) x = __fmaf_rz(x, 4294967296.0f, __uint2float_rz(q[w]));
    return __float_as_uint(x);
}

constexpr uint32_t kSearchKeyOfOne = 0x3f800000u;  // search_key(1)

__device__ __forceinline__ uint4 load_record(uint32_t addr) {
    uint4 v;
#ifdef PVQ_DEBUG
    if (!debug_table_ok(addr, 16)) return make_uint4(0u, 0u, 0u, 0u);
#endif
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t load_bucket(uint32_t addr) {
    uint32_t v;
#ifdef PVQ_DEBUG
    if (!debug_table_ok(addr, 4)) return 0u;
#endif
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// Once the section has arrived in shared memory (at `sec`; `bytes` is its size in the blob): is
// it the section of this (N,K)?  (A table built for another one would send the look-ups
// anywhere.)  If so, the numbers of rows per width go to cnt[1..4].
template <int N, int W>
__device__ __forceinline__ bool search_section_begin(const uint8_t* sec, uint32_t bytes, int K, int (&cnt)[5]) {
    const uint32_t* head = reinterpret_cast<const uint32_t*>(sec);
    if (head[0] != kSearchMagic || head[1] != static_cast<uint32_t>(N) || head[2] != static_cast<uint32_t>(K) ||
        head[3] != bytes)
        return false;
    cnt[0] = 0;
#pragma unroll
    for (int w = 1; w <= 4; ++w) cnt[w] = static_cast<int>(head[8 - w]);
    if (cnt[1] + cnt[2] + cnt[3] + cnt[4] != N || ((cnt[1] | cnt[2] | cnt[3] | cnt[4]) & 3) != 0 ||
        (W < 4 && cnt[4] != 0) || (W < 3 && cnt[3] != 0) || (W < 2 && cnt[2] != 0))
        return false;
    return true;
}

// Entry of PW words of a row stored word plane by word plane (PLANE entries a plane): word w
// sits PLANE words behind word w - 1.  `addr` is the shared address of word 0.
template <int PW, int PLANE>
__device__ __forceinline__ mp<PW> load_planes(uint32_t addr) {
    mp<PW> t;  // the plane offsets go into the loads as immediates
    t.w[0] = load_entry<1, 0>(addr).w[0];
    if constexpr (PW > 1) t.w[1] = load_entry<1, PLANE * 4>(addr).w[0];
    if constexpr (PW > 2) t.w[2] = load_entry<1, 2 * PLANE * 4>(addr).w[0];
    if constexpr (PW > 3) t.w[3] = load_entry<1, 3 * PLANE * 4>(addr).w[0];
    return t;
}

// Four bytes of a thread's slot at once.
__device__ __forceinline__ void store_y4(uint32_t addr, uint32_t val) {
#ifdef PVQ_DEBUG
    if (!debug_slot_ok(addr, 4)) return;
#endif
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(val) : "memory");
}

// From the threshold indices of four positions (a byte each, first position lowest) to their coordinates, all four at
// a time: pulses left after a position m >> 1, before it those of the position before (k for the
// first); their difference is |y|, and y > 0 where m is odd.  No byte borrows from or
// carries into its neighbour: the pulses left never grow, and |y| <= 127.
// The four y_i + 128 go to the word at y, their squares to ssy.
__device__ __forceinline__ void search_coordinates(uint32_t m4, uint32_t& k, uint32_t y, uint32_t& ssy) {
    const uint32_t after = (m4 >> 1) & 0x7f7f7f7fu;
    const uint32_t before = (after << 8) | k;
    const uint32_t mag = before - after;
    ssy = __dp4a(mag, mag, ssy);
    const uint32_t odd = m4 & 0x01010101u;
    const uint32_t pos = (odd << 8) - odd;  // 0xff in the bytes with y > 0
    store_y4(y, (mag ^ ~pos) + 0x80808081u + pos);  // 128 + |y|; else 255 - |y| + 128 - 255: no byte of the sum leaves 1 .. 255
    k = after >> 24;
}

// How a position is searched: the key of q selects a bucket; its entry holds the low key bits of the threshold T[m0] in it, and m0.
// q's own low key bits being larger means q > T[m0] and the index m0 + 1, smaller that it is m0 (a bucket without a threshold
// holds all ones there).  Equal bits leave it open, unless the threshold is its key (below 2^24): then the threads of the warp
// whose bits were equal compare q with T[m0] in full.  A launch of some rounds can afford to rewrite the staged buckets first
// (LONG): an entry is then what, added to twice the key, leaves the index in the top byte, the comparison being the carry into
// it, and all ones below it where the comparison is open (an even number where the threshold is its key).  Four instructions
// less a position; with them and the last four positions looked up, decoder layer 271 -> 257 us.
// Tried and not kept: bucket and key bits from one wide product, and the comparison taken as the borrow of a
// subtraction (decoder layer 271 -> 288 and 284 us: they tie up the pipes that are short); equal bits not looked for but found out
// from the position that follows, and such a group searched again (237 us, but heavy-tailed data have many: N = 32, 96
// bits, Student's t with 3 degrees of freedom, 4096 x 4096 25 -> 70 us); E read before the vote (257 -> 259 us).

// The last four positions at once: the indices of q in row 3, of the q that follows in row 2, and so on depend on q
// alone (no N, K or pulses left in them), and q is small there: at most N(4,k) with k pulses left, some K / 8 of them at
// N = 32.  A QuadTable holds the four indices, first position lowest, of q = 1 .. N(4,kQuadPulses); a larger q is searched.
constexpr uint32_t kQuadPulses = 16;
constexpr uint32_t quad_count(uint32_t n, uint32_t k) {  // V(n,k) = sum over j <= k of N(n,j)
    return n == 0 ? 1u : (n == 1 ? 2u * k + 1u : (n == 2 ? 2u * k * k + 2u * k + 1u : (2u * k + 1u) * (2u * k * k + 2u * k + 3u) / 3u));
}
constexpr uint32_t quad_threshold(uint32_t n, uint32_t m) {  // T_n[m]
    return (m & 1u) ? 2u * quad_count(n, m >> 1) : quad_count(n, m >> 1) + (m > 1u ? quad_count(n, (m >> 1) - 1u) : 0u);
}
constexpr uint32_t kQuadEntries = quad_threshold(3, 2 * kQuadPulses);  // N(4,16) = 11008
struct QuadTable {
    uint32_t m4[kQuadEntries];
};
constexpr QuadTable make_quads() {
    QuadTable t{};
    uint32_t m3 = 0;
    for (uint32_t q = 1; q <= kQuadEntries; ++q) {
        while (quad_threshold(3, m3) < q) ++m3;
        const uint32_t q2 = q + quad_threshold(2, m3 & ~1u) - quad_threshold(3, m3);
        uint32_t m2 = q > 1 && (t.m4[q - 2] & 0xffu) == m3 ? (t.m4[q - 2] >> 8) & 0xffu : 0u;  // from where the q before was
        while (quad_threshold(2, m2) < q2) ++m2;
        const uint32_t q1 = q2 + quad_threshold(1, m2 & ~1u) - quad_threshold(2, m2);
        const uint32_t m1 = q1 == 1 ? 0 : (q1 + 1) / 2;  // thresholds 1, 2, 4, 6, ...
        const uint32_t q0 = q1 + quad_threshold(0, m1 & ~1u) - quad_threshold(1, m1);
        t.m4[q - 1] = m3 | m2 << 8 | m1 << 16 | (q0 - 1) << 24;  // thresholds 1, 2
    }
    return t;
}

// Makes the accepted section ready for the search; all threads, a barrier follows.  `t_off`: where its buckets end.  Records
// afterwards: 32 - shift, the shared addresses of its row of E and of its buckets, the shift.
// The thresholds T are not staged (open comparisons read some, from global memory): the
// increments E sit where T is in the blob, `t_before_e` bytes lower.
template <int N, bool LONG>
__device__ __forceinline__ void search_section_ready(uint8_t* sec, uint32_t t_off, uint32_t t_before_e) {
    uint32_t* recs = reinterpret_cast<uint32_t*>(sec + kSearchHeader);
    if constexpr (LONG) {
        auto first_bucket = [&](int n) { return n < N ? recs[4 * n + 2] + ((kSearchKeyOfOne >> recs[4 * n + 3]) << 2) : t_off; };
        for (int n = threadIdx.x >> 5; n < N; n += blockDim.x >> 5) {
            const uint32_t sh = recs[4 * n + 3], from = first_bucket(n), end = first_bucket(n + 1);
            uint32_t* b = reinterpret_cast<uint32_t*>(sec + from);
            for (uint32_t i = threadIdx.x & 31; from + 4u * i < end; i += 32u) {
                const uint32_t e = b[i];
                // (no threshold: the last key of the bucket, which nothing in it passes, and bit 8, as for one that is its key)
                b[i] = (e << 24) + 0xffffffu - ((e >> 8) & 1u) - 2u * ((((kSearchKeyOfOne >> sh) + i) << sh) + (e >> (32u - sh)));
            }
        }
        __syncthreads();
    }
    if (threadIdx.x < N) {
        uint32_t* rec = recs + 4 * threadIdx.x;
        const uint32_t base = shared_addr(sec);
        rec[1] += base - t_before_e;
        rec[2] += base;
    }
}

// Four positions of GP codes (GP independent chains of dependent table reads, so that one
// thread keeps several reads in flight), in PW-word arithmetic on rows of PW word planes.
// `rec` is the shared address of the record of the first of the four rows (the rows of the
// following positions have the records before it); a record is read once for all chains.
// `t_rows` plus the shared address of a row of E is the global address of the same row of T.
// The four y_i + 128 of chain j go to the word at y + j * ychain, their squares to ssy[j].
template <int W, int PW, int GP, int PLANE, bool LONG>
__device__ __forceinline__ void search_block4(mp<W> (&q)[GP], uint32_t (&k)[GP], uint32_t rec, const uint8_t* t_rows,
                                              uint32_t y, uint32_t ychain, uint32_t (&ssy)[GP]) {
    uint32_t acc[GP];  // the four threshold indices m, a byte each, first position lowest
    mp<PW> v[GP];      // the low PW words of q: the rest is zero by now
#pragma unroll
    for (int j = 0; j < GP; ++j) {
        acc[j] = 0u;
#pragma unroll
        for (int w = 0; w < PW; ++w) v[j].w[w] = q[j].w[w];
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const uint4 r = load_record(rec - static_cast<uint32_t>(s) * 16u);  // 32 - shift, E row, buckets, shift
        uint32_t key[GP], m[GP];  // m: the index; LONG: in the top byte
        bool open[GP], any = false;
#pragma unroll
        for (int j = 0; j < GP; ++j) {
            key[j] = search_key<PW>(v[j].w);
            m[j] = load_bucket(r.z + ((key[j] >> r.w) << 2));
        }
#pragma unroll
        for (int j = 0; j < GP; ++j) {
            if constexpr (LONG) {
                m[j] += key[j] + key[j];
                open[j] = (~m[j] & 0xffffffu) == 0u;
            } else {
                const uint32_t low = key[j] << r.x;  // the key bits below the shift, left-aligned like the entry's
                open[j] = m[j] - low < 256u;
                m[j] = (m[j] & 0xffu) + (low > m[j] ? 1u : 0u);
            }
            any = any || open[j];
        }
        if (__any_sync(kFull, any)) {
#pragma unroll
            for (int j = 0; j < GP; ++j) {
                if (open[j]) {
                    // the row of T in global memory lies where the row of E lies in shared memory
                    const uint32_t* tp = reinterpret_cast<const uint32_t*>(t_rows + r.y + (LONG ? m[j] >> 24 : m[j]) * 4u);
                    mp<PW> t, d;
#pragma unroll
                    for (int w = 0; w < PW; ++w) t.w[w] = tp[w * PLANE];
                    if (mp_sub_borrow<PW>(d, t, v[j])) m[j] += LONG ? 1u << 24 : 1u;
                }
            }
        }
#pragma unroll
        for (int j = 0; j < GP; ++j) {
            const mp<PW> e = load_planes<PW, PLANE>(r.y + ((LONG ? m[j] >> 24 : m[j]) << 2));
            mp_add<PW>(v[j], e);
            acc[j] = LONG ? __byte_perm(acc[j], m[j], 0x7321) : __funnelshift_r(acc[j], m[j], 8);  // the new byte enters at the top
        }
    }
#pragma unroll
    for (int j = 0; j < GP; ++j) {
        search_coordinates(acc[j], k[j], y + static_cast<uint32_t>(j) * ychain, ssy[j]);
#pragma unroll
        for (int w = 0; w < PW; ++w) q[j].w[w] = v[j].w[w];
    }
}

// The points of GP codes: q = N(N,K) - code on entry.  `recs` is the shared address of the
// row records (absolute shared addresses by now), cnt[w] the number of rows done in w words; quads: shared address of a QuadTable,
// or 0: without.
template <int N, int W, int GP, int PLANE, bool LONG>
__device__ __forceinline__ void search_codes(mp<W> (&q)[GP], int K, uint32_t recs, const uint8_t* t_rows, const int (&cnt)[5], uint32_t quads,
                                             uint32_t y, uint32_t ychain, uint32_t (&ssy)[GP]) {
    uint32_t k[GP];
#pragma unroll
    for (int j = 0; j < GP; ++j) k[j] = static_cast<uint32_t>(K);
    uint32_t rec = recs + static_cast<uint32_t>(N - 1) * 16u;
    if constexpr (W >= 4) {
#pragma unroll 1
        for (int b = 0; b < cnt[4]; b += 4, rec -= 64u, y += 4u) search_block4<W, 4, GP, PLANE, LONG>(q, k, rec, t_rows, y, ychain, ssy);
    }
    if constexpr (W >= 3) {
#pragma unroll 1
        for (int b = 0; b < cnt[3]; b += 4, rec -= 64u, y += 4u) search_block4<W, 3, GP, PLANE, LONG>(q, k, rec, t_rows, y, ychain, ssy);
    }
    if constexpr (W >= 2) {
#pragma unroll 1
        for (int b = 0; b < cnt[2]; b += 4, rec -= 64u, y += 4u) search_block4<W, 2, GP, PLANE, LONG>(q, k, rec, t_rows, y, ychain, ssy);
    }
#pragma unroll 1
    for (int b = 0; b < cnt[1]; b += 4, rec -= 64u, y += 4u) {
        if (LONG && b + 4 == cnt[1] && quads != 0u) {  // the last four (N(4,K) is below 2^32: a block of one word)
            uint32_t most = q[0].w[0];
#pragma unroll
            for (int j = 1; j < GP; ++j) most = max(most, q[j].w[0]);
            if (!__any_sync(kFull, most > kQuadEntries)) {
                uint32_t m4[GP];
#pragma unroll
                for (int j = 0; j < GP; ++j) m4[j] = load_bucket(quads + ((q[j].w[0] - 1u) << 2));
#pragma unroll
                for (int j = 0; j < GP; ++j) search_coordinates(m4[j], k[j], y + static_cast<uint32_t>(j) * ychain, ssy[j]);
                break;
            }
        }
        search_block4<W, 1, GP, PLANE, LONG>(q, k, rec, t_rows, y, ychain, ssy);
    }
}

}  // namespace pvq
