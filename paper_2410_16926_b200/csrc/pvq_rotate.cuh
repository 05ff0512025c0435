// Random-sign Hadamard rotation of a row held E consecutive values per lane (Sec. 2.3, Sec. 3.3
// Step 1): x <- (x * s) H_B / sqrt(B) on every block of B consecutive columns, B = E * T0.  The
// Sylvester butterflies (a, b) -> (a + b, a - b) run with strides 1, 2, 4, ..., B/2.  Every sum
// is one fp32 addition, so the result does not depend on which thread makes it.
//   E = 32 (rotate_lanes32): always inside a lane.  After five strides the values of a warp change places through shared
//   memory, a lane then holding those 32 apart, for the next five; what spans warps is done two strides at a time, a
//   thread holding four times eight values.  (Shuffles for the strides between lanes, 160 of them, and a round through
//   shared memory for each larger one: 1999 x 4096, B = 4096, 28.3 us.)
//   E = 8, 16 (rotate_lanes): strides below E inside the lane, E .. 16 E between the lanes of a warp by shuffle (T0
//   divides the lanes of a row, so lane t and its partner t ^ d belong to the same block), larger ones through shared memory.
#pragma once
#include "pvq_quant.cuh"

namespace pvq {

// The signs of one rotation block as bits, a word of E bits per lane; all threads, before a barrier.
// Bit i is value i's; for 32 values: bit 31 - w value 2w + 1's, bit 15 - w value 2w's, so that a shift by w brings
// the signs of a word of two bf16 to where they act.
template <int E>
__device__ __forceinline__ void pack_signs(uint32_t* s_signs, const float* signs, int block) {
    for (int j = threadIdx.x; j < block / E; j += blockDim.x) {
        uint32_t bits = 0;
#pragma unroll
        for (int i = 0; i < E; i += 4) {
            const float4 s = __ldg(reinterpret_cast<const float4*>(signs + j * E + i));
            if constexpr (E == 32)
                bits |= ((s.x < 0.0f ? 0x8000u : 0u) | (s.y < 0.0f ? 0x80000000u : 0u) | (s.z < 0.0f ? 0x4000u : 0u) | (s.w < 0.0f ? 0x40000000u : 0u)) >> (i / 2);
            else
                bits |= (s.x < 0.0f ? 1u << i : 0u) | (s.y < 0.0f ? 2u << i : 0u) | (s.z < 0.0f ? 4u << i : 0u) | (s.w < 0.0f ? 8u << i : 0u);
        }
        s_signs[j] = bits;
    }
}

// The strides 1 .. 16 among 32 values, values i and i + 16 a pair, as far as they are below `span`.
__device__ __forceinline__ void butterflies32(f32x2 (&v)[16], int span) {
    const f32x2 m2 = pack2(-1.0f, -1.0f);
#pragma unroll
    for (int h = 1; h < 16; h <<= 1) {
        if (h >= span) return;
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if ((i & h) == 0) {
                const f32x2 a = v[i], b = v[i + h];
                v[i] = add2(a, b);
                v[i + h] = fma2(b, m2, a);  // a - b: the product is exact
            }
    }
    if (span <= 16) return;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        float a, b;
        unpack2(v[i], a, b);
        v[i] = pack2(__fadd_rn(a, b), __fsub_rn(a, b));
    }
}

// Values in shared memory, 32 to a row.  Piece q of a row holds values 2q, 2q + 16, 2q + 1 and 2q + 17: two pairs, as lanes
// hold them (no register is moved).  The eight pieces are exchanged by the row's number, so that lanes that read
// the same piece of consecutive rows, or the same place of consecutive rows' pieces, hit different banks.
// As byte offsets from a multiple of 128: piece q of a row lies at rotate_row(row) ^ 16 q.
__device__ __forceinline__ uint32_t rotate_row(uint32_t row) { return row * 128u + ((row & 7u) << 4); }

// LEVELS (1 or 2) strides between rows, 2^bit rows apart and twice that: a thread takes the same 32 >> LEVELS places of
// each of the 2 or 4 rows.  `rows` rows, as many as threads.
template <int LEVELS>
__device__ __forceinline__ void butterflies_rows(uint8_t* smem, uint32_t xbuf, uint32_t tid, int bit) {
    constexpr int R = 1 << LEVELS, V = 32 / R, Q = V / 4;
    const uint32_t rest = tid / R, row0 = ((rest >> bit) << (bit + LEVELS)) | (rest & ((1u << bit) - 1u));
    const uint32_t first = (xbuf + rotate_row(row0)) ^ ((tid % R) * (16u * Q)), step = 128u << bit;  // (the rows' numbers agree in their last three bits)
    f32x2 v[R][V / 2];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float4 x = *reinterpret_cast<const float4*>(smem + ((first ^ (16u * q)) + r * step));
            v[r][2 * q] = pack2(x.x, x.y);
            v[r][2 * q + 1] = pack2(x.z, x.w);
        }
    const f32x2 m2 = pack2(-1.0f, -1.0f);
#pragma unroll
    for (int h = 1; h < R; h <<= 1)
#pragma unroll
        for (int r = 0; r < R; ++r)
            if ((r & h) == 0) {
#pragma unroll
                for (int i = 0; i < V / 2; ++i) {
                    const f32x2 a = v[r][i], b = v[r + h][i];
                    v[r][i] = add2(a, b);
                    v[r + h][i] = fma2(b, m2, a);
                }
            }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            float4 x;
            unpack2(v[r][2 * q], x.x, x.y);
            unpack2(v[r][2 * q + 1], x.z, x.w);
            *reinterpret_cast<float4*>(smem + ((first ^ (16u * q)) + r * step)) = x;
        }
}

// 32 values a lane, their signs applied; blocks of 32 * T0 values, T0 a power of two that divides blockDim.x or is below 32.
// xbuf: offset in shared memory, a multiple of 128, of 32 * blockDim.x floats; the rotated values are left there, not yet scaled (FetchRotated).  `barrier`
// is called by all threads where the block has to meet (T0 > 32 only).  A lane's part of xbuf may be overwritten by its warp as
// soon as the warp is through with the function and with FetchRotated.
template <class Barrier>
__device__ __forceinline__ void rotate_lanes32(float (&x)[32], int T0, float scale, uint8_t* smem, uint32_t xbuf, float minus_zero, Barrier&& barrier) {
    const uint32_t tid = threadIdx.x, lane = tid & 31u, mine = xbuf + rotate_row(tid);
    f32x2 v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = pack2(x[i], x[i + 16]);
    butterflies32(v, 32);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        float4 y;
        unpack2(v[2 * q], y.x, y.y);
        unpack2(v[2 * q + 1], y.z, y.w);
        *reinterpret_cast<float4*>(smem + (mine ^ (16u * q))) = y;
    }
    if (T0 > 1) {
        __syncwarp();
        const uint32_t col = xbuf + (tid - lane) * 128u + lane * 4u;  // place `lane` of the warp's rows
        auto at = [&](int row) -> float& { return *reinterpret_cast<float*>(smem + ((col ^ (16u * (row & 7))) + 128u * row)); };
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = pack2(at(i), at(i + 16));
        butterflies32(v, T0);
#pragma unroll
        for (int i = 0; i < 16; ++i) unpack2(v[i], at(i), at(i + 16));
        if (T0 <= 32) {
            __syncwarp();
        } else {
            int bit = 5;
            for (; (2 << bit) < T0; bit += 2) {
                barrier();
                butterflies_rows<2>(smem, xbuf, tid, bit);
            }
            if ((1 << bit) < T0) {
                barrier();
                butterflies_rows<1>(smem, xbuf, tid, bit);
            }
            barrier();
        }
    }
    const f32x2 k2 = pack2(scale, scale);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float4 y = *reinterpret_cast<const float4*>(smem + (mine ^ (16u * q)));
        unpack2(mul2_rounded(pack2(y.x, y.y), k2, minus_zero), x[2 * q], x[2 * q + 16]);
        unpack2(mul2_rounded(pack2(y.z, y.w), k2, minus_zero), x[2 * q + 1], x[2 * q + 17]);
    }
}

// c: the lane's index in its row.  xbuf: E * blockDim.x floats, used when a block spans more than a warp,
// and for the copy of the rotated values that is left there ([i][thread]).
template <int E>
__device__ __forceinline__ void rotate_lanes(float (&x)[E], const uint32_t* s_signs, int block, float scale, int c, float* xbuf,
                                             float minus_zero) {
    constexpr int H = E / 2;
    const int tid = threadIdx.x, T = blockDim.x, T0 = block / E;
    const uint32_t sb = s_signs[c & (T0 - 1)];
    f32x2 v[H];  // values i and i + E/2
    {
        const float minus = -1.0f;
        const f32x2 m2 = pack2(minus, minus);
#pragma unroll
        for (int i = 0; i < H; ++i)  // multiplying by -1 flips the sign bit
            v[i] = pack2(__uint_as_float(__float_as_uint(x[i]) ^ ((sb >> i) << 31)),
                         __uint_as_float(__float_as_uint(x[i + H]) ^ ((sb >> (i + H)) << 31)));
#pragma unroll
        for (int h = 1; h < H; h <<= 1) {
#pragma unroll
            for (int i = 0; i < H; ++i)
                if ((i & h) == 0) {
                    const f32x2 a = v[i], b = v[i + h];
                    v[i] = add2(a, b);
                    v[i + h] = fma2(b, m2, a);  // a - b: the product is exact
                }
        }
    }
#pragma unroll
    for (int i = 0; i < H; ++i) {
        float a, b;
        unpack2(v[i], a, b);
        v[i] = pack2(__fadd_rn(a, b), __fsub_rn(a, b));
    }
    // a + b on the lane that holds a, a - b on the one that holds b: other + sgn * own
    for (int d = 1; d < T0 && d < 32; d <<= 1) {
        const float sgn = (tid & d) != 0 ? -1.0f : 1.0f;
        const f32x2 s2 = pack2(sgn, sgn);
#pragma unroll
        for (int i = 0; i < H; ++i) {
            float a, b;
            unpack2(v[i], a, b);
            v[i] = fma2(v[i], s2, pack2(__shfl_xor_sync(0xffffffffu, a, d), __shfl_xor_sync(0xffffffffu, b, d)));
        }
    }
    for (int d = 32; d < T0; d <<= 1) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < H; ++i) {
            float a, b;
            unpack2(v[i], a, b);
            xbuf[i * T + tid] = a;
            xbuf[(i + H) * T + tid] = b;
        }
        __syncthreads();
        const float sgn = (tid & d) != 0 ? -1.0f : 1.0f;
        const f32x2 s2 = pack2(sgn, sgn);
        const int partner = (tid ^ d) < T ? tid ^ d : tid;  // beyond the block: a thread without a group
#pragma unroll
        for (int i = 0; i < H; ++i) v[i] = fma2(v[i], s2, pack2(xbuf[i * T + partner], xbuf[(i + H) * T + partner]));
    }
    if (T0 > 32) __syncthreads();  // nobody reads a partner's values any more
    const f32x2 k2 = pack2(scale, scale);
#pragma unroll
    for (int i = 0; i < H; ++i) {
        unpack2(mul2_rounded(v[i], k2, minus_zero), x[i], x[i + H]);
        xbuf[i * T + tid] = x[i];
        xbuf[(i + H) * T + tid] = x[i + H];
    }
}

// |x_i| of the calling lane from the copy that rotate_lanes or rotate_lanes32 leaves at xbuf
template <int E>
struct FetchRotated {
    const uint8_t* smem;
    uint32_t xbuf;
    float scale;
    __device__ __forceinline__ float operator()(int i) const {
        if constexpr (E == 32) {
            const uint32_t at = ((xbuf + rotate_row(threadIdx.x)) ^ ((static_cast<uint32_t>(i) & 14u) << 3)) + 8u * (i & 1) + ((i & 16) >> 2);
            return fabsf(__fmul_rn(*reinterpret_cast<const float*>(smem + at), scale));
        } else {
            return fabsf(reinterpret_cast<const float*>(smem + xbuf)[i * blockDim.x + threadIdx.x]);
        }
    }
};

}  // namespace pvq
