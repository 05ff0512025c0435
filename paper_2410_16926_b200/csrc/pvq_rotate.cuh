// Random-sign Hadamard rotation of a row held E consecutive values per lane (Sec. 2.3, Sec. 3.3
// Step 1): x <- (x * s) H_B / sqrt(B) on every block of B consecutive columns, B = E * T0.  The
// Sylvester butterflies (a, b) -> (a + b, a - b) run with strides 1, 2, 4, ..., B/2: below E inside
// the lane, E .. 16 E between the lanes of a warp by shuffle (T0 divides the lanes of a row, so lane t
// and its partner t ^ d belong to the same block), larger ones through shared memory.  Every sum
// is one fp32 addition, so the result does not depend on which of the three a stage takes.
#pragma once
#include "pvq_quant.cuh"

namespace pvq {

// words of signs a lane needs, one bit a value
template <int E>
constexpr int kSignWords = (E + 31) / 32;

// The signs of one rotation block as bits, a word of E bits per lane; all threads, before a barrier.
template <int E>
__device__ __forceinline__ void pack_signs(uint32_t* s_signs, const float* signs, int block) {
    for (int j = threadIdx.x; j < block / E; j += blockDim.x) {
        uint32_t bits = 0;
#pragma unroll
        for (int i = 0; i < E; i += 4) {
            const float4 s = __ldg(reinterpret_cast<const float4*>(signs + j * E + i));
            bits |= (s.x < 0.0f ? 1u << i : 0u) | (s.y < 0.0f ? 2u << i : 0u) | (s.z < 0.0f ? 4u << i : 0u) | (s.w < 0.0f ? 8u << i : 0u);
        }
        s_signs[j] = bits;
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

// |x_i| of the calling lane from the copy rotate_lanes leaves
struct FetchRotated {
    const float* p;  // xbuf + threadIdx.x
    int T;
    __device__ __forceinline__ float operator()(int i) const { return fabsf(p[i * T]); }
};

}  // namespace pvq
