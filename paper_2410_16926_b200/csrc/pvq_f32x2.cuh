// Packed fp32 arithmetic (two values an instruction) and what kernels build on it.
#pragma once
#include <cstdint>

#include "pvq_internal.cuh"

namespace pvq {

// Two fp32 in a register pair: one instruction for two roundings (same results as two scalar
// operations; what it saves is issue slots).
struct f32x2 {
    unsigned long long v;
};
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 a, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f32x2 add2_rd(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
// A product on its own.  Where an addition follows, the rounding of the product has to stay: the
// assembler was seen to merge a mul.rn.f32x2 into a following add.rn.f32x2 (a group's energy then
// came out an ulp off).  mul2_rounded is a multiply-add of a -0 that it cannot see (a kernel
// argument), which changes no result and leaves nothing to merge.
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f32x2 mul2_rounded(f32x2 a, f32x2 b, float minus_zero) { return fma2(a, b, pack2(minus_zero, minus_zero)); }

// Eight coordinates, stored as y + 128 in the bytes of lo and hi, times s, as bf16.  A byte v goes into the low
// mantissa bits of 2^23: the float 2^23 + v, then minus 2^23 + 128.
__device__ __forceinline__ uint4 scale_bytes8(uint32_t lo, uint32_t hi, float s) {
    const f32x2 off = pack2(-8388736.0f, -8388736.0f), s2 = pack2(s, s);
    uint32_t o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const uint32_t w = e < 2 ? lo : hi, at = 0x7540u + 2u * (e & 1);
        float a, b;
        unpack2(mul2(add2(pack2(__uint_as_float(__byte_perm(w, 0x4B000000u, at)), __uint_as_float(__byte_perm(w, 0x4B000000u, at + 1u))), off), s2), a, b);
        o[e] = pack_bf16x2(a, b);
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

}  // namespace pvq
