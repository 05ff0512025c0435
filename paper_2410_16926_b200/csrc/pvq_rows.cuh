// Energy of a row from its groups' energies in shared memory, by the balanced tree over
// contiguous halves (zero padded to a power of two).
#pragma once
#include "pvq_internal.cuh"

namespace pvq {

// Sum of the gp (a power of two, <= 4096) floats at p, computed by one warp; every lane gets the result.
// Lane l takes the gp / 32 consecutive values that start at l * gp / 32 (zeros beyond gp: adding
// +0 changes nothing).
__device__ __forceinline__ float warp_tree_sum(const float* p, int gp, int lane) {
    float v = 0.0f;
    if (gp <= 32) {
        v = lane < gp ? p[lane] : 0.0f;
    } else if (gp == 64) {
        const float2 x = reinterpret_cast<const float2*>(p)[lane];
        v = __fadd_rn(x.x, x.y);
    } else if (gp == 128) {
        const float4 x = reinterpret_cast<const float4*>(p)[lane];
        v = __fadd_rn(__fadd_rn(x.x, x.y), __fadd_rn(x.z, x.w));
    } else if (gp == 256) {
        const float4 x = reinterpret_cast<const float4*>(p)[2 * lane], y = reinterpret_cast<const float4*>(p)[2 * lane + 1];
        v = __fadd_rn(__fadd_rn(__fadd_rn(x.x, x.y), __fadd_rn(x.z, x.w)), __fadd_rn(__fadd_rn(y.x, y.y), __fadd_rn(y.z, y.w)));
    } else {
        // 16 Q values per lane, Q = 1, 2, 4 or 8: a tree over each run of 16, then over the runs
        const int Q = gp >> 9;
        float part[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            part[q] = 0.0f;
            if (q < Q) {
                float t[16];
                const float4* src = reinterpret_cast<const float4*>(p + (lane * Q + q) * 16);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 x = src[j];
                    t[4 * j] = x.x, t[4 * j + 1] = x.y, t[4 * j + 2] = x.z, t[4 * j + 3] = x.w;
                }
                part[q] = tree_sum<16>(t);
            }
        }
        v = tree_sum<8>(part);  // the runs beyond Q are zero
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Energy of the row rl of a tile of rpt rows, for the threads of a warp (whose rows follow one
// another): every warp sums the rows its threads sit in.  For a row of many groups that is one row;
// the same sum is then made by several warps, which costs less than a barrier.
__device__ __forceinline__ float row_energy(const float* s_ss, int gp, int rl, int rpt, int lane) {
    const int lo = __shfl_sync(0xffffffffu, rl, 0);
    const int hi = min(__shfl_sync(0xffffffffu, rl, 31), rpt - 1);
    float mine = 0.0f;
    for (int r = lo; r <= hi; ++r) {
        const float sum = warp_tree_sum(s_ss + r * gp, gp, lane);
        if (r == rl) mine = sum;
    }
    return mine;
}

}  // namespace pvq
