// Copies between global and shared memory by the bulk-copy engine (TMA, untiled form).
// Addresses and sizes are multiples of 16 bytes.
#pragma once
#include <cstdint>

namespace pvq {

// Shared-window address of a pointer into shared memory.
__device__ __forceinline__ uint32_t shared_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbarrier_init_one(uint64_t* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(shared_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbarrier_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// Waits for the phase `parity` of the barrier; false when it has not completed after a bounded
// number of polls (the caller then leaves the kernel instead of spinning).
__device__ __forceinline__ bool mbarrier_wait(uint32_t bar, int parity, int polls = 1 << 22) {
    uint32_t done = 0;
    for (int it = 0; it < polls && !done; ++it) {
        asm volatile(
            "{\n\t"
            ".reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t"
            "}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
    }
    return done != 0u;
}

// Staging in one go: thread 0 arms a barrier with the byte count and issues the copies, global ->
// shared; the data lands while the block does its other set-up, and every thread waits on the
// barrier before it reads.
struct BulkStage {
    uint32_t bar;  // shared address of the mbarrier
};

__device__ __forceinline__ BulkStage bulk_stage_begin(uint64_t* bar_storage) {
    BulkStage st;
    st.bar = shared_addr(bar_storage);
    if (threadIdx.x == 0) {
        mbarrier_init_one(bar_storage);
        mbarrier_init_fence();
    }
    __syncthreads();
    return st;
}

// one thread: announce `total` bytes, then copy the pieces with bulk_stage_copy
__device__ __forceinline__ void bulk_stage_expect(const BulkStage& st, uint32_t total) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(st.bar), "r"(total) : "memory");
}

__device__ __forceinline__ void bulk_stage_copy(const BulkStage& st, void* dst, const void* src, uint32_t bytes) {
    const uint32_t d = shared_addr(dst);
    const uint8_t* s = static_cast<const uint8_t*>(src);
    for (uint32_t off = 0; off < bytes; off += 32768u) {
        const uint32_t n = bytes - off < 32768u ? bytes - off : 32768u;
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(d + off),
                     "l"(s + off), "r"(n), "r"(st.bar)
                     : "memory");
    }
}

// every thread: true once the announced bytes have arrived
__device__ __forceinline__ bool bulk_stage_wait(const BulkStage& st) { return mbarrier_wait(st.bar, 0); }

// Shared -> global.  The threads that wrote the data run bulk_store_fence, then a barrier, then one
// thread copies, commits, and before the shared memory is reused waits until all but the last
// PENDING groups have been read.
__device__ __forceinline__ void bulk_store_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(shared_addr(src)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void bulk_store_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(PENDING) : "memory");
}

}  // namespace pvq
