// TMA (cp.async.bulk.tensor) and mbarrier helpers for sm_103a, written as inline
// PTX. Every wait is bounded in time; on timeout the caller records an error in the
// device status word and leaves.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace cbct {

// Device status word (owned by the geometry, passed to kernels): 0 = ok, otherwise
// an error code set by a kernel that gave up waiting (read and cleared by
// cbct_device_status).
constexpr int kStatusMbarTimeout = 1;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(
                     smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Default limit of every bounded wait in the library's kernels (2 s of %globaltimer).
constexpr uint64_t kWaitLimitNs = 2000000000ull;

// Wait for the phase of `bar` with the given parity; after limit_ns nanoseconds
// record a timeout in *status and return false.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, int *status,
                                          uint64_t limit_ns = kWaitLimitNs) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (global_ns() - t0 > limit_ns) {
            atomicExch(status, kStatusMbarTimeout);
            return false;
        }
    }
}

// Waits inside a loop that a whole warp runs with warp-wide instructions: a lane that left such a
// loop alone would leave the others waiting for it.
// By vote: every lane gets the same answer, and the warp leaves together. The MMA warps take this one:
// what they compute next stays warp-uniform, which tcgen05.mma's operands need (a lane's own answer put
// the 3x3x3 input gradient at 128^3, 32 channels, from 150 to 196 us).
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity, int *status,
                                               uint64_t limit_ns = kWaitLimitNs) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, status, limit_ns));
}
// By staying: a lane whose wait gave up runs on to the loop's end with `alive` false, only looks at
// further barriers and takes no further effect (stores, arrivals). The epilogue warps take this one:
// sixteen of them voting cost the same layer 4 % (154 against 148 us).
__device__ __forceinline__ void mbar_wait_alive(bool &alive, uint64_t *bar, uint32_t parity, int *status,
                                                uint64_t limit_ns = kWaitLimitNs) {
    alive = mbar_wait(bar, parity, status, alive ? limit_ns : 0) && alive;
}

// By leaving, for a loop whose only warp-wide step is one __syncwarp() in each iteration: the lane that
// leaves makes the barriers of its remaining iterations first (any call site counts).
__device__ __forceinline__ void leave_warp_loop(int iterations) {
#pragma unroll 1
    for (; iterations > 0; --iterations) __syncwarp();
}

// What a CTA's threads found: whether one gave up a wait and, if none did, whether one saw something
// odd in its data. Every thread gets the same answer. (A barrier's OR is a vote, not the OR of bits: two
// questions take two votes, the second only where the first found anything.)
struct CtaVote {
    bool gave_up, odd;
};
__device__ __forceinline__ CtaVote cta_vote(bool gave_up, bool odd) {
    if (!__syncthreads_or(gave_up || odd)) return CtaVote{false, false};
    const bool g = __syncthreads_or(gave_up) != 0;
    return CtaVote{g, !g};
}

// 3D tiled TMA load of a box into shared memory, completion counted on `bar`.
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int c0, int c1, int c2, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap *map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// Host: encode a tiled tensor map of rank <= 5 without swizzle, zero fill outside
// (driver entry point looked up through the runtime). strides: bytes, dims 1..rank-1.
int encode_tmap(CUtensorMap *map, CUtensorMapDataType dt, int rank, const void *base, const uint64_t *dims,
                const uint64_t *strides, const uint32_t *box);

}  // namespace cbct
