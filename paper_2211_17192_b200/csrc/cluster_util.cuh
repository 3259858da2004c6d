// What kernels whose CTAs exchange results through one another's shared memory have in common.
#pragma once

#include "common.cuh"

namespace spec {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ uint32_t peer_u32(uint32_t addr, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// Stores into a peer's shared memory that are counted in bytes on the peer's barrier.
__device__ __forceinline__ void send2(const float* here, uint64_t* bar, int rank, float x, float y) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(peer_u32(smem_u32(here), rank)),
                 "r"(__float_as_uint(x)), "r"(__float_as_uint(y)), "r"(peer_u32(smem_u32(bar), rank))
                 : "memory");
}
__device__ __forceinline__ void send4(const float* here, uint64_t* bar, int rank, const float4& v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                     peer_u32(smem_u32(here), rank)),
                 "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)), "r"(__float_as_uint(v.w)),
                 "r"(peer_u32(smem_u32(bar), rank))
                 : "memory");
}
// Waits, with a limit in tries, for the phase of the given parity; false when the limit ran out.
__device__ __forceinline__ bool bar_wait(uint64_t* bar, uint32_t parity, uint32_t limit) {
#pragma unroll 1
    for (uint32_t spin = 0; spin < limit; ++spin) {
        uint32_t done;
        asm volatile(
            "{\n\t"
            ".reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t"
            "}"
            : "=r"(done)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

}  // namespace spec
