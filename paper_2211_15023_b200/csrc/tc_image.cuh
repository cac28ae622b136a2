// Helpers of the kernels that keep images resident in shared memory (tc_resnet.cu, tc_atari.cu).
#pragma once
#include <type_traits>

#include "epilogue.cuh"
#include "tc_ptx.cuh"

namespace accerl {

namespace {

// the waits of these kernels are short and on the critical path of their context: poll (try_wait itself
// suspends the warp for a while) before backing off
__device__ __forceinline__ void image_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status, int code)
{
    mbar_wait_limited(bar, parity, abort_flag, status, code, 2048, kWaitLimitPolls);
}

__device__ __forceinline__ void sts16(uint32_t addr, uint4 v)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint4 lds16(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint4 relu16(uint4 v)
{
    return make_uint4(relu_bytes(v.x), relu_bytes(v.y), relu_bytes(v.z), relu_bytes(v.w));
}

__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

template <int I>
using OpIndex = std::integral_constant<int, I>;

__host__ __device__ constexpr uint32_t idesc_for(int n)
{
    return (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ uint64_t desc(uint32_t hi, uint32_t lo) { return ((uint64_t)hi << 32) | lo; }

}  // namespace

}  // namespace accerl
