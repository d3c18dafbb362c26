// Segments of a persistent launch's items: the words through which a unit (segment, item) learns that
// its item's previous segment is done, and publishes its own.
#pragma once

#include <cstdint>

namespace vx {

// Polls of a segment's wait on its item's previous segment (each with a 256 ns sleep) before it
// gives up: a few seconds, far beyond any segment's duration.
constexpr uint32_t kSegSpinLimit = 1u << 22;

__device__ __forceinline__ int ld_acquire_gpu(const int* p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_gpu(int* p, int v)
{
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

}  // namespace vx
