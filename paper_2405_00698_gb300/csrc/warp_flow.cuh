// Warp-to-warp ordering inside one robot's thread group, in place of group-wide barriers.
//
// The lattice kernels give consecutive masses (or corners) to consecutive threads, and a spring
// reaches at most XY + X + 1 corner ids ahead, so a warp exchanges data only with the D warps
// after it (whose displacements its forward springs read) and the D warps before it (whose force
// planes it gathers), D = (31 + XY + X + 1) / 32.  A step has two phases:
//   A: read rows of the warps w .. w + D, write this warp's plane rows;
//   B: read plane rows of the warps w - D .. w, write this warp's row.
// Before B a warp waits until w - D .. w have finished A, before the next A until w .. w + D have
// finished B.  The same two waits order the overwrites: the readers of this warp's row (A) are
// w - D .. w, and the readers of its plane rows (B) are w .. w + D.
// Each warp owns two mbarriers: `a` counts the A arrivals of w - D .. w, `b` the B arrivals of
// w .. w + D; a warp arrives with one lane per barrier.  A barrier's phase cannot complete twice
// before its owner has seen it, because the owner's own arrival is part of every phase.
// The waits are bounded; one that gives up returns false.
//
// What it gives: 1024 MLP robots 8x8x8 (20 warps each), 2000 steps: 31.7 ms with the group's
// barriers, 29.3 ms with these waits; the adjoint's sweep gains with it too.  (test_wait in place of
// try_wait: 31.5 ms.)  A group of few warps gains nothing, since nearly all of its warps wait for
// one another anyway and a barrier is quicker than an mbarrier's round trip (1000 robots 4x4x4 of
// four warps, 500 steps: 2.35 ms with barriers, 2.64 ms with these waits): the kernels with
// run-time strides keep barriers.
#pragma once

#include <cstdint>

namespace vx {

constexpr uint32_t kFlowSpinLimit = 1u << 20;
constexpr int kFlowWarps = 24;                 // warps of a 768-thread block

// The barriers of a block: per warp, `a` then `b`.
struct FlowBars {
    uint64_t bar[kFlowWarps][2];
};

__device__ __forceinline__ void flow_bar_init(uint64_t* bar, uint32_t count)
{
    const uint32_t p = (uint32_t)__cvta_generic_to_shared(bar);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(p), "r"(count) : "memory");
}

__device__ __forceinline__ void flow_bar_inval(uint64_t* bar)
{
    const uint32_t p = (uint32_t)__cvta_generic_to_shared(bar);
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(p) : "memory");
}

// Once per kernel, by the whole block (followed by a block barrier): the barriers exist, so that
// every later WarpFlow::init can invalidate them first.
__device__ __forceinline__ void flow_create(FlowBars& f)
{
    if (threadIdx.x < 2 * kFlowWarps) flow_bar_init(&f.bar[threadIdx.x >> 1][threadIdx.x & 1], 1);
}

struct WarpFlow {
    uint32_t own;    // shared address of this warp's barriers, bit 0: this lane arrives ahead
                     // (phase A), bit 1: behind (phase B)

    // This warp is warp w of the group's nw participating warps, whose barriers start at f[first];
    // reach: the largest distance in threads between the ends of a spring.
    // All barriers of the group are initialised by their owners; the caller orders that against
    // the group's first arrival with a barrier, and against the previous use with another.
    __device__ __forceinline__ void init(FlowBars& f, int first, int w, int nw, int reach)
    {
        const int lane = threadIdx.x & 31;
        const int D = min((31 + reach) >> 5, nw - 1);
        uint64_t* bar = f.bar[first + w];
        own = (uint32_t)__cvta_generic_to_shared(bar);
        if (lane == 0) {
            flow_bar_inval(bar);
            flow_bar_inval(bar + 1);
            flow_bar_init(bar, (uint32_t)(min(w, D) + 1));
            flow_bar_init(bar + 1, (uint32_t)(min(nw - 1 - w, D) + 1));
        }
        if (lane <= D && w + lane < nw) own |= 1u;
        if (lane <= D && lane <= w) own |= 2u;
    }
    __device__ __forceinline__ static void arrive(uint32_t p)
    {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(p) : "memory");
    }
    __device__ __forceinline__ static bool try_wait(uint32_t p, uint32_t parity)
    {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(p), "r"(parity)
            : "memory");
        return ok != 0;
    }
    __device__ __forceinline__ static bool wait(uint32_t p, uint32_t parity)
    {
        for (uint32_t i = 0; !try_wait(p, parity); ++i)
            if (i >= kFlowSpinLimit) return false;
        return true;
    }
    // End of phase A / B: this warp's writes are published to the warps that wait for them.
    __device__ __forceinline__ void arrive_a() const
    {
        __syncwarp();
        if (own & 1u) arrive((own & ~3u) + 16u * (threadIdx.x & 31u));
    }
    __device__ __forceinline__ void arrive_b() const
    {
        __syncwarp();
        if (own & 2u) arrive((own & ~3u) + 8u - 16u * (threadIdx.x & 31u));
    }
    __device__ __forceinline__ bool wait_a(uint32_t parity) const { return wait(own & ~3u, parity); }
    __device__ __forceinline__ bool wait_b(uint32_t parity) const { return wait((own & ~3u) + 8u, parity); }
};

}  // namespace vx
