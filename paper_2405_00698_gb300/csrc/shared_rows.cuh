// Narrow rows in shared memory: three floats per row, the x and y of all rows first and then their
// z.  A warp's 32 rows move in three wavefronts of 128 bytes (an 8-byte and a 4-byte access per
// lane) where a float4 row with an unused lane takes four, but every access is two instructions
// with an address each: they pay where the strides are compile-time constants and all addresses
// immediate offsets (1024 robots 8x8x8, 2000 steps: 32.1 ms with float4 rows, 30.1 ms narrow, and
// no register spills); with run-time strides float4 rows stay (200 robots 6x9x5 mass-packed, 500
// steps: 2.2 ms, narrow 3.1 ms).
// Force rows are grouped by corner or by thread, 13 directions to a group: 13 is odd, so
// consecutive groups are as free of bank conflicts as consecutive rows, and the direction is an
// immediate offset.
#pragma once

namespace vx {

// The kernel's dynamic shared memory.  Rows are named by byte offsets into it rather than by
// pointers: a pointer kept in a struct loses its address space, and its loads and stores become
// generic ones (4 % of the 8x8x8 step).
extern __shared__ __align__(16) unsigned char lattice_smem[];

struct NarrowRows {
    int xy, z;

    // n rows from byte offset `base` (a multiple of 8) on: 12 n bytes
    __device__ __forceinline__ NarrowRows(int base, int n) : xy(base), z(base + 8 * n) {}
    __device__ __forceinline__ float4 load(int i) const
    {
        const float2 q = *reinterpret_cast<const float2*>(lattice_smem + xy + 8 * i);
        return make_float4(q.x, q.y, *reinterpret_cast<const float*>(lattice_smem + z + 4 * i), 0.f);
    }
    __device__ __forceinline__ void store(int i, float x, float y, float zz) const
    {
        *reinterpret_cast<float2*>(lattice_smem + xy + 8 * i) = make_float2(x, y);
        *reinterpret_cast<float*>(lattice_smem + z + 4 * i) = zz;
    }
};

}  // namespace vx
