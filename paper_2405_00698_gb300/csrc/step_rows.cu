// Resident time stepping of robots of more masses than a lattice block's threads: the per-mass
// scheme of step_lattice.cu with up to three masses per thread of a 1024-thread block, one robot
// per SM, in place of shared-memory float atomics (each a load, an add and a compare-and-swap, six per
// spring: step_resident.cu).
//
// Shared memory holds the displacement of every grid corner and ND force rows per corner, 12 bytes
// each.  With ND = 13 a step is one pass: every mass evaluates its 13 forward springs, keeps the
// force's sum and writes it to its rows; after a barrier it subtracts the rows of its backward
// springs and moves.  A robot whose 13 rows do not fit takes ND = 7: directions 0..6, then 7..12
// through the same rows, one more pair of barriers per step.  The sums run in a fixed order (in the
// two-pass form the first pass's forward and backward springs, then the second's), so runs repeat
// bit for bit.
// The spring parameters of a thread's first mass and of 6 of its second mass's 13 springs live in
// tensor memory (64 of its cells per thread); the others come from the parameter planes (L2) every
// step.
// With more robots than SMs a call's steps run in segments, as in k_step_lattice_seg, the robot's state
// read and published through L2.
// What bounds it: issue and the shared-memory pipe.  Against the atomic kernel, 200 steps: 500 robots
// 9x9x9 of 1000 masses 6.28 -> 3.42 ms (2.90 in segments), 300 robots 10x10x10 of 1300 masses 3.69 -> 2.73 ms, 150 robots
// 11x10x12 of 1700 masses (two passes) 2.62 -> 1.63 ms, 152 full 12x12x12 3.15 -> 2.41 ms.  The row
// addresses are formed anew in every pass: hoisted out of the steps they spilled 300 to 400 bytes.
#include "common.cuh"
#include "physics.cuh"
#include "segments.cuh"
#include "shared_rows.cuh"
#include "tmem.cuh"

namespace vx {
namespace {

constexpr int kRowsThreads = 1024;
constexpr int kRowsCols = 64;            // tensor-memory columns per thread

// Groups of directions whose parameters are loaded together: 0..3, 4..6, 7..10, 11..12.
__host__ __device__ constexpr int group_first(int g) { return g == 0 ? 0 : (g == 1 ? 4 : (g == 2 ? 7 : 11)); }
__host__ __device__ constexpr int group_size(int g) { return g == 0 ? 4 : (g == 1 ? 3 : (g == 2 ? 4 : 2)); }
// Tensor-memory column of group g of a thread's mass j (-1: from the planes), 3 per direction, in
// whole fours.
__host__ __device__ constexpr int group_col(int j, int g)
{
    return j == 0 ? (g == 0 ? 0 : (g == 1 ? 12 : (g == 2 ? 24 : 36))) : (j == 1 && g == 0 ? 44 : (j == 1 && g == 3 ? 56 : -1));
}
__host__ __device__ constexpr int group_quads(int g) { return (3 * group_size(g) + 3) / 4; }

// Force on the near end of a spring along direction D, and the mass update below, in the roundings
// of the atomic kernel (which leaves the fusing of its sums and products to the compiler; checked
// value by value), so that a robot keeps its trajectory up to the order of its sums whichever of
// the two kernels steps it: a contact decided the other way by another rounding would show long
// before the sums' order does.
struct Force {
    float x, y, z;
};
template <int D>
__device__ __forceinline__ Force spring_force(const float4& b, const float4& a, const StepConst& c, float k, float pa,
                                              float pb, float sn, float cs)
{
    constexpr int ox = lattice_dir(D, 0), oy = lattice_dir(D, 1), oz = lattice_dir(D, 2);
    const float ex = ox > 0 ? c.edge : -c.edge, ey = oy > 0 ? c.edge : -c.edge, ez = oz > 0 ? c.edge : -c.edge;
    const float2 dxy = __ffma2_rn(make_float2(a.x, a.y), kMinusOne2, make_float2(b.x, b.y));
    const float dux = dxy.x, duy = dxy.y, duz = __fsub_rn(b.z, a.z);
    const float dx = ox ? __fadd_rn(ex, dux) : dux, dy = oy ? __fadd_rn(ey, duy) : duy, dz = oz ? __fadd_rn(ez, duz) : duz;
    const float l2 = __fmaf_rn(dz, dz, __fmaf_rn(dx, dx, __fmul_rn(dy, dy)));
    const float inv = rsqrtf(l2);
    float d0du = oy ? __fmul_rn(ey, duy) : 0.f;
    if (ox) d0du = oy ? __fmaf_rn(ex, dux, d0du) : __fmul_rn(ex, dux);
    if (oz) d0du = ox || oy ? __fmaf_rn(ez, duz, d0du) : __fmul_rn(ez, duz);
    const float num = __fmaf_rn(2.0f, d0du, __fmaf_rn(duz, duz, __fmaf_rn(dux, dux, __fmul_rn(duy, duy))));
    float rcp;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rcp) : "f"(__fadd_rn(__fmul_rn(l2, inv), lattice_rest<D>(c))));
    const float ext = __fmaf_rn(num, rcp, -__fmaf_rn(pa, sn, __fmul_rn(pb, cs)));
    const float f = l2 > 1e-30f ? __fmul_rn(__fmul_rn(k, ext), inv) : 0.0f;
    return {__fmul_rn(f, dx), __fmul_rn(f, dy), __fmul_rn(f, dz)};
}

__device__ __forceinline__ void move_mass(float4& u, float4& v, float fx, float fy, float fz, const StepConst& c)
{
    fz = __fsub_rn(__fsub_rn(fz, c.weight), c.weight_lo);
    const float z = __fadd_rn(u.w, u.z);
    if (c.ground_on && z < 0.f) {
        const float fn = __fmul_rn(c.k_ground, -z);
        fz = __fmaf_rn(-c.ground_c, v.z, __fadd_rn(fz, fn));
        const float fh = __fsqrt_rn(__fmaf_rn(fx, fx, __fmul_rn(fy, fy)));
        if (fh <= __fmul_rn(c.mu_s, fn)) {
            fx = 0.f; fy = 0.f; v.x = 0.f; v.y = 0.f;
        } else {
            // kinetic friction removes at most |F_h| (saturated: F_h cancelled)
            const float q = __fdiv_rn(__fmaf_rn(c.mu_k, fn, __fmul_rn(c.mu_k_lo, fn)), fh);
            const float s = q >= 1.0f ? 0.0f : __fsub_rn(1.0f, q);
            fx = __fmul_rn(fx, s); fy = __fmul_rn(fy, s);
        }
    }
    integrate(u, v, fx, fy, fz, c);
}

// PER: masses per thread.
template <int ND, int PER>
__global__ void __launch_bounds__(kRowsThreads, 1) k_step_rows(ResidentArgs a)
{
    __shared__ int sh_robot, sh_item, sh_begin, sh_end, sh_seg;
    __shared__ uint32_t sh_tmem;
    const int tid = threadIdx.x, warp = tid >> 5;
    const StepConst c = a.c;
    if (warp == 0) tmem_alloc_warp(&sh_tmem);
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t tm = sh_tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(kRowsCols * (warp >> 2));
    const int cap = (a.max_mass + 1) & ~1;            // corners of the largest robot (even: 8-byte rows)
    const NarrowRows su(0, cap), fb(12 * cap, ND * cap);
    for (;;) {
        if (tid == 0) {
            // unit it: segment it / n_robots of a robot, waiting (bounded) for the robot's previous
            // segment, as in k_step_lattice_seg
            const int it = atomicAdd(a.queue, 1), seg = it / a.n_robots, i = it - seg * a.n_robots;
            sh_robot = seg < a.nseg ? a.order[i] : -1;
            sh_item = i;
            sh_seg = seg;
            sh_begin = seg * a.seg_steps;
            sh_end = min(sh_begin + a.seg_steps, a.nsteps);
            if (seg > 0 && seg < a.nseg) {
                uint32_t k = 0;
                while (ld_acquire_gpu(a.progress + i) < seg) {
                    if (++k >= kSegSpinLimit) { atomicOr(a.status, 8); break; }
                    __nanosleep(256);
                }
            }
        }
        __syncthreads();
        const int r = sh_robot;
        if (r < 0) break;
        const int X = a.pv.dims[3 * r] + 1, XY = X * (a.pv.dims[3 * r + 1] + 1), C = XY * (a.pv.dims[3 * r + 2] + 1);
        const int64_t mo = a.pv.moff[r];
        const int M = a.pv.n_mass[r];
        const float* prm = a.prm + 39 * mo;
        int cidx[PER];
        uint32_t fl[PER];
        float4 u[PER], v[PER];
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int m = tid + j * kRowsThreads;
            const bool in = m < M;
            cidx[j] = in ? a.corner_order[mo + m] : 0;
            fl[j] = in ? a.cflags[mo + cidx[j]] : 0u;
            // (the previous segment's state, written by another SM: read through L2)
            u[j] = in ? __ldcg(a.x + mo + cidx[j]) : make_float4(0.f, 0.f, 0.f, 0.f);
            v[j] = in ? __ldcg(a.v + mo + cidx[j]) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (in) {
                su.store(cidx[j], u[j].x, u[j].y, u[j].z);
            }
        }
        // parameters into tensor memory (absent springs: zeros)
        for_each_dir_in<0, PER>([&](auto tj) {
            constexpr int j = decltype(tj)::value;
            for_each_dir_in<0, 4>([&](auto tg) {
                constexpr int g = decltype(tg)::value, col = group_col(j, g);
                if constexpr (col >= 0) {
                    uint32_t q[4 * group_quads(g)];
#pragma unroll
                    for (int i = 0; i < 4 * group_quads(g); ++i) {
                        const int d = group_first(g) + i / 3, k = i % 3;
                        const bool has = i < 3 * group_size(g) && ((fl[j] >> d) & 1u);
                        q[i] = has ? __float_as_uint(prm[(k * 13 + d) * C + cidx[j]]) : 0u;
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < group_quads(g); ++i)
                        tmem_st4(tm + col + 4 * i, q[4 * i], q[4 * i + 1], q[4 * i + 2], q[4 * i + 3]);
                }
            });
        });
        tmem_wait_st();
        __syncthreads();
        for (int n = sh_begin; n < *(volatile int*)&sh_end; ++n) {
            const float2 sc = a.sc[n];
            float2 Fxy[PER];
            float Fz[PER];
#pragma unroll
            for (int j = 0; j < PER; ++j) { Fxy[j] = make_float2(0.f, 0.f); Fz[j] = 0.f; }
            // groups [G0, G1) of a pass that starts at direction D0
            auto pass = [&](auto tg0, auto tg1, auto td0) {
                constexpr int G0 = decltype(tg0)::value, G1 = decltype(tg1)::value, D0 = decltype(td0)::value;
                constexpr int D1 = group_first(G1 - 1) + group_size(G1 - 1);
                for_each_dir_in<0, PER>([&](auto tj) {
                    constexpr int j = decltype(tj)::value;
                    if ((tid & ~31) + j * kRowsThreads >= M) return;   // whole warps
                    // (opaque copies: the row addresses are formed here, not hoisted out of the steps
                    // and spilled)
                    int ci = cidx[j], xs = X, xys = XY;
                    asm volatile("" : "+r"(ci), "+r"(xs), "+r"(xys));
                    for_each_dir_in<G0, G1 - G0>([&](auto tg) {
                        constexpr int g = decltype(tg)::value, col = group_col(j, g), d0 = group_first(g), nd = group_size(g);
                        float p[4 * group_quads(g)];
                        if constexpr (col >= 0) {
                            uint32_t q[4 * group_quads(g)];
                            __syncwarp();
#pragma unroll
                            for (int i = 0; i < group_quads(g); ++i)
                                tmem_ld4(tm + col + 4 * i, q[4 * i], q[4 * i + 1], q[4 * i + 2], q[4 * i + 3]);
                            tmem_wait_ldn(q);
#pragma unroll
                            for (int i = 0; i < 4 * group_quads(g); ++i) p[i] = __uint_as_float(q[i]);
                        } else {
#pragma unroll
                            for (int i = 0; i < 3 * nd; ++i) {
                                const int d = d0 + i / 3;
                                p[i] = (fl[j] >> d) & 1u ? __ldg(prm + ((i % 3) * 13 + d) * C + ci) : 0.f;
                            }
                        }
                        for_each_dir_in<d0, nd>([&](auto t) {
                            constexpr int d = decltype(t)::value, i = 3 * (d - d0);
                            const bool has = (fl[j] >> d) & 1u;
                            float4 ub = u[j];
                            if (has) ub = su.load(ci + lattice_offset<d>(xs, xys));
                            const Force e = spring_force<d>(ub, u[j], c, p[i], p[i + 1], p[i + 2], sc.x, sc.y);
                            Fxy[j] = __fadd2_rn(Fxy[j], make_float2(e.x, e.y)); Fz[j] = __fadd_rn(Fz[j], e.z);
                            if (has) fb.store(ND * ci + (d - D0), e.x, e.y, e.z);
                        });
                    });
                });
                __syncthreads();
#pragma unroll
                for (int j = 0; j < PER; ++j) {
                    if (!fl[j]) continue;
                    int ci = cidx[j], xs = X, xys = XY;
                    asm volatile("" : "+r"(ci), "+r"(xs), "+r"(xys));
                    for_each_dir_in<D0, D1 - D0>([&](auto t) {
                        constexpr int d = decltype(t)::value;
                        if (!((fl[j] >> (16 + d)) & 1u)) return;
                        const float4 g = fb.load(ND * (ci - lattice_offset<d>(xs, xys)) + (d - D0));
                        Fxy[j] = __ffma2_rn(make_float2(g.x, g.y), kMinusOne2, Fxy[j]); Fz[j] = __fsub_rn(Fz[j], g.z);
                    });
                    if constexpr (D1 == 13) {
                        move_mass(u[j], v[j], Fxy[j].x, Fxy[j].y, Fz[j], c);
                        su.store(cidx[j], u[j].x, u[j].y, u[j].z);
                    }
                }
                __syncthreads();
            };
            if constexpr (ND == 13) {
                pass(DirTag<0>{}, DirTag<4>{}, DirTag<0>{});
            } else {
                pass(DirTag<0>{}, DirTag<2>{}, DirTag<0>{});
                pass(DirTag<2>{}, DirTag<4>{}, DirTag<7>{});
            }
        }
#pragma unroll
        for (int j = 0; j < PER; ++j)
            if (fl[j]) {
                a.x[mo + cidx[j]] = u[j];
                a.v[mo + cidx[j]] = v[j];
            }
        __threadfence();                              // visible before the segment is published
        __syncthreads();
        if (tid == 0) st_release_gpu(a.progress + sh_item, sh_seg + 1);
    }
    tmem_fence_before();                              // every thread has waited for its own accesses
    __syncthreads();
    tmem_fence_after();
    if (warp == 0) tmem_dealloc_warp(sh_tmem);
}

size_t rows_bytes(int nd, int corners) { return 12 * (size_t)((corners + 1) & ~1) * (nd + 1); }

}  // namespace

// Force rows per corner with which robots of up to `corners` corners fit `budget` bytes of shared
// memory: 13, 7, or 0 (none, or more masses than three per thread).
int rows_per_corner(int corners, size_t budget)
{
    if (corners > 3 * kRowsThreads) return 0;
    return rows_bytes(13, corners) <= budget ? 13 : (rows_bytes(7, corners) <= budget ? 7 : 0);
}

// a.max_mass: corners of the largest robot; max_masses: masses of the one with most; min_smem: at
// least so much shared memory per block, so that two blocks (each holds the whole tensor memory)
// never share an SM.
cudaError_t launch_step_rows(const ResidentArgs& a, int nd, int max_masses, size_t min_smem, int grid, cudaStream_t s)
{
    auto kernel = nd == 13 ? k_step_rows<13, 2>
                           : (max_masses <= 2 * kRowsThreads ? k_step_rows<7, 2> : k_step_rows<7, 3>);
    size_t smem = rows_bytes(nd, a.max_mass);
    if (smem < min_smem) smem = min_smem;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<grid, kRowsThreads, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace vx
