// Lattice time stepping with several threads per mass, for populations that leave SMs idle (at
// most one robot per SM): a step's time is then its longest chain, the 13 spring evaluations that
// one thread of the per-corner kernel (step_lattice.cu) makes one after the other.
//
// A robot of nw warps of masses takes R = min(4, 32 / nw) threads per mass, each in its own set
// of nw warps ("role"): role 0 owns the mass, the others are helpers.  Per step
//   phase A: every role evaluates its share of the 13 forward directions (at most 4, 5 or 7 for
//            R = 4, 3, 2) and leaves the forces in the shared force rows; the owner sums its own;
//   phase B: the owner adds the helpers' forces and subtracts the backward springs' in direction
//            order (the loads several at a time), then updates the mass.
// The sums are formed from the same values in the same order as the per-corner kernel's: the same
// bits.  One block per robot, two barriers per step.  With dashpots the coefficient
// 2 zeta sqrt(k m / 2) of each spring is formed once instead of every step.
// What bounds it: latency (0.9 us per step of a 4x4x4 robot).  Against one thread per mass (two
// with dashpots): 30 robots 5x5x5 with dashpots, 2000 steps: 4.47 -> 2.89 ms; 16 robots 4x4x4, 500
// steps: 0.786 -> 0.453 ms; 100 robots 7x7x7 of 299 to 485 masses, 500 steps: 1.12 -> 1.06 ms.
// 1024-thread blocks (64 registers, R = 4 for up to 256 masses) measured 3 % ahead of 768 threads
// on the first, equal on the others; batches of 4 and 6 rows equal.
#include "common.cuh"
#include "physics.cuh"

namespace vx {
namespace {

constexpr int kRolesThreads = 1024;
constexpr int kGatherBatch = 6;      // force rows in flight per batch of the owner's sums

__device__ __forceinline__ void robot_sync(int nthreads)
{
    asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

// One role: directions D0 .. D0 + N - 1; role 0 (D0 == 0) owns the masses.
template <int D0, int N, bool DAMPED, bool RECORD>
__device__ __forceinline__ void run_role(const LatticeArgs& a, float4* su, int r, int lt, int nthreads)
{
    constexpr bool kOwner = D0 == 0;
    const StepConst c = a.c;
    const int nx = a.pv.dims[3 * r], ny = a.pv.dims[3 * r + 1], nz = a.pv.dims[3 * r + 2];
    const int X = nx + 1, XY = (nx + 1) * (ny + 1), C = XY * (nz + 1);
    const int64_t mo = a.pv.moff[r];
    float4* fb = su + C;                        // row 13 a + d: force on a of spring (a, d)
    float4* sv = fb + 13 * C;                   // velocities (dashpots only)
    const bool in = lt < a.pv.n_mass[r];
    const int cidx = in ? a.corner_order[mo + lt] : 0;
    const uint32_t fl = in ? a.cflags[mo + cidx] : 0u;
    const float* prm = a.prm + 39 * mo;
    float pk[N], pa[N], pb[N], cs[DAMPED ? N : 1];
    for_each_dir_in<D0, N>([&](auto t) {
        constexpr int d = decltype(t)::value, i = d - D0;
        const bool has = (fl >> d) & 1u;
        pk[i] = has ? prm[(0 * 13 + d) * C + cidx] : 0.f;
        pa[i] = has ? prm[(1 * 13 + d) * C + cidx] : 0.f;
        pb[i] = has ? prm[(2 * 13 + d) * C + cidx] : 0.f;
        if constexpr (DAMPED) cs[i] = dashpot_coefficient(pk[i], c);
    });
    float4 u = in ? a.u[mo + cidx] : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 v = in ? a.v[mo + cidx] : make_float4(0.f, 0.f, 0.f, 0.f);
    if (kOwner && in) {
        su[cidx] = u;
        if (DAMPED) sv[cidx] = v;
    }
    float2 sc = a.sc[0];
    robot_sync(nthreads);
    for (int n = 0; n < a.nsteps; ++n) {
        const float2 sc_next = a.sc[min(n + 1, a.nsteps - 1)];
        if (!kOwner && in) {                    // the owner's state after the previous step
            u = su[cidx];
            if (DAMPED) v = sv[cidx];
        }
        if (kOwner && a.ckpt_u && in && n % a.ckpt_every == 0) {   // state at the start of segment n / K
            const int64_t o = (int64_t)(n / a.ckpt_every) * a.ckpt_stride + mo + cidx;
            a.ckpt_u[o] = u;
            a.ckpt_v[o] = v;
        }
        float2 Fxy = make_float2(0.f, 0.f);
        float Fz = 0.f;
        // an absent spring takes the corner itself as its far end and has zero parameters: an
        // exact zero force, never read
        if (in) for_each_dir_in<D0, N>([&](auto t) {
            constexpr int d = decltype(t)::value, i = d - D0;
            const bool has = (fl >> d) & 1u;
            float4 ub = u;
            if (has) ub = su[cidx + lattice_offset<d>(X, XY)];
            SpringEval e = spring_eval_ends<d>(ub, u, c.edge, lattice_rest<d>(c), lattice_rest_sq<d>(c), pk[i], pa[i],
                                               pb[i], sc.x, sc.y);
            if constexpr (DAMPED) {
                float4 vb = v;
                if (has) vb = sv[cidx + lattice_offset<d>(X, XY)];
                spring_dashpot_c(e, __fsub_rn(vb.x, v.x), __fsub_rn(vb.y, v.y), __fsub_rn(vb.z, v.z), cs[i]);
            }
            if (kOwner) { Fxy = __fadd2_rn(Fxy, make_float2(e.gx, e.gy)); Fz = __fadd_rn(Fz, e.gz); }
            fb[13 * cidx + d] = make_float4(e.gx, e.gy, e.gz, e.ext);
        });
        robot_sync(nthreads);
        if (kOwner && in) {
            // the helpers' forward springs, then the backward springs (c - offset(d), c), each in
            // direction order; an absent one adds an exact zero
            for_each_batch_in<N, 13, kGatherBatch>([&](auto t0, auto cnt) {
                constexpr int d0 = decltype(t0)::value, nb = decltype(cnt)::value;
                float4 g[nb];
                for_each_dir_in<d0, nb>([&](auto t) {
                    constexpr int d = decltype(t)::value;
                    g[d - d0] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if ((fl >> d) & 1u) g[d - d0] = fb[13 * cidx + d];
                });
                for_each_dir_in<d0, nb>([&](auto t) {
                    const float4 q = g[decltype(t)::value - d0];
                    Fxy = __fadd2_rn(Fxy, make_float2(q.x, q.y)); Fz = __fadd_rn(Fz, q.z);
                });
            });
            for_each_batch_in<0, 13, kGatherBatch>([&](auto t0, auto cnt) {
                constexpr int d0 = decltype(t0)::value, nb = decltype(cnt)::value;
                float4 g[nb];
                for_each_dir_in<d0, nb>([&](auto t) {
                    constexpr int d = decltype(t)::value;
                    g[d - d0] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if ((fl >> (16 + d)) & 1u) g[d - d0] = fb[13 * (cidx - lattice_offset<d>(X, XY)) + d];
                });
                for_each_dir_in<d0, nb>([&](auto t) {
                    const float4 q = g[decltype(t)::value - d0];
                    Fxy = __ffma2_rn(make_float2(q.x, q.y), kMinusOne2, Fxy); Fz = __fsub_rn(Fz, q.z);
                });
            });
            const float4 before = u;
            const unsigned mode = mass_update(u, v, Fxy.x, Fxy.y, Fz, c);
            if constexpr (RECORD) {             // the step's inputs, for the adjoint
                const int64_t o = (int64_t)n * a.rec_stride + mo + cidx;
                a.rec_u[o] = make_float4(before.x, before.y, before.z, __uint_as_float(mode));
                a.rec_f[o] = Fxy;
            }
            su[cidx] = u;
            if (DAMPED) sv[cidx] = v;
        }
        sc = sc_next;
        robot_sync(nthreads);
    }
    if (kOwner && in) {
        a.u[mo + cidx] = u;
        a.v[mo + cidx] = v;
    }
}

template <bool DAMPED, bool RECORD>
__global__ void __launch_bounds__(kRolesThreads, 1) k_step_roles(LatticeArgs a)
{
    extern __shared__ __align__(16) float4 roles_sm[];
    const int r = a.item_robots[a.items[blockIdx.x].x];
    const int nw = (a.pv.n_mass[r] + 31) >> 5, warp = threadIdx.x >> 5;
    if (nw == 0) return;
    const int R = min(4, kRolesThreads / 32 / nw), role = warp / nw;
    const int lt = threadIdx.x - 32 * nw * role, nthreads = 32 * nw * R;
    if (role >= R) return;                      // whole warps; the barriers count the others
    auto run = [&](auto d0, auto n) {
        run_role<decltype(d0)::value, decltype(n)::value, DAMPED, RECORD>(a, roles_sm, r, lt, nthreads);
    };
    if (R == 4) {
        if (role == 0) run(DirTag<0>{}, DirTag<4>{});
        else if (role == 1) run(DirTag<4>{}, DirTag<3>{});
        else if (role == 2) run(DirTag<7>{}, DirTag<3>{});
        else run(DirTag<10>{}, DirTag<3>{});
    } else if (R == 3) {
        if (role == 0) run(DirTag<0>{}, DirTag<5>{});
        else if (role == 1) run(DirTag<5>{}, DirTag<4>{});
        else run(DirTag<9>{}, DirTag<4>{});
    } else {
        if (role == 0) run(DirTag<0>{}, DirTag<7>{});
        else run(DirTag<7>{}, DirTag<6>{});
    }
}

}  // namespace

int roles_max_masses() { return kRolesThreads / 2; }

cudaError_t launch_step_roles(const LatticeArgs& a, int max_corners, cudaStream_t s)
{
    auto kernel = a.c.damped ? k_step_roles<true, false> : (a.rec_u ? k_step_roles<false, true> : k_step_roles<false, false>);
    const size_t smem = sizeof(float4) * (a.c.damped ? 15 : 14) * (size_t)max_corners;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<a.n_items, kRolesThreads, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace vx
