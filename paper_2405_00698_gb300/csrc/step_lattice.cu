// Lattice-gather time stepping: the deterministic, atomic-free resident path (Section II-C:
// spring updates then mass updates each step; Table II constants).
//
// A robot's masses sit on the corners of its voxel grid, and every spring joins a corner to one
// of its 13 "forward" lattice neighbours (offset d with a larger corner id).  Each thread owns
// one corner for the whole call and keeps in registers its displacement u, velocity v and the
// (k, alpha L0, beta L0) of its up-to-13 forward springs.  Per step:
//   phase A: for each forward spring (c, c + off(d)) the owner computes the force f from its own
//            u and the neighbour's u (shared memory), adds f to its own total and writes f to
//            row 13 c + d of the force rows in shared memory;
//   phase B: each thread subtracts rows 13 (c - off(d)) + d of its backward springs, then
//            applies gravity, ground contact with friction and the semi-implicit Euler update in
//            registers and publishes its new u.
// Two waits per step (barriers of the robot's group, or of neighbouring warps, WarpFlow), no
// atomics, and a fixed summation order (own forward springs by direction, then backward springs by
// direction): bit-reproducible.
// Shared memory per robot slot: u, v and 13 force rows per corner, a float4 each, or 12 bytes in the
// instantiations with compile-time strides (shared_rows.cuh).
// The state is the displacement from the rest lattice (rest height z0 in u.w), so a spring
// vector is d0 + (u_b - u_a) with d0 the exact lattice offset and the extension is formed without
// cancellation: l - L0 = (2 d0.du + du.du) / (l + L0).
#include "common.cuh"
#include "physics.cuh"
#include "segments.cuh"
#include "shared_rows.cuh"
#include "warp_flow.cuh"

namespace vx {
namespace {

constexpr int kMaxLatticeThreads = 768;
__device__ __forceinline__ void group_sync(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// DAMPED: spring dashpots of the paper's preset (a separate instantiation, so the undamped path
// keeps its registers).  RECORD: the adjoint's replay of a checkpoint segment, which also writes
// every step's state before the update with its contact mode, and the horizontal spring force
// before contact.
// IMPOSE: some robots take their contact modes from a table (sim_impose_contact_modes).
// GRID8: every item of the launch is one robot of at most 8 voxels along each axis in a 768-thread
// slot.  Its rows in shared memory lie as on the full 9 x 9 x 9 lattice of corners, so the strides
// are compile-time constants and the addresses of the 13 directions immediate offsets; the rows
// are the narrow ones, and the warps wait for their neighbours (WarpFlow) instead of for the
// group: 1024 MLP robots 8x8x8, 2000 steps: 32.8 ms with the group's barriers and float4 rows in
// 13 planes, 31.7 ms with narrow rows, 29.3 ms with the neighbour waits too; 1024 robots 7x8x7, 1000
// steps: 15.4 -> 13.8 ms.  With run-time strides
// the neighbour waits measured within 1 % of the barriers (12 % slower on groups of four warps),
// narrow rows slower.
template <bool DAMPED, bool RECORD, bool IMPOSE, bool GRID8 = false>
__global__ void __launch_bounds__(kMaxLatticeThreads, 1) k_step_lattice(LatticeArgs a)
{
    __shared__ int sh_item[4];
    __shared__ FlowBars sh_flow;
    float4* const sm4 = reinterpret_cast<float4*>(lattice_smem);
    const int tid = threadIdx.x;
    const StepConst c = a.c;
    flow_create(sh_flow);
    for (;;) {
        if (tid == 0) {
            const int it = atomicAdd(a.queue, 1);
            if (it < a.n_items) {
                const int4 item = a.items[it];
                sh_item[0] = item.x; sh_item[1] = item.y; sh_item[2] = item.z; sh_item[3] = 1;
            } else {
                sh_item[3] = 0;
            }
        }
        __syncthreads();
        if (!sh_item[3]) break;
        const int first = sh_item[0], count = sh_item[1], gthreads = sh_item[2];
        const int group = GRID8 ? 0 : tid / gthreads, lt = GRID8 ? tid : tid % gthreads;
        __syncthreads();   // everyone has read the item before thread 0 may overwrite it
        if (group < count) {
            const int r = a.item_robots[first + group];
            const int nx = a.pv.dims[3 * r], ny = a.pv.dims[3 * r + 1], nz = a.pv.dims[3 * r + 2];
            const int X = nx + 1, XY = X * (ny + 1), C = XY * (nz + 1);
            // row strides in shared memory: the grid's own, or those of 9 x 9 x 9 corners
            const int RX = GRID8 ? 9 : X, RXY = GRID8 ? 81 : XY;
            const int64_t mo = a.pv.moff[r];
            const int bar = 1 + group;
            // shared-memory slot of this group (S corners): u, v, then 13 force rows per corner
            // (row 13 a + d: force on a of spring (a, d))
            const int S = GRID8 ? kMaxLatticeThreads : gthreads;
            float4* su = sm4 + (size_t)group * kSlotVec4 * S;
            float4* sv = su + S;               // velocities (read by spring dashpots)
            float4* fb = sv + S;
            const NarrowRows nu(0, kMaxLatticeThreads), nf(12 * kMaxLatticeThreads, 13 * kMaxLatticeThreads);   // GRID8
            // thread lt owns the lt-th mass (ascending corner order: neighbouring threads touch
            // neighbouring shared-memory rows); threads past the mass count only take part in the
            // barriers
            const int M = a.pv.n_mass[r];
            const bool in = lt < M;
            const int cidx = in ? a.corner_order[mo + lt] : 0;
            const int row = GRID8 ? cidx + (cidx / X) * (9 - X) + (cidx / XY) * (81 - 9 * (ny + 1)) : cidx;
            const uint32_t fl = in ? a.cflags[mo + cidx] : 0u;
            float pk[13], pa[13], pb[13];
            const float* prm = a.prm + 39 * mo;
            for_each_dir([&](auto t) {
                constexpr int d = decltype(t)::value;
                const bool has = (fl >> d) & 1u;
                pk[d] = has ? prm[(0 * 13 + d) * C + cidx] : 0.f;
                pa[d] = has ? prm[(1 * 13 + d) * C + cidx] : 0.f;
                pb[d] = has ? prm[(2 * 13 + d) * C + cidx] : 0.f;
            });
            float4 u = in ? a.u[mo + cidx] : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 v = in ? a.v[mo + cidx] : make_float4(0.f, 0.f, 0.f, 0.f);
            const bool mass = (fl >> 31) & 1u;
            const int64_t imp = IMPOSE ? a.imp_off[r] : -1;
            auto put_u = [&] {
                if constexpr (GRID8) nu.store(row, u.x, u.y, u.z);
                else su[cidx] = u;
            };
            if (in) {
                put_u();
                if (DAMPED) sv[cidx] = v;
            }
            // whole warps past the masses take no part in the steps
            const bool warp_in = (lt & ~31) < M;
            const int nw = (M + 31) >> 5;
            WarpFlow flow;
            if (GRID8 && warp_in) flow.init(sh_flow, 0, lt >> 5, nw, 91);
            group_sync(bar, gthreads);
            // a warp of the top layer has no springs upwards: it skips those directions (1 %)
            const bool up = __any_sync(0xffffffffu, fl & 0x1ff0u);
            uint32_t ph = 0;
            if (warp_in) for (int n = 0; n < a.nsteps; ++n, ph ^= 1u) {
                if (a.ckpt_u && in && n % a.ckpt_every == 0) {   // state at the start of segment n / K
                    const int64_t o = (int64_t)(n / a.ckpt_every) * a.ckpt_stride + mo + cidx;
                    a.ckpt_u[o] = u;
                    a.ckpt_v[o] = v;
                }
                const float2 sc = a.sc[n];
                float2 Fxy = make_float2(0.f, 0.f);
                float Fz = 0.f;
                // phase A: forward springs (c, c + offset(d)).  No branch per direction: an
                // absent spring has zero parameters and takes the corner itself as its far end
                // (du = 0, so ext = 0 and the force is an exact zero that leaves the sums' bits
                // unchanged); its force row is never read.  6.5 % faster than skipping it, and
                // 2.6 % more with the far end's load predicated off (u from the register).
                auto forward = [&](auto t) {
                    constexpr int d = decltype(t)::value;
                    const bool has = (fl >> d) & 1u;
                    if constexpr (DAMPED) {
                        // with dashpots an absent spring would also load a velocity and take a
                        // square root: here the branch is cheaper (17 % on 5x5x5 robots)
                        if (!has) return;
                    }
                    float4 ub = u;
                    if (has) ub = GRID8 ? nu.load(row + lattice_offset<d>(RX, RXY)) : su[row + lattice_offset<d>(RX, RXY)];
                    SpringEval e = spring_eval_ends<d>(ub, u, c.edge, lattice_rest<d>(c), lattice_rest_sq<d>(c),
                                                      pk[d], pa[d], pb[d], sc.x, sc.y);
                    if constexpr (DAMPED) {
                        const float4 vb = sv[has ? row + lattice_offset<d>(RX, RXY) : cidx];
                        spring_dashpot(e, __fsub_rn(vb.x, v.x), __fsub_rn(vb.y, v.y), __fsub_rn(vb.z, v.z), pk[d], c);
                    }
                    Fxy = __fadd2_rn(Fxy, make_float2(e.gx, e.gy)); Fz = __fadd_rn(Fz, e.gz);
                    if constexpr (GRID8) nf.store(13 * row + d, e.gx, e.gy, e.gz);
                    else fb[13 * row + d] = make_float4(e.gx, e.gy, e.gz, e.ext);   // (any value in the unused lane)
                };
                if (in) {
                    for_each_dir_in<0, 4>(forward);
                    if (!GRID8 || up) for_each_dir_in<4, 9>(forward);
                }
                if constexpr (GRID8) {
                    flow.arrive_a();
                    if (!flow.wait_a(ph)) { atomicOr(a.status, 8); break; }
                } else {
                    group_sync(bar, 32 * nw);
                }
                // phase B: the backward springs (c - offset(d), c), then the mass update
                for_each_dir([&](auto t) {
                    constexpr int d = decltype(t)::value;
                    if (!((fl >> (16 + d)) & 1u)) return;
                    const int at = 13 * (row - lattice_offset<d>(RX, RXY)) + d;
                    const float4 g = GRID8 ? nf.load(at) : fb[at];   // force on a
                    Fxy = __ffma2_rn(make_float2(g.x, g.y), kMinusOne2, Fxy); Fz = __fsub_rn(Fz, g.z);
                });
                if (mass) {
                    int forced = -1;
                    if constexpr (IMPOSE) {
                        const int64_t gstep = a.imp_step0 + n;
                        if (imp >= 0 && gstep < a.imp_n) forced = a.imp_modes[imp + gstep * C + cidx];
                    }
                    if constexpr (RECORD) {            // replay for the adjoint: the step's inputs
                        const float4 ub4 = u;
                        const unsigned mode = IMPOSE ? mass_update_imposed(u, v, Fxy.x, Fxy.y, Fz, c, forced)
                                                     : mass_update(u, v, Fxy.x, Fxy.y, Fz, c);
                        const int64_t o = (int64_t)n * a.rec_stride + mo + cidx;
                        a.rec_u[o] = make_float4(ub4.x, ub4.y, ub4.z, __uint_as_float(mode));
                        a.rec_f[o] = Fxy;
                    } else if constexpr (IMPOSE) {
                        mass_update_imposed(u, v, Fxy.x, Fxy.y, Fz, c, forced);
                    } else {
                        mass_update(u, v, Fxy.x, Fxy.y, Fz, c);
                    }
                    put_u();
                    if (DAMPED) sv[cidx] = v;
                }
                if constexpr (GRID8) {
                    flow.arrive_b();
                    if (!flow.wait_b(ph)) { atomicOr(a.status, 8); break; }
                } else {
                    group_sync(bar, 32 * nw);
                }
            }
            if (in) {
                a.u[mo + cidx] = u;
                a.v[mo + cidx] = v;
            }
        }
        __syncthreads();
    }
}


// ----------------------------------------------------------------------------------------------
// Segmented queue for the per-corner step (undamped, no imposed modes; RECORD as
// above; GRID8 as above).  With more items than SMs a queue of whole items leaves SMs idle while
// the last wave's robots run all their steps; here every item's steps are cut into a.nseg
// segments of a.seg_steps and the queue holds the (segment, item) units in segment-major order,
// so the last wave waits for one segment.  A unit first waits (thread 0, bounded) until its item's
// previous segment has published progress[item]: that unit lies n_items places earlier in the
// queue and was taken by a running block, so the wait is normally over before it starts, and it
// cannot deadlock (every unit's dependency sits earlier in the queue).  The state passes between
// segments through global memory (stored, fenced, then published; read through L2 after the
// acquire), and every step is the per-corner kernel's arithmetic in its order: the same bits as
// one unit per item (tested).  A separate kernel rather than a template switch of the one above:
// with the switch, the unsegmented instantiations measured 2 % slower.
// ----------------------------------------------------------------------------------------------
template <bool RECORD, bool GRID8>
__global__ void __launch_bounds__(kMaxLatticeThreads, 1) k_step_lattice_seg(LatticeArgs a)
{
    // item (first robot, robots, threads), more work, -, segment, item index, segment's end
    __shared__ int sh_item[8];
    __shared__ FlowBars sh_flow;
    float4* const sm4 = reinterpret_cast<float4*>(lattice_smem);
    const int tid = threadIdx.x;
    const StepConst c = a.c;
    flow_create(sh_flow);
    for (;;) {
        if (tid == 0) {
            const int it = atomicAdd(a.queue, 1);
            if (it < a.n_items * a.nseg) {
                const int seg = it / a.n_items, ii = it - seg * a.n_items;
                const int4 item = a.items[ii];
                sh_item[0] = item.x; sh_item[1] = item.y; sh_item[2] = item.z; sh_item[3] = 1;
                sh_item[5] = seg; sh_item[6] = ii;
                sh_item[7] = min((seg + 1) * a.seg_steps, a.nsteps);
                if (seg > 0) {
                    uint32_t k = 0;
                    while (ld_acquire_gpu(a.progress + ii) < seg) {
                        if (++k >= kSegSpinLimit) { atomicOr(a.status, 8); break; }
                        __nanosleep(256);
                    }
                }
            } else {
                sh_item[3] = 0;
            }
        }
        __syncthreads();
        if (!sh_item[3]) break;
        const int first = sh_item[0], count = sh_item[1], gthreads = sh_item[2];
        const int n_begin = sh_item[5] * a.seg_steps;
        const int group = GRID8 ? 0 : tid / gthreads, lt = GRID8 ? tid : tid % gthreads;
        __syncthreads();   // everyone has read the item before thread 0 may overwrite it
        if (group < count) {
            const int r = a.item_robots[first + group];
            const int nx = a.pv.dims[3 * r], ny = a.pv.dims[3 * r + 1], nz = a.pv.dims[3 * r + 2];
            const int X = nx + 1, XY = X * (ny + 1), C = XY * (nz + 1);
            // row strides in shared memory: the grid's own, or those of 9 x 9 x 9 corners
            const int RX = GRID8 ? 9 : X, RXY = GRID8 ? 81 : XY;
            const int64_t mo = a.pv.moff[r];
            const int bar = 1 + group;
            const int S = GRID8 ? kMaxLatticeThreads : gthreads;
            float4* su = sm4 + (size_t)group * kSlotVec4 * S;
            float4* fb = su + 2 * S;           // (after u and the unused v)
            const NarrowRows nu(0, kMaxLatticeThreads), nf(12 * kMaxLatticeThreads, 13 * kMaxLatticeThreads);   // GRID8
            const int M = a.pv.n_mass[r];
            const bool in = lt < M;
            const int cidx = in ? a.corner_order[mo + lt] : 0;
            const int row = GRID8 ? cidx + (cidx / X) * (9 - X) + (cidx / XY) * (81 - 9 * (ny + 1)) : cidx;
            const uint32_t fl = in ? a.cflags[mo + cidx] : 0u;
            float pk[13], pa[13], pb[13];
            const float* prm = a.prm + 39 * mo;
            for_each_dir([&](auto t) {
                constexpr int d = decltype(t)::value;
                const bool has = (fl >> d) & 1u;
                pk[d] = has ? prm[(0 * 13 + d) * C + cidx] : 0.f;
                pa[d] = has ? prm[(1 * 13 + d) * C + cidx] : 0.f;
                pb[d] = has ? prm[(2 * 13 + d) * C + cidx] : 0.f;
            });
            // the previous segment's state, written by another SM: read through L2
            float4 u = in ? __ldcg(a.u + mo + cidx) : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 v = in ? __ldcg(a.v + mo + cidx) : make_float4(0.f, 0.f, 0.f, 0.f);
            const bool mass = (fl >> 31) & 1u;
            auto put_u = [&] {
                if constexpr (GRID8) nu.store(row, u.x, u.y, u.z);
                else su[cidx] = u;
            };
            if (in) put_u();
            const bool warp_in = (lt & ~31) < M;
            const int nw = (M + 31) >> 5;
            WarpFlow flow;
            if (GRID8 && warp_in) flow.init(sh_flow, 0, lt >> 5, nw, 91);
            group_sync(bar, gthreads);
            // a warp of the top layer has no springs upwards: it skips those directions (1 %)
            const bool up = __any_sync(0xffffffffu, fl & 0x1ff0u);
            uint32_t ph = 0;
            // (the segment's end is re-read from shared memory each step rather than held in a
            // register through the step)
            if (warp_in) for (int n = n_begin; n < *(volatile int*)&sh_item[7]; ++n, ph ^= 1u) {
                if (a.ckpt_u && in && n % a.ckpt_every == 0) {   // state at the start of segment n / K
                    const int64_t o = (int64_t)(n / a.ckpt_every) * a.ckpt_stride + mo + cidx;
                    a.ckpt_u[o] = u;
                    a.ckpt_v[o] = v;
                }
                const float2 sc = a.sc[n];
                float2 Fxy = make_float2(0.f, 0.f);
                float Fz = 0.f;
                // phase A: forward springs, branch-free (an absent spring is an exact zero force)
                auto forward = [&](auto t) {
                    constexpr int d = decltype(t)::value;
                    const bool has = (fl >> d) & 1u;
                    float4 ub = u;
                    if (has) ub = GRID8 ? nu.load(row + lattice_offset<d>(RX, RXY)) : su[row + lattice_offset<d>(RX, RXY)];
                    SpringEval e = spring_eval_ends<d>(ub, u, c.edge, lattice_rest<d>(c), lattice_rest_sq<d>(c),
                                                      pk[d], pa[d], pb[d], sc.x, sc.y);
                    Fxy = __fadd2_rn(Fxy, make_float2(e.gx, e.gy)); Fz = __fadd_rn(Fz, e.gz);
                    if constexpr (GRID8) nf.store(13 * row + d, e.gx, e.gy, e.gz);
                    else fb[13 * row + d] = make_float4(e.gx, e.gy, e.gz, e.ext);   // (any value in the unused lane)
                };
                if (in) {
                    for_each_dir_in<0, 4>(forward);
                    if (!GRID8 || up) for_each_dir_in<4, 9>(forward);
                }
                if constexpr (GRID8) {
                    flow.arrive_a();
                    if (!flow.wait_a(ph)) { atomicOr(a.status, 8); break; }
                } else {
                    group_sync(bar, 32 * nw);
                }
                // phase B: backward springs in direction order, then the mass update
                if (in) for_each_dir([&](auto t) {
                    constexpr int d = decltype(t)::value;
                    if (!((fl >> (16 + d)) & 1u)) return;
                    const int at = 13 * (row - lattice_offset<d>(RX, RXY)) + d;
                    const float4 g = GRID8 ? nf.load(at) : fb[at];   // force on a
                    Fxy = __ffma2_rn(make_float2(g.x, g.y), kMinusOne2, Fxy); Fz = __fsub_rn(Fz, g.z);
                });
                if (mass) {
                    if constexpr (RECORD) {            // the step's inputs, for the adjoint
                        const float4 ub4 = u;
                        const unsigned mode = mass_update(u, v, Fxy.x, Fxy.y, Fz, c);
                        const int64_t o = (int64_t)n * a.rec_stride + mo + cidx;
                        a.rec_u[o] = make_float4(ub4.x, ub4.y, ub4.z, __uint_as_float(mode));
                        a.rec_f[o] = Fxy;
                    } else {
                        mass_update(u, v, Fxy.x, Fxy.y, Fz, c);
                    }
                    put_u();
                }
                if constexpr (GRID8) {
                    flow.arrive_b();
                    if (!flow.wait_b(ph)) { atomicOr(a.status, 8); break; }
                } else {
                    group_sync(bar, 32 * nw);
                }
            }
            if (in) {
                a.u[mo + cidx] = u;
                a.v[mo + cidx] = v;
                __threadfence();                   // visible before the segment is published
            }
        }
        __syncthreads();
        if (tid == 0) st_release_gpu(a.progress + sh_item[6], sh_item[5] + 1);
    }
}


// ----------------------------------------------------------------------------------------------
// Direction-compacted variant of the same step.  In the per-corner kernel above a warp spends an
// evaluation on direction d whenever any of its 32 corners has a spring along d, so partly
// filled grids pay for absent springs.  Here thread t's slot d holds the t-th existing spring of
// direction d (the direction-major packed list), so along every direction the busy threads are
// 0 .. n_d - 1 and whole warps past n_d skip it: the cost of phase A follows the spring count.
// Per step:
//   phase A: slot d of every thread below n_d evaluates its spring (a, a + off(d)) from the shared
//            positions and writes the force on a to plane d at index a;
//   phase B: each mass thread adds its forward planes (index c) and subtracts its backward planes
//            (index c - off(d)) in direction order, then the mass update.
// Same arithmetic (compile-time directions), same per-mass summation order (forward by direction,
// then backward by direction) and same initial zero as the per-corner kernel: the two give
// identical bits.  It trades instructions for shared-memory traffic (phase A also reads u_a and
// phase B also reads the forward planes).
// ----------------------------------------------------------------------------------------------
template <bool DAMPED>
__global__ void __launch_bounds__(kMaxLatticeThreads, 1) k_step_lattice_compact(LatticeArgs a)
{
    extern __shared__ __align__(16) float4 sm4[];
    __shared__ int sh_item[4];
    __shared__ int sh_nd[kMaxLatticeThreads / 64][16];   // per group: springs per direction
    const int tid = threadIdx.x;
    const StepConst c = a.c;
    for (;;) {
        if (tid == 0) {
            const int it = atomicAdd(a.queue, 1);
            if (it < a.n_items) {
                const int4 item = a.items[it];
                sh_item[0] = item.x; sh_item[1] = item.y; sh_item[2] = item.z; sh_item[3] = 1;
            } else {
                sh_item[3] = 0;
            }
        }
        __syncthreads();
        if (!sh_item[3]) break;
        const int first = sh_item[0], count = sh_item[1], gthreads = sh_item[2];
        const int group = tid / gthreads, lt = tid % gthreads;
        __syncthreads();
        if (group < count) {
            const int r = a.item_robots[first + group];
            const int nx = a.pv.dims[3 * r], ny = a.pv.dims[3 * r + 1];
            const int X = nx + 1, XY = (nx + 1) * (ny + 1);
            const int64_t mo = a.pv.moff[r];
            const int bar = 1 + group;
            const int S = gthreads;
            float4* su = sm4 + (size_t)group * kSlotVec4 * S;
            float4* sv = su + S;
            float4* fb = sv + S;
            int* nd = sh_nd[group];
            const int M = a.pv.n_mass[r];
            const bool in = lt < M;
            const int cidx = in ? a.corner_order[mo + lt] : 0;
            const uint32_t fl = in ? a.cflags[mo + cidx] : 0u;
            // springs per direction = corners with that forward bit
            if (lt < 13) nd[lt] = 0;
            group_sync(bar, gthreads);
            for_each_dir([&](auto t) {
                constexpr int d = decltype(t)::value;
                const unsigned w = __ballot_sync(0xffffffffu, (fl >> d) & 1u);
                if ((lt & 31) == 0 && w) atomicAdd(&nd[d], __popc(w));
            });
            group_sync(bar, gthreads);
            // slot d: the lt-th spring of direction d, at list offset (springs of directions < d) + lt
            const float4* __restrict__ list = a.spack + a.pv.soff[r];
            float pk[13], pa[13], pb[13];
            uint32_t cpack[5];                                     // the slots' corners a, 10 bits each
            uint32_t has = 0u;
#pragma unroll
            for (int i = 0; i < 5; ++i) cpack[i] = 0u;
            int base = 0;
            for_each_dir([&](auto t) {
                constexpr int d = decltype(t)::value;
                const int n_d = nd[d];
                const bool h = lt < n_d;
                const float4 p = h ? list[base + lt] : make_float4(0.f, 0.f, 0.f, 0.f);
                pk[d] = p.x; pa[d] = p.y; pb[d] = p.z;
                cpack[d / 3] |= (__float_as_uint(p.w) & 0x3ffu) << (10 * (d % 3));
                has |= (h ? 1u : 0u) << d;
                base += n_d;
            });
            float4 u = in ? a.u[mo + cidx] : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 v = in ? a.v[mo + cidx] : make_float4(0.f, 0.f, 0.f, 0.f);
            if (in) {
                su[cidx] = u;
                if (DAMPED) sv[cidx] = v;
            }
            group_sync(bar, gthreads);
            for (int n = 0; n < a.nsteps; ++n) {
                if (a.ckpt_u && in && n % a.ckpt_every == 0) {
                    const int64_t o = (int64_t)(n / a.ckpt_every) * a.ckpt_stride + mo + cidx;
                    a.ckpt_u[o] = u;
                    a.ckpt_v[o] = v;
                }
                const float2 sc = a.sc[n];
                // phase A: this thread's slot of every direction.  The corner words are re-read
                // as opaque values every step so the compiler decodes them where used instead of
                // keeping 13 decoded corners (and their neighbours) live across the loop.
#pragma unroll
                for (int i = 0; i < 5; ++i) asm volatile("" : "+r"(cpack[i]));
                asm volatile("" : "+r"(has));
                for_each_dir([&](auto t) {
                    constexpr int d = decltype(t)::value;
                    if (!((has >> d) & 1u)) return;
                    const int ca = (int)((cpack[d / 3] >> (10 * (d % 3))) & 0x3ffu);
                    const int cb = ca + lattice_offset<d>(X, XY);
                    const float4 ua = su[ca];
                    const float4 ub = su[cb];
                    SpringEval e = spring_eval_ends<d>(ub, ua, c.edge, lattice_rest<d>(c), lattice_rest_sq<d>(c),
                                                      pk[d], pa[d], pb[d], sc.x, sc.y);
                    if constexpr (DAMPED) {
                        const float4 va = sv[ca];
                        const float4 vb = sv[cb];
                        spring_dashpot(e, __fsub_rn(vb.x, va.x), __fsub_rn(vb.y, va.y), __fsub_rn(vb.z, va.z), pk[d], c);
                    }
                    fb[d * S + ca] = make_float4(e.gx, e.gy, e.gz, e.ext);
                });
                group_sync(bar, gthreads);
                // phase B: the forces of this mass's springs in direction order, then the update
                if (in) {
                    float Fx = 0.f, Fy = 0.f, Fz = 0.f;
                    for_each_dir([&](auto t) {
                        constexpr int d = decltype(t)::value;
                        if (!((fl >> d) & 1u)) return;
                        const float4 g = fb[d * S + cidx];
                        Fx = __fadd_rn(Fx, g.x); Fy = __fadd_rn(Fy, g.y); Fz = __fadd_rn(Fz, g.z);
                    });
                    for_each_dir([&](auto t) {
                        constexpr int d = decltype(t)::value;
                        if (!((fl >> (16 + d)) & 1u)) return;
                        const float4 g = fb[d * S + cidx - lattice_offset<d>(X, XY)];
                        Fx = __fsub_rn(Fx, g.x); Fy = __fsub_rn(Fy, g.y); Fz = __fsub_rn(Fz, g.z);
                    });
                    mass_update(u, v, Fx, Fy, Fz, c);
                    su[cidx] = u;
                    if (DAMPED) sv[cidx] = v;
                }
                group_sync(bar, gthreads);
            }
            if (in) {
                a.u[mo + cidx] = u;
                a.v[mo + cidx] = v;
            }
        }
        __syncthreads();
    }
}

// ----------------------------------------------------------------------------------------------
// Mass-packed variant of the per-corner step.  The kernel above gives every robot a slot sized
// by its grid corners, and threads past the robot's mass count only join the barriers: an
// evolved 8x8x8 robot of ~400 masses leaves half of a 768-thread block idle.  Here a block's
// 768 threads are shared by several robots, each group sized by its mass count (a multiple of
// 32 threads), so a block runs as many masses as it has threads.  What makes that fit in shared
// memory is grouping the force rows by the thread slot of the spring's far end (the reader)
// instead of by corner: a robot needs 13 rows per thread (T threads) and its displacements by
// corner (C entries), not 13 rows per corner.  The far end's slot rides in
// the .w lane of its shared displacement, which the spring evaluation loads anyway.
// Per step:
//   phase A: for each forward spring (c, c + off(d)) the owner computes the force f from its own
//            displacement and the far end's, adds f to its own total, and writes f into row d
//            of the far end's slot (absent springs write a never-read row per lane);
//   phase B: each thread subtracts its own slot's rows of its backward springs (contiguous,
//            conflict-free), then the mass update.
// The sums run over the same values in the same order as the per-corner kernel (own forward
// springs by direction, then backward springs by direction): identical bits, so the adjoint's
// replay (which runs the per-corner kernel) reproduces a run of this one.
// ----------------------------------------------------------------------------------------------
template <bool DAMPED>
__global__ void __launch_bounds__(kMaxLatticeThreads, 1) k_step_lattice_packed(LatticeArgs a)
{
    __shared__ int sh_item[3];
    float4* const sm4 = reinterpret_cast<float4*>(lattice_smem);
    const int tid = threadIdx.x;
    const StepConst c = a.c;
    for (;;) {
        if (tid == 0) {
            const int it = atomicAdd(a.queue, 1);
            if (it < a.n_items) {
                const int4 item = a.items[it];
                sh_item[0] = item.x; sh_item[1] = item.y; sh_item[2] = 1;
            } else {
                sh_item[2] = 0;
            }
        }
        __syncthreads();
        if (!sh_item[2]) break;
        const int first = sh_item[0], count = sh_item[1];
        __syncthreads();   // everyone has read the item before thread 0 may overwrite it
        // this thread's group: the one whose thread range [t0, t0 + T) holds it (groups are
        // whole warps; threads past the last group only wait for the next item)
        int group = -1;
        int4 gi = make_int4(0, 0, 0, 0);
        for (int j = 0; j < count; ++j) {
            const int4 q = a.groups[first + j];
            if (tid >= q.y && tid < q.y + q.z) { group = j; gi = q; }
        }
        if (group >= 0) {
            const int r = gi.x, T = gi.z, lt = tid - gi.y;
            const int nx = a.pv.dims[3 * r], ny = a.pv.dims[3 * r + 1], nz = a.pv.dims[3 * r + 2];
            const int X = nx + 1, XY = (nx + 1) * (ny + 1), C = XY * (nz + 1);
            const int64_t mo = a.pv.moff[r];
            const int bar = 1 + group;
            float4* su = sm4 + gi.w;                 // displacements by corner, slot in .w
            float4* fb = su + C;                     // row 13 t + d: thread t's backward spring d; then 32
                                                     // rows for absent springs (never read)
            float4* sv = fb + 13 * T + 32;           // velocities by corner (dashpots only)
            const int M = a.pv.n_mass[r];
            const bool in = lt < M;
            const int cidx = in ? a.corner_order[mo + lt] : 0;
            const uint32_t fl = in ? a.cflags[mo + cidx] : 0u;
            const float slot = __int_as_float(13 * lt);   // this thread's first force row
            const int junk = 13 * T + (lt & 31);          // this lane's row for absent springs
            float pk[13], pa[13], pb[13];
            const float* prm = a.prm + 39 * mo;
            for_each_dir([&](auto t) {
                constexpr int d = decltype(t)::value;
                const bool has = (fl >> d) & 1u;
                pk[d] = has ? prm[(0 * 13 + d) * C + cidx] : 0.f;
                pa[d] = has ? prm[(1 * 13 + d) * C + cidx] : 0.f;
                pb[d] = has ? prm[(2 * 13 + d) * C + cidx] : 0.f;
            });
            float4 u = in ? a.u[mo + cidx] : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 v = in ? a.v[mo + cidx] : make_float4(0.f, 0.f, 0.f, 0.f);
            if (in) {
                su[cidx] = make_float4(u.x, u.y, u.z, slot);
                if (DAMPED) sv[cidx] = v;
            }
            group_sync(bar, T);
            for (int n = 0; n < a.nsteps; ++n) {
                if (a.ckpt_u && in && n % a.ckpt_every == 0) {   // state at the start of segment n / K
                    const int64_t o = (int64_t)(n / a.ckpt_every) * a.ckpt_stride + mo + cidx;
                    a.ckpt_u[o] = u;
                    a.ckpt_v[o] = v;
                }
                const float2 sc = a.sc[n];
                float2 Fxy = make_float2(0.f, 0.f);
                float Fz = 0.f;
                // phase A: forward springs, no branch per direction (an absent spring has zero
                // parameters and the corner itself as far end: an exact zero force)
                auto forward = [&](auto t) {
                    constexpr int d = decltype(t)::value;
                    const bool has = (fl >> d) & 1u;
                    if constexpr (DAMPED) {
                        if (!has) return;
                    }
                    float4 ub = u;
                    if (has) ub = su[cidx + lattice_offset<d>(X, XY)];
                    SpringEval e = spring_eval_ends<d>(ub, u, c.edge, lattice_rest<d>(c), lattice_rest_sq<d>(c),
                                                      pk[d], pa[d], pb[d], sc.x, sc.y);
                    if constexpr (DAMPED) {
                        const float4 vb = sv[cidx + lattice_offset<d>(X, XY)];
                        spring_dashpot(e, __fsub_rn(vb.x, v.x), __fsub_rn(vb.y, v.y), __fsub_rn(vb.z, v.z), pk[d], c);
                    }
                    Fxy = __fadd2_rn(Fxy, make_float2(e.gx, e.gy)); Fz = __fadd_rn(Fz, e.gz);
                    const int row = has ? __float_as_int(ub.w) + d : junk;
                    fb[row] = make_float4(e.gx, e.gy, e.gz, e.ext);
                };
                if (in) for_each_dir(forward);
                group_sync(bar, T);
                // phase B: backward springs (c - offset(d), c) from this slot's rows, then the update
                if (in) {
                    for_each_dir([&](auto t) {
                        constexpr int d = decltype(t)::value;
                        if (!((fl >> (16 + d)) & 1u)) return;
                        const float4 g = fb[13 * lt + d];   // force on the spring's first end
                        Fxy = __ffma2_rn(make_float2(g.x, g.y), kMinusOne2, Fxy); Fz = __fsub_rn(Fz, g.z);
                    });
                    if ((fl >> 31) & 1u) {
                        mass_update(u, v, Fxy.x, Fxy.y, Fz, c);
                        su[cidx] = make_float4(u.x, u.y, u.z, slot);
                        if (DAMPED) sv[cidx] = v;
                    }
                }
                group_sync(bar, T);
            }
            if (in) {
                a.u[mo + cidx] = u;
                a.v[mo + cidx] = v;
            }
        }
        __syncthreads();
    }
}

// ----------------------------------------------------------------------------------------------
// Segmented queue for the mass-packed step (undamped): the packed items' steps cut into a.nseg
// segments, queued segment-major, each unit waiting (bounded) for its item's previous segment
// and publishing its own, exactly as k_step_lattice_seg does for the per-corner step; the step
// itself is k_step_lattice_packed's undamped arithmetic in its order (the same bits as whole runs).
// ----------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kMaxLatticeThreads, 1) k_step_lattice_packed_seg(LatticeArgs a)
{
    // item (first group, groups), more work, -, -, segment, item index, segment's end
    __shared__ int sh_item[8];
    float4* const sm4 = reinterpret_cast<float4*>(lattice_smem);
    const int tid = threadIdx.x;
    const StepConst c = a.c;
    for (;;) {
        if (tid == 0) {
            const int it = atomicAdd(a.queue, 1);
            if (it < a.n_items * a.nseg) {
                const int seg = it / a.n_items, ii = it - seg * a.n_items;
                const int4 item = a.items[ii];
                sh_item[0] = item.x; sh_item[1] = item.y; sh_item[2] = 1;
                sh_item[5] = seg; sh_item[6] = ii;
                sh_item[7] = min((seg + 1) * a.seg_steps, a.nsteps);
                if (seg > 0) {
                    uint32_t k = 0;
                    while (ld_acquire_gpu(a.progress + ii) < seg) {
                        if (++k >= kSegSpinLimit) { atomicOr(a.status, 8); break; }
                        __nanosleep(256);
                    }
                }
            } else {
                sh_item[2] = 0;
            }
        }
        __syncthreads();
        if (!sh_item[2]) break;
        const int first = sh_item[0], count = sh_item[1];
        const int n_begin = sh_item[5] * a.seg_steps;
        __syncthreads();   // everyone has read the item before thread 0 may overwrite it
        int group = -1;
        int4 gi = make_int4(0, 0, 0, 0);
        for (int j = 0; j < count; ++j) {
            const int4 q = a.groups[first + j];
            if (tid >= q.y && tid < q.y + q.z) { group = j; gi = q; }
        }
        if (group >= 0) {
            const int r = gi.x, T = gi.z, lt = tid - gi.y;
            const int nx = a.pv.dims[3 * r], ny = a.pv.dims[3 * r + 1], nz = a.pv.dims[3 * r + 2];
            const int X = nx + 1, XY = (nx + 1) * (ny + 1), C = XY * (nz + 1);
            const int64_t mo = a.pv.moff[r];
            const int bar = 1 + group;
            float4* su = sm4 + gi.w;                 // (as in k_step_lattice_packed)
            float4* fb = su + C;
            const int M = a.pv.n_mass[r];
            const bool in = lt < M;
            const int cidx = in ? a.corner_order[mo + lt] : 0;
            const uint32_t fl = in ? a.cflags[mo + cidx] : 0u;
            const float slot = __int_as_float(13 * lt);   // this thread's first force row
            const int junk = 13 * T + (lt & 31);          // this lane's row for absent springs
            float pk[13], pa[13], pb[13];
            const float* prm = a.prm + 39 * mo;
            for_each_dir([&](auto t) {
                constexpr int d = decltype(t)::value;
                const bool has = (fl >> d) & 1u;
                pk[d] = has ? prm[(0 * 13 + d) * C + cidx] : 0.f;
                pa[d] = has ? prm[(1 * 13 + d) * C + cidx] : 0.f;
                pb[d] = has ? prm[(2 * 13 + d) * C + cidx] : 0.f;
            });
            // the previous segment's state, written by another SM: read through L2
            float4 u = in ? __ldcg(a.u + mo + cidx) : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 v = in ? __ldcg(a.v + mo + cidx) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (in) su[cidx] = make_float4(u.x, u.y, u.z, slot);
            group_sync(bar, T);
            for (int n = n_begin; n < *(volatile int*)&sh_item[7]; ++n) {
                if (a.ckpt_u && in && n % a.ckpt_every == 0) {   // state at the start of segment n / K
                    const int64_t o = (int64_t)(n / a.ckpt_every) * a.ckpt_stride + mo + cidx;
                    a.ckpt_u[o] = u;
                    a.ckpt_v[o] = v;
                }
                const float2 sc = a.sc[n];
                float2 Fxy = make_float2(0.f, 0.f);
                float Fz = 0.f;
                auto forward = [&](auto t) {
                    constexpr int d = decltype(t)::value;
                    const bool has = (fl >> d) & 1u;
                    float4 ub = u;
                    if (has) ub = su[cidx + lattice_offset<d>(X, XY)];
                    SpringEval e = spring_eval_ends<d>(ub, u, c.edge, lattice_rest<d>(c), lattice_rest_sq<d>(c),
                                                      pk[d], pa[d], pb[d], sc.x, sc.y);
                    Fxy = __fadd2_rn(Fxy, make_float2(e.gx, e.gy)); Fz = __fadd_rn(Fz, e.gz);
                    const int row = has ? __float_as_int(ub.w) + d : junk;
                    fb[row] = make_float4(e.gx, e.gy, e.gz, e.ext);
                };
                if (in) for_each_dir(forward);
                group_sync(bar, T);
                if (in) {
                    for_each_dir([&](auto t) {
                        constexpr int d = decltype(t)::value;
                        if (!((fl >> (16 + d)) & 1u)) return;
                        const float4 g = fb[13 * lt + d];   // force on the spring's first end
                        Fxy = __ffma2_rn(make_float2(g.x, g.y), kMinusOne2, Fxy); Fz = __fsub_rn(Fz, g.z);
                    });
                    if ((fl >> 31) & 1u) {
                        mass_update(u, v, Fxy.x, Fxy.y, Fz, c);
                        su[cidx] = make_float4(u.x, u.y, u.z, slot);
                    }
                }
                group_sync(bar, T);
            }
            if (in) {
                a.u[mo + cidx] = u;
                a.v[mo + cidx] = v;
                __threadfence();                   // visible before the segment is published
            }
        }
        __syncthreads();
        if (tid == 0) st_release_gpu(a.progress + sh_item[6], sh_item[5] + 1);
    }
}

}  // namespace

int lattice_max_threads() { return kMaxLatticeThreads; }

cudaError_t launch_step_lattice_packed(const LatticeArgs& a, int grid, size_t smem, cudaStream_t s)
{
    // a segmented queue (a.nseg > 1; the host sets it only for undamped robots)
    auto kernel = a.nseg > 1 ? k_step_lattice_packed_seg
                : (a.c.damped ? k_step_lattice_packed<true> : k_step_lattice_packed<false>);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<grid, kMaxLatticeThreads, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_step_lattice(const LatticeArgs& a, int grid, int threads, cudaStream_t s)
{
    size_t smem = sizeof(float4) * kSlotVec4 * (size_t)threads;
    const bool grid8 = a.grid8 && !a.c.damped;
    // a segmented queue (a.nseg > 1; the host sets it only for undamped per-corner items without
    // imposed modes, recording only on robots of at most 8 voxels along each axis)
    if (a.nseg > 1) {
        auto kseg = a.rec_u ? k_step_lattice_seg<true, true>
                  : (grid8 ? k_step_lattice_seg<false, true> : k_step_lattice_seg<false, false>);
        cudaError_t e = cudaFuncSetAttribute(kseg, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kseg<<<grid, threads, smem, s>>>(a);
        return cudaGetLastError();
    }
    auto kernel = a.imp_modes ? (a.rec_u ? k_step_lattice<false, true, true> : k_step_lattice<false, false, true>)
                : a.rec_u ? (grid8 ? k_step_lattice<false, true, false, true> : k_step_lattice<false, true, false>)
                : (grid8 && !a.spack) ? k_step_lattice<false, false, false, true>
                : a.spack ? (a.c.damped ? k_step_lattice_compact<true> : k_step_lattice_compact<false>)
                : a.c.damped ? k_step_lattice<true, false, false> : k_step_lattice<false, false, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<grid, threads, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace vx
