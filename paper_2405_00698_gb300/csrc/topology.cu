// Largest connected component, mass / spring topology and initial state.  Integer work is
// deterministic and matches the definition exactly:
//   * components are 6-connected sets of occupied voxels; the kept one is the largest, ties
//     broken toward the component holding the smallest linear voxel index;
//   * masses are the corners of kept voxels in ascending corner id;
//   * springs are the distinct corner pairs of kept voxels, sorted by (a, b), with stiffness and
//     actuation terms averaged over the kept voxels sharing the pair (Section II-A, Table II).
//
// Components by union-find: every voxel starts as its own parent, each pair of occupied face
// neighbours is united by hooking the larger root under the smaller (atomicMin), so a root is
// its component's smallest voxel index.
// Everything about a corner follows from the eight voxels around it: the masks of its forward and
// backward springs are tests of their occupancy bits, and a forward spring's parameters are means
// over a fixed subset of them, so each corner loads the eight once (w, kappa, amplitude, and the
// phase's sine and cosine, formed once per voxel).
//
// Robots of at most kSmallCorners corners: one block per robot does all of it (labels in shared
// memory).  Larger robots: a few launches over (robot, chunk of voxels or corners), joined by
// per-chunk counts.  What bounds it: for large populations the writes (64 robots 40x40x40: 1.8 GB of
// parameters and springs in 0.40 ms of 0.91), for small ones the latency of the labelling and of
// the scan.  Device time, before (one block per robot, labels propagated through device memory by
// rounds, every spring's voxels read for each of three passes) -> now: 64 robots 40x40x40 6.37 ->
// 0.84 ms, 5 robots 37x22x29 2.11 -> 0.12 ms, 2048 uneven robots of 4 to 12 voxels per axis 1.09 ->
// 0.45 ms, 1024 robots 8x8x8 0.53 -> 0.25 ms, 16 robots 4x4x4 49 -> 22 us.
// (Springs stored by each thread at its own place in the list: 1.23 ms instead of 0.40 for the 64
// large robots; unions without run starts and path halving: 0.35 ms instead of 0.13.)
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "physics.cuh"

namespace vx {
namespace {

constexpr int kSmallCorners = 4096;
constexpr int kChunk = 512;          // corners per block of the large robots' launches
constexpr int kVoxChunk = 4096;      // voxels per block of their labelling

// One robot of the population.
struct Grid {
    int nx, ny, nz, V, cx, cy, cz, C;
    int64_t vo, mo, so;
    __device__ __forceinline__ Grid(const PopView& pv, int r)
        : nx(pv.dims[3 * r]), ny(pv.dims[3 * r + 1]), nz(pv.dims[3 * r + 2]), V(nx * ny * nz), cx(nx + 1), cy(ny + 1),
          cz(nz + 1), C(cx * cy * cz), vo(pv.voff[r]), mo(pv.moff[r]), so(pv.soff[r])
    {
    }
};

// Root of a's set, labels in shared or device memory.  Every walk halves its path (a node's parent
// becomes its grandparent).  Parents only decrease, so a stale value is still an ancestor and every
// walk ends; a halving store that overtakes a hook made meanwhile loses nothing, because whoever
// hooks a node that has a parent already goes on to unite that parent.
__device__ __forceinline__ int find_root(int* label, int a)
{
    volatile int* l = label;
    int p = l[a];
    while (p != a) {
        const int q = l[p];
        if (q != p) l[a] = q;
        a = p;
        p = q;
    }
    return a;
}

// The same without halving, for the pass that replaces every label by its root: a halving store
// could put an older ancestor back over a root already written.
__device__ __forceinline__ int final_root(const int* label, int a)
{
    const volatile int* l = label;
    for (int p = l[a]; p != a; p = l[a]) a = p;
    return a;
}

// Unite the sets of a and b: the larger root is hooked under the smaller; when another thread has
// hooked it meanwhile, its parent is united instead.
__device__ __forceinline__ void unite(int* label, int a, int b)
{
    a = find_root(label, a);
    b = find_root(label, b);
    while (a != b) {
        if (a < b) { const int t = a; a = b; b = t; }
        const int old = atomicMin(label + a, b);
        if (old == a) return;
        a = old;
    }
}

// Components of a run of n voxels of a robot in shared memory (label[i] for voxel v0 + i; whole
// block, n padded to whole warps by the caller's loop): first every voxel's label is the start of
// its run of occupied voxels along x within the warp's 32 voxels, then the runs are united along
// x across warps and along y and z, once per pair of runs (a pair whose x predecessors are
// occupied too has been united by those).  Neighbours before v0 are left to the caller.
__device__ __forceinline__ void label_runs(const Grid& g, const uint8_t* raw, int v0, int n, int* label)
{
    const int lane = threadIdx.x & 31;
    for (int i0 = (int)(threadIdx.x & ~31u); i0 < n; i0 += blockDim.x) {
        const int i = i0 + lane;
        const bool occ = i < n && raw[i] != 0;
        const unsigned gaps = ~__ballot_sync(0xffffffffu, occ) & ((1u << lane) - 1u);
        const int start = max(gaps ? 32 - __clz(gaps) : 0, lane - (v0 + i) % g.nx);
        if (i < n) label[i] = occ ? i - (lane - start) : -1;
    }
    __syncthreads();
    const int layer = g.nx * g.ny;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        if (label[i] < 0) continue;
        const int v = v0 + i;
        const bool before = i > 0 && v % g.nx > 0 && label[i - 1] >= 0;    // its x predecessor
        if (before && (i & 31) == 0) unite(label, i, i - 1);
        if (i >= g.nx && (v / g.nx) % g.ny > 0 && label[i - g.nx] >= 0 &&
            !(before && i > g.nx && label[i - 1 - g.nx] >= 0))
            unite(label, i, i - g.nx);
        if (i >= layer && label[i - layer] >= 0 && !(before && i > layer && label[i - 1 - layer] >= 0))
            unite(label, i, i - layer);
    }
    __syncthreads();
}

// Add the number of this warp's lanes with the same root (< 0: none) to count[root].
__device__ __forceinline__ void count_roots(int* count, int root)
{
    const unsigned peers = __match_any_sync(__activemask(), root);
    if (root >= 0 && (int)(__ffs(peers) - 1) == (int)(threadIdx.x & 31)) atomicAdd(count + root, __popc(peers));
}

__device__ __forceinline__ unsigned long long size_key(int count, int v)
{
    return ((unsigned long long)count << 32) | (unsigned)(0x7fffffff - v);
}
__device__ __forceinline__ int key_root(unsigned long long key)
{
    return key == 0ull ? -1 : 0x7fffffff - (int)(key & 0xffffffffull);
}

// Kept voxel's parameters: (w, kappa, amplitude, cos phi) and sin phi.
__device__ __forceinline__ void voxel_params_out(const TopoArgs& a, int64_t v, int m)
{
    float s, c;
    sincosf(a.phi[v], &s, &c);
    const float w = a.w[v];
    a.vox_q[v] = make_float4(w, a.kappa[v], w * a.mc.amp[m], c);
    a.vox_s[v] = s;
}

// Which of the eight voxels around a corner (bit x + 2 y + 4 z; 0: the voxel before it along the
// axis, 1: after) hold both the corner and its neighbour along sign * direction d.
__host__ __device__ constexpr unsigned around_mask(int d, int sign)
{
    unsigned m = 0;
    for (int b = 0; b < 8; ++b) {
        bool in = true;
        for (int ax = 0; ax < 3; ++ax) {
            const int o = sign * lattice_dir(d, ax), bit = (b >> ax) & 1;
            if (o > 0 && bit != 1) in = false;
            if (o < 0 && bit != 0) in = false;
        }
        if (in) m |= 1u << b;
    }
    return m;
}

// Robot-local index of voxel b around the corner at (ci, cj, ck); -1 outside the grid.
__device__ __forceinline__ int around_voxel(const Grid& g, int ci, int cj, int ck, int b)
{
    const int x = ci - 1 + (b & 1), y = cj - 1 + ((b >> 1) & 1), z = ck - 1 + (b >> 2);
    const bool in = x >= 0 && x < g.nx && y >= 0 && y < g.ny && z >= 0 && z < g.nz;
    return in ? x + g.nx * (y + g.ny * z) : -1;
}

// Occupancy bits of the voxels around a corner; kept(v): whether robot-local voxel v is kept.
template <class Kept>
__device__ __forceinline__ unsigned around_bits(const Grid& g, int c, Kept&& kept)
{
    const int ci = c % g.cx, cj = (c / g.cx) % g.cy, ck = c / (g.cx * g.cy);
    unsigned occ = 0;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const int v = around_voxel(g, ci, cj, ck, b);
        if (v >= 0 && kept(v)) occ |= 1u << b;
    }
    return occ;
}

// A corner's flags: forward springs bits 0..12, backward springs (a spring from corner c -
// offset(d) to c) bits 16..28, mass bit 31.
__device__ __forceinline__ uint32_t corner_flags(unsigned occ)
{
    uint32_t fl = occ ? 0x80000000u : 0u;
    for_each_dir([&](auto t) {
        constexpr int d = decltype(t)::value;
        constexpr unsigned f = around_mask(d, 1), b = around_mask(d, -1);
        if (occ & f) fl |= 1u << d;
        if (occ & b) fl |= 1u << (16 + d);
    });
    return fl;
}

// Initial pose of a corner: the lattice with the lowest mass layer at z = 0, at rest.  State is
// indexed by corner and kept as the displacement u from this rest lattice (small, hence precise in
// float32), with the rest height z0 in the fourth lane: u = (ux, uy, uz, z0).
__device__ __forceinline__ void corner_pose(const TopoArgs& a, const Grid& g, int c, int zmin)
{
    const int ci = c % g.cx, cj = (c / g.cx) % g.cy, ck = c / (g.cx * g.cy);
    const float4 p = make_float4((float)(ci * a.edge), (float)(cj * a.edge), (float)((ck - zmin) * a.edge), 0.f);
    a.x0[g.mo + c] = p;
    a.x[g.mo + c] = make_float4(0.f, 0.f, 0.f, p.z);
    a.v[g.mo + c] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// The forward springs of a warp's 32 corners from c0 on: the lattice kernels' parameter planes
// [3][13][C] and the robot's spring list.  The list is ordered by corner, so the warp's springs are
// one stretch of it: they are put together in shared memory (up to 416 entries: parameters, and the
// far end's mass with the lane of the near one) and leave in whole sectors.
constexpr int kWarpSprings = 13 * 32;
constexpr int kWarpSpringBytes = kWarpSprings * (16 + 4);
__device__ __forceinline__ void warp_springs(const TopoArgs& a, const Grid& g, int c0, unsigned char* sm)
{
    float4* sh_p = reinterpret_cast<float4*>(sm);
    uint32_t* sh_b = reinterpret_cast<uint32_t*>(sh_p + kWarpSprings);
    const int lane = threadIdx.x & 31, c = c0 + lane;
    const uint32_t fl = c < g.C ? a.cflags[g.mo + c] : 0u;
    float* prm = a.prm + 39 * g.mo;
    float w[8], kappa[8], amp[8], cph[8], sph[8];
    unsigned occ = 0;
    const int ci = c % g.cx, cj = (c / g.cx) % g.cy, ck = c / (g.cx * g.cy);
    if (fl & 0x1fffu) {
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const int v = around_voxel(g, ci, cj, ck, b);
            w[b] = kappa[b] = amp[b] = cph[b] = sph[b] = 0.f;
            if (v >= 0 && a.mat[g.vo + v] != 0) {
                occ |= 1u << b;
                const float4 q = a.vox_q[g.vo + v];
                w[b] = q.x; kappa[b] = q.y; amp[b] = q.z; cph[b] = q.w;
                sph[b] = a.vox_s[g.vo + v];
            }
        }
    }
    int at = c < g.C ? a.corner_spring[g.mo + c] : 0;
    const int m = c < g.C ? a.corner_mass[g.mo + c] : -1;
    const int first = __shfl_sync(0xffffffffu, at, 0);
    int total = __popc(fl & 0x1fffu);
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    at -= first;
    for_each_dir([&](auto t) {
        constexpr int d = decltype(t)::value;
        constexpr unsigned around = around_mask(d, 1);
        constexpr int cls = (lattice_dir(d, 0) != 0) + (lattice_dir(d, 1) != 0) + (lattice_dir(d, 2) != 0);
        float k = 0.f, al = 0.f, be = 0.f, L0 = 0.f;
        if ((fl >> d) & 1u) {
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                if (!((around >> b) & 1u)) continue;
                if ((occ >> b) & 1u) {
                    k = __fmaf_rn(w[b], kappa[b], k);
                    al = __fmaf_rn(amp[b], cph[b], al);
                    be = __fmaf_rn(amp[b], sph[b], be);
                }
            }
            const float inv = 1.0f / (float)__popc(occ & around);
            k *= inv; al *= inv; be *= inv;
            L0 = cls == 1 ? a.rest1 : (cls == 2 ? a.rest2 : a.rest3);
            const int b = a.corner_mass[g.mo + c + lattice_offset<d>(g.cx, g.cx * g.cy)];
            sh_p[at] = make_float4(L0, k, al, be);
            sh_b[at] = (uint32_t)b | ((uint32_t)lane << 27);
            ++at;
        }
        if (c < g.C) {
            prm[(0 * 13 + d) * g.C + c] = k;
            prm[(1 * 13 + d) * g.C + c] = al * L0;
            prm[(2 * 13 + d) * g.C + c] = be * L0;
        }
    });
    __syncwarp();
    const int64_t out = g.so + first;
    for (int i0 = 0; i0 < total; i0 += 32) {
        const int i = i0 + lane;
        const uint32_t e = i < total ? sh_b[i] : 0u;
        const int ma = __shfl_sync(0xffffffffu, m, e >> 27);
        if (i < total) {
            a.spr_ab[out + i] = make_int2(ma, (int)(e & 0x7ffffffu));
            a.spr_p[out + i] = sh_p[i];
        }
    }
    __syncwarp();                                         // the warp's entries may be overwritten
}

// The atomic kernel's copy of the springs, direction-major (all springs of direction 0, then
// direction 1, ...), and within a direction interleaved over the residue of the corner id mod 32:
// round j holds the j-th spring (by ascending corner) of every residue that has one, in residue
// order.  Consecutive entries then have corners that differ mod 32, so a warp's float atomics and
// float4 loads at either endpoint fall on distinct shared-memory banks, also in sparse robots,
// where ascending corners leave gaps.  Packed as (k, alpha L0, beta L0, corner a | corner b << 14 |
// direction << 28) from the parameter planes.  A warp takes a direction, lane l the corners
// a = l (mod 32); whole blocks only (sh: 13 ints).
__device__ void pack_springs(const TopoArgs& a, const Grid& g, int* sh)
{
    const uint32_t* cflags = a.cflags + g.mo;
    const float* prm = a.prm + 39 * g.mo;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = (blockDim.x + 31) >> 5;
    for (int d = warp; d < 13; d += nwarps) {
        int cnt = 0;
        for (int c = lane; c < g.C; c += 32) cnt += (int)((cflags[c] >> d) & 1u);
        for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        if (lane == 0) sh[d] = cnt;
    }
    __syncthreads();
    float4* pack = a.spr_pack + g.so;
    for (int d = warp; d < 13; d += nwarps) {
        int base = 0;
        for (int e = 0; e < d; ++e) base += sh[e];
        const int off = lattice_dir(d, 0) + g.cx * (lattice_dir(d, 1) + g.cy * lattice_dir(d, 2));
        const int end = base + sh[d];
        for (int c = lane; base < end; c += 32) {        // one round per turn: each lane's next spring
            while (c < g.C && !((cflags[c] >> d) & 1u)) c += 32;
            const unsigned m = __ballot_sync(0xffffffffu, c < g.C);
            if (c < g.C)
                pack[base + __popc(m & ((1u << lane) - 1u))] =
                    make_float4(prm[d * g.C + c], prm[(13 + d) * g.C + c], prm[(26 + d) * g.C + c],
                                __uint_as_float((unsigned)c | ((unsigned)(c + off) << 14) | ((unsigned)d << 28)));
            base += __popc(m);
        }
    }
}

// Exclusive prefix over the block's threads of two counts at once (each total below 2^31); the
// totals in *ta, *tb.  sh: 2 x 32 ints.
__device__ __forceinline__ int2 block_scan2(int x, int y, int2* sh, int* ta, int* tb)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    int px = x, py = y;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int qx = __shfl_up_sync(0xffffffffu, px, o), qy = __shfl_up_sync(0xffffffffu, py, o);
        if (lane >= o) { px += qx; py += qy; }
    }
    if (lane == 31) sh[warp] = make_int2(px, py);
    __syncthreads();
    int bx = 0, by = 0, sx = 0, sy = 0;
    for (int i = 0; i < nw; ++i) {
        const int2 q = sh[i];
        if (i < warp) { bx += q.x; by += q.y; }
        sx += q.x; sy += q.y;
    }
    __syncthreads();                                      // sh may be reused
    *ta = sx;
    *tb = sy;
    return make_int2(bx + px - x, by + py - y);
}

// Robots of at most kSmallCorners corners: block b takes robot a.robots[b] (NULL: robot b).
// Dynamic shared memory: labels and component sizes (ints) of the largest robot's voxels, then
// the warps' springs.
__global__ void __launch_bounds__(512) k_topology_small(TopoArgs a, int max_vox)
{
    extern __shared__ __align__(16) int topo_sm[];
    __shared__ int2 sh_scan[32];
    __shared__ unsigned long long sh_best;
    __shared__ int sh_zmin, sh_cnt[13];
    const int r = a.robots ? a.robots[blockIdx.x] : blockIdx.x;
    const int tid = threadIdx.x, T = blockDim.x;
    const Grid g(a.pv, r);
    int* label = topo_sm;
    int* count = topo_sm + max_vox;
    const uint8_t* raw = a.mat_raw + g.vo;
    for (int v = tid; v < g.V; v += T) count[v] = 0;
    if (tid == 0) { sh_best = 0ull; sh_zmin = INT_MAX; }
    label_runs(g, raw, 0, g.V, label);
    for (int v = tid; v < g.V; v += T) {
        const int root = raw[v] ? final_root(label, v) : -1;
        if (root >= 0) label[v] = root;
        count_roots(count, root);
    }
    __syncthreads();
    for (int v = tid; v < g.V; v += T)
        if (count[v] > 0) atomicMax(&sh_best, size_key(count[v], v));
    __syncthreads();
    const int best = key_root(sh_best);
    for (int v = tid; v < g.V; v += T) {
        const int m = best >= 0 && label[v] == best ? raw[v] : 0;
        a.mat[g.vo + v] = (uint8_t)m;
        if (m) voxel_params_out(a, g.vo + v, m);
    }
    // masses in ascending corner order, and where each corner's springs start
    int M = 0, S = 0;
    for (int c0 = 0; c0 < g.C; c0 += T) {
        const int c = c0 + tid;
        uint32_t fl = 0;
        if (c < g.C) {
            const unsigned occ = around_bits(g, c, [&](int v) { return best >= 0 && label[v] == best; });
            fl = corner_flags(occ);
            a.cflags[g.mo + c] = fl;
        }
        const int mass = (int)(fl >> 31);
        int tm, ts;
        const int2 p = block_scan2(mass, __popc(fl & 0x1fffu), sh_scan, &tm, &ts);
        if (c < g.C) {
            a.corner_mass[g.mo + c] = mass ? M + p.x : -1;
            a.corner_spring[g.mo + c] = S + p.y;
            if (mass) {
                a.mass_corner[g.mo + M + p.x] = c;
                if (M + p.x == 0) sh_zmin = c / (g.cx * g.cy);      // the lowest mass is the first
            }
        }
        M += tm;
        S += ts;
    }
    if (tid == 0) {
        a.pv.n_mass[r] = M;
        a.pv.n_spring[r] = S;
    }
    __syncthreads();
    const int zmin = sh_zmin == INT_MAX ? 0 : sh_zmin;
    for (int c = tid; c < g.C; c += T) corner_pose(a, g, c, zmin);
    // (the labels have been read: their shared memory takes the warps' springs)
    unsigned char* sh_springs = reinterpret_cast<unsigned char*>(topo_sm) + (tid >> 5) * kWarpSpringBytes;
    for (int c0 = tid & ~31; c0 < g.C; c0 += T) warp_springs(a, g, c0, sh_springs);
    if (!a.spr_pack) return;
    __syncthreads();
    pack_springs(a, g, sh_cnt);
}

// ---- larger robots: blockIdx.y = entry of a.robots, blockIdx.x = chunk ------------------------

// Components within chunks of kVoxChunk voxels; the robot's totals cleared.
__global__ void __launch_bounds__(512) k_topo_label(TopoArgs a)
{
    __shared__ int label[kVoxChunk];
    const int r = a.robots[blockIdx.y];
    const Grid g(a.pv, r);
    const int v0 = blockIdx.x * kVoxChunk, n = min(kVoxChunk, g.V - v0);
    if (n <= 0) return;
    const uint8_t* raw = a.mat_raw + g.vo + v0;
    if (blockIdx.x == 0 && threadIdx.x == 0) { a.best[r] = 0ull; a.zmin[r] = INT_MAX; }
    label_runs(g, raw, v0, n, label);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        a.label[g.vo + v0 + i] = raw[i] ? v0 + final_root(label, i) : -1;
        a.count[g.vo + v0 + i] = 0;
    }
}

// Unions across the chunks' borders.
__global__ void __launch_bounds__(512) k_topo_merge(TopoArgs a)
{
    const Grid g(a.pv, a.robots[blockIdx.y]);
    const int v0 = blockIdx.x * kVoxChunk, n = min(kVoxChunk, g.V - v0), layer = g.nx * g.ny;
    if (n <= 0 || v0 == 0) return;
    const uint8_t* raw = a.mat_raw + g.vo;
    int* label = a.label + g.vo;
    for (int i = threadIdx.x; i < min(n, layer); i += blockDim.x) {
        const int v = v0 + i;
        if (raw[v] == 0) continue;
        // (a pair whose x predecessors cross the border too and are occupied is theirs to unite)
        const bool before = v % g.nx > 0 && raw[v - 1];
        if (i < 1 && before) unite(label, v, v - 1);
        if (i < g.nx && (v / g.nx) % g.ny > 0 && raw[v - g.nx] && !(before && i > 0 && raw[v - 1 - g.nx]))
            unite(label, v, v - g.nx);
        if (v >= layer && raw[v - layer] && !(before && i > 0 && raw[v - 1 - layer])) unite(label, v, v - layer);
    }
}

// Component sizes.
__global__ void __launch_bounds__(512) k_topo_count(TopoArgs a)
{
    const Grid g(a.pv, a.robots[blockIdx.y]);
    const int v0 = blockIdx.x * kVoxChunk, n = min(kVoxChunk, g.V - v0);
    int* label = a.label + g.vo;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int v = v0 + i;
        int root = label[v];
        if (root >= 0) {
            root = final_root(label, root);
            label[v] = root;
        }
        count_roots(a.count + g.vo, root);
    }
}

// The kept component.
__global__ void __launch_bounds__(512) k_topo_best(TopoArgs a)
{
    const int r = a.robots[blockIdx.y];
    const Grid g(a.pv, r);
    const int v0 = blockIdx.x * kVoxChunk, n = min(kVoxChunk, g.V - v0);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int c = a.count[g.vo + v0 + i];
        if (c > 0) atomicMax(a.best + r, size_key(c, v0 + i));
    }
}

// Kept materials and voxel parameters; the corners' flags, and the chunks' masses and springs.
__global__ void __launch_bounds__(kChunk) k_topo_flags(TopoArgs a)
{
    __shared__ int2 sh_scan[32];
    const int r = a.robots[blockIdx.y];
    const Grid g(a.pv, r);
    const int c0 = blockIdx.x * kChunk, c = c0 + threadIdx.x;
    if (c0 >= g.C) return;
    const int best = key_root(a.best[r]);
    const int* label = a.label + g.vo;
    if (c < g.V) {
        const int m = best >= 0 && label[c] == best ? a.mat_raw[g.vo + c] : 0;
        a.mat[g.vo + c] = (uint8_t)m;
        if (m) voxel_params_out(a, g.vo + c, m);
    }
    uint32_t fl = 0;
    if (c < g.C) {
        const unsigned occ = around_bits(g, c, [&](int v) { return best >= 0 && label[v] == best; });
        fl = corner_flags(occ);
        a.cflags[g.mo + c] = fl;
    }
    int tm, ts;
    block_scan2((int)(fl >> 31), __popc(fl & 0x1fffu), sh_scan, &tm, &ts);
    if (threadIdx.x == 0) a.chunk[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = make_int2(tm, ts);
    if (fl >> 31) atomicMin(a.zmin + r, c / (g.cx * g.cy));
}

// Mass indices, where each corner's springs start, the initial pose.
__global__ void __launch_bounds__(kChunk) k_topo_scan(TopoArgs a)
{
    __shared__ int2 sh_scan[32];
    const int r = a.robots[blockIdx.y];
    const Grid g(a.pv, r);
    const int c0 = blockIdx.x * kChunk, c = c0 + threadIdx.x;
    if (c0 >= g.C) return;
    const int2* chunk = a.chunk + (int64_t)blockIdx.y * gridDim.x;
    int bm = 0, bs = 0;                                   // totals of the chunks before this one
    for (int i = threadIdx.x; i < (int)blockIdx.x; i += kChunk) { bm += chunk[i].x; bs += chunk[i].y; }
    int M, S;
    block_scan2(bm, bs, sh_scan, &M, &S);
    const uint32_t fl = c < g.C ? a.cflags[g.mo + c] : 0u;
    const int mass = (int)(fl >> 31);
    int tm, ts;
    const int2 p = block_scan2(mass, __popc(fl & 0x1fffu), sh_scan, &tm, &ts);
    if (c < g.C) {
        a.corner_mass[g.mo + c] = mass ? M + p.x : -1;
        a.corner_spring[g.mo + c] = S + p.y;
        if (mass) a.mass_corner[g.mo + M + p.x] = c;
        const int zmin = a.zmin[r];
        corner_pose(a, g, c, zmin == INT_MAX ? 0 : zmin);
    }
    if (threadIdx.x == 0 && c0 + kChunk >= g.C) {
        a.pv.n_mass[r] = M + tm;
        a.pv.n_spring[r] = S + ts;
    }
}

constexpr int kSpringThreads = 128;
__global__ void __launch_bounds__(kSpringThreads) k_topo_springs(TopoArgs a)
{
    __shared__ __align__(16) unsigned char sm[kSpringThreads / 32 * kWarpSpringBytes];
    const Grid g(a.pv, a.robots[blockIdx.y]);
    const int c0 = blockIdx.x * kSpringThreads + (int)(threadIdx.x & ~31u);
    if (c0 < g.C) warp_springs(a, g, c0, sm + (threadIdx.x >> 5) * kWarpSpringBytes);
}

__global__ void __launch_bounds__(416) k_topo_pack(TopoArgs a)
{
    __shared__ int sh_cnt[13];
    const Grid g(a.pv, a.robots[blockIdx.x]);
    pack_springs(a, g, sh_cnt);
}

}  // namespace

int topology_small_corners() { return kSmallCorners; }
size_t topology_chunks(int max_corners) { return (size_t)((max_corners + kChunk - 1) / kChunk); }

cudaError_t launch_topology_small(const TopoArgs& a, int n, int max_vox, int max_corners, int num_sms, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    // a block alone on its SM takes 512 threads; several share it with 256 each (1024 robots 8x8x8:
    // 0.48 ms the whole call, 0.51 with 512 and 0.54 with 128 threads)
    const int T = std::min((max_corners + 127) / 128 * 128, n <= num_sms ? 512 : 256);
    const size_t smem = std::max(2 * sizeof(int) * (size_t)max_vox, (size_t)(T / 32) * kWarpSpringBytes);
    cudaError_t e = cudaFuncSetAttribute(k_topology_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_topology_small<<<n, T, smem, s>>>(a, max_vox);
    return cudaGetLastError();
}

cudaError_t launch_topology_large(const TopoArgs& a, int n, int max_vox, int max_corners, cudaStream_t s, int* launches)
{
    if (n == 0) return cudaSuccess;
    const dim3 vox((max_vox + kVoxChunk - 1) / kVoxChunk, n), cor((max_corners + kChunk - 1) / kChunk, n);
    k_topo_label<<<vox, 512, 0, s>>>(a);
    if (vox.x > 1) k_topo_merge<<<vox, 512, 0, s>>>(a);
    k_topo_count<<<vox, 512, 0, s>>>(a);
    k_topo_best<<<vox, 512, 0, s>>>(a);
    k_topo_flags<<<cor, kChunk, 0, s>>>(a);
    k_topo_scan<<<cor, kChunk, 0, s>>>(a);
    k_topo_springs<<<dim3((max_corners + kSpringThreads - 1) / kSpringThreads, n), kSpringThreads, 0, s>>>(a);
    if (a.spr_pack) k_topo_pack<<<n, 416, 0, s>>>(a);
    *launches = 6 + (vox.x > 1) + (a.spr_pack != nullptr);
    return cudaGetLastError();
}

}  // namespace vx
