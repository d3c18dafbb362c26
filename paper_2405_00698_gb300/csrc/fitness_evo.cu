// Fitness reduction and the evolutionary step, fully on the GPU (Section II-C: "crossover,
// mutation and elite selection ... fully parallel"; Table I).
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace vx {
namespace {

// ----------------------------------------------------------------------------------------------
// Fitness: centroid x displacement, FP64 warp-shuffle block reduction, one block per robot.
// The state is the displacement u from the rest pose, so the centroid displacement is the mean
// of u_x (u = 0 at the start).
// ----------------------------------------------------------------------------------------------
// A robot of more than kFitChunk corners is cut into chunks, a block each: the chunks' sums go to
// `partial`, and the robot's last block to arrive adds them in chunk order (64 robots 40x40x40: 283
// -> 40 us, 158 MB; one robot 64x64x64: 0.43 ms -> 26 us the whole call).  kFitLoads masses per
// thread are in flight at a time.
constexpr int kFitThreads = 256;
constexpr int kFitLoads = 4;
constexpr int kFitChunk = 4096;

__global__ void __launch_bounds__(kFitThreads)
k_fitness(PopView pv, const int* __restrict__ mass_corner, const float4* __restrict__ u,
          const float4* __restrict__ x0, float dead_bound, double* partial, int* arrived, double* __restrict__ out)
{
    __shared__ double sh_sum[kFitThreads / 32];
    const int r = blockIdx.x, chunk = blockIdx.y, chunks = gridDim.y;
    const int M = pv.n_mass[r], m0 = chunk * kFitChunk, m1 = min(M, m0 + kFitChunk);
    const int64_t mo = pv.moff[r];
    double s = 0.0;
    int dead = 0;
    for (int m = m0 + threadIdx.x; m < m1; m += kFitLoads * kFitThreads) {
        float4 d[kFitLoads], q[kFitLoads];
#pragma unroll
        for (int i = 0; i < kFitLoads; ++i) {
            const int mi = m + i * kFitThreads;
            if (mi < m1) {
                const int64_t c = mo + mass_corner[mo + mi];
                d[i] = u[c];
                q[i] = x0[c];
            } else {
                d[i] = q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
#pragma unroll
        for (int i = 0; i < kFitLoads; ++i) {
            const float px = q[i].x + d[i].x, py = q[i].y + d[i].y, pz = q[i].z + d[i].z;
            if (!(fabsf(px) <= dead_bound) || !(fabsf(py) <= dead_bound) || !(fabsf(pz) <= dead_bound))
                dead = 1;   // catches NaN too
            s += (double)d[i].x;
        }
    }
    dead = __syncthreads_or(dead);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh_sum[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double t = 0.0;
    for (int i = 0; i < kFitThreads / 32; ++i) t += sh_sum[i];
    if (chunks > 1) {
        // a dead chunk's sum is marked by a NaN
        double* sums = partial + (int64_t)r * chunks;
        __stcg(sums + chunk, dead ? NAN : t);
        __threadfence();
        if (atomicAdd(arrived + r, 1) != chunks - 1) return;
        __threadfence();
        t = 0.0;
        dead = 0;
        for (int i = 0; i < chunks; ++i) {
            const double q = __ldcg(sums + i);
            dead |= isnan(q);
            t += q;
        }
        arrived[r] = 0;                                   // for the next call
    }
    out[r] = M == 0 ? 0.0 : (dead ? -INFINITY : t / M);
}

// ----------------------------------------------------------------------------------------------
// Counter-based random numbers: SplitMix64 (Steele, Lea and Flood, OOPSLA 2014).  Output
// number `ctr` of the stream seeded with `seed` is the SplitMix64 finaliser applied to
// seed + (ctr + 1) * golden-gamma.
// ----------------------------------------------------------------------------------------------
enum { kParentA = 0, kParentB = 1, kMask = 2, kMutate = 3, kU1 = 4, kU2 = 5, kCross = 6 };

// A draw is the high 32 bits of the output for (generation, child, gene, purpose), fields packed as
// generation | child (16 bits) | gene (26 bits) | purpose (3 bits): see row_draw.

// Rank by counting: the rank of robot i is the number of robots ordered before it
// (larger fitness, or equal fitness and smaller index; NaN counts as -infinity).  The fitness
// values are compared as order-preserving 64-bit integer keys (the same order and the same ties
// as the floating-point comparison; -0 and +0 share a key), which runs on the integer pipes
// instead of the few FP64 units.
__device__ __forceinline__ unsigned long long rank_key(double x)
{
    if (isnan(x)) x = -INFINITY;
    if (x == 0.0) x = 0.0;                               // -0 and +0 compare equal
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// A warp ranks kRankPer robots: its lanes share the comparisons with all others, tile by tile from
// shared memory, so 1024 robots spread over 32 blocks (one thread per robot, as before, left all but
// 4 SMs idle: 17 us; now 6.7).
constexpr int kRankThreads = 256;
constexpr int kRankPer = 4;

__global__ void __launch_bounds__(kRankThreads) k_rank(const double* __restrict__ f, int P, int* __restrict__ order)
{
    __shared__ unsigned long long tile[kRankThreads];
    const int lane = threadIdx.x & 31;
    const int i0 = (blockIdx.x * (kRankThreads / 32) + (threadIdx.x >> 5)) * kRankPer;
    unsigned long long key[kRankPer];
    int rank[kRankPer];
#pragma unroll
    for (int k = 0; k < kRankPer; ++k) {
        key[k] = i0 + k < P ? rank_key(f[i0 + k]) : ~0ull;
        rank[k] = 0;
    }
    for (int base = 0; base < P; base += kRankThreads) {
        __syncthreads();
        const int j = base + threadIdx.x;
        tile[threadIdx.x] = j < P ? rank_key(f[j]) : 0ull;   // (0: before no robot, see below)
        __syncthreads();
#pragma unroll
        for (int t = lane; t < kRankThreads; t += 32) {
            const unsigned long long kg = tile[t];
            const int jj = base + t;
#pragma unroll
            for (int k = 0; k < kRankPer; ++k) rank[k] += (kg > key[k]) || (kg == key[k] && jj < i0 + k);
        }
    }
    // entries past P have key 0, below every robot's (the least is that of -infinity), so they count
    // for none
#pragma unroll
    for (int k = 0; k < kRankPer; ++k) {
        for (int o = 16; o > 0; o >>= 1) rank[k] += __shfl_xor_sync(0xffffffffu, rank[k], o);
        if (lane == 0 && i0 + k < P) order[rank[k]] = i0 + k;
    }
}

// The generator's finaliser; high 32 bits.
constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;
__device__ __forceinline__ uint32_t mix(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return (uint32_t)((z ^ (z >> 31)) >> 32);
}

// Draw number `purpose` of gene j of a row whose counters start at `ctr0` (generation and child
// packed above gene and purpose): z = seed + (ctr + 1) gamma with the row's part added up before.
__device__ __forceinline__ uint32_t row_draw(uint64_t z0, uint32_t j, uint32_t purpose)
{
    return mix(z0 + (uint64_t)j * (8ull * kGamma) + purpose * kGamma);
}

// A block takes kChildGenes genes of a row.  Elite rows copy their genome; child rows pick parents,
// crossover mask and mutation from the counter-based generator.  A gene mutates with probability
// 0.1 or so, so nearly every warp holds a mutating lane: the warp queues its mutating genes in
// shared memory and evaluates the Gaussian for 32 of them at a time instead of for each warp of 32
// genes (1024 genomes of 20,998 genes: 152 -> 66 us, 78 with one gene per lane in flight; 107 MB
// through device memory, 16 us; the generator's 64-bit products are what is left).
constexpr int kChildThreads = 256;
constexpr int kChildGenes = 16 * kChildThreads;

__device__ __forceinline__ float mutated(uint64_t z0, uint32_t j, float g, float sigma)
{
    const float u1 = ((float)row_draw(z0, j, kU1) + 1.0f) * 2.3283064365386963e-10f;
    const float u2 = (float)row_draw(z0, j, kU2) * 2.3283064365386963e-10f;
    const float z = sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
    return g + sigma * z;
}

__global__ void __launch_bounds__(kChildThreads)
k_children(const float* __restrict__ gin, float* __restrict__ gout, const int* __restrict__ order, int P, int G,
           int E, uint64_t seed, uint64_t gen, uint32_t thresh, float sigma, uint32_t keep,
           int* __restrict__ parents, uint8_t* __restrict__ mask)
{
    __shared__ uint32_t sh_j[kChildThreads / 32][64];
    __shared__ float sh_g[kChildThreads / 32][64];
    const int c = blockIdx.y, j0 = blockIdx.x * kChildGenes, j1 = min(G, j0 + kChildGenes);
    const size_t row = (size_t)c * G;
    if (c < E) {
        const float* src = gin + (size_t)order[c] * G;
#pragma unroll 8
        for (int j = j0 + threadIdx.x; j < j1; j += kChildThreads) {
            gout[row + j] = src[j];
            if (mask) mask[row + j] = 0;
        }
        if (parents && blockIdx.x == 0 && threadIdx.x == 0) {
            parents[2 * c] = order[c];
            parents[2 * c + 1] = order[c];
        }
        return;
    }
    const uint64_t z0 = seed + (((((gen << 16) | (uint64_t)c) << 26) << 3) + 1ull) * kGamma;
    const uint32_t ua = row_draw(z0, 0, kParentA);
    const uint32_t ub = row_draw(z0, 0, kParentB);
    const int pa = order[(int)(((uint64_t)ua * (uint64_t)E) >> 32)];
    const int pb = order[(int)(((uint64_t)ub * (uint64_t)E) >> 32)];
    if (parents && blockIdx.x == 0 && threadIdx.x == 0) {
        parents[2 * c] = pa;
        parents[2 * c + 1] = pb;
    }
    const float* A = gin + (size_t)pa * G;
    const float* Bp = gin + (size_t)pb * G;
    // crossover rate below 1: some children copy parent A (a draw per child)
    const bool copy_a = keep != 0u && row_draw(z0, 0, kCross) < keep;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* qj = sh_j[warp];
    float* qg = sh_g[warp];
    int queued = 0;                                       // of the warp, below 32 between rounds
    constexpr int kU = 4;                                // genes per lane and round
    uint64_t z = z0 + (uint64_t)(j0 + 32 * kU * warp + lane) * (8ull * kGamma);
    for (int jb = j0 + 32 * kU * warp; jb < j1;
         jb += kU * kChildThreads, z += (uint64_t)kU * kChildThreads * (8ull * kGamma)) {
        bool mut[kU];
        float g[kU];
        uint32_t m[kU];
#pragma unroll
        for (int i = 0; i < kU; ++i) {
            const int j = jb + 32 * i + lane;
            const uint64_t zi = z + (uint64_t)(32 * i) * (8ull * kGamma);
            m[i] = copy_a ? 1u : mix(zi + kMask * kGamma) >> 31;
            mut[i] = j < j1 && mix(zi + kMutate * kGamma) < thresh;
            g[i] = j < j1 ? (m[i] ? A[j] : Bp[j]) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < kU; ++i) {
            const int j = jb + 32 * i + lane;
            if (j < j1 && !mut[i]) gout[row + j] = g[i];
            if (mask && j < j1) mask[row + j] = (uint8_t)m[i];
            const unsigned w = __ballot_sync(0xffffffffu, mut[i]);
            if (mut[i]) {
                const int at = queued + __popc(w & ((1u << lane) - 1u));
                qj[at] = (uint32_t)j;
                qg[at] = g[i];
            }
            queued += __popc(w);
            __syncwarp();
            if (queued >= 32) {
                queued -= 32;                             // the last 32 of the queue
                const uint32_t jm = qj[queued + lane];
                gout[row + jm] = mutated(z0, jm, qg[queued + lane], sigma);
                __syncwarp();
            }
        }
    }
    if (lane < queued) gout[row + qj[lane]] = mutated(z0, qj[lane], qg[lane], sigma);
}

// sin and cos of w t for the steps of one call, FP64 then rounded to float:
// phase = (2 pi freq) (step dt), evaluated in that order.
__global__ void k_sincos(double omega, double dt, int64_t step0, int n, float2* out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double t = __dmul_rn((double)(step0 + i), dt);
    const double ph = __dmul_rn(omega, t);
    double s, c;
    sincos(ph, &s, &c);
    out[i] = make_float2((float)s, (float)c);
}

// Gather a per-mass float4 state into packed float[3] rows; `add` (optional) is added first
// (rest lattice + displacement = position).
__global__ void k_compact(PopView pv, const int* __restrict__ mass_corner,
                          const float4* __restrict__ src, const float4* __restrict__ add,
                          float* __restrict__ dst, const int64_t* __restrict__ dst_off)
{
    const int r = blockIdx.x;
    const int M = pv.n_mass[r];
    const int64_t mo = pv.moff[r], d = dst_off[r];
    for (int m = threadIdx.x; m < M; m += blockDim.x) {
        const int64_t c = mo + mass_corner[mo + m];
        float4 p = src[c];
        if (add) {
            const float4 q = add[c];
            p.x += q.x; p.y += q.y; p.z += q.z;
        }
        dst[3 * (d + m) + 0] = p.x;
        dst[3 * (d + m) + 1] = p.y;
        dst[3 * (d + m) + 2] = p.z;
    }
}

}  // namespace

int fitness_chunks(int max_corners) { return std::max(1, (max_corners + kFitChunk - 1) / kFitChunk); }

cudaError_t launch_fitness(PopView pv, const int* mass_corner, const float4* u, const float4* x0,
                           float dead_bound, int chunks, double* partial, int* arrived, double* out, cudaStream_t s)
{
    if (pv.P == 0) return cudaSuccess;
    k_fitness<<<dim3(pv.P, chunks), kFitThreads, 0, s>>>(pv, mass_corner, u, x0, dead_bound, partial, arrived, out);
    return cudaGetLastError();
}

namespace {

// dL/df weights of the E best robots in rank order (1 for the j-th ranked robot when j < E and
// its fitness is finite, 0 for every other robot).
__global__ void k_elite_weights(const int* __restrict__ order, const double* __restrict__ f, int P, int E,
                                double* __restrict__ w)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= P) return;
    const int r = order[j];
    w[r] = (j < E && isfinite(f[r])) ? 1.0 : 0.0;
}

}  // namespace

cudaError_t launch_elite_weights(const int* order, const double* fitness, int P, int E, double* w, cudaStream_t s)
{
    k_elite_weights<<<(P + 255) / 256, 256, 0, s>>>(order, fitness, P, E, w);
    return cudaGetLastError();
}

cudaError_t launch_evo_rank(const double* fitness, int P, int* order, cudaStream_t s)
{
    constexpr int per_block = kRankThreads / 32 * kRankPer;
    k_rank<<<(P + per_block - 1) / per_block, kRankThreads, 0, s>>>(fitness, P, order);
    return cudaGetLastError();
}

cudaError_t launch_evo_children(const float* gin, float* gout, const int* order, int P, int G,
                                int E, uint64_t seed, uint64_t gen, uint32_t thresh, float sigma,
                                uint32_t keep, int* parents, uint8_t* mask, cudaStream_t s)
{
    const dim3 grid((G + kChildGenes - 1) / kChildGenes, P);
    k_children<<<grid, kChildThreads, 0, s>>>(gin, gout, order, P, G, E, seed, gen, thresh, sigma, keep, parents,
                                  mask);
    return cudaGetLastError();
}

cudaError_t launch_sincos_table(double omega, double dt, int64_t step0, int n, float2* out,
                                cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    k_sincos<<<(n + 255) / 256, 256, 0, s>>>(omega, dt, step0, n, out);
    return cudaGetLastError();
}

cudaError_t launch_compact_state(PopView pv, const int* mass_corner, const float4* src,
                                 const float4* add, float* dst, const int64_t* dst_off, cudaStream_t s)
{
    if (pv.P == 0) return cudaSuccess;
    k_compact<<<pv.P, 256, 0, s>>>(pv, mass_corner, src, add, dst, dst_off);
    return cudaGetLastError();
}

}  // namespace vx

// ----------------------------------------------------------------------------------------------
// Population diversity (logged per generation beside the fitness, Fig. 3(b) "diversity"):
//   genome: root of the mean pairwise squared distance, from the identity
//           mean_{i != j} |g_i - g_j|^2 = 2 P / (P - 1) * mean_i |g_i - mean g|^2;
//   morphology: mean over robot pairs of the fraction of voxels whose kept materials differ,
//           from per-voxel material counts c_k: differing pairs = (P^2 - sum_k c_k^2) / 2.
// FP64 accumulation, atomics into two FP64 totals.
// ----------------------------------------------------------------------------------------------
namespace vx {
namespace {

// A block takes kSpreadCols genes (or voxels), its thread rows share the population's rows; before,
// a thread took a whole column and most SMs stood empty (1024 genomes of
// 20,998 genes: 250 -> 142 us; 1024 robots 8x8x8: 412 -> 10 us).
constexpr int kSpreadCols = 32;
constexpr int kSpreadRows = 8;       // (the FP64 units bound it; 32 rows: 171 us)
constexpr int kMorphRows = 32;       // (8: 23 us)

__global__ void __launch_bounds__(kSpreadCols * kSpreadRows)
k_genome_spread(const float* __restrict__ g, int P, int G, double* __restrict__ total)
{
    __shared__ double sh[2][kSpreadRows][kSpreadCols];
    const int x = threadIdx.x, y = threadIdx.y, j = blockIdx.x * kSpreadCols + x;
    double s = 0.0, s2 = 0.0;
    if (j < G) {
#pragma unroll 8
        for (int i = y; i < P; i += kSpreadRows) {
            const double v = (double)g[(size_t)i * G + j];
            s += v;
            s2 += v * v;
        }
    }
    sh[0][y][x] = s;
    sh[1][y][x] = s2;
    __syncthreads();
    if (y != 0) return;
#pragma unroll
    for (int i = 1; i < kSpreadRows; ++i) {
        s += sh[0][i][x];
        s2 += sh[1][i][x];
    }
    double acc = s2 - s * s / P;                           // sum_i (g_ij - mean_j)^2 (0 past the last gene)
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (x == 0) atomicAdd(total, acc);
}

__global__ void __launch_bounds__(kSpreadCols * kMorphRows)
k_morph_spread(const uint8_t* __restrict__ mat, int P, int V, double* __restrict__ total)
{
    __shared__ int sh_c[kSpreadCols][kNumMat];
    const int x = threadIdx.x, y = threadIdx.y, v = blockIdx.x * kSpreadCols + x;
    if (y < kNumMat) sh_c[x][y] = 0;
    __syncthreads();
    int c[kNumMat] = {0, 0, 0, 0, 0};
    if (v < V) {
#pragma unroll 4
        for (int i = y; i < P; i += kMorphRows) {
            const int m = mat[(size_t)i * V + v] % kNumMat;
#pragma unroll
            for (int k = 0; k < kNumMat; ++k) c[k] += m == k;
        }
#pragma unroll
        for (int k = 0; k < kNumMat; ++k)
            if (c[k]) atomicAdd(&sh_c[x][k], c[k]);
    }
    __syncthreads();
    if (y != 0) return;
    double acc = 0.0;
    if (v < V) {
        double eq = 0.0;
        for (int k = 0; k < kNumMat; ++k) eq += (double)sh_c[x][k] * sh_c[x][k];
        acc = ((double)P * P - eq) * 0.5;                  // pairs of robots that differ at voxel v
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (x == 0) atomicAdd(total, acc);
}

}  // namespace

cudaError_t launch_diversity(const float* genomes, int P, int G, const uint8_t* mat, int V, double* totals,
                             cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(totals, 0, 2 * sizeof(double), s);
    if (e != cudaSuccess) return e;
    const dim3 block(kSpreadCols, kSpreadRows);
    if (genomes && G > 0) k_genome_spread<<<(G + kSpreadCols - 1) / kSpreadCols, block, 0, s>>>(genomes, P, G, totals);
    if (mat && V > 0)
        k_morph_spread<<<(V + kSpreadCols - 1) / kSpreadCols, dim3(kSpreadCols, kMorphRows), 0, s>>>(mat, P, V, totals + 1);
    return cudaGetLastError();
}

}  // namespace vx

// ----------------------------------------------------------------------------------------------
// Lamarckian gradient step on genome rows [w | kappa | phi] (gradient-assisted co-design): for
// listed row r (every row when there is no list) and gene j, genome <- clamp(fmaf(eta_seg, d, genome), lo_j, hi_j) with d the
// adjoint's gradient of voxel j mod V of robot r (robot r's voxels start at voff[r]) and eta_seg
// the step of the gene's segment.
// ----------------------------------------------------------------------------------------------
namespace vx {
namespace {

__global__ void k_grad_step(float* __restrict__ genomes, int G, int64_t V, const int64_t* __restrict__ voff,
                            const float* __restrict__ g_w, const float* __restrict__ g_kappa,
                            const float* __restrict__ g_phi, const int* __restrict__ rows, float eta_w,
                            float eta_kappa, float eta_phi, const float* __restrict__ lo,
                            const float* __restrict__ hi)
{
    const int r = rows ? rows[blockIdx.y] : blockIdx.y;
    float* row = genomes + (size_t)r * G;
    const int64_t base = voff[r];
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < G; j += gridDim.x * blockDim.x) {
        const int seg = (int)(j / V);
        const int64_t v = j - seg * V;
        const float* grad = seg == 0 ? g_w : (seg == 1 ? g_kappa : g_phi);
        const float eta = seg == 0 ? eta_w : (seg == 1 ? eta_kappa : eta_phi);
        float x = __fmaf_rn(eta, grad[base + v], row[j]);
        if (lo) x = fmaxf(x, lo[j]);
        if (hi) x = fminf(x, hi[j]);
        row[j] = x;
    }
}

}  // namespace

cudaError_t launch_grad_step(float* genomes, int G, int64_t V, const int64_t* voff, const float* g_w,
                             const float* g_kappa, const float* g_phi, const int* rows, int n_rows,
                             float eta_w, float eta_kappa, float eta_phi, const float* lo,
                             const float* hi, cudaStream_t s)
{
    if (n_rows == 0 || G == 0) return cudaSuccess;
    const int T = 256;
    int bx = (G + T - 1) / T;
    if (bx > 64) bx = 64;
    k_grad_step<<<dim3(bx, n_rows), T, 0, s>>>(genomes, G, V, voff, g_w, g_kappa, g_phi, rows, eta_w,
                                               eta_kappa, eta_phi, lo, hi);
    return cudaGetLastError();
}

}  // namespace vx
