"""The work a user of the library has it do, as measurable cases.

A case is one pass through the public entry points (voxsim.Simulator, voxsim.fitness_function,
codesign): evaluating a population (decode, topology, stepping, fitness), one co-design generation
of genomes, gradients of the fitness, the genetic operators alone, exporting a trajectory.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2405_00698_gb300 import codesign
from paper_2405_00698_gb300 import voxsim as vs
from paper_2405_00698_gb300 import workloads as W

DIRS = ((1, 0, 0), (-1, 1, 0), (0, 1, 0), (1, 1, 0), (-1, -1, 1), (0, -1, 1), (1, -1, 1),
        (-1, 0, 1), (0, 0, 1), (1, 0, 1), (-1, 1, 1), (0, 1, 1), (1, 1, 1))
GENOME = W.GENOME_LEN


# ------------------------------------------------------------------------------------------
# The cases
# ------------------------------------------------------------------------------------------

def listed():
    return [
        # a handful of small robots over a short horizon, scored from the host: the smallest call,
        # where launches and waits count
        dict(name="evaluate_16x4", kind="evaluate", robots=16, nx=4, ny=4, nz=4, fill=0.0, steps=100,
             physics="config", where="host"),
        # the paper's own experiment: 30 robots of 5x5x5, Table II physics with dashpots, scored and bred
        dict(name="paper_30x5", kind="paper", robots=30, nx=5, ny=5, nz=5, steps=2000),
        # the main workload: one generation of MLP-encoded robots through the co-design loop
        dict(name="codesign_1024x8", kind="codesign", robots=1024, nx=8, ny=8, nz=8, steps=10000),
        # the same loop while trying things out: fewer robots, a ragged grid, a shorter horizon
        dict(name="codesign_200x6x9x5", kind="codesign", robots=200, nx=6, ny=9, nz=5, steps=500),
        # a mixed archive of body plans of many sizes scored in one call
        dict(name="uneven_2048", kind="uneven", robots=2048, lo=4, hi=12, steps=300),
        # mid-sized robots (more corners than one lattice block), densely filled
        dict(name="evaluate_150x11x10x12", kind="evaluate", robots=150, nx=11, ny=10, nz=12, fill=0.9,
             steps=200, physics="config", where="device"),
        # the large-robot workload: state streamed from device memory
        dict(name="large_64x40", kind="evaluate", robots=64, nx=40, ny=40, nz=40, fill=0.7, steps=500,
             physics="config", where="device"),
        # a few large robots on a ragged grid
        dict(name="large_5x37x22x29", kind="evaluate", robots=5, nx=37, ny=22, nz=29, fill=0.6, steps=200,
             physics="config", where="host"),
        # gradient-assisted co-design: one generation of parameter genomes with the elites' gradient step
        dict(name="lamarckian_512x8", kind="lamarckian", robots=512, nx=8, ny=8, nz=8, steps=2000, every=100),
        # the fitness as an autograd function on small robots of a ragged grid
        dict(name="gradient_40x7x5x6", kind="gradient", robots=40, nx=7, ny=5, nz=6, steps=300, every=50),
        # and on robots too large for one SM
        dict(name="gradient_4x28", kind="gradient", robots=4, nx=28, ny=28, nz=28, steps=100, every=25),
        # the genetic operators alone on a population of MLP genomes
        dict(name="evolve_1024", kind="evolve", robots=1024, genes=GENOME),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("evaluate", "evaluate", "large", "paper", "codesign", "uneven", "lamarckian", "gradient",
                       "gradient_large", "evolve"))
    axes = lambda lo, hi: dict(nx=rng.randint(lo, hi), ny=rng.randint(lo, hi), nz=rng.randint(lo, hi))  # noqa: E731
    if kind == "evaluate":
        return dict(kind="evaluate", robots=_log(rng, 12, 1200), **axes(3, 12), fill=rng.choice((0.0, 0.5, 0.7, 0.9)),
                    steps=_log(rng, 60, 400), physics="config", where=rng.choice(("host", "device")))
    if kind == "large":
        return dict(kind="evaluate", robots=_log(rng, 2, 48), **axes(17, 40), fill=rng.choice((0.6, 0.7, 0.85)),
                    steps=_log(rng, 50, 300), physics="config", where=rng.choice(("host", "device")))
    if kind == "paper":
        return dict(kind="paper", robots=_log(rng, 16, 300), **axes(4, 7), steps=_log(rng, 500, 3000))
    if kind == "codesign":
        return dict(kind="codesign", robots=_log(rng, 64, 1024), **axes(4, 8), steps=_log(rng, 300, 5000))
    if kind == "uneven":
        return dict(kind="uneven", robots=_log(rng, 100, 2048), lo=rng.randint(3, 6), hi=rng.randint(8, 13),
                    steps=_log(rng, 50, 300))
    if kind == "lamarckian":
        return dict(kind="lamarckian", robots=_log(rng, 64, 512), **axes(4, 8), steps=_log(rng, 200, 1500),
                    every=rng.choice((50, 100)))
    if kind == "gradient":
        return dict(kind="gradient", robots=_log(rng, 8, 300), **axes(3, 8), steps=_log(rng, 60, 400),
                    every=rng.choice((20, 50, 100)))
    if kind == "gradient_large":
        return dict(kind="gradient", robots=_log(rng, 1, 8), **axes(14, 30), steps=_log(rng, 20, 120),
                    every=rng.choice((10, 25, 50)))
    return dict(kind="evolve", robots=_log(rng, 30, 2000), genes=rng.choice((GENOME, _log(rng, 300, 21000))))


# ------------------------------------------------------------------------------------------
# Inputs and one pass
# ------------------------------------------------------------------------------------------

def _rng(seed):
    return np.random.default_rng([seed & 0x7fffffff, 77])


def _dims(case):
    return (case["nx"], case["ny"], case["nz"])


def _uneven(rng, P, lo, hi):
    """Body plans on ragged grids: the voxels nearest (in a noisy distance) to a random seed voxel,
    a fraction U[0.3, 0.9] of each grid, materials uniform over the four non-empty ones."""
    dims, grids = rng.integers(lo, hi + 1, size=(P, 3)).astype(np.int32), []
    for nx, ny, nz in dims:
        V = int(nx) * int(ny) * int(nz)
        k, j, i = np.unravel_index(np.arange(V), (nz, ny, nx))
        c = rng.integers(0, (nx, ny, nz))
        far = np.abs(i - c[0]) + np.abs(j - c[1]) + np.abs(k - c[2]) + 2.0 * rng.random(V)
        n = max(1, int(rng.uniform(0.3, 0.9) * V))
        mat = rng.integers(1, W.N_MAT, size=V, dtype=np.uint8)
        mat[np.argpartition(far, n - 1)[n:]] = 0
        grids.append(mat)
    return dims, np.concatenate(grids)


def _materials(rng, case):
    """Every voxel uniform over the five materials (fill 0), or occupied with probability `fill`."""
    n = case["robots"] * case["nx"] * case["ny"] * case["nz"]
    if case["fill"] == 0.0:
        return rng.integers(0, W.N_MAT, size=n, dtype=np.uint8)
    mat = rng.integers(1, W.N_MAT, size=n, dtype=np.uint8)
    mat[rng.random(n, dtype=np.float32) >= case["fill"]] = 0
    return mat


def _params(rng, case):
    """Fixed morphologies with per-voxel weight, stiffness and phase (the differentiation workload)."""
    mat = _materials(rng, dict(case, fill=0.0))
    n = mat.size
    w = rng.uniform(0.5, 1.0, n).astype(np.float32)
    kappa = np.asarray(W.CONFIG.k_mat, np.float32)[mat]
    phi = np.asarray(W.CONFIG.phase_mat, np.float32)[mat] + rng.uniform(-0.5, 0.5, n).astype(np.float32)
    return mat, w, kappa, phi.astype(np.float32)


def _inputs(case, seed):
    """The case's arrays on the host, from the seed alone."""
    rng, kind = _rng(seed), case["kind"]
    P = case["robots"]
    if kind == "evaluate":
        return dict(dims=np.tile(np.asarray(_dims(case), np.int32), (P, 1)), mats=_materials(rng, case))
    if kind == "uneven":
        dims, mats = _uneven(rng, P, case["lo"], case["hi"])
        return dict(dims=dims, mats=mats)
    if kind == "paper":
        mats = _materials(rng, dict(case, fill=0.0))
        return dict(dims=np.tile(np.asarray(_dims(case), np.int32), (P, 1)), mats=mats,
                    genomes=W.one_hot_logits(mats).reshape(P, -1))
    if kind in ("gradient", "lamarckian"):
        mat, w, kappa, phi = _params(rng, case)
        return dict(dims=np.tile(np.asarray(_dims(case), np.int32), (P, 1)), mats=mat, w=w, kappa=kappa, phi=phi)
    raise ValueError(kind)


def _mlp_genomes(seed, P):
    """MLP genomes (each layer uniform in +-1/sqrt(fan_in)) and the encoding matrix, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7fffffff)
    scale = torch.cat([torch.full((i * o + o,), 1.0 / math.sqrt(i)) for i, o in W.LAYERS]).cuda()
    genomes = (torch.rand(P, GENOME, generator=g, device="cuda") * 2 - 1) * scale
    return genomes, 2.0 * torch.randn(W.PE_M, 3, generator=g, device="cuda")


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


class State:
    pass


def prepare(case, seed):
    s, kind, P = State(), case["kind"], case["robots"]
    s.case = case
    if kind == "evolve":
        g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7fffffff)
        s.genomes = torch.randn(P, case["genes"], generator=g, device="cuda") * 0.1
        s.out = torch.empty_like(s.genomes)
        s.fitness = torch.randn(P, generator=g, device="cuda", dtype=torch.float64)
        s.sim = vs.Simulator(W.CONFIG)
        return s
    s.sim = vs.Simulator(W.PAPER if kind == "paper" else W.CONFIG)
    if kind == "codesign":
        s.genomes, s.B = _mlp_genomes(seed, P)
        return s
    d = _inputs(case, seed)
    s.dims = d["dims"]
    s.fitness = torch.empty(P, dtype=torch.float64, device="cuda")
    if kind in ("evaluate", "uneven"):
        s.mats = d["mats"] if case.get("where", "host") == "host" else _gpu(d["mats"])
    elif kind == "paper":
        s.genomes = _gpu(d["genomes"])
        s.out = torch.empty_like(s.genomes)
    elif kind == "gradient":
        s.mats = _gpu(d["mats"])
        s.leaves = [_gpu(d[k]).requires_grad_(True) for k in ("w", "kappa", "phi")]
        s.weights = _gpu(_rng(seed + 1).uniform(0.5, 1.5, P))
        s.function = vs.fitness_function()
    else:
        s.mats = _gpu(d["mats"])
        s.rows = _gpu(np.concatenate([d[k].reshape(P, -1) for k in ("w", "kappa", "phi")], axis=1))
        s.bounds = codesign.param_bounds(s.rows.shape[1] // 3)
    return s


def run(s):
    c, sim = s.case, s.sim
    kind = c["kind"]
    if kind in ("evaluate", "uneven"):
        sim.set_population(s.dims, s.mats)
        sim.step(c["steps"])
        if c.get("where", "host") == "host":
            fitness = sim.fitness()
        else:
            fitness = sim.fitness(s.fitness)
        masses, springs = sim.counts()
        return dict(fitness=fitness, masses=masses, springs=springs)
    if kind == "paper":
        sim.set_population(s.dims, s.genomes, vs.MODE_LOGITS)
        sim.step(c["steps"])
        sim.fitness(s.fitness)
        sim.evo_generation(s.fitness, s.genomes, s.out, W.PAPER_EVOLUTION, 0)
        return dict(fitness=s.fitness, genomes=s.out)
    if kind == "codesign":
        records, genomes = codesign.run(sim, s.genomes, s.B, _dims(c), 1, c["steps"])
        r = records[0]
        return dict(best=r.best, mean=r.mean, median=r.median, dead=r.dead, spring_updates=r.spring_updates,
                    genome_diversity=r.genome_diversity, morphology_diversity=r.morphology_diversity,
                    genomes=genomes)
    if kind == "gradient":
        f = s.function.apply(sim, s.dims, s.mats, *s.leaves, c["steps"], c["every"])
        return dict(fitness=f.detach(), gradients=list(torch.autograd.grad((f * s.weights).sum(), s.leaves)))
    if kind == "lamarckian":
        rows = s.rows.clone()            # the loop moves the elites' rows in place
        _, bred = codesign.run_lamarckian(sim, s.mats, rows, _dims(c), 1, c["steps"], eta=(1e-2, 1e4, 1e-2),
                                          checkpoint=c["every"], bounds=s.bounds, log=False)
        return dict(moved=rows, bred=bred)
    sim.evo_generation(s.fitness, s.genomes, s.out, W.Evolution(), 3)
    return dict(genomes=s.out)


# ------------------------------------------------------------------------------------------
# What a pass cannot do without
# ------------------------------------------------------------------------------------------

def _springs(nx, ny, nz, p):
    """Expected springs and masses of a grid whose voxels are kept with probability p."""
    X, Y, Z = nx + 1, ny + 1, nz + 1
    edges = nx * Y * Z + ny * X * Z + nz * X * Y
    faces = 2 * (nx * ny * Z + nx * nz * Y + ny * nz * X)
    s = edges * (1 - (1 - p) ** 4) + faces * (1 - (1 - p) ** 2) + 4 * nx * ny * nz * p
    return s, X * Y * Z * (1 - (1 - p) ** 8)


def work(case):
    P, kind = case["robots"], case["kind"]
    if kind == "evolve":
        n = P * case["genes"]
        return dict(bytes=8 * n + 8 * P, flops=2 * n)
    steps = case["steps"]
    if kind == "uneven":
        a = 0.5 * (case["lo"] + case["hi"])
        nx = ny = nz = a
        p = 0.6
    else:
        nx, ny, nz = _dims(case)
        p = case.get("fill") or 0.8
        if kind == "codesign":
            p = 0.7
    S, M = (P * v for v in _springs(nx, ny, nz, p))
    V = P * nx * ny * nz
    size = {"evaluate": 1, "uneven": 1, "paper": 40, "codesign": 0, "gradient": 25, "lamarckian": 37}[kind] * V
    if kind == "codesign":
        size = 8 * P * GENOME
    passes = 3 if kind in ("gradient", "lamarckian") else 1
    flops = passes * steps * (45.0 * S + 30.0 * M)
    if kind == "codesign":
        flops += 2.0 * V * sum(i * o for i, o in W.LAYERS)
    # a robot of more than 10,000 corners does not stay on chip: its springs' parameters and its
    # masses' state go through device memory every step
    if (nx + 1) * (ny + 1) * (nz + 1) > 10000:
        size += passes * steps * (12.0 * S + 64.0 * M)
    return dict(bytes=size + 8 * P, flops=flops)


# ------------------------------------------------------------------------------------------
# The same results in 64 bits
# ------------------------------------------------------------------------------------------

def _largest_component(mat):
    """mat [P, nz, ny, nx]: only the largest face-connected component of occupied voxels (ties: the
    one holding the smallest voxel index)."""
    P, V = mat.shape[0], mat[0].numel()
    big = V + 1
    occ = mat > 0
    lab = torch.where(occ, torch.arange(V, device=mat.device).reshape(mat.shape[1:]).expand_as(mat), big)
    while True:
        m = lab.clone()
        for ax in (1, 2, 3):
            n = lab.shape[ax]
            if n > 1:
                lo, hi = lab.narrow(ax, 0, n - 1), lab.narrow(ax, 1, n - 1)
                m.narrow(ax, 0, n - 1).copy_(torch.minimum(m.narrow(ax, 0, n - 1), hi))
                m.narrow(ax, 1, n - 1).copy_(torch.minimum(m.narrow(ax, 1, n - 1), lo))
        m = torch.where(occ, m, big)
        flat = torch.cat([m.reshape(P, V), torch.full((P, 2), big, device=mat.device)], 1)
        m = torch.minimum(m, torch.gather(flat, 1, m.reshape(P, V)).reshape(m.shape))
        m = torch.where(occ, m, big)
        if torch.equal(m, lab):
            break
        lab = m
    count = torch.zeros(P, V + 2, dtype=torch.int64, device=mat.device)
    count.scatter_add_(1, lab.reshape(P, V), torch.ones_like(lab.reshape(P, V)))
    count[:, V:] = 0
    best = count.argmax(1)              # the first of the largest
    return torch.where(occ & (lab == best.reshape(P, 1, 1, 1)), mat, torch.zeros_like(mat))


def _ends(d):
    """Slices (z, y, x) of the two ends of the springs along direction d."""
    a, b = [], []
    for o in (d[2], d[1], d[0]):
        lo, hi, al = slice(None, -1), slice(1, None), slice(None)
        a.append(al if o == 0 else (lo if o > 0 else hi))
        b.append(al if o == 0 else (hi if o > 0 else lo))
    return tuple(a), tuple(b)


def _around(v, d):
    """Sum of a per-voxel quantity over the voxels that hold both ends of each spring along d."""
    for ax, o in ((1, d[2]), (2, d[1]), (3, d[0])):
        if o == 0:
            pad = list(v.shape)
            pad[ax] = 1
            z = torch.zeros(pad, dtype=v.dtype, device=v.device)
            v = torch.cat([v, z], ax) + torch.cat([z, v], ax)
    return v


class _Exact:
    """A batch of robots on one grid shape, in float64."""

    def __init__(self, mat, phys):
        self.phys = phys
        self.mat = _largest_component(mat)
        kept = (self.mat > 0).double()
        self.kept = kept
        self.mass = torch.zeros([s + (1 if i else 0) for i, s in enumerate(mat.shape)], dtype=torch.bool,
                                device=mat.device)
        for dz in (0, 1):
            for dy in (0, 1):
                for dx in (0, 1):
                    n = mat.shape
                    self.mass[:, dz:dz + n[1], dy:dy + n[2], dx:dx + n[3]] |= self.mat > 0
        self.M = self.mass.flatten(1).sum(1)
        n = [_around(kept, d) for d in DIRS]
        self.share = [torch.where(c > 0, 1.0 / c.clamp(min=1), torch.zeros_like(c)) for c in n]
        self.S = sum((c > 0).flatten(1).sum(1) for c in n)
        layer = torch.arange(self.mass.shape[1], device=mat.device).reshape(1, -1, 1, 1)
        low = torch.where(self.mass, layer, 1 << 30).flatten(1).min(1).values.reshape(-1, 1, 1, 1)
        self.z0 = ((layer - low) * phys.edge).double().expand_as(self.mass)

    def springs(self, w, kappa, phi):
        """Per direction (k, alpha, beta): means over the kept voxels that share the spring."""
        amp = torch.tensor(self.phys.amp_mat, dtype=torch.float64, device=w.device)[self.mat.long()]
        k, al, be = w * kappa * self.kept, w * amp * torch.cos(phi) * self.kept, w * amp * torch.sin(phi) * self.kept
        return [tuple(_around(q, d) * self.share[i] for q in (k, al, be)) for i, d in enumerate(DIRS)]

    def step(self, u, v, springs, n):
        """u, v [3, P, z, y, x] after one more step."""
        p = self.phys
        t = n * p.dt
        sn, cs = math.sin(2 * math.pi * p.freq * t), math.cos(2 * math.pi * p.freq * t)
        F = torch.zeros_like(u)
        for d, (k, al, be) in zip(DIRS, springs):
            a, b = _ends(d)
            sa, sb = (slice(None), slice(None)) + a, (slice(None), slice(None)) + b
            d0 = torch.tensor(d, dtype=torch.float64, device=u.device).reshape(3, 1, 1, 1, 1) * p.edge
            L0 = p.edge * math.sqrt(sum(o * o for o in d))
            du = u[sb] - u[sa]
            num = ((2 * d0 + du) * du).sum(0)
            ln = torch.sqrt(L0 * L0 + num)
            f = k * (num / (ln + L0) - L0 * (al * sn + be * cs)) / ln
            if p.spring_zeta > 0:
                dv = v[sb] - v[sa]
                f = f + 2 * p.spring_zeta * torch.sqrt(k * p.mass / 2) * ((d0 + du) * dv).sum(0) / (ln * ln)
            g = f * (d0 + du)
            F[sa] += g
            F[sb] -= g
        Fx, Fy, Fz = F
        Fz = Fz - p.mass * p.gravity
        z = self.z0 + u[2]
        down = (z < 0) & self.mass
        fn = torch.where(down, -z * p.k_ground, torch.zeros_like(z))
        Fz = Fz + fn
        if p.ground_zeta > 0:
            cg = 2 * p.ground_zeta * math.sqrt(p.k_ground * p.mass)
            Fz = Fz - torch.where(down, cg * v[2], torch.zeros_like(z))
        fh2 = Fx * Fx + Fy * Fy
        fh = torch.sqrt(torch.where(fh2 > 0, fh2, torch.ones_like(fh2)))
        stick = down & (torch.where(fh2 > 0, fh, torch.zeros_like(fh)) <= p.mu_s * fn)
        left = torch.where(down, (1 - p.mu_k * fn / fh).clamp(min=0), torch.ones_like(fh))
        zero = torch.zeros_like(fh)
        Fx, Fy = torch.where(stick, zero, Fx * left), torch.where(stick, zero, Fy * left)
        vx, vy = torch.where(stick, zero, v[0]), torch.where(stick, zero, v[1])
        v = p.damping * (torch.stack([vx, vy, v[2]]) + (p.dt / p.mass) * torch.stack([Fx, Fy, Fz]))
        v = v * self.mass
        return u + p.dt * v, v

    def start(self):
        u = torch.zeros((3,) + tuple(self.mass.shape), dtype=torch.float64, device=self.mass.device)
        return u, torch.zeros_like(u)

    def fitness(self, u):
        return torch.where(self.M > 0, (u[0] * self.mass).flatten(1).sum(1) / self.M.clamp(min=1),
                           torch.zeros_like(self.M, dtype=torch.float64))


def _padded(dims, mats):
    """All robots on one grid: the voxels past a robot's own grid are empty."""
    n = dims.max(0)
    out = np.zeros((len(dims), n[2], n[1], n[0]), np.uint8)
    o = 0
    for r, (nx, ny, nz) in enumerate(dims):
        V = int(nx) * int(ny) * int(nz)
        out[r, :nz, :ny, :nx] = mats[o:o + V].reshape(nz, ny, nx)
        o += V
    return _gpu(out)


def _table(values, mat):
    """Per-voxel constants as the library takes them: rounded to float32."""
    return torch.tensor(values, dtype=torch.float32, device=mat.device).double()[mat.long()]


def _draws(seed, gen, child, gene, purpose):
    """High 32 bits of SplitMix64 output ((((gen << 16 | child) << 26 | gene) << 3) | purpose)."""
    with np.errstate(over="ignore"):
        ctr = ((((np.uint64(gen) << np.uint64(16)) | child) << np.uint64(26) | gene) << np.uint64(3)) | np.uint64(purpose)
        z = np.uint64(seed) + (ctr + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return (z ^ (z >> np.uint64(31))) >> np.uint64(32)


def _bred(fitness, genomes, evo, gen):
    """The genetic operators in 64 bits (uniform crossover for every child)."""
    P, G = genomes.shape
    E = evo.elites(P)
    order = np.argsort(-np.where(np.isnan(fitness), -np.inf, fitness), kind="stable")
    out = np.empty((P, G))
    out[:E] = genomes[order[:E]]
    gene = np.arange(G, dtype=np.uint64)
    for c in range(E, P):
        cu = np.uint64(c)
        pa, pb = (order[int(_draws(evo.seed, gen, cu, np.uint64(0), q)) * E >> 32] for q in (0, 1))
        row = np.where(_draws(evo.seed, gen, cu, gene, 2) >> np.uint64(31) == 1, genomes[pa], genomes[pb])
        hit = np.flatnonzero(_draws(evo.seed, gen, cu, gene, 3) < evo.mut_threshold())
        h = hit.astype(np.uint64)
        u1 = (_draws(evo.seed, gen, cu, h, 4).astype(np.float64) + 1) / 2.0 ** 32
        u2 = _draws(evo.seed, gen, cu, h, 5).astype(np.float64) / 2.0 ** 32
        row = row.astype(np.float64)
        row[hit] += evo.sigma * np.sqrt(-2 * np.log(u1)) * np.cos(2 * np.pi * u2)
        out[c] = row
    return out


def _spread(g):
    P = g.shape[0]
    return math.sqrt(2.0 * float((g.double() - g.double().mean(0)).square().sum()) / (P - 1))


def exact(case, seed):
    kind, P = case["kind"], case["robots"]
    if kind == "evolve":
        s = prepare(case, seed)
        return dict(genomes=_bred(s.fitness.cpu().numpy(), s.genomes.cpu().numpy(), W.Evolution(), 3))
    if kind == "codesign":
        # the MLP rounds to bfloat16 between its layers, so its near ties and all that follows
        # from them have no 64-bit value
        genomes, _ = _mlp_genomes(seed, P)
        return dict(best=None, mean=None, median=None, dead=None, spring_updates=None,
                    genome_diversity=_spread(genomes), morphology_diversity=None, genomes=None)
    if kind == "lamarckian":
        return None                     # thousands of steps across contact switches
    d = _inputs(case, seed)
    phys = W.PAPER if kind == "paper" else W.CONFIG
    mat = _padded(d["dims"], d["mats"])
    if case["steps"] * mat.numel() > 3e9:
        return None                     # over about 20 seconds
    e = _Exact(mat, phys)
    if kind != "gradient":
        m = _padded(d["dims"], d["mats"])
        springs = e.springs(torch.ones_like(e.kept), _table(phys.k_mat, m), _table(phys.phase_mat, m))
        u, v = e.start()
        for n in range(case["steps"]):
            u, v = e.step(u, v, springs, n)
        f = e.fitness(u)
        if kind == "paper":
            return dict(fitness=f, genomes=None)
        return dict(fitness=f, masses=e.M.int(), springs=e.S.int())
    # gradient: the steps' states, then their transposes from last to first (contact modes fixed)
    shape = mat.shape
    leaves = [_gpu(d[k]).double().reshape(shape).requires_grad_(True) for k in ("w", "kappa", "phi")]
    springs = e.springs(*leaves)
    held = [tuple(q.detach().requires_grad_(True) for q in s) for s in springs]
    flat = [q for s in held for q in s]
    u, v = e.start()
    states = []
    with torch.no_grad():
        for n in range(case["steps"]):
            states.append((u, v))
            u, v = e.step(u, v, held, n)
        f = e.fitness(u)
    weights = _gpu(_rng(seed + 1).uniform(0.5, 1.5, P))
    uf = u.detach().requires_grad_(True)
    gu, = torch.autograd.grad((e.fitness(uf) * weights).sum(), uf)
    gv = torch.zeros_like(gu)
    total = [torch.zeros_like(q) for q in flat]
    for n in reversed(range(case["steps"])):
        a, b = (q.detach().requires_grad_(True) for q in states.pop())
        un, vn = e.step(a, b, held, n)
        gu, gv, *gp = torch.autograd.grad([un, vn], [a, b] + flat, [gu, gv])
        for t, g in zip(total, gp):
            t += g
    grads = torch.autograd.grad([q for s in springs for q in s], leaves, total)
    return dict(fitness=f, gradients=[g.reshape(-1) for g in grads])
