"""The lattice kernels chosen by population size and grid: several threads per mass when robots leave
SMs idle, and compile-time row strides for robots of at most 8 voxels along each axis.  Both give
the streamed kernel's bits (one thread per corner, every spring evaluated at both ends in the same
order)."""
import numpy as np
import pytest

from paper_2405_00698_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# full grids: 256 masses (four threads each), 288 and 320 (three), 343, 504 and 512 (two)
ROLES = [(7, 7, 3), (7, 5, 5), (7, 7, 4), (6, 6, 6), (8, 7, 6), (7, 7, 7), (1, 1, 1)]
GRID8 = [(8, 8, 8), (7, 8, 8), (8, 7, 8), (8, 8, 6), (5, 8, 8)]


def population(dims, fill, seed):
    rng = np.random.default_rng(seed)
    return W.make_population(dims, [W.bernoulli_grid(rng, d, fill) for d in dims])


def run(pop, phys, steps, **kw):
    from paper_2405_00698_gb300 import voxsim as vs
    sim = vs.Simulator(phys, **kw)
    sim.set_population_from(pop)
    for n in steps:
        sim.step(n)
    x, v, off = sim.state()
    f = sim.fitness()
    sim.close()
    return x, v, off, f


@pytest.mark.parametrize("phys", [W.CONFIG, W.PAPER], ids=["config", "paper"])
@pytest.mark.parametrize("dims", ROLES, ids=str)
def test_several_threads_per_mass(dims, phys):
    from paper_2405_00698_gb300 import voxsim as vs
    pop = population([dims] * 3 + [(2, 3, 1)], 1.0, 11)
    a = run(pop, phys, (60, 7))
    b = run(pop, phys, (60, 7), path=vs.PATH_STREAMED)
    for p, q in zip(a, b):
        assert np.array_equal(p, q)


def test_one_too_many_masses_keeps_the_plain_kernel():
    from paper_2405_00698_gb300 import voxsim as vs
    pop = population([(7, 7, 8), (7, 7, 3)], 1.0, 12)      # 576 masses: no second thread fits
    a = run(pop, W.CONFIG, (50,))
    b = run(pop, W.CONFIG, (50,), path=vs.PATH_STREAMED)
    for p, q in zip(a, b):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("steps", [(40, 3), (600,)], ids=["whole", "segments"])
def test_compile_time_strides(steps):
    from paper_2405_00698_gb300 import voxsim as vs
    pop = population(GRID8 * 40, 0.8, 13)
    a = run(pop, W.CONFIG, steps)
    b = run(pop, W.CONFIG, steps, path=vs.PATH_STREAMED)
    for p, q in zip(a, b):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("copies", [1, 40], ids=["several threads per mass", "compile-time strides"])
def test_gradients_on_mixed_grids(copies):
    """The same robots' gradients with and without a small robot beside them, which takes the
    population to the run-time strides.  Only the order of the voxel sums differs: at most 76 springs
    of 3 terms around a voxel, each sum off by half a unit in the last place per term."""
    import torch
    from paper_2405_00698_gb300 import voxsim as vs
    got = []
    for extra in ([], [(3, 3, 3)]):
        dims = [d for d in GRID8 for _ in range(copies)]
        pop = population(dims + extra, 0.7, 14)            # (the same robots first)
        full = population(dims + [(3, 3, 3)], 0.7, 14)
        w, kappa, phi = (q[:pop.mats.size] for q in W.voxel_params(np.random.default_rng(15), full))
        sim = vs.Simulator(W.CONFIG)
        leaves = [torch.from_numpy(q).cuda() for q in (w, kappa, phi)]
        sim.set_checkpointing(20)
        sim.set_population(pop.dims, (torch.from_numpy(pop.mats).cuda(), *leaves), vs.MODE_PARAMS)
        sim.step(50)
        g = [torch.empty_like(q) for q in leaves]
        dl = torch.ones(pop.P, dtype=torch.float64, device="cuda")
        sim.backward(dl, *g)
        n = int(pop.voxel_off[len(dims)])
        got.append([q[:n].cpu().numpy() for q in g])
        sim.close()
    for p, q in zip(*got):
        assert np.abs(p - q).max() <= 228 * 2.0 ** -24 * np.abs(q).max()
