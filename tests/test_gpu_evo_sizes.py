"""The genetic operators and the diversity where their loops end: populations and genomes around the
blocks' and warps' sizes, mutation rates that fill or never fill a warp's queue, ties and NaN in the
ranking."""
import numpy as np
import pytest

from paper_2405_00698_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (population, genes, mutation rate, crossover rate)
SIZES = [(1, 1, 0.1, 1.0), (2, 31, 1.0, 1.0), (33, 33, 0.5, 0.4), (31, 2047, 0.1, 1.0), (32, 2048, 0.0, 1.0),
         (65, 2049, 0.9, 1.0), (257, 300, 0.1, 0.4), (300, 65, 1.0, 1.0)]


@pytest.mark.parametrize("P,G,rate,cross", SIZES)
def test_generation_against_the_oracle(P, G, rate, cross):
    import torch
    from oracle import oracle as orc
    from paper_2405_00698_gb300 import voxsim as vs
    orc.build()
    rng = np.random.default_rng(P * 1000 + G)
    g = rng.standard_normal((P, G)).astype(np.float32)
    f = rng.integers(0, max(2, P // 3), P).astype(np.float64)      # ties
    f[rng.integers(0, P, P // 8)] = np.nan
    f[rng.integers(0, P, P // 8)] = -np.inf
    f[rng.integers(0, P, P // 8)] = -0.0
    evo = W.Evolution(mut_rate=rate, cross_rate=cross)
    sim = vs.Simulator(W.CONFIG)
    out = torch.empty(P, G, device="cuda")
    parents = torch.empty(P, 2, dtype=torch.int32, device="cuda")
    mask = torch.empty(P, G, dtype=torch.uint8, device="cuda")
    sim.evo_generation(torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda(), out, evo, 5, parents, mask)
    ref = orc.evo_generation(f, g, evo.elites(P), evo.seed, 5, evo.mut_threshold(), evo.sigma,
                             keep_threshold=evo.keep_threshold())
    assert np.array_equal(parents.cpu().numpy(), ref["parents"])
    assert np.array_equal(mask.cpu().numpy(), ref["mask"])
    # sigma sqrt(-2 ln u) <= 0.05 * 6.7, its float32 functions off by a few units in the last place
    assert np.allclose(out.cpu().numpy(), ref["genomes"], rtol=1e-6, atol=1e-6)
    sim.close()


@pytest.mark.parametrize("P,dims,G", [(2, (1, 1, 1), 1), (7, (3, 11, 1), 33), (33, (4, 4, 5), 31), (100, (8, 8, 8), 500)])
def test_diversity(P, dims, G):
    import torch
    from oracle import oracle as orc
    from paper_2405_00698_gb300 import voxsim as vs
    orc.build()
    rng = np.random.default_rng(P)
    pop = W.population_uniform(P, dims, P)
    g = rng.standard_normal((P, G)).astype(np.float32)
    sim = vs.Simulator(W.CONFIG)
    sim.set_population_from(pop)
    genome, morph = sim.diversity(torch.from_numpy(g).cuda())
    kept = sim.voxels()["kept"].reshape(P, -1)
    sim.close()
    assert abs(genome - orc.genome_diversity(g)) <= 1e-12 * genome
    assert abs(morph - orc.morphology_diversity(kept)) <= 1e-12
