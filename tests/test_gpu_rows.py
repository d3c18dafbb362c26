"""Robots of more masses than a lattice block's threads on the per-mass kernel of 1024-thread blocks:
one and two passes over the directions, one to three masses per thread, corner counts of either
parity, several robots per SM's queue; against the streamed kernel and the oracle."""
import numpy as np
import pytest

from paper_2405_00698_gb300 import workloads as W

from .parity import check_population

pytestmark = pytest.mark.gpu

# grid, fill: corners, masses
ROBOTS = [((9, 9, 9), 1.0),      # 1000 corners, one mass per thread, one pass
          ((8, 8, 10), 1.0),     # 891 corners (odd)
          ((10, 10, 10), 0.9),   # 1331, two masses per thread
          ((12, 11, 9), 1.0),    # 1560 corners, two passes
          ((12, 12, 12), 1.0),   # 2197 corners, three masses per thread
          ((15, 14, 9), 0.95)]   # 2400 corners


def population(seed, copies=1):
    rng = np.random.default_rng(seed)
    dims = [d for d, _ in ROBOTS for _ in range(copies)]
    return W.make_population(dims, [W.bernoulli_grid(rng, d, f) for d, f in ROBOTS for _ in range(copies)])


def run(pop, steps, **kw):
    from paper_2405_00698_gb300 import voxsim as vs
    sim = vs.Simulator(W.CONFIG, **kw)
    sim.set_population_from(pop)
    for n in steps:
        sim.step(n)
    x, v, off = sim.state()
    f = sim.fitness()
    sim.close()
    return x, v, off, f


@pytest.mark.parametrize("i", range(len(ROBOTS)), ids=[str(d) for d, _ in ROBOTS])
def test_each_size_against_the_oracle(i):
    from oracle import oracle as orc
    orc.build()
    pop = population(21).subset([i, i])
    x, _, off, f = run(pop, (90, 10))
    ref = orc.run_population(pop, W.CONFIG, 100)
    check_population(orc, pop, W.CONFIG, 100, f, x, off, ref)


def test_queue_repeats_and_agrees_with_streamed():
    """200 robots on one persistent launch: the same bits twice, and the streamed kernel's positions
    up to the order of each mass's 26 force terms (float32 displacements of 20 steps, below 1e-3 m)."""
    from paper_2405_00698_gb300 import voxsim as vs
    pop = population(22, copies=34)
    a, b = run(pop, (20,)), run(pop, (20,))
    for p, q in zip(a, b):
        assert np.array_equal(p, q)
    s = run(pop, (20,), path=vs.PATH_STREAMED)
    assert np.array_equal(a[2], s[2])
    assert np.abs(a[0] - s[0]).max() <= 1e-6


def test_segments_repeat_the_whole_run():
    """More robots than SMs: the steps of one call run in segments from 64 steps on; the state must be
    that of calls too short to be cut, bit for bit."""
    pop = population(23, copies=34)
    a, b = run(pop, (165,)), run(pop, (60, 60, 45))
    for p, q in zip(a, b):
        assert np.array_equal(p, q)
