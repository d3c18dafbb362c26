"""More robots than SMs: a call of 64 steps or more runs in segments (per-corner and packed lattice).
The state must be that of calls too short to be cut, bit for bit."""
import numpy as np
import pytest

from paper_2405_00698_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def run(pop, steps):
    from paper_2405_00698_gb300 import voxsim as vs
    sim = vs.Simulator(W.CONFIG)
    sim.set_population_from(pop)
    for n in steps:
        sim.step(n)
    x, v, _ = sim.state()
    sim.close()
    return x, v


@pytest.mark.parametrize("robots, dims, fill", [(200, (6, 9, 5), 0.8), (160, (8, 8, 8), 0.9), (900, (4, 4, 4), 0.7),
                                                (400, (8, 8, 8), 0.3)])
def test_segments_repeat_the_whole_run(robots, dims, fill):
    rng = np.random.default_rng(23)
    pop = W.make_population([dims] * robots, [W.bernoulli_grid(rng, dims, fill) for _ in range(robots)])
    (xa, va), (xb, vb) = run(pop, (165,)), run(pop, (60, 60, 45))
    assert np.array_equal(xa, xb) and np.array_equal(va, vb)
