"""The streamed step's launches: robots named in the launch's arguments (up to 16) or read from their
list, one wave of blocks or several, with and without dashpots.  Every corner's arithmetic is the
same in all of them, so a robot's state does not depend on the others' number: the same bits."""
import numpy as np
import pytest

from paper_2405_00698_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def run(pop, steps, config, **kw):
    from paper_2405_00698_gb300 import voxsim as vs
    sim = vs.Simulator(config, **kw)
    sim.set_population_from(pop)
    sim.step(steps)
    x, v, off = sim.state()
    sim.close()
    return x, v, off


@pytest.mark.parametrize("robots, dims", [(16, [(3, 4, 2), (5, 2, 3)]), (17, [(4, 4, 4), (2, 3, 5), (1, 1, 1)]),
                                          (16, [(21, 21, 21), (9, 20, 17)]), (17, [(21, 21, 21), (20, 22, 19)])])
@pytest.mark.parametrize("config", [W.CONFIG, W.PAPER], ids=["undamped", "damped"])
def test_state_independent_of_the_population(robots, dims, config):
    from paper_2405_00698_gb300 import voxsim as vs
    rng = np.random.default_rng(31)
    grids = [dims[i % len(dims)] for i in range(robots)]
    pop = W.make_population(grids, [W.bernoulli_grid(rng, d, 0.8) for d in grids])
    x, v, off = run(pop, 13, config, path=vs.PATH_STREAMED)
    for i in (0, robots - 1):
        xs, vs_, _ = run(pop.subset([i]), 13, config, path=vs.PATH_STREAMED)
        assert np.array_equal(x[off[i]:off[i + 1]], xs)
        assert np.array_equal(v[off[i]:off[i + 1]], vs_)
