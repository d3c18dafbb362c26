"""Host materials are checked eight at a time: an id out of range is found wherever it stands."""
import numpy as np
import pytest

from paper_2405_00698_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 8, 9, 27])
@pytest.mark.parametrize("bad", [5, 127, 128, 132, 255])
def test_out_of_range_ids_are_refused(n, bad):
    from paper_2405_00698_gb300 import voxsim as vs
    sim = vs.Simulator(W.CONFIG)
    for at in range(n):
        m = np.full(n, 4, np.uint8)
        m[at] = bad
        with pytest.raises(vs.VoxsimError) as e:
            sim.set_population([(n, 1, 1)], m)
        assert e.value.status == vs.SIM_EINVAL and f"id {bad} at voxel {at}" in str(e.value)
    sim.set_population([(n, 1, 1)], np.full(n, 4, np.uint8))
    assert sim.counts()[0][0] == 4 * (n + 1)
    sim.close()
