"""Temporal-blocking launches over many grids, whose arguments travel with the launch for up to
12 and up to 104 grids of a group and lie in a table on the device beyond that (and for launches of
fewer than four steps): every member equals the same grid stepped alone, bit for bit, and
more strips than fit the arguments equal the whole grid.
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("members", [2, 24, 26, 209, 212])
def test_members_equal_the_grids_alone(members):
    import paper_2204_10323_gb300 as F
    probs = [inputs.random_small(5 + 7 * k % 140, 4 + 5 * k % 37, 40 + k) for k in range(members)]
    ens = F.Ensemble(probs)
    ens.set_kernel(F.KERNEL_TILED, 4)
    ens.step(22)                                      # whole epochs and a launch of two steps
    for k in list(range(0, members, 17)) + [members - 1]:
        sim = F.Sim(probs[k], kernel=F.KERNEL_STREAM)
        sim.step(22)
        for a, b in zip(ens.members[k].state(), sim.state()):
            assert np.array_equal(a, b), k
        sim.close()
    ens.close()


@pytest.mark.parametrize("parts", [12, 13, 105])
def test_many_strips_equal_the_whole_grid(parts):
    import paper_2204_10323_gb300 as F
    p = inputs.random_small(130, 430, 3)
    sim, dec = F.Sim(p, kernel=F.KERNEL_TILED), F.Decomp(p, parts, 4, kernel=F.KERNEL_TILED)
    for s in (sim, dec):
        s.step(26)
        s.sync()
    for a, b in zip(sim.state(), dec.state()):
        assert np.array_equal(a, b)
    sim.close()
    dec.close()
