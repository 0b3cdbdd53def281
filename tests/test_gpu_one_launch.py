"""Every step of a call in one launch on lattices of a single tile, where the same
thread block reads every address again two steps after it was rewritten."""
import numpy as np
import pytest

from paper_2407_01651_gb300 import pf
from paper_2407_01651_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 4), (128, 4), (100, 32), (129, 33)])
@pytest.mark.parametrize("precision,thermal", [("fp32", 0), ("fp32", 1), ("fp64", 0), ("fp16", 0)])
def test_one_launch_gives_the_bits_of_single_steps(shape, precision, thermal):
    nx, ny = shape
    sims = []
    for one in (True, False):
        sim = pf.Simulation([shape], dict(wl.BASE_PARAMS, thermal=thermal, g=1e-5), precision)
        sim.set_step_config(1, 32)
        sim.init_fields(0, [(nx / 3, ny / 2, 0.4)], 3.0, [(3 * nx / 4, ny / 2, 3.0)])
        if one:
            sim.set_launch(0, 2)
            sim.step(9)
        else:
            for _ in range(9):
                sim.step(1)
        sims.append(sim)
    assert np.array_equal(sims[0].get_state(), sims[1].get_state())
    f, g = sims[0].fields(), sims[1].fields()
    assert all(np.array_equal(f[k], g[k]) for k in f)
